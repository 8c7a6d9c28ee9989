"""The gather of dense tiles where a block takes several chunks of 1024 pieces in
turn (more chunks than blocks for them, 608), of tiles at the box's faces and
inside: a particle's sums don't depend on the others, so that all particles and a
sparse part of them give the same bits; the part against the oracle to the FP32
bound of the parity tests, 1e-5 relative L2.
"""

import dataclasses
import math

import numpy as np
import pytest

import erpp_inputs as I

pytestmark = pytest.mark.gpu
DX = 2 * math.pi / 64


@pytest.fixture(scope="module")
def erpp(oracle_lib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1405_6969_gb300 as pkg
    return pkg


@pytest.mark.parametrize("n,sigma", [((192, 64, 24), 1.0), ((192, 64, 24), 1.5),
                                     ((181, 57, 23), 1.0)])
def test_many_chunks(erpp, oracle_lib, n, sigma):
    import torch
    w = dataclasses.replace(I.CFG_SMALL, n=n, L=tuple(v * DX for v in n), sigma_over_dx=sigma,
                            kmax=2.0)
    rng = np.random.default_rng(4)
    corners = np.array([[0, 0, 0], [80, 34, 10], [170, 20, 15], [100, 50, 18]]).T[:, :, None]
    x = ((corners + np.array([8, 6, 4])[:, None, None] * rng.random((3, 4, 60000))) *
         DX * (1 - 1e-9)).reshape(3, -1)
    u = np.random.default_rng(5).standard_normal((3,) + n[::-1]).astype(np.float32)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()  # noqa: E731
    ctx = erpp.Context(w.params(), precision="fp32")
    up = ctx.interpolate(cu(u), cu(x))
    few = np.ascontiguousarray(x[:, ::600])
    alone = ctx.interpolate(cu(u), cu(few))
    ctx.check()
    assert torch.equal(alone, up[:, ::600])
    ref = oracle_lib.gather(w.params(), few, u.astype(np.float64))
    assert float(np.linalg.norm(alone.cpu().numpy() - ref) / np.linalg.norm(ref)) < 1e-5

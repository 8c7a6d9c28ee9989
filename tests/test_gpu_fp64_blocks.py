"""The plain FP64 kernels' two block sizes (8 particles for at most 50000, else 32):
a particle's sums don't depend on its block, so that gathers of 50000 and of 50001
particles agree bit for bit on those they share, and sources to the rounding of
atomic additions.

Tolerance: the FP64 bound of the parity tests, 1e-12 relative L2.
"""

import dataclasses
import math

import numpy as np
import pytest

import erpp_inputs as I

pytestmark = pytest.mark.gpu

MANY = 50001


@pytest.fixture(scope="module")
def erpp(oracle_lib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1405_6969_gb300 as pkg
    return pkg


def rel(a, b):
    return float(np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b))


@pytest.mark.parametrize("normalize", [True, False])
@pytest.mark.parametrize("n,sigma", [((34, 33, 40), 1.0), ((7, 40, 9), 1.0), ((40, 37, 36), 2.5),
                                     ((64, 36, 40), 5.0)])
def test_block_sizes(erpp, oracle_lib, n, sigma, normalize):
    import torch
    dx = 2 * math.pi / 64
    w = dataclasses.replace(I.CFG_SMALL, n=n, L=tuple(v * dx for v in n), sigma_over_dx=sigma,
                            shear_rate=0.3)
    p = w.params(normalize=normalize)
    rng = np.random.default_rng(1)
    x = rng.random((3, MANY)) * np.array(w.L)[:, None] * (1 - 1e-12)
    x[1, 77] = np.nan  # reported and left out
    D = rng.standard_normal(x.shape)
    u = rng.standard_normal((3,) + n[::-1])
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()  # noqa: E731
    ctx = erpp.Context(w.params(), precision="fp64", normalize=normalize)
    many, few = ctx.interpolate(cu(u), cu(x)), ctx.interpolate(cu(u), cu(x[:, :-1]))
    ok = torch.arange(MANY - 1, device="cuda") != 77
    assert torch.equal(many[:, :-1][:, ok], few[:, ok])
    some = np.r_[0:70, 78:200, MANY - 70:MANY]
    assert rel(many[:, torch.as_tensor(some).cuda()],
               oracle_lib.gather(p, np.ascontiguousarray(x[:, some]), u)) < 1e-12
    x[1, 77] = 0.0
    ref = oracle_lib.scatter(p, np.ascontiguousarray(x[:, :300]), np.ascontiguousarray(D[:, :300]))
    D[:, 300:] = 0.0
    with pytest.raises(erpp.ErppError):
        ctx.check()
    assert rel(ctx.scatter_source(cu(x), cu(D)), ref) < 1e-12
    assert rel(ctx.scatter_source(cu(x[:, :-1]), cu(D[:, :-1])), ref) < 1e-12
    ctx.check()

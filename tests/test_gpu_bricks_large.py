"""Bricks beyond those that one scan kernel takes (131072): the source and the adjoint
of a box of 132000, against the tile kernels (FP32 bound of the parity tests, 1e-5
relative L2) and the warp-per-particle kernel (the same bits).
"""

import dataclasses
import math

import numpy as np
import pytest

import erpp_inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def erpp(oracle_lib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1405_6969_gb300 as pkg
    return pkg


def test_more_bricks_than_one_scan(erpp):
    import torch
    n = (8, 2000, 2100)
    assert 8 * math.prod(-(-v // 16) for v in n) > 131072
    w = dataclasses.replace(I.CFG_SMALL, n=n, L=tuple(v * 2 * math.pi / 64 for v in n))
    rng = np.random.default_rng(1)
    x = torch.as_tensor(rng.random((3, 120000)) * np.array(w.L)[:, None] * (1 - 1e-12)).cuda()
    D = torch.as_tensor(rng.standard_normal(x.shape)).cuda()
    R = torch.randn((3,) + n[::-1], device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    got = []
    for mode in ("merge", "cluster"):
        ctx = erpp.Context(w.params(), precision="fp32")
        ctx.set_scatter_mode(mode)
        S = ctx.scatter_source(x, D)
        assert ctx.debug_last_route() == ({"source"} if mode == "merge" else set())
        dD, dx = ctx.scatter_backward(x, D, R)
        assert ctx.debug_last_route() == ({"adjoint"} if mode == "merge" else set())
        ctx.check()
        got.append((S, dD, dx))
    (S, dD, dx), (T, eD, ex) = got
    assert float((S - T).norm() / T.norm()) < 1e-5
    assert torch.equal(dD, eD) and torch.equal(dx, ex)

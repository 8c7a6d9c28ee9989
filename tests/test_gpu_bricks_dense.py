"""Dense bricks of the source: quarters of a region that nothing reaches beside a
brick of more particles than a list entry can count, and forces that are not finite.

Tolerance: the FP32 bound of the parity tests, 1e-5 relative L2.
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


def box(n, sigma=1.0):
    return dataclasses.replace(I.CFG_SMALL, n=n, L=tuple(v * DX for v in n), sigma_over_dx=sigma)


def cuda(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("sigma", [1.0, 1.5])
def test_untouched_quarters(erpp, oracle_lib, sigma):
    """20000 particles in one plane of cells of one brick."""
    n = (48, 32, 48)
    w = box(n, sigma)
    rng = np.random.default_rng(1)
    x = (np.array([24, 8, 16])[:, None] + np.array([8, 8, 1])[:, None] * rng.random((3, 20000))) * DX
    D = rng.standard_normal(x.shape)
    ctx = erpp.Context(w.params(), precision="fp32")
    S = ctx.scatter_source(cuda(x), cuda(D))
    assert ctx.debug_last_route() == {"source"}
    ctx.check()
    S = S.cpu().numpy()
    ref = oracle_lib.scatter(w.params(), x, D)
    assert rel(S, ref) < 1e-5
    reach = int(math.floor(3 * sigma)) + 1
    inside = np.zeros(n[2], dtype=bool)
    inside[16 - reach:17 + reach + 1] = True
    assert not S[:, ~inside].any() and S[:, 16].any()


# whole regions of several batches, and quarters of dense ones; rows that are no
# multiple of 16 bytes; axes shorter than a region
ODD = [((64, 64, 48), 59000, 1.0), ((24, 20, 18), 18000, 1.0), ((33, 31, 30), 20000, 1.5),
       ((16, 40, 40), 30000, 1.0)]


@pytest.mark.parametrize("n,particles,sigma", ODD, ids=["x".join(map(str, o[0])) for o in ODD])
def test_forces_that_are_not_finite(erpp, oracle_lib, n, particles, sigma):
    """Dense boxes: NaN and infinite components reach the nodes in their particles'
    windows, as in the tiles, and no others; through a step too."""
    import torch
    w = box(n, sigma)
    rng = np.random.default_rng(2)
    x = rng.random((3, particles)) * np.array(w.L)[:, None] * (1 - 1e-12)
    D = rng.standard_normal(x.shape)
    bad = {(0, 5): np.nan, (1, 5): np.inf, (2, 900): -np.inf, (0, 901): np.inf, (0, 902): -np.inf}
    x[:, 902] = x[:, 901]  # their sum is no number
    clean = D.copy()
    for (c, i), v in bad.items():
        D[c, i] = v
        clean[c, i] = 0.0
    got = []
    for mode in ("merge", "cluster"):
        ctx = erpp.Context(w.params(), precision="fp32")
        ctx.set_scatter_mode(mode)
        S = ctx.scatter_source(cuda(x), cuda(D)).cpu().numpy()
        assert ctx.debug_last_route() == ({"source"} if mode == "merge" else set())
        du, _ = ctx.gather_backward(cuda(x), torch.zeros(S.shape, device="cuda"), cuda(D))
        ctx.check()
        got.append((S, du.cpu().numpy()))
    ref = oracle_lib.scatter(w.params(), x, clean)
    for a, b in zip(*got):
        assert np.isnan(a).any() and np.isposinf(a).any() and np.isneginf(a).any()
        for kind in (np.isnan, np.isposinf, np.isneginf):
            assert np.array_equal(kind(a), kind(b))
    fin = np.isfinite(got[0][0])
    assert fin.any() and rel(got[0][0][fin], ref[fin]) < 1e-5
    # a step whose velocity of one particle is infinite
    one = torch.ones(particles, device="cuda", dtype=torch.float64)
    v = 0.01 * clean
    v[2, 77] = np.inf
    masks = []
    for mode in ("merge", "cluster"):
        ctx = erpp.Context(w.params(), precision="fp32")
        ctx.set_scatter_mode(mode)
        P = erpp.ParticleState(cuda(x), cuda(v), cuda(x), cuda(1e-3 * clean), 0.01 * one, 1000 * one)
        masks.append(np.isfinite(ctx.step(torch.zeros(S.shape, device="cuda"), P).cpu().numpy()))
    assert not masks[0].all() and np.array_equal(masks[0], masks[1])


def test_sparse_regions_leave_them_out(erpp, oracle_lib):
    """Fewer than 1024 particles around a region: the other forces' sums alone."""
    w = box((96, 96, 80))
    rng = np.random.default_rng(3)
    x = rng.random((3, 4000)) * np.array(w.L)[:, None] * (1 - 1e-12)
    D = rng.standard_normal(x.shape)
    clean = D.copy()
    D[0, 7], D[1, 8] = np.nan, np.inf
    clean[0, 7] = clean[1, 8] = 0.0
    ctx = erpp.Context(w.params(), precision="fp32")
    S = ctx.scatter_source(cuda(x), cuda(D)).cpu().numpy()
    assert ctx.debug_last_route() == {"source"}
    assert rel(S, oracle_lib.scatter(w.params(), x, clean)) < 1e-5

"""Which calls the brick kernels serve, and the brick adjoint at sizes that it
serves.

The adjoint takes bricks where the particles pay for the sort and for staging
their tiles: sparse clouds and small ones keep the warp-per-particle kernel
(256^3 nodes with 10k particles took 148 us from bricks, 67 with a warp each).  The
cases of the brick tests are checked to run the kernels that they are for.

Tolerance: the FP32 bound of the parity tests, 1e-5 relative L2.
"""

import dataclasses
import math

import numpy as np
import pytest

import erpp_inputs as I

pytestmark = pytest.mark.gpu

TOL = 1e-5
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


def cuda(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def rel(a, b):
    return float(np.linalg.norm(a.cpu().numpy() - b) / max(np.linalg.norm(b), 1e-300))


def cloud(n, particles, sigma=1.0, seed=1, **over):
    w = dataclasses.replace(I.CFG_SMALL, n=n, L=tuple(v * DX for v in n), sigma_over_dx=sigma,
                            shear_rate=0.5, **over)
    rng = np.random.default_rng(seed)
    x = rng.random((3, particles)) * np.array(w.L)[:, None] * (1 - 1e-12)
    return w, x, rng.standard_normal(x.shape)


# box, particles, whether the source and whether the adjoint take bricks
ROUTES = [((96, 96, 80), 40, True, False), ((96, 96, 80), 4999, True, False),
          ((96, 96, 80), 5000, True, True), ((256, 128, 128), 14000, True, False),
          ((256, 128, 128), 15000, True, True), ((90, 83, 85), 13999, True, False),
          ((90, 83, 85), 14000, True, True), ((131, 128, 128), 32000, True, False),
          ((131, 128, 128), 33000, True, True), ((64, 64, 64), 12000, False, False),
          ((40, 40, 40), 16384, True, True)]


@pytest.mark.parametrize("n,particles,source,adjoint", ROUTES,
                         ids=["x".join(map(str, r[0])) + f"_{r[1]}" for r in ROUTES])
def test_routes(erpp, n, particles, source, adjoint):
    import torch
    w, x, D = cloud(n, particles)
    ctx = erpp.Context(w.params(), precision="fp32")
    u = torch.zeros((3,) + n[::-1], dtype=torch.float32, device="cuda")
    want = lambda *on: {k for k, v in zip(("source", "adjoint"), on) if v}  # noqa: E731
    ctx.scatter_source(cuda(x), cuda(D))
    assert ctx.debug_last_route() == want(source, False)
    ctx.scatter_backward(cuda(x), cuda(D), u)
    assert ctx.debug_last_route() == want(False, adjoint)
    ctx.gather_backward(cuda(x), u, cuda(D))
    assert ctx.debug_last_route() == want(source, adjoint)
    ctx.gather_backward(cuda(x), u, cuda(D), need_du=False)
    assert ctx.debug_last_route() == want(False, adjoint)
    # an unaligned field's rows are staged word by word
    buf = torch.zeros(u.numel() + 4, dtype=torch.float32, device="cuda")
    ctx.scatter_backward(cuda(x), cuda(D), buf[1:1 + u.numel()].view_as(u))
    dense = particles >= 14000 and n[0] * n[1] * n[2] * 0.015 <= particles
    assert ctx.debug_last_route() == want(False, adjoint and dense)
    ctx.set_scatter_mode("cluster")
    ctx.gather_backward(cuda(x), u, cuda(D))
    assert not ctx.debug_last_route()
    ctx.check()


def test_brick_tests_run_bricks(erpp):
    """The cases of the brick tests take the source from bricks."""
    from test_gpu_bricks import CASES, positions
    for name, (w, opts) in CASES.items():
        x = positions(w)
        ctx = erpp.Context(w.params(), precision="fp32", **opts)
        ctx.scatter_source(cuda(x), cuda(np.zeros(x.shape)))
        assert ctx.debug_last_route() == {"source"}, name
        ctx.close()


# aligned and odd rows, axes shorter than a brick and one node past a region,
# windows of 2 to 10 nodes, raw weights, unequal spacings; particles enough for
# the adjoint to take bricks
ADJOINT = {
    "ragged_90x83x85": ((90, 83, 85), 14500, {}, {}),
    "even_96x96x80_raw": ((96, 96, 80), 6000, {}, dict(normalize=False)),
    "odd_rows_91x97x81": ((91, 97, 81), 14500, dict(sigma=1.5), {}),
    "even_96x97x81_wide": ((96, 97, 81), 7000, dict(sigma=1.5), {}),
    "thin_x_9x300x170": ((9, 300, 170), 14500, {}, {}),
    "one_past_a_region_17x289x81": ((17, 289, 81), 14500, {}, {}),
    "shorter_than_a_brick_7x160x257": ((7, 160, 257), 14500, {}, {}),
    "shorter_than_a_brick_8x160x257": ((8, 160, 257), 7000, {}, {}),
    "windows_of_two_88x88x81": ((88, 88, 81), 7000, dict(cutoff=1.1), {}),
    "windows_of_ten_88x90x85": ((88, 90, 85), 7000, dict(sigma=1.6), {}),
    "stretched_81x96x90": ((81, 96, 90), 14500, dict(stretch=(1.0, 0.8, 1.3)), {}),
}


@pytest.mark.parametrize("name", ADJOINT)
def test_adjoints(erpp, oracle_lib, name):
    """The bits of the warp-per-particle kernel, and the oracle's values."""
    import torch
    n, particles, over, opts = ADJOINT[name]
    over = dict(over)
    stretch = over.pop("stretch", (1.0, 1.0, 1.0))
    sigma = over.pop("sigma", 1.0)
    w, x, D = cloud(n, particles, sigma, **over)
    w = dataclasses.replace(w, L=tuple(v * DX * s for v, s in zip(n, stretch)))
    # some particles on nodes and next to the upper faces
    L = np.array(w.L)[:, None]
    x = x / (np.array(n)[:, None] * DX) * L
    nodes = np.arange(64) % np.array(n)[:, None]
    x[:, :64] = np.minimum(nodes * (L / np.array(n)[:, None]), np.nextafter(L, 0))
    x[:, 64:66] = np.nextafter(L, 0)
    R = np.random.default_rng(6).standard_normal((3,) + n[::-1]).astype(np.float32)
    got = []
    for mode in ("merge", "cluster"):
        ctx = erpp.Context(w.params(), precision="fp32", **opts)
        ctx.set_scatter_mode(mode)
        dD, dxs = ctx.scatter_backward(cuda(x), cuda(D), cuda(R))
        assert ("adjoint" in ctx.debug_last_route()) == (mode == "merge")
        _, dxg = ctx.gather_backward(cuda(x), cuda(R), cuda(D), need_du=False)
        assert ("adjoint" in ctx.debug_last_route()) == (mode == "merge")
        ctx.check()
        got.append((dD, dxs, dxg))
    for a, b in zip(*got):
        assert torch.equal(a, b)
    p = w.params(**opts)
    rdD, rdx = oracle_lib.scatter_backward(p, x, D, R.astype(np.float64))
    assert rel(got[0][0], rdD) < TOL and rel(got[0][1], rdx) < TOL
    rdx = oracle_lib.gather_backward(p, x, R.astype(np.float64), D)[1]
    assert rel(got[0][2], rdx) < TOL


def test_invalid_particles(erpp):
    """Positions outside the box are reported; their gradients are zeros."""
    import torch
    w, x, D = cloud((90, 83, 85), 14500)
    x[1, 33], x[0, 34], x[2, 35] = np.nan, -1e-3, w.L[2]
    R = np.random.default_rng(8).standard_normal((3, 85, 83, 90)).astype(np.float32)
    ctx = erpp.Context(w.params(), precision="fp32")
    dD, dx = ctx.scatter_backward(cuda(x), cuda(D), cuda(R))
    assert ctx.debug_last_route() == {"adjoint"}
    with pytest.raises(erpp.ErppError):
        ctx.check()
    assert not dD[:, 33:36].any() and not dx[:, 33:36].any()
    assert dD.isfinite().all() and (dD[:, 36:] != 0).all()
    assert torch.isfinite(dx).all()


def test_wait_runs_out(erpp):
    """The bounded wait for the staged field gives up with a status, and the
    next call works."""
    import torch
    w, x, D = cloud((96, 96, 80), 9000)
    R = torch.ones((3, 80, 96, 96), dtype=torch.float32, device="cuda")
    ctx = erpp.Context(w.params(), precision="fp32")
    ctx.debug_set_wait(limit_ns=2_000_000, stall=True)
    ctx.scatter_backward(cuda(x), cuda(D), R)
    with pytest.raises(erpp.ErppError) as ei:
        ctx.check()
    assert ei.value.status == 6  # ERPP_ETIMEOUT
    ctx.debug_set_wait(0, False)
    dD, _ = ctx.scatter_backward(cuda(x), cuda(D), R)
    ctx.check()
    assert dD.isfinite().all()

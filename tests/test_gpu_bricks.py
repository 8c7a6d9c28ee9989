"""The brick kernels (particles sorted by 8^3-cell bricks, erpp_bricks.cu)
against the FP64 oracle where they can go wrong: boxes that are not multiples
of the brick or the 16^3 region, axes shorter than a region (periodic images of
the same brick on both sides), windows of 2 to 10 nodes, dense bricks (more
particles than one staged batch, and than the ordered ones), raw weights,
particles on faces and nodes, values that are not finite.

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


def cuda(a, dtype=None):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype or torch.float64).cuda()


def rel(a, b):
    a = np.asarray(a, dtype=np.float64)
    b = np.asarray(b, dtype=np.float64)
    return float(np.linalg.norm((a - b).ravel()) / max(np.linalg.norm(b.ravel()), 1e-300))


def work(n, particles, sigma=1.0, cloud="uniform", std=0.3, cutoff=3.0, stretch=(1, 1, 1)):
    return dataclasses.replace(I.CFG_SMALL, name="bricks", n=n,
                               L=tuple(v * DX * s for v, s in zip(n, stretch)),
                               n_particles=particles, sigma_over_dx=sigma, cloud=cloud,
                               cluster_std=std, n_clusters=7, kmax=2.0, shear_rate=0.5,
                               cutoff=cutoff)


# at least 120 regions of 16^3 nodes, or a quarter of a particle per node
# and 16384 particles, so that the library's rule takes the brick kernels
CASES = {
    "ragged_90x83x85": (work((90, 83, 85), 5000), {}),
    "even_96x96x80_raw": (work((96, 96, 80), 5000), dict(normalize=False)),
    "few_regions_80x74x90": (work((80, 74, 90), 5000), {}),
    "rows_of_odd_length_91x97x81": (work((91, 97, 81), 9000, 1.5, "clusters"), {}),
    "thin_x_9x300x170": (work((9, 300, 170), 4000), {}),
    "one_past_a_region_17x289x81": (work((17, 289, 81), 4000), {}),
    "shorter_than_a_brick_7x160x257": (work((7, 160, 257), 6000), {}),
    "windows_of_two_88x88x81": (work((88, 88, 81), 5000, cutoff=1.1), {}),
    "windows_of_ten_88x90x85": (work((88, 90, 85), 4000, 1.6), {}),
    "stretched_81x96x90": (work((81, 96, 90), 5000, stretch=(1.0, 0.8, 1.3)), {}),
    "dense_24x20x18": (work((24, 20, 18), 18000), {}),
    "dense_wide_33x31x30": (work((33, 31, 30), 20000, 1.5, "clusters"), {}),
    # whole regions of several batches; dense regions, by quarters, among others
    "several_batches_64x64x48": (work((64, 64, 48), 59000), {}),
    "dense_and_not_64x50x39": (work((64, 50, 39), 32000, 1.0, "clusters", 0.15), {}),
    "one_brick_of_many_16x16x16": (work((16, 16, 16), 30000, 1.0, "clusters", 0.05), {}),
}


def positions(w):
    """The cloud, and particles on nodes, faces and next to the upper faces."""
    x = I.make_particles(w, None).x
    L = np.array(w.L)[:, None]
    n = np.array(w.n)[:, None]
    k = np.arange(40)
    special = np.concatenate([(k % n) * (L / n), ((8 * k) % n) * (L / n),
                              np.nextafter(L, 0) * np.ones((3, 3)), np.zeros((3, 2)),
                              np.array([[-0.0]] * 3)], axis=1)
    return np.concatenate([x, np.minimum(special, np.nextafter(L, 0))], axis=1)


@pytest.mark.parametrize("name", CASES)
def test_source(erpp, oracle_lib, name):
    import torch
    w, opts = CASES[name]
    p = w.params(**opts)
    x = positions(w)
    D = np.random.default_rng(3).standard_normal(x.shape)
    ctx = erpp.Context(w.params(), precision="fp32", **opts)
    S = ctx.scatter_source(cuda(x), cuda(D))
    ctx.check()
    ref = oracle_lib.scatter(p, x, D)
    assert rel(S.cpu().numpy(), ref) < TOL
    # the other halo form goes through the tile kernels
    other = erpp.Context(w.params(), precision="fp32", **opts)
    other.set_scatter_mode("cluster")
    T = other.scatter_source(cuda(x), cuda(D))
    other.check()
    assert rel(T.cpu().numpy(), ref) < TOL
    if "one_brick" not in name:  # bricks of more than 4096 members keep the order of arrival
        S2 = ctx.scatter_source(cuda(x), cuda(D))
        assert torch.equal(S, S2)


def test_source_unaligned_output(erpp, oracle_lib):
    """S at an address that is a multiple of 4 bytes only."""
    import torch
    w, _ = CASES["even_96x96x80_raw"]
    x = positions(w)
    D = np.random.default_rng(4).standard_normal(x.shape)
    ctx = erpp.Context(w.params(), precision="fp32")
    nn = 3 * 96 * 96 * 80
    buf = torch.full((nn + 8,), 7.0, dtype=torch.float32, device="cuda")
    S = buf[1:1 + nn].view(3, 80, 96, 96)
    ctx.scatter_source(cuda(x), cuda(D), S=S)
    ctx.check()
    assert rel(S.cpu().numpy(), oracle_lib.scatter(w.params(), x, D)) < TOL
    assert buf[0].item() == 7.0 and (buf[1 + nn:] == 7.0).all()


def test_invalid_particles_and_forces(erpp, oracle_lib):
    """A particle outside the box or NaN is reported and skipped; a force that
    is not finite gives no source and leaves the others alone."""
    w, _ = CASES["ragged_90x83x85"]
    x = positions(w)
    D = np.random.default_rng(5).standard_normal(x.shape)
    keep = np.ones(x.shape[1], dtype=bool)
    xb = x.copy()
    xb[0, 10] = np.nan
    xb[1, 700] = w.L[1]
    xb[2, 701] = -1e-3
    keep[[10, 700, 701]] = False
    Db = D.copy()
    Db[1, 50] = np.nan
    Db[2, 51] = np.inf
    D0 = D.copy()
    D0[1, 50] = D0[2, 51] = 0.0
    ctx = erpp.Context(w.params(), precision="fp32")
    S = ctx.scatter_source(cuda(xb), cuda(Db))
    with pytest.raises(erpp.ErppError):
        ctx.check()
    ref = oracle_lib.scatter(w.params(), np.ascontiguousarray(x[:, keep]),
                             np.ascontiguousarray(D0[:, keep]))
    assert rel(S.cpu().numpy(), ref) < TOL
    ctx.scatter_source(cuda(x), cuda(np.zeros_like(D)), S=S)
    ctx.check()
    assert not S.any()


def test_gather_of_dense_tiles(erpp, oracle_lib):
    """Tiles of more than 1024 pieces are gathered by several blocks: every
    particle of a cluster inside one tile, next to sparse tiles, equals the
    oracle's and, bit for bit, the gather of the same particle in a sparse
    cloud (its sums do not depend on its neighbours)."""
    import torch
    w = work((72, 40, 24), 6000, 1.0, "clusters", 0.08)
    x = I.make_particles(w, None).x
    grid, _ = I.make_grid(w)
    u = cuda(grid, torch.float32)
    ctx = erpp.Context(w.params(), precision="fp32")
    up = ctx.interpolate(u, cuda(x))
    ctx.check()
    assert rel(up.cpu().numpy(), oracle_lib.gather(w.params(), x, grid)) < TOL
    few = np.ascontiguousarray(x[:, ::60])
    alone = ctx.interpolate(u, cuda(few))
    ctx.check()
    assert torch.equal(alone, up[:, ::60])


ADJOINT = ["ragged_90x83x85", "even_96x96x80_raw", "rows_of_odd_length_91x97x81",
           "thin_x_9x300x170", "one_past_a_region_17x289x81", "shorter_than_a_brick_7x160x257",
           "windows_of_two_88x88x81", "windows_of_ten_88x90x85", "stretched_81x96x90",
           "dense_24x20x18", "dense_wide_33x31x30", "one_brick_of_many_16x16x16"]


@pytest.mark.parametrize("name", ADJOINT)
def test_adjoints(erpp, oracle_lib, name):
    """The adjoints from sorted particles: the bits of the warp-per-particle
    kernel (which contexts in another halo mode keep) and the oracle's values."""
    import torch
    w, opts = CASES[name]
    p = w.params(**opts)
    x = positions(w)
    rng = np.random.default_rng(6)
    D = rng.standard_normal(x.shape)
    R = rng.standard_normal((3,) + tuple(w.n)[::-1]).astype(np.float32)
    got = []
    for mode in ("merge", "cluster"):
        ctx = erpp.Context(w.params(), precision="fp32", **opts)
        ctx.set_scatter_mode(mode)
        dD, dxs = ctx.scatter_backward(cuda(x), cuda(D), cuda(R, torch.float32))
        _, dxg = ctx.gather_backward(cuda(x), cuda(R, torch.float32), cuda(D), need_du=False)
        ctx.check()
        got.append((dD, dxs, dxg))
    for a, b in zip(*got):
        assert torch.equal(a, b)
    rdD, rdx = oracle_lib.scatter_backward(p, x, D, R.astype(np.float64))
    assert rel(got[0][0].cpu().numpy(), rdD) < TOL and rel(got[0][1].cpu().numpy(), rdx) < TOL
    rdx = oracle_lib.gather_backward(p, x, R.astype(np.float64), D)[1]
    assert rel(got[0][2].cpu().numpy(), rdx) < TOL


def test_adjoint_of_invalid_particles(erpp, oracle_lib):
    """A position outside the box is reported; its gradients are zeros."""
    w, _ = CASES["ragged_90x83x85"]
    x = positions(w)
    x[1, 33] = np.nan
    D = np.random.default_rng(7).standard_normal(x.shape)
    R = np.random.default_rng(8).standard_normal((3,) + tuple(w.n)[::-1]).astype(np.float32)
    import torch
    ctx = erpp.Context(w.params(), precision="fp32")
    dD, dx = ctx.scatter_backward(cuda(x), cuda(D), cuda(R, torch.float32))
    with pytest.raises(erpp.ErppError):
        ctx.check()
    assert not dD[:, 33].any() and not dx[:, 33].any()
    assert dD.isfinite().all() and (dD[:, 34:] != 0).all()


def test_adjoint_wait_runs_out(erpp):
    """The bounded wait for the staged field gives up with a status, and the
    next call works."""
    import torch
    w, _ = CASES["even_96x96x80_raw"]
    x = positions(w)
    D = np.ones(x.shape)
    R = torch.ones((3,) + tuple(w.n)[::-1], dtype=torch.float32, device="cuda")
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

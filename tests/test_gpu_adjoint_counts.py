"""The adjoints for the smallest particle counts and around the particles that
a block of the brick adjoint takes (96), in boxes that the brick kernels serve:
uniform clouds, and all particles in one brick (more than 96 there are shared
among blocks); windows of at most 7 nodes and of 9.

Results: the bits of the warp-per-particle kernel, which contexts in another
halo mode keep, and the oracle's values to the FP32 bound of the parity tests,
1e-5 relative L2.
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


def rel(a, b):
    return float(np.linalg.norm(a.cpu().numpy() - b) / max(np.linalg.norm(b), 1e-300))


BOXES = [((96, 96, 80), 1.0), ((90, 83, 85), 1.0), ((91, 97, 81), 1.5)]


@pytest.mark.parametrize("cloud", ["uniform", "one_brick"])
@pytest.mark.parametrize("particles", [1, 31, 95, 96, 97, 193])
@pytest.mark.parametrize("n,sigma", BOXES, ids=["x".join(map(str, b)) for b, _ in BOXES])
def test_few_particles(erpp, oracle_lib, n, sigma, particles, cloud):
    import torch
    w = dataclasses.replace(I.CFG_SMALL, n=n, L=tuple(v * DX for v in n), sigma_over_dx=sigma,
                            n_particles=particles, shear_rate=0.5)
    p = w.params()
    rng = np.random.default_rng(particles)
    side = np.array(w.L)[:, None] if cloud == "uniform" else np.full((3, 1), 8 * DX * (1 - 1e-9))
    x = rng.random((3, particles)) * side
    D = rng.standard_normal(x.shape)
    R = rng.standard_normal((3,) + n[::-1]).astype(np.float32)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()  # noqa: E731
    got = []
    for mode in ("merge", "cluster"):
        ctx = erpp.Context(p, precision="fp32")
        ctx.set_scatter_mode(mode)
        dD, dxs = ctx.scatter_backward(cu(x), cu(D), cu(R))
        du, dxg = ctx.gather_backward(cu(x), cu(R), cu(D))
        ctx.check()
        got.append((dD, dxs, dxg, du))
    for a, b in zip(got[0][:3], got[1][:3]):
        assert torch.equal(a, b)
    dD, dxs, dxg, du = got[0]
    rdD, rdx = oracle_lib.scatter_backward(p, x, D, R.astype(np.float64))
    assert rel(dD, rdD) < TOL and rel(dxs, rdx) < TOL
    rdu, rdx = oracle_lib.gather_backward(p, x, R.astype(np.float64), D)
    assert rel(dxg, rdx) < TOL and rel(du, rdu) < TOL


@pytest.mark.parametrize("sigma", [1.0, 1.5])
def test_blocks_of_many_chunks(erpp, oracle_lib, sigma):
    """More further chunks than blocks for them (608): a block stages tiles at
    the box's faces (copied row by row) and inside (one TMA box) in turn into the
    same shared memory."""
    import torch
    n = (96, 80, 96)
    w = dataclasses.replace(I.CFG_SMALL, n=n, L=tuple(v * DX for v in n), sigma_over_dx=sigma,
                            shear_rate=0.5)
    p = w.params()
    rng = np.random.default_rng(2)
    corners = np.array([[0, 0, 0], [40, 32, 40], [88, 72, 88], [24, 40, 56]]).T[:, :, None]
    x = ((corners + 8 * rng.random((3, 4, 20000))) * DX * (1 - 1e-9)).reshape(3, -1)
    assert sum(c // 96 for c in [20000] * 4) > 608
    D = rng.standard_normal(x.shape)
    R = rng.standard_normal((3,) + n[::-1]).astype(np.float32)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()  # noqa: E731
    got = []
    for mode in ("merge", "cluster"):
        ctx = erpp.Context(p, precision="fp32")
        ctx.set_scatter_mode(mode)
        got.append(ctx.scatter_backward(cu(x), cu(D), cu(R)))
        ctx.check()
    for a, b in zip(*got):
        assert torch.equal(a, b)
    few = np.ascontiguousarray(x[:, ::40])
    rdD, rdx = oracle_lib.scatter_backward(p, few, np.ascontiguousarray(D[:, ::40]),
                                           R.astype(np.float64))
    assert rel(got[0][0][:, ::40], rdD) < TOL and rel(got[0][1][:, ::40], rdx) < TOL

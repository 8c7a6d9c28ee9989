"""The general force's gather (the velocity and its Laplacian) on tiles of
several batches: tiles of 64 x 16 nodes in x and y, whose staged field leaves
shared memory for two blocks per SM with half the pieces a batch only, cut short
at the box's edges, and the smaller tiles of a small box; windows of 6 and of 9
nodes.  A particle's sums don't depend on the others of its tile, so that all
particles together and sixteenths of them, whose tiles hold few pieces, give the
same bits (test_gpu_full_force.py compares with the oracle).
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


@pytest.mark.parametrize("n,particles,sigma", [
    ((128, 33, 20), 16000, 1.0),
    ((70, 18, 9), 9000, 1.0),
    ((128, 20, 18), 9000, 1.5),
    ((30, 32, 28), 9000, 1.0),
])
def test_dense_tiles(erpp, n, particles, sigma):
    import torch
    w = dataclasses.replace(
        I.CFG_SMALL.scaled("ffd", n, particles, L=tuple(k * DX for k in n)),
        radius=0.005, rho_ratio=10.0, sigma_over_dx=sigma, kmax=2.0)
    p = w.params(gravity=(0.0, -0.3, -1.0))
    grid, field = I.make_grid(w)
    u = torch.as_tensor(np.ascontiguousarray(grid), dtype=torch.float32).cuda()
    st = I.make_particles(w, field)

    def steps(at):
        part = dataclasses.replace(
            st, **{k: np.ascontiguousarray(getattr(st, k)[..., at])
                   for k in ("x", "v", "D", "x_prev", "radius", "rho_p") if hasattr(st, k)})
        ctx = erpp.Context(p, precision="fp32", full_force=True)
        ps = erpp.ParticleState.from_numpy(part)
        for k in range(2):
            ctx.step(u, ps, first_step=(k == 0))
        ctx.check()
        return [getattr(ps, name).cpu().numpy() for name in ("x", "v", "D")]

    together = steps(slice(None))
    for q in range(16):
        for a, b in zip(together, steps(slice(q, None, 16))):
            assert np.array_equal(a[..., q::16], b)

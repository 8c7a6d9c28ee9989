"""The plain FP64 kernels at the sizes where their blocks can go wrong: particle
counts around a block's 32, windows of 2 to 31 nodes (rows beyond the buffered
64, one to sixteen lanes rows at a time), axes barely longer than the window,
and the step that keeps the gather's weights for its source.

Tolerance: the FP64 bound of the parity tests, 1e-12 relative L2.
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


def rel(a, b):
    return float(np.linalg.norm(a.cpu().numpy() - b) / max(np.linalg.norm(b), 1e-300))


CASES = [((34, 33, 40), 1, 1.0, 3.0), ((34, 33, 40), 31, 1.0, 3.0), ((34, 33, 40), 33, 1.5, 3.0),
         ((20, 18, 16), 64, 1.0, 1.1), ((40, 37, 36), 97, 2.5, 3.0), ((64, 36, 40), 50, 5.0, 3.0),
         ((7, 40, 9), 200, 1.0, 3.0)]


@pytest.mark.parametrize("n,particles,sigma,cutoff", CASES)
def test_step_and_parts(erpp, oracle_lib, n, particles, sigma, cutoff):
    import torch
    dx = 2 * math.pi / 64
    w = dataclasses.replace(I.CFG_SMALL, n=n, L=tuple(v * dx for v in n), sigma_over_dx=sigma,
                            cutoff=cutoff, n_particles=particles, kmax=3.0, shear_rate=0.3)
    p = w.params(gravity=(0.0, 0.0, -1.0))
    grid = np.random.default_rng(1).standard_normal((3,) + n[::-1])
    st = I.make_particles(w, None)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()  # noqa: E731
    ctx = erpp.Context(p, precision="fp64")
    assert rel(ctx.interpolate(cu(grid), cu(st.x)), oracle_lib.gather(p, st.x, grid)) < 1e-12
    assert rel(ctx.scatter_source(cu(st.x), cu(st.D)), oracle_lib.scatter(p, st.x, st.D)) < 1e-12
    ps = erpp.ParticleState.from_numpy(st)
    ref = st.copy()
    for _ in range(2):
        S = ctx.step(cu(grid), ps, first_step=False)
        ctx.check()
        S_ref = oracle_lib.step(p, grid, ref, first_step=False)
        assert rel(S, S_ref) < 1e-12
        assert rel(ps.D, ref.D) < 1e-12 and rel(ps.v, ref.v) < 1e-12

"""Particles exactly on grid nodes in boxes whose r_c / dx rounds to just below
an integer on some axis (c' = 3 - 2^-51): the window s - c' .. s + c' of such a
particle rounds to three nodes below it, one more than floor(c').  The tiles'
halos and the binning's bounds have to cover it.

Tolerance: the FP32 bound of the parity tests, 1e-5 relative L2.
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


def _reach(w):
    p = w.params()
    rc = p["cutoff"] * math.sqrt((2.0 * p["nu"]) * p["eps_R"])
    return [rc * (p["n"][a] / p["L"][a]) for a in range(3)]


BOXES = [(30, 83, 24), (90, 83, 24), (90, 24, 83), (30, 24, 83)]


@pytest.mark.parametrize("mode", ["merge", "cluster", "xclip"])
@pytest.mark.parametrize("n", BOXES, ids=["x".join(map(str, b)) for b in BOXES])
def test_particles_on_nodes(erpp, oracle_lib, n, mode):
    import torch
    dx = 2 * math.pi / 64
    w = dataclasses.replace(I.CFG_SMALL, n=n, L=tuple(v * dx for v in n), kmax=3.0)
    assert any(2.9 < c < 3.0 for c in _reach(w))  # the boxes are what they are meant to be
    rng = np.random.default_rng(8)
    nodes = np.stack([rng.integers(0, v, 400) for v in n]).astype(np.float64)
    x = nodes * (np.array(w.L) / np.array(n))[:, None]
    grid, _ = I.make_grid(w)
    D = rng.standard_normal(x.shape)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()  # noqa: E731
    ctx = erpp.Context(w.params(), precision="fp32")
    ctx.set_scatter_mode(mode)
    S = ctx.scatter_source(cu(x), cu(D))
    up = ctx.interpolate(cu(grid).float().contiguous(), cu(x))
    ctx.check()
    ref = oracle_lib.scatter(w.params(), x, D)
    rup = oracle_lib.gather(w.params(), x, grid)
    rel = lambda a, b: float(np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b))  # noqa: E731
    assert rel(S, ref) < 1e-5 and rel(up, rup) < 1e-5

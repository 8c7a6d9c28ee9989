"""Tiles whose staged field leaves one block per SM: the gather takes half batches
there, the compensated scatter 512 threads.  Tiles of 18 rows and more, by request and
by the box's size; windows of 6 nodes and of 9, and boxes whose r_c / dx rounds to
just below 3.

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


CASES = [((128, 274, 10), 9000, 1.0, 0), ((70, 50, 20), 9000, 1.0, 20), ((70, 50, 20), 9000, 1.5, 16),
         ((181, 45, 19), 9000, 1.0, 22), ((32, 64, 40), 12000, 1.0, 0), ((33, 64, 40), 12000, 1.0, 24)]


@pytest.mark.parametrize("kahan", [False, True])
@pytest.mark.parametrize("n,particles,sigma,tile_y", CASES,
                         ids=["x".join(map(str, c[0])) + f"_{c[2]}" for c in CASES])
def test_large_tiles(erpp, oracle_lib, n, particles, sigma, tile_y, kahan):
    import torch
    w = dataclasses.replace(I.CFG_SMALL, n=n, L=tuple(v * 0.05 for v in n), sigma_over_dx=sigma,
                            shear_rate=0.5, kmax=2.0)
    rng = np.random.default_rng(3)
    x = rng.random((3, particles)) * np.array(w.L)[:, None] * (1 - 1e-12)
    D = rng.standard_normal(x.shape)
    u = rng.standard_normal((3,) + n[::-1]).astype(np.float32)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()  # noqa: E731
    ctx = erpp.Context(w.params(), precision="fp32", kahan=kahan)
    if tile_y:
        ctx.set_tiling(tile_y=tile_y)
    ctx.set_scatter_mode("xclip" if n[0] == 33 else "merge")
    up = ctx.interpolate(cu(u), cu(x)).cpu().numpy()
    S = ctx.scatter_source(cu(x), cu(D)).cpu().numpy()
    ctx.check()
    ref, Sr = oracle_lib.gather(w.params(), x, u.astype(np.float64)), oracle_lib.scatter(w.params(), x, D)
    assert np.linalg.norm(up - ref) / np.linalg.norm(ref) < 1e-5
    assert np.linalg.norm(S - Sr) / np.linalg.norm(Sr) < 1e-5

"""Dense bricks of the source: quarters of a region that nothing reaches beside a
brick of more particles than a list entry can count.

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

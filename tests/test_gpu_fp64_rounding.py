"""Rounding of the FP64 gather: its error against extended precision (the host's long
double, 64 bits of mantissa or more).

Bound: 2.3e-16 rms of the mean velocity.  A division per weight and pairwise sums of
the weights leave 1.9e-16 (a few roundings of 2^-53 each, independent); weights from a
rounded reciprocal and a running sum 2.7e-16.
"""

import math

import numpy as np
import pytest

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


def gather(x, u, n, L, nu, eps, cutoff):
    """The gather of normalised weights in long double; windows and positions in units
    of the spacing as the library rounds them."""
    ld = np.longdouble
    s2, dV, J, W = ld(2) * ld(nu) * ld(eps), ld(1), [], []
    for a in range(3):
        c, s = cutoff * math.sqrt(2 * nu * eps) * (n[a] / L[a]), x[a] * (n[a] / L[a])
        lo, hi, k = np.ceil(s - c), np.floor(s + c), np.arange(12)
        dx = ld(L[a]) / ld(n[a])
        dV = dV * dx
        j = lo[:, None] + k
        d = (j.astype(ld) - s[:, None].astype(ld)) * dx
        w = np.where(j <= hi[:, None], np.exp(-d * d / (2 * s2)), ld(0))
        W.append(w / (dx * w.sum(1, keepdims=True)))
        J.append(np.mod(j.astype(np.int64), n[a]))
    idx = ((J[2][:, :, None, None] * n[1] + J[1][:, None, :, None]) * n[0] + J[0][:, None, None, :])
    w = W[2][:, :, None, None] * W[1][:, None, :, None] * W[0][:, None, None, :]
    return np.stack([dV * (u[c].reshape(-1)[idx].astype(ld) * w).sum((1, 2, 3)) for c in range(3)])


@pytest.mark.parametrize("n,sigma", [((64, 64, 64), 1.0), ((64, 48, 72), 1.5)])
def test_gather_rounding(erpp, n, sigma):
    import torch
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision on this host")
    dx, nu = 2 * math.pi / 64, 0.01
    L, eps = tuple(v * dx for v in n), (sigma * dx) ** 2 / (2 * nu)
    x = np.random.default_rng(5).random((3, 1500)) * np.array(L)[:, None]
    z, y, i = np.meshgrid(*[np.arange(k) for k in n[::-1]], indexing="ij")
    u = np.stack([np.sin(2 * np.pi * i / n[0]) * np.cos(2 * np.pi * y / n[1]) + 0.5,
                  np.cos(4 * np.pi * z / n[2]) * 1.3 + 0.2,
                  np.sin(2 * np.pi * (i + y) / n[0]) + 0.7])
    ctx = erpp.Context(dict(n=n, L=L, nu=nu, rho_f=1.0, eps_R=eps, cutoff=3.0, dt=1e-3),
                       precision="fp64")
    up = ctx.interpolate(torch.as_tensor(u).cuda(), torch.as_tensor(x).cuda()).cpu().numpy()
    ref = gather(x, u, n, L, nu, eps, 3.0)
    err = (up - ref) / np.abs(ref).mean()
    assert float(np.sqrt((err ** 2).mean())) < 2.3e-16

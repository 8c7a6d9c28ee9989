"""Performance cases of the coupling library: what its users have it do.

Each case is one pass through the public entry points of
``paper_1405_6969_gb300``: the coupling step on boxes from 32^3 nodes and a
thousand particles to 512 x 256 x 256 nodes and a million (FP32 and FP64, the
other weights, the compensated scatter, the general force), the gather alone,
the source and the gather with their adjoints, many boxes in one graph, and the
step coupled to the fluid stand-in.  Contexts are made with their default
options, as a program that does not tune makes them.

``exact`` is the same arithmetic in 64 bits in plain PyTorch: truncated
Gaussian weights per axis, App. A.5's closed form for the removed disturbance,
Stokes drag or the general force, explicit Euler, the exact Stokes step.
"""

from __future__ import annotations

import math

import torch

import paper_1405_6969_gb300 as erpp

PI = math.pi


def _case(name, kind, n, particles, **over):
    c = dict(name=name, kind=kind, nx=n[0], ny=n[1], nz=n[2], particles=particles,
             dx=2 * PI / 256, sigma=1.0, cloud="uniform", shear=0.0, precision="fp32",
             weights="gaussian", normalize=True, kahan=False, full_force=False, boxes=1)
    c.update(over)
    return c


def listed():
    return [
        # a first look at a small box: a thousand particles, one step at a
        # time from Python, where launches and latency are all there is
        _case("step_32cube_1k", "step", (32, 32, 32), 1000, dx=2 * PI / 32),
        # the production run: homogeneous-shear box, a million particles of
        # three Stokes numbers
        _case("step_shear512_1M", "step", (512, 256, 256), 1_000_000, shear=1.0),
        # clustered particles (preferential concentration) with a wider kernel
        _case("step_clusters128_100k", "step", (128, 128, 128), 100_000, dx=2 * PI / 128,
              sigma=1.5, cloud="clusters", shear=1.0),
        # a box whose rows are not a multiple of 16 bytes, with the raw
        # (unnormalised) Gaussian
        _case("step_ragged_raw_60k", "step", (181, 122, 95), 60_000, dx=2 * PI / 128,
              normalize=False),
        # the gather alone: fluid velocity at tracers for statistics
        _case("interpolate_256cube_1M", "interpolate", (256, 256, 256), 1_000_000, shear=1.0),
        # optimisation over particle positions and forces: the source and its
        # adjoint through autograd
        _case("source_adjoint_128cube_100k", "source_adjoint", (128, 128, 128), 100_000,
              dx=2 * PI / 128, sigma=1.5),
        # optimisation over the field and positions: the gather and its adjoint
        _case("gather_adjoint_96x101x90_50k", "gather_adjoint", (96, 101, 90), 50_000,
              dx=2 * PI / 96, sigma=1.5),
        # the double-precision step of a reference run
        _case("step_fp64_128cube_100k", "step", (128, 128, 128), 100_000, dx=2 * PI / 128,
              precision="fp64"),
        # the classical particle-in-cell coupling, for comparison runs
        _case("step_pic_256cube_500k", "step", (256, 256, 256), 500_000, weights="pic"),
        # the general force (Faxen, added mass, one-step memory)
        _case("step_full_force_192cube_300k", "step", (192, 192, 192), 300_000,
              dx=2 * PI / 192, full_force=True),
        # many independent boxes stepped as one graph: 64^3 to 128^3 nodes,
        # 1e3 to 2e5 particles each
        _case("batch_12_boxes", "batch", (64, 64, 64), 0, boxes=12),
        # the two-way coupled loop: step with the compensated scatter, then the
        # fluid stand-in driven by the source
        _case("coupled_kahan_256x128x128_200k", "coupled", (256, 128, 128), 200_000,
              dx=2 * PI / 128, kahan=True, shear=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["interpolate", "source_adjoint", "gather_adjoint", "batch",
                                      "coupled"])
    if kind == "batch":
        return _drop_name(_case("", "batch", (64, 64, 64), 0, boxes=rng.randint(3, 12),
                                sigma=rng.choice([1.0, 1.0, 1.5]),
                                shear=rng.choice([0.0, 1.0])))
    option = rng.choice(["plain"] * 4 + ["raw", "kahan", "fp64", "pic", "point", "full_force"]) \
        if kind in ("step", "coupled") else "plain"
    heavy = kind.endswith("adjoint") or kind == "coupled" or option in ("fp64", "full_force")
    top = 2 ** 21 if heavy else 2 ** 25
    while True:
        n = tuple(_log_int(rng, 30, 192 if heavy else 512) for _ in range(3))
        if rng.random() < 0.5:  # rows of whole 16-byte chunks as often as not
            n = (max(32, n[0] // 16 * 16), n[1], n[2])
        nodes = n[0] * n[1] * n[2]
        if 2 ** 15 <= nodes <= top:
            break
    particles = max(200, min(int(nodes * math.exp(rng.uniform(math.log(0.008), math.log(0.08)))),
                             100_000 if heavy else 1_000_000))
    over = dict(dx=0.02 + 0.08 * rng.random(), sigma=rng.choice([1.0, 1.0, 1.5]),
                cloud=rng.choice(["uniform", "uniform", "clusters"]),
                shear=rng.choice([0.0, 1.0]))
    if option == "raw":
        over["normalize"] = False
    elif option == "kahan":
        over["kahan"] = True
    elif option == "fp64":
        over["precision"] = "fp64"
    elif option in ("pic", "point"):
        over["weights"] = option
    elif option == "full_force":
        over["full_force"] = True
    return _drop_name(_case("", kind, n, particles, **over))


def _drop_name(c):
    return {k: v for k, v in c.items() if k != "name"}


# ---- inputs -------------------------------------------------------------

def _params(case):
    n = (case["nx"], case["ny"], case["nz"])
    sigma = case["sigma"] * case["dx"]
    nu = 0.01
    return dict(n=n, L=tuple(v * case["dx"] for v in n), nu=nu, rho_f=1.0,
                eps_R=sigma * sigma / (2 * nu), cutoff=3.0, dt=1e-3, gravity=(0.0, -1.0, 0.0),
                shear_rate=case["shear"])


def _wrap(x, L):
    x = torch.remainder(x, L)
    return torch.where(x >= L, torch.zeros_like(x), x)


def _field(case, gen):
    """A divergence-free random field of the box's longest waves, unit rms."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    m = [torch.fft.fftfreq(v, 1.0 / v, device="cuda", dtype=torch.float64) for v in (nz, ny)]
    mx = torch.arange(nx // 2 + 1, device="cuda", dtype=torch.float64)
    k = (mx[None, None, :] / nx, m[1][None, :, None] / ny, m[0][:, None, None] / nz)
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    low = (k2 > 0) & (k2 <= (6.0 / min(nx, ny, nz)) ** 2)
    at = low.nonzero(as_tuple=True)
    amp = torch.randn((2, 3, at[0].numel()), generator=gen, device="cuda", dtype=torch.float64)
    amp = torch.complex(amp[0], amp[1])
    kk = torch.stack([k[0].expand_as(k2)[at], k[1].expand_as(k2)[at], k[2].expand_as(k2)[at]])
    amp = amp - kk * (kk * amp).sum(0) / (kk * kk).sum(0)
    u = torch.empty((3, nz, ny, nx), device="cuda", dtype=torch.float32)
    for c in range(3):
        spec = torch.zeros(k2.shape, device="cuda", dtype=torch.complex64)
        spec[at] = amp[c].to(torch.complex64)
        g = torch.fft.irfftn(spec, s=(nz, ny, nx))
        u[c] = g / g.square().mean().sqrt().clamp_min(1e-30)
    return u.to(torch.float64) if case["precision"] == "fp64" else u


def _cloud(case, gen):
    p = _params(case)
    N = case["particles"]
    L = torch.tensor(p["L"], device="cuda", dtype=torch.float64)[:, None]
    kw = dict(generator=gen, device="cuda", dtype=torch.float64)
    x = torch.rand((3, N), **kw) * L
    if case["cloud"] == "clusters":
        # fifty clusters a few grid spacings wide
        centre = torch.rand((3, 50), **kw) * L
        which = torch.randint(0, 50, (N,), generator=gen, device="cuda")
        x = centre[:, which] + 1.2 * case["dx"] * torch.randn((3, N), **kw)
    return _wrap(x, L).contiguous()


def _particles(case, u, gen):
    """Positions, velocities near the fluid's, the previous position and
    force, and the radii and density of three Stokes numbers."""
    p = _params(case)
    N = case["particles"]
    kw = dict(generator=gen, device="cuda", dtype=torch.float64)
    L = torch.tensor(p["L"], device="cuda", dtype=torch.float64)[:, None]
    x = _cloud(case, gen)
    j = [(x[a] / case["dx"]).long().clamp_max(p["n"][a] - 1) for a in range(3)]
    slip = 0.05 * torch.randn((3, N), **kw)
    v = u[:, j[2], j[1], j[0]].double() + slip
    v[0] += case["shear"] * x[1]
    x_prev = _wrap(x - p["dt"] * v, L).contiguous()
    tau_eta = (case["sigma"] * case["dx"]) ** 2 / p["nu"]
    st = torch.tensor([0.1, 1.0, 10.0], device="cuda", dtype=torch.float64)
    tau = st[torch.randint(0, 3, (N,), generator=gen, device="cuda")] * tau_eta
    rho = torch.full((N,), 200.0 if case["full_force"] else 1000.0, device="cuda",
                     dtype=torch.float64)
    radius = torch.sqrt(4.5 * p["nu"] * tau / rho)
    D = 6 * PI * p["nu"] * radius * 0.05 * torch.randn((3, N), **kw)
    return x, v.contiguous(), x_prev, D, radius, rho


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _boxes(case, seed):
    """The boxes of a batch: sizes from the box's number, contents from the seed."""
    out = []
    for i in range(case["boxes"]):
        r = torch.rand(2, generator=torch.Generator().manual_seed(1000 + i)).tolist()
        g = (64, 96, 128)[int(3 * r[0])]
        out.append(dict(case, nx=g, ny=g, nz=g, dx=2 * PI / g,
                        particles=int(round(1000 * 200 ** r[1]))))
    return out


def _inputs(case, seed):
    gen = _gen(seed)
    if case["kind"] == "source_adjoint":
        p = _params(case)
        x = _cloud(case, gen)
        D = torch.randn(x.shape, generator=gen, device="cuda", dtype=torch.float64)
        R = torch.randn((3,) + p["n"][::-1], generator=gen, device="cuda", dtype=torch.float32)
        return x, D, R
    u = _field(case, gen)
    if case["kind"] == "interpolate":
        return u, _cloud(case, gen)
    if case["kind"] == "gather_adjoint":
        x = _cloud(case, gen)
        return u, x, torch.randn(x.shape, generator=gen, device="cuda", dtype=torch.float64)
    return u, _particles(case, u, gen)


def _context(case):
    return erpp.Context(_params(case), precision=case["precision"], normalize=case["normalize"],
                        kahan=case["kahan"], weights=case["weights"],
                        full_force=case["full_force"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        boxes = []
        for i, b in enumerate(_boxes(case, seed)):
            u, parts = _inputs(dict(b, kind="step"), seed * 1009 + i)
            boxes.append((_params(b), u, erpp.ParticleState(*parts), torch.empty_like(u)))
        return dict(kind=kind, boxes=boxes, batch=erpp.Batch(boxes))
    st = dict(kind=kind, ctx=_context(case))
    if kind == "source_adjoint":
        x, D, R = _inputs(case, seed)
        st.update(x=x.requires_grad_(), D=D.requires_grad_(), R=R)
    elif kind == "gather_adjoint":
        u, x, g = _inputs(case, seed)
        st.update(u=u.requires_grad_(), x=x.requires_grad_(), g=g)
    elif kind == "interpolate":
        st["u"], st["x"] = _inputs(case, seed)
    else:
        st["u"], parts = _inputs(case, seed)
        st["particles"] = erpp.ParticleState(*parts)
        if case["full_force"]:  # the run's first step, which starts the history
            st["ctx"].step(st["u"], st["particles"], first_step=True)
        if kind == "coupled":
            st["fluid"] = erpp.StokesFluid(_params(case), precision=case["precision"])
    return st


def _state_out(P):
    return dict(x=P.x, v=P.v, x_prev=P.x_prev, D=P.D)


def run(state):
    kind = state["kind"]
    if kind == "step":
        P = state["particles"]
        S = state["ctx"].step(state["u"], P)
        return dict(_state_out(P), S=S)
    if kind == "interpolate":
        return state["ctx"].interpolate(state["u"], state["x"])
    if kind == "source_adjoint":
        x, D = state["x"], state["D"]
        S = erpp.ScatterSource.apply(state["ctx"], x, D)
        gx, gD = torch.autograd.grad(S, (x, D), state["R"])
        return dict(S=S.detach(), gx=gx, gD=gD)
    if kind == "gather_adjoint":
        u, x = state["u"], state["x"]
        up = erpp.Interpolate.apply(state["ctx"], u, x)
        gu, gx = torch.autograd.grad(up, (u, x), state["g"])
        return dict(up=up.detach(), gu=gu, gx=gx)
    if kind == "batch":
        state["batch"].step()
        return [dict(_state_out(P), S=S) for _, _, P, S in state["boxes"]]
    # coupled
    P = state["particles"]
    S = state["ctx"].step(state["u"], P)
    state["fluid"].step(state["u"], S)
    return dict(_state_out(P), S=S, u=state["u"])


def work(case):
    if case["kind"] == "batch":
        w = [work(dict(b, kind="step")) for b in _boxes(case, 0)]
        return {k: sum(i[k] for i in w) for k in ("bytes", "flops")}
    nodes, N = case["nx"] * case["ny"] * case["nz"], case["particles"]
    real = 8 if case["precision"] == "fp64" else 4
    grid, kind = 3 * nodes * real, case["kind"]
    stencil = 8 if case["weights"] == "pic" else (6 * case["sigma"]) ** 3
    point = (64 if case["weights"] == "point" else stencil) * 6  # gather, 3 components
    spread = stencil * 6
    if kind == "interpolate":
        return {"bytes": grid + 48 * N, "flops": point * N}
    if kind == "source_adjoint":  # S; R, x, D; the two gradients
        return {"bytes": 2 * grid + 48 * N + 48 * N, "flops": (spread + 2 * point) * N}
    if kind == "gather_adjoint":  # u; g, x; the two gradients
        return {"bytes": 2 * grid + 24 * N + 24 * N + 48 * N, "flops": (spread + 2 * point) * N}
    w = {"bytes": 2 * grid + 208 * N, "flops": (point + spread) * N}
    if case["full_force"]:  # the previous velocity and its Laplacian, kept
        w["bytes"] += 96 * N
        w["flops"] += point * N
    if kind == "coupled":  # u read once more is u written back
        w["bytes"] += grid
        w["flops"] += 2 * 3 * 2.5 * nodes * math.log2(nodes)
    return w


# ---- the same in 64 bits ------------------------------------------------

class _Stencil:
    """Truncated per-axis weights of every particle, and the node indices."""

    def __init__(self, p, x, weights, normalize):
        self.p, self.dV = p, 1.0
        self.j, self.w, self.dw, self.d2w = [], [], [], []
        s2 = 2 * p["nu"] * p["eps_R"]
        for a in range(3):
            n, L = p["n"][a], p["L"][a]
            dx, s = L / n, x[a] * (n / L)
            self.dV *= dx
            if weights == "pic":
                lo, f = torch.floor(s), s - torch.floor(s)
                w = torch.stack([1 - f, f], 1) / dx
                dw = d2w = torch.zeros_like(w)
            elif weights == "point":
                lo = torch.floor(s) - 1
                f = s - lo - 1
                w = torch.stack([-f * (f - 1) * (f - 2) / 6, (f * f - 1) * (f - 2) / 2,
                                 -f * (f + 1) * (f - 2) / 2, f * (f * f - 1) / 6], 1) / dx
                dw = d2w = torch.zeros_like(w)
            else:
                c = p["cutoff"] * math.sqrt(s2) * (n / L)
                lo, hi = torch.ceil(s - c), torch.floor(s + c)
                k = torch.arange(int(2 * c) + 2, device=x.device, dtype=torch.float64)
                d = (lo[:, None] + k - s[:, None]) * dx
                w = torch.exp(-d * d / (2 * s2)) / math.sqrt(2 * PI * s2)
                w = torch.where(lo[:, None] + k <= hi[:, None], w, torch.zeros_like(w))
                A, B = d / s2, d * d / s2 ** 2 - 1 / s2
                if normalize:
                    w = w / (dx * w.sum(1, keepdim=True))
                    m1 = dx * (w * A).sum(1, keepdim=True)
                    m2 = dx * (w * B).sum(1, keepdim=True)
                    dw, d2w = w * (A - m1), w * (B - 2 * A * m1 - m2 + 2 * m1 * m1)
                else:
                    dw, d2w = w * A, w * B
            k = torch.arange(w.shape[1], device=x.device)
            self.j.append(torch.remainder(lo.long()[:, None] + k, n))
            self.w.append(w)
            self.dw.append(dw)
            self.d2w.append(d2w)

    def nodes(self):
        nx, ny, _ = self.p["n"]
        jx, jy, jz = self.j
        return (jz[:, :, None, None] * ny + jy[:, None, :, None]) * nx + jx[:, None, None, :]

    def contract(self, U, wx, wy, wz):
        return torch.einsum("czyxp,px,py,pz->cp", U, wx, wy, wz)

    def values(self, u):
        """u at the stencil nodes, [3, z, y, x, p]."""
        idx = self.nodes()
        return torch.stack([u[c].reshape(-1)[idx] for c in range(3)]).permute(0, 2, 3, 4, 1)


def _chunks(x, rows=50_000):
    return [slice(s, min(s + rows, x.shape[1])) for s in range(0, x.shape[1], rows)]


def _gather64(p, u, x, weights="gaussian", normalize=True, laplacian=False, v=None):
    """u_p (with the mean shear); also its Laplacian, or (with v) the
    derivative of u_p . v in the position and u_p without the shear."""
    up, more = torch.empty_like(x), torch.empty_like(x)
    for c in _chunks(x):
        st = _Stencil(p, x[:, c], weights, normalize)
        U = st.values(u).double()
        w = st.w
        up[:, c] = st.dV * st.contract(U, *w)
        if laplacian:
            more[:, c] = st.dV * (st.contract(U, st.d2w[0], w[1], w[2]) +
                                  st.contract(U, w[0], st.d2w[1], w[2]) +
                                  st.contract(U, w[0], w[1], st.d2w[2]))
        elif v is not None:
            for a in range(3):
                ww = [st.dw[b] if a == b else w[b] for b in range(3)]
                more[a, c] = st.dV * (st.contract(U, *ww) * v[:, c]).sum(0)
    if v is None:
        up[0] += p["shear_rate"] * x[1]
    return up, more


def _scatter64(p, x, D, weights="gaussian", normalize=True, scale=None):
    n = p["n"]
    S = torch.zeros((3, n[0] * n[1] * n[2]), device=x.device, dtype=torch.float64)
    scale = -1.0 / p["rho_f"] if scale is None else scale
    for c in _chunks(x):
        st = _Stencil(p, x[:, c], weights, normalize)
        W = torch.einsum("pz,py,px->pzyx", st.w[2], st.w[1], st.w[0])
        idx = st.nodes().reshape(-1)
        for a in range(3):
            S[a].index_add_(0, idx, (W * (scale * D[a, c])[:, None, None, None]).reshape(-1))
    return S.reshape((3,) + n[::-1])


def _self64(p, r, D, weights):
    """App. A.5's closed form and its Laplacian (2 d/ds2 of it)."""
    s2 = 2 * p["nu"] * (p["eps_R"] + p["dt"])
    if weights != "point":
        s2 += 2 * p["nu"] * p["eps_R"]
    pref = -(p["dt"] / p["rho_f"]) / (2 * PI * s2) ** 1.5
    rr = r.square().sum(0).sqrt()
    eta = rr / math.sqrt(2 * s2)
    e = torch.exp(-eta * eta)
    big = eta.clamp_min(0.5)
    F = (0.5 * math.sqrt(PI) * torch.erf(big) - big * torch.exp(-big * big)) / (2 * big ** 3)
    dF = torch.exp(-big * big) / big - 3 * F / big
    Fs, dFs, term = torch.zeros_like(eta), torch.zeros_like(eta), torch.ones_like(eta)
    for k in range(20):
        Fs, dFs = Fs + term / (2 * k + 3), dFs + 2 * k * term / (2 * k + 3)
        term = -term * eta * eta / (k + 1)
    small = eta < 0.5
    F = torch.where(small, Fs, F)
    dF = torch.where(small, dFs / eta.clamp_min(1e-300), dF)
    de = -2 * eta * e
    rh = r / rr.clamp_min(1e-300)
    Dr = (D * rh).sum(0)
    B = (e - F) * D - Dr * (e - 3 * F) * rh
    dB = (de - dF) * D - Dr * (de - 3 * dF) * rh
    return pref * B, -(pref / s2) * (3 * B + eta * dB)


def _step64(case, u, parts, first=False, kept=None):
    """One step; returns the new particles, S and what the general force keeps."""
    p, weights = _params(case), case["weights"]
    x, v, x_prev, D, radius, rho = parts
    L = torch.tensor(p["L"], device=x.device, dtype=torch.float64)[:, None]
    g = torch.tensor(p["gravity"], device=x.device, dtype=torch.float64)[:, None]
    dt, mu = p["dt"], p["nu"] * p["rho_f"]
    ut, Lt = _gather64(p, u, x, weights, case["normalize"], laplacian=case["full_force"])
    if weights != "pic" and not first:
        r = x - x_prev
        r = r - L * torch.round(r / L)
        vs, ls = _self64(p, r, D, weights)
        ut, Lt = ut - vs, Lt - ls
    m_p = 4.0 / 3.0 * PI * radius ** 3 * rho
    if case["full_force"]:
        u0, L0 = (ut, Lt) if kept is None else kept
        a2, m_f = radius ** 2, 4.0 / 3.0 * PI * radius ** 3 * p["rho_f"]
        cB = 12 * mu * a2 * math.sqrt(PI / (p["nu"] * dt))
        dq = ut + a2 / 6 * Lt - u0 - a2 / 6 * L0
        F = (6 * PI * mu * radius * (ut + a2 / 6 * Lt - v) + m_f * (ut - u0) / dt +
             0.5 * m_f * (ut + a2 / 10 * Lt - u0 - a2 / 10 * L0) / dt + cB * dq)
        dv = (F + (m_p - m_f) * g) / ((m_p + 0.5 * m_f) / dt + cB)
        Dn = F - (0.5 * m_f / dt + cB) * dv
    else:
        Dn = 6 * PI * mu * radius * (ut - v)
        dv = dt * (Dn / m_p + (1 - p["rho_f"] / rho) * g)
    xn = x + dt * v
    xn = torch.where(xn < 0, xn + L, xn)
    xn = torch.where(xn >= L, xn - L, xn)
    S = _scatter64(p, x, Dn, "pic" if weights == "pic" else "gaussian", case["normalize"])
    return (xn, v + dv, x, Dn, radius, rho), S, (ut, Lt)


def _stokes64(p, u, S):
    k, t = [], []
    for a, shape in ((0, (1, 1, -1)), (1, (1, -1, 1)), (2, (-1, 1, 1))):
        n = p["n"][a]
        m = torch.fft.fftfreq(n, 1.0 / n, device=u.device, dtype=torch.float64)
        k.append((2 * PI / p["L"][a] * m).reshape(shape))
        if n % 2 == 0:  # the Nyquist wave counts with either sign
            m = m.clone()
            m[n // 2] = -m[n // 2]
        t.append((2 * PI / p["L"][a] * m).reshape(shape))
    h = torch.fft.fftn(u + p["dt"] * S, dim=(1, 2, 3))
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    inv = torch.where(k2 > 0, 0.5 / k2, torch.zeros_like(k2))
    q = [sum(w[a] * h[a] for a in range(3)) * inv for w in (k, t)]
    decay = torch.exp(-p["nu"] * p["dt"] * k2)
    return torch.stack([torch.fft.ifftn(decay * (h[a] - k[a] * q[0] - t[a] * q[1])).real
                        for a in range(3)])


def exact(case, seed):
    kind, p = case["kind"], _params(case)
    if kind == "batch":
        return [exact(dict(b, kind="step", exact_seed=seed * 1009 + i), seed)
                for i, b in enumerate(_boxes(case, seed))]
    got = _inputs(case, case.get("exact_seed", seed))
    if kind == "source_adjoint":
        x, D, R = got
        G, h = _gather64(p, R, x, v=D)
        # the gather's dV is the source's -1 / rho_f
        n, L = p["n"], p["L"]
        to = -1.0 / (p["rho_f"] * (L[0] / n[0]) * (L[1] / n[1]) * (L[2] / n[2]))
        return dict(S=_scatter64(p, x, D), gx=to * h, gD=to * G)
    if kind == "interpolate":
        return _gather64(p, *got)[0]
    if kind == "gather_adjoint":
        u, x, g = got
        n, L = p["n"], p["L"]
        dV = (L[0] / n[0]) * (L[1] / n[1]) * (L[2] / n[2])
        h = _gather64(p, u, x, v=g)[1]
        h[1] += p["shear_rate"] * g[0]
        return dict(up=_gather64(p, u, x)[0], gu=_scatter64(p, x, g, scale=dV), gx=h)
    u, parts = got
    kept = None
    if case["full_force"]:
        parts, _, kept = _step64(case, u, parts, first=True)
    parts, S, _ = _step64(case, u, parts, kept=kept)
    out = dict(x=parts[0], v=parts[1], x_prev=parts[2], D=parts[3], S=S)
    if kind == "coupled":
        out["u"] = _stokes64(p, u.double(), S)
    return out

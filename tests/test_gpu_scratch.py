"""Scratch of the brick kernels and of the FP64 step: made by the calls that use
it, and left where captured graphs expect it.

Replays are compared bit for bit with the same call issued directly.
"""

import dataclasses
import math

import numpy as np
import pytest

import erpp_inputs as I

pytestmark = pytest.mark.gpu

DX = 2 * math.pi / 64
N = (96, 96, 80)


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


def box():
    return dataclasses.replace(I.CFG_SMALL, n=N, L=tuple(v * DX for v in N), shear_rate=0.5)


def cloud(particles, seed):
    rng = np.random.default_rng(seed)
    x = rng.random((3, particles)) * np.array(box().L)[:, None] * (1 - 1e-12)
    return cuda(x), cuda(rng.standard_normal(x.shape))


def free_bytes():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_only_sorting_calls_take_it(erpp):
    """A context that interpolates has no arrays for the sort (76 bytes a
    particle); the first source makes them."""
    import torch
    particles = 1_000_000
    x, D = cloud(particles, 1)
    u = torch.zeros((3,) + N[::-1], device="cuda")
    S, up = torch.empty_like(u), torch.empty_like(x)
    ctx = erpp.Context(box().params(), precision="fp32")
    ctx.interpolate(u, x, out=up)
    start = free_bytes()
    ctx.scatter_source(x, D, S=S)
    assert ctx.debug_last_route() == {"source"}
    assert start - free_bytes() > 70 * particles
    ctx.check()
    # in another halo mode neither call takes them
    other = erpp.Context(box().params(), precision="fp32")
    other.set_scatter_mode("cluster")
    other.interpolate(u, x, out=up)
    start = free_bytes()
    other.scatter_source(x, D, S=S)
    assert start - free_bytes() < 10 * particles


def graph_of(call):
    import torch
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        call()
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    return graph


@pytest.mark.parametrize("later", ["adjoint", "source"])
def test_captured_calls_outlive_larger_ones(erpp, later):
    """A step and a backward call, captured, replay after a larger backward call
    on the same context; the backward call also after a larger source."""
    import torch
    x, D = cloud(9000, 2)
    xl, Dl = cloud(60000, 3)
    R = torch.randn((3,) + N[::-1], device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    ctx = erpp.Context(box().params(), precision="fp32")
    one = torch.ones(9000, device="cuda", dtype=torch.float64)
    start = [x, 0.01 * D, x.clone(), 1e-3 * D]
    P = erpp.ParticleState(*[t.clone() for t in start], 0.01 * one, 1000 * one)
    S = torch.empty_like(R)
    dx = {}

    def backward():
        dx["dD"], dx["dx"] = ctx.scatter_backward(x, D, R)

    def step():
        ctx.step(R, P, S=S)

    def restore():
        for t, s in zip((P.x, P.v, P.x_prev, P.D), start):
            t.copy_(s)

    graphs = [graph_of(backward)]
    kept = dict(dx)  # the graph's outputs
    backward()
    assert ctx.debug_last_route() == {"adjoint"}
    ref = dict(dx)
    if later == "adjoint":
        graphs.append(graph_of(step))
        restore()
        step()
        assert ctx.debug_last_route() == {"source"}
        ref_step = [t.clone() for t in (S, P.x, P.v, P.D)]
        large = [ctx.scatter_backward(xl, Dl, R)]
        assert ctx.debug_last_route() == {"adjoint"}
    else:
        large = [(ctx.scatter_source(xl, Dl),)]
        assert ctx.debug_last_route() == {"source"}
    fill = torch.full((1 << 24,), float("nan"), device="cuda")  # freed memory would not keep
    for t in kept.values():
        t.zero_()
    graphs[0].replay()
    assert all(torch.equal(kept[k], ref[k]) for k in ref)
    if later == "adjoint":
        restore()
        S.zero_()
        graphs[1].replay()
        assert all(torch.equal(a, b) for a, b in zip((S, P.x, P.v, P.D), ref_step))
        again = [ctx.scatter_backward(xl, Dl, R)]
    else:
        again = [(ctx.scatter_source(xl, Dl),)]
    assert all(torch.equal(a, b) for a, b in zip(large[0], again[0]))
    ctx.check()
    del fill


def test_capture_without_it(erpp):
    """A source captured before any call has sorted allocates nothing: the tile
    kernels are recorded, and give the source to FP32 rounding."""
    import torch
    x, D = cloud(9000, 4)
    u = torch.zeros((3,) + N[::-1], device="cuda")
    ctx = erpp.Context(box().params(), precision="fp32")
    ctx.interpolate(u, x)  # the other scratch
    S = torch.empty_like(u)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.scatter_source(x, D, S=S)
    assert not ctx.debug_last_route()
    graph.replay()
    T = ctx.scatter_source(x, D)
    assert ctx.debug_last_route() == {"source"}
    ctx.check()
    assert float((S - T).norm() / T.norm()) < 1e-5


def test_fp64_step_keeps_weights_only(erpp, oracle_lib):
    """An FP64 context that interpolates or forms sources holds the gathered
    velocity alone (24 bytes a particle); the first step makes the array of the
    weights (24 (xs + 1), xs = 7 here), and a step captured before that does
    without it, with the same results."""
    import torch
    particles = 400_000
    x, D = cloud(particles, 5)
    u = torch.zeros((3,) + N[::-1], device="cuda", dtype=torch.float64)
    S, up = torch.empty_like(u), torch.empty_like(x)
    ctx = erpp.Context(box().params(), precision="fp64")
    start = free_bytes()
    ctx.interpolate(u, x, out=up)
    ctx.scatter_source(x, D, S=S)
    assert start - free_bytes() < 40 * particles
    one = torch.ones(particles, device="cuda", dtype=torch.float64)
    state = lambda: erpp.ParticleState(x.clone(), 0.01 * D, x.clone(), 1e-3 * D,  # noqa: E731
                                       0.01 * one, 1000 * one)
    P = state()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.step(u, P, S=S)
    graph.replay()
    start = free_bytes()
    Q, T = state(), torch.empty_like(u)
    start = free_bytes()
    ctx.step(u, Q, S=T)
    assert start - free_bytes() > 180 * particles
    ctx.check()
    assert torch.equal(P.D, Q.D) and torch.equal(P.v, Q.v) and torch.equal(P.x, Q.x)
    assert float((S - T).norm() / T.norm()) < 1e-12  # atomics: the order of additions

"""Calls of one context on two streams at a time that share no memory of the caller's: each gives the same bits
as alone."""
import numpy as np
import pytest

from tests.gpu_common import dev, host, need_gpu, pair, torch
from workloads import diamond8_24, draw_x0

pytestmark = pytest.mark.gpu


def _beside(first, second, reps=20):
    """first() and second() on a stream each, reps times with nothing between them."""
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(reps):
        with torch.cuda.stream(s1):
            first()
        with torch.cuda.stream(s2):
            second()
    torch.cuda.synchronize()


def _empty(*shape):
    return torch.zeros(shape, dtype=torch.complex128, device="cuda")


def test_project_beside_h_psi_and_itself():
    need_gpu()
    ctx, _, _ = pair(diamond8_24())
    x, y = dev(draw_x0(1, 64, ctx.n)), dev(draw_x0(2, 48, ctx.n))
    h, p, q, r = _empty(64, ctx.n), _empty(48, 32), _empty(64, 32), _empty(48, 32)
    ctx.apply_h(x, h)
    ctx.project(y, p)
    ctx.project(x, q)
    ref = host(h).copy(), host(p).copy(), host(q).copy()
    for t in (h, p, q):
        t.zero_()
    _beside(lambda: ctx.apply_h(x, h), lambda: ctx.project(y, p))
    _beside(lambda: ctx.project(x, q), lambda: ctx.project(y, r))
    assert all(np.array_equal(host(t), v) for t, v in zip((h, p, q, r), (*ref, ref[1])))
    ctx.close()


def _blocks(ctx):
    return [(dev(draw_x0(i, k, ctx.n)), dev(draw_x0(10 + i, k, m))) for i, (k, m) in
            enumerate([(160, 80), (96, 96), (130, 70), (200, 60), (128, 64), (150, 75)])]


def test_rotations_and_grams_beside_each_other():
    """More streams than the context keeps memory for, each with its own rotation, and Grams and H psi between."""
    need_gpu()
    ctx, _, _ = pair(diamond8_24())
    blocks = _blocks(ctx)
    outs = [_empty(c.shape[1], ctx.n) for _, c in blocks]
    ref = []
    for (y, c), o in zip(blocks, outs):
        ctx.rotate(y, c, o)
        ref.append(host(o).copy())
        o.zero_()
    y0 = blocks[3][0]
    g, h = _empty(200, 200), _empty(200, ctx.n)
    ctx.gram(y0, y0, g)
    ctx.apply_h(y0, h)
    gref, href = host(g).copy(), host(h).copy()
    streams = [torch.cuda.Stream() for _ in range(8)]
    for _ in range(10):
        for s, (y, c), o in zip(streams, blocks, outs):
            with torch.cuda.stream(s):
                ctx.rotate(y, c, o)
        with torch.cuda.stream(streams[6]):
            ctx.gram(y0, y0, g)
        with torch.cuda.stream(streams[7]):
            ctx.apply_h(y0, h)
    torch.cuda.synchronize()
    assert all(np.array_equal(host(o), r) for o, r in zip(outs, ref))
    assert np.array_equal(host(g), gref) and np.array_equal(host(h), href)
    ctx.close()


def _captured(call):
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        call()
    return graph


def test_replayed_graphs_beside_each_other_and_a_call():
    need_gpu()
    ctx, _, _ = pair(diamond8_24())
    (ya, ca), (yb, cb), (yc, cc) = _blocks(ctx)[:3]
    a, b, c = (_empty(z.shape[1], ctx.n) for z in (ca, cb, cc))
    ref = []
    for y, z, o in ((ya, ca, a), (yb, cb, b), (yc, cc, c)):
        ctx.rotate(y, z, o)
        ref.append(host(o).copy())
        o.zero_()
    ga, gb = _captured(lambda: ctx.rotate(ya, ca, a)), _captured(lambda: ctx.rotate(yb, cb, b))
    streams = [torch.cuda.Stream() for _ in range(3)]
    for _ in range(10):
        for s, call in zip(streams, (ga.replay, gb.replay, lambda: ctx.rotate(yc, cc, c))):
            with torch.cuda.stream(s):
                call()
    torch.cuda.synchronize()
    assert all(np.array_equal(host(o), r) for o, r in zip((a, b, c), ref))
    del ga, gb
    ctx.close()


def test_memory_of_captured_calls_is_used_again():
    """Graphs made and dropped one after the other hold the memory of a few at a time, not of all."""
    need_gpu()
    ctx, _, _ = pair(diamond8_24())
    y, c = dev(draw_x0(1, 160, ctx.n)), dev(draw_x0(2, 160, 80))
    out = _empty(80, ctx.n)
    planes = 16 * 160 * 2 * 2 * ctx.n               # bytes of one call's residues
    _captured(lambda: ctx.rotate(y, c, out))
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    for _ in range(24):
        graph = _captured(lambda: ctx.rotate(y, c, out))
        graph.replay()
        torch.cuda.synchronize()
        del graph
    torch.cuda.empty_cache()
    assert before - torch.cuda.mem_get_info()[0] < 8 * planes
    ctx.close()


def test_field_solvers_beside_h_psi():
    need_gpu()
    ctx, _, _ = pair(diamond8_24())
    x = dev(draw_x0(1, 64, ctx.n))
    rho = dev(np.random.default_rng(2).uniform(0.1, 1.0, ctx.n))
    h, v, e, u = _empty(64, ctx.n), *(torch.zeros_like(rho) for _ in range(3))
    ctx.apply_h(x, h)
    ctx.hartree(rho, v)
    ctx.xc_pbe(rho, e, u)
    ref = [host(t).copy() for t in (h, v, e, u)]
    for t in (h, v, e, u):
        t.zero_()

    def fields():
        ctx.hartree(rho, v)
        ctx.xc_pbe(rho, e, u)

    _beside(lambda: ctx.apply_h(x, h), fields)
    assert all(np.array_equal(host(t), r) for t, r in zip((h, v, e, u), ref))
    ctx.close()


def test_first_call_while_another_stream_is_captured():
    """A rotation that needs its memory allocated, on a stream of its own, in the middle of a capture on another one."""
    need_gpu()
    one, two = pair(diamond8_24())[0], pair(diamond8_24())[0]
    y, c = dev(draw_x0(1, 96, one.n)), dev(draw_x0(2, 96, 64))
    a, b = _empty(64, one.n), _empty(64, one.n)
    other, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        one.rotate(y, c, a)
        with torch.cuda.stream(other):
            two.rotate(y, c, b)
    other.synchronize()
    graph.replay()
    assert np.any(host(b)) and np.array_equal(host(a), host(b))
    del graph
    one.close()
    two.close()

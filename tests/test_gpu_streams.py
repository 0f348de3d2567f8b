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

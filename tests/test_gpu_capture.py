"""Calls whose scratch grows on demand, inside a CUDA graph: captured as the context's first call,
replayed after larger calls have grown the scratch, and compared with the same calls outside."""
import numpy as np
import pytest

from tests.gpu_common import dev, host, need_gpu, pair, torch
from workloads import diamond8_24, draw_x0

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["project", "rotate"])
def test_first_call_captured_then_outgrown(call):
    need_gpu()
    ctx, _, _ = pair(diamond8_24())
    y, c = dev(draw_x0(1, 48, ctx.n)), dev(draw_x0(2, 48, 24))
    big, bigc = dev(draw_x0(3, 160, ctx.n)), dev(draw_x0(4, 160, 160))

    def empty(*shape):
        return torch.zeros(shape, dtype=torch.complex128, device="cuda")

    out, again, wide = (empty(48, 32), empty(48, 32), empty(160, 32)) if call == "project" else \
        (empty(24, ctx.n), empty(24, ctx.n), empty(160, ctx.n))

    def run(a, b, o):
        ctx.project(a, o) if call == "project" else ctx.rotate(a, b, o)

    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        run(y, c, out)
    run(big, bigc, wide)
    graph.replay()
    run(y, c, again)
    assert np.array_equal(host(out), host(again)) and np.any(host(out))
    del graph
    ctx.close()

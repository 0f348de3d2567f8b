"""The FP32 passes on every length that their plan takes in one, two or three stages (radices 2 to 16): the
kinetic term there and back against numpy's FP64 transforms.

Tolerance (2-norm, relative to the largest factor times the input): at most three stages on each of three axes, there
and back, and a stage rounds its outputs to 2^-24 of their norm (sums and twiddle products in all)."""
import numpy as np
import pytest

from tests.gpu_common import R, dev, host, need_gpu, torch
from workloads import draw_x0

pytestmark = pytest.mark.gpu
GRIDS = [(2, 3, 4), (5, 6, 8), (9, 10, 12), (15, 16, 18), (20, 24, 25), (27, 30, 32), (36, 40, 45), (48, 50, 54), (60, 64, 72),
         (75, 80, 81), (90, 96, 100), (108, 120, 4), (6, 125, 128)]


@pytest.mark.parametrize("turn", [0, 1, 2])
@pytest.mark.parametrize("N", GRIDS)
def test_fp32_kinetic_on_every_length(N, turn):
    need_gpu()
    N = N[turn:] + N[:turn]
    if (N[0] | 1) * N[1] * 8 > 227 * 1024 or N[0] * N[2] * 8 > 227 * 1024:
        pytest.skip("a plane that does not fit shared memory")
    L = tuple(0.21 * n for n in N)
    f = 0.5 * sum(np.meshgrid(*[(2 * np.pi / L[a] * np.fft.fftfreq(N[a], 1 / N[a])) ** 2 for a in (2, 1, 0)], indexing="ij"))
    ctx = R.Context(L, N, np.zeros(N[0] * N[1] * N[2]))
    x = draw_x0(3, 2, ctx.n).astype(np.complex64)
    h = torch.empty(2, ctx.n, dtype=torch.complex64, device="cuda")
    ctx.apply_h(dev(x), h, R.MIXED)
    for got, v in zip(host(h), x):
        ref = np.fft.ifftn(np.fft.fftn(v.reshape(f.shape).astype(complex)) * f).reshape(-1)
        assert np.linalg.norm(got - ref) <= 18 * 2.0 ** -24 * f.max() * np.linalg.norm(v)
    ctx.close()

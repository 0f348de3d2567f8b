"""The fixed-point FP64 transforms: every radix chain and odd planes against numpy's FP64 FFT, blocks of
very different and extreme magnitude, zero and non-finite bands.

Tolerance (2-norm, relative to the largest factor times the input): an FP64 transform and its inverse
round some 2 log2 n times, each time by at most 2^-53 of the norm, and the fixed-point form less;
their sum stays below 4 log2 n 2^-53."""
import numpy as np
import pytest

from tests.gpu_common import R, dev, host, need_gpu, torch
from workloads import draw_x0

pytestmark = pytest.mark.gpu
GRIDS = [(2, 2, 2), (3, 4, 5), (8, 9, 10), (16, 12, 15), (25, 27, 2), (32, 36, 48), (5, 125, 6), (128, 3, 64),
         (81, 20, 54), (120, 120, 4), (4, 120, 120), (96, 2, 128)]


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def _setup(N):
    L = tuple(0.21 * n for n in N)
    g2 = sum(np.meshgrid(*[(2 * np.pi / L[a] * np.fft.fftfreq(N[a], 1 / N[a])) ** 2 for a in (2, 1, 0)], indexing="ij"))
    return R.Context(L, N, np.zeros(N[0] * N[1] * N[2])), g2


def _round_trip(x, f):
    return np.fft.ifftn(np.fft.fftn(x.reshape(f.shape)) * f).reshape(-1)


def _tpa(g2, t):
    x = 0.5 * g2 / t
    p = 27 + 18 * x + 12 * x ** 2 + 8 * x ** 3
    return p / (p + 16 * x ** 4)


@pytest.mark.parametrize("N", GRIDS)
def test_kinetic_and_tpa_on_every_radix_chain(N):
    ctx, g2 = _setup(N)
    tol = 4 * max(np.log2(ctx.n), 2) * 2.0 ** -53
    x = draw_x0(3, 5, ctx.n)
    x[1] *= 10.0 ** np.linspace(-14, 3, ctx.n)      # planes of very different size
    x[2] *= 1e-250
    x[3] *= 1e250
    x[4] = 0.0
    h, w = torch.empty(5, ctx.n, dtype=torch.complex128, device="cuda"), torch.empty(5, ctx.n, dtype=torch.complex128, device="cuda")
    ctx.apply_h(dev(x), h)
    t = np.array([0.7, 2.0, 1e-15, 5.0, 1.0])
    ctx.precondition_tpa(dev(x), w, dev(t))
    h, w = host(h), host(w)
    for b in range(5):
        s = max(np.abs(x[b]).max(), 1e-300)
        nx = np.linalg.norm(x[b] / s)
        assert np.linalg.norm(h[b] / s - _round_trip(x[b] / s, 0.5 * g2)) <= tol * 0.5 * g2.max() * nx
        k = _tpa(g2, t[b] if t[b] >= 1e-12 else 1.0)
        assert np.linalg.norm(w[b] / s - _round_trip(x[b] / s, k)) <= tol * nx
    assert np.all(h[4] == 0) and np.all(w[4] == 0)
    # a power of two passes through exactly
    h2 = torch.empty(1, ctx.n, dtype=torch.complex128, device="cuda")
    ctx.apply_h(dev(x[:1] * 2.0 ** 40), h2)
    assert np.array_equal(host(h2)[0], h[0] * 2.0 ** 40)
    ctx.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_non_finite_value_reaches_its_band_only(bad):
    ctx, g2 = _setup((24, 20, 18))
    x = draw_x0(3, 3, ctx.n)
    x[1, 1234] = bad
    w = torch.empty(3, ctx.n, dtype=torch.complex128, device="cuda")
    ctx.precondition_tpa(dev(x), w, dev(np.ones(3)))
    w = host(w)
    assert not np.any(np.isfinite(w[1]))
    for b in (0, 2):
        assert np.allclose(w[b], _round_trip(x[b], _tpa(g2, 1.0)), rtol=0, atol=1e-13)
    ctx.close()


def test_field_solvers_on_fields_of_any_size():
    ctx, g2 = _setup((27, 20, 32))
    rng = np.random.default_rng(5)
    rho = rng.uniform(0.0, 1.0, ctx.n)
    f = np.where(g2 > 0, 4 * np.pi / np.where(g2 > 0, g2, 1), 0.0)
    tol = 4 * np.log2(ctx.n) * 2.0 ** -53
    for s in (1.0, 2.0 ** -300, 2.0 ** 300, 0.0):
        v = torch.empty(ctx.n, dtype=torch.float64, device="cuda")
        ctx.hartree(dev(rho * s), v)
        ref = _round_trip(rho, f).real * s
        assert np.linalg.norm(host(v) - ref) <= tol * f.max() * np.linalg.norm(rho * s) + 0.0
    ctx.close()

"""FP64 Gram matrices and rotations by residue arithmetic: operands that one scale for many values could
cost bits."""
import numpy as np
import pytest

from tests.gpu_common import R, dev, host, need_gpu, torch

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def _ctx(N):
    need_gpu()
    return R.Context((5.0, 5.0, 5.0), N, np.zeros(N[0] * N[1] * N[2]))


def _empty(real, *shape):
    return torch.empty(shape, dtype=torch.float64 if real else torch.complex128, device="cuda")


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("N", [(20, 20, 20), (64, 64, 64), (96, 96, 96)])
def test_gram_of_uniform_rows(N, real):
    """A plane wave with k = 0 rounds every value the same way.  A value is at least 2^61 / sqrt(2 n) units,
    2^50.6 for 96^3, so that two operands are off by at most 2 x 2^-51.6 = 5.3 x 2^-53; the result's, the
    scale's and the reference's roundings add five more at most."""
    ctx = _ctx(N)
    v = np.array([1 / 3, 0.1, 1e-7 / 7, 12345.678]) * (1.0 if real else 1.0 + 1.0j)
    a = np.repeat(v[:, None], ctx.n, 1)
    g = _empty(real, 4, 4)
    before = ctx.launch_count()
    (ctx.gram_real if real else ctx.gram)(dev(a), dev(a), g)
    assert ctx.launch_count() - before > 5          # the residue passes ran
    ref = np.outer(v.conj(), v) * ctx.n * ctx.dV
    assert np.all(np.abs(host(g) - ref) <= 12 * EPS * np.abs(ref))
    ctx.close()

"""FP64 Gram matrices and rotations by residue arithmetic on the tensor cores: against numpy at the
sizes where tiles, K-blocks, chunks of points and padded bands begin and end, with rows of very
different magnitude, and with inputs that are handed back to the FP64 kernels.

Tolerance: the integers are formed from operands rounded to 2^-59 of their row's norm, so an entry
is off by at most 2^-57 |a| |b| (twice for the two operands, sqrt(2) for the parts) plus its own
rounding; numpy's blocked FP64 sums are good to a few 2^-53 |a| |b|.  8 x 2^-53 covers both."""
import numpy as np
import pytest

from tests.gpu_common import R, dev, host, need_gpu, torch
from workloads import draw_x0, draw_x0_real

pytestmark = pytest.mark.gpu
TOL = 8 * 2.0 ** -53


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def _ctx(N):
    return R.Context((5.0, 5.0, 5.0), N, np.zeros(N[0] * N[1] * N[2]))


def _draw(seed, rows, n, real):
    x = (draw_x0_real if real else draw_x0)(seed, rows, n)
    rng = np.random.default_rng(seed)
    x *= 10.0 ** rng.uniform(-12, 6, (rows, 1))            # rows of very different norm
    x[:, : n // 2] *= 10.0 ** rng.uniform(-9, 0, n // 2)   # and points
    return x


def _norm(x, axis):
    return np.linalg.norm(x, axis=axis)


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("N,na,nb", [((30, 30, 30), 128, 128), ((30, 30, 30), 129, 127), ((27, 25, 15), 257, 96),
                                     ((32, 32, 32), 144, 300), ((64, 64, 48), 145, 143)])
def test_gram_at_the_edges(N, na, nb, real):
    ctx = _ctx(N)
    a, b = _draw(1, na, ctx.n, real), _draw(2, nb, ctx.n, real)
    a[3] = 0.0
    g = torch.empty((na, nb), dtype=torch.float64 if real else torch.complex128, device="cuda")
    before = ctx.launch_count()
    (ctx.gram_real if real else ctx.gram)(dev(a), dev(b), g)
    assert ctx.launch_count() - before > 5          # the residue passes ran
    ref = a.conj() @ b.T * ctx.dV
    bound = _norm(a, 1)[:, None] * _norm(b, 1)[None] * ctx.dV
    assert np.all(np.abs(host(g) - ref) <= TOL * bound)
    ctx.close()


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("N,k,m,base", [((30, 30, 30), 128, 128, False), ((27, 25, 15), 193, 65, True),
                                        ((32, 32, 32), 321, 131, True), ((64, 64, 48), 200, 67, False),
                                        ((25, 25, 15), 1090, 260, False)])
def test_rotation_at_the_edges(N, k, m, base, real):
    ctx = _ctx(N)
    y, c = _draw(3, k, ctx.n, real), _draw(4, k, m, real)
    y[:, 7] = 0.0
    b = (draw_x0_real if real else draw_x0)(5, m, ctx.n) if base else None
    out = torch.empty((m, ctx.n), dtype=torch.float64 if real else torch.complex128, device="cuda")
    rotate = ctx.rotate_real if real else ctx.rotate
    ref = c.T @ y
    bound = _norm(c, 0)[:, None] * _norm(y, 0)[None]
    if base:
        t = dev(b)
        rotate(dev(y), dev(c), t, base=t, sign=-1)        # in place
        out, ref, bound = t, b - ref, bound + np.abs(b)
    else:
        rotate(dev(y), dev(c), out)
    assert np.all(np.abs(host(out) - ref) <= TOL * bound)
    ctx.close()


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("N,na,nb", [((9, 2, 10), 3, 5), ((5, 5, 8), 3, 5), ((6, 6, 6), 1, 16), ((8, 10, 6), 17, 9),
                                     ((30, 20, 15), 1, 8)])
def test_gram_of_few_points_and_rows(N, na, nb, real):
    ctx = _ctx(N)   # 180 points: the FP64 kernels; from 200 on the residue passes
    a, b = _draw(7, na, ctx.n, real), _draw(8, nb, ctx.n, real)
    g = torch.empty((na, nb), dtype=torch.float64 if real else torch.complex128, device="cuda")
    (ctx.gram_real if real else ctx.gram)(dev(a), dev(b), g)
    ref = a.conj() @ b.T * ctx.dV
    assert np.all(np.abs(host(g) - ref) <= TOL * _norm(a, 1)[:, None] * _norm(b, 1)[None] * ctx.dV)
    y, c = _draw(9, nb + 32, ctx.n, real), _draw(10, nb + 32, na, real)
    out = torch.empty((na, ctx.n), dtype=g.dtype, device="cuda")
    (ctx.rotate_real if real else ctx.rotate)(dev(y), dev(c), out)
    assert np.all(np.abs(host(out) - c.T @ y) <= TOL * _norm(c, 0)[:, None] * _norm(y, 0)[None])
    ctx.close()


@pytest.mark.parametrize("bad", [np.inf, np.nan, 1e200, 1e-200])
def test_inputs_that_the_fp64_kernels_take(bad):
    ctx = _ctx((30, 30, 30))
    a, b = draw_x0(1, 130, ctx.n), draw_x0(2, 120, ctx.n)
    if np.isfinite(bad):
        a[5] *= bad
    else:
        a[5, 11] = bad
    g = torch.empty((130, 120), dtype=torch.complex128, device="cuda")
    ctx.gram(dev(a), dev(b), g)
    got = host(g)
    with np.errstate(all="ignore"):
        ref = a.conj() @ b.T * ctx.dV
    rest = np.arange(130) != 5
    bound = _norm(a[rest], 1)[:, None] * _norm(b, 1)[None] * ctx.dV
    assert np.all(np.abs(got[rest] - ref[rest]) <= TOL * bound)
    if np.isfinite(bad):
        assert np.all(np.abs(got[5] / bad - ref[5] / bad) <= TOL * _norm(a[5] / bad, 0) * _norm(b, 1) * ctx.dV)
    else:
        assert not np.any(np.isfinite(got[5]))
    # the rotation in place: the update happens once
    base = draw_x0(6, 120, ctx.n)
    c = draw_x0(7, 130, 120)
    t = dev(base)
    ctx.rotate(dev(a), dev(c), t, base=t, sign=-1)
    got = host(t)
    keep = np.isfinite(a).all(axis=0)
    with np.errstate(all="ignore"):
        ref = base - c.T @ a
        bound = np.abs(base) + _norm(c, 0)[:, None] * _norm(a, 0)[None]
    assert np.all(np.abs(got - ref)[:, keep] <= TOL * bound[:, keep])
    assert keep.all() or not np.any(np.isfinite(got[:, ~keep]))
    ctx.close()

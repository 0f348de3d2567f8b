"""FP64 Gram matrices and rotations by residue arithmetic: operands that one scale for many values could
cost bits."""
import numpy as np
import pytest

from oracle.gamma import lobpcg_gamma
from oracle.lobpcg import lobpcg
from tests.gpu_common import R, dev, host, need_gpu, pair, torch
from workloads import draw_x0, draw_x0_real, small_cell

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


def _draw(seed, rows, n, real):
    return (draw_x0_real if real else draw_x0)(seed, rows, n)


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("N,k,m", [((32, 32, 32), 128, 128), ((27, 25, 15), 193, 65)])
def test_rotation_of_rows_of_any_size(N, k, m, real):
    """Rows 2^-120 to 2^60 apart.  The scaled rows are rounded to 2^-bits of the largest one of a point, with
    bits = 62 - h and 2^h < 2 sqrt(2 k): in the norm of an output row at most 4 k 2^-62 (1.5 x 2^-53 for 193), the
    result to another 2^-53.  Rows and coefficients whose powers of two cancel give the same bits; an FP64 sum is good to
    some 2^-53 of sum |c| |y|, and eight of them cover both sides."""
    ctx = _ctx(N)
    y, s = _draw(3, k, ctx.n, real), 2.0 ** np.random.default_rng(11).integers(-120, 60, k)
    rotate, out = (ctx.rotate_real if real else ctx.rotate), _empty(real, m, ctx.n)
    before = ctx.launch_count()
    rotate(dev(y * s[:, None]), dev(np.eye(k, m).astype(y.dtype)), out)
    assert ctx.launch_count() - before > 5          # the residue passes ran
    off = np.linalg.norm(host(out) / s[:m, None] - y[:m], axis=1)
    assert np.all(off <= 4 * EPS * np.linalg.norm(y[:m], axis=1))
    c = _draw(4, k, m, real)
    rotate(dev(y), dev(c), out)
    plain = host(out).copy()
    assert np.all(np.abs(plain - c.T @ y) <= 8 * EPS * (np.abs(c).T @ np.abs(y)))
    rotate(dev(y * s[:, None]), dev(c / s[:, None]), out)
    assert np.array_equal(plain, host(out))
    ctx.close()


@pytest.mark.parametrize("real", [False, True])
def test_rotation_of_two_segments(real):
    """The solvers' rotations of X and [W P] as two sums (45 rows each, no multiple of a K-block) at a size where
    they run as residues: four iterations against the oracle's, to the LOBPCG tests' bars."""
    need_gpu()
    wl = small_cell(N=(32, 30, 32), L=(8.0, 7.5, 8.0), natom=4, nband=45, rcut=2.5)
    ctx, ham, _ = pair(wl)
    x0 = wl.x0_real(45) if real else wl.x0()
    x = dev(x0)
    eig, res, stats, _ = (ctx.lobpcg_real if real else ctx.lobpcg)(x, ctx.lobpcg_opts(maxit=4, tol=0.0))
    o = (lobpcg_gamma if real else lobpcg)(ham, x0, maxit=4, tol=0.0)
    assert stats.iterations == o.iterations
    assert np.max(np.abs(eig - o.eig)) < 1e-9
    assert np.max(np.abs(res - o.resnorm)) < 1e-7
    charge = np.abs(host(x)) ** 2
    assert np.max(np.abs(charge - np.abs(o.X) ** 2)) < 1e-7 * np.max(charge)
    ctx.close()


@pytest.mark.parametrize("real", [False, True])
def test_rows_anywhere_in_the_range(real):
    """Powers of two of rows cancel to the bit wherever in the range they lie, and values without a normal number count:
    a row of them against numpy's product of the scaled rows, to 8 x 2^-53 of their norms' product."""
    ctx = _ctx((20, 20, 20))
    x = _draw(1, 20, ctx.n, real)
    gram = ctx.gram_real if real else ctx.gram
    ref, g = _empty(real, 20, 20), _empty(real, 20, 20)
    gram(dev(x), dev(x), ref)
    gram(dev(x * 2.0 ** -450), dev(x * 2.0 ** 450), g)
    assert np.array_equal(host(ref), host(g))
    gram(dev(x * 2.0 ** 900), dev(x * 2.0 ** -900), g)
    assert np.array_equal(host(ref), host(g))
    for bits in (3, 20, 40):
        a = x.copy()
        a[4] = np.round(x[4].real * 2.0 ** bits)
        b = a.copy()
        b[4] = np.ldexp(a[4].real, -1074)
        gram(dev(b), dev(x * 2.0 ** 390), g)
        got = host(g) * np.where(np.arange(20) == 4, 2.0 ** (1074 - 390), 2.0 ** -390)[:, None]
        bound = np.linalg.norm(a, axis=1)[:, None] * np.linalg.norm(x, axis=1)[None] * ctx.dV
        assert np.all(np.abs(got - a.conj() @ x.T * ctx.dV) <= 8 * EPS * bound), bits
    ctx.close()


@pytest.mark.parametrize("real", [False, True])
def test_a_point_of_subnormal_values_leaves_the_others(real):
    ctx = _ctx((24, 24, 24))
    y, c = _draw(5, 128, ctx.n, real), _draw(6, 128, 128, real)
    rotate, one, two = (ctx.rotate_real if real else ctx.rotate), _empty(real, 128, ctx.n), _empty(real, 128, ctx.n)
    rotate(dev(y), dev(c), one)
    k = np.arange(1.0, 129.0)
    y[:, 5] = np.ldexp(k, -1074)
    rotate(dev(y), dev(c), two)
    rest = np.arange(ctx.n) != 5
    one, two = host(one), host(two)
    assert np.array_equal(one[:, rest], two[:, rest])
    got = np.ldexp(two[:, 5].real, 1074)
    assert np.all(np.abs(got - (c.T @ k).real) <= 1.0)          # whole numbers of 2^-1074, rounded twice
    ctx.close()


@pytest.mark.parametrize("real", [False, True])
def test_short_memory_changes_no_bit(real):
    """Chunks of points as small as 4,096 where the device's memory is nearly all taken."""
    N = (64, 64, 64)
    ctx, short = _ctx(N), _ctx(N)
    a, b, c = (dev(_draw(i, k, ctx.n if i < 3 else 96, real)) for i, k in ((1, 160), (2, 160), (3, 160)))
    rows = {}
    for name, x in (("all", ctx), ("short", short)):
        g, o = _empty(real, 160, 160), _empty(real, 96, ctx.n)
        if name == "short":
            if real:                                # the packed rows' workspace, before there is no room for it
                x.apply_h_real(a, torch.empty_like(a))
            torch.cuda.empty_cache()
            held = torch.empty(torch.cuda.mem_get_info()[0] - 700_000_000, dtype=torch.uint8, device="cuda")
        (x.gram_real if real else x.gram)(a, b, g)
        (x.rotate_real if real else x.rotate)(a, c, o)
        rows[name] = host(g).copy(), host(o).copy()
    del held
    torch.cuda.empty_cache()
    assert all(np.array_equal(p, q) for p, q in zip(rows["all"], rows["short"]))
    ctx.close()
    short.close()


def test_more_rows_than_a_grid_has_blocks():
    """70,000 rows: the FP64 kernels, one after the other.  Sums of n products err by some sqrt(n) 2^-53 of the sum of the
    magnitudes, 15 and 265 here; four times that is allowed."""
    ctx = _ctx((6, 6, 6))
    a, b, c = draw_x0(1, 70000, ctx.n), draw_x0(2, 1, ctx.n), draw_x0(3, 70000, 1)
    g, o = _empty(False, 70000, 1), _empty(False, 1, ctx.n)
    ctx.gram(dev(a), dev(b), g)
    assert np.all(np.abs(host(g) - a.conj() @ b.T * ctx.dV) <= 60 * EPS * (np.abs(a) @ np.abs(b).T * ctx.dV))
    ctx.rotate(dev(a), dev(c), o)
    assert np.all(np.abs(host(o) - c.T @ a) <= 1060 * EPS * (np.abs(c).T @ np.abs(a)))
    ctx.close()

"""The fixed-point FP64 transforms at the ends of the range: orbitals without a normal number, and per-G
factors far below the largest one of the grid."""
import numpy as np
import pytest

from oracle.grid import Grid, kb_projectors, local_potential
from oracle.hamiltonian import Hamiltonian
from tests.gpu_common import R, dev, host, need_gpu, torch
from workloads import draw_e_kb, draw_x0

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("natom", [0, 4])
@pytest.mark.parametrize("bits", [3, 20, 40])
def test_subnormal_orbitals(bits, natom):
    """Orbitals whose values are whole numbers of 2^-1074, of at most `bits` bits.  In these units T and V psi are
    rounded to whole numbers once or twice each, and their sum is whole: off by at most 2, beside the FP64
    form's 1e-12 of the largest value.  With projectors, every subnormal step of an atom's coefficients
    rounds to half a unit as well, in any FP64 form: some 16 disc sums (norm 0.6, dV 0.018: 0.2), the projection
    (0.5), times E c <= 1.2 (0.5), by four projectors of at most 1, 0.6, 0.6, 0.6, and the coefficients of the
    discs (1.2): 5 an atom, 20 where all four overlap."""
    need_gpu()
    N, L = (24, 20, 16), (6.0, 5.0, 4.5)
    pos = np.random.default_rng(3).uniform(0.0, 1.0, (4, 3)) * np.array(L)
    g = Grid(L=L, N=N)
    v = local_potential(g, pos, 4.0, 0.6)
    if natom:
        e = draw_e_kb(4, 4, 4)
        ham = Hamiltonian(g, v, kb_projectors(g, pos, 1.0, 2.0, e, 4))
        ctx = R.Context(L, N, v, pos, 1.0, 2.0, e, 4)
    else:
        ham, ctx = Hamiltonian(g, v), R.Context(L, N, v)
    x = draw_x0(3, 2, ctx.n)
    x = np.round(x.real * 2.0 ** (bits - 3)) + 1j * np.round(x.imag * 2.0 ** (bits - 3))
    x[1, : ctx.n // 2] = 0.0                     # planes of zeros beside them
    h = torch.empty(2, ctx.n, dtype=torch.complex128, device="cuda")
    ctx.apply_h(dev(np.ldexp(x.view(np.float64), -1074).view(np.complex128)), h)
    got = np.ldexp(host(h).view(np.float64), 1074)
    ref = ham.apply(x).view(np.float64)
    assert np.max(np.abs(got - ref)) <= 2.0 + 5.0 * natom + 1e-12 * np.max(np.abs(ref))
    ctx.close()


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_factors_far_below_the_largest(axis):
    """A plane wave of alternating signs along one axis of a cell of very unequal grid spacings: its transform is
    exact, so the result is the input times one factor, and that keeps FP64's relative precision
    however small it is (the largest kinetic factor is 2^41 times the smallest here).  Roundings of 2^-53: G^2
    from G 3, the kinetic and the Hartree factor 4, the rational TPA function twice those of x and 14, the
    result and its product with 1/n 2."""
    need_gpu()
    N, L = (16, 24, 12), (30000.0, 100.0, 3.0)
    ctx = R.Context(L, N, np.zeros(N[0] * N[1] * N[2]))
    i = np.meshgrid(*[np.arange(m) for m in N[::-1]], indexing="ij")[2 - axis]
    x = (1.0 - 2.0 * (i % 2)).reshape(-1)
    g2 = (np.longdouble(np.pi) * N[axis] / np.longdouble(L[axis])) ** 2
    h = torch.empty(1, ctx.n, dtype=torch.complex128, device="cuda")

    def close(got, factor, roundings):
        return np.all(np.abs(got - x * float(factor)) <= roundings * 2.0 ** -53 * float(factor))

    ctx.apply_h(dev(x[None] + 0j), h)
    assert close(host(h)[0], g2 / 2, 10)
    v = torch.empty(ctx.n, dtype=torch.float64, device="cuda")
    ctx.hartree(dev(x), v)
    assert close(host(v), 4 * np.longdouble(np.pi) / g2, 10)
    for t in (1.0, 1e-3, 1e-6, 1e-9, 1e-12):
        ctx.precondition_tpa(dev(x[None] + 0j), h, dev(np.array([t])))
        q = g2 / 2 / np.longdouble(t)
        p = 27 + q * (18 + q * (12 + 8 * q))
        assert close(host(h)[0], p / (p + 16 * q ** 4), 24), t
    ctx.close()

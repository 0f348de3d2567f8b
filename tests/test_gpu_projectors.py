"""The Kleinman-Bylander discs against the oracle's point tables: windows beyond a warp, atoms across
every cell edge, one and four projectors, more discs in a plane than are staged at a time, planes
that leave room for two, bands of very different size.

Tolerances are those of the operator tests: 1e-12 of max |H psi| and 1e-13 of max |p| in FP64;
2e-6 of max |H psi| in FP32, plus a rounding of 2^-24 for each of the at most natom overlapping
terms."""
import numpy as np
import pytest

from oracle.grid import Grid, kb_projectors
from oracle.hamiltonian import Hamiltonian
from tests.gpu_common import R, dev, host, need_gpu, rel_err, torch
from workloads import draw_e_kb, draw_x0

pytestmark = pytest.mark.gpu

CASES = [((20, 18, 15), (6.0, 5.0, 4.5), 3, 2.2, 4), ((64, 40, 30), (8.0, 8.2, 8.4), 5, 3.9, 4),
         ((30, 32, 25), (6.0, 6.0, 6.0), 90, 2.9, 4), ((120, 120, 4), (24.0, 24.0, 6.0), 12, 2.9, 4),
         ((24, 27, 16), (6.0, 6.0, 6.0), 4, 2.5, 1), ((96, 3, 128), (10.0, 6.1, 10.0), 4, 3.0, 4)]


@pytest.mark.parametrize("N,L,natom,rcut,nproj", CASES)
def test_discs_match_the_oracle(N, L, natom, rcut, nproj):
    need_gpu()
    rng = np.random.default_rng(natom)
    pos = rng.uniform(0.0, 1.0, (natom, 3)) * np.array(L)
    pos[0] = 0.0                                    # an atom on the cell's corner
    e = draw_e_kb(natom, natom, nproj)
    g = Grid(L=L, N=N)
    P = kb_projectors(g, pos, 1.0, rcut, e, nproj)
    ham = Hamiltonian(g, np.zeros(g.n), P)
    ctx = R.Context(L, N, np.zeros(N[0] * N[1] * N[2]), pos, 1.0, rcut, e, nproj)
    x = draw_x0(7, 5, ctx.n)
    x[1] *= 1e-30
    x[2] *= 1e30
    x[3] = 0.0
    ref = ham.apply(x)
    h = torch.empty(5, ctx.n, dtype=torch.complex128, device="cuda")
    ctx.apply_h(dev(x), h)
    h = host(h)
    for b in (0, 1, 2, 4):
        assert rel_err(h[b], ref[b]) < 1e-12, b
    assert np.all(h[3] == 0)
    p = torch.empty(5, natom * nproj, dtype=torch.complex128, device="cuda")
    ctx.project(dev(x), p)
    q = ham.project(x).T
    for b in (0, 1, 2, 4):
        assert rel_err(host(p)[b], q[b]) < 1e-13, b
    h32 = torch.empty(2, ctx.n, dtype=torch.complex64, device="cuda")
    ctx.apply_h(dev(x[[0, 4]].astype(np.complex64)), h32, R.MIXED)
    h32 = host(h32)
    tol = 2e-6 + natom * 2.0 ** -24
    assert rel_err(h32[0], ref[0]) < tol and rel_err(h32[1], ref[4]) < tol
    ctx.close()

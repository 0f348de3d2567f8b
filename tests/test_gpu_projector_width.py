"""Kleinman-Bylander projectors against the oracle's point tables from widths well above the grid's spacing to
far below it, where an axis' largest factor is some e^-65 and only the normalisation makes it count.

Tolerances: the operator tests' 1e-12 of max |H psi| in FP64, for the projections too (the exponents reach 200, so
that both sides' factors are off by 200 x 2^-53 and normalised), 2e-6 in FP32."""
import numpy as np
import pytest

from oracle.grid import Grid, kb_projectors
from oracle.hamiltonian import Hamiltonian
from tests.gpu_common import R, dev, host, need_gpu, rel_err, torch
from workloads import draw_e_kb, draw_x0

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nproj", [1, 4])
@pytest.mark.parametrize("rc", [1.0, 0.2, 0.05, 0.035])
def test_projectors_of_any_width(rc, nproj):
    need_gpu()
    N, L = (12, 15, 10), (9.6, 9.0, 8.0)
    pos = np.random.default_rng(3).uniform(0.0, 1.0, (5, 3)) * np.array(L)
    e = draw_e_kb(5, 5, nproj)
    g = Grid(L=L, N=N)
    ham = Hamiltonian(g, np.zeros(g.n), kb_projectors(g, pos, rc, 1.9, e, nproj))
    ctx = R.Context(L, N, np.zeros(g.n), pos, rc, 1.9, e, nproj)
    x = draw_x0(7, 2, ctx.n)
    h = torch.empty(2, ctx.n, dtype=torch.complex128, device="cuda")
    ctx.apply_h(dev(x), h)
    assert rel_err(host(h), ham.apply(x)) < 1e-12
    p = torch.empty(2, 5 * nproj, dtype=torch.complex128, device="cuda")
    ctx.project(dev(x), p)
    assert rel_err(host(p), ham.project(x).T) < 1e-12
    h32 = torch.empty(2, ctx.n, dtype=torch.complex64, device="cuda")
    ctx.apply_h(dev(x.astype(np.complex64)), h32, R.MIXED)
    assert rel_err(host(h32), ham.apply(x)) < 2e-6
    ctx.close()

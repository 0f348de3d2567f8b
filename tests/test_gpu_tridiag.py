"""The double-float tridiagonalisation at the sizes where rows per CTA (16 CTAs), pieces of a row (the
table's steps at 3, 17 and 25 rows) and blocks of columns change.  Tolerances: 48-bit double-float,
a few units a step over at most 448 steps, 2e-11 |A|; orthonormality is the inverse iteration's, 3e-10."""
import numpy as np
import pytest

from tests.gpu_common import R, dev, host, need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [2, 3, 15, 16, 31, 33, 49, 129, 257, 272, 385, 401, 447])
def test_sizes_around_the_rows_of_a_cta(k):
    need_gpu()
    rng = np.random.default_rng(k)
    a = rng.standard_normal((k, k)) + 1j * rng.standard_normal((k, k))
    a = a + a.conj().T
    if k == 33:
        a[5:, :5] = a[:5, 5:] = 0       # a column that is reduced already
    ctx = R.Context((5.0, 5.0, 5.0), (6, 6, 6), np.zeros(216))
    ctx.set_dense(R.DENSE_DF)
    keep = max(1, k // 3)
    z = torch.empty((k, keep), dtype=torch.complex128, device="cuda")
    lam, Z = ctx.eigh(dev(a), keep, z), host(z)
    nrm = np.linalg.norm(a, 2)
    assert np.max(np.abs(lam - np.linalg.eigvalsh(a)[:keep])) < 2e-11 * nrm
    assert np.max(np.abs(Z.conj().T @ Z - np.eye(keep))) < 3e-10
    assert np.max(np.abs(a @ Z - Z * lam)) < 2e-11 * nrm
    ctx.close()

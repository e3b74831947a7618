"""The allocation-free scaling on matrices with NaN and infinite entries, and
with entries at both ends of the double range: a line's maximum leaves NaN
entries out (fmax), an infinite one gives the factor infinity.  The Ruiz passes
are maxima, square roots and divisions, each correctly rounded, so numpy's are
the same bits."""

import numpy as np
import pytest
import scipy.sparse as sp

from paper_2311_12180_gb300 import pdlp as P

pytestmark = pytest.mark.gpu


def _ruiz(K, iters):
    rows = np.repeat(np.arange(K.shape[0]), np.diff(K.indptr))
    v, D1, D2 = K.data.copy(), np.ones(K.shape[0]), np.ones(K.shape[1])
    with np.errstate(all="ignore"):
        for _ in range(iters):
            r, s = np.zeros(K.shape[0]), np.zeros(K.shape[1])
            np.fmax.at(r, rows, np.abs(v))
            np.fmax.at(s, K.indices, np.abs(v))
            r, s = (np.where(f > 0.0, np.sqrt(f), 1.0) for f in (r, s))
            v = v / r[rows] / s[K.indices]
            D1, D2 = D1 / r, D2 / s
    return v, D1, D2


@pytest.mark.parametrize("m,n", [(1, 1), (7, 40), (300, 170)])
@pytest.mark.parametrize("values", ["nan", "inf", "nan and inf", "range"])
def test_ruiz_passes_on_extreme_entries(m, n, values):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(m + n)
    mask = rng.random((m, n)) < 0.3
    mask[:, 0] = True
    K = sp.csr_matrix(mask.astype(np.float64))
    K.data = rng.standard_normal(K.nnz)
    pick = rng.random(K.nnz) < 0.05
    pick[0] = True  # the first row has one; in the smallest matrix nothing else
    if "nan" in values:
        K.data[pick] = np.where(rng.random(pick.sum()) < 0.5, np.nan, -np.nan)
    if "inf" in values:
        K.data[np.roll(pick, 3) if K.nnz > 3 else pick] = -np.inf
    if values == "range":
        K.data *= 10.0 ** rng.integers(-305, 305, K.nnz)
        K.data[pick] = 5e-324
    KT = K.T.tocsr()
    KT.sort_indices()
    dev = torch.device("cuda", 0)
    t = lambda a, dt: torch.tensor(np.ascontiguousarray(a), dtype=dt, device=dev)
    d = [t(K.indptr, torch.int32), t(K.indices, torch.int32), t(K.data, torch.float64),
         t(KT.indptr, torch.int32), t(KT.indices, torch.int32), t(KT.data, torch.float64)]
    D1, D2 = torch.empty(m, dtype=torch.float64, device=dev), torch.empty(n, dtype=torch.float64, device=dev)
    P.pdlp_scale_device_noalloc(m, n, *(a.data_ptr() for a in d), 4, -1.0, D1.data_ptr(), D2.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    v, r1, r2 = _ruiz(K, 4)
    vt = sp.csr_matrix((np.arange(K.nnz) + 1.0, K.indices, K.indptr), shape=(m, n)).T.tocsr()
    vt.sort_indices()
    for got, want in ((D1, r1), (D2, r2), (d[2], v), (d[5], v[vt.data.astype(np.int64) - 1])):
        np.testing.assert_array_equal(got.cpu().numpy(), want)

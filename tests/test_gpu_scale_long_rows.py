"""The allocation-free scaling where rows and columns are of very different
lengths: the rows that get a warp each (more than 48 entries) next to the ones
that share one, and few long lines.  The Ruiz passes bit for bit, the
Pock-Chambolle pass up to the order of its sums."""

import numpy as np
import pytest
import scipy.sparse as sp

from paper_2311_12180_gb300 import pdlp as P
from test_gpu_scale_nonfinite import _ruiz

pytestmark = pytest.mark.gpu


def _matrix(lens, n, seed=0):
    rng = np.random.default_rng(seed)
    lens = np.minimum(np.asarray(lens, dtype=np.int64), n)
    ptr = np.concatenate([[0], np.cumsum(lens)])
    start = rng.integers(0, n, lens.size)
    rows = np.repeat(np.arange(lens.size), lens)
    cols = (start[rows] + 7919 * (np.arange(ptr[-1]) - ptr[rows])) % n  # distinct in a row: n is no multiple of 7919
    K = sp.csr_matrix((rng.standard_normal(ptr[-1]) * 10.0 ** rng.integers(-3, 4, ptr[-1]), cols, ptr), shape=(lens.size, n))
    K.sort_indices()
    return K


class _Scaler:
    def __init__(self, K):
        import torch

        self.torch, self.K, self.KT = torch, K, K.T.tocsr()
        self.KT.sort_indices()
        dev = torch.device("cuda", 0)
        t = lambda a, dt: torch.tensor(np.ascontiguousarray(a), dtype=dt, device=dev)
        self.d = [t(a, dt) for M in (K, self.KT)
                  for a, dt in ((M.indptr, torch.int32), (M.indices, torch.int32), (M.data, torch.float64))]
        self.D = [torch.empty(k, dtype=torch.float64, device=dev) for k in K.shape]

    def __call__(self, pc_alpha):
        P.pdlp_scale_device_noalloc(*self.K.shape, *(a.data_ptr() for a in self.d), 10, pc_alpha, self.D[0].data_ptr(),
                                    self.D[1].data_ptr(), self.torch.cuda.current_stream().cuda_stream)

    def results(self):
        self.torch.cuda.synchronize()
        return [a.cpu().numpy() for a in (self.d[2], self.D[0], self.D[1], self.d[5])]


rng = np.random.default_rng(1)
SHAPES = {
    "one row": ([3000], 5000),
    "around the limit": (np.arange(40, 60), 999),
    "long in a group": ([3, 49, 0, 1, 48, 4000, 50, 2] * 5 + [7], 4500),
    "adjacent long": (np.concatenate([np.full(12000, 4), np.full(70, 2500), np.full(100, 3)]), 30000),
    "wide": (np.full(60, 3001), 20011),
    "tall": (rng.integers(0, 30, 11000), 150),
    "mixed": (np.where(rng.random(3000) < 0.1, rng.integers(49, 400, 3000), rng.integers(0, 49, 3000)), 700),
}


@pytest.mark.parametrize("shape", SHAPES)
def test_rows_of_all_lengths(shape):
    pytest.importorskip("torch")
    K = _matrix(*SHAPES[shape])
    ruiz = _Scaler(K)
    ruiz(-1.0)
    got = ruiz.results()
    v, r1, r2 = _ruiz(K, 10)
    for a, b in zip(got, (v, r1, r2)):
        np.testing.assert_array_equal(a, b)
    both = _Scaler(K)
    both(1.0)
    v2, D1, D2, vt = both.results()
    rows = np.repeat(np.arange(K.shape[0]), np.diff(K.indptr))
    s1, s2 = np.zeros(K.shape[0]), np.zeros(K.shape[1])
    np.add.at(s1, rows, np.abs(v))
    np.add.at(s2, K.indices, np.abs(v))
    s1, s2 = (np.where(f > 0.0, np.sqrt(f), 1.0) for f in (s1, s2))
    for a, b in ((v2, v / s1[rows] / s2[K.indices]), (D1, r1 / s1), (D2, r2 / s2)):
        np.testing.assert_allclose(a, b, rtol=1e-12)  # sums of up to 1e4 terms in another order
    Kt = sp.csr_matrix((v2, K.indices, K.indptr), shape=K.shape).T.tocsr()
    Kt.sort_indices()
    assert np.array_equal(Kt.data, vt)  # K' stays the exact transpose


def test_few_long_columns_cost_no_more_than_their_entries():
    """The time of 300 columns of about 6000 entries against that of as many
    entries spread over 20000 columns; one warp per eight columns made it 13
    times as long, a warp per column 1.5 to 2 times."""
    torch = pytest.importorskip("torch")
    times = []
    for K in (_matrix(np.full(10007, 180), 300), _matrix(np.full(20000, 90), 20000)):
        s = _Scaler(K)
        best = np.inf
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            s(1.0)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        times.append(best)
    assert times[0] < 6.0 * times[1], times

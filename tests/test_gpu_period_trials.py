"""Rejected trials in the one-launch check period, on one cluster and on the
whole GPU: the shortest primal half-steps, one right after another's totals,
so the reuse of the partial sums of ||dx||^2 is exercised where a CTA can be
furthest ahead.  Bit for bit the step kernels' results."""

import numpy as np
import pytest

import lpgen
from paper_2311_12180_gb300 import pdlp as P

pytestmark = pytest.mark.gpu

SMS = 152  # of a GB300


def _ragged(m, n, longest, most):
    """Rows of up to `longest` entries among rows of fewer than `most`, and a dense column."""
    rng = np.random.default_rng(9)
    lens = np.concatenate([[longest, 0, 0, 1024, 1025, 49, 48, 47, 33, 32, 31], rng.integers(0, most, m - 11)])
    row_ptr, cols = lpgen._sample_rows(rng, lens, n)
    rows = np.repeat(np.arange(m, dtype=np.int64), np.diff(row_ptr))
    key = np.unique(np.concatenate([rows * n + cols, np.arange(100, 400, dtype=np.int64) * n + 7]))
    rows, cols = key // n, key % n
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=m))])
    return lpgen.plant(rng, m, n, m // 3, row_ptr, cols, rng.standard_normal(cols.size), np.zeros(n), np.full(n, 10.0))


@pytest.mark.parametrize("shape", [(700, 3000, 2500, 6), (9000, 30000, 20000, 12)])  # one cluster, the whole GPU
@pytest.mark.parametrize("period", [8, 64])
def test_rejected_trials_equal_the_step_kernels(shape, period):
    N = 400
    with P.Solver(_ragged(*shape), check_period=period) as s:
        assert s.layout()["period_ctas"] == (16 if shape[0] == 700 else SMS)
        runs = []
        for _ in range(3):
            a = s.solve(tol=1e-14, max_iter=N)
            runs.append((a, s.info()))
        s.begin(tol=1e-14, max_iter=N)
        s.time_kernels(N)
        b = s.finish()
        ib = s.info()
    assert ib["attempts"] >= b[3] + 3  # trials were rejected
    for a, ia in runs:
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[2:] == b[2:]
        assert all(ia[f] == ib[f] for f in ("attempts", "restarts", "checks", "omega", "eta_hat", "pobj", "dobj"))

"""The one-launch check period (small LPs) against the FP64 oracle, and bit for
bit against the step and check kernels, where its rules change: one cluster or the whole GPU, the matrix resident in shared
memory or not, the largest LPs that still take it and the first that do not,
no rows at all, long rows next to empty ones, FP32 values and a QP.

Tolerance: both sides compute the same formulas in FP64 and differ only in
summation order, O(1e-16) per step, which adaptive-step PDHG amplifies by at
most a few orders of magnitude over these horizons: rtol 1e-9 with a floor of
1e-9 max|x|, as in the parity tests."""

import numpy as np
import pytest

import lpgen
import oracle
from paper_2311_12180_gb300 import pdlp as P

pytestmark = pytest.mark.gpu


def _large(m, n, nnz):
    return lpgen.large_lp(4, m=m, n=n, nnz=nnz)


def _ragged():
    """Rows of 1 to 2500 entries and empty ones; a column of 300 entries."""
    rng = np.random.default_rng(9)
    m, n = 700, 3000
    lens = np.concatenate([[2500, 0, 0, 1024, 1025, 49, 48, 47, 33, 32, 31], rng.integers(0, 6, m - 11)])
    row_ptr, cols = lpgen._sample_rows(rng, lens, n)
    rows = np.repeat(np.arange(m, dtype=np.int64), np.diff(row_ptr))
    key = np.unique(np.concatenate([rows * n + cols, np.arange(100, 400, dtype=np.int64) * n + 7]))
    rows, cols = key // n, key % n
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=m))])
    return lpgen.plant(rng, m, n, 300, row_ptr, cols, rng.standard_normal(cols.size), np.zeros(n), np.full(n, 10.0))


def _no_rows():
    rng = np.random.default_rng(3)
    n = 77
    return lpgen.plant(rng, 0, n, 0, np.zeros(1, np.int64), np.zeros(0, np.int64), np.zeros(0), np.zeros(n), np.ones(n))


CASES = {
    "one_column": lambda: lpgen.random_boxed_lp(1, 1, 1, 1),
    "one_cluster": lambda: lpgen.tiny_lp(5, m_eq=300, m_ineq=200, n=1100, density=0.03),
    "whole_gpu": lambda: _large(3000, 6000, 60000),
    "resident_edge": lambda: _large(61000, 120000, 1200000),
    "not_resident": lambda: _large(110000, 220000, 2200000),
    "step_kernels": lambda: _large(170000, 330000, 3300000),
    "ragged": _ragged,
}


@pytest.mark.parametrize("case,bits,qp,period,N", [
    ("one_column", 64, False, 4, 10),
    ("one_cluster", 64, False, 16, 50),
    ("one_cluster", 32, True, 64, 40),
    ("whole_gpu", 64, False, 16, 50),
    ("whole_gpu", 32, False, 64, 40),
    ("resident_edge", 64, True, 16, 20),
    ("not_resident", 64, False, 16, 20),
    ("not_resident", 32, False, 64, 20),
    ("step_kernels", 64, False, 16, 20),
    ("ragged", 64, False, 8, 40),
])
def test_period_matches_oracle(case, bits, qp, period, N):
    lp = CASES[case]()
    if qp:
        lp = lpgen.planted_qp(lp, seed=2)
    with P.Solver(lp, check_period=period, value_bits=bits) as s:
        x, y, st, it = s.solve(tol=1e-14, max_iter=N)
        info = s.info()
        # the general path: the step and check kernels one by one, bit for bit the same
        s.begin(tol=1e-14, max_iter=N)
        s.time_kernels(-(-N // period))
        x2, y2, st2, it2 = s.finish()
    r = oracle.solve(lp, tol=1e-14, max_iter=N, check_period=period, **({"step_value_bits": 32} if bits == 32 else {}))
    assert np.array_equal(x, x2) and np.array_equal(y, y2) and (st, it) == (st2, it2)
    assert (st, it) == (r.status, r.iters)
    assert info["attempts"] == r.attempts and info["restarts"] == r.restarts
    np.testing.assert_allclose(x, r.x, rtol=1e-9, atol=1e-9 * max(1.0, np.abs(r.x).max()))
    np.testing.assert_allclose(y, r.y, rtol=1e-9, atol=1e-9 * max(1.0, np.abs(r.y).max()))


@pytest.mark.parametrize("case,period,N", [("one_cluster", 8, 700), ("whole_gpu", 16, 400), ("ragged", 8, 400)])
def test_long_runs_equal_the_step_kernels(case, period, N):
    """Many checks and restarts, and rejected trials where the LP has them: the same bits."""
    lp = CASES[case]()
    with P.Solver(lp, check_period=period) as s:
        a = s.solve(tol=1e-14, max_iter=N)
        ia = s.info()
        s.begin(tol=1e-14, max_iter=N)
        s.time_kernels(N)
        b = s.finish()
        ib = s.info()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[2:] == b[2:]
    assert all(ia[f] == ib[f] for f in ("attempts", "restarts", "checks", "omega", "eta_hat", "pobj", "dobj", "rp_norm"))
    assert ia["restarts"] > 0


def test_no_rows():
    lp = _no_rows()
    with P.Solver(lp) as s:
        x, y, st, it = s.solve(tol=1e-8, max_iter=10_000)
    r = oracle.solve(lp, tol=1e-8, max_iter=10_000)
    assert st == r.status == P.OPTIMAL and y.size == 0
    assert abs(float(lp.c @ x) - lp.obj_star) <= 1e-6 * (1 + abs(lp.obj_star))


def test_two_solvers_on_two_streams_share_nothing():
    """Two solvers stepping in turn without waiting give what each gives alone."""
    a_lp, b_lp = lpgen.tiny_lp(1), _large(3000, 6000, 60000)
    with P.Solver(a_lp) as a, P.Solver(b_lp) as b:
        ra, rb = a.solve(tol=1e-14, max_iter=256), b.solve(tol=1e-14, max_iter=256)
        a.begin(tol=1e-14, max_iter=256)
        b.begin(tol=1e-14, max_iter=256)
        for _ in range(8):
            a.run_periods(1)
            b.run_periods(1)
        fa, fb = a.finish(), b.finish()
    assert np.array_equal(ra[0], fa[0]) and np.array_equal(ra[1], fa[1])
    assert np.array_equal(rb[0], fb[0]) and np.array_equal(rb[1], fb[1])

"""Which LPs run a check period in one launch: those whose iteration it makes
shorter.  Shapes on both sides of each line (stored entries, long rows, slices
with the matrix resident or not, long rows on one cluster, FP32 values), and the
step kernels' bits on all of them."""

import numpy as np
import pytest

import lpgen
from paper_2311_12180_gb300 import pdlp as P

pytestmark = pytest.mark.gpu

SMS = 152  # of a GB300


def _rows(m, n, k):
    rng = np.random.default_rng(1)
    row_ptr, cols = lpgen._sample_rows(rng, np.full(m, k), n)
    return lpgen.plant(rng, m, n, m // 3, row_ptr, cols, rng.standard_normal(cols.size), np.zeros(n), np.full(n, 10.0))


def _transport(sources, sinks):
    fam = lpgen.transport_family(0, sources, sinks)
    return lpgen.transport_lp(fam, lpgen.transport_thetas(1, 0)[0], 0)


CASES = [
    ("cluster", lambda: lpgen.tiny_lp(1), 16),
    ("FP32 2e5", lambda: lpgen.large_lp(3, m=10000, n=20000, nnz=200000), SMS),
    ("FP32 5e5", lambda: lpgen.large_lp(3, m=25000, n=50000, nnz=500000), 0),
    ("340 long rows", lambda: _rows(170, 170, 70), 16),
    ("600 long rows", lambda: _rows(300, 300, 100), SMS),
    ("power law 2e6", lambda: lpgen.large_lp(3, m=100000, n=200000, nnz=2000000), SMS),
    ("power law 2.4e6", lambda: lpgen.large_lp(3, m=120000, n=240000, nnz=2400000), 0),
    ("14000 long rows", lambda: _rows(7000, 7000, 60), SMS),
    ("29000 long rows", lambda: _rows(15000, 15000, 60), 0),
    ("16900 slices, resident", lambda: _transport(600, 900), SMS),
    ("18800 slices", lambda: _transport(600, 1000), 0),
    ("15600 slices, not resident", lambda: _rows(250000, 250000, 5), 0),
]


@pytest.mark.parametrize("name,lp,ctas", CASES, ids=[c[0] for c in CASES])
def test_path(name, lp, ctas):
    with P.Solver(lp(), check_period=16, value_bits=32 if "FP32" in name else 64) as s:
        assert s.layout()["period_ctas"] == ctas
        a = s.solve(tol=1e-14, max_iter=40)
        s.begin(tol=1e-14, max_iter=40)
        s.time_kernels(3)
        b = s.finish()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[2:] == b[2:]

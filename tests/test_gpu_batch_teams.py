"""Teams of 4, 8 and 16 CTAs on the same large LPs: the size follows from the
batch's composition, the results must not."""

import numpy as np
import pytest

import lpgen
import oracle
from paper_2311_12180_gb300 import pdlp as P

pytestmark = pytest.mark.gpu

N = 24  # short horizon: identical decisions, and rounding differences (x10 in ten iterations) stay below 1e-9


def large(kind):
    if kind == "odd":  # row and column counts that are no multiple of a warp
        return lpgen.tiny_lp(43, m_eq=601, m_ineq=598, n=3001, density=0.02)
    if kind == "wide":  # fewer rows than one CTA has threads
        return lpgen.tiny_lp(44, m_eq=21, m_ineq=18, n=2999, density=0.4)
    return lpgen.tiny_lp(45, m_eq=1500, m_ineq=1499, n=301, density=0.05)  # tall


@pytest.mark.parametrize("kind", ["odd", "wide", "tall"])
def test_team_size_does_not_change_the_results(kind):
    lp = large(kind)
    assert lp.val.size >= 32768  # a team's LP
    small = lpgen.batch_lps(20, seed=5, m_lo=10, m_hi=60)
    got = {}
    for copies in (34, 17, 2):  # one full round of teams of 4, of 8, and a nearly empty chip
        with P.BatchSolver(small + [lp] * copies) as b:
            s = b.stats()
            xs, ys, st, it = b.solve(tol=1e-14, max_iter=N)
        assert s["team_lps"] == copies
        for i in range(len(small), len(small) + copies):
            got.setdefault(int(s["team_size"]), []).append((xs[i], ys[i], st[i], it[i]))
    assert set(got) == {4, 8, 16}
    r = oracle.solve(lp, tol=1e-14, max_iter=N)
    x0, y0, st0, it0 = got[4][0]
    assert st0 == r.status and it0 == r.iters
    np.testing.assert_allclose(x0, r.x, rtol=1e-9, atol=1e-9 * max(1.0, np.abs(r.x).max()))
    np.testing.assert_allclose(y0, r.y, rtol=1e-9, atol=1e-9 * max(1.0, np.abs(r.y).max()))
    for size, runs in got.items():
        for x, y, st, it in runs:
            assert st == st0 and it == it0 and np.array_equal(x, x0) and np.array_equal(y, y0), size

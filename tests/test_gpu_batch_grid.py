"""A batch holds the SMs it has use for: no more teams than large LPs, no more
single CTAs than small ones, so that batches on several streams fit side by
side; the results do not depend on it."""

import threading

import numpy as np
import pytest

import lpgen
from paper_2311_12180_gb300 import pdlp as P

pytestmark = pytest.mark.gpu

SMS = 152  # of a GB300


def _lps(small, large):
    lps = [lp for lp in lpgen.batch_lps(small + 10, seed=5, m_lo=10, m_hi=80) if lp.val.size < 32768][:small]
    return lps + [lpgen.tiny_lp(60 + i, m_eq=500, m_ineq=500, n=2200, density=0.02) for i in range(large)]


@pytest.mark.parametrize("small,large", [(20, 1), (19, 1), (30, 6), (60, 0), (0, 20), (140, 3), (170, 0), (18, 1)])
def test_grid_follows_the_batch(small, large):
    lps = _lps(small, large)
    with P.BatchSolver(lps) as b:
        s = b.stats()
        xs, ys, st, it = b.solve(tol=1e-14, max_iter=40)
    with_teams = small + large >= 20 and large > 0
    assert s["team_lps"] == (large if with_teams else 0)
    if with_teams:
        assert s["grid"] <= min(SMS, large * s["team_size"] + small)
    else:
        assert s["grid"] == min(SMS, small + large)
    # each small LP as in a batch of its own kind
    with P.BatchSolver(lps[:small][:19] or lps[:1]) as b:
        x2, y2, st2, it2 = b.solve(tol=1e-14, max_iter=40)
    for i in range(min(small, 19)):
        assert np.array_equal(xs[i], x2[i]) and np.array_equal(ys[i], y2[i]) and (st[i], it[i]) == (st2[i], it2[i])


def test_concurrent_batches_equal_batches_alone():
    sets = [_lps(20, 1), _lps(60, 0), _lps(30, 6), _lps(25, 2)]
    batches = [P.BatchSolver(s) for s in sets]
    alone = [b.solve(tol=1e-14, max_iter=130) for b in batches]
    got = [None] * len(sets)

    def work(i):
        got[i] = batches[i].solve(tol=1e-14, max_iter=130)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sets))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for b in batches:
        b.close()
    for a, g in zip(alone, got):
        assert all(np.array_equal(u, v) for k in (0, 1) for u, v in zip(a[k], g[k]))
        assert np.array_equal(a[2], g[2]) and np.array_equal(a[3], g[3])

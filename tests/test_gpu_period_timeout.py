"""The one-launch period's grid barrier gives up after 2 s: the call that sees it
fails, and whatever comes next on the same solver starts afresh.  The wait is
made to run out by a CTA that leaves at once (PDLP_TEST_PERIOD_STALL)."""

import numpy as np
import pytest

import lpgen
from paper_2311_12180_gb300 import pdlp as P

pytestmark = pytest.mark.gpu

STALL = "PDLP_TEST_PERIOD_STALL"


@pytest.fixture(scope="module")
def lp():
    return lpgen.large_lp(4, m=3000, n=6000, nnz=60000)  # a period on the whole GPU


def _same(a, b):
    return np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[2:] == b[2:]


def _timed_out(call):
    with pytest.raises(P.PdlpError) as e:
        call()
    assert e.value.code == P.ERR_CUDA and "timed out" in str(e.value)


def test_solve_reports_the_timeout_and_the_next_is_normal(lp, monkeypatch):
    with P.Solver(lp, check_period=16) as s:
        ok = s.solve(tol=1e-14, max_iter=200)
        monkeypatch.setenv(STALL, "1")
        _timed_out(lambda: s.solve(tol=1e-14, max_iter=200))
        monkeypatch.delenv(STALL)
        assert _same(s.solve(tol=1e-14, max_iter=200), ok)


def test_poll_reports_the_timeout_and_begin_or_set_state_clear_it(lp, monkeypatch):
    with P.Solver(lp, check_period=16) as s:
        ok = s.solve(tol=1e-14, max_iter=200)
        s.begin(tol=1e-14, max_iter=200)
        s.run_periods(3)
        state = s.get_state()
        for recover in (lambda: s.begin(tol=1e-14, max_iter=200), lambda: s.set_state(state)):
            monkeypatch.setenv(STALL, "1")
            s.begin(tol=1e-14, max_iter=200)
            s.run_periods(2)
            _timed_out(s.poll)
            _timed_out(s.poll)  # and again until the state is written anew
            monkeypatch.delenv(STALL)
            recover()
            assert _same(s.resume(), ok)

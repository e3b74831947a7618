"""Solvers of small LPs on several threads and streams: the path of a period
follows from how many have work in flight, the results must not."""

import threading

import numpy as np
import pytest

import lpgen
from paper_2311_12180_gb300 import pdlp as P

pytestmark = pytest.mark.gpu

N = 700


def _same(a, b):
    return np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[2:] == b[2:]


def test_concurrent_solves_equal_solves_alone():
    lps = [lpgen.large_lp(1, m=3000, n=6000, nnz=60000), lpgen.large_lp(2, m=20000, n=40000, nnz=400000),
           lpgen.large_lp(3, m=5000, n=10000, nnz=100000), lpgen.tiny_lp(4)]
    solvers = [P.Solver(lp, check_period=16) for lp in lps]
    alone = [s.solve(tol=1e-14, max_iter=N) for s in solvers]
    got = [[] for _ in lps]
    gate = threading.Barrier(len(lps))

    def work(i):
        gate.wait()
        for _ in range(1 + 3 * (i % 2)):  # some end while others go on: both paths within a solve
            got[i].append(solvers[i].solve(tol=1e-14, max_iter=N))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(lps))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    again = [s.solve(tol=1e-14, max_iter=N) for s in solvers]
    for s in solvers:
        s.close()
    for i, want in enumerate(alone):
        assert len(got[i]) == 1 + 3 * (i % 2) and all(_same(g, want) for g in got[i] + [again[i]]), i

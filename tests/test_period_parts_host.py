"""Where the one-launch check period keeps its partial sums (csrc/pdlp_period.cuh),
no GPU: no place is read by one CTA while another may write it, by the order
of the phases and barriers, and all of them fit the room a solver reserves.

Barrier numbers: trial t passes barriers 2 t + 1 (after the primal half-step)
and 2 t + 2 (after the dual one).  An access lies behind the wait of barrier
`after` and before the arrival at barrier `before`; one CTA's access is ordered
before another's if it comes before the arrival at a barrier whose wait the
other is behind."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("parts") / "period_parts_host")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-x", "cu", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "paper_2311_12180_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "period_parts_host.cpp"), "-o", out], check=True)
    return out


@pytest.mark.parametrize("cluster,grid,groups", [
    (1, 16, (1, 1, 1, 1, 1, 1)), (1, 16, (5, 3, 5, 3, 2, 2)), (1, 16, (512,) * 6),
    (0, 152, (1, 1, 1, 1, 1, 1)), (0, 152, (151, 152, 153, 303, 7, 7)), (0, 152, (608, 608, 304, 456, 1064, 1215)),
    (0, 152, (1216,) * 6), (0, 148, (1183,) * 6),
])
def test_partial_sums_are_not_written_while_they_are_read(exe, cluster, grid, groups):
    text = " ".join(map(str, (cluster, grid) + groups))
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    room = int(out[0])
    spans = [tuple(map(int, line.split())) for line in out[1:10]]
    primal, dual, once = spans[:4], spans[4], spans[5:]
    assert max(at + n for at, n in spans) <= room
    overlap = lambda p, q: p[0] < q[0] + q[1] and q[0] < p[0] + p[1]
    places = [primal[0], primal[1], dual, *once]
    assert not any(overlap(p, q) for i, p in enumerate(places) for q in places[:i])
    writes, reads = [], []  # (place, after, before)
    for t in range(4):
        writes += [(primal[t], 2 * t, 2 * t + 1),      # spread warps, in the primal half-step
                   (primal[t], 2 * t, 2 * t + 2),      # a warp's last, between arrival and wait
                   (primal[t], 2 * t + 1, 2 * t + 2),  # whole groups, with the dual sums
                   (dual, 2 * t + 1, 2 * t + 2)]
        reads += [(primal[t], 2 * t + 2, 2 * t + 3), (dual, 2 * t + 2, 2 * t + 3)]  # the totals
    for p, r_after, r_before in reads:
        for q, w_after, w_before in writes:
            if overlap(p, q):
                assert r_before <= w_after or w_before <= r_after, (p, r_after, w_after)

"""The solver's host driver (csrc/pdlp_capi.cu) on a stand-in for the CUDA
runtime, no GPU: what it answers when a call of the runtime fails."""

import os
import shutil
import subprocess

import pytest

from paper_2311_12180_gb300 import pdlp as P

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _build(out, *sources):
    """sources: (file, "cu" or "" to compile as its suffix says), or an object file."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    csrc = os.path.join(ROOT, "paper_2311_12180_gb300", "csrc")
    flags = ["-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-I", csrc, "-I", os.path.join(ROOT, "include")]
    objs = []
    for src, lang in sources:
        if src.endswith(".o"):
            objs.append(src)
            continue
        objs.append(os.path.join(os.path.dirname(out), os.path.basename(src) + ".o"))
        subprocess.run([nvcc, *flags, *(["-x", lang] if lang else []), "-c", src, "-o", objs[-1]], check=True)
    subprocess.run([nvcc, "-cudart", "none", *objs, "-lpthread", "-o", out], check=True)
    return out


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    here, csrc = os.path.join(ROOT, "tests"), os.path.join(ROOT, "paper_2311_12180_gb300", "csrc")
    return _build(str(tmp_path_factory.mktemp("solver") / "solver_host"), (os.path.join(here, "cuda_runtime_host.cpp"), ""),
                  (os.path.join(here, "solver_host.cpp"), "cu"), (os.path.join(csrc, "pdlp_capi.cu"), ""))


def _with_library_object(out, driver, obj):
    from paper_2311_12180_gb300 import _build as B

    B.build()
    here = os.path.join(ROOT, "tests")
    return _build(str(out / "host"), (os.path.join(here, "cuda_runtime_host.cpp"), ""), (os.path.join(here, driver), "cu"),
                  (os.path.join(B.OBJDIR, obj), ""))


@pytest.fixture(scope="module")
def batch_exe(tmp_path_factory):
    return _with_library_object(tmp_path_factory.mktemp("batch"), "batch_host.cpp", "pdlp_batch.cu.o")


@pytest.fixture(scope="module")
def mlp_exe(tmp_path_factory):
    return _with_library_object(tmp_path_factory.mktemp("mlp"), "mlp_host.cpp", "pdlp_mlp.cu.o")


def _run(exe, *args):
    out = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, check=True).stdout.strip().split("\n")
    rows = []
    for line in out:
        w = line.split()
        rows.append((w[0], int(w[1]), {w[i]: int(w[i + 1]) for i in range(2, len(w), 2)}))
    return rows


def test_a_failed_capture_leaves_no_period_to_run(exe):
    quad, begin, run, begin2, run2 = _run(exe, "capture")
    assert quad[1] == P.OK and begin[1] == P.ERR_CUDA
    assert run[1] == P.ERR_INVALID and run[2]["graph"] == 0  # "call pdlp_begin first"
    assert begin2[1] == P.OK and run2[1] == P.OK and run2[2]["graph"] == 2


@pytest.mark.parametrize("scenario", ["refused", "refused later"])
def test_a_period_that_does_not_fit_falls_back_to_the_step_kernels(exe, scenario):
    begin, run, finish, _, ctas = _run(exe, scenario)
    assert begin[1] == P.OK and run[1] == P.OK and finish[1] == P.OK
    assert run[2]["graph"] == 2 and ctas[1] == 0
    assert (begin[2]["check"], begin[2]["period"]) == ((2, 0) if scenario == "refused" else (0, 1))


def test_another_launch_error_is_reported(exe):
    begin, *_, ctas = _run(exe, "broken")
    assert begin[1] == P.ERR_CUDA and ctas[1] == 152


def test_several_solvers_share_the_gpu_as_step_kernels(exe):
    rows = _run(exe, "several")
    assert all(r[1] == P.OK for r in rows)
    got = [(r[0], r[2]["graph"], r[2]["period"]) for r in rows]
    assert got == [("begin_a", 0, 1), ("run_a", 0, 2),                   # a alone
                   ("begin_b", 0, 2), ("run_b", 1, 2), ("run_a", 2, 2),  # both in flight
                   ("finish_a", 2, 2), ("run_b", 2, 3), ("poll_b", 2, 3),  # b alone
                   ("run_a", 2, 4), ("run_b", 3, 4),                     # a alone, then both
                   ("run_b", 3, 5),                                      # a destroyed
                   ("poll_b", 3, 5), ("run_b", 4, 5), ("run_b", 4, 6),   # beside a network, then alone
                   ("begin_c", 4, 7), ("run_c", 4, 8),                   # a cluster beside b
                   ("run_c", 5, 8), ("begin_c", 5, 8), ("run_c", 5, 9)]  # beside a batch, then not


@pytest.mark.parametrize("resident,small,large", [(152, 60, 40), (100, 60, 40), (40, 60, 40), (16, 60, 40), (20, 30, 1),
                                                  (4, 30, 1), (10, 170, 0)])
def test_a_batch_fits_its_grid_to_the_stream(batch_exe, resident, small, large):
    """Launches that the runtime refuses as too large are repeated with fewer
    teams, in create (which times short solves) and in solve; a batch without
    large LPs has no CTAs that must be resident together."""
    create, solve = _run(batch_exe, resident, small, large)
    assert create[1] == P.OK and solve[1] == P.OK
    assert solve[2]["grid"] == create[2]["grid"] > 0
    assert create[2]["in_flight"] == solve[2]["in_flight"] == 1 and create[2]["left"] == solve[2]["left"] == 0
    if large:
        assert resident / 4 < create[2]["grid"] <= resident or create[2]["grid"] == 4 <= resident
    else:
        assert create[2]["grid"] == 152


def test_page_locked_chunks_come_where_a_large_pageable_prediction_pays_for_them(mlp_exe):
    rows = _run(mlp_exe, 0)
    assert all(r[1] == P.OK and r[2]["written"] for r in rows)
    assert [(r[0], r[2]["pinned"], r[2]["streams"]) for r in rows] == [
        ("create", 0, 1), ("small", 0, 1), ("locked", 0, 1), ("written", 0, 1), ("first", 0, 1), ("second", 1, 9),
        ("batches", 1, 9), ("big", 1, 10), ("written", 1, 10), ("once", 2, 18)]
    assert [r[2]["in_flight"] for r in rows] == [0, 1, 1, 1, 1, 1, 1, 0, 1, 1] and rows[-1][2]["left"] == 0


def test_predictions_without_page_locked_memory(mlp_exe):
    rows = _run(mlp_exe, 1)
    assert all(r[1] == P.OK and r[2]["written"] for r in rows)
    assert [r[2]["pinned"] for r in rows] == [0, 0, 0, 0, 0, 1, 1, 1, 1, 2]  # asked for once a network


@pytest.mark.parametrize("scenario", ["captured", "captured graph"])
def test_periods_are_refused_on_a_stream_under_capture(exe, scenario):
    begin, refused, run = _run(exe, scenario)
    assert begin[1] == P.OK and refused[1] == P.ERR_CUDA and run[1] == P.OK
    kind = "period" if scenario == "captured" else "graph"
    assert refused[2][kind] == begin[2][kind] and run[2][kind] == begin[2][kind] + 2

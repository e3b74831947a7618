"""Calls on a stream that the caller captures: check periods are refused on
either path (they would be recorded, not run), and the solver goes on
normally; the allocation-free scaling can be captured and replayed."""

import numpy as np
import pytest

import lpgen
from paper_2311_12180_gb300 import pdlp as P
from test_gpu_scale_long_rows import SHAPES, _matrix, _Scaler

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [2000, 60000, 3000000])  # one cluster, the whole GPU, the step kernels' graph
def test_periods_are_refused_under_capture(size):
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    with P.Solver(lpgen.large_lp(1, m=size // 20, n=size // 10, nnz=size), stream=stream.cuda_stream) as s:
        ok = s.solve(tol=1e-14, max_iter=130)
        s.begin(tol=1e-14, max_iter=130)
        stream.synchronize()
        x = torch.zeros(4, device="cuda")
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
            x += 1
            with pytest.raises(P.PdlpError) as e:
                s.run_periods(1)
        assert e.value.code == P.ERR_CUDA
        graph.replay()
        torch.cuda.synchronize()
        assert x.tolist() == [1.0] * 4  # the caller's capture is whole
        a = s.resume()
    assert np.array_equal(a[0], ok[0]) and np.array_equal(a[1], ok[1]) and a[2:] == ok[2:]


@pytest.mark.parametrize("shape", ["mixed", "adjacent long"])  # a warp a row; lists of long rows
def test_scaling_under_capture(shape):
    torch = pytest.importorskip("torch")
    K = _matrix(*SHAPES[shape])
    plain = _Scaler(K)
    plain(1.0)
    want = plain.results()
    captured = _Scaler(K)
    fresh = [t.clone() for t in captured.d]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured(1.0)
    for _ in range(2):
        for t, f in zip(captured.d, fresh):
            t.copy_(f)
        graph.replay()
        assert all(np.array_equal(a, b) for a, b in zip(captured.results(), want))

"""Predictions whose batches are above 8 MB each: several staged batches in one
call (the pinned chunks and the device buffer used again), a short last batch,
and destinations that are fresh, written before, half written, or page-locked
(the written and the page-locked one are copied to directly)."""

import mmap

import numpy as np
import pytest

from paper_2311_12180_gb300 import pdlp as P
from paper_2311_12180_gb300 import warmstart

pytestmark = pytest.mark.gpu


def test_several_staged_batches_and_a_page_locked_destination():
    torch = pytest.importorskip("torch")
    in_dim, out_dim, batch, count, guard = 5, 60501, 48, 130, 5000
    X = np.random.default_rng(3).standard_normal((count, in_dim)).astype(np.float32)
    with P.Mlp(in_dim, 32, out_dim, max_batch=batch) as net:
        assert 4 * batch * out_dim > 8 << 20
        net.set_params(warmstart.init_params(in_dim, 32, out_dim, 7))
        small = np.concatenate([net.predict(X[i:i + 8]) for i in range(0, count, 8)])  # 1.9 MB each: never staged
        size = guard + count * out_dim + guard
        locked = torch.empty(size, dtype=torch.float32).pin_memory().numpy()
        written = np.full(size, 1.5, dtype=np.float32)
        fresh = [np.frombuffer(mmap.mmap(-1, 4 * size), dtype=np.float32) for _ in range(3)]
        half = np.frombuffer(mmap.mmap(-1, 4 * size), dtype=np.float32)
        half[: size // 2] = 2.0
        for buf in (fresh[0], locked, fresh[1], written, half, fresh[2], fresh[2]):
            buf[:guard] = buf[-guard:] = 1.5
            Y = buf[guard:guard + count * out_dim]
            P._check(P.lib().pdlp_mlp_predict(net.h, count, P._ptr(X), P._ptr(Y)))
            assert np.array_equal(Y.reshape(count, out_dim), small)
            assert np.all(buf[:guard] == 1.5) and np.all(buf[guard + count * out_dim:] == 1.5)

"""Predictions whose batches are above 8 MB each: several staged batches in one
call (the pinned chunks and the device buffer used again), a short last batch,
and a page-locked destination, which is copied to directly."""

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
        plain = np.empty(guard + count * out_dim + guard, dtype=np.float32)
        locked = torch.empty(plain.size, dtype=torch.float32).pin_memory().numpy()
        for buf in (plain, locked, plain):
            buf[:] = 1.5
            Y = buf[guard:guard + count * out_dim]
            P._check(P.lib().pdlp_mlp_predict(net.h, count, P._ptr(X), P._ptr(Y)))
            assert np.array_equal(Y.reshape(count, out_dim), small)
            assert np.all(buf[:guard] == 1.5) and np.all(buf[guard + count * out_dim:] == 1.5)

"""Predictions of more than 8 MB reach pageable memory in chunks, on several
threads; nothing outside the result may change."""

import numpy as np
import pytest

from paper_2311_12180_gb300 import pdlp as P
from paper_2311_12180_gb300 import warmstart

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 3])  # page-aligned or not
@pytest.mark.parametrize("max_batch", [16, 64])  # several chunks of the workspace, one
def test_large_prediction_into_a_fresh_buffer(offset, max_batch):
    in_dim, out_dim, count, guard = 5, 60501, 40, 40000
    net = P.Mlp(in_dim, 32, out_dim, max_batch=max_batch)
    net.set_params(warmstart.init_params(in_dim, 32, out_dim, 7))
    X = np.random.default_rng(3).standard_normal((count, in_dim)).astype(np.float32)
    small = np.concatenate([net.predict(X[i:i + 8]) for i in range(0, count, 8)])  # 1.9 MB each
    buf = np.empty(guard + offset + count * out_dim + guard, dtype=np.float32)
    buf[:guard + offset] = 1.5
    buf[guard + offset + count * out_dim:] = 2.5
    Y = buf[guard + offset:guard + offset + count * out_dim]
    assert Y.nbytes > 8 << 20
    P._check(P.lib().pdlp_mlp_predict(net.h, count, P._ptr(X), P._ptr(Y)))
    assert np.array_equal(Y.reshape(count, out_dim), small)
    assert np.all(buf[:guard + offset] == 1.5) and np.all(buf[guard + offset + count * out_dim:] == 2.5)
    net.close()

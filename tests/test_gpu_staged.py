"""Searches whose rows are gathered through shared memory: every width that has the staged kernel, narrow and wide graph
rows, and the batch sizes around which the launch changes between it and the plain kernel. All equal the oracle's."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, dev_index, run

pytestmark = pytest.mark.gpu


# 16 one-warp teams per SM with plain gathers, 20 with staged ones
@pytest.mark.parametrize("d", [36, 128, 132, 256, 260, 320, 324, 384, 388])
@pytest.mark.parametrize("r", [20, 90])
def test_widths_and_batch_sizes(d, r):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(d + r)
    n, nq = 4000, 20 * sms + 1
    X = rng.standard_normal((n, d)).astype(np.float32)
    X /= np.linalg.norm(X, axis=1, keepdims=True)
    Q = rng.standard_normal((nq, d)).astype(np.float32)
    adj = rng.integers(0, n, (n, r)).astype(np.uint32)
    adj[:, r // 2] = adj[:, 0]
    idx = dev_index(X, adj, 0)
    for L in (100, 300):
        ref = oracle.beam_search(X, adj, 0, Q[:60], 10, L, max_visits=16384)
        for m in (16 * sms, 16 * sms + 1, 17 * sms + 1, 20 * sms, 20 * sms + 1):
            got = run(idx, Q[:m], 10, L)
            assert_same([g[:60] for g in got], ref, f"L {L}, {m} queries")
        for table in (-1, 10):                  # the bitmap alone; a table of ids
            idx.set_tuning(L, 1, table)
            assert_same(run(idx, Q[:60], 10, L), ref, f"L {L}, table {table}")
        idx.set_tuning(L, 1, 0)
        assert_same(run(idx, Q[:60], 10, L), ref, f"L {L}, one warp")
        idx.close()
        idx = dev_index(X, adj, 0)
    idx.close()

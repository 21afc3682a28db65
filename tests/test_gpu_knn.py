"""Edges of the tensor-core kNN: tile, block and K-step remainders, X ranges merged
from several CTA pairs, ties, and orders of X that fill the candidate buffers."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _knn(T, X, kk):
    import torch

    import paper_2408_08933_gb300 as pkg

    ids, dist = pkg.knn(torch.from_numpy(T).to("cuda:0"), torch.from_numpy(X).to("cuda:0"), kk)
    torch.cuda.synchronize()
    return ids.cpu().numpy().view(np.uint32), dist.cpu().numpy()


@pytest.mark.parametrize("nt,n,d,kk", [
    (1, 1, 8, 1), (2, 128, 16, 128), (127, 129, 24, 100), (128, 255, 40, 64), (129, 256, 56, 50), (255, 257, 64, 10),
    (256, 1023, 72, 100), (257, 1025, 200, 100), (511, 4097, 248, 100), (513, 5000, 320, 100), (40, 30_011, 512, 100),
    (1, 40_000, 32, 100)])
def test_knn_tile_edges(nt, n, d, kk):
    rng = np.random.default_rng(nt * 7 + n)
    X = rng.standard_normal((n, d)).astype(np.float32)
    T = rng.standard_normal((nt, d)).astype(np.float32)
    ids, dist = _knn(T, X, kk)
    s64 = T.astype(np.float64) @ X.astype(np.float64).T
    # BF16 rounding moves a score by at most 2^-8 |t||x| (both operands rounded), so a row whose score is above the
    # 129th best by twice that is surely among the 128 candidates
    slack = 2.0 ** -7 * np.linalg.norm(T, axis=1) * np.linalg.norm(X, axis=1).max()
    order = np.argsort(-s64, axis=1, kind="stable")
    for r in range(0, nt, max(1, nt // 50)):
        assert len(set(ids[r].tolist())) == kk and ids[r].max() < n
        assert np.all(np.diff(dist[r]) >= 0)
        assert dist[r, 0] == -oracle.dot_fixed(T[r], X[ids[r, 0]])
        edge = s64[r, order[r, 128]] + slack[r] if n > 128 else -np.inf
        sure = [c for c in order[r, :kk] if s64[r, c] > edge]
        # ... and comes back in place, up to exchanges within FP32 rounding
        assert set(sure) <= set(ids[r].tolist())
        got = s64[r, ids[r, :len(sure)]]
        assert np.all(np.abs(got - s64[r, order[r, :len(sure)]]) <= 1e-5 * np.linalg.norm(T[r]) * d ** 0.5)


@pytest.mark.parametrize("n_distinct,copies,nt", [(1, 5000, 3), (40, 500, 300), (3, 20_000, 5)])
def test_knn_mass_ties_keep_the_lowest_ids(n_distinct, copies, nt):
    rng = np.random.default_rng(copies)
    base = rng.standard_normal((n_distinct, 64)).astype(np.float32)
    T = rng.standard_normal((nt, 64)).astype(np.float32)
    which = rng.permutation(np.repeat(np.arange(n_distinct), copies))
    ids, _ = _knn(T, base[which], 100)
    best = np.argmax(T.astype(np.float64) @ base.astype(np.float64).T, axis=1)
    for r in range(nt):
        assert ids[r].tolist() == np.flatnonzero(which == best[r])[:100].tolist()


@pytest.mark.parametrize("reverse", [False, True])
def test_knn_sorted_rows(reverse):
    # every row of X beats (or none beats) all before it: buffers fill at once, or never again
    rng = np.random.default_rng(5)
    t = rng.standard_normal(64)
    t /= np.linalg.norm(t)
    n = 12_000
    X = (np.linspace(0.1, 4.0, n)[:, None] * t[None, :]).astype(np.float32)
    T = (t[None, :] * np.linspace(0.5, 2.0, 200)[:, None]).astype(np.float32)
    if reverse:
        X = np.ascontiguousarray(X[::-1])
    ids, _ = _knn(T, X, 10)
    # BF16 merges about 4.0 * 2^-9 of the scale per step, 24 rows: the best 10 lie well inside the best 128
    want = np.arange(10) if reverse else n - 1 - np.arange(10)
    for r in range(0, 200, 9):
        assert set(ids[r].tolist()) == set(want.tolist())


def test_a_destroyed_index_gives_the_pool_back():
    import torch
    from gpu_util import dev_index

    rng = np.random.default_rng(6)
    X = rng.standard_normal((10_000, 64)).astype(np.float32)
    T = rng.standard_normal((1000, 64)).astype(np.float32)
    first = _knn(T, X, 50)
    held = torch.cuda.mem_get_info()[0]
    dev_index(X[:100], np.full((100, 8), 0xFFFFFFFF, np.uint32), 0).close()
    # the least a call holds: candidate buffers of 3 MB per pair, at least one pair per 256 T rows
    assert torch.cuda.mem_get_info()[0] - held >= 4 * 3 << 20
    again = _knn(T, X, 50)
    assert np.array_equal(first[0], again[0]) and np.array_equal(first[1], again[1])


def test_the_library_s_own_handles_leave_the_pool():
    import torch
    from gpu_util import dev_index
    from test_gpu_insert import CASES, _case

    import paper_2408_08933_gb300 as pkg

    rng = np.random.default_rng(7)
    X = rng.standard_normal((10_000, 64)).astype(np.float32)
    _knn(rng.standard_normal((1000, 64)).astype(np.float32), X, 50)
    B, T, knn, entry, adj, nout, cnt, _ = _case(*CASES[1])
    Bd, Ad = torch.from_numpy(B).to("cuda:0"), torch.from_numpy(adj.view(np.int32)).to("cuda:0")
    pkg.insert(Bd, Ad, entry, CASES[1][1], T, knn[:, 0], nout.copy(), cnt.copy(), *CASES[1][2:])   # searches by a handle of its own
    idx = dev_index(X[:100], np.full((100, 8), 0xFFFFFFFF, np.uint32), 0)
    held = torch.cuda.mem_get_info()[0]
    idx.close()
    assert torch.cuda.mem_get_info()[0] - held >= 4 * 3 << 20     # it was there until the program's handle went


def test_the_pool_is_given_back_on_request():
    import torch

    import paper_2408_08933_gb300 as pkg

    rng = np.random.default_rng(8)
    X = rng.standard_normal((10_000, 64)).astype(np.float32)
    T = rng.standard_normal((1000, 64)).astype(np.float32)
    first = _knn(T, X, 50)
    held = torch.cuda.mem_get_info()[0]
    pkg.roar_knn_release()
    assert torch.cuda.mem_get_info()[0] - held >= 4 * 3 << 20
    again = _knn(T, X, 50)
    assert np.array_equal(first[0], again[0]) and np.array_equal(first[1], again[1])
    pkg.roar_knn_release()
    pkg.roar_knn_release()      # nothing left to give

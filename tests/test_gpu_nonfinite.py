"""Sums that are NaN order as +inf: queries and rows that are not finite walk a defined path, and ids stay in range."""
import numpy as np
import pytest

import oracle
from gpu_util import dev_index, run

pytestmark = pytest.mark.gpu


def _data(n, d, r, nq):
    rng = np.random.default_rng(n + d)
    X = rng.standard_normal((n, d)).astype(np.float32)
    X /= np.linalg.norm(X, axis=1, keepdims=True)
    Q = rng.standard_normal((nq, d)).astype(np.float32)
    Q[:, 0] = np.abs(Q[:, 0]) + 0.5
    return X, Q, rng.integers(0, n, (n, r)).astype(np.uint32)


def _index(X, adj, dtype):
    if dtype == "f32":
        return dev_index(X, adj, 0)
    if dtype == "bf16":
        return dev_index(X, adj, 0, dtype="bf16", trav=oracle.quant_bf16(X).view(np.int16))
    codes, scales = oracle.quant_e4m3(X)
    return dev_index(X, adj, 0, dtype="fp8", trav=codes, scales=scales)


def _same(got, ref):
    for g, w, what in zip(got, ref, ("ids", "dist", "visits", "hops", "status")):
        assert np.array_equal(g, w), what


# the bitmap alone at 200 columns is the staged gather; a team of 0 is the untuned choice
@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("tw,table", [(0, 0), (1, 0), (1, -1), (4, 10)])
@pytest.mark.parametrize("d,L", [(32, 60), (200, 300)])
def test_nan_queries(dtype, tw, table, d, L):
    X, Q, adj = _data(3000, d, 64, 20)
    Q[::2, d // 2] = np.nan
    # all distances equal: the walk of a zero query, whose ties are broken by id
    Z = np.where(np.isnan(Q).any(1, keepdims=True), np.float32(0), Q)
    kw = {}
    if dtype == "bf16":
        kw = {"dtype": dtype, "Xt": oracle.quant_bf16(X)}
    elif dtype == "fp8":
        kw = dict(zip(("Xt", "scales"), oracle.quant_e4m3(X)), dtype=dtype)
    ref = list(oracle.beam_search(X, adj, 0, Z, 10, L, max_visits=16384, **kw))
    ref[1] = np.where(np.isnan(Q).any(1, keepdims=True), np.float32(np.inf), ref[1])
    idx = _index(X, adj, dtype)
    if tw:
        idx.set_tuning(L, tw, table)
    _same(run(idx, Q, 10, L), ref)
    idx.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("tw", [0, 1])
def test_nan_rows(dtype, tw):
    X, Q, adj = _data(3000, 32, 64, 20)
    bad = np.random.default_rng(1).random(3000) < 0.3
    bad[0] = False
    Y, Z = X.copy(), X.copy()
    Y[bad, 3] = np.nan
    Z[bad] = 0.0
    Z[bad, 0] = -np.inf        # the same distance, +inf, without a NaN: every query's first element is positive
    ref = oracle.beam_search(Z, adj, 0, Q, 10, 200, max_visits=16384,
                             **({} if dtype == "f32" else {"dtype": dtype, "Xt": oracle.quant_bf16(Z)}))
    idx = _index(Y, adj, dtype)
    if tw:
        idx.set_tuning(200, tw)
    _same(run(idx, Q, 10, 200), ref)
    idx.close()

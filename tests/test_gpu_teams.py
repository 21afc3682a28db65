"""Hand-off between the warps of a team: searches whose hops mostly bring no new row, and batches in which bad (k, L) are
skipped between good queries. Every query equals the oracle's, in every one of several launches."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, dev_index, run

pytestmark = pytest.mark.gpu


def _case(seed, n=400, d=32, r=32):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, d)).astype(np.float32)
    X /= np.linalg.norm(X, axis=1, keepdims=True)
    Q = rng.standard_normal((64, d)).astype(np.float32)
    adj = np.tile(np.arange(1, r + 1, dtype=np.uint32), (n, 1))   # every hop after the first brings nothing ...
    adj[5, :6] = np.arange(100, 106)                              # ... but for a few rows
    adj[9, :3] = np.arange(200, 203)
    return X, Q, adj


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("tw", [0, 1, 2, 4, 8])
def test_hops_without_new_rows(dtype, tw):
    X, Q, adj = _case(1)
    codes = scales = None
    if dtype == "bf16":
        codes = oracle.quant_bf16(X)
    elif dtype == "fp8":
        codes, scales = oracle.quant_e4m3(X)
    kw = {} if dtype == "f32" else {"dtype": dtype, "Xt": codes, "scales": scales}
    idx = dev_index(X, adj, 0, dtype=dtype, trav=codes.view(np.int16) if dtype == "bf16" else codes, scales=scales)
    for L in (7, 40, 200):          # a full pool, and pools whose last hops bring nothing
        if tw:
            idx.set_tuning(L, tw)
        ref = oracle.beam_search(X, adj, 0, Q, 5, L, max_visits=16384, **kw)
        for again in range(5):
            assert_same(run(idx, Q, 5, L), ref, f"L {L} launch {again}")
    idx.close()


@pytest.mark.parametrize("tw", [0, 1, 2, 4, 8])
def test_bad_parameters_between_good_queries(tw):
    import torch

    X, Q, adj = _case(2)
    nq = len(Q)
    ks, Ls = np.full(nq, 5, np.int32), np.full(nq, 40, np.int32)
    ks[1::4], Ls[2::4], ks[6::8] = 0, 300, 41      # k = 0; L past L_max; k past L; some in a row
    ok = (ks >= 1) & (Ls <= 64) & (ks <= Ls)
    ref = oracle.beam_search(X, adj, 0, Q, 5, 40, max_visits=16384)
    idx = dev_index(X, adj, 0)
    if tw:
        idx.set_tuning(64, tw)
    out = idx.uneven_outputs(np.maximum(ks, 1))
    off = out[0].cpu().numpy()
    for again in range(5):
        for t in out[1:]:
            t.fill_(-7)
        idx.search_uneven(*(torch.from_numpy(a).to("cuda:0") for a in (Q, ks, Ls)), 64, out)
        torch.cuda.synchronize()
        ids, st, vis = out[1].cpu().numpy().view(np.uint32), out[5].cpu().numpy(), out[3].cpu().numpy()
        assert st.tolist() == [0 if o else 1 for o in ok], again
        for i in range(nq):
            if ok[i]:
                assert np.array_equal(ids[off[i]:off[i] + 5], ref[0][i]) and vis[i] == ref[2][i], (again, i)
            else:
                assert vis[i] == 0, (again, i)
    idx.close()

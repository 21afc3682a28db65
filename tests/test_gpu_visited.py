"""The compact visited table and the pool merge of the search kernels, where they can go wrong: rows that repeat an id,
ids whose slot value is the free mark, tables that overflow into the bitmap, tiny sets, wide graph rows, and every team
size and batch size the launch rules tell apart. Everything equals the oracle's search."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, dev_index, run

pytestmark = pytest.mark.gpu


def _graph(rng, n, r, special=None):
    adj = rng.integers(0, n, (n, r)).astype(np.uint32)
    adj[:, 1::5] = adj[:, 0::5][:, :adj[:, 1::5].shape[1]]           # the same id twice in a row
    if special is not None:
        adj[rng.random((n, r)) < 0.05] = rng.choice(special)
    pad = rng.integers(r // 2, r + 1, n)
    adj[np.arange(r)[None, :] >= pad[:, None]] = 0xFFFFFFFF
    return adj


def _unit(rng, n, d):
    x = rng.standard_normal((n, d)).astype(np.float32)
    return x / np.linalg.norm(x, axis=1, keepdims=True)


@pytest.mark.parametrize("n,d,r,L,k,nq", [
    (33, 8, 8, 10, 5, 3), (100, 16, 64, 100, 10, 40), (5000, 64, 64, 3, 1, 200), (5000, 64, 96, 33, 10, 50),
    (5000, 132, 128, 128, 100, 20), (20_000, 200, 33, 31, 10, 700), (20_000, 40, 70, 500, 10, 30),
    (3000, 300, 48, 1024, 100, 8)])
def test_sizes_teams_and_repeated_ids(n, d, r, L, k, nq):
    rng = np.random.default_rng(n + L)
    X, Q, adj = _unit(rng, n, d), _unit(rng, nq, d), _graph(rng, n, r)
    ref = oracle.beam_search(X, adj, 0, Q, k, L, max_visits=16384)
    idx = dev_index(X, adj, 0)
    assert_same(run(idx, Q, k, L), ref, "automatic")
    for tw, hash_log2 in ((1, 0), (2, 0), (4, -1), (8, 0), (1, 10)):
        idx.set_tuning(L, tw, hash_log2)
        assert_same(run(idx, Q, k, L), ref, f"team {tw} table {hash_log2}")
    idx.close()


def test_values_that_equal_the_free_mark():
    # 23-bit ids over 2^7 buckets: 16 bits in a slot, so 0xFFFF is a possible value; the entry and many neighbours have it
    n, L = 5_000_000, 10
    u = np.arange(n, dtype=np.uint64)
    h = (u * 2654435769) & ((1 << 23) - 1)
    special = u[(h & 0xFFFF) == 0xFFFF].astype(np.uint32)
    assert len(special) > 20
    rng = np.random.default_rng(1)
    X, Q = _unit(rng, n, 4), _unit(rng, 300, 4)
    adj = _graph(rng, n, 8, special)
    ref = oracle.beam_search(X, adj, int(special[0]), Q, 5, L, max_visits=16384)
    idx = dev_index(X, adj, int(special[0]))
    assert_same(run(idx, Q, 5, L), ref)
    assert_same(run(idx, Q, 5, L), ref, "bitmap clean after the first batch")
    idx.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("cap", [16384, 900])
def test_full_buckets_go_to_the_bitmap(dtype, cap):
    # a full grid of wide searches: few slots per query for many visits (and a visit cap that ends them in the middle)
    n, d, L, nq = 300_000, 16, 400, 5000
    rng = np.random.default_rng(2)
    X, Q, adj = _unit(rng, n, d), _unit(rng, nq, d), _graph(rng, n, 64)
    codes = scales = None
    if dtype == "bf16":
        codes = oracle.quant_bf16(X)
    elif dtype == "fp8":
        codes, scales = oracle.quant_e4m3(X)
    kw = {} if dtype == "f32" else {"dtype": dtype, "Xt": codes, "scales": scales}
    ref = oracle.beam_search(X, adj, 7, Q[:48], 10, L, max_visits=cap, **kw)
    idx = dev_index(X, adj, 7, dtype=dtype, trav=codes.view(np.int16) if dtype == "bf16" else codes, scales=scales,
                    max_visits=cap)
    for again in range(2):
        got = run(idx, Q, 10, L)
        assert_same([g[:48] for g in got], ref, f"pass {again}")
    idx.close()


def test_a_plan_outlives_the_scratch_it_was_captured_with():
    # a small captured batch (wide teams, few scratch slots), then a batch that needs more scratch, then the plan again
    import torch

    n, d, r = 20_000, 32, 32
    rng = np.random.default_rng(6)
    X, Q, adj = _unit(rng, n, d), _unit(rng, 4000, d), _graph(rng, n, r)
    k = np.full(20, 10, np.int32)
    L = np.arange(60, 80).astype(np.int32)
    idx = dev_index(X, adj, 3)
    out = idx.uneven_outputs(k)
    plan = idx.plan_uneven(torch.from_numpy(Q[:20]).to("cuda:0"), torch.from_numpy(k).to("cuda:0"),
                           torch.from_numpy(L).to("cuda:0"), 80, out)
    assert_same(run(idx, Q, 5, 10), oracle.beam_search(X, adj, 3, Q, 5, 10, max_visits=16384), "large batch")
    for _ in range(2):
        plan.launch()
        torch.cuda.synchronize()
        ids = out[1].cpu().numpy().view(np.uint32).reshape(20, 10)
        for i in range(20):
            ref = oracle.beam_search(X, adj, 3, Q[i:i + 1], 10, int(L[i]), max_visits=16384)
            assert np.array_equal(ids[i], ref[0][0]), i
    plan.close()
    idx.close()


def test_a_small_warm_up_is_enough_before_a_capture():
    import torch

    n, d, r, nq = 20_000, 32, 32, 3000
    rng = np.random.default_rng(8)
    X, Q, adj = _unit(rng, n, d), _unit(rng, nq, d), _graph(rng, n, r)
    idx = dev_index(X, adj, 3)
    q = torch.from_numpy(Q).to("cuda:0")
    out = (torch.empty((nq, 10), dtype=torch.int32, device="cuda:0"), torch.empty((nq, 10), device="cuda:0"),
           *(torch.empty(nq, dtype=torch.int32, device="cuda:0") for _ in range(3)))
    idx.search(q[:1], 10, 40)                 # one query: a wide team
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        idx.search(q, 10, 40, out=out)
    g.replay()
    torch.cuda.synchronize()
    got = [o.cpu().numpy() for o in out]
    got = (got[0].view(np.uint32), got[1], got[2].view(np.uint32), got[3].view(np.uint32), got[4])
    assert_same(got, oracle.beam_search(X, adj, 3, Q, 10, 40, max_visits=16384))
    idx.close()


def test_a_small_warm_up_is_enough_for_the_staged_gather():
    # the bitmap alone at 129 to 256 columns: the large launch stages its gathers, with more CTAs per SM
    import torch

    n, d, r, nq = 20_000, 200, 32, 4000
    rng = np.random.default_rng(9)
    X, Q, adj = _unit(rng, n, d), _unit(rng, nq, d), _graph(rng, n, r)
    idx = dev_index(X, adj, 3)
    idx.set_hash_log2(-1)
    q = torch.from_numpy(Q).to("cuda:0")
    out = (torch.empty((nq, 10), dtype=torch.int32, device="cuda:0"), torch.empty((nq, 10), device="cuda:0"),
           *(torch.empty(nq, dtype=torch.int32, device="cuda:0") for _ in range(3)))
    idx.search(q[:1], 10, 40)                 # one query: a wide team
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        idx.search(q, 10, 40, out=out)
    g.replay()
    torch.cuda.synchronize()
    got = [o.cpu().numpy() for o in out]
    got = (got[0].view(np.uint32), got[1], got[2].view(np.uint32), got[3].view(np.uint32), got[4])
    assert_same(got, oracle.beam_search(X, adj, 3, Q, 10, 40, max_visits=16384))
    idx.close()


@pytest.mark.parametrize("nq", [1, 3000])
def test_a_table_too_large_for_one_warp_teams_is_refused_for_any_batch(nq):
    import torch

    rng = np.random.default_rng(10)
    X, Q, adj = _unit(rng, 1000, 32), _unit(rng, nq, 32), _graph(rng, 1000, 32)
    idx = dev_index(X, adj, 3)
    idx.set_hash_log2(15)                     # 4 teams x 128 KB
    with pytest.raises(Exception, match="shared memory"):
        idx.search(torch.from_numpy(Q).to("cuda:0"), 10, 40)
    idx.close()


def test_tuned_wide_teams_allocate_scratch_for_themselves_only():
    import torch

    n, L = 1_000_000, 40
    rng = np.random.default_rng(11)
    X, Q, adj = _unit(rng, n, 8), _unit(rng, 50, 8), _graph(rng, n, 8)
    idx = dev_index(X, adj, 0)
    idx.set_tuning(L, 8)
    q = torch.from_numpy(Q).to("cuda:0")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    idx.search(q, 10, L)
    torch.cuda.synchronize()
    # 32 warps per SM at most, hence 4 teams; a bitmap and a visit log each (allocations come in 2 MB pages, and
    # torch takes up to 20 MB for the outputs)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    slots = 4 * sms * (n // 8 + 4 * (16384 + 128))
    assert free - torch.cuda.mem_get_info()[0] <= slots + (64 << 20)
    idx.close()


def test_a_captured_search_keeps_its_scratch():
    # a capture at L = 500, then a search at L = 100 whose launches keep more CTAs resident and replace the scratch
    import torch

    n, d, r, nq = 20_000, 200, 32, 3000
    rng = np.random.default_rng(12)
    X, Q, adj = _unit(rng, n, d), _unit(rng, nq, d), _graph(rng, n, r)
    idx = dev_index(X, adj, 3)
    q = torch.from_numpy(Q).to("cuda:0")

    def outputs():
        return (torch.empty((nq, 10), dtype=torch.int32, device="cuda:0"), torch.empty((nq, 10), device="cuda:0"),
                *(torch.empty(nq, dtype=torch.int32, device="cuda:0") for _ in range(3)))

    out, other = outputs(), outputs()
    idx.search(q, 10, 500, out=out)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        idx.search(q, 10, 500, out=out)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    idx.search(q, 10, 100, out=other)
    torch.cuda.synchronize()
    # the larger scratch came on top of the graph's: one bitmap and visit log at least for each query of the batch
    assert free - torch.cuda.mem_get_info()[0] >= nq * (n // 8 + 4 * 16384)
    for _ in range(2):
        for o in out:
            o.zero_()
        g.replay()
        torch.cuda.synchronize()
        got = [o.cpu().numpy()[:300] for o in out]
        got = (got[0].view(np.uint32), got[1], got[2].view(np.uint32), got[3].view(np.uint32), got[4])
        assert_same(got, oracle.beam_search(X, adj, 3, Q[:300], 10, 500, max_visits=16384))
    idx.close()


@pytest.mark.parametrize("table,cap", [(0, 1), (-1, 2), (13, 0)])
def test_tuned_caps_and_tables_bound_the_scratch(table, cap):
    import torch

    n, L = 1_000_000, 40
    rng = np.random.default_rng(13)
    X, Q, adj = _unit(rng, n, 8), _unit(rng, 50, 8), _graph(rng, n, 8)
    idx = dev_index(X, adj, 0)
    idx.set_tuning(L, 1, table, cap)
    q = torch.from_numpy(Q).to("cuda:0")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    idx.search(q, 10, L)
    torch.cuda.synchronize()
    # CTAs of 4 teams: as many per SM as the cap says, or as four tables of 32 KB leave in 228 KB: one
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    slots = 4 * max(cap, 1) * sms * (n // 8 + 4 * (16384 + 128))
    assert free - torch.cuda.mem_get_info()[0] <= slots + (64 << 20)
    idx.close()


def test_a_small_warm_up_is_enough_with_a_table_of_ids():
    # 8,192 slots: one CTA of four one-warp teams per SM, but three CTAs of two two-warp teams
    import torch

    n, d, r, nq = 20_000, 32, 32, 700
    rng = np.random.default_rng(14)
    X, Q, adj = _unit(rng, n, d), _unit(rng, nq, d), _graph(rng, n, r)
    idx = dev_index(X, adj, 3)
    idx.set_hash_log2(13)
    q = torch.from_numpy(Q).to("cuda:0")
    out = (torch.empty((nq, 10), dtype=torch.int32, device="cuda:0"), torch.empty((nq, 10), device="cuda:0"),
           *(torch.empty(nq, dtype=torch.int32, device="cuda:0") for _ in range(3)))
    idx.search(q[:1], 10, 40)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        idx.search(q, 10, 40, out=out)
    g.replay()
    torch.cuda.synchronize()
    got = [o.cpu().numpy() for o in out]
    got = (got[0].view(np.uint32), got[1], got[2].view(np.uint32), got[3].view(np.uint32), got[4])
    assert_same(got, oracle.beam_search(X, adj, 3, Q, 10, 40, max_visits=16384))
    idx.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
def test_short_searches_of_sets_past_eight_million_rows(dtype):
    # 24-bit ids need 2^8 buckets for 16 bits in a slot, more than the visits of these searches ask for
    n = (1 << 23) + 1000
    rng = np.random.default_rng(15)
    X = rng.standard_normal((n, 4), dtype=np.float32)
    Q = rng.standard_normal((3000, 4), dtype=np.float32)
    adj = rng.integers(0, n, (n, 8), dtype=np.uint32)
    adj[:, 7] = adj[:, 0]
    u = np.arange(n, dtype=np.uint32)
    special = u[((u * np.uint32(2654435769)) & 0xFFFF) == 0xFFFF]       # the free mark as slot value
    adj[::3, 5] = rng.choice(special, len(adj[::3]))
    codes = scales = None
    if dtype == "bf16":
        codes = (X.view(np.uint32) >> 16).astype(np.uint16)              # any codes will do
    elif dtype == "fp8":
        codes, scales = rng.integers(0, 127, (n, 4), dtype=np.uint8), np.full(n, 0.5, np.float32)
    kw = {} if dtype == "f32" else {"dtype": dtype, "Xt": codes, "scales": scales}
    idx = dev_index(X, adj, n - 1, dtype=dtype, trav=codes.view(np.int16) if dtype == "bf16" else codes, scales=scales)
    for L in (10, 22):
        ref = oracle.beam_search(X, adj, n - 1, Q, 5, L, max_visits=16384, **kw)
        for m in (3000, 100):
            assert_same(run(idx, Q[:m], 5, L), [r[:m] for r in ref], f"L {L}, {m} queries")
    idx.close()

// Beam-search dispatch: kernel choice, shared-memory sizing, occupancy and launch.
// The kernels themselves are in roar_search_kernel.cuh (one translation unit
// per traversal type).
#include <algorithm>
#include <cmath>

#include "roar_internal.cuh"

namespace roar {

namespace {

int nch_for(int d) { return search_nch(d); }

int threads_for(int tw) { return 32 * (tw > kWarpsPerBlock ? tw : kWarpsPerBlock); }

}  // namespace

int teams_per_block(int tw) { return threads_for(tw) / (32 * tw); }

static const void *search_kernel(const SearchArgs &a, int tw) {
    const int nch = nch_for(a.d), rpl = a.rmax <= 64 ? 2 : 4;
    if (a.bi_off) return (a.dtype == 0 && tw == 1) ? kernel_table_bi(nch, rpl) : nullptr;
    const bool staged = a.staged != 0;
    switch (a.dtype) {
        case 0: return kernel_table<0>(nch, rpl, tw, staged);
        case 1: return kernel_table<1>(nch, rpl, tw, staged);
        case 2: return kernel_table<2>(nch, rpl, tw, staged);
        default: return nullptr;
    }
}

static size_t stage_of(const SearchArgs &a) {
    return a.staged ? stage_bytes(stage_rows(search_nch(a.d)), a.d >> 2) : 0;
}

// Shared memory a CTA can have. A kernel is allowed all of it, never the size
// of one launch: launches of other sizes by other threads share the kernel.
constexpr size_t kMaxSmem = 227 * 1024;
static cudaError_t allow_smem(const void *fn) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
}

int search_blocks_per_sm(const SearchArgs &a, int tw) {
    const void *fn = search_kernel(a, tw);
    if (!fn) return 0;
    const size_t smem = search_smem_per_team(a, stage_of(a)) * teams_per_block(tw);
    if (smem > kMaxSmem || allow_smem(fn) != cudaSuccess) return 0;
    int blocks = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fn, threads_for(tw), smem) != cudaSuccess)
        return 0;
    const int cap = kMaxWarpsPerSm * 32 / threads_for(tw);
    return blocks < cap ? blocks : cap;
}

// Visited rows of one query of beam width L, about (measured on 1M rows of
// d = 200 and 512: 592 / 2,899 / 4,343 / 7,430 / 11,498 at L = 10 / 100 / 200 /
// 500 / 1000; fewer on smaller sets).
static double visits_for(int L) { return 128.0 * std::pow((double)L, 2.0 / 3.0); }

// Whether a launch does better with staged gathers and the bitmap alone than with
// the compact table (`table`: there is room for one) or with plain gathers. On
// GB300 one-warp FP32 searches, start with the plain side; us:
// - queries that fill a fifth CTA per SM but no more, where four leave a second
//   round: 300,000 x 160, 3,000 queries, L = 100 1,724 / 1,485, L = 320 3,838 / 2,690.
//   Short searches of narrow rows gain nothing (300,000 x 100, L = 60 equal), nor
//   does a second round of a few queries unless the searches are long (300,000 x
//   128, 2,440 queries: L = 100 1,117 / 1,276, L = 320 2,730 / 2,292);
// - 257 to 384 columns, whose plain batches leave lanes idle: all of one round
//   (300,000 x 320, L = 100: 1,220 queries 1,679 / 1,588, 3,000 2,571 / 2,029), and
//   larger launches up to 320 columns while the bitmaps stay in L2 (30,000 x 320,
//   10,000 queries, L = 200 5,241 / 4,381; 1M x 320 the other way round).
// Without a table staged gathers pay from 129 columns on, as said at search_staged
// (d = 100 2.39 / 2.35 ms).
static bool staged_pays(const SearchArgs &a, int L, int64_t nq, int sms, bool table) {
    if (a.bi_off || !search_staged(a.dtype, a.d, 1, a.lcap)) return false;
    SearchArgs plain = a, stg = a;
    plain.staged = plain.ct_log2 = plain.hash_log2 = 0;
    stg = plain;
    stg.staged = 1;
    const int64_t teams = (int64_t)teams_per_block(1) * sms, four = search_blocks_per_sm(plain, 1) * teams,
                  five = search_blocks_per_sm(stg, 1) * teams;
    const int nch = search_nch(a.d);
    if (!table && nch >= 2) return true;
    if (nch == 4)
        return nq <= five || (a.d <= 320 && (double)five * (double)a.n / 8.0 <= 128.0 * (1 << 20));
    const bool few_more = nq <= four + four / 16 && L <= (nch == 2 ? 128 : 256);
    return nq > four && nq <= five && !few_more && (nch == 2 || L > 96);
}

void choose_visited(SearchArgs &a, int hash, int tw, int L, int64_t nq, int sms) {
    a.hash_log2 = hash > 0 ? hash : 0;
    a.ct_log2 = 0;
    a.staged = 0;
    if (hash == 0 && tw == 1 && staged_pays(a, L, nq, sms, true)) {
        a.staged = 1;
        return;
    }
    if (hash == 0) {
        // The compact table: twice the visits expected, or less, as long as the
        // CTAs this launch can use stay resident. Measured on GB300, 1M rows,
        // 10,000 queries, against the bitmap alone: FP32 d = 200 L = 100 4.99 ms
        // (bitmap 6.01, a larger table with fewer CTAs 5.61), L = 500 17.0
        // (18.6); BF16 d = 200 L = 100 4.64 (5.21); FP8 4.78 (4.99). It has to
        // hold a quarter of the visits to help (FP8 L = 350 with 1,024 slots
        // 12.23, bitmap 12.13), and two thirds while the bitmaps of all warps fit
        // half of L2 (100k rows, FP32 L = 200 3.81 / 3.92, L = 500 8.94 / 8.68).
        const int bps = search_blocks_per_sm(a, tw), tpb = teams_per_block(tw);
        const int64_t need = (nq + (int64_t)tpb * sms - 1) / ((int64_t)tpb * sms);
        const int64_t want = std::min<int64_t>(std::max<int64_t>(need, 1), bps);
        const double est = std::min(visits_for(L), (double)a.n);
        // A slot keeps 16 of an id's bits and the bucket stands for the rest, so
        // sets past 2^21 rows need a table of some size however few the visits
        // (10M x 64, 10,000 queries, FP32 L = 10 909 us with the bitmap alone, 627
        // with 4,096 slots; L = 15 1,276 and 860). A full grid of one-warp BF16 / FP8
        // teams has room for 2,048 slots, hence 8.4M rows; past that the bitmap is
        // as good as a table of ids for short searches too (FP8 L = 15 1,395 us, a
        // table of 1,024 ids 1,488).
        int bits = 1;   // of the ids
        while (bits < 31 && ((int64_t)1 << bits) < a.n) ++bits;
        const int least = std::max(9, bits - 16 + kCtBucketLog2);
        int lg = least;
        while (lg < 15 && (double)(1 << lg) < 2.0 * est) ++lg;
        auto resident = [&](int x) {
            a.ct_log2 = x;
            const size_t smem = search_smem_per_team(a, 0) * tpb;
            return smem > kMaxSmem ? 0 : (int64_t)(228 * 1024 / (smem + 1024));
        };
        while (lg >= least && resident(lg) < want) --lg;
        a.ct_log2 = 0;
        const double bitmaps = (double)std::min<int64_t>(nq, want * tpb * sms) * (double)a.n / 8.0;
        const double share = bitmaps <= 64.0 * (1 << 20) ? 1.5 : 4.0;
        if (lg >= least && lg <= 15 && (double)(1 << lg) * share >= est) {
            bits = std::max(bits, lg - kCtBucketLog2);
            a.ct_log2 = lg;
            a.ct_rem = bits - (lg - kCtBucketLog2);
            a.ct_mask = (uint32_t)(((uint64_t)1 << bits) - 1);
        }
    }
    // (With the table the staged gather would need its bytes: 5.1-5.4 ms at 1M x 200,
    // 10,000 queries, L = 100, 4.99 without it.)
    if (!a.ct_log2 && tw == 1 && staged_pays(a, L, nq, sms, false)) a.staged = 1;
}

cudaError_t launch_search(const SearchArgs &a, int blocks, int tw, cudaStream_t s, bool configure) {
    const void *fn = search_kernel(a, tw);
    if (!fn || blocks <= 0) return cudaErrorInvalidValue;
    const size_t smem = search_smem_per_team(a, stage_of(a)) * teams_per_block(tw);
    cudaError_t e = cudaSuccess;
    if (configure) {  // already done by search_blocks_per_sm when planning
        e = allow_smem(fn);
        if (e != cudaSuccess) return e;
    }
    e = cudaMemsetAsync(a.work, 0, sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    void *args[] = {const_cast<SearchArgs *>(&a)};
    return cudaLaunchKernel(fn, dim3(blocks), dim3(threads_for(tw)), args, smem, s);
}

}  // namespace roar

// Tensor-core scores with a fused running top-C (the kNN step of the index
// construction, Sec. 4.2.1): S = T . X^T in BF16 with FP32 accumulation on the
// 5th-generation tensor cores, never written to memory.
//
// Two CTAs of a cluster (a pair on neighbouring SMs) work on one block of 256
// rows of T with cta_group::2 MMAs of M = N = 256: each CTA keeps its own 128
// rows resident in shared memory and holds their scores in its own TMEM, and
// each loads only its half of every X tile, which the MMA of the pair reads from
// both shared memories. A unit of work is one block of T rows and one range of
// X tiles; the pairs are persistent and take units in turn, so a few T rows
// still use every SM (the X ranges' lists are merged afterwards), and the
// candidate buffers belong to a CTA, not to a row of T.
//
// Warp roles per CTA: warp 0 stages operands by TMA (2-D tensor maps, 64-column
// boxes in the 128-byte-swizzled K-major layout; both CTAs' copies count their
// bytes on the leader's barriers); warp 1 owns TMEM and, in the leader CTA
// (rank 0), issues every tcgen05.mma into one of two alternating accumulators;
// K steps that hold only the padding of d to 64 columns are not issued (d =
// 200: 13 of 16). The 16 other warps read TMEM with tcgen05.ld, one row of T
// per thread, and filter the scores: per row a running threshold (the C-th best
// score so far) decides which enter the row's candidate buffer. The buffers are
// trimmed back to about their best C each time the X rows seen have doubled,
// which raises the thresholds. The best C of a row are those first in (score
// descending, id ascending) order, whatever the units, the sets and the trims.
//
// What bounds it (GB300, 131,072 T rows x 1M x 200, whole call; 90.1 ms as one
// CTA per 256 T rows with lane 0 in the MMA loop): the MMAs alone run at 90 % of
// the measured BF16 burst (35 ms), reading TMEM and testing the scores beside
// them 42 ms, accepting about 1,900 scores per T row and trimming 49 ms. What
// brought it there: the MMA warp kept uniform (79 -> 64 ms: its operands had
// been moved to uniform registers for every MMA, longer than the MMA took);
// trims at the same tiles in all warps instead of each list as it fills (62 ->
// 55: every cut held up the pair's MMAs); 16 epilogue warps in two sets that
// take alternate tiles, one 64-column TMEM load at a time (55 -> 49: a load waits
// for its turn between the MMAs, whatever its width).
//
// Every mbarrier wait is bounded (wait_ns of wall time per wait): on timeout
// the kernel sets *err, waits for its copies and for the MMAs it has issued,
// frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "roar_knn_tc.cuh"

namespace roar {

roar_status cuda_fail(cudaError_t e, const char *what);

namespace {

constexpr int kTM = 128;           // T rows in one CTA (TMEM lanes); the pair's MMA has M = 256
constexpr int kKC = 64;            // K elements per staged chunk (128 bytes per row)
constexpr int kC = 128;            // candidates kept per row
constexpr int kMaxStages = 16;
constexpr int kCols = 128;         // columns of a tile one epilogue warp filters
constexpr int kTrimMost = 384;     // entries of a row a trim takes in registers (12 per lane)
constexpr int kSegCut = 256;       // a segment of a row's candidate buffer with more entries is cut at once;
constexpr int kSegCap = kSegCut + kCols;     // so that it can take another tile's
constexpr uint64_t kDrainNs = 2000000000ull;  // bound of the final wait for issued MMAs and copies
constexpr int kTmemCols = 512;     // 2 accumulators of 256 columns
constexpr uint32_t kChunkA = kTM * kKC * 2;   // 16 KB: one CTA's T rows, a 64-wide K chunk
constexpr unsigned kFull = 0xFFFFFFFFu;

constexpr int kTN = 256;           // X rows per tile: the MMA's N, two accumulators of which fill TMEM
constexpr int kSegs = 2 * (kTN / kCols);      // epilogue warps per 32 rows: two sets x kTN / kCols
constexpr int kEpiWarps = 4 * kSegs;
constexpr int kThreads = (2 + kEpiWarps) * 32;
constexpr uint32_t kChunkB = (uint32_t)(kTN / 2) * kKC * 2;   // 16 KB: one CTA's half of a tile's K chunk
// Instruction descriptor, kind::f16: D = F32 (bits 4-5 = 1), A = B = BF16
// (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bit 17,
// M >> 4 at bit 24.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTN >> 3) << 17) |
                            ((uint32_t)((2 * kTM) >> 4) << 24);

// One call's units: blocks of 256 T rows x `splits` ranges of X tiles.
struct KnnUnits {
    int64_t nt, n, tiles;
    int nkc, ksteps;         // 64-column chunks, 16-column MMA steps
    int splits;
    int64_t units;
};

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// True in one lane of the (converged) warp, the same one every time.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xFFFFFFFF;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}

// The shared::cluster address of a shared-memory location of CTA `rank`.
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

__device__ __forceinline__ int64_t ld_cluster_s64(uint32_t addr) {
    int64_t v;
    asm volatile("ld.shared::cluster.s64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
    return v;
}

// All threads of both CTAs (each always gets here: every wait before it is bounded).
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}

// Shared-memory matrix descriptor of the 128-byte-swizzled K-major layout TMA
// writes: rows of 128 bytes (64 BF16 of K), the 16-byte pieces of row r at
// piece ^ (r % 8), 8-row atoms 1024 bytes apart (stride offset, >> 4 at bit
// 32); the atoms are 1024-byte aligned (base offset 0). Start address >> 4 in
// the low 14 bits, descriptor version 1 at bit 46, swizzle mode 2 (128-byte)
// in bits 61-63. A K step of 16 elements advances the start by 32 bytes.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Arm a barrier for `bytes` of asynchronous copies (one arrival).
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

// TMA: the box at (x = column, y = row) of the 2-D tensor map to this CTA's
// shared memory; completion counted in bytes on `bar` (a shared::cluster
// address: the leader's barrier).
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int32_t x, int32_t y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count));
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase with the given parity: gives up (and raises the
// CTA's abort flag) after wait_ns of wall time, or as soon as another role
// aborted. wait_ns == 0 gives up as soon as the phase is found incomplete
// (a test setting: it makes the timeout path run without any fault).
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort, uint64_t wait_ns) {
    if (wait_ns == 0) {
        if (mbar_test(bar, parity)) return true;
        *abort = 1;
        return false;
    }
    uint64_t deadline = 0;
    for (uint32_t i = 0;; ++i) {
        if (mbar_try(bar, parity)) return true;
        if (*abort) return false;
        if ((i & 63) == 0) {
            const uint64_t now = global_ns();
            if (deadline == 0) deadline = now + wait_ns;
            else if (now > deadline) {
                *abort = 1;
                return false;
            }
        }
    }
}

// Bounded wait that ignores the abort flag: the final wait for issued MMAs and
// copies (they always complete; the bound only keeps the wait finite).
__device__ __forceinline__ bool mbar_drain(uint64_t *bar, uint32_t parity) {
    uint64_t deadline = 0;
    for (uint32_t i = 0;; ++i) {
        if (mbar_try(bar, parity)) return true;
        if ((i & 63) == 0) {
            const uint64_t now = global_ns();
            if (deadline == 0) deadline = now + kDrainNs;
            else if (now > deadline) return false;
        }
    }
}

// Arrive on a barrier of either CTA (a shared::cluster address).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The barrier at this offset in both CTAs gets one arrival once this thread's
// earlier MMAs have completed.
__device__ __forceinline__ void tc_commit_pair(uint64_t *bar) {
    const uint16_t mask = 3;
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_addr(bar)),
        "h"(mask)
        : "memory");
}

// Issue a load of 64 consecutive FP32 columns of this thread's TMEM lane; the
// registers are valid only after tc_wait_ld. (One load of 64: between the
// MMAs' own accesses TMEM serves about one load per MMA, whatever its width.)
__device__ __forceinline__ void tc_ld64_issue(uint32_t taddr, uint32_t (&a)[32], uint32_t (&b)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%64];"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15]), "=r"(a[16]), "=r"(a[17]), "=r"(a[18]), "=r"(a[19]), "=r"(a[20]), "=r"(a[21]), "=r"(a[22]), "=r"(a[23]), "=r"(a[24]), "=r"(a[25]), "=r"(a[26]), "=r"(a[27]), "=r"(a[28]), "=r"(a[29]), "=r"(a[30]), "=r"(a[31]), "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7]), "=r"(b[8]), "=r"(b[9]), "=r"(b[10]), "=r"(b[11]), "=r"(b[12]), "=r"(b[13]), "=r"(b[14]), "=r"(b[15]), "=r"(b[16]), "=r"(b[17]), "=r"(b[18]), "=r"(b[19]), "=r"(b[20]), "=r"(b[21]), "=r"(b[22]), "=r"(b[23]), "=r"(b[24]), "=r"(b[25]), "=r"(b[26]), "=r"(b[27]), "=r"(b[28]), "=r"(b[29]), "=r"(b[30]), "=r"(b[31])
        : "r"(taddr));
}

// Wait for this thread's TMEM loads. The registers of the loads pass through
// the statement, so no use of them can be scheduled before the wait.
__device__ __forceinline__ void tc_wait_ld(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}

// Orders later uses of `r` after the preceding (volatile) wait.
__device__ __forceinline__ void reg_after_wait(uint32_t (&r)[32]) {
    asm volatile(""
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31]));
}

// Order-preserving map of a finite float to uint32 (larger float, larger key).
__device__ __forceinline__ uint32_t f2key(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float key2f(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// 32 columns of a row's scores: columns lim and up can no longer be taken.
__device__ __forceinline__ void mask_past(uint32_t (&r)[32], int lim) {
#pragma unroll
    for (int i = 0; i < 32; ++i)
        if (i >= lim) r[i] = 0xFF800000u;   // -inf
}

// Bit g: the maximum of columns 8 g .. 8 g + 7 beats the threshold.
__device__ __forceinline__ uint32_t group_hits(const uint32_t (&r)[32], float thr) {
    uint32_t m = 0;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const uint32_t *v = r + 8 * g;
        float x = max3(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]));
        x = max3(x, __uint_as_float(v[3]), __uint_as_float(v[4]));
        x = max3(x, __uint_as_float(v[5]), __uint_as_float(v[6]));
        x = fmaxf(x, __uint_as_float(v[7]));
        if (x > thr) m |= 1u << g;
    }
    return m;
}

// Appends the columns of the groups in `hit` (the same in all lanes) that beat
// the row's threshold to its buffer: predicated, without a branch per score.
__device__ __forceinline__ void take(const uint32_t (&r)[32], uint32_t hit, float thr, uint32_t id0, uint64_t &end) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        if (hit & (1u << g)) {
#pragma unroll
            for (int i = 8 * g; i < 8 * g + 8; ++i)
                asm volatile(
                    "{\n .reg .pred p;\n setp.gt.f32 p, %1, %2;\n @p st.global.v2.b32 [%0], {%3, %4};\n"
                    " @p add.u64 %0, %0, 8;\n}\n"
                    : "+l"(end)
                    : "f"(__uint_as_float(r[i])), "f"(thr), "r"(r[i]), "r"(id0 + i)
                    : "memory");
        }
    }
}

// 64 columns of a row's scores, `left` of them within n, ids from id0: those
// that beat the threshold go to the row's buffer. Most lie below it: one bit
// per 8 columns tells whether any row of the warp takes one there.
__device__ __forceinline__ void filter(uint32_t (&ra)[32], uint32_t (&rb)[32], int64_t left, float thr, uint32_t id0,
                                       uint64_t &end) {
    if (left < 64) {   // the last tile
        mask_past(ra, (int)max(left, (int64_t)0));
        mask_past(rb, (int)max(left - 32, (int64_t)0));
    }
    uint32_t hit = group_hits(ra, thr) | group_hits(rb, thr) << 4;
    hit = __reduce_or_sync(kFull, hit);
    if (hit & 0xFu) take(ra, hit, thr, id0, end);
    if (hit & 0xF0u) take(rb, hit >> 4, thr, id0 + 32, end);
}

// A row's candidates: up to kSegs segments of kSegCap entries (score, id), read
// as one list.
template <int kSegs>
struct RowList {
    uint2 *base;
    int m[kSegs];
    __device__ __forceinline__ int size() const {
        int t = 0;
#pragma unroll
        for (int e = 0; e < kSegs; ++e) t += m[e];
        return t;
    }
    // Entry j < size().
    __device__ __forceinline__ uint2 at(int j) const {
        const uint2 *p = base;
#pragma unroll
        for (int e = 0; e + 1 < kSegs; ++e) {
            if (p == base + e * kSegCap && j >= m[e]) {
                j -= m[e];
                p += kSegCap;
            }
        }
        return p[j];
    }
};

// The whole warp picks the best `keep` of a list of at most 32 kPer entries in
// (score descending, id ascending) order and calls put(i, entry) for each, i =
// 0 .. keep - 1 in list order; returns the keep-th best score. That score's key
// is found bit by bit, from the highest bit in which the keys differ, stopping
// as soon as a prefix holds exactly `keep`; among entries of that key the
// lowest ids are kept, found the same way when there are too many. All 32
// lanes call it with the same arguments, after the lanes that wrote the list
// have passed a barrier with them. put may overwrite the list.
template <int kPer, class List, class Put>
__device__ __forceinline__ float warp_cut(const List &list, int keep, int lane, Put &&put) {
    const int m = list.size();
    uint32_t key[kPer], id[kPer];
    uint32_t kmax = 0, kmin = 0xFFFFFFFFu;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int j = i * 32 + lane;
        const uint2 e = j < m ? list.at(j) : make_uint2(0u, 0u);
        key[i] = j < m ? f2key(__uint_as_float(e.x)) : 0u;
        id[i] = e.y;
        kmax = max(kmax, key[i]);
        if (j < m) kmin = min(kmin, key[i]);
    }
    kmax = __reduce_max_sync(kFull, kmax);
    kmin = __reduce_min_sync(kFull, kmin);
    uint32_t t = kmin, idt = 0xFFFFFFFFu;
    if (m > keep) {
        if (kmax != kmin) {
            int bit = 31 - __clz(kmax ^ kmin);
            t = bit == 31 ? 0u : kmax & ~((2u << bit) - 1u);   // the common prefix
            for (; bit >= 0; --bit) {
                const uint32_t c = t | (1u << bit);
                uint32_t cnt = 0;
#pragma unroll
                for (int i = 0; i < kPer; ++i) cnt += key[i] >= c ? 1u : 0u;
                cnt = __reduce_add_sync(kFull, cnt);
                if ((int)cnt >= keep) t = c;
                if ((int)cnt == keep) {
                    uint32_t low = 0xFFFFFFFFu;
#pragma unroll
                    for (int i = 0; i < kPer; ++i) low = key[i] >= c ? min(low, key[i]) : low;
                    t = __reduce_min_sync(kFull, low);
                    break;
                }
            }
        }
        uint32_t above = 0, ties = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            above += key[i] > t ? 1u : 0u;
            ties += key[i] == t ? 1u : 0u;
        }
        above = __reduce_add_sync(kFull, above);
        ties = __reduce_add_sync(kFull, ties);
        const uint32_t room = (uint32_t)keep - above;
        if (ties > room) {   // idt: the room-th lowest id of the ties
            idt = 0;
            for (int bit = 30; bit >= 0; --bit) {
                const uint32_t c = idt | (1u << bit);
                uint32_t below = 0;
#pragma unroll
                for (int i = 0; i < kPer; ++i) below += key[i] == t && id[i] < c ? 1u : 0u;
                if (__reduce_add_sync(kFull, below) < room) idt = c;
            }
        }
    }
    __syncwarp();  // every lane has read the list before it is rewritten
    const uint32_t lt = (1u << lane) - 1u;
    int pos = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const bool take = i * 32 + lane < m && (key[i] > t || (key[i] == t && id[i] <= idt));
        const uint32_t b = __ballot_sync(kFull, take);
        if (take) put(pos + __popc(b & lt), make_uint2(__float_as_uint(key2f(key[i])), id[i]));
        pos += __popc(b);
    }
    __syncwarp();
    return key2f(t);
}

// Cuts every segment of a row that holds more than kC entries to its best kC.
template <int kSegs>
__device__ __noinline__ void cut_segments(RowList<kSegs> &l, int lane) {
#pragma unroll 1
    for (int e = 0; e < kSegs; ++e) {
        RowList<1> one;
        one.base = l.base + e * kSegCap;
        int me = 0;
#pragma unroll
        for (int x = 0; x < kSegs; ++x)
            if (x == e) me = l.m[x];
        if (me <= kC) continue;
        one.m[0] = me;
        uint2 *const dst = one.base;
        warp_cut<kSegCap / 32>(one, kC, lane, [&](int i, uint2 v) { dst[i] = v; });
#pragma unroll
        for (int x = 0; x < kSegs; ++x)
            if (x == e) l.m[x] = kC;
    }
}

// The whole warp trims kRows rows at once (their latencies overlap) to their
// best kC to kC + kTrimSlack candidates, which it writes to their first
// segments: a score key t is searched as in warp_cut, but the search ends as
// soon as the entries of key t and up are that few (ties may leave more). Rows
// of more than kTrimMost entries are cut exactly. Rows of at most kC entries
// keep them all. kept[r]: entries left. thr[r]: the row's best kC of all X rows
// so far score at least this, so a later one (of higher id) has to beat it.
constexpr int kTrimSlack = 24;
template <int kRows, int kSegs>
__device__ __forceinline__ void warp_trim(RowList<kSegs> (&l)[kRows], int (&kept)[kRows], float (&thr)[kRows], int lane) {
    constexpr int kPer = kTrimMost / 32;
    int m[kRows];
    bool wide = false;
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        m[r] = l[r].size();
        wide |= m[r] > kTrimMost;
    }
    if (wide) {   // lists that filled faster than their share
#pragma unroll 1
        for (int r = 0; r < kRows; ++r) {
            RowList<kSegs> x = l[0];
#pragma unroll
            for (int y = 1; y < kRows; ++y)
                if (y == r) x = l[y];
            cut_segments<kSegs>(x, lane);
            const int n = min(x.size(), kC);
            const bool more = x.size() > kC;
            const float t = warp_cut<4 * kSegs>(x, kC, lane, [&](int i, uint2 v) { x.base[i] = v; });
#pragma unroll
            for (int y = 0; y < kRows; ++y) {
                if (y == r) {
                    kept[y] = n;
                    thr[y] = more || n == kC ? t : -__int_as_float(0x7f800000);
                }
            }
        }
        return;
    }
    uint32_t key[kRows][kPer], id[kRows][kPer], t[kRows], kmin[kRows];
    int bit[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int j = i * 32 + lane;
            const uint2 e = j < m[r] ? l[r].at(j) : make_uint2(0xFFFFFFFFu, 0u);   // (key 0)
            key[r][i] = e.x;
            id[r][i] = e.y;
        }
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        uint32_t hi = 0, lo = 0xFFFFFFFFu;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            key[r][i] = f2key(__uint_as_float(key[r][i]));
            hi = max(hi, key[r][i]);
            if (i * 32 + lane < m[r]) lo = min(lo, key[r][i]);
        }
        hi = __reduce_max_sync(kFull, hi);
        kmin[r] = __reduce_min_sync(kFull, lo);
        bit[r] = 31 - __clz(hi ^ kmin[r]);                        // -1: all keys equal
        t[r] = bit[r] >= 31 ? 0u : hi & ~((2u << bit[r]) - 1u);   // the common prefix (hi itself at -1)
        kept[r] = m[r];
    }
    for (;;) {
        bool more = false;
        uint32_t c[kRows], cnt[kRows];
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            const bool act = bit[r] >= 0 && kept[r] > kC + kTrimSlack;
            more |= act;
            c[r] = act ? t[r] | (1u << bit[r]) : 0xFFFFFFFFu;   // above every key
            cnt[r] = 0;
#pragma unroll
            for (int i = 0; i < kPer; ++i) cnt[r] += key[r][i] >= c[r] ? 1u : 0u;
        }
        if (!more) break;   // (uniform: reduced values)
#pragma unroll
        for (int r = 0; r < kRows; ++r) cnt[r] = __reduce_add_sync(kFull, cnt[r]);
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            if ((int)cnt[r] >= kC) {
                t[r] = c[r];
                kept[r] = (int)cnt[r];
            }
            --bit[r];
        }
    }
    __syncwarp();  // every lane has read the lists before they are rewritten
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        t[r] = max(t[r], kmin[r]);
        int pos = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const bool take = i * 32 + lane < m[r] && key[r][i] >= t[r];
            const uint32_t w = __ballot_sync(kFull, take);
            if (take) l[r].base[pos + __popc(w & lt)] = make_uint2(__float_as_uint(key2f(key[r][i])), id[r][i]);
            pos += __popc(w);
        }
        thr[r] = kept[r] >= kC ? key2f(t[r]) : -__int_as_float(0x7f800000);
    }
    __syncwarp();
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
knn_tc_kernel(const KnnUnits u, int stages, uint2 *__restrict__ scratch, uint2 *__restrict__ out_e,
              uint32_t *__restrict__ out_i, int *__restrict__ err, uint64_t wait_ns,
              const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB) {
    extern __shared__ __align__(1024) unsigned char smem[];
    // full, a_full, acc_empty: used in the leader; empty, a_empty, acc_full: in both CTAs
    __shared__ uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], acc_full[2], acc_empty[2], a_full, a_empty,
        drain_bar;
    __shared__ int64_t issued_ops;   // copy operations this CTA's producer has issued
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ int seg_cnt[kSegs][kTM];   // entries per segment and row, at a trim
    __shared__ float row_thr[kTM];              // and what it gives
    __shared__ int row_kept[kTM];
    volatile int *abort_v = &abort_flag;

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(kFull, tid >> 5, 0);   // uniform over the warp, and seen to be
    const uint32_t rank = cluster_rank();
    const int64_t pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int nkc = u.nkc;
    // TMA's 128-byte swizzle repeats every 1024 bytes: start the operands there
    // (the same offset in both CTAs).
    const uint32_t a_base = (smem_addr(smem) + 1023u) & ~1023u;
    const uint32_t b_base = a_base + (uint32_t)nkc * kChunkA;
    auto first_row = [&](int64_t unit) { return (unit / u.splits) * (2 * kTM); };
    auto first_tile = [&](int64_t unit) { return (unit % u.splits) * u.tiles / u.splits; };
    auto last_tile = [&](int64_t unit) { return (unit % u.splits + 1) * u.tiles / u.splits; };

    if (tid == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], kEpiWarps);   // one arrival per epilogue warp of its set in both CTAs
        }
        mbar_init(&a_full, 1);
        mbar_init(&a_empty, 1);
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        issued_ops = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // both CTAs' barriers are initialised
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    // The producer's copy operations in order: per unit the T rows (one
    // operation), then one per K chunk of every tile. Issues operations
    // [from, to), waiting for free buffers unless `waits` is false, and returns
    // how many operations are issued in all (stops at a wait that gives up).
    auto produce = [&](int64_t from, int64_t to, bool waits) -> int64_t {
        int64_t op = 0;
        int s = 0;
        uint32_t wrap = 0, ui = 0;
        const uint32_t abar = map_rank(smem_addr(&a_full), 0), fbar = map_rank(smem_addr(&full_bar[0]), 0);
        for (int64_t unit = pair; unit < u.units; unit += npairs, ++ui) {
            const int64_t m0 = first_row(unit) + kTM * rank, t1 = last_tile(unit);
            if (op >= to) return op;
            if (op >= from) {
                if (waits && ui > 0 && !mbar_wait(&a_empty, (ui - 1) & 1, abort_v, wait_ns)) return op;
                if (rank == 0) mbar_expect_tx(&a_full, 2u * (uint32_t)nkc * kChunkA);
                for (int c = 0; c < nkc; ++c)
                    tma_load_2d(a_base + (uint32_t)c * kChunkA, &tmA, c * kKC, (int32_t)m0, abar);
            }
            ++op;
            for (int64_t t = first_tile(unit); t < t1; ++t) {
                const int32_t x0 = (int32_t)(t * kTN + (kTN / 2) * rank);
                for (int c = 0; c < nkc; ++c) {
                    if (op >= to) return op;
                    if (op >= from) {
                        if (waits && wrap > 0 && !mbar_wait(&empty_bar[s], (wrap - 1) & 1, abort_v, wait_ns)) return op;
                        if (rank == 0) mbar_expect_tx(&full_bar[s], 2u * kChunkB);
                        tma_load_2d(b_base + (uint32_t)s * kChunkB, &tmB, c * kKC, x0, fbar + 8u * s);
                    }
                    ++op;
                    if (++s == stages) {
                        s = 0;
                        ++wrap;
                    }
                }
            }
        }
        return op;
    };

    if (warp == 0) {
        if (lane == 0) issued_ops = produce(0, INT64_MAX, true);
        __syncwarp();
    } else if (warp == 1) {
        // ---- MMA issue (leader) ----
        // The whole warp walks the tiles together and one elected lane issues:
        // in warp-uniform code the descriptors stay in uniform registers. (With
        // lane 0 alone in the loop, every MMA's operands were moved there first,
        // which took longer than the MMA.)
        if (rank == 0) {
            bool issued = false, ok = true;
            const bool elected = elect_one();
            // Descriptors of the operand bases; a chunk or a K step moves the
            // start address field (bytes >> 4).
            const uint64_t adesc0 = smem_desc_sw128(a_base), bdesc0 = smem_desc_sw128(b_base);
            int s = 0;
            uint32_t wrap = 0, ui = 0, acc = 0;
            auto wait = [&](uint64_t *bar, uint32_t parity) {
                return __all_sync(kFull, mbar_wait(bar, parity, abort_v, wait_ns));
            };
            for (int64_t unit = pair; unit < u.units && ok; unit += npairs, ++ui) {
                if (!wait(&a_full, ui & 1)) break;
                const int64_t t1 = last_tile(unit);
                for (int64_t t = first_tile(unit); t < t1 && ok; ++t, ++acc) {
                    const uint32_t b = acc & 1, ub = acc >> 1;
                    if (ub > 0 && !wait(&acc_empty[b], (ub - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    for (int c = 0; c < nkc; ++c) {
                        if (!wait(&full_bar[s], wrap & 1)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint64_t bd0 = bdesc0 + (((uint32_t)s * kChunkB) >> 4);
                        const uint64_t ad0 = adesc0 + (((uint32_t)c * kChunkA) >> 4);
                        const uint32_t d0 = tmem + b * kTN;
                        const int steps = u.ksteps - c * (kKC / 16);   // past the last one: zero padding
                        if (elected) {
#pragma unroll
                            for (int ks = 0; ks < kKC / 16; ++ks) {
                                if (ks < steps)
                                    tc_mma(d0, ad0 + ks * 2, bd0 + ks * 2, kIdesc, (c > 0 || ks > 0) ? 1u : 0u);
                            }
                            tc_commit_pair(&empty_bar[s]);
                        }
                        issued = true;
                        if (++s == stages) {
                            s = 0;
                            ++wrap;
                        }
                    }
                    if (ok && elected) tc_commit_pair(&acc_full[b]);
                }
                if (ok && elected) tc_commit_pair(&a_empty);
            }
            // Every MMA the elected lane issued has finished (it may still be
            // writing TMEM and reading shared memory after an abort) before
            // the CTAs free their TMEM and exit.
            if (issued && elected) {
                asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 smem_addr(&drain_bar))
                             : "memory");
                if (!mbar_drain(&drain_bar, 0)) *abort_v = 1;
            }
        }
        __syncwarp();
    } else {
        // ---- epilogue: filter each tile's scores into the row buffers ----
        // Two sets of 8 warps take the tiles in turn (each its own
        // accumulator), so that one set's TMEM loads overlap the other's
        // filtering. kSegs warps share 32 rows (one per lane): each filters its
        // kCols columns of its tiles into its own segment of the rows' buffers.
        // They meet (named barrier) only where the lists are trimmed, which
        // depends on the tile number alone. After an abort (`dead`) a warp still
        // comes to every such barrier.
        const int q = warp & 3;              // TMEM lanes 32 q .. 32 q + 31
        const int grp = (warp - 2) >> 2;
        const uint32_t set = grp & 1;
        const int seg = grp, col0 = (grp >> 1) * kCols;
        const int row0 = 32 * q;             // of the CTA's rows
        uint2 *const wbuf = scratch + ((int64_t)blockIdx.x * kTM + row0) * (kSegs * kSegCap);
        const uint64_t mybuf =
            (uint64_t)__cvta_generic_to_global(wbuf + (int64_t)(lane * kSegs + seg) * kSegCap);
        const uint32_t taddr = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(set * kTN + col0);
        const uint32_t ebar = map_rank(smem_addr(&acc_empty[set]), 0);
        const float ninf = -__int_as_float(0x7f800000);
        auto meet = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + q), "n"(32 * kSegs) : "memory"); };
        auto list_of = [&](int r) {
            RowList<kSegs> l;
            l.base = wbuf + (int64_t)r * (kSegs * kSegCap);
#pragma unroll
            for (int e = 0; e < kSegs; ++e) l.m[e] = seg_cnt[e][row0 + r];
            return l;
        };
        uint32_t acc = 0;
        bool dead = false;
        for (int64_t unit = pair; unit < u.units; unit += npairs) {
            const int64_t wrow0 = first_row(unit) + kTM * rank + 32 * q;
            int cnt = 0;
            uint64_t end = mybuf;                                   // where the row's next entry goes
            float thr = wrow0 + lane < u.nt ? ninf : -ninf;         // rows past the end take nothing
            const int64_t t0 = first_tile(unit), t1 = last_tile(unit);
            for (int64_t t = t0; t < t1; ++t, ++acc) {
                const bool mine = (acc & 1) == set;
                // The warp leaves together: the TMEM loads below are warp-collective.
                if (mine && !dead &&
                    !__all_sync(kFull, mbar_wait(&acc_full[set], (acc >> 1) & 1, abort_v, wait_ns)))
                    dead = true;
                if (mine && !dead) {
                    uint32_t full = __ballot_sync(kFull, cnt > kSegCut);
                    while (full) {   // filled before its trim is due, or left so by ties
                        const int src = __ffs(full) - 1;
                        full &= full - 1;
                        RowList<1> one;
                        one.base = wbuf + (int64_t)(src * kSegs + seg) * kSegCap;
                        one.m[0] = __shfl_sync(kFull, cnt, src);
                        const float th = warp_cut<kSegCap / 32>(one, kC, lane, [&](int i, uint2 v) { one.base[i] = v; });
                        if (lane == src) {
                            thr = fmaxf(thr, th);
                            cnt = kC;
                            end = mybuf + 8 * kC;
                        }
                    }
                    tc_fence_after();
#pragma unroll 1
                    for (int c = 0; c < kCols; c += 64) {
                        uint32_t r0[32], r1[32];
                        tc_ld64_issue(taddr + c, r0, r1);
                        tc_wait_ld(r0);
                        reg_after_wait(r1);
                        if (c + 64 == kCols) {   // the scores are in registers: the accumulator is free
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive_cluster(ebar);
                        }
                        const int64_t n0 = t * kTN + col0 + c;
                        filter(r0, r1, u.n - n0, thr, (uint32_t)n0, end);
                    }
                    cnt = (int)((end - mybuf) >> 3);
                    __syncwarp();
                }
                // Trim the lists each time the rows of X seen have doubled
                // (about kC new entries per row each).
                const uint32_t seen = (uint32_t)(t + 1 - t0);
                if (seen * kTN < 2 * kC || (seen & (seen - 1)) != 0) continue;
                seg_cnt[seg][row0 + lane] = cnt;
                meet();
                if (!dead) {
                    constexpr int kRows = 2;
#pragma unroll 1
                    for (int r = seg * (32 / kSegs); r < (seg + 1) * (32 / kSegs) && wrow0 + r < u.nt; r += kRows) {
                        RowList<kSegs> l[kRows];
                        int kept[kRows];
                        float th[kRows];
#pragma unroll
                        for (int x = 0; x < kRows; ++x) l[x] = list_of(r + x);
                        warp_trim<kRows, kSegs>(l, kept, th, lane);
#pragma unroll
                        for (int x = 0; x < kRows; ++x) {
                            if (lane == 0) {
                                row_thr[row0 + r + x] = th[x];
                                row_kept[row0 + r + x] = kept[x];
                            }
                        }
                    }
                }
                meet();
                // A warp that skipped its rows saw the abort flag before this barrier.
                if (__any_sync(kFull, *abort_v != 0)) dead = true;
                if (!dead) {
                    thr = fmaxf(thr, row_thr[row0 + lane]);
                    cnt = seg == 0 && wrow0 + lane < u.nt ? row_kept[row0 + lane] : 0;   // (no row past the end is trimmed)
                    end = mybuf + 8 * cnt;
                }
            }
            // The unit's lists: the best kC of each row, padded with 0xFFFFFFFF.
            seg_cnt[seg][row0 + lane] = cnt;
            meet();
            if (__any_sync(kFull, *abort_v != 0)) dead = true;
            for (int r = seg * (32 / kSegs); r < (seg + 1) * (32 / kSegs) && !dead && wrow0 + r < u.nt; ++r) {
                RowList<kSegs> l = list_of(r);
                if (l.size() > kTrimMost) cut_segments<kSegs>(l, lane);
                const int64_t o = ((wrow0 + r) * u.splits + unit % u.splits) * kC;
                auto put = [&](int i, uint2 v) {
                    if (u.splits > 1) out_e[o + i] = v;
                    else out_i[o + i] = v.y;
                };
                constexpr int kPer = 4 * kSegs > kTrimMost / 32 ? 4 * kSegs : kTrimMost / 32;
                warp_cut<kPer>(l, kC, lane, put);
                for (int i = l.size() + lane; i < kC; i += 32) put(i, make_uint2(0xFF800000u, 0xFFFFFFFFu));
            }
            meet();   // the buffers are free for the next unit
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    // No copy may still be landing when a CTA exits. After an abort the two
    // producers may have stopped at different operations, and the leader's
    // barriers count both CTAs' bytes: the one behind issues what it is behind
    // (its buffers are free: the other has seen them so), then the leader waits,
    // bounded, for the last phase armed on every barrier.
    if (warp == 0 && lane == 0) {
        const int64_t mine = issued_ops, theirs = ld_cluster_s64(map_rank(smem_addr(&issued_ops), rank ^ 1));
        if (mine < theirs) produce(mine, theirs, false);
        if (rank == 0) {
            const int64_t ops = mine > theirs ? mine : theirs;
            int64_t left = ops, na = 0, nb = 0;   // operations issued on T rows and on X chunks
            for (int64_t unit = pair; unit < u.units && left > 0; unit += npairs) {
                const int64_t ch = (last_tile(unit) - first_tile(unit)) * nkc;
                ++na;
                --left;
                nb += left < ch ? left : ch;
                left -= left < ch ? left : ch;
            }
            bool drained = na == 0 || mbar_drain(&a_full, (uint32_t)(na - 1) & 1);
            for (int i = 0; i < stages && i < nb; ++i)
                drained = mbar_drain(&full_bar[i], (uint32_t)((nb - 1 - i) / stages) & 1) && drained;
            if (!drained) *abort_v = 1;
        }
    }
    __syncthreads();
    cluster_sync();
    if (*abort_v && tid == 0) atomicExch(err, 1);
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
    }
}

// The best kC of a row from its `splits` lists (each padded at its end), in the
// kernel's order: one warp per row, lists taken in turn while the running kC
// fit beside them in 32 entries per lane.
struct FlatList {
    const uint2 *p;
    int m;
    __device__ __forceinline__ int size() const { return m; }
    __device__ __forceinline__ uint2 at(int j) const { return p[j]; }
};
__global__ void __launch_bounds__(128) knn_merge_kernel(const uint2 *__restrict__ e, int64_t nt, int splits,
                                                        uint32_t *__restrict__ out) {
    __shared__ uint2 buf[4][1024];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * 4 + w;
    if (row >= nt) return;
    uint2 *const b = buf[w];
    int m = 0;
    for (int s = 0; s < splits; ++s) {
        const uint2 *src = e + (row * splits + s) * kC;
        for (int j0 = 0; j0 < kC; j0 += 32) {
            const uint2 v = src[j0 + lane];
            const unsigned have = __ballot_sync(kFull, v.y != 0xFFFFFFFFu);
            if (v.y != 0xFFFFFFFFu) b[m + __popc(have & ((1u << lane) - 1u))] = v;
            m += __popc(have);
        }
        __syncwarp();
        if (m > kC && (m > 1024 - kC || s + 1 == splits)) {
            warp_cut<32>(FlatList{b, m}, kC, lane, [&](int i, uint2 v) { b[i] = v; });
            m = kC;
        }
    }
    for (int j = lane; j < kC; j += 32) out[row * kC + j] = j < m ? b[j].y : 0xFFFFFFFFu;
}

int knn_tc_stages(int nkc) {
    return std::min(kMaxStages, (220 * 1024 - nkc * (int)kChunkA) / (int)kChunkB);
}

size_t knn_tc_smem_bytes(int nkc) {
    const size_t need = (size_t)nkc * kChunkA + (size_t)knn_tc_stages(nkc) * kChunkB + 1024;
    return need < 120 * 1024 ? 120 * 1024 : need;  // one CTA per SM: it holds all 512 TMEM columns
}

// cuTensorMapEncodeTiled, looked up through the runtime (no link to the
// driver library).
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
    static EncodeTiledFn fn = []() -> EncodeTiledFn {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// A BF16 matrix [rows][dp] (row-major, dp % 16 == 0 so rows are 32-byte
// multiples) read in boxes of 64 columns x box_rows rows with the 128-byte
// swizzle; reads past the last row or column return zeros.
bool make_map(CUtensorMap *m, const __nv_bfloat16 *base, int64_t rows, int dp, int box_rows) {
    const EncodeTiledFn fn = encode_tiled();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)dp, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)dp * 2u};
    const cuuint32_t box[2] = {(cuuint32_t)kKC, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1u, 1u};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16 *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// CTA pairs that run at once (one CTA per SM).
cudaError_t resident_pairs(size_t smem, int *pairs) {
    cudaError_t e = cudaFuncSetAttribute(knn_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         222 * 1024);   // the most any width needs: calls of several threads share it
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 2;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(pairs, knn_tc_kernel, &cfg);
    if (e == cudaSuccess && *pairs < 1) e = cudaErrorInvalidConfiguration;
    return e;
}

}  // namespace

// Every number of X ranges is priced in rows of X swept by the busiest pair:
// ceil(units / pairs) units of n / splits rows each, plus kUnitRows per unit for
// what a unit costs before its thresholds filter (measured on GB300: 10,000 T
// rows x 1M x 200 7.0 ms with 80,000, 7.2 with 40,000, 7.6 with 10,000).
cudaError_t knn_tc_plan(int64_t nt, int64_t n, int d, KnnPlan *p) {
    constexpr double kUnitRows = 80000.0;
    p->nkc = (d + kKC - 1) / kKC;
    p->ksteps = (d + 15) / 16;
    int pairs = 0;
    const cudaError_t e = resident_pairs(knn_tc_smem_bytes(p->nkc), &pairs);
    if (e != cudaSuccess) return e;
    const int64_t blocks = (nt + 2 * kTM - 1) / (2 * kTM), tiles = (n + kTN - 1) / kTN;
    const int most = (int)std::max<int64_t>(1, std::min<int64_t>(pairs, tiles / 4));
    double best = 1e300;
    for (int s = 1; s <= most; ++s) {
        const int64_t waves = (blocks * s + pairs - 1) / pairs;
        const double cost = (double)waves * ((double)n / s + kUnitRows);
        if (cost < best * 0.98) {
            best = cost;
            p->splits = s;
        }
    }
    p->units = blocks * p->splits;
    p->pairs = (int)std::min<int64_t>(pairs, p->units);
    p->scratch_bytes = (size_t)p->pairs * 2 * kTM * kSegs * kSegCap * sizeof(uint2);
    p->lists_bytes = p->splits > 1 ? (size_t)nt * p->splits * kC * sizeof(uint2) : 0;
    return cudaSuccess;
}

// T rows of whole waves of the kernel (every pair one block) at width d.
int64_t knn_tc_wave_rows(int d) {
    int pairs = 0;
    if (resident_pairs(knn_tc_smem_bytes((d + kKC - 1) / kKC), &pairs) != cudaSuccess) {
        cudaGetLastError();
        pairs = 1;
    }
    return (int64_t)pairs * 2 * kTM;
}

// Candidates (best 128 per row, unsorted, 0xFFFFFFFF padded) of nt rows of T16
// against X16 (rows of dp columns, d rounded up to 16 with zeros) into cand
// [nt][128].
cudaError_t knn_tc_launch(const KnnPlan &p, const __nv_bfloat16 *T16, int64_t nt, const __nv_bfloat16 *X16, int64_t n,
                          int dp, void *scratch, void *lists, uint32_t *cand, int *err, uint64_t wait_ns,
                          cudaStream_t s) {
    alignas(64) CUtensorMap tmA, tmB;
    if (!make_map(&tmA, T16, nt, dp, kTM) || !make_map(&tmB, X16, n, dp, kTN / 2)) return cudaErrorInvalidValue;
    const int stages = knn_tc_stages(p.nkc);
    if (stages < 2) return cudaErrorInvalidValue;
    const size_t smem = knn_tc_smem_bytes(p.nkc);
    KnnUnits u;
    u.nt = nt;
    u.n = n;
    u.tiles = (n + kTN - 1) / kTN;
    u.nkc = p.nkc;
    u.ksteps = p.ksteps;
    u.splits = p.splits;
    u.units = p.units;
    knn_tc_kernel<<<2 * p.pairs, kThreads, smem, s>>>(u, stages, (uint2 *)scratch, (uint2 *)lists, cand, err, wait_ns, tmA,
                                                      tmB);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && p.splits > 1) {
        knn_merge_kernel<<<(unsigned)((nt + 3) / 4), 128, 0, s>>>((const uint2 *)lists, nt, p.splits, cand);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace roar

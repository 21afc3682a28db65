// AcquireNeighbors (Alg. 3, Sec. 4.2.3) for many nodes at once on the GPU: the
// pruning step of index construction (projection and connectivity
// enhancement keep, for node x, the candidates c that are closer to x than to
// every neighbour already kept).
//
// One CTA per node x (one warp where there are few candidates):
//   1. delta(x, c) = -dot(x, c) for every candidate, in the search's fixed FP32
//      order (score_rows: element i on lane (i >> 2) & 31, fmaf, xor
//      butterfly), padding ids (0xFFFFFFFF) dropped;
//   2. the candidates sorted by (delta, id) in shared memory (bitonic sort of
//      64-bit keys);
//   3. Alg. 3 in that order: skip x itself and ids already kept; keep the
//      first; keep any later c with delta(x, c) < delta(c, r) for every kept r;
//      stop at M; with fill, top up to M from the remaining candidates in
//      order.
// Every decision is taken in FP32 with those exact sums, so the result is
// defined without reference to any particular sort or launch shape.
//
// Step 3 looks sequential, but a candidate only depends on the rows kept before
// it. The kept rows sit in shared memory; each warp holds the rows of G
// candidates in registers and tests them against every kept row, two at a
// time, leaving as soon as all its candidates are out. The few of a chunk
// (all warps' candidates) that pass are then kept one at a time in order, each
// newly kept row being tested against the chunk's remaining ones only. So a
// candidate's row is read once and a kept row once per G candidates, from
// shared memory; one warp per node with the kept rows read from L1 / L2 for
// every candidate was bound by that traffic (65,536 nodes x 516 candidates,
// 1M x 200: about 540 GB through L2, 68.6 ms; this form
// 13.1 ms: 4.1 ms scoring, which is the rows' DRAM traffic at the copy rate,
// 0.6 ms sorting, the rest the tests, bound by their latency).
#include <algorithm>

#include "roar_search_kernel.cuh"

namespace roar {
roar_status cuda_fail(cudaError_t e, const char *what);
void set_error(const char *msg);
bool aligned(const void *p, size_t a);
}  // namespace roar

namespace roar {
namespace {

constexpr int kAcqMaxCand = 1024;   // candidates per node (sort capacity)
constexpr int kAcqMaxM = 64;        // kept neighbours per node
// Shared memory for kept rows per CTA: three CTAs per SM stay resident; kept
// rows past it (wide rows with a large M) are read from global memory.
constexpr int kAcqRowBytes = 64 * 1024;

// Candidates a warp holds in registers at a time (16-byte chunks: G * NCH <= 8).
template <int NCH>
__host__ __device__ constexpr int acq_group() {
    return NCH <= 2 ? 4 : (NCH <= 4 ? 2 : 1);
}

// The order of (distance, id) as one integer; -0 counts as +0, as in the
// float comparison.
__device__ __forceinline__ unsigned long long acq_key(float dist, uint32_t id) {
    const uint32_t u = __float_as_uint(dist + 0.0f);
    return ((unsigned long long)((u & 0x80000000u) ? ~u : (u | 0x80000000u)) << 32) | id;
}
__device__ __forceinline__ float acq_dist(unsigned long long key) {
    const uint32_t k = (uint32_t)(key >> 32);
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

template <int NCH>
__device__ __forceinline__ void load_query(const float *X, uint32_t u, int d4, float4 (&qr)[NCH], int lane) {
    const float4 *r = reinterpret_cast<const float4 *>(X) + (size_t)u * d4;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        const int ch = lane + 32 * c;
        qr[c] = ch < d4 ? __ldg(r + ch) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// Launch shape. Measured on GB300 (65,536 nodes x 516 candidates, 1M x 200, M =
// 32): 4 warps per CTA and 5 CTAs per SM 12.6-13.1 ms; 4 CTAs 14.0 ms, 6 (spilling)
// 17.8 ms; 8 warps per CTA 16.7-19.5 ms, 2 warps 16.4 ms. Rows of d > 256 hold
// more registers per candidate and more shared memory per node: there 8 warps,
// 2 CTAs per SM (20,000 nodes, d = 512: 7.5 ms, 4 warps 8.3-10.0 ms).
template <int NCH>
struct AcqShape {
    static constexpr int W = NCH <= 2 ? 4 : 8;
    static constexpr int kMinBlocks = NCH <= 2 ? 5 : 2;
    static constexpr int kKept = 2;                          // kept rows tested at a time
    static constexpr int kScoreRows = NCH >= 8 ? 1 : 8 / NCH;   // step 1: rows per batch (12 / NCH spilled)
};

// Tests a warp's candidates qc (distance to x of candidate g on the lanes
// whose reduced sum is g's: dc) against the kept rows r0 .. r1 - 1 and clears
// the losers' bits in `alive` (bit g * RS). Rows below scap are in shared
// memory, later ones are read from X.
template <int NCH, int G>
__device__ __forceinline__ uint32_t acq_test(uint32_t alive, const float4 (&qc)[G][NCH], float dc, int r0, int r1,
                                             const float4 *rows, int scap, const uint32_t *res, const float *X,
                                             int d4, int lane) {
    constexpr int RB = AcqShape<NCH>::kKept, RS = reduce_stride<RB * G>();
    for (int r = r0; r < r1 && alive; r += RB) {
        float s[RB * G];
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            const int rr = min(r + b, r1 - 1);   // an odd last row is tested twice
            const float4 *row = rr < scap ? rows + (size_t)rr * d4
                                          : reinterpret_cast<const float4 *>(X) + (size_t)res[rr] * d4;
#pragma unroll
            for (int g = 0; g < G; ++g) s[b * G + g] = 0.0f;
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
                const int ch = lane + 32 * c;
                if (ch < d4) {
                    const float4 x = row[ch];
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        s[b * G + g] = fmaf(qc[g][c].x, x.x, s[b * G + g]);
                        s[b * G + g] = fmaf(qc[g][c].y, x.y, s[b * G + g]);
                        s[b * G + g] = fmaf(qc[g][c].z, x.z, s[b * G + g]);
                        s[b * G + g] = fmaf(qc[g][c].w, x.w, s[b * G + g]);
                    }
                }
            }
        }
        const float rd = -reduce_rows<RB * G>(s, lane);
        uint32_t out = __ballot_sync(kFull, !(dc < rd));
#pragma unroll
        for (int b = 1; b < RB; ++b) out |= out >> (RS * G * b);
        alive &= ~out;
    }
    return alive;
}

template <int NCH>
__global__ void __launch_bounds__(32 * AcqShape<NCH>::W, AcqShape<NCH>::kMinBlocks)
acquire_kernel(const float *__restrict__ X, int64_t n, int d, const uint32_t *__restrict__ xs, int64_t nx,
               const uint32_t *__restrict__ cand, int cstride, const int32_t *__restrict__ ncand, int M,
               int fill, uint32_t *__restrict__ out, int32_t *__restrict__ out_cnt,
               uint32_t *__restrict__ sorted_out, int keycap, int scap) {
    constexpr int W = AcqShape<NCH>::W, B = AcqShape<NCH>::kScoreRows;
    constexpr int G = acq_group<NCH>();
    constexpr int RS = reduce_stride<AcqShape<NCH>::kKept * G>();
    constexpr int T = 32 * W, kPer = (kAcqMaxCand + T - 1) / T;
    static_assert(W * G <= 32, "a chunk's survivors fit one word");
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t res[kAcqMaxM], masks[2][W];
    __shared__ int s_nv, s_bad;
    const int d4 = d >> 2;
    float4 *rows = reinterpret_cast<float4 *>(smem);                                    // scap kept rows
    unsigned long long *key = reinterpret_cast<unsigned long long *>(rows + (size_t)scap * d4);   // [keycap]
    uint32_t *ci = reinterpret_cast<uint32_t *>(key);                                   // before the sort:
    float *cd = reinterpret_cast<float *>(ci + keycap);                                 // ids, then distances
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int64_t i = blockIdx.x; i < nx; i += gridDim.x) {
        const uint32_t x = xs[i];
        const int nc = min(max(ncand[i], 0), cstride);
        const uint32_t *ci_g = cand + (size_t)i * cstride;
        if (tid == 0) {
            s_nv = 0;
            s_bad = (int64_t)x >= n;
        }
        __syncthreads();
        // 0. validate and compact the candidate ids (padding dropped; any order).
        for (int b0 = 32 * w; b0 < nc; b0 += T) {
            const int j = b0 + lane;
            const uint32_t u = j < nc ? ci_g[j] : kNone;
            const bool ok = u != kNone && (int64_t)u < n;
            if (u != kNone && !ok) s_bad = 1;
            const unsigned m = __ballot_sync(kFull, ok);
            int p = 0;
            if (lane == 0 && m) p = atomicAdd(&s_nv, __popc(m));
            p = __shfl_sync(kFull, p, 0);
            if (ok) ci[p + __popc(m & ((1u << lane) - 1u))] = u;
        }
        __syncthreads();
        const int nv = s_nv;
        if (s_bad) {
            for (int j = tid; j < M; j += T) out[(size_t)i * M + j] = kNone;
            if (sorted_out)
                for (int j = tid; j < cstride; j += T) sorted_out[(size_t)i * cstride + j] = kNone;
            if (tid == 0) out_cnt[i] = -1;
            __syncthreads();
            continue;
        }
        // 1. delta(x, c) for every candidate.
        {
            float4 qr[NCH];
            load_query<NCH>(X, x, d4, qr, lane);
            score_rows<0, NCH, B>(X, nullptr, d, d4, qr, ci, nv, cd, lane, w * B, W * B);
        }
        __syncthreads();
        // 2. bitonic sort of the (delta, id) keys over the next power of two,
        // padded with the largest key. Warp w compares the pairs
        // [w * Q, (w + 1) * Q), so a step of distance j <= Q stays inside the
        // warp's own elements and needs no CTA barrier.
        int P = 2;
        while (P < nv) P <<= 1;
        {
            unsigned long long k[kPer];
#pragma unroll
            for (int e = 0; e < kPer; ++e) {
                const int j = tid + e * T;
                k[e] = j < nv ? acq_key(cd[j], ci[j]) : ~0ull;
            }
            __syncthreads();
#pragma unroll
            for (int e = 0; e < kPer; ++e) {
                const int j = tid + e * T;
                if (j < P) key[j] = k[e];
            }
            __syncthreads();
        }
        const int Q = max(1, P / 2 / W);
        for (int k = 2; k <= P; k <<= 1) {
            for (int j = k >> 1; j > 0; j >>= 1) {
                if (w * Q < P / 2) {
                    for (int p = w * Q + lane; p < (w + 1) * Q; p += 32) {
                        const int a = ((p & ~(j - 1)) << 1) | (p & (j - 1)), b = a + j;
                        const unsigned long long ka = key[a], kb = key[b];
                        if ((ka > kb) == ((a & k) == 0)) {
                            key[a] = kb;
                            key[b] = ka;
                        }
                    }
                }
                const int next = j > 1 ? j >> 1 : k;   // the next step's distance
                if (j > Q || next > Q) __syncthreads();
                else __syncwarp();
            }
        }
        __syncthreads();
        // 3. Alg. 3 over the sorted candidates, W * G at a time.
        int nr = 0, buf = 0;
        float4 qc[G][NCH];
        for (int t0 = 0; t0 < nv && nr < M; t0 += W * G) {
            const int tw = t0 + w * G;
            uint32_t alive = 0;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int t = tw + g;
                // equal ids are neighbours in the order: the second of a pair is
                // rejected or already kept whatever became of the first
                if (t < nv && (uint32_t)key[t] != x && (t == 0 || (uint32_t)key[t - 1] != (uint32_t)key[t]))
                    alive |= 1u << (g * RS);
                load_query<NCH>(X, (uint32_t)key[min(t, nv - 1)], d4, qc[g], lane);
            }
            const int mine = tw + (lane / RS) % G;
            const float dc = mine < nv ? acq_dist(key[mine]) : 0.0f;
            alive = acq_test<NCH, G>(alive, qc, dc, 0, nr, rows, scap, res, X, d4, lane);
            for (;;) {
                if (lane == 0) {
                    uint32_t m = 0;
#pragma unroll
                    for (int g = 0; g < G; ++g) m |= ((alive >> (g * RS)) & 1u) << (w * G + g);
                    masks[buf][w] = m;
                }
                __syncthreads();
                const uint32_t all = __reduce_or_sync(kFull, lane < W ? masks[buf][lane] : 0u);
                buf ^= 1;
                if (!all || nr == M) break;
                const int f = __ffs(all) - 1;   // the nearest survivor is kept
                if (f / G == w) {
                    if (nr < scap) {
#pragma unroll
                        for (int c = 0; c < NCH; ++c) {
                            // picked by masks: selects made the compiler index qc in local memory
                            uint4 v = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                            for (int g = 0; g < G; ++g) {
                                const uint32_t m = f % G == g ? ~0u : 0u;
                                v.x |= __float_as_uint(qc[g][c].x) & m;
                                v.y |= __float_as_uint(qc[g][c].y) & m;
                                v.z |= __float_as_uint(qc[g][c].z) & m;
                                v.w |= __float_as_uint(qc[g][c].w) & m;
                            }
                            if (lane + 32 * c < d4)
                                reinterpret_cast<uint4 *>(rows)[(size_t)nr * d4 + lane + 32 * c] = v;
                        }
                    }
                    if (lane == 0) res[nr] = (uint32_t)key[t0 + f];
                    alive &= ~(1u << ((f % G) * RS));
                }
                ++nr;
                __syncthreads();
                if (nr < M)
                    alive = acq_test<NCH, G>(alive, qc, dc, nr - 1, nr, rows, scap, res, X, d4, lane);
            }
        }
        __syncthreads();
        if (fill && w == 0) {
            for (int t = 0; t < nv && nr < M; ++t) {
                const uint32_t c = (uint32_t)key[t];
                if (c == x) continue;
                const bool dupl = (lane < nr && res[lane] == c) || (lane + 32 < nr && res[lane + 32] == c);
                if (__any_sync(kFull, dupl)) continue;
                if (lane == 0) res[nr] = c;
                ++nr;
                __syncwarp();
            }
        }
        // 4. outputs (warp 0 holds the final count).
        if (w == 0) {
            for (int j = lane; j < M; j += 32) out[(size_t)i * M + j] = j < nr ? res[j] : kNone;
            if (lane == 0) out_cnt[i] = nr;
        }
        if (sorted_out)
            for (int j = tid; j < cstride; j += T) sorted_out[(size_t)i * cstride + j] = j < nv ? (uint32_t)key[j] : kNone;
        __syncthreads();
    }
}

// Nodes of few candidates: one warp per node, its own arrays in shared memory,
// the kept rows read through L1. A CTA per node spends such a node on its
// barriers. (The rule and its figures: acquire_few_most.)
constexpr int kAcqFewCand = 40;
constexpr int kAcqFewSlots = 64;    // the sort's: the next power of two
struct AcqFew {                     // per warp
    float cd[kAcqFewSlots], rd[kAcqMaxM];
    uint32_t ci[kAcqFewSlots], res[kAcqMaxM];
};
static_assert(kAcqFewCand <= kAcqFewSlots, "the padded candidates fit");

__device__ __forceinline__ bool acq_less(float da, uint32_t ia, float db, uint32_t ib) {
    return da < db || (da == db && ia < ib);
}

template <int NCH>
__global__ void __launch_bounds__(128)
acquire_few_kernel(const float *__restrict__ X, int64_t n, int d, const uint32_t *__restrict__ xs, int64_t nx,
                   const uint32_t *__restrict__ cand, int cstride, const int32_t *__restrict__ ncand, int M,
                   int fill, uint32_t *__restrict__ out, int32_t *__restrict__ out_cnt,
                   uint32_t *__restrict__ sorted_out) {
    constexpr int B = batch_rows<0, NCH>();
    __shared__ AcqFew sm[4];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    AcqFew &S = sm[w];
    const int d4 = d >> 2;
    for (int64_t i = (int64_t)blockIdx.x * 4 + w; i < nx; i += (int64_t)gridDim.x * 4) {
        const uint32_t x = xs[i];
        const int nc = min(max(ncand[i], 0), cstride);
        const uint32_t *ci_g = cand + (size_t)i * cstride;
        bool bad = (int64_t)x >= n;
        int nv = 0;
        for (int b0 = 0; b0 < nc; b0 += 32) {
            const int j = b0 + lane;
            const uint32_t u = j < nc ? ci_g[j] : kNone;
            const bool ok = u != kNone && (int64_t)u < n;
            if (u != kNone && !ok) bad = true;
            const unsigned m = __ballot_sync(kFull, ok);
            if (ok) S.ci[nv + __popc(m & ((1u << lane) - 1u))] = u;
            nv += __popc(m);
        }
        if (__any_sync(kFull, bad)) {
            for (int j = lane; j < M; j += 32) out[(size_t)i * M + j] = kNone;
            if (sorted_out)
                for (int j = lane; j < cstride; j += 32) sorted_out[(size_t)i * cstride + j] = kNone;
            if (lane == 0) out_cnt[i] = -1;
            __syncwarp();
            continue;
        }
        __syncwarp();
        float4 qr[NCH];
        load_query<NCH>(X, x, d4, qr, lane);
        score_rows<0, NCH, B>(X, nullptr, d, d4, qr, S.ci, nv, S.cd, lane);
        // bitonic sort over the next power of two, padded with (+inf, kNone)
        int P = 1;
        while (P < nv) P <<= 1;
        for (int j = nv + lane; j < P; j += 32) {
            S.cd[j] = __int_as_float(0x7f800000);
            S.ci[j] = kNone;
        }
        __syncwarp();
        for (int k = 2; k <= P; k <<= 1) {
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int t = lane; t < P; t += 32) {
                    const int o = t ^ j;
                    if (o > t) {
                        const float da = S.cd[t], db = S.cd[o];
                        const uint32_t ia = S.ci[t], ib = S.ci[o];
                        if ((t & k) == 0 ? acq_less(db, ib, da, ia) : acq_less(da, ia, db, ib)) {
                            S.cd[t] = db;
                            S.cd[o] = da;
                            S.ci[t] = ib;
                            S.ci[o] = ia;
                        }
                    }
                }
                __syncwarp();
            }
        }
        int nr = 0;
        auto kept = [&](uint32_t c) {
            return __any_sync(kFull, (lane < nr && S.res[lane] == c) || (lane + 32 < nr && S.res[lane + 32] == c));
        };
        for (int t = 0; t < nv && nr < M; ++t) {
            const uint32_t c = S.ci[t];
            if (c == x || kept(c)) continue;
            if (nr > 0) {
                float4 qc[NCH];
                load_query<NCH>(X, c, d4, qc, lane);
                score_rows<0, NCH, B>(X, nullptr, d, d4, qc, S.res, nr, S.rd, lane);
                const float dc = S.cd[t];
                const bool viol = (lane < nr && !(dc < S.rd[lane])) || (lane + 32 < nr && !(dc < S.rd[lane + 32]));
                if (__any_sync(kFull, viol)) continue;
            }
            if (lane == 0) S.res[nr] = c;
            ++nr;
            __syncwarp();
        }
        if (fill) {
            for (int t = 0; t < nv && nr < M; ++t) {
                const uint32_t c = S.ci[t];
                if (c == x || kept(c)) continue;
                if (lane == 0) S.res[nr] = c;
                ++nr;
                __syncwarp();
            }
        }
        for (int j = lane; j < M; j += 32) out[(size_t)i * M + j] = j < nr ? S.res[j] : kNone;
        if (sorted_out)
            for (int j = lane; j < cstride; j += 32) sorted_out[(size_t)i * cstride + j] = j < nv ? S.ci[j] : kNone;
        if (lane == 0) out_cnt[i] = nr;
        __syncwarp();
    }
}

// The most candidates per node for which one warp per node is the better form (or
// as good, depending on M and fill). Measured on GB300, one warp per node / one
// CTA per node, us, M = 16, no fill, 40,000 nodes: d = 200: 8 candidates 98 / 299,
// 16 449 / 661, 24 744 / 956, 32 1,021 / 1,072, 40 1,374 / 1,260; d = 64: 32 740 / 761,
// 40 1,020 / 948; d = 512: 24 1,296 / 1,873, 40 2,466 / 2,521, 48 2,993 / 2,642; d =
// 1024: 8 523 / 854, 16 1,485 / 1,431, 24 2,814 / 2,029 (M = 32 with fill: 16 and
// 20 candidates 1.16 to 1.3 times as fast for 520 to 1,024 columns). Fewer nodes than
// warps that run at once are better spread over CTAs: at 100 nodes a CTA is faster
// from 12 candidates on (d = 200, 24 candidates 36 / 22), at 800 from 32, at 2,000 from
// 32 (d = 128, 68 / 53) or 16 (d = 1024, 104 / 85).
template <int NCH>
int acquire_few_most(int64_t nx, int sms) {
    if (nx < 4 * (int64_t)sms) return 8;
    if (nx < 8 * (int64_t)sms) return NCH >= 8 ? 12 : 24;
    if (nx < 16 * (int64_t)sms) return NCH >= 8 ? 12 : NCH >= 2 ? 32 : 24;
    return NCH >= 8 ? 20 : NCH >= 4 ? kAcqFewCand : 32;
}

template <int NCH>
cudaError_t launch_acquire(const float *X, int64_t n, int d, const uint32_t *xs, int64_t nx, const uint32_t *cand,
                           int cstride, const int32_t *ncand, int M, int fill, uint32_t *out, int32_t *out_cnt,
                           uint32_t *sorted_out, cudaStream_t s) {
    constexpr int W = AcqShape<NCH>::W;
    int dev = 0, sms = 0, per = 0;
    const auto fn = acquire_kernel<NCH>;
    int keycap = 2;
    while (keycap < cstride) keycap <<= 1;
    const int scap = std::min(M, kAcqRowBytes / (d * 4));
    const size_t smem = (size_t)scap * d * 4 + (size_t)keycap * 8;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && cstride <= acquire_few_most<NCH>(nx, sms)) {
        const int64_t few = std::min<int64_t>((nx + 3) / 4, (int64_t)sms * 16);
        acquire_few_kernel<NCH><<<(unsigned)few, 128, 0, s>>>(X, n, d, xs, nx, cand, cstride, ncand, M, fill, out,
                                                             out_cnt, sorted_out);
        return cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kAcqRowBytes + 8 * kAcqMaxCand);   // any launch's
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, 32 * W, smem);
    if (e != cudaSuccess) return e;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>(nx, (int64_t)sms * std::max(1, per)));
    fn<<<(unsigned)blocks, 32 * W, smem, s>>>(X, n, d, xs, nx, cand, cstride, ncand, M, fill, out, out_cnt,
                                              sorted_out, keycap, scap);
    return cudaGetLastError();
}

}  // namespace

cudaError_t acquire_launch(const float *X, int64_t n, int d, const uint32_t *xs, int64_t nx, const uint32_t *cand,
                           int cstride, const int32_t *ncand, int M, int fill, uint32_t *out, int32_t *out_cnt,
                           uint32_t *sorted_out, cudaStream_t s) {
    switch (search_nch(d)) {
        case 1: return launch_acquire<1>(X, n, d, xs, nx, cand, cstride, ncand, M, fill, out, out_cnt, sorted_out, s);
        case 2: return launch_acquire<2>(X, n, d, xs, nx, cand, cstride, ncand, M, fill, out, out_cnt, sorted_out, s);
        case 4: return launch_acquire<4>(X, n, d, xs, nx, cand, cstride, ncand, M, fill, out, out_cnt, sorted_out, s);
        default: return launch_acquire<8>(X, n, d, xs, nx, cand, cstride, ncand, M, fill, out, out_cnt, sorted_out, s);
    }
}

}  // namespace roar

using namespace roar;

extern "C" roar_status roar_acquire(const float *X, int64_t n, int32_t d, const uint32_t *xs, int64_t nx,
                                    const uint32_t *cand, int32_t cand_stride, const int32_t *ncand, int32_t M,
                                    int32_t fill, uint32_t *out, int32_t *out_cnt, uint32_t *sorted_out,
                                    void *stream) {
    if (n < 1 || n >= (int64_t)kIdMask || d < 4 || d % 4 != 0 || d > 1024 || nx < 0 || M < 1 || M > kAcqMaxM ||
        cand_stride < 0 || cand_stride > kAcqMaxCand) {
        set_error("roar_acquire: need n >= 1, d % 4 == 0 and 4 <= d <= 1024, 1 <= M <= 64, "
                  "0 <= cand_stride <= 1024");
        return ROAR_EINVAL;
    }
    if (nx == 0) return ROAR_OK;
    if (!X || !xs || !ncand || !out || !out_cnt || (cand_stride > 0 && !cand) || !aligned(X, 16)) {
        set_error("roar_acquire: bad pointer (X must be 16-byte aligned)");
        return ROAR_EINVAL;
    }
    cudaError_t e = acquire_launch(X, n, d, xs, nx, cand, cand_stride, ncand, M, fill ? 1 : 0, out, out_cnt,
                                   sorted_out, (cudaStream_t)stream);
    return e == cudaSuccess ? ROAR_OK : cuda_fail(e, "roar_acquire");
}

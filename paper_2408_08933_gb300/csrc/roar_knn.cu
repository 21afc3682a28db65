// Dense steps: reduced-precision copies of the base rows, and the exact
// k-nearest-neighbour search of many queries against the base set, which is
// the preprocessing step of RoarGraph's construction ("ground truths of the
// training queries", Sec. 4.2.1) and also yields the evaluation ground truth
// (Sec. 2.1.1).
//
// kNN pipeline per block of query rows:
//   1. BF16 copies of both sides (round to nearest even);
//   2. scores on the 5th-generation tensor cores with a fused running top-C
//      per row (roar_knn_tc.cu): no score matrix is written;
//   3. the C candidates are re-scored with exact FP32 dot products (the
//      search's fixed order) and the first kk in (distance, id) order are kept.
// With C > kk the BF16 rounding of step 2 only has to keep the true top-kk
// inside the top-C, which a margin of C - kk ranks makes near-certain; the
// returned distances are exact FP32 values.
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <atomic>
#include <cstdio>
#include <mutex>

#include "roar_knn_tc.cuh"

namespace roar {

roar_status cuda_fail(cudaError_t e, const char *what);
void set_error(const char *msg);
bool aligned(const void *p, size_t a);

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

__device__ __forceinline__ bool less_entry(float da, uint32_t ia, float db, uint32_t ib) {
    return da < db || (da == db && ia < ib);
}

// One warp per row, any alignment. BF16: round to nearest even, scale 1.
__global__ void quantize_bf16_kernel(const float *__restrict__ X, int64_t n, int d,
                                     __nv_bfloat16 *__restrict__ out) {
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= n) return;
    const float *x = X + row * d;
    __nv_bfloat16 *o = out + row * d;
    for (int i = lane; i < d; i += 32) o[i] = __float2bfloat16_rn(x[i]);
}

// One warp per row, any alignment. FP8-E4M3: s = maxabs / 448 (IEEE division), code = E4M3(x / s)
// rounded to nearest even and saturated to +-448; an all-zero row gets s = 1.
__global__ void quantize_fp8_kernel(const float *__restrict__ X, int64_t n, int d,
                                    uint8_t *__restrict__ out, float *__restrict__ scales) {
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= n) return;
    const float *x = X + row * d;
    float m = 0.0f;
    for (int i = lane; i < d; i += 32) m = fmaxf(m, fabsf(x[i]));
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
    const float s = (m == 0.0f) ? 1.0f : __fdiv_rn(m, 448.0f);
    if (lane == 0) scales[row] = s;
    uint8_t *o = out + row * d;
    for (int i = lane; i < d; i += 32)
        o[i] = (uint8_t)__nv_cvt_float_to_fp8(__fdiv_rn(x[i], s), __NV_SATFINITE, __NV_E4M3);
}

// The same for 16-byte-aligned rows, bound by HBM: 16 bytes per lane and load, each
// element read once. Measured on GB300, 1M x 512 to FP8: 486 us (5.3 TB/s) with a
// second read of the row and one-byte stores, 363 us (7.0 TB/s) so.

__device__ __forceinline__ uint2 to_bf16x4(const float4 &v) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    return make_uint2(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b));
}

// BF16, m 16-byte chunks: rows need no padding, so they are one array and no lane
// idles at a row's end. (Lanes dealt to rows, 32 at most, with loads that leave
// nothing in the caches: 300,000 x 200 67 us, x 256 77, x 512 145, x 1,024 284;
// an element per lane and load 87, 69, 131, 259; so 53, 67, 130 and 255.)
__global__ void __launch_bounds__(256) quantize_bf16_flat_kernel(const float4 *__restrict__ X, int64_t m,
                                                                 uint2 *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * 512 + threadIdx.x, j = i + 256;
    float4 v, w;
    if (i < m) v = __ldg(X + i);
    if (j < m) w = __ldg(X + j);
    if (i < m) out[i] = to_bf16x4(v);
    if (j < m) out[j] = to_bf16x4(w);
}

// BF16 rows of d4 16-byte chunks into rows of dp4 8-byte ones, zeros past d4: LPR
// lanes per row (a power of two, so narrow rows fill the warp too).
template <int LPR>
__global__ void __launch_bounds__(256) quantize_bf16_vec_kernel(const float4 *__restrict__ X, int64_t n, int d4, int dp4,
                                                                uint2 *__restrict__ out) {
    const int64_t row = (int64_t)blockIdx.x * (256 / LPR) + threadIdx.x / LPR;
    if (row >= n) return;
    const float4 *x = X + row * d4;
    uint2 *o = out + row * dp4;
#pragma unroll 4
    for (int c = threadIdx.x % LPR; c < dp4; c += LPR) {
        const float4 v = c < d4 ? __ldcs(x + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        o[c] = to_bf16x4(v);
    }
}

// FP8 rows of d4 chunks on LPR lanes, at most LPR * NCH chunks, held in registers
// between the row's maximum and the codes.
template <int LPR, int NCH>
__global__ void __launch_bounds__(256) quantize_fp8_vec_kernel(const float4 *__restrict__ X, int64_t n, int d4,
                                                               uint32_t *__restrict__ out, float *__restrict__ scales) {
    const int64_t row = (int64_t)blockIdx.x * (256 / LPR) + threadIdx.x / LPR;
    const int l = threadIdx.x % LPR;
    float4 v[NCH];
    float m = 0.0f;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        const int ch = l + LPR * c;
        v[c] = row < n && ch < d4 ? __ldcs(X + row * d4 + ch) : make_float4(0.f, 0.f, 0.f, 0.f);
        m = fmaxf(m, fmaxf(fmaxf(fabsf(v[c].x), fabsf(v[c].y)), fmaxf(fabsf(v[c].z), fabsf(v[c].w))));
    }
#pragma unroll
    for (int o = LPR / 2; o >= 1; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
    if (row >= n) return;
    const float s = (m == 0.0f) ? 1.0f : __fdiv_rn(m, 448.0f);
    if (l == 0) scales[row] = s;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        const int ch = l + LPR * c;
        if (ch >= d4) break;
        const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(__fdiv_rn(v[c].x, s), __fdiv_rn(v[c].y, s)),
                                                     __NV_SATFINITE, __NV_E4M3);
        const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(__fdiv_rn(v[c].z, s), __fdiv_rn(v[c].w, s)),
                                                     __NV_SATFINITE, __NV_E4M3);
        out[row * d4 + ch] = lo | (hi << 16);
    }
}

// Exact FP32 re-scoring of C candidates per query row, then the first kk in
// (distance, id) order. One warp per row; dot products use the fixed order
// (element i on lane (i >> 2) & 31, fmaf, xor butterfly).
template <int C>
__global__ void rescore_kernel(const float *__restrict__ T, int64_t nt, const float *__restrict__ X,
                               int d, const uint32_t *__restrict__ cand, int kk,
                               uint32_t *__restrict__ ids, float *__restrict__ dist, const int *__restrict__ err) {
    __shared__ float sd[4][C];
    __shared__ uint32_t si[4][C];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * 4 + w;
    if (row >= nt || *err) return;   // after a timeout the candidates were not written
    const int d4 = d >> 2;   // d <= 512: at most 4 chunks per lane
    const float4 *q4 = reinterpret_cast<const float4 *>(T + row * d);
    float4 qv[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int ch = lane + 32 * c;
        qv[c] = ch < d4 ? __ldg(q4 + ch) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    // G candidates at a time, so that their row loads are in flight together;
    // each candidate's sum keeps its own order (chunks in increasing index).
    constexpr int G = 4;
    static_assert(C % G == 0, "candidates come in groups of G");
    for (int j0 = 0; j0 < C; j0 += G) {
        uint32_t u[G];
        float s[G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            u[g] = cand[row * C + j0 + g];
            s[g] = 0.0f;
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int ch = lane + 32 * c;
            if (ch >= d4) break;
            float4 b[G];
#pragma unroll
            for (int g = 0; g < G; ++g)
                b[g] = u[g] != 0xFFFFFFFFu ? __ldg(reinterpret_cast<const float4 *>(X + (int64_t)u[g] * d) + ch)
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int g = 0; g < G; ++g) {
                s[g] = fmaf(qv[c].x, b[g].x, s[g]);
                s[g] = fmaf(qv[c].y, b[g].y, s[g]);
                s[g] = fmaf(qv[c].z, b[g].z, s[g]);
                s[g] = fmaf(qv[c].w, b[g].w, s[g]);
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) s[g] = s[g] + __shfl_xor_sync(kFull, s[g], o);
            if (lane == 0) {
                sd[w][j0 + g] = (u[g] != 0xFFFFFFFFu) ? -s[g] : __int_as_float(0x7f800000);
                si[w][j0 + g] = u[g];
            }
        }
    }
    __syncwarp();
    for (int j = lane; j < C; j += 32) {
        const float dj = sd[w][j];
        const uint32_t ij = si[w][j];
        int r = 0;
        for (int x = 0; x < C; ++x) r += less_entry(sd[w][x], si[w][x], dj, ij) ? 1 : 0;
        if (r < kk) {
            ids[row * kk + r] = ij;
            dist[row * kk + r] = dj;
        }
    }
}

}  // namespace

// BF16 copy in rows of dp >= d columns (zeros past d); X 16-byte and out 8-byte aligned.
static cudaError_t quantize_bf16_vec(const float *X, int64_t n, int d, int dp, void *out, cudaStream_t s) {
    const int d4 = d / 4, dp4 = dp / 4;
    const float4 *x = reinterpret_cast<const float4 *>(X);
    uint2 *o = reinterpret_cast<uint2 *>(out);
    if (dp == d) quantize_bf16_flat_kernel<<<(unsigned)((n * d4 + 511) / 512), 256, 0, s>>>(x, n * d4, o);
    else if (dp4 <= 8) quantize_bf16_vec_kernel<8><<<(unsigned)((n + 31) / 32), 256, 0, s>>>(x, n, d4, dp4, o);
    else if (dp4 <= 16) quantize_bf16_vec_kernel<16><<<(unsigned)((n + 15) / 16), 256, 0, s>>>(x, n, d4, dp4, o);
    else quantize_bf16_vec_kernel<32><<<(unsigned)((n + 7) / 8), 256, 0, s>>>(x, n, d4, dp4, o);
    return cudaGetLastError();
}

static cudaError_t quantize_fp8_vec(const float *X, int64_t n, int d, void *out, float *scales, cudaStream_t s) {
    const int d4 = d / 4;
    const float4 *x = reinterpret_cast<const float4 *>(X);
    uint32_t *o = reinterpret_cast<uint32_t *>(out);
    const unsigned rows8 = (unsigned)((n + 7) / 8);
    if (d4 <= 8) quantize_fp8_vec_kernel<8, 1><<<(unsigned)((n + 31) / 32), 256, 0, s>>>(x, n, d4, o, scales);
    else if (d4 <= 16) quantize_fp8_vec_kernel<16, 1><<<(unsigned)((n + 15) / 16), 256, 0, s>>>(x, n, d4, o, scales);
    else if (d4 <= 32) quantize_fp8_vec_kernel<32, 1><<<rows8, 256, 0, s>>>(x, n, d4, o, scales);
    else if (d4 <= 64) quantize_fp8_vec_kernel<32, 2><<<rows8, 256, 0, s>>>(x, n, d4, o, scales);
    else if (d4 <= 128) quantize_fp8_vec_kernel<32, 4><<<rows8, 256, 0, s>>>(x, n, d4, o, scales);
    else quantize_fp8_vec_kernel<32, 8><<<rows8, 256, 0, s>>>(x, n, d4, o, scales);
    return cudaGetLastError();
}

roar_status quantize_bf16_pad(const float *X, int64_t n, int d, int dp, void *out, cudaStream_t s) {
    const cudaError_t e = quantize_bf16_vec(X, n, d, dp, out, s);
    return e == cudaSuccess ? ROAR_OK : cuda_fail(e, "quantize_bf16");
}

}  // namespace roar

using namespace roar;

extern "C" roar_status roar_quantize(const float *X, int64_t n, int32_t d, roar_dtype dtype,
                                     void *out, float *scales, void *stream) {
    if (n < 0 || d < 4 || d % 4 != 0 || d > 1024) return ROAR_EINVAL;
    if (n == 0) return ROAR_OK;
    if (!X || !out) return ROAR_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t blocks = (n + 7) / 8;
    if (blocks > 0x7FFFFFFF) return ROAR_EINVAL;
    cudaError_t e = cudaSuccess;
    // Rows are multiples of 16 bytes, so the first one's alignment is every one's.
    if (dtype == ROAR_BF16 && aligned(X, 16) && aligned(out, 8)) {
        e = quantize_bf16_vec(X, n, d, d, out, s);
    } else if (dtype == ROAR_BF16) {
        quantize_bf16_kernel<<<(unsigned)blocks, 256, 0, s>>>(X, n, d, (__nv_bfloat16 *)out);
    } else if (dtype == ROAR_FP8_E4M3) {
        if (!scales) return ROAR_EINVAL;
        if (aligned(X, 16) && aligned(out, 4)) e = quantize_fp8_vec(X, n, d, out, scales, s);
        else quantize_fp8_kernel<<<(unsigned)blocks, 256, 0, s>>>(X, n, d, (uint8_t *)out, scales);
    } else {
        return ROAR_EINVAL;
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    return e == cudaSuccess ? ROAR_OK : cuda_fail(e, "roar_quantize");
}

namespace roar {
// Wall-time limit of each bounded wait in the tensor-core kernel: 2 s by
// default, far above any legitimate wait there.
constexpr int64_t kKnnWaitDefaultNs = 2000000000ll;
static std::atomic<int64_t> g_knn_wait_ns{kKnnWaitDefaultNs};
}  // namespace roar

extern "C" roar_status roar_knn_set_wait_limit_ns(int64_t ns) {
    g_knn_wait_ns.store(ns < 0 ? kKnnWaitDefaultNs : ns);
    return ROAR_OK;
}

namespace roar {
// A call whose buffers fit kKnnPoolKeep bytes takes them from a private
// stream-ordered pool per device, which keeps at most that much between calls:
// it then allocates nothing, while cudaMalloc and cudaFree of five buffers took
// longer than its kernels (GB300, 1,000 x 10,000 x 64: 680 us per call, 333 us so).
// Larger calls allocate and free for themselves: pool memory above the limit is
// given back at every synchronisation, and mapping it again took longer than
// cudaMalloc (10,000 x 1M x 200: 7.24 ms from the pool, 7.05 ms without).
constexpr uint64_t kKnnPoolKeep = 320ull << 20;   // a full grid's candidate buffers (239 MB) and small operands
constexpr int kMaxDevices = 128;
static std::mutex g_knn_pool_mu;
static cudaMemPool_t g_knn_pools[kMaxDevices] = {};
static cudaError_t knn_pool(cudaMemPool_t *pool) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_knn_pool_mu);
    if (!g_knn_pools[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        e = cudaMemPoolCreate(&p, &props);
        uint64_t keep = kKnnPoolKeep;
        if (e == cudaSuccess) e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
        if (e != cudaSuccess) {
            if (p) cudaMemPoolDestroy(p);
            return e;
        }
        g_knn_pools[dev] = p;
    }
    *pool = g_knn_pools[dev];
    return cudaSuccess;
}
// Gives back what the device's pool holds and no call is using.
void knn_pool_trim(int dev) {
    if (dev < 0 || dev >= kMaxDevices) return;
    std::lock_guard<std::mutex> lock(g_knn_pool_mu);
    if (g_knn_pools[dev]) cudaMemPoolTrimTo(g_knn_pools[dev], 0);
}
}  // namespace roar

extern "C" roar_status roar_knn_release(void) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "roar_knn_release");
    knn_pool_trim(dev);
    return ROAR_OK;
}

extern "C" roar_status roar_knn(const float *T, int64_t nt, const float *X, int64_t n, int32_t d,
                                int32_t kk, uint32_t *ids, float *dist, void *stream) {
    constexpr int C = 128;
    if (nt < 0 || n < 1 || n >= 0x7FFFFFFF || d < 8 || d % 8 != 0 || d > 512 || kk < 1 || kk > C ||
        kk > n) {
        set_error("roar_knn: need n >= kk, 1 <= kk <= 128, d % 8 == 0, 8 <= d <= 512");
        return ROAR_EINVAL;
    }
    if (nt == 0) return ROAR_OK;
    if (!T || !X || !ids || !dist || !aligned(T, 16) || !aligned(X, 16)) return ROAR_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int dp = (d + 15) / 16 * 16;   // BF16 operand rows padded to whole MMA steps of K
    // Query rows per launch: whole waves of the kernel, about 131,072 at most.
    const int64_t wave = knn_tc_wave_rows(d);
    const int64_t RB = std::min<int64_t>(nt, std::max<int64_t>(wave, 131072 / wave * wave));
    KnnPlan whole, rest;   // of a launch of RB rows and of the last one
    __nv_bfloat16 *t16 = nullptr, *x16 = nullptr;
    void *scratch = nullptr, *lists = nullptr;
    uint32_t *cand = nullptr;
    int *err = nullptr;
    const uint64_t wait_ns = (uint64_t)g_knn_wait_ns.load();
    roar_status rc = ROAR_OK;
    int herr = 0;
    cudaError_t e = knn_tc_plan(RB, n, d, &whole);
    if (e == cudaSuccess) e = knn_tc_plan(nt % RB ? nt % RB : RB, n, d, &rest);
    if (e != cudaSuccess) return cuda_fail(e, "roar_knn: launch plan");
    const size_t lists_bytes = std::max(whole.lists_bytes, rest.lists_bytes);
    const size_t sizes[6] = {(size_t)nt * dp * 2, (size_t)n * dp * 2, std::max(whole.scratch_bytes, rest.scratch_bytes),
                             lists_bytes, (size_t)RB * C * 4, sizeof(int)};
    void **const buffers[6] = {(void **)&t16, (void **)&x16, &scratch, &lists, (void **)&cand, (void **)&err};
    size_t total = 0;
    for (size_t b : sizes) total += b;
    const bool pooled = total <= kKnnPoolKeep;
    cudaMemPool_t pool = nullptr;
    if (pooled) e = knn_pool(&pool);
    for (int i = 0; i < 6 && e == cudaSuccess; ++i)
        if (sizes[i]) e = pooled ? cudaMallocFromPoolAsync(buffers[i], sizes[i], pool, s) : cudaMalloc(buffers[i], sizes[i]);
    if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, sizeof(int), s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("roar_knn: out of device memory");
        rc = ROAR_ENOMEM;
        goto done;
    }
    if ((rc = quantize_bf16_pad(T, nt, d, dp, t16, s)) != ROAR_OK) goto done;
    if ((rc = quantize_bf16_pad(X, n, d, dp, x16, s)) != ROAR_OK) goto done;
    for (int64_t r0 = 0; r0 < nt; r0 += RB) {
        const int64_t rb = std::min(RB, nt - r0);
        e = knn_tc_launch(rb == RB ? whole : rest, t16 + r0 * dp, rb, x16, n, dp, scratch, lists, cand, err, wait_ns, s);
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "roar_knn: tensor-core scores");
            goto done;
        }
        rescore_kernel<C><<<(unsigned)((rb + 3) / 4), 128, 0, s>>>(T + r0 * d, rb, X, d, cand, kk,
                                                                 ids + r0 * kk, dist + r0 * kk, err);
        e = cudaGetLastError();
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "roar_knn: rescore");
            goto done;
        }
    }
    e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) rc = cuda_fail(e, "roar_knn");
    else if (herr) {
        set_error("roar_knn: a tensor-core wait timed out");
        rc = ROAR_ETIMEOUT;
    }
done:
    for (void **p : buffers) {
        if (*p && pooled) cudaFreeAsync(*p, s);
        else cudaFree(*p);
    }
    return rc;
}

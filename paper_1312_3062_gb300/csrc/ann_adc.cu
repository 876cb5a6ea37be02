// ann_adc.cu -- Graph-D-ADC (Sec. 5.4) on sm_103a: the method as the coarse
// quantizer of an inverted file whose residuals are product-quantized.
//
//  - pq_encode_kernel: the code of every reference, one thread per
//    (reference, part); the part's codebook sits in shared memory and every
//    lane of a warp reads the same codeword (broadcast).
//  - adc_rerank_kernel: one CTA per query.  The visited lists (the coarse
//    search's result, in order) are taken two at a time: the CTA builds the
//    asymmetric-distance tables of both q - c against every codeword in shared
//    memory, reading each codeword once, then keys the lists' members by m
//    table lookups, a member's code being one load.  A candidate enters a
//    pending buffer only when it beats the current T-th best; when the buffer
//    fills, a bisection over the (key, id) values finds the T-th of it and the
//    rest is dropped.  Only the final T are sorted.  The result, the T smallest
//    (key, id) of all candidates, does not depend on the order in which
//    candidates arrive.
//    Bound by the tables' float32 issue (m x ks x d / m x 3 operations a list,
//    two at a time in one instruction) and the lookups' shared-memory bank
//    conflicts.  A bitonic sort of the whole buffer at every merge, codes read
//    byte by byte and one list's table at a time took 6.08 ms for 10,000
//    queries, m = 16, ks = 256, L = 10,000; this takes 2.04 ms.
// Codes and keys are decided in float32 (the precision of the lookup tables
// of asymmetric distance computation) with every operation rounded: each
// distance is within (dp + m + 8) * 2^-24 * sum_t (|a_t| + |w_t|)^2 of the
// real one (a = x - c or q - c, w the codeword), so a code or a rank differs
// from the real-valued one of Sec. 5.4 only at near-ties of that size.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "ann_device.cuh"
#include "ann_internal.cuh"

namespace ann {
namespace {

constexpr int ENC_THREADS = 128;
constexpr int ENC_MAX_DP = 32;       // dims per part held in registers
constexpr int RR_THREADS = 256;
constexpr int RR_PER_THREAD = 4;
constexpr int RR_CHUNK = RR_THREADS * RR_PER_THREAD;  // candidates keyed per pass
constexpr int RR_BUF = 2048;         // candidates kept, at least T + RR_CHUNK
constexpr int RR_MAX_T = 128;

template <int DT>
__device__ __forceinline__ float elem(const void *X, int64_t i) {
    if (DT == ANN_U8) return (float)((const uint8_t *)X)[i];
    return ((const float *)X)[i];
}

template <int DT>
__global__ void __launch_bounds__(ENC_THREADS) pq_encode_kernel(const void *__restrict__ X, int64_t N, int d,
                                                                const float *__restrict__ centers, int64_t K,
                                                                const int32_t *__restrict__ assign, int m, int ks,
                                                                const float *__restrict__ codebooks,
                                                                uint8_t *__restrict__ codes) {
    extern __shared__ float cbs[];  // part j's codebook, ks * dp
    const int j = blockIdx.y;
    const int dp = d / m;
    for (int e = threadIdx.x; e < ks * dp; e += blockDim.x) cbs[e] = codebooks[(int64_t)j * ks * dp + e];
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int64_t a = assign[i];
    if (a < 0 || a >= K) {  // no such list: code 0 (rejected on the host for valid inputs)
        codes[i * m + j] = 0;
        return;
    }
    float r[ENC_MAX_DP];
#pragma unroll
    for (int t = 0; t < ENC_MAX_DP; t++)
        if (t < dp) r[t] = __fsub_rn(elem<DT>(X, i * d + j * dp + t), centers[a * d + j * dp + t]);
    float best = INFINITY;
    int arg = 0;
    for (int k = 0; k < ks; k++) {
        const float *w = cbs + k * dp;
        float s = 0.0f;
#pragma unroll
        for (int t = 0; t < ENC_MAX_DP; t++)
            if (t < dp) {
                const float e = __fsub_rn(r[t], w[t]);
                s = __fadd_rn(s, __fmul_rn(e, e));
            }
        if (s < best) {
            best = s;
            arg = k;
        }
    }
    codes[i * m + j] = (uint8_t)arg;
}

// The products are single ones: a two-wide multiply and the two-wide add after
// it came back as one fused operation, without the product's rounding.
__device__ __forceinline__ uint64_t square2(uint64_t a) {
    float x, y;
    unpack2(a, x, y);
    return pack2(__fmul_rn(x, x), __fmul_rn(y, y));
}

// Keep T of the n values in buf (n > T), the smallest ones, in any order: the
// T-th by bisection, every thread counting its own values, then compaction (of
// values equal to the T-th, from a list visited twice, as many as fit).
// Returns the T-th value or, when exactly T lie below it, one before the next.
__device__ uint64_t cta_keep_smallest(uint64_t *buf, unsigned n, int T, unsigned *s_n) {
    constexpr int PER = RR_BUF / RR_THREADS, WARPS = RR_THREADS / 32;
    uint64_t e[PER];
    uint64_t lo = ~0ull, hi = 0;  // of the values
#pragma unroll
    for (int i = 0; i < PER; i++) {
        const unsigned at = threadIdx.x + RR_THREADS * i;
        e[i] = at < n ? buf[at] : ~0ull;
        if (at < n) {
            lo = e[i] < lo ? e[i] : lo;
            hi = e[i] > hi ? e[i] : hi;
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        const uint64_t l = __shfl_xor_sync(0xffffffffu, lo, off), h = __shfl_xor_sync(0xffffffffu, hi, off);
        lo = l < lo ? l : lo;
        hi = h > hi ? h : hi;
    }
    __syncthreads();  // every value is in a register: the buffer serves the warps' results
    int *s_sum = (int *)(buf + 2 * WARPS);
    if ((threadIdx.x & 31) == 0) {
        buf[threadIdx.x >> 5] = lo;
        buf[WARPS + (threadIdx.x >> 5)] = hi;
    }
    __syncthreads();
    for (int i = 0; i < WARPS; i++) {
        lo = buf[i] < lo ? buf[i] : lo;
        hi = buf[WARPS + i] > hi ? buf[WARPS + i] : hi;
    }
    while (lo < hi) {  // at or below hi there are at least T values
        const uint64_t mid = lo + (hi - lo) / 2;
        int c = 0;
#pragma unroll
        for (int i = 0; i < PER; i++) c += e[i] <= mid;
        c = __reduce_add_sync(0xffffffffu, c);
        __syncthreads();  // the last sums have been read
        if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = c;
        __syncthreads();
        c = 0;
#pragma unroll
        for (int i = 0; i < WARPS; i++) c += s_sum[i];
        if (c >= T) hi = mid;
        else lo = mid + 1;
        if (c == T) break;
    }
    __syncthreads();
    if (threadIdx.x == 0) *s_n = 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; i++)
        if (e[i] < hi) buf[atomicAdd(s_n, 1u)] = e[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; i++)
        if (e[i] == hi) {
            const unsigned at = atomicAdd(s_n, 1u);
            if (at < (unsigned)T) buf[at] = e[i];
        }
    __syncthreads();
    if (threadIdx.x == 0) *s_n = (unsigned)T;
    __syncthreads();
    return hi;
}

// m bytes of a code, CB (16, 8, 4 or 1) at a time, each as a lookup added to key
template <int CB>
__device__ __forceinline__ float adc_key(const uint8_t *cx, int m, const float *table, int ks) {
    float key = 0.0f;
    for (int j = 0; j < m; j += CB) {
        uint32_t w[CB >= 4 ? CB / 4 : 1];
        if (CB == 16) {
            const uint4 v = __ldg((const uint4 *)(cx + j));
            w[0] = v.x, w[1 % (CB / 4 + (CB < 4))] = v.y, w[2 % (CB / 4 + (CB < 4))] = v.z, w[3 % (CB / 4 + (CB < 4))] = v.w;
        } else if (CB == 8) {
            const uint2 v = __ldg((const uint2 *)(cx + j));
            w[0] = v.x, w[1 % (CB / 4 + (CB < 4))] = v.y;
        } else if (CB == 4) {
            w[0] = __ldg((const uint32_t *)(cx + j));
        } else {
            w[0] = cx[j];
        }
#pragma unroll
        for (int i = 0; i < CB; i++) key = __fadd_rn(key, table[(j + i) * ks + ((w[i / 4] >> (8 * (i & 3))) & 255u)]);
    }
    return key;
}

// NL lists at a time (their tables side by side); CB bytes of a code per load
template <int NL, int CB>
__global__ void __launch_bounds__(RR_THREADS) adc_rerank_kernel(
    const float *__restrict__ Q, int d, const int32_t *__restrict__ lists, int w, const int64_t *__restrict__ offsets,
    int64_t K, const int32_t *__restrict__ members, const float *__restrict__ centers,
    const uint8_t *__restrict__ codes, int m, int ks, const float *__restrict__ codebooks, int64_t L, int T,
    int32_t *__restrict__ out_ids, float *__restrict__ out_keys, int64_t *__restrict__ out_seen) {
    extern __shared__ __align__(16) uint8_t sm[];
    uint64_t *buf = (uint64_t *)sm;                            // RR_BUF candidates
    float *table = (float *)(sm + sizeof(uint64_t) * RR_BUF);  // NL x m * ks
    float *rq = table + (NL * m * ks + 3) / 4 * 4;             // NL x d: q - c of the current lists
    __shared__ unsigned s_n;
    const int64_t b = blockIdx.x;
    const float *q = Q + b * d;
    const int dp = d / m;
    if (threadIdx.x == 0) s_n = 0;
    uint64_t thr = ~0ull;  // a candidate has to be below it
    int64_t seen = 0;
    int li = 0;
    while (li < w && seen < L) {
        // the next NL valid lists, in order (the same in every thread)
        int64_t cur[NL];
        int nl = 0;
        while (li < w && nl < NL) {
            const int64_t c = lists[b * w + li++];
            if (c >= 0 && c < K) cur[nl++] = c;
        }
        if (nl == 0) break;
#pragma unroll
        for (int l = 0; l < NL; l++)
            if (l < nl)
                for (int t = threadIdx.x; t < d; t += RR_THREADS)
                    rq[l * d + t] = __fsub_rn(q[t], centers[cur[l] * d + t]);
        __syncthreads();
        for (int e = threadIdx.x; e < m * ks; e += RR_THREADS) {
            const int j = e / ks;
            const float *cw = codebooks + (int64_t)e * dp;
            const float *r0 = rq + j * dp;
            uint64_t s2 = 0;  // two lists' sums
            if ((dp & 3) == 0) {
                // the codeword as 16-byte loads; the same operations in the same order
                for (int t = 0; t < dp; t += 4) {
                    const float4 w4 = __ldg((const float4 *)(cw + t)), a4 = *(const float4 *)(r0 + t);
                    const float4 b4 = NL == 2 ? *(const float4 *)(r0 + d + t) : a4;
                    const float ww[4] = {w4.x, w4.y, w4.z, w4.w}, ra[4] = {a4.x, a4.y, a4.z, a4.w};
                    const float rb[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const uint64_t ee = sub2(pack2(ra[u], rb[u]), pack2(ww[u], ww[u]));
                        s2 = add2(s2, square2(ee));
                    }
                }
            } else {
                for (int t = 0; t < dp; t++) {
                    const float wt = __ldg(cw + t);
                    const uint64_t ee = sub2(pack2(r0[t], NL == 2 ? r0[d + t] : 0.f), pack2(wt, wt));
                    s2 = add2(s2, square2(ee));
                }
            }
            table[e] = __uint_as_float((uint32_t)s2);
            if (NL == 2) table[m * ks + e] = __uint_as_float((uint32_t)(s2 >> 32));
        }
        __syncthreads();
#pragma unroll
        for (int l = 0; l < NL; l++) {
            if (l >= nl || seen >= L) continue;  // uniform
            const int64_t lo = offsets[cur[l]];
            const int64_t size = offsets[cur[l] + 1] - lo;
            const int64_t take = size < L - seen ? size : L - seen;
            const float *tab = table + l * m * ks;
            for (int64_t base = 0; base < take; base += RR_CHUNK) {
#pragma unroll
                for (int u = 0; u < RR_PER_THREAD; u++) {
                    const int64_t p = base + u * RR_THREADS + threadIdx.x;
                    if (p < take) {
                        const int32_t x = __ldg(members + lo + p);
                        const float key = adc_key<CB>(codes + (int64_t)x * m, m, tab, ks);
                        const uint64_t v = ((uint64_t)__float_as_uint(key) << 32) | (uint32_t)x;
                        if (v < thr) buf[atomicAdd(&s_n, 1u)] = v;
                    }
                }
                __syncthreads();
                // every thread takes the count of this chunk into a register, and
                // no thread may add to it for the next chunk before all have read
                // it, so the decision is the same in every thread
                const unsigned n = s_n;
                __syncthreads();
                // room for a whole chunk, and a limit as soon as there are T
                if (n > RR_BUF - RR_CHUNK || (thr == ~0ull && n > (unsigned)(2 * T)))
                    if (n > (unsigned)T) thr = cta_keep_smallest(buf, n, T, &s_n);
            }
            seen += take;
        }
        __syncthreads();  // the tables are rebuilt for the next lists
    }
    __syncthreads();
    unsigned n = s_n;
    if (n > (unsigned)T) {
        cta_keep_smallest(buf, n, T, &s_n);
        n = (unsigned)T;
    }
    // the final T <= 128 in order, by one warp
    if (threadIdx.x < 32) {
        uint64_t v[RR_MAX_T / 32];
#pragma unroll
        for (int i = 0; i < RR_MAX_T / 32; i++) {
            const unsigned at = threadIdx.x * (RR_MAX_T / 32) + i;
            v[i] = at < n ? buf[at] : ~0ull;
        }
        reg_bitonic_sort<RR_MAX_T / 32>(v);
#pragma unroll
        for (int i = 0; i < RR_MAX_T / 32; i++) {
            const int r = threadIdx.x * (RR_MAX_T / 32) + i;
            if (r < T) {
                out_ids[b * T + r] = v[i] == ~0ull ? -1 : (int32_t)(uint32_t)v[i];
                if (out_keys) out_keys[b * T + r] = v[i] == ~0ull ? INFINITY : __uint_as_float((uint32_t)(v[i] >> 32));
            }
        }
    }
    if (out_seen && threadIdx.x == 0) out_seen[b] = seen;
}

}  // namespace
}  // namespace ann

extern "C" int ann_pq_encode(const void *data, int dtype, int64_t N, int32_t d, const float *centers, int64_t K,
                             const int32_t *assign, int32_t m, int32_t ks, const float *codebooks, uint8_t *codes,
                             void *stream) {
    using namespace ann;
    ANN_ARG(dtype == ANN_U8 || dtype == ANN_F32, "dtype must be ANN_U8 or ANN_F32");
    ANN_ARG(N >= 0 && N < (1ll << 31), "N out of range");
    ANN_ARG(m >= 1 && m <= 65535 && d >= m && d % m == 0, "d must be a positive multiple of m");
    ANN_ARG(d / m <= ENC_MAX_DP, "at most 32 dims per part");
    ANN_ARG(ks >= 1 && ks <= 256, "ks must be in [1, 256]");
    ANN_ARG(K >= 1, "K must be >= 1");
    ANN_ARG(N == 0 || (data && centers && assign && codebooks && codes), "null pointer");
    if (N == 0) return ANN_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t smem = sizeof(float) * (size_t)ks * (size_t)(d / m);
    dim3 grid((unsigned)((N + ENC_THREADS - 1) / ENC_THREADS), (unsigned)m);
    if (dtype == ANN_U8)
        pq_encode_kernel<ANN_U8><<<grid, ENC_THREADS, smem, s>>>(data, N, d, centers, K, assign, m, ks,
                                                                 codebooks, codes);
    else
        pq_encode_kernel<ANN_F32><<<grid, ENC_THREADS, smem, s>>>(data, N, d, centers, K, assign, m, ks,
                                                                  codebooks, codes);
    ANN_CUDA(cudaGetLastError());
    return ANN_OK;
}

extern "C" int ann_adc_rerank(const float *queries, int64_t nq, int32_t d, const int32_t *lists, int32_t w,
                              const int64_t *offsets, int64_t K, const int32_t *members, const float *centers,
                              const uint8_t *codes, int32_t m, int32_t ks, const float *codebooks, int64_t L,
                              int32_t T, int32_t *out_ids, float *out_keys, int64_t *out_seen, void *stream) {
    using namespace ann;
    ANN_ARG(nq >= 0 && nq < (1ll << 31), "nq out of range");
    ANN_ARG(m >= 1 && m <= 64 && d >= m && d % m == 0, "d must be a multiple of m, m <= 64");
    ANN_ARG(ks >= 1 && ks <= 256, "ks must be in [1, 256]");
    ANN_ARG(T >= 1 && T <= RR_MAX_T, "T must be in [1, 128]");
    ANN_ARG(w >= 1 && K >= 1 && L >= 0, "w >= 1, K >= 1, L >= 0");
    ANN_ARG(nq == 0 || (queries && lists && offsets && members && centers && codes && codebooks && out_ids),
            "null pointer");
    if (nq == 0) return ANN_OK;
    int dev = 0, optin = 0;
    ANN_CUDA(cudaGetDevice(&dev));
    ANN_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    // what limits m * ks is one list's table beside the buffer
    auto bytes = [&](int nl) {
        return sizeof(uint64_t) * RR_BUF + sizeof(float) * (size_t)nl * ((size_t)m * (size_t)ks + (size_t)d);
    };
    ANN_ARG(bytes(1) + 64 <= (size_t)optin, "m * ks tables too large for shared memory");
    cudaStream_t s = (cudaStream_t)stream;
    // two lists' tables share the codeword loads while three CTAs still fit an SM
    const bool two = w > 1 && bytes(2) + 1024 <= (size_t)optin / 3;
    const size_t smem = bytes(two ? 2 : 1) + 16;  // the residuals start on a 16-byte boundary
    const uintptr_t ca = (uintptr_t)codes | (uintptr_t)m;  // alignment of every code
    auto run = [&](auto kernel) -> int {
        ANN_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kernel<<<(unsigned)nq, RR_THREADS, smem, s>>>(queries, d, lists, w, offsets, K, members, centers, codes, m, ks,
                                                      codebooks, L, T, out_ids, out_keys, out_seen);
        return ANN_OK;
    };
    int r;
    if ((ca & 15) == 0) r = two ? run(adc_rerank_kernel<2, 16>) : run(adc_rerank_kernel<1, 16>);
    else if ((ca & 7) == 0) r = two ? run(adc_rerank_kernel<2, 8>) : run(adc_rerank_kernel<1, 8>);
    else if ((ca & 3) == 0) r = two ? run(adc_rerank_kernel<2, 4>) : run(adc_rerank_kernel<1, 4>);
    else r = two ? run(adc_rerank_kernel<2, 1>) : run(adc_rerank_kernel<1, 1>);
    if (r != ANN_OK) return r;
    ANN_CUDA(cudaGetLastError());
    return ANN_OK;
}

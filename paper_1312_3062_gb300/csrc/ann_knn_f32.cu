// ann_knn_f32.cu -- exact k-NN of float32 rows (ground truth of Sec. 5.1 and
// the exact R-NN graph of Sec. 3.1 / Sec. 4.1) with the dot products on the
// tensor cores.
//
// Keys are the float32 nearest to the exact squared distance, exactly as in
// the SIMT kernel of ann_knn.cu.  The tensor cores only choose candidates:
//   1. Every row is split into bf16 parts, x = xh + xl + (dropped rest);
//      one bf16 tensor-core GEMM (cuBLAS, float32 accumulation) over the
//      concatenations [xh | xh | xl] and [qh | ql | qh] (inner length 3 d)
//      gives <q, x> ~ qh.xh + ql.xh + qh.xl for a tile of query rows against
//      every reference row; the approximate key a(x) = |q|^2 + |x|^2 - 2<q, x> is off
//      the exact one by at most eps(q) (a bound from the dropped terms and the
//      accumulation length, times a safety factor; see eps_row).
//   2. One pass over a query row's dot products finds a_k, the k-th smallest
//      a(x), and every x with a(x) <= a_k + 2 eps.  The k references with
//      a(x) <= a_k have exact keys <= a_k + eps, so the true k-th key is
//      <= a_k + eps, and every true neighbour y has
//      a(y) <= exact(y) + eps <= a_k + 2 eps: these x are the candidates (at
//      most kCap per row).
//   3. The candidates' exact keys (double-float, one rounding) decide the k
//      smallest by (key, id).
// Rows whose candidate list overflows are recomputed by the exact SIMT kernel.
#include <cublas_v2.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "ann_device.cuh"
#include "ann_internal.cuh"

namespace ann {

constexpr int kCap = 512;  // candidates per row kept for exact rescoring

static std::mutex g_blas_mu;
static cublasHandle_t g_blas[64];
static std::mutex g_blas_use[64];  // a handle's stream is set per call: one caller at a time

static int blas_handle(cublasHandle_t *out) {
    int dev = 0;
    ANN_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(ANN_ERR_ARG, "device ordinal out of range");
    std::lock_guard<std::mutex> g(g_blas_mu);
    if (!g_blas[dev]) {
        if (cublasCreate(&g_blas[dev]) != CUBLAS_STATUS_SUCCESS) return fail(ANN_ERR_CUDA, "cublasCreate failed");
    }
    *out = g_blas[dev];
    return ANN_OK;
}

// |x|^2 of every row in fp64 (products of floats are exact in fp64)
__global__ void norms_f32_kernel(const float *X, int64_t N, int d, double *n64, float *n32) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const float *row = X + i * d;
    double s = 0.0;
    for (int j = 0; j < d; j++) {
        const double v = (double)__ldg(row + j);
        s += v * v;
    }
    n64[i] = s;
    n32[i] = (float)s;
}

__global__ void max_norm_kernel(const double *n64, int64_t N, unsigned long long *out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) atomicMax(out, (unsigned long long)__double_as_longlong(n64[i]));  // non-negative doubles order as bits
}

// split x into bf16 xh = rn(x) and xl = rn(x - xh), |x - xh - xl| <= 2^-18 |x|,
// and store each row as three blocks of d: (h, h, l) for references,
// (h, l, h) for queries, so that one inner product of length 3 d pairs
// xh.qh + xh.ql + xl.qh
// (ld >= 3 d elements per row; what lies beyond 3 d and beyond `rows` is zero)
__global__ void split_bf16_kernel(const float *X, int64_t rows, int64_t rows_padded, int d, int ld, int query_order,
                                  __nv_bfloat16 *out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int w = d + (ld - 3 * d);  // one thread per value and one per padding element
    if (i >= rows_padded * w) return;
    const int64_t r = i / w;
    const int j = (int)(i - r * w);
    __nv_bfloat16 *o = out + r * ld;
    if (j >= d) {
        o[2 * d + j] = __float2bfloat16_rn(0.f);
        return;
    }
    const float v = r < rows ? X[r * d + j] : 0.f;
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    const __nv_bfloat16 l = __float2bfloat16_rn(v - __bfloat162float(h));
    o[j] = h;
    o[d + j] = query_order ? l : h;
    o[2 * d + j] = query_order ? h : l;
}

// Error bound of a(x) for query norm qn and the largest reference norm xn.
// Per coordinate the three products miss at most 3 * 2^-18 |q_i x_i| (the
// dropped ql.xl term and the rounding of ql, xl); the float32 sum of the
// n = 3 d + 16 rounded terms adds at most gamma_n times their magnitudes.
// All magnitudes sum to at most (qn + xn) / 2 (Cauchy-Schwarz), and the key
// doubles the dot product; the bound is then taken four times over.
__device__ __forceinline__ double eps_row(int d, double qn, double xn) {
    const double u = 1.0 / 16777216.0;
    const double n = 3.0 * d + 16.0;
    return 4.0 * (n * u / (1.0 - n * u) + 3.0 / 262144.0) * (qn + xn) + 1e-30;
}

__device__ __forceinline__ float approx_key(float dot, float qn, float xn) {
    const float a = qn + xn - 2.0f * dot;
    return a > 0.f ? a : 0.f;
}

constexpr int kScanThreads = 256;
constexpr int kScanVec = 4;     // 16-byte loads in flight per lane
constexpr int kScanBuf = 2048;  // a row's possible candidates during the pass
constexpr int kScanStep = 4 * kScanVec * kScanThreads;

// The smallest b with at least k of the CTA's values at or below it, values
// being bits of non-negative floats; below(b) counts this thread's.
template <class F>
__device__ __forceinline__ uint32_t cta_kth(int k, int *s_sum, F below) {
    uint32_t lo = 0, hi = 0x7f800000u;  // everything lies at or below hi, or there are fewer than k
    while (lo < hi) {
        const uint32_t mid = lo + (hi - lo) / 2;
        const int w = __reduce_add_sync(0xffffffffu, below(mid));
        __syncthreads();  // the last sum has been read
        if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = w;
        __syncthreads();
        int c = 0;
#pragma unroll
        for (int i = 0; i < kScanThreads / 32; i++) c += s_sum[i];
        if (c >= k) hi = mid;
        else lo = mid + 1;
    }
    return hi;
}

// One CTA per row.  The k-th smallest of the threads' minima over the first
// kScanStep columns is at least a_k; whatever lies within 2 eps of that goes
// to a shared buffer (about k N / kScanStep values of a row in random order).
// A buffer more than half full is cut to the k-th smallest value in it, plus
// 2 eps, which is again at least a_k + 2 eps; at the end that value is a_k.
// Should more than half a buffer lie that close, a_k comes from a bisection
// over the whole row (many equal rows: such rows mostly end in the exact scan).
// Bound by reading the dot products (HBM).  Two passes with 4-byte loads and
// warp-sorted lists, one for a_k and one for the candidates, took 33 ms for the
// 40 GB of 100,003 rows, one such pass 17.6 ms; this one takes 9.4 ms
// (4.3 TB/s).
__global__ void __launch_bounds__(kScanThreads)
    f32_scan_kernel(const float *D, int64_t ldD, int64_t q0, int64_t N, int d, const float *qn32, const float *rn32,
                    const double *qn64, const unsigned long long *xmax, int exclude_self, int k, uint32_t *cand,
                    int32_t *ncand) {
    __shared__ uint64_t buf[kScanBuf];
    __shared__ uint32_t s_cnt, s_out;
    __shared__ int s_sum[kScanThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t r = blockIdx.x, q = q0 + r;
    if (tid == 0) s_cnt = s_out = 0;
    const float qn = qn32[q];
    // limits in float32, rounded up: never fewer candidates than in fp64
    const float e2 = __double2float_ru(2.0 * eps_row(d, qn64[q], __longlong_as_double((long long)*xmax)));
    const float *row = D + r * ldD;
    const int64_t self = exclude_self ? q : -1;
    float lim = 0.f;
    bool full = false;
    for (int64_t c0 = 0; c0 < N && !full; c0 += kScanStep) {
        float a[kScanVec][4];
        const int64_t c1 = c0 + 4 * tid;
#pragma unroll
        for (int u = 0; u < kScanVec; u++) {
            const int64_t c = c1 + (int64_t)(4 * kScanThreads) * u;
            float4 dv = make_float4(0.f, 0.f, 0.f, 0.f), xv = dv;
            if (c < N) {  // rows of D and the norms are padded to multiples of four
                dv = __ldcs((const float4 *)(row + c));
                xv = __ldg((const float4 *)(rn32 + c));
            }
            a[u][0] = approx_key(dv.x, qn, xv.x);
            a[u][1] = approx_key(dv.y, qn, xv.y);
            a[u][2] = approx_key(dv.z, qn, xv.z);
            a[u][3] = approx_key(dv.w, qn, xv.w);
        }
        if (c0 + kScanStep > N || (self >= c0 && self < c0 + kScanStep))  // what is no neighbour
#pragma unroll
            for (int u = 0; u < kScanVec; u++)
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int64_t c = c1 + (int64_t)(4 * kScanThreads) * u + j;
                    if (c >= N || c == self) a[u][j] = __int_as_float(0x7fc00000);  // never at or below a limit
                }
        if (c0 == 0) {
            float mn = __int_as_float(0x7f800000);
#pragma unroll
            for (int u = 0; u < kScanVec; u++)
#pragma unroll
                for (int j = 0; j < 4; j++) mn = fminf(mn, a[u][j]);
            const uint32_t mb = __float_as_uint(mn);
            lim = __fadd_ru(__uint_as_float(cta_kth(k, s_sum, [&](uint32_t b) { return (int)(mb <= b); })), e2);
        }
        auto append = [&](float v, uint32_t id) {
            const uint32_t at = atomicAdd(&s_cnt, 1u);
            if (at < kScanBuf) buf[at] = ((uint64_t)__float_as_uint(v) << 32) | id;
        };
        // cut the buffer to the entries that can still matter
        auto refine = [&]() {
            uint64_t e[kScanBuf / kScanThreads];
            const uint32_t n = s_cnt;
#pragma unroll
            for (int i = 0; i < kScanBuf / kScanThreads; i++) {
                const uint32_t at = tid + kScanThreads * i;
                e[i] = at < n ? buf[at] : ~0ull;
            }
            const uint32_t kth = cta_kth(k, s_sum, [&](uint32_t b) {
                int c = 0;
#pragma unroll
                for (int i = 0; i < kScanBuf / kScanThreads; i++) c += (uint32_t)(e[i] >> 32) <= b;
                return c;
            });
            lim = __fadd_ru(__uint_as_float(kth), e2);
            __syncthreads();
            if (tid == 0) s_cnt = 0;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kScanBuf / kScanThreads; i++)
                if (e[i] != ~0ull && __uint_as_float((uint32_t)(e[i] >> 32)) <= lim) buf[atomicAdd(&s_cnt, 1u)] = e[i];
            __syncthreads();
            full = s_cnt > kScanBuf / 2;
        };
        const uint32_t before = s_cnt;  // at most half a buffer; every thread reads it before any adds to it
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kScanVec; u++) {
            const float mn = fminf(fminf(a[u][0], a[u][1]), fminf(a[u][2], a[u][3]));
            if (mn <= lim)
#pragma unroll
                for (int j = 0; j < 4; j++)
                    if (a[u][j] <= lim) append(a[u][j], (uint32_t)(c1 + (4 * kScanThreads) * u + j));
        }
        __syncthreads();
        if (s_cnt > kScanBuf) {
            // too many at once: take the step again a quarter at a time (a
            // quarter of a step fills half a buffer at most)
            __syncthreads();
            if (tid == 0) s_cnt = before;
            __syncthreads();
#pragma unroll
            for (int u = 0; u < kScanVec; u++) {
                if (full) break;
#pragma unroll
                for (int j = 0; j < 4; j++)
                    if (a[u][j] <= lim) append(a[u][j], (uint32_t)(c1 + (4 * kScanThreads) * u + j));
                __syncthreads();
                if (s_cnt > kScanBuf / 2) refine();
                __syncthreads();
            }
        } else if (s_cnt > kScanBuf / 2) {
            refine();
        }
        __syncthreads();
    }
    auto key_at = [&](int64_t c) { return approx_key(row[c], qn, rn32[c]); };
    uint32_t kth;
    if (!full) {
        uint64_t e[kScanBuf / kScanThreads];
        const uint32_t n = s_cnt;
#pragma unroll
        for (int i = 0; i < kScanBuf / kScanThreads; i++)
            e[i] = tid + kScanThreads * i < n ? buf[tid + kScanThreads * i] : ~0ull;
        kth = cta_kth(k, s_sum, [&](uint32_t b) {
            int c = 0;
#pragma unroll
            for (int i = 0; i < kScanBuf / kScanThreads; i++) c += (uint32_t)(e[i] >> 32) <= b;
            return c;
        });
    } else {
        kth = cta_kth(k, s_sum, [&](uint32_t b) {
            int n = 0;
            for (int64_t c = tid; c < N; c += kScanThreads) n += c != self && __float_as_uint(key_at(c)) <= b;
            return n;
        });
    }
    lim = __fadd_ru(__uint_as_float(kth), e2);
    uint32_t *out = cand + r * kCap;
    auto put = [&](uint32_t id) {
        const uint32_t at = atomicAdd(&s_out, 1u);
        if (at < kCap) out[at] = id;
    };
    __syncthreads();
    if (!full) {
        for (uint32_t i = tid; i < s_cnt; i += kScanThreads)
            if (__uint_as_float((uint32_t)(buf[i] >> 32)) <= lim) put((uint32_t)buf[i]);
    } else {
        for (int64_t c = tid; c < N; c += kScanThreads)
            if (c != self && key_at(c) <= lim) put((uint32_t)c);
    }
    __syncthreads();
    if (tid == 0) ncand[r] = (int32_t)s_out;
}

// Exact keys of the candidates and the k smallest by (key, id).  Rows whose
// candidates overflowed go to the fallback list.
// VEC: both row sets start on 16-byte boundaries (d is a multiple of 4).
template <bool VEC>
__global__ void f32_rescore_kernel(const float *X, const float *Qm, int d, int64_t rows, int64_t q0,
                                   const uint32_t *cand, const int32_t *ncand, int k, int32_t *out_ids,
                                   uint32_t *out_keys, int32_t *fb_rows, int32_t *fb_count) {
    const int lane = threadIdx.x & 31;
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (r >= rows) return;
    const int64_t q = q0 + r;
    const int nc = ncand[r];
    if (nc > kCap) {
        if (lane == 0) fb_rows[atomicAdd(fb_count, 1)] = (int32_t)q;
        return;
    }
    const float *qv = Qm + q * d;
    uint64_t mine = ~0ull;
    for (int b0 = 0; b0 < nc; b0 += 32) {
        const int i = b0 + lane;
        uint64_t v = ~0ull;
        if (i < nc) {
            const uint32_t x = cand[r * kCap + i];
            // each lane its own row, summed in dimension order
            const float *xv = X + (int64_t)x * d;
            float hi = 0.f, lo = 0.f;
            if (!VEC)
                for (int j = 0; j < d; j++) df_acc_sqdiff(__ldg(xv + j), __ldg(qv + j), hi, lo);
#pragma unroll 4
            for (int j = 0; VEC && j < d / 4; j++) {
                const float4 a = __ldg((const float4 *)xv + j), b = __ldg((const float4 *)qv + j);
                df_acc_sqdiff(a.x, b.x, hi, lo);
                df_acc_sqdiff(a.y, b.y, hi, lo);
                df_acc_sqdiff(a.z, b.z, hi, lo);
                df_acc_sqdiff(a.w, b.w, hi, lo);
            }
            v = ((uint64_t)__float_as_uint(__fadd_rn(hi, lo)) << 32) | x;
        }
        unsigned m = __ballot_sync(0xffffffffu, v < __shfl_sync(0xffffffffu, mine, k - 1));
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1;
            const uint64_t cv = __shfl_sync(0xffffffffu, v, src);
            if (cv < __shfl_sync(0xffffffffu, mine, k - 1)) {
                const int pos = __popc(__ballot_sync(0xffffffffu, mine < cv));
                const uint64_t up = __shfl_up_sync(0xffffffffu, mine, 1);
                if (lane == pos) mine = cv;
                else if (lane > pos) mine = up;
            }
        }
    }
    if (lane < k) {
        const bool have = mine != ~0ull;
        out_ids[q * k + lane] = have ? (int32_t)(uint32_t)mine : -1;
        if (out_keys) out_keys[q * k + lane] = have ? (uint32_t)(mine >> 32) : 0x7f800000u;
    }
}

// implemented in ann_knn.cu: exact SIMT k-NN of the selected query rows
int knn_f32_rows(const float *refs, int64_t N, const float *queries, const int32_t *rows, int64_t nrows, int d,
                 int k, int exclude_self, int32_t *out_ids, uint32_t *out_keys, cudaStream_t s);

int knn_f32_tensor(const float *refs, int64_t N, const float *queries, int64_t nq, int d, int k, int exclude_self,
                   int32_t *out_ids, uint32_t *out_keys, cudaStream_t s) {
    cublasHandle_t h;
    int rc = blas_handle(&h);
    if (rc != ANN_OK) return rc;
    int dev = 0;
    ANN_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> use(g_blas_use[dev]);
    // Rows of the operands and of the dot products are padded to 16 bytes and
    // the columns of D with them: cuBLAS has its tensor-core kernels for this
    // part only for aligned operands (100,003 rows of 384: 171 ms in a kernel
    // of an older part, 12.3 ms padded).
    const int ld = (3 * d + 7) / 8 * 8;
    const int64_t Np = (N + 63) / 64 * 64;
    // Tile of query rows: the tile's dot products take about 2 GB, or up to 8 GB
    // to make it 512 rows, below which reading all reference rows for it costs
    // more than the products.
    const int64_t rows8 = std::max<int64_t>(32, ((int64_t)1 << 31) / Np / 32 * 32);
    int64_t tm = std::max(((int64_t)1 << 29) / Np / 256 * 256, std::min<int64_t>(512, rows8));
    if (tm > nq) tm = nq;
    const bool shared = queries == refs && nq <= N;  // queries are the first nq reference rows
    __nv_bfloat16 *x3 = nullptr, *q3 = nullptr;
    double *rn64 = nullptr, *qn64 = nullptr;
    float *rn32 = nullptr, *qn32 = nullptr, *D = nullptr;
    unsigned long long *xmax = nullptr;
    uint32_t *cand = nullptr;
    int32_t *ncand = nullptr, *fb_rows = nullptr, *fb_count = nullptr;
    auto release = [&]() {
        void *ps[] = {rn64, rn32, shared ? nullptr : qn64, shared ? nullptr : qn32, D, xmax, cand, ncand,
                      fb_rows, fb_count, x3, q3};
        for (void *p : ps)
            if (p) cudaFreeAsync(p, s);
    };
#define F32_ALLOC(p, bytes)                                                     \
    do {                                                                        \
        cudaError_t _e = cudaMallocAsync((void **)&(p), (bytes), s);            \
        if (_e != cudaSuccess) {                                                \
            release();                                                          \
            return cuda_fail(_e, "cudaMallocAsync(float32 k-NN workspace)");    \
        }                                                                       \
    } while (0)
    F32_ALLOC(rn64, 8 * N);
    F32_ALLOC(rn32, 4 * Np);
    if (shared) {
        qn64 = rn64;
        qn32 = rn32;
    } else {
        F32_ALLOC(qn64, 8 * nq);
        F32_ALLOC(qn32, 4 * nq);
    }
    F32_ALLOC(D, 4 * (size_t)tm * Np);
    F32_ALLOC(xmax, 8);
    F32_ALLOC(cand, 4 * (size_t)tm * kCap);
    F32_ALLOC(ncand, 4 * tm);
    F32_ALLOC(fb_rows, 4 * nq);
    F32_ALLOC(fb_count, 4);
    F32_ALLOC(x3, 2 * (size_t)Np * ld);
    F32_ALLOC(q3, 2 * (size_t)nq * ld);
#undef F32_ALLOC
    const int64_t w = d + (ld - 3 * d);
    split_bf16_kernel<<<(unsigned)((Np * w + 255) / 256), 256, 0, s>>>(refs, N, Np, d, ld, 0, x3);
    split_bf16_kernel<<<(unsigned)((nq * w + 255) / 256), 256, 0, s>>>(queries, nq, nq, d, ld, 1, q3);
    norms_f32_kernel<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(refs, N, d, rn64, rn32);
    if (!shared) norms_f32_kernel<<<(unsigned)((nq + 255) / 256), 256, 0, s>>>(queries, nq, d, qn64, qn32);
    cudaMemsetAsync(xmax, 0, 8, s);
    cudaMemsetAsync(fb_count, 0, 4, s);
    max_norm_kernel<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(rn64, N, xmax);
    if (cublasSetStream(h, s) != CUBLAS_STATUS_SUCCESS) {
        release();
        return fail(ANN_ERR_CUDA, "cublasSetStream failed");
    }
    const float one = 1.f, zero = 0.f;
    for (int64_t q0 = 0; q0 < nq; q0 += tm) {
        const int64_t rows = std::min<int64_t>(tm, nq - q0);
        // D (column-major Np x rows) = X3^T Q3: row r of the tile is D + r * Np
        const cublasStatus_t st = cublasGemmEx(h, CUBLAS_OP_T, CUBLAS_OP_N, (int)Np, (int)rows, ld, &one, x3,
                                               CUDA_R_16BF, ld, q3 + q0 * ld, CUDA_R_16BF, ld, &zero, D, CUDA_R_32F,
                                               (int)Np, CUBLAS_COMPUTE_32F, CUBLAS_GEMM_DEFAULT);
        if (st != CUBLAS_STATUS_SUCCESS) {
            release();
            return fail(ANN_ERR_CUDA, "cublasGemmEx (float32 k-NN) failed: status " + std::to_string((int)st));
        }
        const unsigned grid = (unsigned)((rows * 32 + 255) / 256);
        f32_scan_kernel<<<(unsigned)rows, kScanThreads, 0, s>>>(D, Np, q0, N, d, qn32, rn32, qn64, xmax,
                                                                   exclude_self, k, cand, ncand);
        if ((((uintptr_t)refs | (uintptr_t)queries) & 15) == 0)
            f32_rescore_kernel<true><<<grid, 256, 0, s>>>(refs, queries, d, rows, q0, cand, ncand, k, out_ids,
                                                          out_keys, fb_rows, fb_count);
        else
            f32_rescore_kernel<false><<<grid, 256, 0, s>>>(refs, queries, d, rows, q0, cand, ncand, k, out_ids,
                                                           out_keys, fb_rows, fb_count);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) {
            release();
            return cuda_fail(e, "float32 k-NN kernels");
        }
    }
    int32_t nfb = 0;
    cudaError_t e = cudaMemcpyAsync(&nfb, fb_count, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        release();
        return cuda_fail(e, "float32 k-NN fallback count");
    }
    if (nfb > 0) rc = knn_f32_rows(refs, N, queries, fb_rows, nfb, d, k, exclude_self, out_ids, out_keys, s);
    release();
    return rc;
}

}  // namespace ann

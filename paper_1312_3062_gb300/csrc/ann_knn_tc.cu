// ann_knn_tc.cu -- exact k nearest neighbours of uint8 vectors on the 5th
// generation tensor cores (tcgen05) of sm_103a: the R-NN neighbourhood graph
// of Sec. 3.1 / Sec. 4.1 and the linear-scan ground truth of Sec. 5.1.
//
// Keys are ||q||^2 + ||x||^2 - 2 q.x.  Bytes 0..255 are exact in bf16 and the
// inner product is taken over d + 16 elements: a row's last 16 hold -1, -1, -1
// on the query side and ||x||^2 / 2 in three bf16 pieces (bits 16.., 8..15,
// 0..7) on the reference side, so the accumulator is q.x - ||x||^2 / 2, a
// multiple of 1/2 below 2^23 in magnitude like every partial sum of it: exact
// in fp32.  The key is ||q||^2 - 2 acc, so an epilogue thread (one query row)
// only looks for accumulators above a limit.
//
// One CTA per SM, persistent over items (128 query rows, a range of reference
// tiles):
//   warp 0      TMA producer: the query rows (A) once per item, reference
//               tiles (B, 256 rows) through a 2-stage ring
//   warp 1      allocates 512 TMEM columns; one lane issues tcgen05.mma
//               (M=128, N=256, K=16) into one of two 256-column accumulators
//   warps 2..9  epilogue, two warps (column halves) per TMEM lane quadrant:
//               tcgen05.ld of 32 columns, the maxima of groups of four with
//               three-input instructions (about 0.6 instructions per key)
//               against the limit; groups that pass are appended whole, without
//               branches, to a per-row buffer (global memory, in L2).  The
//               buffers are emptied into sorted lists of K entries in
//               registers, all 32 rows of a warp at once, after 1, 2, 4, 8, ...
//               tiles of an item: a limit that is one doubling old lets about
//               k more references through, so this costs k log2(tiles)
//               insertions a row against k ln(N / k) with a limit that is
//               always new, but the two accumulators in flight hide only one
//               tile's time, and the epilogue warps now stop together a dozen
//               times an item and not each at its own hundreds of insertions
//               (graph of 400,000 rows, k = 20: 56.6 -> 34.1 ms).  The
//               first limit is the k-th best of the maxima of the first tile's
//               groups of four columns.  The two column halves of a row share
//               the k/2-th keys of their lists (the larger one bounds the row's
//               k-th), and the lists of a row's ranges their k-th keys.
// A second kernel merges the lists of a row.
// Measured: graph of 400,000 x 128 rows, k = 20: 34.1 ms (1190 TFLOP/s of
// distances, 1340 with the slab); 138 ms with norms added and sorted insertions
// into shared memory in the epilogue.  10,000 queries against 1M rows, k = 10:
// 2.4 ms, 9.7 before (79 CTAs, no ranges).
// The leaf step of the approximate graph (knn_u8_leaves) is the same kernel with
// other items: rows in leaf order, and 128 rows of a leaf against that leaf.
// Every mbarrier wait is bounded; on timeout the CTA records an error and
// every role leaves its loop, so the kernel always returns and frees TMEM.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "ann_device.cuh"
#include "ann_internal.cuh"

namespace ann {
namespace tc {

constexpr int BM = 128;           // query rows per block (TMEM lanes)
constexpr int BN = 256;           // reference rows per tile (accumulator columns)
constexpr int BK = 64;            // bf16 elements per TMA box row (128 B, one swizzle row)
constexpr int STAGES = 2;
constexpr int NUM_THREADS = 320;  // 10 warps

constexpr int SLAB = 16;          // the extra inner-product elements
constexpr int CAP = 64;           // pending groups of four columns per row and epilogue warp

struct Params {
    int64_t nq, N;
    int d, k, exclude_self;
    int nsplit;                   // ranges of reference tiles per block of query rows
    int levels, leaf_blocks;      // leaves: halvings of [0, N), 128-row blocks of the largest leaf
    const uint32_t *ids;          // leaves: the id of the row at each position
    const uint32_t *qnorm;
    uint32_t *row_limit;          // per query row: the smallest k-th key of its lists so far
    uint64_t *lists;              // [row][2 * nsplit][k], ascending, ~0 padded
    float4 *pend;                 // [CTA][8 epilogue warps][CAP][32 rows]: four accumulators
    int *pend_col;                // and the id of the first one's reference
    int *error;
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// bounded wait (2 s) for the phase with the given parity; false on timeout or
// when another role has already recorded an error
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *err) {
    const uint32_t a = smem_u32(bar);
    if (*err) return false;
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t it = 0;; it++) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((it & 255) == 255) {
            if (*err) return false;
            if (globaltimer_ns() - t0 > 2000000000ull) break;
        }
    }
    *err = 1;
    return false;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(smem_u32(dst)),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row atoms 1024 B apart
__device__ __forceinline__ uint64_t smem_desc(const void *p) {
    const uint64_t addr = smem_u32(p);
    uint64_t d = 0;
    d |= (addr >> 4) & 0x3FFFull;            // start address
    d |= (uint64_t)1 << 16;                  // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;        // stride byte offset: next 8-row atom
    d |= (uint64_t)1 << 46;                  // descriptor version for sm_100-class tensor cores
    d |= (uint64_t)2 << 61;                  // layout: 128-byte swizzle
    return d;
}

// the slab's tiles: K-major, 32-byte rows, 32-byte swizzle, 8-row atoms 256 B apart
__device__ __forceinline__ uint64_t slab_desc(const void *p) {
    uint64_t d = 0;
    d |= ((uint64_t)smem_u32(p) >> 4) & 0x3FFFull;
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(256 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)6 << 61;                  // layout: 32-byte swizzle
    return d;
}

// instruction descriptor: kind::f16, A and B bf16, D f32, both K-major, M x N
__host__ __device__ constexpr uint32_t instr_desc(int M, int N) {
    return (1u << 4)                   // D format f32
           | (1u << 7)                 // A format bf16
           | (1u << 10)                // B format bf16
           | ((uint32_t)(N >> 3) << 17)
           | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
// the loads issued so far have arrived; the registers pass through so that no
// use of them moves before the wait
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])::"memory");
}

// shared memory plan (bytes, 1024-aligned tiles)
struct Smem {
    __host__ __device__ static constexpr int a_bytes(int d) { return BM * (d + SLAB) * 2; }
    __host__ __device__ static constexpr int b_bytes(int d) { return BN * (d + SLAB) * 2; }
};

// A row's list: K (key - ||q||^2, id) pairs in registers, ascending; the first
// K - k are held at -infinity so that the last is the k-th best.  References
// come in ascending id order, so an equal key belongs behind.
template <int K>
struct RowList {
    float key[K];
    int id[K];
    __device__ __forceinline__ void clear(int k) {
#pragma unroll
        for (int i = 0; i < K; i++) {
            key[i] = i < K - k ? -__int_as_float(0x7f800000) : __int_as_float(0x7f800000);
            id[i] = -1;
        }
    }
    __device__ __forceinline__ void insert(float v, int x) {
#pragma unroll
        for (int i = K - 1; i >= 0; i--) {
            const bool here = v < key[i], before = i > 0 && v < key[i > 0 ? i - 1 : 0];
            key[i] = before ? key[i > 0 ? i - 1 : 0] : (here ? v : key[i]);
            id[i] = before ? id[i > 0 ? i - 1 : 0] : (here ? x : id[i]);
        }
    }
};

// leaf `s` of `levels` halvings of [0, N): its positions [lo, hi)
__device__ __forceinline__ void leaf_range(int64_t N, int levels, int64_t s, int64_t &lo, int64_t &hi) {
    lo = 0;
    hi = N;
    for (int k = levels - 1; k >= 0; k--) {
        const int64_t m = lo + (hi - lo) / 2;
        if ((s >> k) & 1) lo = m;
        else hi = m;
    }
}

// One item: query rows [row0, row1), at most BM of them, against the
// references [ref0, ref1).
struct Item {
    int64_t row0, row1, ref0, ref1, split;
    __device__ __forceinline__ int64_t tiles() const { return (ref1 - ref0 + BN - 1) / BN; }
};

template <bool LEAF>
__device__ __forceinline__ int64_t num_items(const Params &p) {
    return LEAF ? ((int64_t)p.leaf_blocks << p.levels) : (p.nq + BM - 1) / BM * p.nsplit;
}

// false: there is nothing to do (a leaf with fewer blocks than the largest)
template <bool LEAF>
__device__ __forceinline__ bool get_item(const Params &p, int64_t it, Item &I) {
    if (LEAF) {
        leaf_range(p.N, p.levels, it / p.leaf_blocks, I.ref0, I.ref1);
        I.row0 = I.ref0 + it % p.leaf_blocks * BM;
        I.row1 = I.ref1;
        I.split = 0;
        return I.row0 < I.ref1;
    }
    // split-major: CTAs of one wave share their tiles
    const int64_t nblocks = (p.nq + BM - 1) / BM, per = ((p.N + BN - 1) / BN + p.nsplit - 1) / p.nsplit;
    I.split = it / nblocks;
    I.row0 = it % nblocks * BM;
    I.row1 = p.nq;
    I.ref0 = I.split * per * BN;
    I.ref1 = I.ref0 + per * BN < p.N ? I.ref0 + per * BN : p.N;
    return true;
}

template <int K, bool LEAF>
__global__ void __launch_bounds__(NUM_THREADS, 1)
    knn_tc_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapAs,
                  const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapBs, Params prm) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    // align the dynamic shared memory base to 1024 bytes (swizzle atoms)
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int d = prm.d, k = prm.k;
    const int kch = d / BK;                       // 128-byte-wide TMA boxes per row block
    uint8_t *sA = smem;                           // kch x [BM rows x 128 B], then [BM rows x 32 B]
    uint8_t *sB = sA + Smem::a_bytes(d);          // STAGES x (kch x [BN rows x 128 B], then [BN rows x 32 B])
    uint64_t *bars = (uint64_t *)(sB + STAGES * Smem::b_bytes(d));
    uint64_t *full = bars;                        // STAGES
    uint64_t *empty = bars + STAGES;              // STAGES
    uint64_t *tfull = bars + 2 * STAGES;          // 2
    uint64_t *tempty = bars + 2 * STAGES + 2;     // 2
    uint64_t *afull = bars + 2 * STAGES + 4;      // 1
    uint64_t *aempty = bars + 2 * STAGES + 5;     // 1
    uint64_t *mdone = bars + 2 * STAGES + 6;      // 1: every MMA issued so far has completed
    uint32_t *tmem_slot = (uint32_t *)(bars + 2 * STAGES + 7);
    __shared__ int s_err;
    // per item (mod 4), column half and row: the ceil(k/2)-th key of the half's
    // list.  A half runs at most two tiles, so two items, ahead of the other; it
    // clears its entry for item n + 2 when it starts item n.
    __shared__ float s_half[4][2][BM];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t nitems = num_items<LEAF>(prm);
    Item I;

    if (threadIdx.x == 0) {
        s_err = 0;
        for (int s = 0; s < STAGES; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; a++) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], 8);  // one arrival per epilogue warp
        }
        mbar_init(afull, 1);
        mbar_init(aempty, 1);
        mbar_init(mdone, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = threadIdx.x; i < 4 * 2 * BM; i += NUM_THREADS) (&s_half[0][0][0])[i] = __int_as_float(0x7f800000);
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;
    volatile int *err = &s_err;

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            int64_t g = 0;  // global tile counter (ring position)
            int64_t nb = 0;
            int64_t last_use[STAGES];
            for (int s = 0; s < STAGES; s++) last_use[s] = -1;
            int64_t a_loads = 0;
            for (int64_t it = blockIdx.x; it < nitems && !*err; it += gridDim.x) {
                if (!get_item<LEAF>(prm, it, I)) continue;
                const int64_t nt = I.tiles();
                if (nb > 0 && !mbar_wait(aempty, (uint32_t)((nb - 1) & 1), err)) break;
                mbar_expect_tx(afull, (uint32_t)Smem::a_bytes(d));
                for (int c = 0; c < kch; c++)
                    tma_load_2d(sA + c * BM * 128, &mapA, afull, c * BK, (int)I.row0);
                tma_load_2d(sA + kch * BM * 128, &mapAs, afull, 0, 0);
                a_loads++;
                nb++;
                bool ok = true;
                for (int64_t t = 0; t < nt; t++, g++) {
                    const int s = (int)(g % STAGES);
                    const int64_t use = g / STAGES;
                    if (use > 0 && !mbar_wait(&empty[s], (uint32_t)((use - 1) & 1), err)) {
                        ok = false;
                        break;
                    }
                    uint8_t *dst = sB + s * Smem::b_bytes(d);
                    mbar_expect_tx(&full[s], (uint32_t)Smem::b_bytes(d));
                    for (int c = 0; c < kch; c++)
                        tma_load_2d(dst + c * BN * 128, &mapB, &full[s], c * BK, (int)(I.ref0 + t * BN));
                    tma_load_2d(dst + kch * BN * 128, &mapBs, &full[s], 0, (int)(I.ref0 + t * BN));
                    last_use[s] = use;
                }
                if (!ok) break;
            }
            // do not leave copies in flight: wait (bounded) for the last load of every buffer
            volatile int drain_err = 0;
            for (int s = 0; s < STAGES; s++)
                if (last_use[s] >= 0) mbar_wait(&full[s], (uint32_t)(last_use[s] & 1), &drain_err);
            if (a_loads > 0) mbar_wait(afull, (uint32_t)((a_loads - 1) & 1), &drain_err);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            const uint32_t idesc = instr_desc(BM, BN);
            int64_t g = 0, u = 0;  // ring position, accumulator use counter
            int64_t nb = 0;
            for (int64_t it = blockIdx.x; it < nitems && !*err; it += gridDim.x) {
                if (!get_item<LEAF>(prm, it, I)) continue;
                const int64_t nt = I.tiles();
                if (!mbar_wait(afull, (uint32_t)(nb & 1), err)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                nb++;
                bool ok = true;
                for (int64_t t = 0; t < nt; t++, g++, u++) {
                    const int s = (int)(g % STAGES);
                    const int acc = (int)(u & 1);
                    const int64_t ause = u >> 1;
                    if ((ause > 0 && !mbar_wait(&tempty[acc], (uint32_t)((ause - 1) & 1), err)) ||
                        !mbar_wait(&full[s], (uint32_t)((g / STAGES) & 1), err)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t dcol = tmem_base + (uint32_t)(acc * BN);
                    const uint8_t *b0 = sB + s * Smem::b_bytes(d);
                    for (int c = 0; c < kch; c++)
                        for (int kk = 0; kk < BK / 16; kk++) {
                            uint64_t ad = smem_desc(sA + c * BM * 128 + kk * 32);
                            uint64_t bd = smem_desc(b0 + c * BN * 128 + kk * 32);
                            mma_bf16(dcol, ad, bd, idesc, (c | kk) != 0);
                        }
                    mma_bf16(dcol, slab_desc(sA + kch * BM * 128), slab_desc(b0 + kch * BN * 128), idesc, 1);
                    mma_commit(&empty[s]);     // B stage free once these MMAs are done
                    mma_commit(&tfull[acc]);   // accumulator ready for the epilogue
                }
                if (!ok) break;
                mma_commit(aempty);            // query block may be replaced
            }
            // every MMA issued has completed before TMEM is released (bounded wait)
            mma_commit(mdone);
            volatile int drain_err = 0;
            mbar_wait(mdone, 0, &drain_err);
        }
    } else {
        // ---------------- epilogue ----------------
        const int ew = warp - 2;              // 0..7
        const int quad = warp & 3;            // TMEM lane quadrant this warp may access
        const int half = ew >> 2;             // column half
        const int row = quad * 32 + lane;     // row of the block
        const size_t slot0 = ((size_t)blockIdx.x * 8 + ew) * CAP * 32 + lane;
        float4 *mypend = prm.pend + slot0;
        int *mycol = prm.pend_col + slot0;
        const float inf = __int_as_float(0x7f800000);
        const int k2 = K - k + (k + 1) / 2 - 1;  // list entry of the ceil(k/2)-th best
        int64_t u = 0;
        uint32_t n_it = 0;
        for (int64_t it = blockIdx.x; it < nitems && !*err; it += gridDim.x) {
            if (!get_item<LEAF>(prm, it, I)) continue;
            volatile float *my_half = &s_half[n_it & 3][half][row], *other_half = &s_half[n_it & 3][half ^ 1][row];
            *(volatile float *)&s_half[(n_it + 2) & 3][half][row] = inf;
            float own_half = inf;
            n_it++;
            const int64_t nt = I.tiles();
            const int64_t qrow = I.row0 + row;
            const bool valid_row = qrow < I.row1;
            const uint32_t qn = valid_row ? prm.qnorm[qrow] : 0u;
            const float qnf = (float)qn;
            uint32_t *limit = prm.row_limit + (valid_row ? qrow : 0);
            RowList<K> list;
            list.clear(k);
            int cnt = 0;                           // pending entries
            // accumulators above lim may belong to the k best; rows past the end take none
            float lim = valid_row ? -inf : inf;
            if (valid_row && *(volatile uint32_t *)limit != 0xffffffffu)
                lim = -0.5f * ((float)(*(volatile uint32_t *)limit + 1) - qnf);
            auto flush = [&]() {
                const int most = __reduce_max_sync(0xffffffffu, cnt);
                const uint32_t other = *(volatile uint32_t *)limit;  // arrives while the entries go in
                float4 en = make_float4(-inf, -inf, -inf, -inf);
                int cn = 0;
                if (cnt > 0) {
                    en = mypend[0];
                    cn = mycol[0];
                }
                for (int i = 0; i < most; i++) {
                    float a[4] = {en.x, en.y, en.z, en.w};
                    const int c = cn;
                    if (i >= cnt) a[0] = a[1] = a[2] = a[3] = -inf;
                    if (i + 1 < cnt) {  // the next group's load flies while this one goes in
                        en = mypend[(i + 1) * 32];
                        cn = mycol[(i + 1) * 32];
                    }
#pragma unroll
                    for (int j = 0; j < 4; j++)
                        if (c + j >= I.ref1 || (prm.exclude_self && c + j == qrow)) a[j] = -inf;
                    for (;;) {  // the best of the four first, the lower id of equal ones
                        const float b = fmaxf(fmaxf(a[0], a[1]), fmaxf(a[2], a[3]));
                        const float v = -2.0f * b;  // -inf becomes an infinite key, which goes nowhere
                        if (!__any_sync(0xffffffffu, v < list.key[K - 1])) break;
                        const int j = a[0] == b ? 0 : (a[1] == b ? 1 : (a[2] == b ? 2 : 3));
                        list.insert(v, c + j);
#pragma unroll
                        for (int q = 0; q < 4; q++)
                            if (q == j) a[q] = -inf;
                    }
                }
                cnt = 0;
                if (valid_row) {
                    // own list: a later reference needs a smaller key; another
                    // list's bound: an equal key may still win by its id
                    float t = list.key[K - 1];
                    if (t < inf) atomicMin(limit, (uint32_t)(t + qnf));
                    if (other != 0xffffffffu) t = fminf(t, (float)(other + 1) - qnf);
                    lim = fmaxf(lim, -0.5f * t);
#pragma unroll
                    for (int i = 0; i < K; i++) own_half = i == k2 ? list.key[i] : own_half;
                    *my_half = own_half;
                }
            };
            bool ok = true;
            int64_t next = 1;  // tiles after which the buffers are emptied next
            for (int64_t t = 0; t < nt; t++, u++) {
                const int acc = (int)(u & 1);
                if (!mbar_wait(&tfull[acc], (uint32_t)((u >> 1) & 1), err)) {
                    ok = false;
                    break;
                }
                __syncwarp();
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // k rows lie at or below the larger of the halves' keys; an equal one may still win by its id
                lim = fmaxf(lim, -0.5f * fmaxf(own_half, *other_half) - 0.5f);
                const uint32_t tcol =
                    tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * BN + half * (BN / 2));
                const int rid0 = (int)(I.ref0 + t * BN) + half * (BN / 2);
                const int kk = k + (prm.exclude_self ? 1 : 0);
                if (t == 0 && rid0 + BN / 2 <= I.ref1 && kk <= 32) {
                    // k distinct references (and the row itself) lie at or above the kk-th group maximum
                    float gm[32];
#pragma unroll
                    for (int c = 0; c < 4; c++) {
                        uint32_t v[32];
                        tmem_ld32(tcol + 32 * c, v);
                        tmem_wait(v);
#pragma unroll
                        for (int g = 0; g < 8; g++)
                            gm[8 * c + g] = fmaxf(fmaxf(__uint_as_float(v[4 * g]), __uint_as_float(v[4 * g + 1])),
                                                  fmaxf(__uint_as_float(v[4 * g + 2]), __uint_as_float(v[4 * g + 3])));
                    }
#pragma unroll
                    for (int w = 2; w <= 32; w <<= 1)
#pragma unroll
                        for (int j = w >> 1; j > 0; j >>= 1)
#pragma unroll
                            for (int i = 0; i < 32; i++)
                                if ((i ^ j) > i) {
                                    const float x = gm[i], y = gm[i ^ j];
                                    const bool down = (i & w) == 0;  // descending overall
                                    gm[i] = down ? fmaxf(x, y) : fminf(x, y);
                                    gm[i ^ j] = down ? fminf(x, y) : fmaxf(x, y);
                                }
                    float bound = gm[0];
#pragma unroll
                    for (int i = 1; i < 32; i++) bound = i == kk - 1 ? gm[i] : bound;
                    if (valid_row) lim = fmaxf(lim, bound - 0.5f);  // accumulators are multiples of 1/2
                }
                auto take = [&](const uint32_t (&v)[32], int cb) __attribute__((always_inline)) {
                    float m[8];
#pragma unroll
                    for (int g = 0; g < 8; g++)
                        m[g] = fmaxf(fmaxf(fmaxf(__uint_as_float(v[4 * g]), __uint_as_float(v[4 * g + 1])),
                                           __uint_as_float(v[4 * g + 2])), __uint_as_float(v[4 * g + 3]));
                    const float mx = fmaxf(fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])),
                                           fmaxf(fmaxf(m[4], m[5]), fmaxf(m[6], m[7])));
                    if (!__any_sync(0xffffffffu, mx > lim)) return;
#pragma unroll
                    for (int g = 0; g < 8; g++)
                        if (m[g] > lim) {
                            mypend[cnt * 32] = make_float4(__uint_as_float(v[4 * g]), __uint_as_float(v[4 * g + 1]),
                                                           __uint_as_float(v[4 * g + 2]), __uint_as_float(v[4 * g + 3]));
                            mycol[cnt * 32] = rid0 + cb + 4 * g;
                            cnt++;
                        }
                };
                uint32_t va[32], vb[32];
                tmem_ld32(tcol, va);
                tmem_wait(va);
                tmem_ld32(tcol + 32, vb);
                take(va, 0);
                tmem_wait(vb);
                tmem_ld32(tcol + 64, va);
                take(vb, 32);
                tmem_wait(va);
                tmem_ld32(tcol + 96, vb);
                take(va, 64);
                tmem_wait(vb);
                // every column of this half is in registers: the accumulator may be overwritten
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty[acc]);
                take(vb, 96);
                // a tile adds up to 32 groups
                if (t + 1 == next || t + 1 == nt || __any_sync(0xffffffffu, cnt > CAP - BN / 8)) {
                    if (t + 1 == next) next *= 2;
                    flush();
                }
            }
            if (!ok) break;
            // this warp's list for its rows and column half; merged by a second kernel
            if (valid_row) {
                uint64_t *dst = prm.lists + ((size_t)qrow * 2 * prm.nsplit + 2 * I.split + half) * k;
#pragma unroll
                for (int i = 0; i < K; i++)
                    if (i >= K - k)
                        dst[i - (K - k)] = list.key[i] < inf
                                               ? ((uint64_t)(uint32_t)(list.key[i] + qnf) << 32) |
                                                     (LEAF ? prm.ids[list.id[i]] : (uint32_t)list.id[i])
                                               : ~0ull;
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base));
    }
    if (threadIdx.x == 0 && s_err) atomicExch(prm.error, 1);
}

// merge the nl sorted lists of every row, one warp per row: the k smallest by
// (key, id), entry `lane` of a warp-held ascending list
__global__ void merge_lists_kernel(const uint64_t *lists, int64_t nq, int nl, int k, int32_t *out_ids,
                                   uint32_t *out_keys) {
    const int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (q >= nq) return;
    const uint64_t *src = lists + (size_t)q * nl * k;
    uint64_t mine = lane < k ? src[lane] : ~0ull;
    for (int b = k; b < nl * k; b += 32) {
        const uint64_t v = b + lane < nl * k ? src[b + lane] : ~0ull;
        unsigned m = __ballot_sync(0xffffffffu, v < __shfl_sync(0xffffffffu, mine, k - 1));
        while (m) {
            const int from = __ffs(m) - 1;
            m &= m - 1;
            const uint64_t c = __shfl_sync(0xffffffffu, v, from);
            if (c >= __shfl_sync(0xffffffffu, mine, k - 1)) continue;
            const int pos = __popc(__ballot_sync(0xffffffffu, mine < c));
            const uint64_t up = __shfl_up_sync(0xffffffffu, mine, 1);
            if (lane == pos) mine = c;
            else if (lane > pos) mine = up;
        }
    }
    if (lane < k) {
        const bool have = mine != ~0ull;
        out_ids[q * k + lane] = have ? (int32_t)(uint32_t)mine : -1;
        if (out_keys) out_keys[q * k + lane] = have ? (uint32_t)(mine >> 32) : 0xffffffffu;
    }
}

// Rows as bf16 (bytes are exact), their squared norms and, for references, the
// slab of norm pieces.  Four bytes per thread, d / 4 threads per row.  With an
// order (leaves), row r is the one of id order[r] & idmask; its id and the
// largest key of its list so far (graph: R per id) go out too.
__global__ void prep_rows_kernel(const uint8_t *X, int64_t N, int d, uint16_t *rows, uint32_t *norm, uint16_t *slab,
                                 const uint64_t *order = nullptr, uint64_t idmask = 0, const uint64_t *graph = nullptr,
                                 int R = 0, uint32_t *ids = nullptr, uint32_t *limit = nullptr) {
    const int tpr = d / 4;  // 16 or 32
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t r = i / tpr;
    const int w = (int)(i - r * tpr);
    const int64_t src = r >= N ? 0 : (order ? (int64_t)(order[r] & idmask) : r);
    const uint32_t v = r < N ? __ldg((const uint32_t *)X + src * tpr + w) : 0u;
    uint32_t s = __dp4a(v, v, 0u);
    for (int off = tpr / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (r >= N) return;
    auto bf = [](float f) { return __float_as_uint(f) >> 16; };
    const uint32_t b0 = bf((float)(v & 255u)), b1 = bf((float)((v >> 8) & 255u));
    const uint32_t b2 = bf((float)((v >> 16) & 255u)), b3 = bf((float)(v >> 24));
    *(uint2 *)(rows + 4 * i) = make_uint2(b0 | (b1 << 16), b2 | (b3 << 16));
    if (w == 0) norm[r] = s;
    if (ids && w == 1) {
        ids[r] = (uint32_t)src;
        limit[r] = (uint32_t)(graph[src * R + R - 1] >> 32);
    }
    if (slab && w < 2) {
        const uint32_t hi = bf((float)(s >> 16) * 32768.0f), mid = bf((float)((s >> 8) & 255u) * 128.0f);
        const uint32_t low = bf((float)(s & 255u) * 0.5f);
        *(uint4 *)(slab + r * SLAB + 8 * w) = w == 0 ? make_uint4(hi | (mid << 16), low, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
    }
}

// the query side of the slab: -1, -1, -1 and zeros, BM rows
__global__ void query_slab_kernel(uint16_t *slab) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < BM * SLAB) slab[i] = i % SLAB < 3 ? 0xbf80u : 0u;
}

// ---- driver entry point for tensor-map encoding (no link against libcuda) ----
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static std::once_flag once;
    static EncodeTiledFn fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    });
    return fn;
}

// tiles of box_rows x BK elements with the 128-byte swizzle, or of the slab's
// box_rows x 16 with the 32-byte one
static int make_map(CUtensorMap *map, const uint16_t *base, int64_t rows, int d, int box_rows) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return fail(ANN_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
    cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)d * 2};
    cuuint32_t box[2] = {(cuuint32_t)(d == SLAB ? SLAB : BK), (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void *)base, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE,
                     d == SLAB ? CU_TENSOR_MAP_SWIZZLE_32B : CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(ANN_ERR_CUDA, "cuTensorMapEncodeTiled failed");
    return ANN_OK;
}

size_t smem_bytes(int d) {
    return 1024 /* alignment slack */ + (size_t)Smem::a_bytes(d) + (size_t)STAGES * Smem::b_bytes(d) +
           (2 * STAGES + 7) * 8 + 16;
}

// Ranges of reference tiles per block of query rows: the count with the
// smallest makespan, waves x (tiles per range + what a new range costs in
// tiles: the query rows' load and the insertions until its limits settle).
// 10,000 queries are 79 blocks, half the SMs of this part; split 25 ways they
// make 13 full waves.  At most 64 ranges: each keeps two lists of k pairs per
// query row, 33 KB a row at k = 32; so calls of up to 128 queries use 64 SMs.
int choose_split(int64_t nblocks, int64_t ntiles, int nsm, int k) {
    const int64_t extra = 8 + k;
    int best = 1;
    int64_t cost = -1;
    for (int ns = 1; ns <= 64 && ns <= ntiles; ns++) {
        const int64_t per = (ntiles + ns - 1) / ns;
        if ((ntiles + per - 1) / per != ns) continue;  // an empty last range
        const int64_t c = (nblocks * ns + nsm - 1) / nsm * (per + extra);
        if (cost < 0 || c < cost) {
            cost = c;
            best = ns;
        }
    }
    return best;
}

template <int K, bool LEAF>
cudaError_t launch_k(unsigned grid, size_t smem, cudaStream_t s, const CUtensorMap *m, const Params &prm) {
    const cudaError_t e =
        cudaFuncSetAttribute(knn_tc_kernel<K, LEAF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) knn_tc_kernel<K, LEAF><<<grid, NUM_THREADS, smem, s>>>(m[0], m[1], m[2], m[3], prm);
    return e;
}

// list capacity 8, 16, 24 or 32
template <bool LEAF>
cudaError_t launch_tc(unsigned grid, size_t smem, cudaStream_t s, const CUtensorMap *m, const Params &prm) {
    return prm.k <= 8    ? launch_k<8, LEAF>(grid, smem, s, m, prm)
           : prm.k <= 16 ? launch_k<16, LEAF>(grid, smem, s, m, prm)
           : prm.k <= 24 ? launch_k<24, LEAF>(grid, smem, s, m, prm)
                         : launch_k<32, LEAF>(grid, smem, s, m, prm);
}

}  // namespace tc

// Exact k-NN of uint8 rows on the tensor cores.  Requires d in {64, 128}, k <= 32.
int knn_u8_tensor(const uint8_t *refs, int64_t N, const uint8_t *queries, int64_t nq, int d, int k,
                  int exclude_self, int32_t *out_ids, uint32_t *out_keys, cudaStream_t s) {
    using namespace tc;
    const size_t smem = smem_bytes(d);
    int dev = 0, nsm = 0;
    ANN_CUDA(cudaGetDevice(&dev));
    ANN_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const bool shared = queries == refs && nq <= N;  // queries are the first nq reference rows
    const int64_t nblocks = (nq + BM - 1) / BM, ntiles = (N + BN - 1) / BN;
    const int nsplit = choose_split(nblocks, ntiles, nsm, k), nl = 2 * nsplit;
    uint16_t *rb = nullptr, *qb = nullptr, *rslab = nullptr, *qslab = nullptr;
    uint32_t *rn = nullptr, *qn = nullptr, *limit = nullptr;
    int *derr = nullptr;
    uint64_t *lists = nullptr;
    float4 *pend = nullptr;
    int *pend_col = nullptr;
    const unsigned grid = (unsigned)std::min<int64_t>(nblocks * nsplit, nsm);
    AsyncBufs bufs(s);  // every buffer below is released on return
    ANN_CUDA(bufs.alloc(&pend, (size_t)grid * 8 * CAP * 32 * 16));
    ANN_CUDA(bufs.alloc(&pend_col, (size_t)grid * 8 * CAP * 32 * 4));
    ANN_CUDA(bufs.alloc(&lists, (size_t)nq * nl * k * 8));
    ANN_CUDA(bufs.alloc(&rb, (size_t)N * d * 2));
    ANN_CUDA(bufs.alloc(&rslab, (size_t)N * SLAB * 2));
    ANN_CUDA(bufs.alloc(&qslab, (size_t)BM * SLAB * 2));
    ANN_CUDA(bufs.alloc(&rn, (size_t)N * 4));
    ANN_CUDA(bufs.alloc(&limit, (size_t)nq * 4));
    ANN_CUDA(bufs.alloc(&derr, sizeof(int)));
    ANN_CUDA(cudaMemsetAsync(derr, 0, sizeof(int), s));
    ANN_CUDA(cudaMemsetAsync(limit, 0xff, (size_t)nq * 4, s));
    const int tpr = d / 4;
    query_slab_kernel<<<(BM * SLAB + 255) / 256, 256, 0, s>>>(qslab);
    prep_rows_kernel<<<(unsigned)((N * tpr + 255) / 256), 256, 0, s>>>(refs, N, d, rb, rn, rslab);
    if (shared) {
        qb = rb;
        qn = rn;
    } else {
        ANN_CUDA(bufs.alloc(&qb, (size_t)nq * d * 2));
        ANN_CUDA(bufs.alloc(&qn, (size_t)nq * 4));
        prep_rows_kernel<<<(unsigned)((nq * tpr + 255) / 256), 256, 0, s>>>(queries, nq, d, qb, qn, nullptr);
    }
    CUtensorMap m[4];
    int r = make_map(&m[0], qb, nq, d, BM);
    if (r == ANN_OK) r = make_map(&m[1], qslab, BM, SLAB, BM);
    if (r == ANN_OK) r = make_map(&m[2], rb, N, d, BN);
    if (r == ANN_OK) r = make_map(&m[3], rslab, N, SLAB, BN);
    if (r != ANN_OK) return r;
    Params prm{nq, N, d, k, exclude_self, nsplit, 0, 0, nullptr, qn, limit, lists, pend, pend_col, derr};
    const cudaError_t e = launch_tc<false>(grid, smem, s, m, prm);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(knn_tc_kernel)");
    merge_lists_kernel<<<(unsigned)((nq * 32 + 255) / 256), 256, 0, s>>>(lists, nq, nl, k, out_ids, out_keys);
    ANN_CUDA(cudaGetLastError());
    int herr = 0;
    ANN_CUDA(cudaMemcpyAsync(&herr, derr, sizeof(int), cudaMemcpyDeviceToHost, s));
    ANN_CUDA(cudaStreamSynchronize(s));
    if (herr) return fail(ANN_ERR_TIMEOUT, "knn_tc_kernel: a pipeline wait timed out");
    return ANN_OK;
}

// ---- the leaf step of the approximate graph ----

int LeafTc::prepare(int64_t N_, int d_, int R_, int levels_, cudaStream_t s) {
    using namespace tc;
    N = N_, d = d_, R = R_, levels = levels_;
    int dev = 0;
    ANN_CUDA(cudaGetDevice(&dev));
    ANN_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    ANN_CUDA(bufs.alloc(&lists, (size_t)N * 2 * R * 8));
    ANN_CUDA(bufs.alloc(&rb, (size_t)N * d * 2));
    ANN_CUDA(bufs.alloc(&rslab, (size_t)N * SLAB * 2));
    ANN_CUDA(bufs.alloc(&qslab, (size_t)BM * SLAB * 2));
    ANN_CUDA(bufs.alloc(&norm, (size_t)N * 4));
    ANN_CUDA(bufs.alloc(&limit, (size_t)N * 4));
    ANN_CUDA(bufs.alloc(&ids, (size_t)N * 4));
    ANN_CUDA(bufs.alloc(&err, sizeof(int)));
    ANN_CUDA(bufs.alloc(&pend, (size_t)nsm * 8 * CAP * 32 * sizeof(float4)));
    ANN_CUDA(bufs.alloc(&pend_col, (size_t)nsm * 8 * CAP * 32 * 4));
    ANN_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s));
    query_slab_kernel<<<(BM * SLAB + 255) / 256, 256, 0, s>>>(qslab);
    ANN_CUDA(cudaGetLastError());
    return ANN_OK;
}

int LeafTc::round(const uint8_t *X, const uint64_t *order, uint64_t idmask, const uint64_t *graph, cudaStream_t s) {
    using namespace tc;
    const int tpr = d / 4;
    prep_rows_kernel<<<(unsigned)((N * tpr + 255) / 256), 256, 0, s>>>(X, N, d, rb, norm, rslab, order, idmask, graph, R,
                                                                       ids, limit);
    CUtensorMap m[4];
    int r = make_map(&m[0], rb, N, d, BM);
    if (r == ANN_OK) r = make_map(&m[1], qslab, BM, SLAB, BM);
    if (r == ANN_OK) r = make_map(&m[2], rb, N, d, BN);
    if (r == ANN_OK) r = make_map(&m[3], rslab, N, SLAB, BN);
    if (r != ANN_OK) return r;
    const int64_t largest = (N + (1ll << levels) - 1) >> levels;
    const int blocks = (int)((largest + BM - 1) / BM);
    Params prm{N, N, d, R, 1, 1, levels, blocks, ids, norm, limit, lists, pend, pend_col, err};
    const unsigned grid = (unsigned)std::min<int64_t>((int64_t)blocks << levels, nsm);
    const cudaError_t e = launch_tc<true>(grid, smem_bytes(d), s, m, prm);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(knn_tc_kernel)");
    ANN_CUDA(cudaGetLastError());
    return ANN_OK;
}

}  // namespace ann

// ann_search.cu -- host side of Algorithm 1 (Sec. 4.2): launch planning, the
// plain, persistent (CUDA graph, autotuned) forms and the C entry point.  The
// device code is in ann_search_dev.cuh.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <map>
#include <memory>
#include <mutex>
#include <set>
#include <tuple>
#include <vector>

#include "ann_search_dev.cuh"

namespace ann {

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static int g_num_sms = 0;
static size_t g_smem_optin = 0;

static int device_props() {
    if (g_num_sms) return ANN_OK;
    int dev;
    ANN_CUDA(cudaGetDevice(&dev));
    cudaDeviceProp prop;
    ANN_CUDA(cudaGetDeviceProperties(&prop, dev));
    g_num_sms = prop.multiProcessorCount;
    g_smem_optin = prop.sharedMemPerBlockOptin;
    // stream-ordered scratch allocations reuse the pool instead of returning memory at every sync
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
        uint64_t keep = ~0ull;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    }
    return ANN_OK;
}

// Budgets from this size on, in launches with more queries than fit otherwise,
// keep the queue's overflow and the visited set in per-warp global scratch, so
// the shared-memory slice of a query no longer grows with its budget.
static const int kWindowedFromT = 1024;

// Launch shape of the main loop for a budget bucket.
struct Tune {
    int warps;                         // per CTA
    bool stage;                        // stage the next pop's neighbour vectors (cp.async)
    int spill_heap = (int)kSpillHeap;  // large budgets: queue entries kept in shared memory
};

// The dynamic shared-memory limit of a kernel is a property of the function,
// read again whenever a launch (or a graph node) is checked, so it is raised
// once to the device's opt-in maximum rather than set per launch: a captured
// graph may hold nodes of one kernel with different sizes.
template <class F>
static cudaError_t occupancy_of(F kernel, bool &raised, size_t smem, int threads, int *blocks_per_sm) {
    if (!raised) {
        cudaError_t e =
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g_smem_optin);
        if (e != cudaSuccess) return e;
        raised = true;
    }
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kernel, threads, smem);
}

// main_kernel of a type, a layout and a register budget, as fn(kernel, index)
template <class Fn>
static auto with_main(int dtype, bool sp, bool wide, Fn fn) {
    if (dtype == ANN_U8) {
        if (sp && wide) return fn(main_kernel<ANN_U8, true, kMainCtasWide>, 0);
        return sp ? fn(main_kernel<ANN_U8, true, kMainCtas>, 1) : fn(main_kernel<ANN_U8, false, kMainCtas>, 2);
    }
    return sp ? fn(main_kernel<ANN_F32, true, kMainCtas>, 3) : fn(main_kernel<ANN_F32, false, kMainCtas>, 4);
}

static cudaError_t main_occupancy(int dtype, bool sp, bool wide, size_t smem, int threads, int *blocks) {
    static bool raised[5] = {};
    return with_main(dtype, sp, wide,
                     [&](auto kernel, int i) { return occupancy_of(kernel, raised[i], smem, threads, blocks); });
}

static cudaError_t resume_occupancy(const DevIndex &ix, bool sp, size_t smem, int threads, int *blocks) {
    static bool raised[4] = {};
    if (ix.ngroups > 0) return config_grouped(ix.dtype, sp, smem, threads, blocks);
    if (ix.dtype == ANN_U8)
        return sp ? occupancy_of(resume_kernel<ANN_U8, true, false>, raised[0], smem, threads, blocks)
                  : occupancy_of(resume_kernel<ANN_U8, false, false>, raised[1], smem, threads, blocks);
    return sp ? occupancy_of(resume_kernel<ANN_F32, true, false>, raised[2], smem, threads, blocks)
              : occupancy_of(resume_kernel<ANN_F32, false, false>, raised[3], smem, threads, blocks);
}

static cudaError_t prologue_occupancy(const DevIndex &ix, size_t smem, int threads, int *blocks) {
    static bool raised[2] = {};
    if (ix.ngroups > 0) return config_grouped_prologue(ix.dtype, smem, threads, blocks);
    return ix.dtype == ANN_U8 ? occupancy_of(prologue_kernel<ANN_U8, false>, raised[0], smem, threads, blocks)
                              : occupancy_of(prologue_kernel<ANN_F32, false>, raised[1], smem, threads, blocks);
}

// one kernel of a search: its layout and launch shape
struct Shape {
    WarpLayout L;
    dim3 grid, block;
    size_t smem = 0;
    int warps = 0;  // resident warps at most
};

// The shape that keeps the most warps resident for slices of L.total bytes
// (ties go to more warps per CTA), for `count` queries at most: few queries
// spread over the SMs one warp to a CTA.  waves > 1: more CTAs than fit.
template <class Occ>
static int fit_shape(Shape &sh, int max_warps, int64_t count, int waves, Occ occ) {
    if (sh.L.total > g_smem_optin) return fail(ANN_ERR_CAPACITY, "per-query state exceeds shared memory");
    const int64_t spread = (count + g_num_sms - 1) / g_num_sms;
    if (max_warps > spread) max_warps = (int)std::max<int64_t>(1, spread);
    int best = 0, best_w = 1, best_blocks = 1;
    for (int w = 1; w <= max_warps; w++) {
        const size_t smem = (size_t)w * sh.L.total;
        if (smem > g_smem_optin) break;
        int blocks = 0;
        const cudaError_t e = occ(smem, 32 * w, &blocks);
        if (e != cudaSuccess) return cuda_fail(e, "search kernel configuration");
        if (blocks * w >= best) {
            best = blocks * w;
            best_w = w;
            best_blocks = std::max(1, blocks);
        }
    }
    int64_t grid = std::min<int64_t>((count + best_w - 1) / best_w, (int64_t)g_num_sms * best_blocks * waves);
    if (grid < 1) grid = 1;
    sh.grid = dim3((unsigned)grid);
    sh.block = dim3(32 * best_w);
    sh.smem = (size_t)best_w * sh.L.total;
    sh.warps = (int)std::min<int64_t>(grid, (int64_t)g_num_sms * best_blocks) * best_w;
    return ANN_OK;
}

// Launch configuration of one search: its three kernels and their workspace.
struct LaunchCfg {
    SearchArgs A;
    Shape pro, main, res;
    uint64_t main_stride, res_stride;  // global scratch per warp (large budgets)
    uint64_t main_spill, main_hash, res_spill, res_hash;
    bool win, wide;
    bool whole;                        // resume_kernel alone
    int64_t total, chunk;              // queries, and queries per pass over the three kernels
    // offsets into the workspace
    size_t o_rec, o_bk, o_bi, o_susp, o_save, o_scratch, bytes;
};

// A pass holds the records and first bridge batches of at most kChunk queries
// (4.7 KB each), and states of suspended ones up to kSaveBytes; queries
// that find no room there start again when they are resumed.  Where the device
// has no room for that, passes and states are a quarter as large (`shrink`
// times over), down to 128 queries: 7 MB for budgets below 1024, 40 MB for the
// largest (the scratch of as many warps).
static const int64_t kChunk = 32768;
static const size_t kSaveBytes = (size_t)256 << 20;
static const int kMaxShrink = 4;

static int plan_launch(const SearchArgs &base, int capT, const int32_t *list, const int32_t *list_count,
                       int64_t list_len, LaunchCfg &cfg, const Tune *tune = nullptr, int shrink = 0) {
    // the buckets of a batch (their counts are on the device) share its queries
    const size_t save_bytes = (list_count ? kSaveBytes / 4 : kSaveBytes) >> (2 * shrink);
    SearchArgs A = base;
    const DevIndex &ix = A.ix;
    const bool grouped = ix.ngroups > 0;
    const Tune tn = tune ? *tune : Tune{kMainWarps, true, (int)kSpillHeap};
    // Large budgets keep the queue's tail and the visited set in global memory
    // so that an SM holds more queries; while all queries of the launch are
    // resident with everything in shared memory, that is the shorter chain (no
    // visited-set probe in L2 at every step): 128 queries of SIFT-shaped rows,
    // T = 1024 / 2048 / 4096: 0.88 / 2.58 / 17.3 -> 0.68 / 2.05 / 14.3 ms.
    // (the form of a launch does not depend on how its main loop is tuned)
    cfg.main.L = main_layout(ix.dtype, ix.d, capT, A.kmax, ix.b, ix.R, true, false, (uint32_t)tn.spill_heap);
    const int64_t fit = (int64_t)(g_smem_optin / (cfg.main.L.total + 1024)) * g_num_sms;
    // bridge batch: budgets below the windowed kernels pop few bridges
    auto res_layout = [&](bool w, bool split) {
        return make_layout(ix.dtype, ix.d, ix.P, ix.n, ix.PA, capT, A.kmax, w ? 128 : 64, ix.b, ix.R, true, grouped, w,
                           (uint32_t)tn.spill_heap, split);
    };
    const bool win =
        capT >= kWindowedFromT && (list_len > fit || res_layout(false, false).total > g_smem_optin);
    A.capT = capT;
    A.bcap = win ? 128 : 64;
    A.bstore = (int)(kFirstEnough + kFirstCap);
    A.list = list;
    A.list_count = list_count;
    A.list_len = list_len;
    cfg.win = win;
    cfg.wide = list_len > (int64_t)g_num_sms * kMainWarps * kMainCtas;
    cfg.total = list_len;
    cfg.chunk = std::min(list_len, kChunk >> (2 * shrink));
    cfg.pro.L = prologue_layout(ix.dtype, ix.d, ix.P, ix.n, ix.PA, (int)kFirstCap, grouped, win);
    cfg.main.L = main_layout(ix.dtype, ix.d, capT, A.kmax, ix.b, ix.R, tn.stage, win, (uint32_t)tn.spill_heap);
    cfg.res.L = res_layout(win, true);
    if (cfg.res.L.total > g_smem_optin) cfg.res.L = res_layout(win, false);
    // rows so wide (float32 from about 20,000 dimensions) that a query fills an
    // SM: what holds it leanest runs it alone
    const bool lean = cfg.pro.L.total > g_smem_optin || cfg.main.L.total > g_smem_optin;
    int r = ANN_OK;
    if (!lean)
        r = fit_shape(cfg.pro, 4, cfg.chunk, 8, [&](size_t smem, int threads, int *blocks) {
            return prologue_occupancy(ix, smem, threads, blocks);
        });
    if (r == ANN_OK && !lean)
        r = fit_shape(cfg.main, tn.warps, cfg.chunk, 1, [&](size_t smem, int threads, int *blocks) {
            return main_occupancy(ix.dtype, win, cfg.wide, smem, threads, blocks);
        });
    if (r == ANN_OK)
        r = fit_shape(cfg.res, 6, cfg.chunk, 1, [&](size_t smem, int threads, int *blocks) {
            return resume_occupancy(ix, win, smem, threads, blocks);
        });
    if (r != ANN_OK) return r;
    // One kernel while it holds all queries at once: the others only pay when
    // there are more queries than that, and a suspended one would come after
    // all that were not.  SIFT-shaped rows, P = 2 x n = 64, 600 queries, T = 64 /
    // 256 / 2048: three kernels 232 / 298 / 1406 us, one 207 / 252 / 1186 us.
    cfg.whole = lean || cfg.res.warps >= list_len;
    A.whole = cfg.whole;
    auto al = [](uint64_t x) { return (x + 255) & ~(uint64_t)255; };
    // A sorted window serves many batches of bridges, and has no use for more
    // than a budget of that size can pop: 1024 entries at least, sorted in global
    // memory, made 300 queries of T = 64 (3 x 32 dictionaries, GIST-shaped) 0.77 ms,
    // 192 (what a walk can trim) 0.53.
    const uint32_t gcap = (uint32_t)std::min(8192, std::max(192, 2 * capT));
    A.gcap = gcap;
    // per-warp scratch: the queue's overflow, then the visited set; the
    // resuming kernel's starts with its sorted bridge windows
    const uint64_t spill = al(8ull * (uint64_t)capT), hash = al(4ull * cfg.main.L.hash_slots);
    cfg.main_spill = 0;
    cfg.main_hash = spill;
    cfg.main_stride = win ? spill + hash : 0;
    cfg.res_spill = al((uint64_t)gcap * 24);
    cfg.res_hash = cfg.res_spill + spill;
    cfg.res_stride = win ? cfg.res_hash + hash : cfg.res_spill;
    // a suspended query's state
    A.save_rbuf = kSaveHeader;
    A.save_heap = A.save_rbuf + (A.kmax > 32 ? 8u * (uint32_t)A.kmax : 0u);
    A.save_hash = align_up(A.save_heap + 8u * cfg.main.L.heap_cap, 16);
    A.save_spill = A.save_hash + 4u * cfg.main.L.hash_slots;
    A.save_stride = al(A.save_spill + (win ? 8ull * (uint64_t)capT : 0ull));
    A.nslots = (uint32_t)std::min<int64_t>(cfg.chunk, (int64_t)(save_bytes / A.save_stride));
    size_t o = 256;  // counters
    // records, first batches and states are the three kernels' only
    const size_t held = cfg.whole ? 0 : (size_t)cfg.chunk;
    cfg.o_rec = o;   o = al(o + sizeof(QRec) * held);
    cfg.o_bk = o;    o = al(o + 8 * (size_t)A.bstore * held);
    cfg.o_bi = o;    o = al(o + 4 * (size_t)A.bstore * held);
    cfg.o_susp = o;  o = al(o + 4 * held);
    cfg.o_save = o;  o = al(o + (cfg.whole ? 0 : (size_t)A.nslots * A.save_stride));
    cfg.o_scratch = o;
    o = al(o + std::max(cfg.whole ? 0 : cfg.main.warps * cfg.main_stride, cfg.res.warps * cfg.res_stride));
    cfg.bytes = o;
    cfg.A = A;
    return ANN_OK;
}

// the kernels of every pass over the queries: number first .. last of the three,
// or the resuming one alone
static int do_launch(LaunchCfg &cfg, uint8_t *ws, cudaStream_t stream, int first = 0, int last = 2) {
    SearchArgs &A = cfg.A;
    const bool u8 = A.ix.dtype == ANN_U8, grouped = A.ix.ngroups > 0;
    A.counters = (int32_t *)ws;
    A.rec = (QRec *)(ws + cfg.o_rec);
    A.bkeys = (uint64_t *)(ws + cfg.o_bk);
    A.bidxs = (uint32_t *)(ws + cfg.o_bi);
    A.susp = (int32_t *)(ws + cfg.o_susp);
    A.save = ws + cfg.o_save;
    A.gscratch = ws + cfg.o_scratch;
    A.chunk = cfg.chunk;
    for (A.base = 0; A.base < cfg.total; A.base += cfg.chunk) {
        if (cfg.whole) first = last = 2;
        if (first <= 0) {
            const Shape &s = cfg.pro;
            A.L = s.L;
            if (grouped) launch_grouped_prologue(A.ix.dtype, s.grid, s.block, s.smem, stream, A);
            else if (u8) prologue_kernel<ANN_U8, false><<<s.grid, s.block, s.smem, stream>>>(A);
            else prologue_kernel<ANN_F32, false><<<s.grid, s.block, s.smem, stream>>>(A);
        }
        if (first <= 1 && last >= 1) {
            const Shape &s = cfg.main;
            A.L = s.L;
            A.spill_off = cfg.main_spill;
            A.hash_off = cfg.main_hash;
            A.wstride = cfg.main_stride;
            with_main(A.ix.dtype, cfg.win, cfg.wide, [&](auto kernel, int) {
                kernel<<<s.grid, s.block, s.smem, stream>>>(A);
                return 0;
            });
        }
        if (last >= 2) {
            const Shape &s = cfg.res;
            A.L = s.L;
            A.spill_off = cfg.res_spill;
            A.hash_off = cfg.res_hash;
            A.wstride = cfg.res_stride;
            if (grouped) {
                launch_grouped(A.ix.dtype, cfg.win, s.grid, s.block, s.smem, stream, A);
            } else if (u8) {
                if (cfg.win) resume_kernel<ANN_U8, true, false><<<s.grid, s.block, s.smem, stream>>>(A);
                else resume_kernel<ANN_U8, false, false><<<s.grid, s.block, s.smem, stream>>>(A);
            } else {
                if (cfg.win) resume_kernel<ANN_F32, true, false><<<s.grid, s.block, s.smem, stream>>>(A);
                else resume_kernel<ANN_F32, false, false><<<s.grid, s.block, s.smem, stream>>>(A);
            }
        }
    }
    ANN_CUDA(cudaGetLastError());
    return ANN_OK;
}

// plan + stream-ordered workspace + launch
static int launch_search(const SearchArgs &base, int capT, cudaStream_t stream, const int32_t *list,
                         int64_t list_len) {
    for (int shrink = 0;; shrink++) {
        LaunchCfg cfg;
        int r = plan_launch(base, capT, list, nullptr, list_len, cfg, nullptr, shrink);
        if (r != ANN_OK) return r;
        uint8_t *ws = nullptr;
        const cudaError_t e = cudaMallocAsync((void **)&ws, cfg.bytes, stream);
        if (e != cudaSuccess) {
            r = cuda_fail(e, "cudaMallocAsync(search workspace)");
            if (r == ANN_ERR_OOM && shrink < kMaxShrink) continue;
            return r;
        }
        r = do_launch(cfg, ws, stream);
        cudaFreeAsync(ws, stream);
        return r;
    }
}

__global__ void max_kernel(const int32_t *v, int64_t n, int32_t *out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) atomicMax(out, v[i]);
}

// ---- persistent mode: bucket queries by budget on the device ----
static const int kBuckets = 7;  // capT = 128 << i  (128 .. 8192)

__global__ void bucket_kernel(int64_t nq, const int32_t *T, int32_t T_all, int32_t *counts, int32_t *lists) {
    // counts[kBuckets], lists[kBuckets * nq]
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nq) return;
    int t = T ? T[i] : T_all;
    int bkt = 0;
    while (bkt < kBuckets - 1 && t > (128 << bkt)) bkt++;
    int pos = atomicAdd(&counts[bkt], 1);
    lists[(int64_t)bkt * nq + pos] = (int32_t)i;
}

// Device memory that the kernels of recorded plans work in.  The plans of one
// stream share it: they run one after another, which `done`, recorded behind
// every launch, also ensures where a stream's handle does not (a handle that
// was destroyed and given out again, the per-thread default stream).
struct Workspace {
    uint8_t *p = nullptr;
    size_t bytes = 0;
    cudaEvent_t done = nullptr;
    const void *last = nullptr;  // the graph launched last
    ~Workspace() {
        if (done) cudaEventDestroy(done);
        if (p) cudaFree(p);
    }
};

struct Plan {
    cudaGraphExec_t exec = nullptr;
    int32_t *scratch = nullptr;     // counts[kBuckets], lists[kBuckets*nq], then a word for autotune()
    std::shared_ptr<Workspace> ws;  // the buckets' workspaces, one after another
    uint64_t last_use = 0;          // for evicting the least recently used plan
};

// plans kept per index, and bytes of their workspaces; beyond either the least
// recently used ones go
static const size_t kMaxPlans = 32, kMaxPlanBytes = (size_t)16 << 30;

struct PlanKey {
    const void *queries;
    int64_t nq;
    const int32_t *k, *T;
    int32_t k_all, T_all, kmax;
    int32_t *out_ids;
    void *out_keys;
    int32_t *out_status;
    int64_t *out_stats;
    cudaStream_t stream;
    bool operator<(const PlanKey &o) const {
        return std::tie(queries, nq, k, T, k_all, T_all, kmax, out_ids, out_keys, out_status, out_stats, stream) <
               std::tie(o.queries, o.nq, o.k, o.T, o.k_all, o.T_all, o.kmax, o.out_ids, o.out_keys, o.out_status,
                        o.out_stats, o.stream);
    }
};

struct PlanCache {
    std::mutex mu;
    uint64_t clock = 0;
    std::map<PlanKey, Plan> plans;
    // measured best launch shape of (bucket capacity, kmax, LaunchCfg::win, LaunchCfg::wide)
    std::map<std::tuple<int, int, bool, bool>, Tune> tuned;
};

void free_plans(ann_index *ix) {
    if (!ix->plans) return;
    PlanCache *pc = (PlanCache *)ix->plans;
    for (auto &kv : pc->plans) {
        if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
        if (kv.second.scratch) cudaFree(kv.second.scratch);
    }
    delete pc;
    ix->plans = nullptr;
}

// bytes of the distinct workspaces of an index's plans
static size_t held_bytes(const PlanCache *pc) {
    std::set<const Workspace *> seen;
    size_t b = 0;
    for (auto &kv : pc->plans)
        if (seen.insert(kv.second.ws.get()).second) b += kv.second.ws->bytes;
    return b;
}

// a workspace of at least `need` bytes that a plan of this stream has already
static std::shared_ptr<Workspace> workspace_of(const PlanCache *pc, cudaStream_t s, size_t need) {
    for (auto &kv : pc->plans)
        if (kv.first.stream == s && kv.second.ws->bytes >= need) return kv.second.ws;
    return nullptr;
}

// The least recently used plan goes, once what was launched in its workspace
// has finished (its stream may be gone).
static int evict_plan(PlanCache *pc) {
    auto old = pc->plans.begin();
    for (auto it = pc->plans.begin(); it != pc->plans.end(); ++it)
        if (it->second.last_use < old->second.last_use) old = it;
    ANN_CUDA(cudaEventSynchronize(old->second.ws->done));
    old->second.ws->last = nullptr;  // nothing left to wait for, and the graph's address may come back
    cudaGraphExecDestroy(old->second.exec);
    cudaFree(old->second.scratch);
    pc->plans.erase(old);
    return ANN_OK;
}

// budgets of the buckets one persistent batch may use
static void bucket_range(const int32_t *T, int32_t T_all, int &b0, int &b1) {
    b1 = kBuckets - 1;
    if (!T) {
        b1 = 0;
        while (b1 < kBuckets - 1 && T_all > (128 << b1)) b1++;
    }
    b0 = T ? 0 : b1;
}

static int bucket_cap(int bkt) { return (128 << bkt) > kMaxT ? kMaxT : (128 << bkt); }

// the budget a bucket's kernels are sized for: a uniform one is known
static int sized_for(int bkt, const int32_t *T, int32_t T_all) {
    return T ? bucket_cap(bkt) : std::max(32, std::min((int)T_all, bucket_cap(bkt)));
}

// the main loop's launch shape that was measured for a bucket run in cfg's form
static Tune *tuned_for(PlanCache *pc, int bkt, const LaunchCfg &cfg) {
    auto it = pc->tuned.find({bucket_cap(bkt), cfg.A.kmax, cfg.win, cfg.wide});
    return it == pc->tuned.end() ? nullptr : &it->second;
}

// streams and events of the fork/join; they must outlive the capture
struct ForkSet {
    cudaStream_t side[kBuckets] = {};
    cudaEvent_t fork = nullptr, join[kBuckets] = {};
    int nside = 0;
    ~ForkSet() {
        for (int i = 0; i < nside; i++) {
            if (join[i]) cudaEventDestroy(join[i]);
            if (side[i]) cudaStreamDestroy(side[i]);
        }
        if (fork) cudaEventDestroy(fork);
    }
};

// one bucket's launch, in its measured shape if it has one: the whole batch in
// order, or (per-query T) its list
static int plan_bucket(PlanCache *pc, const SearchArgs &A, int64_t nq, const int32_t *T, int32_t T_all,
                       int32_t *scratch, int bkt, LaunchCfg &cfg, int shrink) {
    const int capT = sized_for(bkt, T, T_all);
    const int32_t *list = T ? scratch + kBuckets + (int64_t)bkt * nq : nullptr, *count = T ? scratch + bkt : nullptr;
    int r = plan_launch(A, capT, list, count, nq, cfg, nullptr, shrink);
    if (r != ANN_OK || cfg.whole) return r;
    const Tune *tn = tuned_for(pc, bkt, cfg);
    return tn ? plan_launch(A, capT, list, count, nq, cfg, tn, shrink) : ANN_OK;
}

// One replay of the persistent form.  A uniform budget is one bucket and the
// queries are taken in order; otherwise a device pass sorts them into buckets
// first.  The buckets run concurrently on forked streams (largest budget
// first), each with a workspace of its own: a bucket's last queries leave most
// SMs idle, above all those that pop many bridges.
static int record_persistent(PlanCache *pc, const SearchArgs &A, int64_t nq, const int32_t *T, int32_t T_all,
                             int32_t *scratch, uint8_t *wscratch, size_t wbytes, int shrink, cudaStream_t s,
                             ForkSet &fs) {
    int32_t *counts = scratch, *lists = scratch + kBuckets;
    if (T) {
        ANN_CUDA(cudaMemsetAsync(counts, 0, sizeof(int32_t) * kBuckets, s));
        bucket_kernel<<<(unsigned)((nq + 255) / 256), 256, 0, s>>>(nq, T, T_all, counts, lists);
        ANN_CUDA(cudaGetLastError());
    }
    int b0, b1;
    bucket_range(T, T_all, b0, b1);
    int rc = ANN_OK;
    for (int bkt = b1; bkt >= b0 && rc == ANN_OK; bkt--) {
        LaunchCfg cfg;
        rc = plan_bucket(pc, A, nq, T, T_all, scratch, bkt, cfg, shrink);
        if (rc != ANN_OK) break;
        if (cfg.bytes > wbytes) {
            rc = fail(ANN_ERR_CAPACITY, "search workspace smaller than its kernels need");
            break;
        }
        uint8_t *ws = wscratch;
        wscratch += cfg.bytes;
        wbytes -= cfg.bytes;
        if (b0 == b1) {
            rc = do_launch(cfg, ws, s);
            continue;
        }
        if (!fs.fork) {
            if (cudaEventCreateWithFlags(&fs.fork, cudaEventDisableTiming) != cudaSuccess ||
                cudaEventRecord(fs.fork, s) != cudaSuccess) {
                rc = cuda_fail(cudaGetLastError(), "fork event");
                break;
            }
        }
        const int i = fs.nside;
        if (cudaStreamCreateWithFlags(&fs.side[i], cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&fs.join[i], cudaEventDisableTiming) != cudaSuccess) {
            rc = cuda_fail(cudaGetLastError(), "side stream");
            break;
        }
        fs.nside++;
        if (cudaStreamWaitEvent(fs.side[i], fs.fork, 0) != cudaSuccess) {
            rc = cuda_fail(cudaGetLastError(), "fork");
            break;
        }
        rc = do_launch(cfg, ws, fs.side[i]);
        if (rc != ANN_OK) break;
        if (cudaEventRecord(fs.join[i], fs.side[i]) != cudaSuccess || cudaStreamWaitEvent(s, fs.join[i], 0) != cudaSuccess) {
            rc = cuda_fail(cudaGetLastError(), "join");
            break;
        }
    }
    return rc;
}

// Launch shapes of the main loop worth measuring for a bucket: as many warps
// per CTA as the kernel takes, fewer (finer granularity), without cp.async
// staging, and, for large budgets, other shared-memory heap capacities (a
// smaller heap leaves room for more resident queries, a larger one moves
// entries out less often).  All give identical results.
static std::vector<Tune> tune_candidates(int capT, bool win) {
    std::vector<Tune> c{Tune{kMainWarps, true}, Tune{kMainWarps / 2, true}, Tune{kMainWarps, false}};
    if (win)
        for (int hc : {256, 1024})
            if (hc < capT) c.push_back(Tune{kMainWarps, true, hc});
    return c;
}

// Measure the candidates of every bucket this batch fills whose form has no
// measured choice yet, on (a prefix of) the batch itself, and keep the fastest.
// They are planned as the replay will be, for the batch's size; a device count
// keeps a run to its share of the queries.
static int autotune(PlanCache *pc, const SearchArgs &A, int64_t nq, const int32_t *T, int32_t T_all,
                    int32_t *scratch, cudaStream_t s) {
    int b0, b1;
    bucket_range(T, T_all, b0, b1);
    LaunchCfg c0[kBuckets];  // the default shapes
    bool todo[kBuckets] = {}, any = false;
    for (int bkt = b0; bkt <= b1; bkt++) {
        const int r = plan_launch(A, sized_for(bkt, T, T_all), nullptr, nullptr, nq, c0[bkt]);
        if (r != ANN_OK) return r;
        todo[bkt] = !c0[bkt].whole && !tuned_for(pc, bkt, c0[bkt]);  // whole: the main loop's shape is not used
        any |= todo[bkt];
    }
    if (!any) return ANN_OK;
    int32_t *counts = scratch, *lists = scratch + kBuckets, *tcount = lists + (int64_t)kBuckets * nq;
    int32_t hc[kBuckets] = {0};
    if (T) {
        ANN_CUDA(cudaMemsetAsync(counts, 0, sizeof(int32_t) * kBuckets, s));
        bucket_kernel<<<(unsigned)((nq + 255) / 256), 256, 0, s>>>(nq, T, T_all, counts, lists);
        ANN_CUDA(cudaGetLastError());
        ANN_CUDA(cudaMemcpyAsync(hc, counts, sizeof(hc), cudaMemcpyDeviceToHost, s));
        ANN_CUDA(cudaStreamSynchronize(s));
    } else {
        hc[b1] = (int32_t)nq;
    }
    cudaEvent_t e0, e1;
    ANN_CUDA(cudaEventCreate(&e0));
    ANN_CUDA(cudaEventCreate(&e1));
    int rc = ANN_OK;
    for (int bkt = b0; bkt <= b1 && rc == ANN_OK; bkt++) {
        // a list shorter than one round of the resident warps takes as long as its
        // longest queries in every shape (2,000 GIST-shaped queries over seven
        // buckets: 26 ms, 315 ms to measure them, 26 ms after): left open
        if (!todo[bkt] || (T && hc[bkt] < c0[bkt].main.warps)) continue;
        const int capT = sized_for(bkt, T, T_all);
        const std::vector<Tune> cands = tune_candidates(capT, c0[bkt].win);
        const int32_t *list = T ? lists + (int64_t)bkt * nq : nullptr;
        // tune on up to four rounds of the default shape's resident warps
        const int32_t ntune = (int32_t)std::min<int64_t>(std::min<int64_t>(hc[bkt], c0[bkt].chunk),
                                                         4 * (int64_t)c0[bkt].main.warps);
        if (cudaMemcpyAsync(tcount, &ntune, sizeof(ntune), cudaMemcpyHostToDevice, s) != cudaSuccess) {
            rc = cuda_fail(cudaGetLastError(), "autotune count");
            break;
        }
        float best_ms = 0.f;
        int best = -1;
        for (size_t ci = 0; ci < cands.size() && rc == ANN_OK; ci++) {
            LaunchCfg cfg;
            if (plan_launch(A, capT, list, tcount, nq, cfg, &cands[ci]) != ANN_OK || cfg.whole) continue;
            cfg.total = cfg.chunk;  // the run's queries are in the first pass
            uint8_t *ws = nullptr;
            if (cudaMallocAsync((void **)&ws, cfg.bytes, s) != cudaSuccess) continue;
            float ms_min = 0.f;
            for (int rep = 0; rep < 2 && rc == ANN_OK; rep++) {
                rc = do_launch(cfg, ws, s, 0, 0);
                cudaEventRecord(e0, s);
                if (rc == ANN_OK) rc = do_launch(cfg, ws, s, 1, 1);
                cudaEventRecord(e1, s);
                if (rc != ANN_OK) break;
                cudaError_t ce = cudaEventSynchronize(e1);
                if (ce != cudaSuccess) {
                    rc = cuda_fail(ce, "autotune run");
                    break;
                }
                float ms = 0.f;
                cudaEventElapsedTime(&ms, e0, e1);
                if (rep == 0 || ms < ms_min) ms_min = ms;
                if (ms > 50.f) break;  // long runs: one measurement is enough
            }
            cudaFreeAsync(ws, s);
            if (rc == ANN_OK && ms_min > 0.f && (best < 0 || ms_min < best_ms)) {
                best_ms = ms_min;
                best = (int)ci;
            }
        }
        cudaGetLastError();  // a candidate that failed to configure is simply not chosen
        if (rc == ANN_OK && best >= 0)
            pc->tuned[{bucket_cap(bkt), A.kmax, c0[bkt].win, c0[bkt].wide}] = cands[best];
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return rc;
}

int search_launch_list(const ann_index *ix, const void *queries, int64_t nq, const int32_t *k, const int32_t *T,
                       int32_t kmax, int capT, const int32_t *list, int64_t count, int32_t *out_ids, void *out_keys,
                       int32_t *out_status, cudaStream_t stream) {
    int r = device_props();
    if (r != ANN_OK) return r;
    if (nq == 0 || count == 0) return ANN_OK;
    SearchArgs A{};
    A.ix = ix->dev;
    A.queries = queries;
    A.nq = nq;
    A.k = k;
    A.T = T;
    A.kmax = kmax;
    A.out_ids = out_ids;
    A.out_keys = out_keys;
    A.out_status = out_status;
    if (capT > kMaxT) capT = kMaxT;
    if (capT < 32) capT = 32;
    return launch_search(A, capT, stream, list, count);
}

int search_bucket_of(int32_t T) {
    int b = 0;
    while (b < kBuckets - 1 && T > (128 << b)) b++;
    return b;
}

int search_bucket_cap(int bucket) { return bucket_cap(bucket); }

int search_num_buckets() { return kBuckets; }

}  // namespace ann

using namespace ann;

extern "C" int ann_search_batch(const ann_index *index, const void *queries, int64_t nq, const int32_t *k,
                                const int32_t *T, int32_t k_all, int32_t T_all, int32_t kmax, int32_t mode,
                                int32_t *out_ids, void *out_keys, int32_t *out_status, int64_t *out_stats,
                                void *stream) {
    ANN_ARG(index != nullptr, "index is NULL");
    ANN_ARG(nq >= 0 && nq < (1ll << 31), "nq out of range");
    ANN_ARG(kmax >= 1 && kmax <= kMaxK, "kmax must be in [1, 128]");
    ANN_ARG(mode == ANN_MODE_PLAIN || mode == ANN_MODE_PERSISTENT, "mode must be 0 (plain) or 1 (persistent)");
    ANN_ARG(nq == 0 || (queries && out_ids), "queries and out_ids are required");
    ANN_ARG(((uintptr_t)queries & 15) == 0, "queries must be 16-byte aligned");
    if (!k) ANN_ARG(k_all >= 0 && k_all <= kmax, "k_all must be in [0, kmax]");
    if (!T) ANN_ARG(T_all >= 0 && T_all <= kMaxT, "T_all must be in [0, 8192]");
    int r = device_props();
    if (r != ANN_OK) return r;
    if (nq == 0) return ANN_OK;
    cudaStream_t s = (cudaStream_t)stream;
    SearchArgs A{};
    A.ix = index->dev;
    A.queries = queries;
    A.nq = nq;
    A.k = k;
    A.T = T;
    A.k_all = k_all;
    A.T_all = T_all;
    A.kmax = kmax;
    A.out_ids = out_ids;
    A.out_keys = out_keys;
    A.out_status = out_status;
    A.out_stats = out_stats;
    if (mode == ANN_MODE_PLAIN) {
        // sized for the largest budget in the batch
        int capT = T_all;
        if (T) {
            int32_t *dmax = nullptr, hmax = 0;
            AsyncBufs bufs(s);  // released at the end of this block
            ANN_CUDA(bufs.alloc(&dmax, sizeof(int32_t)));
            ANN_CUDA(cudaMemsetAsync(dmax, 0, sizeof(int32_t), s));
            max_kernel<<<(unsigned)((nq + 255) / 256), 256, 0, s>>>(T, nq, dmax);
            ANN_CUDA(cudaMemcpyAsync(&hmax, dmax, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
            ANN_CUDA(cudaStreamSynchronize(s));
            capT = hmax;
        }
        if (capT > kMaxT) capT = kMaxT;
        if (capT < 32) capT = 32;
        return launch_search(A, capT, s, nullptr, nq);
    }
    // persistent: bucket by budget, the buckets' kernels side by side, replayed as a CUDA graph
    ann_index *ixm = const_cast<ann_index *>(index);
    if (!ixm->plans) ixm->plans = new PlanCache();
    PlanCache *pc = (PlanCache *)ixm->plans;
    PlanKey key{queries, nq, k, T, k_all, T_all, kmax, out_ids, out_keys, out_status, out_stats, s};
    std::lock_guard<std::mutex> g(pc->mu);
    auto it = pc->plans.find(key);
    if (it == pc->plans.end() && pc->plans.size() >= kMaxPlans) {
        const int er = evict_plan(pc);
        if (er != ANN_OK) return er;
    }
    if (it == pc->plans.end()) {
        Plan p;
        ANN_CUDA(cudaMalloc(&p.scratch, sizeof(int32_t) * (kBuckets + (size_t)kBuckets * nq + 1)));
        auto drop = [&p](int code) {
            cudaFree(p.scratch);
            return code;
        };
        r = autotune(pc, A, nq, T, T_all, p.scratch, s);
        if (r != ANN_OK) return drop(r);
        int b0, b1, shrink = 0;
        bucket_range(T, T_all, b0, b1);
        for (;; shrink++) {
            size_t need = 0;
            for (int bkt = b0; bkt <= b1; bkt++) {
                LaunchCfg cfg;
                r = plan_bucket(pc, A, nq, T, T_all, p.scratch, bkt, cfg, shrink);
                if (r != ANN_OK) return drop(r);
                need += cfg.bytes;
            }
            p.ws = workspace_of(pc, s, need);
            if (p.ws) break;
            while (held_bytes(pc) + need > kMaxPlanBytes && !pc->plans.empty())
                if ((r = evict_plan(pc)) != ANN_OK) return drop(r);
            p.ws = std::make_shared<Workspace>();
            cudaError_t e = cudaEventCreateWithFlags(&p.ws->done, cudaEventDisableTiming);
            if (e != cudaSuccess) return drop(cuda_fail(e, "cudaEventCreateWithFlags"));
            e = cudaMalloc((void **)&p.ws->p, need);
            if (e == cudaSuccess) {
                p.ws->bytes = need;
                break;
            }
            r = cuda_fail(e, "cudaMalloc(search workspace)");
            if (r != ANN_ERR_OOM || shrink == kMaxShrink) return drop(r);
        }
        cudaStream_t cap;
        cudaError_t ce = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
        if (ce != cudaSuccess) return drop(cuda_fail(ce, "cudaStreamCreateWithFlags"));
        cudaGraph_t graph;
        ce = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
        if (ce != cudaSuccess) {
            cudaStreamDestroy(cap);
            return drop(cuda_fail(ce, "cudaStreamBeginCapture"));
        }
        int rr;
        {
            ForkSet fs;
            rr = record_persistent(pc, A, nq, T, T_all, p.scratch, p.ws->p, p.ws->bytes, shrink, cap, fs);
            ce = cudaStreamEndCapture(cap, &graph);
        }
        cudaStreamDestroy(cap);
        if (rr != ANN_OK || ce != cudaSuccess) {
            if (ce == cudaSuccess) cudaGraphDestroy(graph);
            return drop(rr != ANN_OK ? rr : cuda_fail(ce, "cudaStreamEndCapture"));
        }
        ce = cudaGraphInstantiate(&p.exec, graph, 0);
        cudaGraphDestroy(graph);
        if (ce != cudaSuccess) return drop(cuda_fail(ce, "cudaGraphInstantiate"));
        it = pc->plans.emplace(key, p).first;
    }
    it->second.last_use = ++pc->clock;
    Plan &plan = it->second;
    Workspace &ws = *plan.ws;
    if (ws.last && ws.last != plan.exec) ANN_CUDA(cudaStreamWaitEvent(s, ws.done, 0));
    ANN_CUDA(cudaGraphLaunch(plan.exec, s));
    ws.last = plan.exec;
    ANN_CUDA(cudaEventRecord(ws.done, s));
    return ANN_OK;
}

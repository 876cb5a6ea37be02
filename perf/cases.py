"""The work that a user of this library has it do, as cases that can be timed
and compared: searches of single queries, of batches and of a served request
stream, and every step of the index build.

A case is a dict of plain values; `op` says which public entry point it calls.
Data are seeded mixtures of the families of `datagen` (uint8: means U[0,255],
sigma 20; float32: folded, L2-normalised), drawn on the GPU.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1312_3062_gb300 import ann, datagen

DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _search(name, **kw):
    c = dict(name=name, op="search", dtype="u8", N=1_000_000, d=128, comp=1000, R=20, P=4, n=256, nq=10_000,
             T=512, T_hi=0, k=10, mode="plain")
    c.update(kw)
    return c


def listed():
    return [
        # one query against a small index: a call's own latency
        _search("search_one_tiny", N=10_000, comp=156, R=10, P=2, n=64, nq=1, T=256),
        # the SIFT-shaped 1M index, its 10,000 queries at the budget of recall@10 = 0.9
        _search("search_sift1m_T371", T=371),
        # the served index's regime: components of 10,000 points (as the 10M rows have) with few dictionary words
        # to a component, and its budget of recall@10 = 0.9, in the replayed form
        _search("search_served_T2392", comp=10_000, R=16, n=50, T=2392, mode="persistent"),
        # float32 GIST-shaped rows, every query its own k and its own budget from 64 to 8192
        _search("search_gist_uneven", dtype="f32", N=200_000, d=384, comp=2000, P=3, n=128, nq=2000, T=64, T_hi=8192,
                k=0, mode="persistent"),
        # a burst of requests of 1 to 512 queries to the server, with the paper's 50-word dictionaries
        dict(name="serve_mix_4x50", op="serve", dtype="u8", N=1_000_000, d=128, comp=5000, R=16, P=4, n=50, nreq=48),
        # ground truth: the queries of a benchmark against all rows
        dict(name="truth_u8_1m", op="knn", dtype="u8", N=1_000_000, d=128, comp=1000, nq=10_000, k=10),
        # exact neighbourhood graphs
        dict(name="graph_u8_400k", op="graph", dtype="u8", N=400_000, d=128, comp=1000, k=20),
        dict(name="graph_f32_100k", op="graph", dtype="f32", N=100_003, d=384, comp=2000, k=20),
        # the approximate neighbourhood graph of a 1M-row set
        dict(name="graph_approx_1m", op="approx", dtype="u8", N=1_000_000, d=128, comp=1000, k=16, rounds=4, leaf=1000,
             iters=1),
        # per-part dictionaries from a training sample
        dict(name="centers_u8_200k", op="centers", dtype="u8", N=200_000, d=128, comp=1000, P=4, n=256, iters=10),
        # the bridge graph of an index, and its lists read back
        dict(name="index_u8_200k", op="index", dtype="u8", N=200_000, d=128, comp=1000, R=20, P=4, n=256, t=100, b=5),
        # Graph-D-ADC: re-ranking the members of the lists of 10,000 queries, 16 bytes per code
        dict(name="rerank_m16_L10000", op="rerank", dtype="u8", N=1_000_000, d=128, comp=1000, w=25, m=16, ks=256,
             L=10_000, T=100, nq=10_000),
    ]


def _logu(rng, lo, hi):
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# dimension and dictionaries that go together: (d, P, n); d % P == 0 and n^P <= 2^32
_U8_SHAPES = [(128, 4, 256), (128, 4, 50), (128, 4, 100), (128, 2, 64), (128, 2, 256), (64, 4, 64), (64, 2, 128),
              (96, 3, 128), (96, 4, 33), (192, 3, 100)]
_F32_SHAPES = [(384, 3, 128), (384, 4, 50), (512, 4, 64), (128, 4, 256), (100, 2, 100), (96, 3, 64)]


def draw(rng):
    op = rng.choice(["search", "search", "search", "search", "serve", "knn", "graph", "approx", "centers", "index",
                     "rerank"])
    dtype = rng.choice(["u8", "u8", "f32"])
    comp = _logu(rng, 150, 10_000)
    d, P, n = rng.choice(_U8_SHAPES if dtype == "u8" else _F32_SHAPES)
    if op == "search":
        N = _logu(rng, 10_000, 300_000 if dtype == "u8" else 60_000)
        nq = _logu(rng, 1, 10_000)
        T = _logu(rng, 32, max(64, min(4096, 6_000_000 // nq)))
        return dict(op=op, dtype=dtype, N=N, d=d, comp=comp, R=rng.choice([8, 10, 16, 20, 32]), P=P, n=n, nq=nq, T=T,
                    T_hi=rng.choice([0, 0, min(8192, 2 * T)]), k=rng.choice([0, 1, 10, 10, 32, 100]),
                    mode=rng.choice(["plain", "plain", "persistent"]))
    if op == "serve":
        return dict(op=op, dtype=dtype, N=_logu(rng, 10_000, 200_000 if dtype == "u8" else 40_000), d=d, comp=10_000,
                    R=rng.choice([10, 16, 20]), P=P, n=n, nreq=_logu(rng, 1, 48))
    if op == "knn":
        N = _logu(rng, 5_000, 500_000 if dtype == "u8" else 100_000)
        return dict(op=op, dtype=dtype, N=N, d=d, comp=comp, nq=_logu(rng, 1, 10_000), k=rng.choice([1, 10, 20, 32]))
    if op == "graph":
        return dict(op=op, dtype=dtype, N=_logu(rng, 8_200, 150_000 if dtype == "u8" else 60_000), d=d, comp=comp,
                    k=rng.choice([8, 10, 16, 20, 32]))
    if op == "approx":
        return dict(op=op, dtype="u8", N=_logu(rng, 20_000, 1_000_000), d=rng.choice([64, 96, 128]), comp=comp,
                    k=rng.choice([8, 10, 16, 20, 32]), rounds=rng.choice([2, 4]), leaf=_logu(rng, 300, 4_000),
                    iters=rng.choice([0, 1, 2]))
    if op == "centers":
        return dict(op=op, dtype=dtype, N=_logu(rng, 2_000, 150_000), d=d, comp=comp, P=P, n=n,
                    iters=rng.choice([3, 5, 10]))
    if op == "index":
        return dict(op=op, dtype=dtype, N=_logu(rng, 10_000, 150_000 if dtype == "u8" else 40_000), d=d, comp=comp,
                    R=rng.choice([10, 16, 20]), P=P, n=n, t=rng.choice([10, 50, 100]), b=rng.choice([1, 5, 8]))
    N = _logu(rng, 20_000, 1_000_000)
    return dict(op=op, dtype=dtype, N=N, d=128, comp=_logu(rng, 200, 5_000), w=_logu(rng, 1, 60),
                m=rng.choice([4, 8, 16, 32]), ks=rng.choice([16, 100, 256]), L=_logu(rng, 300, 30_000),
                T=rng.choice([1, 10, 100, 128]), nq=_logu(rng, 1, 5_000))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rows(gen, means, rows, dtype):
    out = torch.empty((rows, means.shape[1]), dtype=torch.uint8 if dtype == "u8" else torch.float32, device=DEV)
    for lo in range(0, rows, 250_000):
        hi = min(rows, lo + 250_000)
        which = torch.randint(0, means.shape[0], (hi - lo,), generator=gen, device=DEV)
        x = torch.randn((hi - lo, means.shape[1]), generator=gen, device=DEV)
        if dtype == "u8":
            out[lo:hi] = (means[which] + 20.0 * x).round_().clamp_(0, 255).to(torch.uint8)
        else:
            x = (means[which] + 0.15 * x).abs_()
            out[lo:hi] = x / x.norm(dim=1, keepdim=True)
    return out


def _data(case, seed):
    """Rows of the case's mixture, about `comp` rows to a component, and a function that draws more."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    ncomp = max(1, case["N"] // case["comp"])
    means = torch.rand((ncomp, case["d"]), generator=gen, device=DEV) * (255.0 if case["dtype"] == "u8" else 1.0)
    return _rows(gen, means, case["N"], case["dtype"]), means, lambda rows: _rows(gen, means, rows, case["dtype"])


def _init_rows(case, rows, seed):
    return np.random.default_rng(seed).permutation(rows)[:case["n"]].astype(np.int64)


def _directions(case, seed):
    levels = datagen.rp_levels(case["N"], case["leaf"])
    while levels and case["N"] >> levels < case["k"] + 1:
        levels -= 1
    return torch.from_numpy(datagen.rp_directions(seed, case["rounds"], levels, case["d"])).to(DEV)


def _graph(case, X, seed):
    """A neighbourhood graph for a search: exact, but for larger uint8 sets whose rows the tensor cores don't take."""
    if case["dtype"] == "u8" and case["d"] not in (64, 128) and case["N"] > 50_000:
        dirs = _directions(dict(case, rounds=4, leaf=1000, k=case["R"]), seed)
        return ann.ann_build_knn_graph_approx(X, case["R"], dirs, 1)[0]
    return ann.ann_build_knn_graph(X, case["R"])[0]


def _centers(case, X, seed):
    sample = X[:20_000]
    return ann.ann_train_centers(sample, case["P"], case["n"], 4, _init_rows(case, len(sample), seed))


def _index(case, X, seed):
    return ann.Index.create(X, _graph(case, X, seed), _centers(case, X, seed), t=100, b=5)


class Server:
    """A server over an index, as a program holds it."""

    def __init__(self, index):
        self.index = index
        self.handle = ctypes.c_void_p()
        ann.check(ann.lib.ann_server_create(index.handle, 256 << 20, 4, ctypes.byref(self.handle)))

    def submit(self, q, k, T):
        ticket = ctypes.c_uint64()
        ann.check(ann.lib.ann_serve_submit(self.handle, q.ctypes.data, len(q), k.ctypes.data, T.ctypes.data,
                                           ctypes.byref(ticket)))
        return ticket.value

    def poll(self, ticket, ids, keys, status):
        return ann.check(ann.lib.ann_serve_poll(self.handle, ticket, ids.ctypes.data, keys.ctypes.data,
                                                status.ctypes.data)) == ann.ANN_OK

    def __del__(self):
        ann.lib.ann_server_destroy(self.handle)


def prepare(case, seed):
    case = {k: v for k, v in case.items() if k != "name"}
    X, means, more = _data(case, seed)
    s = dict(case=case, X=X)
    rng = np.random.default_rng(seed)
    op = case["op"]
    if op == "search":
        s["index"] = _index(case, X, seed)
        nq = case["nq"]
        s["Q"] = more(nq)
        T = case["T"]
        if case["T_hi"]:  # each query its own budget, log-uniform
            T = np.exp(rng.uniform(math.log(case["T"]), math.log(case["T_hi"] + 1), nq)).astype(np.int32)
            T = torch.from_numpy(np.clip(T, case["T"], case["T_hi"])).to(DEV)
        k = case["k"]
        if not k:  # each query its own k
            k = torch.from_numpy(rng.choice(np.array([1, 10, 100], np.int32), nq)).to(DEV)
        s.update(k=k, T=T, kmax=case["k"] or 100)
        key = torch.int32 if case["dtype"] == "u8" else torch.float32
        s["out"] = (torch.empty((nq, s["kmax"]), dtype=torch.int32, device=DEV),
                    torch.empty((nq, s["kmax"]), dtype=key, device=DEV),
                    torch.empty((nq,), dtype=torch.int32, device=DEV))
    elif op == "serve":
        s["server"] = Server(_index(case, X, seed))
        plan = np.random.default_rng(case["nreq"])  # the requests' sizes and k: the same for every seed
        sizes = np.clip(np.floor(np.exp(plan.uniform(0.0, math.log(513.0), case["nreq"]))), 1, 512).astype(int)
        Q = more(int(sizes.sum())).cpu().numpy()
        k = plan.choice(np.array([1, 10, 100], np.int32), len(Q))
        T = rng.choice(np.array([128, 512, 2048], np.int32), len(Q))
        at = np.concatenate([[0], np.cumsum(sizes)])
        s["requests"] = [(np.ascontiguousarray(Q[a:b]), k[a:b].copy(), T[a:b].copy()) for a, b in zip(at, at[1:])]
    elif op == "knn":
        s["Q"] = more(case["nq"])
    elif op == "approx":
        s["dirs"] = _directions(case, seed)
    elif op == "centers":
        s["init"] = _init_rows(case, case["N"], seed)
    elif op == "index":
        # a graph of the right shape: the bridge graph does not read it
        s["G"] = torch.randint(0, case["N"], (case["N"], case["R"]), dtype=torch.int32, device=DEV)
        s["C"] = _centers(case, X, seed)
        # room for the lists: how many bridges have one depends on the rows
        rows = min(case["n"] ** case["P"], 8 * case["N"])
        s["out"] = np.full(rows, -1, np.int64), np.full((rows, case["b"]), -1, np.int32)
    elif op == "rerank":
        # the mixture's means as coarse centers, every row in its nearest one's list
        K, m, ks, dp = len(means), case["m"], case["ks"], case["d"] // case["m"]
        nearest = torch.cat([torch.cdist(x.float(), means).argmin(1) for x in X.split(100_000)]).to(torch.int32)
        members = torch.argsort(nearest, stable=True)
        rest = (X[:50_000].float() - means[nearest[:50_000].long()])
        books = rest[torch.from_numpy(rng.permutation(len(rest))[:ks]).to(DEV)].reshape(ks, m, dp)
        books = books.permute(1, 0, 2).contiguous()
        Q = more(case["nq"]).float()
        w = min(case["w"], K)
        s.update(Q=Q, centers=means.contiguous(), books=books, members=members.to(torch.int32),
                 offsets=torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV),
                                    torch.bincount(nearest.long(), minlength=K).cumsum(0)]),
                 lists=torch.cdist(Q, means).topk(w, largest=False).indices.to(torch.int32),
                 codes=ann.ann_pq_encode(X, means.contiguous(), nearest, books))
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    case = s["case"]
    op = case["op"]
    if op == "search":
        mode = ann.ANN_MODE_PERSISTENT if case["mode"] == "persistent" else ann.ANN_MODE_PLAIN
        ids, keys, status = s["out"]
        return ann.ann_search_batch(s["index"], s["Q"], s["k"], s["T"], kmax=s["kmax"], mode=mode, out_ids=ids,
                                    out_keys=keys, out_status=status)
    if op == "serve":
        server, todo, out = s["server"], [], []
        for q, k, T in s["requests"]:
            todo.append(server.submit(q, k, T))
            kmax = int(k.max())
            out.append((np.empty((len(q), kmax), np.int32),
                        np.empty((len(q), kmax), np.int32 if case["dtype"] == "u8" else np.float32),
                        np.empty(len(q), np.int32)))
        waiting = list(zip(todo, out))
        while waiting:
            waiting = [(t, o) for t, o in waiting if not server.poll(t, *o)]
        return {name: np.concatenate([o[i].reshape(-1) for o in out]) for i, name in enumerate(("ids", "keys", "status"))}
    if op == "knn":
        return ann.ann_exact_knn(s["X"], s["Q"], case["k"])
    if op == "graph":
        return ann.ann_build_knn_graph(s["X"], case["k"])
    if op == "approx":
        return ann.ann_build_knn_graph_approx(s["X"], case["k"], s["dirs"], case["iters"])
    if op == "centers":
        return ann.ann_train_centers(s["X"], case["P"], case["n"], case["iters"], s["init"])
    if op == "index":
        index = ann.Index.create(s["X"], s["G"], s["C"], t=case["t"], b=case["b"])
        ids, refs = index.bridges()
        index.free()
        m = min(len(ids), len(s["out"][0]))
        s["out"][0][:m], s["out"][1][:m] = ids[:m], refs[:m]
        return len(ids), *s["out"]
    return ann.ann_adc_rerank(s["Q"], s["lists"], s["offsets"], s["members"], s["centers"], s["codes"], s["books"],
                              case["L"], case["T"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    op, N, d = case["op"], case["N"], case["d"]
    es = 1 if case["dtype"] == "u8" else 4
    if op in ("search", "serve"):
        if op == "search":
            nq, T = case["nq"], case["T"]
            if case["T_hi"]:
                T = (case["T_hi"] - T) / math.log(case["T_hi"] / T)
            kmax = case["k"] or 100
        else:
            nq, T, kmax = case["nreq"] * 82, 896, 100
        # every discovered row once, the query, its part tables and the results
        return {"bytes": nq * (T * d * es + d * es + kmax * 8) + case["n"] * d * es,
                "flops": nq * (3.0 * T * d + 3.0 * case["n"] * d)}
    if op == "knn":
        return {"bytes": (N + case["nq"]) * d * es + case["nq"] * case["k"] * 8, "flops": 2.0 * N * case["nq"] * d}
    if op == "graph":
        return {"bytes": N * d * es + N * case["k"] * 8, "flops": 2.0 * N * N * d}
    if op == "approx":
        levels = datagen.rp_levels(N, case["leaf"])
        leaf = N / (1 << levels)
        pairs = N * case["rounds"] * leaf + N * case["iters"] * case["k"] ** 2
        return {"bytes": N * d + N * case["k"] * 8, "flops": 2.0 * d * (pairs + N * case["rounds"] * levels)}
    if op == "centers":
        return {"bytes": N * d * es, "flops": 3.0 * N * d * case["n"] * case["iters"]}
    if op == "index":
        # rows and graph in, the index's copies out, a (bridge, key, row) triple per row and bridge written and read
        return {"bytes": 2 * N * (d * es + 4 * case["R"]) + 24 * N * case["t"], "flops": 3.0 * N * d * case["n"]}
    K = max(1, N // case["comp"])
    seen = min(case["L"], case["w"] * case["comp"], N)
    lists = min(case["w"], K, -(-seen // case["comp"]))
    return {"bytes": N * (case["m"] + 4) + case["nq"] * (4 * d + case["T"] * 8),
            "flops": case["nq"] * (3.0 * lists * case["ks"] * d + seen * case["m"])}


# ---------------------------------------------------------------------------
# the same in 64 bits, without this library's code
# ---------------------------------------------------------------------------
def exact(case, seed):
    """Keys in 64 bits of the exact neighbour searches and of the re-ranking.  The other outputs are whole numbers,
    or keys of a search whose ids follow from its own order of visits."""
    op = case["op"]
    if op in ("knn", "graph") and case["dtype"] == "f32":
        if op == "graph" and case["N"] > 120_000:
            return None
        s = prepare(case, seed)
        X = s["X"].double()
        Q = X if op == "graph" else s["Q"].double()
        xn, keys = (X * X).sum(1), []
        for lo in range(0, len(Q), 8192):
            q = Q[lo:lo + 8192]
            D = (q * q).sum(1)[:, None] + xn[None] - 2.0 * (q @ X.T)
            if op == "graph":
                D[torch.arange(len(q), device=DEV), torch.arange(lo, lo + len(q), device=DEV)] = math.inf
            at = D.topk(case["k"], largest=False).indices
            # the chosen keys again without cancellation
            keys.append(torch.stack([((q - X[at[:, j]]) ** 2).sum(1) for j in range(case["k"])], 1).sort(1).values)
        return [None, torch.cat(keys)]
    if op == "rerank":
        s = prepare(case, seed)
        w, m, T, L, nq = s["lists"].shape[1], case["m"], case["T"], case["L"], case["nq"]
        off, members, codes = s["offsets"], s["members"].long(), s["codes"].long()
        books, centers = s["books"].double(), s["centers"].double()
        all_keys = []
        for lo in range(0, nq, 50):
            q, lists = s["Q"][lo:lo + 50].double(), s["lists"][lo:lo + 50].long()
            B = len(q)
            r = (q[:, None] - centers[lists]).reshape(B, w, m, -1)
            table = torch.stack([((r[:, :, j, None] - books[j]) ** 2).sum(-1) for j in range(m)], 2)  # B, w, m, ks
            size = off[lists + 1] - off[lists]
            end = size.cumsum(1)
            p = torch.arange(min(L, int(end.max())), device=DEV).expand(B, -1).contiguous()
            li = torch.searchsorted(end, p, right=True)
            have = li < w
            li = li.clamp(max=w - 1)
            x = members[(off[lists] + size - end).gather(1, li).add(p).clamp(0, len(members) - 1)]
            keys = torch.zeros_like(p, dtype=torch.float64)
            flat = table.reshape(B, -1)
            for j in range(m):
                keys += flat.gather(1, (li * m + j) * case["ks"] + codes[:, j][x])
            keys[~have] = math.inf
            if keys.shape[1] < T:
                keys = torch.cat([keys, torch.full((B, T - keys.shape[1]), math.inf, dtype=keys.dtype, device=DEV)], 1)
            all_keys.append(keys.topk(T, largest=False).values)
        return [None, torch.cat(all_keys), None]
    return None

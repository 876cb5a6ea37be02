"""Index-build kernels at the edges of their tiles and of their dispatch rules,
against the CPU oracle (whole numbers exactly; fp64 centers within the rounding
of a differently ordered sum)."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_1312_3062_gb300 import datagen  # noqa: E402


@pytest.fixture(scope="module")
def ann():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1312_3062_gb300 import _build
    _build.build()
    from paper_1312_3062_gb300 import ann as mod
    return mod


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("kind,N,d,P,n", [("u8", 300, 16, 1, 1), ("u8", 129, 16, 4, 64), ("u8", 1000, 100, 4, 65),
                                          ("u8", 2049, 96, 2, 256), ("ties", 600, 64, 4, 70),
                                          ("f32", 257, 100, 2, 64), ("f32", 900, 264, 2, 130),
                                          ("far", 513, 96, 3, 33), ("huge", 300, 32, 2, 8)])
def test_kmeans_tile_edges_and_rows_left_to_fp64(ann, kind, N, d, P, n):
    rng = np.random.default_rng(N)
    if kind == "ties":  # many equidistant centers: every row needs the fp64 scan and its tie rule
        X = rng.integers(0, 3, size=(N, d)).astype(np.uint8) * 2
    elif kind == "u8":
        X = datagen.mixture(N, N, d, 9, np.uint8)
    elif kind == "far":  # float32 cannot separate the centers
        X = (4096.0 + rng.standard_normal((N, d)) * 0.01).astype(np.float32)
    elif kind == "huge":  # squares overflow float32, not fp64
        X = (rng.standard_normal((N, d)) * 1e25).astype(np.float32)
    else:
        X = datagen.mixture(N, N, d, 9, np.float32)
    init = rng.permutation(N)[:n]
    want = oracle.kmeans(X, P, n, 2, init)
    got, got64 = ann.ann_train_centers(dev(X), P, n, 2, init, want_f64=True)
    if X.dtype == np.uint8:
        np.testing.assert_array_equal(got64.cpu().numpy(), want)
        np.testing.assert_array_equal(got.cpu().numpy(), oracle.round_centers(want, np.uint8))
    else:
        # sums of up to N equal-sized terms in another order: N * 2^-53 relative to the largest term
        np.testing.assert_allclose(got64.cpu().numpy(), want, rtol=0, atol=N * 2.0 ** -52 * np.abs(X).max())


@pytest.mark.parametrize("N,dtype", [((1 << 24) + 300, "u8"), ((1 << 24) + 1, "f32"), ((1 << 31) + 4096, "u8")])
def test_kmeans_rows_beyond_one_pass_and_beyond_32_bits(ann, N, dtype):
    # two equal centers leave every row near them to the fp64 scan; rows of both clusters in the last pass
    d, tail = 16, 200
    if torch.cuda.mem_get_info()[0] < 2 * N * d * (1 if dtype == "u8" else 4):
        pytest.skip("not enough device memory")
    X = torch.empty((N, d), dtype=torch.uint8 if dtype == "u8" else torch.float32, device="cuda")
    X.random_(0, 4)
    X[:2] = 1
    X[2] = 250
    X[-tail:] = 240
    _, got = ann.ann_train_centers(X, 1, 3, 1, np.arange(3), want_f64=True)
    low = torch.zeros(d, dtype=torch.float64, device="cuda")
    for r in range(0, N, 1 << 24):  # whole numbers below 2^53
        low += X[r:r + (1 << 24)].sum(0, dtype=torch.float64)
    del X
    torch.cuda.empty_cache()
    near = low.cpu().numpy() - (250 + 240 * tail)
    want = np.stack([near / (N - tail - 1), np.ones(d), np.full(d, (250 + 240 * tail) / (tail + 1))])
    np.testing.assert_array_equal(got[0].cpu().numpy(), want)


@pytest.mark.parametrize("kind,N,d,P,n,t,b", [("u8", 70, 64, 4, 256, 100, 5),    # a buffer smaller than the candidates
                                              ("u8", 33, 48, 2, 256, 700, 2),    # t beyond the buffer's first size
                                              ("u8", 40, 96, 3, 33, 1, 5),
                                              ("u8", 40, 64, 4, 3, 500, 8),      # every bridge is among the t nearest
                                              ("equal", 35, 64, 4, 64, 100, 3),  # all keys equal: ranks decide
                                              ("f32", 45, 60, 4, 128, 100, 5), ("f32", 40, 36, 2, 100, 100, 1),
                                              ("f32equal", 33, 16, 4, 48, 100, 5)])
def test_bridge_lists_where_candidates_are_cut(ann, kind, N, d, P, n, t, b):
    dt = np.float32 if kind.startswith("f32") else np.uint8
    rng = np.random.default_rng(N)
    if kind.endswith("equal"):
        X = np.ones((N, d), dt)
        C = np.full((P, n, d // P), 3, dt)
    else:
        X = datagen.mixture(N, N, d, 4, dt)
        C = rng.integers(0, 256, (P, n, d // P)).astype(dt) if dt == np.uint8 else \
            rng.random((P, n, d // P)).astype(dt) * 0.2
    want = oracle.bridge_graph(X, C, t, b)
    ix = ann.Index.create(dev(X), dev(np.zeros((N, 4), np.int32)), dev(C), t=t, b=b)
    ids, refs = ix.bridges()
    np.testing.assert_array_equal(ids, want["bridges"])
    lens = np.diff(want["offsets"])
    np.testing.assert_array_equal((refs >= 0).sum(1), lens)
    np.testing.assert_array_equal(refs[refs >= 0], want["refs"])


@pytest.mark.parametrize("N,nq,d,k,shift", [(8192, 256, 60, 1, 0), (8193, 257, 100, 32, 0), (9001, 300, 4, 20, 0),
                                            (8257, 259, 384, 10, 1), (10_003, 256, 36, 7, 3)])
def test_f32_knn_odd_sizes_and_alignments(ann, N, nq, d, k, shift):
    X, Q = datagen.mixture(N, N, d, 9, np.float32), datagen.mixture(N, nq, d, 9, np.float32)

    def at(a):  # rows that start `shift` floats off a 16-byte boundary
        flat = torch.empty(a.size + shift, dtype=torch.float32, device="cuda")
        flat[shift:] = dev(a.reshape(-1))
        return flat[shift:].view(a.shape)

    ids, keys = ann.ann_exact_knn(at(X), at(Q), k)
    want_ids, want_keys = oracle.exact_knn(X, Q, k)
    np.testing.assert_array_equal(ids.cpu().numpy(), want_ids)
    np.testing.assert_allclose(keys.cpu().numpy(), want_keys, rtol=1e-5)


def test_f32_knn_with_millions_of_references(ann):
    # more references than a tile of 256 query rows takes in 2 GB; two tiles and a remainder
    N, nq, d, k = 2_200_003, 1100, 4, 10
    X, Q = np.random.default_rng(1).random((N, d), np.float32), np.random.default_rng(2).random((nq, d), np.float32)
    ids, keys = ann.ann_exact_knn(dev(X), dev(Q), k)
    sel = np.r_[0, 511, 512, 1023, 1024, nq - 1]
    want_ids, want_keys = oracle.exact_knn(X, np.ascontiguousarray(Q[sel]), k)
    np.testing.assert_array_equal(ids.cpu().numpy()[sel], want_ids)
    np.testing.assert_allclose(keys.cpu().numpy()[sel], want_keys, rtol=1e-5)


@pytest.mark.parametrize("kind", ["descending", "late_cluster", "ties"])
def test_f32_knn_when_the_first_columns_mislead(ann, kind):
    # the candidate limit starts from the first 4096 columns: here those are
    # the farthest rows, the near ones come all at once, or most are equal
    N, nq, d, k = 20_011, 256, 32, 20
    X, Q = datagen.mixture(5, N, d, 6, np.float32), datagen.mixture(6, nq, d, 6, np.float32)
    Q[1:] = Q[0] + 0.001 * Q[1:]
    dist = ((X - Q[0]) ** 2).sum(1)
    if kind == "descending":
        X = X[np.argsort(-dist)]
    elif kind == "late_cluster":
        X[4096:12_000] = Q[0] + 0.1 * X[4096:12_000]
    else:
        X[3000:9000] = X[3000]
    X = np.ascontiguousarray(X)
    ids, keys = ann.ann_exact_knn(dev(X), dev(Q), k)
    want_ids, want_keys = oracle.exact_knn(X, Q, k)
    np.testing.assert_array_equal(ids.cpu().numpy(), want_ids)
    np.testing.assert_allclose(keys.cpu().numpy(), want_keys, rtol=1e-5)


@pytest.mark.parametrize("kind,N,nq,d,k", [
    ("mix", 5, 1, 64, 8), ("mix", 255, 127, 128, 1), ("mix", 256, 128, 64, 9), ("mix", 257, 129, 128, 16),
    ("mix", 3001, 33, 128, 17), ("mix", 20_011, 700, 64, 25), ("mix", 70_003, 3, 128, 32), ("mix", 40_000, 2500, 128, 10),
    ("black_white", 3000, 300, 128, 20), ("white", 700, 130, 128, 32), ("equal", 2000, 140, 64, 24),
    ("descending", 9000, 200, 128, 10), ("graph", 2500, 0, 128, 24), ("graph", 1100, 0, 64, 31)])
def test_u8_tensor_knn_tile_edges_and_extreme_rows(ann, kind, N, nq, d, k):
    rng = np.random.default_rng(N + k)
    X, Q = datagen.mixture(N, N, d, 7, np.uint8), datagen.mixture(N, max(nq, 1), d, 7, np.uint8)
    if kind == "black_white":    # the largest norms and products
        X, Q = (rng.integers(0, 2, X.shape) * 255).astype(np.uint8), (rng.integers(0, 2, Q.shape) * 255).astype(np.uint8)
    elif kind == "white":
        X[:] = 255
        Q[::2] = 255
        Q[1::2] = 0
    elif kind == "equal":        # every key equal: ids decide, also across the lists of a row
        X[:] = X[0]
    elif kind == "descending":   # every tile beats the ones before it
        X = X[np.argsort(-((X.astype(np.int64) - Q[0]) ** 2).sum(1), kind="stable")]
        Q[:] = Q[0]
    if kind == "graph":
        ids, keys = ann.ann_build_knn_graph(dev(X), k)
        want_ids, want_keys = oracle.exact_knn(X, X, k, exclude_self=True)
    else:
        ids, keys = ann.ann_exact_knn(dev(X), dev(Q), k)
        want_ids, want_keys = oracle.exact_knn(X, Q, k)
    np.testing.assert_array_equal(ids.cpu().numpy(), want_ids)
    np.testing.assert_array_equal(ann.keys_as_uint32(keys).astype(np.float64),
                                  np.where(np.isinf(want_keys), 4294967295.0, want_keys))


@pytest.mark.parametrize("m,dp,ks,w,T,L,shift", [(16, 8, 256, 6, 100, 10**9, 0), (8, 5, 37, 1, 128, 900, 0),
                                                 (2, 4, 101, 3, 1, 5000, 0), (12, 3, 100, 5, 128, 10**9, 0),
                                                 (5, 12, 16, 4, 33, 3333, 0), (16, 4, 256, 5, 128, 10**9, 4),
                                                 (3, 4, 1, 4, 77, 10**9, 0)])
def test_adc_rerank_is_bit_exact_in_its_stated_order(ann, m, dp, ks, w, T, L, shift):
    # the float32 operations of ann.h in their order, with numpy; lists of up to 3,000 members (the buffer is cut
    # several times), a list visited twice, absent lists, codes off their natural alignment, one codeword (all keys tie)
    rng = np.random.default_rng(m * 1000 + ks)
    d, N, K, nq = m * dp, 9000, 7, 5
    C = rng.standard_normal((K, d)).astype(np.float32)
    books = rng.standard_normal((m, ks, dp)).astype(np.float32)
    codes = rng.integers(0, ks, (N, m)).astype(np.uint8)
    assign = np.sort(rng.choice(K, N, p=[.34, .3, .2, .1, .05, .009, .001]))
    members = np.argsort(assign, kind="stable").astype(np.int32)
    offsets = np.concatenate([[0], np.cumsum(np.bincount(assign, minlength=K))]).astype(np.int64)
    Q = rng.standard_normal((nq, d)).astype(np.float32)
    lists = np.stack([rng.permutation(K)[:w] for _ in range(nq)]).astype(np.int32)
    lists[0, -1] = lists[0, 0]
    lists[1, 0] = -1
    flat = torch.empty(codes.size + shift, dtype=torch.uint8, device="cuda")
    flat[shift:] = dev(codes.reshape(-1))
    ids, keys, seen = ann.ann_adc_rerank(dev(Q), dev(lists), dev(offsets), dev(members), dev(C),
                                         flat[shift:].view(N, m), dev(books), L, T)
    for i in range(nq):
        got, total = [np.zeros(0, np.uint64)], 0
        for c in lists[i]:
            if c < 0 or total >= L:
                continue
            x = members[offsets[c]:offsets[c + 1]][:L - total]
            total += len(x)
            r = (Q[i] - C[c]).reshape(m, 1, dp)
            table = np.zeros((m, ks), np.float32)
            for t in range(dp):
                e = r[:, :, t] - books[:, :, t]
                table = table + e * e
            key = np.zeros(len(x), np.float32)
            for j in range(m):
                key = key + table[j, codes[x, j]]
            got.append(np.stack([key.view(np.uint32).astype(np.uint64) << 32 | x.astype(np.uint64)]).reshape(-1))
        best = np.sort(np.concatenate(got))[:T]
        assert int(seen[i]) == total
        np.testing.assert_array_equal(ids[i].cpu().numpy()[:len(best)], (best & 0xffffffff).astype(np.int32))
        np.testing.assert_array_equal(keys[i].cpu().numpy().view(np.uint32)[:len(best)], (best >> 32).astype(np.uint32))
        assert np.all(ids[i].cpu().numpy()[len(best):] == -1)


@pytest.mark.parametrize("kind,N,d,R,rounds,levels,iters", [
    ("mix", 193, 64, 8, 1, 0, 0), ("mix", 1539, 128, 32, 2, 1, 0), ("mix", 4100, 128, 20, 3, 3, 1),
    ("mix", 5003, 64, 16, 2, 3, 1), ("mix", 3001, 128, 1, 2, 4, 0), ("mix", 5099, 128, 25, 3, 3, 0),
    ("equal", 1500, 64, 12, 2, 2, 1), ("few", 5000, 128, 24, 3, 3, 1), ("mix", 97, 64, 8, 1, 0, 0)])
def test_approx_graph_leaves_on_the_tensor_cores(ann, kind, N, d, R, rounds, levels, iters):
    X = datagen.mixture(N, N, d, 11, np.uint8)
    if kind == "equal":      # every key equal: ids decide
        X[:] = X[0]
    elif kind == "few":      # many equal rows, so equal keys in one leaf and across rounds
        X = np.ascontiguousarray(X[np.random.default_rng(1).integers(0, 30, N)])
    dirs = datagen.rp_directions(N, rounds, levels, d)
    gi, gk = ann.ann_build_knn_graph_approx(dev(X), R, dev(dirs), iters)
    oi, ok = oracle.knn_graph_approx(X, R, dirs, iters)
    np.testing.assert_array_equal(gi.cpu().numpy(), oi)
    np.testing.assert_array_equal(gk.cpu().numpy().view(np.uint32), ok.astype(np.uint32))


def test_widest_lists_and_plain_searches_can_be_captured(ann):
    """Calls that wait for nothing on the host: recorded into a CUDA graph once, replayed on other queries."""
    N, nq, d, k, T = 3000, 5000, 128, 32, 200
    X, Q = datagen.mixture(3, N, d, 9, np.uint8), datagen.mixture(4, nq, d, 9, np.uint8)
    Xd, Qd = dev(X), dev(Q)
    G, _ = ann.ann_build_knn_graph(Xd, 10)
    C = ann.ann_train_centers(Xd, 4, 16, 2, np.arange(16))
    ix = ann.Index.create(Xd, G, C, t=100, b=5)

    def calls(q):
        s = torch.cuda.current_stream()
        return (*ann.ann_exact_knn(Xd, q[:200], k, stream=s), *ann.ann_search_batch(ix, q, 10, T, mode=0, stream=s)[:2],
                *ann.ann_search_batch(ix, q[:64], 10, 2000, mode=0, stream=s)[:2])

    want = [x.cpu().numpy() for x in calls(Qd)]
    buf = torch.zeros_like(Qd)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        got = calls(buf)
    for _ in range(2):
        buf.copy_(Qd)
        g.replay()
        for a, b in zip(got, want):
            np.testing.assert_array_equal(a.cpu().numpy(), b)
            a.zero_()


@pytest.mark.parametrize("dtype,N,nq,d,k", [(np.uint8, 3000, 200, 64, 10), (np.uint8, 3000, 200, 64, 31),
                                            (np.uint8, 3000, 200, 128, 10), (np.uint8, 3000, 200, 128, 32),
                                            (np.float32, 8192, 256, 36, 10), (np.float32, 8192, 255, 36, 10)])
def test_exact_knn_can_be_captured_whatever_its_sizes(ann, dtype, N, nq, d, k):
    X, Q = dev(datagen.mixture(3, N, d, 9, dtype)), dev(datagen.mixture(4, nq, d, 9, dtype))
    want = ann.ann_exact_knn(X, Q, k)
    buf = torch.zeros_like(Q)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        got = ann.ann_exact_knn(X, buf, k, stream=torch.cuda.current_stream())
    buf.copy_(Q)
    g.replay()
    for a, b in zip(got, want):
        assert torch.equal(a, b)

"""Launches of more queries than one kernel holds run as prologue, main loop and
resumed queries; smaller ones as one kernel from start to end.  Both give the
same results, counters included, and the oracle's on a sample."""
from __future__ import annotations

import ctypes

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


# the last uint8 cases pop more bridges than the prologue leaves: nearly every query is resumed, with budgets of 8192
# more of them than there are slots for their states
@pytest.mark.parametrize("dtype,N,d,comps,P,n,R,T,k,mode", [
    (np.uint8, 4000, 128, 4, 4, 16, 16, 300, 10, 0), (np.uint8, 4000, 64, 40, 2, 64, 20, 900, 100, 1),
    (np.uint8, 4000, 128, 40, 4, 24, 10, 1024, 33, 0), (np.float32, 3000, 96, 20, 3, 20, 20, 700, 10, 1),
    (np.float32, 3000, 512, 20, 4, 12, 16, 1500, 1, 0), (np.uint8, 9000, 32, 3, 2, 128, 8, 8192, 10, 0),
    (np.uint8, 2500, 48, 60, 3, 33, 32, 31, 5, 1)])
def test_many_queries_equal_few_and_the_oracle(ann, dtype, N, d, comps, P, n, R, T, k, mode):
    rng = np.random.default_rng(N + T)
    X = datagen.mixture(T, N, d, comps, dtype)
    nq = 6000
    Q = datagen.mixture(T, nq, d, comps, dtype)
    C = ann.ann_train_centers(dev(X), P, n, 2, rng.permutation(N)[:n])
    G, _ = ann.ann_build_knn_graph(dev(X), R)
    ix = ann.Index.create(dev(X), G, C, t=100, b=5)

    def search(q, m):
        st = torch.zeros((len(q), ann.ANN_NSTATS), dtype=torch.int64, device="cuda")
        ids, keys, status = ann.ann_search_batch(ix, q, k, T, mode=m, out_stats=st)
        torch.cuda.synchronize()
        cols = [ann.STAT_NAMES.index(s) for s in ("discovered", "ref_pops", "bridge_pops", "max_q")]
        return [x.cpu().numpy() for x in (ids, keys, status, st[:, cols])]

    Qd = dev(Q)
    many = search(Qd, mode)
    few = [np.concatenate(x) for x in zip(*(search(Qd[i:i + 150].contiguous(), 0) for i in range(0, nq, 150)))]
    for a, b in zip(many, few):
        np.testing.assert_array_equal(a, b)
    sel = rng.permutation(nq)[:24]
    ids, refs = ix.bridges()
    bg = dict(bridges=ids, offsets=np.concatenate([[0], np.cumsum((refs >= 0).sum(1))]).astype(np.int64),
              refs=refs[refs >= 0])
    wi, wk, ws = oracle.search(X, G.cpu().numpy(), C.cpu().numpy(), bg, Q[sel], k, T, kmax=k, nthreads=8)
    np.testing.assert_array_equal(many[0][sel], wi)
    np.testing.assert_array_equal(many[3][sel, 1], ws["ref_pops"])
    np.testing.assert_array_equal(many[3][sel, 2], ws["nonempty_bridge_pops"])


# rows so wide that one query fills an SM: beside a budget's queue and visited set in shared memory (T = 8192), and
# beside no more than the prologue's first batch (T = 32; also more queries than SMs)
@pytest.mark.parametrize("d,T,nq", [(24_000, 8192, 12), (24_000, 8192, 300), (55_728, 32, 12), (55_728, 32, 300)])
def test_rows_as_wide_as_shared_memory(ann, d, T, nq):
    rng = np.random.default_rng(d)
    N, P, n, k = 300, 2, 256, 10
    X = datagen.mixture(1, N, d, 4, np.float32)
    Q = datagen.mixture(2, nq, d, 4, np.float32)
    C = np.ascontiguousarray(X[rng.permutation(N)[:n]].reshape(n, P, d // P).transpose(1, 0, 2))
    G, _ = ann.ann_build_knn_graph(dev(X), 8)
    ix = ann.Index.create(dev(X), G, dev(C), t=20, b=5)
    ids, refs = ix.bridges()
    bg = dict(bridges=ids, offsets=np.concatenate([[0], np.cumsum((refs >= 0).sum(1))]).astype(np.int64),
              refs=refs[refs >= 0])
    sel = rng.permutation(nq)[:12]
    want = oracle.search(X, G.cpu().numpy(), C, bg, Q[sel], k, T, kmax=k, nthreads=8)[0]
    for mode in (0, 1):
        got, _, status = ann.ann_search_batch(ix, dev(Q), k, T, mode=mode)
        torch.cuda.synchronize()
        assert not status.any()
        np.testing.assert_array_equal(got.cpu().numpy()[sel], want)


def test_launch_shapes_are_measured_for_the_form_that_runs(ann):
    # the runs that measure take their workspace from the device's memory pool, recorded plans do not: the pool's mark
    # shows which call measured
    cu, pool = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p()
    torch.zeros(1, device="cuda")
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    N, nq = 4000, 6000
    X, Q = dev(datagen.mixture(1, N, 64, 10, np.uint8)), dev(datagen.mixture(2, nq, 64, 10, np.uint8))
    G, _ = ann.ann_build_knn_graph(X, 10)
    ix = ann.Index.create(X, G, ann.ann_train_centers(X, 4, 16, 2, np.arange(16)), t=100, b=5)

    def measures(q, T):
        mark = ctypes.c_uint64(0)
        torch.cuda.synchronize()
        assert cu.cuMemPoolSetAttribute(pool, 8, ctypes.byref(mark)) == 0  # CU_MEMPOOL_ATTR_USED_MEM_HIGH
        ids, _, _ = ann.ann_search_batch(ix, q, 10, T, mode=1)
        torch.cuda.synchronize()
        assert cu.cuMemPoolGetAttribute(pool, 8, ctypes.byref(mark)) == 0
        assert torch.equal(ids, ann.ann_search_batch(ix, q, 10, T, mode=0)[0])
        return mark.value > 0

    assert not measures(Q[:1], 600)   # one kernel alone: nothing to choose
    assert measures(Q, 600)
    assert not measures(Q, 700)       # the same bucket and form
    assert measures(Q, 1024)          # the same bucket, but queues that spill
    T = torch.full((nq,), 600, dtype=torch.int32, device="cuda")
    assert not measures(Q, T)         # sized for its bucket, as budgets of 1024 are
    T[:100] = 3000                    # a bucket with too few queries to tell: left to a batch that fills it
    assert not measures(Q, T)
    assert measures(Q, 3000)
    assert not measures(Q, 3000)
    ix.free()


@pytest.mark.parametrize("mode,T", [(0, 40), (1, 40), (0, 1200), (1, "mixed")])
def test_batches_of_more_than_one_pass(ann, mode, T):
    # records and first batches are held for 32,768 queries at a time; with budgets of their own the lists of queries are
    # counted on the device, and one of them ends in the second pass
    N, nq = 3000, 33_001
    X, Q = dev(datagen.mixture(3, N, 64, 30, np.uint8)), dev(datagen.mixture(4, nq, 64, 30, np.uint8))
    G, _ = ann.ann_build_knn_graph(X, 8)
    ix = ann.Index.create(X, G, ann.ann_train_centers(X, 4, 16, 2, np.arange(16)), t=50, b=5)
    if T == "mixed":
        T = torch.full((nq,), 90, dtype=torch.int32, device="cuda")
        T[5:nq:400] = 300
    for _ in range(2):
        got = ann.ann_search_batch(ix, Q, 10, T, mode=mode)
        torch.cuda.synchronize()
        for lo in range(0, nq, 6000):
            part = T[lo:lo + 6000].contiguous() if torch.is_tensor(T) else T
            want = ann.ann_search_batch(ix, Q[lo:lo + 6000].contiguous(), 10, part, mode=0)
            for a, b in zip(got, want):
                assert torch.equal(a[lo:lo + 6000], b)
        for a in got:
            a.zero_()
    ix.free()


# the prologue's rules: budgets below 256 walk up to the reach only, dictionaries with c2 groups (4 x 8) or one prefix
# part look at every batch's references; few cells, so that queries pop many bridges and walks end at the limit
@pytest.mark.parametrize("dtype,d,P,n,T", [(np.uint8, 64, 4, 8, 64), (np.uint8, 64, 4, 8, 300), (np.uint8, 128, 2, 64, 255),
                                           (np.uint8, 128, 2, 64, 256), (np.float32, 48, 3, 16, 100),
                                           (np.float32, 64, 2, 32, 33), (np.uint8, 96, 3, 30, 1)])
def test_first_batches_of_bridges(ann, dtype, d, P, n, T):
    N, nq, k = 5000, 4000, 10
    rng = np.random.default_rng(T)
    X, Q = datagen.mixture(T, N, d, 300, dtype), datagen.mixture(T, nq, d, 300, dtype)
    C = ann.ann_train_centers(dev(X), P, n, 2, rng.permutation(N)[:n])
    G, _ = ann.ann_build_knn_graph(dev(X), 8)
    ix = ann.Index.create(dev(X), G, C, t=100, b=5)
    Qd = dev(Q)

    def search(q):
        st = torch.zeros((len(q), ann.ANN_NSTATS), dtype=torch.int64, device="cuda")
        out = ann.ann_search_batch(ix, q, k, T, out_stats=st)
        return [*out, st[:, [ann.STAT_NAMES.index(x) for x in ("discovered", "ref_pops", "bridge_pops", "max_q")]]]

    many = search(Qd)
    few = [torch.cat(x) for x in zip(*(search(Qd[i:i + 150].contiguous()) for i in range(0, nq, 150)))]
    for a, b in zip(many, few):
        assert torch.equal(a, b)
    sel = rng.permutation(nq)[:16]
    ids, refs = ix.bridges()
    bg = dict(bridges=ids, offsets=np.concatenate([[0], np.cumsum((refs >= 0).sum(1))]).astype(np.int64),
              refs=refs[refs >= 0])
    want = oracle.search(X, G.cpu().numpy(), C.cpu().numpy(), bg, Q[sel], k, T, kmax=k, nthreads=8)[0]
    np.testing.assert_array_equal(many[0].cpu().numpy()[sel], want)
    assert (ix.info()["groups"] > 0) == (P == 4)
    ix.free()

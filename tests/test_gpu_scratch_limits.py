"""Calls whose scratch does not fit the device fall back to forms that need
less, with the same results.  The device's current memory pool, from which the
library takes its stream-ordered scratch, is replaced by one of a limited size
(CUDA driver API), so that an allocation fails without filling the device."""
from __future__ import annotations

import contextlib
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

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


class PoolProps(ctypes.Structure):  # CUmemPoolProps
    _fields_ = [("allocType", ctypes.c_int), ("handleTypes", ctypes.c_int), ("location_type", ctypes.c_int),
                ("location_id", ctypes.c_int), ("security", ctypes.c_void_p), ("maxSize", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


@contextlib.contextmanager
def pool_of(mbytes):
    cu = ctypes.CDLL("libcuda.so.1")
    torch.zeros(1, device="cuda")  # the primary context is current
    torch.cuda.synchronize()
    props = PoolProps(allocType=1, location_type=1, location_id=torch.cuda.current_device(), maxSize=mbytes << 20)
    device = ctypes.c_int(props.location_id)
    small, before, p = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_uint64()
    assert cu.cuDeviceGetMemPool(ctypes.byref(before), device) == 0
    assert cu.cuMemPoolCreate(ctypes.byref(small), ctypes.byref(props)) == 0
    assert cu.cuDeviceSetMemPool(device, small) == 0
    try:
        # the limit holds: twice its size is refused
        assert cu.cuMemAllocAsync(ctypes.byref(p), ctypes.c_size_t(mbytes << 21), None) == 2
        yield
        torch.cuda.synchronize()
    finally:
        assert cu.cuDeviceSetMemPool(device, before) == 0
        torch.cuda.synchronize()
        assert cu.cuMemPoolDestroy(small) == 0


@pytest.mark.parametrize("N,R,levels,mbytes", [(60_000, 16, 4, 64), (6000, 8, 0, 32)])
def test_approx_graph_leaves_without_the_tensor_cores_scratch(ann, N, R, levels, mbytes):
    # lists and pending groups of the tensor-core leaves take some 90 and 55 MB, the rest 18 and 1 MB
    X = dev(datagen.mixture(N, N, 128, 11, np.uint8))
    dirs = dev(datagen.rp_directions(N, 2, levels, 128))
    want = ann.ann_build_knn_graph_approx(X, R, dirs, 1)
    with pool_of(mbytes):
        got = ann.ann_build_knn_graph_approx(X, R, dirs, 1)
    for a, b in zip(got, want):
        assert torch.equal(a, b)


def test_a_call_that_ran_out_of_memory_does_not_fail_the_next(ann):
    X = dev(datagen.mixture(5, 300_000, 64, 11, np.uint8))
    dirs = dev(datagen.rp_directions(5, 1, 3, 64))
    with pool_of(32):
        with pytest.raises(ann.AnnError) as e:  # 38 MB of rows
            ann.ann_build_knn_graph_approx(X, 16, dirs, 0)
        assert e.value.code == ann.ANN_ERR_OOM
        few = X[:1000]
        got = ann.ann_build_knn_graph_approx(few, 16, dirs, 0)
    for a, b in zip(got, ann.ann_build_knn_graph_approx(few, 16, dirs, 0)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("d,k", [(64, 32), (128, 10)])
def test_exact_knn_without_the_tensor_cores_scratch(ann, d, k):
    X, Q = dev(datagen.mixture(6, 20_000, d, 11, np.uint8)), dev(datagen.mixture(7, 300, d, 11, np.uint8))
    want = ann.ann_exact_knn(X, Q, k)
    with pool_of(32):  # the pending groups alone are 50 MB
        got = ann.ann_exact_knn(X, Q, k)
    for a, b in zip(got, want):
        assert torch.equal(a, b)


@pytest.mark.parametrize("nq,T,mbytes", [(10_000, 400, 64), (1500, 900, 32), (3000, 3000, 96)])
def test_plain_search_in_smaller_passes(ann, nq, T, mbytes):
    # records and first batches of 10,000 queries take 47 MB, the scratch of a full device some 90 MB (T = 400), 73 MB
    # for 1500 queries in one kernel, and 330 MB (T = 3000)
    N = 4000
    X = dev(datagen.mixture(8, N, 128, 40, np.uint8))
    Q = dev(datagen.mixture(9, nq, 128, 40, np.uint8))
    G, _ = ann.ann_build_knn_graph(X, 10)
    ix = ann.Index.create(X, G, ann.ann_train_centers(X, 4, 24, 2, np.arange(24)), t=100, b=5)

    def search():
        st = torch.zeros((nq, ann.ANN_NSTATS), dtype=torch.int64, device="cuda")
        out = ann.ann_search_batch(ix, Q, 10, T, mode=0, out_stats=st)
        return [*out, st[:, [ann.STAT_NAMES.index(s) for s in ("discovered", "ref_pops", "bridge_pops", "max_q")]]]

    want = search()
    with pool_of(mbytes):
        got = search()
    for a, b in zip(got, want):
        assert torch.equal(a, b)


@pytest.fixture(scope="module")
def mixed(ann):
    N, nq = 4000, 10_000
    X = dev(datagen.mixture(8, N, 128, 40, np.uint8))
    Q = dev(datagen.mixture(9, nq, 128, 40, np.uint8))
    G, _ = ann.ann_build_knn_graph(X, 10)
    C = ann.ann_train_centers(X, 4, 24, 2, np.arange(24))
    T = dev(np.random.default_rng(1).choice([40, 200, 500, 1000, 1500, 2500], nq).astype(np.int32))
    want = ann.ann_search_batch(ann.Index.create(X, G, C, t=100, b=5), Q, 10, T, mode=0)[0]
    return (lambda: ann.Index.create(X, G, C, t=100, b=5)), Q, T, want


def taken():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_plans_of_one_stream_share_a_workspace(ann, mixed):
    make, Q, T, want = mixed
    ix, outs = make(), [torch.empty_like(want) for _ in range(12)]
    ann.ann_search_batch(ix, Q, 10, T, mode=1)  # launch shapes are measured here
    before = taken()
    for turn in range(2):
        for i, o in enumerate(outs):
            ann.ann_search_batch(ix, Q, 10, T, mode=1, out_ids=o)
            if (turn, i) == (0, 0):
                first = taken() - before
    grown = taken() - before
    for o in outs:
        assert torch.equal(o, want)
    # a graph, its lists and outputs for each plan, but not a workspace (about 2 GB)
    assert grown - first < 1 << 29, (first, grown)
    # other streams side by side, each with a workspace of its own
    streams = [torch.cuda.Stream() for _ in range(3)]
    torch.cuda.synchronize()
    for o in outs:
        o.zero_()
    torch.cuda.synchronize()
    for _ in range(3):
        for i, o in enumerate(outs):
            ann.ann_search_batch(ix, Q, 10, T, mode=1, out_ids=o, stream=streams[i % 3])
    torch.cuda.synchronize()
    for o in outs:
        assert torch.equal(o, want)
    ix.free()


def test_workspaces_of_many_streams_are_bounded(ann, mixed):
    make, Q, T, want = mixed
    ix, streams = make(), [torch.cuda.Stream() for _ in range(14)]
    before = taken()
    outs = [torch.empty_like(want) for _ in streams]
    torch.cuda.synchronize()
    for _ in range(2):
        for s, o in zip(streams, outs):
            ann.ann_search_batch(ix, Q, 10, T, mode=1, out_ids=o, stream=s)
    # 14 workspaces of about 2 GB do not fit in 16 GB: the least recently used plans went
    assert taken() - before < (16 << 30) + (1 << 30)
    for o in outs:
        assert torch.equal(o, want)
    ix.free()


def test_a_plan_in_what_memory_is_left(ann, mixed):
    make, Q, T, want = mixed
    torch.cuda.empty_cache()
    ix = make()
    ann.ann_search_batch(ix, Q[:3000], 10, T[:3000], mode=1)  # launch shapes are measured here
    torch.cuda.synchronize()
    rest = torch.empty(torch.cuda.mem_get_info()[0] - (5 << 28), dtype=torch.uint8, device="cuda")  # leaves 1.25 GB
    out = torch.empty_like(want)
    ann.ann_search_batch(ix, Q, 10, T, mode=1, out_ids=out)
    torch.cuda.synchronize()
    del rest
    torch.cuda.empty_cache()
    assert torch.equal(out, want)
    ix.free()

"""Calls whose fast form the device cannot take: the other form has to answer.

A device without room is a memory pool with a limit, made current for the
calls under test; nothing is filled.
"""
import contextlib
import ctypes as C

import numpy as np
import pytest

from lpmake import INF

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_16182_gb300 import lpp, synth  # noqa: E402


class PoolProps(C.Structure):  # CUmemPoolProps
    _fields_ = [("alloc_type", C.c_int), ("handle_types", C.c_int), ("loc_type", C.c_int), ("loc_id", C.c_int),
                ("win32", C.c_void_p), ("max_size", C.c_size_t), ("usage", C.c_ushort), ("reserved", C.c_ubyte * 54)]


@contextlib.contextmanager
def pool_limit(max_bytes):
    """Device 0's stream-ordered allocations come from a pool of max_bytes."""
    cu = C.CDLL("libcuda.so.1")
    old, pool = C.c_void_p(), C.c_void_p()
    props = PoolProps(alloc_type=1, loc_type=1, loc_id=0, max_size=max_bytes)  # pinned, on device 0
    assert cu.cuDeviceGetMemPool(C.byref(old), 0) == 0
    assert cu.cuMemPoolCreate(C.byref(pool), C.byref(props)) == 0
    try:
        assert cu.cuDeviceSetMemPool(0, pool) == 0
        yield
    finally:
        assert cu.cuDeviceSetMemPool(0, old) == 0
        assert cu.cuMemPoolDestroy(pool) == 0


def wide(n, m=64, seed=0):
    """m rows of two entries each and n columns, most of them empty."""
    r = np.random.default_rng(seed)
    return synth.LP(m=m, n=n, row_ptr=np.arange(0, 2 * m + 1, 2, dtype=np.int32),
                    col_idx=np.arange(2 * m, dtype=np.int32), val=r.choice([-1.0, 2.0], 2 * m),
                    c=r.integers(-2, 3, n).astype(float), lhs=np.full(m, -INF), rhs=np.full(m, 3.0),
                    lb=np.full(n, -5.0), ub=np.full(n, 5.0))


def test_primal_postsolve_without_device_memory():
    r = lpp.presolve(wide(9_000_001))  # two vectors: 72 MB or more
    red = r.reduced()
    assert red.n > 0
    x = np.random.default_rng(1).standard_normal(red.n)
    want = np.where(r.col_kind != 0, r.col_val, np.nan)
    want[red.col_map] = x
    # a second record, none of whose arrays is on the host yet
    q = lpp.presolve(wide(9_000_001))
    with pool_limit(1 << 22):
        np.testing.assert_array_equal(q.postsolve_primal(x), want)
    np.testing.assert_array_equal(q.postsolve_primal(x), want)
    torch.cuda.synchronize()  # no error is left behind


def launches():
    f = lpp.load()._ZN3lpp12launch_countEv  # kernels the library has launched
    f.restype = C.c_int64
    return f()


# up to 65,536 columns
@pytest.mark.parametrize("n", [300, 65_536])
@pytest.mark.parametrize("first", ["postsolve", "records"])
def test_a_repeated_primal_postsolve_is_host_work(n, first):
    r = lpp.presolve(wide(n))
    red = r.reduced()
    r.info
    x, y = np.random.default_rng(2).standard_normal((2, red.n))
    if first == "records":
        r.col_kind
    a = r.postsolve_primal(x)
    k = launches()
    b = r.postsolve_primal(y)
    np.testing.assert_array_equal(r.postsolve_primal(x), a)
    assert launches() == k
    for got, sol in ((a, x), (b, y)):
        want = np.where(r.col_kind != 0, r.col_val, np.nan)
        want[red.col_map] = sol
        np.testing.assert_array_equal(got, want)


def test_primal_postsolve_waits_for_no_other_stream():
    lp = wide(65_537)
    warm = lpp.presolve(lp)
    x = np.random.default_rng(3).standard_normal(warm.info.n_red)
    want = warm.postsolve_primal(x)
    for r in (lpp.presolve(lp), warm):
        r.info
        torch.cuda._sleep(1_000_000_000)  # about half a second on the default stream
        busy = torch.cuda.Event()
        busy.record()
        got = r.postsolve_primal(x)
        assert not busy.query()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(got, want)


class SmResource(C.Structure):  # CUdevResource of streaming multiprocessors
    _fields_ = [("type", C.c_int), ("pad", C.c_ubyte * 92), ("sms", C.c_uint), ("rest", C.c_ubyte * 44)]


@contextlib.contextmanager
def small_stream(sms):
    """A stream that owns a part of the device of at least `sms` SMs (a green context's)."""
    cu = C.CDLL("libcuda.so.1")
    torch.cuda.current_stream()  # the device's primary context is there
    every, part, count = SmResource(), SmResource(), C.c_uint(1)
    desc, ctx, stream = C.c_void_p(), C.c_void_p(), C.c_void_p()
    assert cu.cuDeviceGetDevResource(0, C.byref(every), 1) == 0
    assert cu.cuDevSmResourceSplitByCount(C.byref(part), C.byref(count), C.byref(every), None, 0, sms) == 0
    assert cu.cuDevResourceGenerateDesc(C.byref(desc), C.byref(part), 1) == 0
    assert cu.cuGreenCtxCreate(C.byref(ctx), desc, 0, 1) == 0
    try:
        assert cu.cuGreenCtxStreamCreate(C.byref(stream), ctx, 1, 0) == 0  # non-blocking
        yield stream.value, part.sms, every.sms
        assert cu.cuStreamSynchronize(stream) == 0
        assert cu.cuStreamDestroy(stream) == 0
    finally:
        assert cu.cuGreenCtxDestroy(ctx) == 0


@pytest.mark.parametrize("m", [300, 30_000])
def test_presolve_on_a_stream_with_few_sms(m):
    """Its cooperative kernels hold two blocks per SM: the larger LP's are refused there."""
    lp = synth.skewed(5, m=m, n=3 * m // 2, target_nnz=10 * m, row_cap=9000)
    want = lpp.presolve(lp)
    with small_stream(8) as (stream, sms, every):
        assert sms <= every // 2
        got = lpp.presolve(lp, stream=stream)
        a, b = got.reduced(), want.reduced()
        x = np.random.default_rng(4).standard_normal(b.n)
        np.testing.assert_array_equal(got.postsolve_primal(x), want.postsolve_primal(x))
        got.close()
    assert want.rounds == got.rounds
    for k in ("row_ptr", "col_idx", "val", "c", "lhs", "rhs", "lb", "ub", "obj_offset", "row_map", "col_map", "csc_ptr",
              "csc_idx", "csc_val"):
        np.testing.assert_array_equal(getattr(a, k), getattr(b, k))


def at(offset, a):
    """The array on the device, `offset` bytes past a 256-byte boundary; keeps its memory."""
    raw = torch.zeros(offset + a.nbytes + 8, dtype=torch.uint8, device="cuda")
    raw[offset:offset + a.nbytes] = torch.from_numpy(a.view(np.uint8)).cuda()
    return raw, raw.data_ptr() + offset


@pytest.mark.parametrize("timing", [0, 1])
@pytest.mark.parametrize("shift", [0, 4, 8, 12, 1, 6])
def test_device_inputs_off_the_boundaries(shift, timing):
    """Device arrays that start off a boundary of their elements are copied, as host arrays are."""
    lp = synth.skewed(6, m=3000, n=4500, target_nnz=30000, row_cap=2000)
    keep, s = [], lpp.LpStruct(lp.m, lp.n, lp.val.size, on_device=1)
    for k, v in lp.arrays().items():
        raw, p = at(shift, np.ascontiguousarray(v, np.int32 if k in ("row_ptr", "col_idx") else np.float64))
        keep.append(raw)
        setattr(s, k, p)
    torch.cuda.synchronize()
    red, rec = C.c_void_p(), C.c_void_p()
    o = lpp.opts(timing=timing)
    assert lpp.load().lpp_presolve(C.byref(s), C.byref(o), C.byref(red), C.byref(rec)) == 0
    a, b = lpp.Result(red.value, rec.value).reduced(), lpp.presolve(lp, timing=timing).reduced()
    for k in ("row_ptr", "col_idx", "val", "c", "lhs", "rhs", "lb", "ub", "row_map", "col_map", "csc_ptr", "csc_idx",
              "csc_val"):
        np.testing.assert_array_equal(getattr(a, k), getattr(b, k))


def test_free_pinned_buffers_are_bounded():
    """Of five buffers of 1 GiB given back, at most the cache's 4 GiB stay pinned; one of them serves
    the next request of their size."""
    L, cu = lpp.load(), C.CDLL("libcuda.so.1")
    get, put = L._ZN3lpp16pinned_get_sizedEm, L._ZN3lpp10pinned_putEPv
    get.restype, get.argtypes, put.restype, put.argtypes = C.c_void_p, [C.c_size_t], None, [C.c_void_p]
    torch.cuda.synchronize()

    def pinned(p):
        kind = C.c_uint(0)
        return cu.cuPointerGetAttribute(C.byref(kind), 2, C.c_uint64(p)) == 0  # memory type

    ps = [get(1 << 30) for _ in range(5)]
    assert len(set(ps)) == 5 and all(pinned(p) for p in ps)
    for p in ps:
        put(p)
    left = [p for p in ps if pinned(p)]
    assert 1 <= len(left) <= 4
    q = get(1 << 30)
    assert q in left
    put(q)

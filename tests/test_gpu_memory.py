"""Idle memory of the library's pool with most of the device taken: the bound
holds by whichever function, context and order C is freed, a caller can have
it given back, and other allocations of the process get what is idle."""
import ctypes
import gc

import pytest

from paper_2106_14402_gb300 import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SR = "plus_times_f64"
MB = 1 << 20


@pytest.fixture(scope="module")
def cb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_14402_gb300 import cb as _cb
    _cb.load()
    return _cb


@pytest.fixture(scope="module")
def big(cb):
    """An operand whose square takes some GB, and the bytes of that square."""
    P = gen.rmat(16, 16, *gen.RMAT_ABCD, seed=980)
    dA = cb.DeviceCSR.from_host(P.with_values(gen.random_values(SR, P.nnz, 981)), SR)
    c_bytes = 12 * cb.spgemm(SR, dA, dA, ctx=cb.Context()).nnz
    assert c_bytes > 3 << 30
    return dA, c_bytes


def free_bytes():
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def product(cb, A, ctx):
    """C = A.A in arrays of the library, as a bare cb_csr."""
    sa, sc, opts = A.as_struct(), cb.cb_csr(), cb.make_opts()
    ctx.check(ctx.lib.cb_spgemm_ex(ctx.handle, 2, ctypes.byref(sa), ctypes.byref(sa), ctypes.byref(sc),
                                   ctypes.byref(opts)))
    return sc


@pytest.fixture
def others():
    """Takes all of the device but `left` bytes for the length of a test."""
    hold = []
    yield lambda left: hold.append(torch.empty(free_bytes() - left, dtype=torch.uint8, device="cuda"))
    hold.clear()
    free_bytes()


def idle_limit(beside):
    """What the pool may keep idle with `beside` bytes of the device free (a
    quarter of the device is more here), and a piece of slack."""
    return max(beside // 2, 1 << 30) + 64 * MB


@pytest.mark.parametrize("how", ["async", "async, other context", "free", "free after the context"])
def test_idle_bound_holds(cb, big, others, how):
    dA, c_bytes = big
    ctx, other = cb.Context(), cb.Context(torch.cuda.Stream())
    x = torch.ones(9, dtype=torch.int64, device="cuda")
    other.check(other.lib.cb_exclusive_scan(other.handle, x.data_ptr(), 8, x.data_ptr()))
    others(c_bytes + (4 << 30))
    base = free_bytes()
    sc = product(cb, dA, ctx)
    lib = ctx.lib
    if how == "free after the context":
        del ctx
    beside = free_bytes()
    in_use = base - beside - c_bytes           # workspaces
    if how.startswith("async"):
        lib.cb_csr_free_async((other if "other" in how else ctx).handle, ctypes.byref(sc))
    else:
        lib.cb_csr_free(ctypes.byref(sc))
    held = base - free_bytes()
    assert held <= in_use + idle_limit(beside), (held >> 20, in_use >> 20, beside >> 20)


def test_bound_does_not_rise_with_what_was_freed(cb, big, others):
    """Memory freed earlier, by any function, is not counted as in use."""
    dA, c_bytes = big
    before = free_bytes()
    for _ in range(3):
        ctx = cb.Context()
        ctx.lib.cb_csr_free(ctypes.byref(product(cb, dA, ctx)))
        del ctx
    assert before - free_bytes() <= 64 * MB
    ctx = cb.Context()
    others(c_bytes + (4 << 30))
    base = free_bytes()
    sc = product(cb, dA, ctx)
    beside = free_bytes()
    in_use = base - beside - c_bytes
    ctx.lib.cb_csr_free_async(ctx.handle, ctypes.byref(sc))
    held = base - free_bytes()
    assert held <= in_use + idle_limit(beside), (held >> 20, in_use >> 20, beside >> 20)


def test_other_allocations_get_idle_memory(cb, big, others):
    dA, c_bytes = big
    ctx = cb.Context(torch.cuda.Stream())
    before = free_bytes()
    cb.spgemm(SR, dA, dA, ctx=ctx)
    assert before - free_bytes() >= c_bytes
    others(-c_bytes // 2)                      # half of C more than is free


def test_trim_gives_idle_memory_back(cb, big):
    dA, c_bytes = big
    ctx = cb.Context()
    before = free_bytes()
    C = cb.spgemm(SR, dA, dA, ctx=ctx)
    in_use = before - free_bytes() - c_bytes
    del C
    for keep in (1 << 30, 0):
        ctx.trim(keep)
        assert before - free_bytes() <= in_use + keep + 64 * MB
    C = cb.spgemm(SR, dA, dA, ctx=ctx)         # what is in use stays
    ctx.trim()
    assert 12 * C.nnz == c_bytes and int(C.row_ptr[-1]) == C.nnz
    with pytest.raises(cb.CBError):
        ctx.trim(-1)
    cb.Context().trim()                        # nothing allocated yet


def test_idle_memory_counts_as_free_for_the_bitmaps(cb, big, others):
    """A second call keeps the heavy rows' bitmaps (and with them the (or,and)
    read-out, one launch less) where the first one did, although the first
    one's C is now idle memory."""
    P, _ = big
    A = cb.DeviceCSR(P.nrows, P.ncols, P.row_ptr, P.col, torch.ones(P.nnz, dtype=torch.uint8, device="cuda"))
    bits = 32768 * int((cb.row_stats(A, A)[0].clamp(max=P.ncols) > 512).sum())
    before = free_bytes()
    ctx = cb.Context()
    C = cb.spgemm("or_and_bool", A, A, ctx=ctx)
    want, c_bytes = ctx.stats()["kernels"], 5 * C.nnz
    in_use = before - free_bytes() - c_bytes
    assert in_use >= bits
    del C, ctx
    ctx = cb.Context()
    others(4 * bits + in_use + c_bytes // 4)
    for _ in range(2):
        cb.spgemm("or_and_bool", A, A, ctx=ctx)
        assert ctx.stats()["kernels"] == want

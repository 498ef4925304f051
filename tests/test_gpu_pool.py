"""The context's memory pool: what a call frees serves the next one, the idle
part stays within a quarter of the device's memory, contexts on several
threads and streams do not disturb each other, and everything goes back with
the context."""
import gc
import threading

import pytest

import oracle
from paper_2106_14402_gb300 import gen
from parity import compare_rows

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_14402_gb300 import cb as _cb
    _cb.load()
    return _cb


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()


def test_idle_memory_is_bounded_and_given_back(cb):
    sr = "plus_times_f64"
    P = gen.rmat(14, 16, *gen.RMAT_ABCD, seed=900)
    A = P.with_values(gen.random_values(sr, P.nnz, 901))
    dA = cb.DeviceCSR.from_host(A, sr)
    cb.spgemm(sr, dA, dA, ctx=cb.Context())  # modules loaded
    gc.collect()
    before, total = free_bytes()
    ctx = cb.Context()
    first = cb.spgemm(sr, dA, dA, ctx=ctx)
    c_bytes = 12 * first.nnz
    del first
    gc.collect()
    held = before - free_bytes()[0]
    assert held <= total // 4 + (256 << 20)
    for _ in range(3):                      # later calls fit what the first one freed
        C = cb.spgemm(sr, dA, dA, ctx=ctx)
        del C
    gc.collect()
    assert before - free_bytes()[0] <= held + c_bytes // 2
    del ctx
    gc.collect()
    assert before - free_bytes()[0] <= 64 << 20


def test_c_outlives_its_context(cb):
    sr = "plus_times_i64"
    P = gen.rmat(10, 8, *gen.RMAT_ABCD, seed=902)
    A = P.with_values(gen.random_values(sr, P.nnz, 903))
    dA = cb.DeviceCSR.from_host(A, sr)
    want = oracle.spgemm(sr, A, A)
    lib = cb.load()
    import ctypes
    ctx = cb.Context()
    sa, sc, opts = dA.as_struct(), cb.cb_csr(), cb.make_opts()
    ctx.check(lib.cb_spgemm_ex(ctx.handle, 1, ctypes.byref(sa), ctypes.byref(sa), ctypes.byref(sc),
                               ctypes.byref(opts)))
    torch.cuda.synchronize()
    del ctx
    gc.collect()
    dev = dA.row_ptr.device
    C = cb.DeviceCSR(sc.nrows, sc.ncols, cb._wrap(sc.row_ptr, sc.nrows + 1, torch.int64, None, dev),
                     cb._wrap(sc.col, sc.nnz, torch.int32, None, dev),
                     cb._wrap(sc.val, sc.nnz, torch.int64, None, dev))
    compare_rows(sr, C.to_host(), want)
    lib.cb_csr_free(ctypes.byref(sc))


def test_contexts_on_threads_and_streams(cb):
    sr = "min_plus_u32"
    P = gen.rmat(12, 16, *gen.RMAT_ABCD, seed=904)
    A = P.with_values(gen.random_values(sr, P.nnz, 905))
    dA = cb.DeviceCSR.from_host(A, sr)
    want = oracle.spgemm(sr, A, A)
    torch.cuda.synchronize()
    errors = []

    def work():
        try:
            stream = torch.cuda.Stream()
            ctx = cb.Context(stream)
            for k in range(8):
                C = cb.spgemm(sr, dA, dA, ctx=ctx)
                stream.synchronize()
                if k % 4 == 3:
                    compare_rows(sr, C.to_host(), want)
        except Exception as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work) for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]

"""A queued validation stops the call before any kernel reads through a bad
index: the call fails with CB_ERR_INDEX, caller buffers stay untouched and the
context serves the next product (one-launch, work-queue and two-phase shapes;
arrays on and off a 16-byte boundary)."""
import numpy as np
import pytest

import oracle
from paper_2106_14402_gb300 import gen
from parity import compare_rows

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
CB_ERR_INDEX = 4
SR = "min_plus_u32"


@pytest.fixture(scope="module")
def cb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_14402_gb300 import cb as _cb
    _cb.load()
    return _cb


def operand(cb, M, off=0):
    d = cb.DeviceCSR.from_host(M, SR)
    if off:
        col = torch.empty(M.nnz + off, dtype=torch.int32, device="cuda")
        col[off:] = d.col
        d = cb.DeviceCSR(d.nrows, d.ncols, d.row_ptr, col[off:], d.val)
    return d


@pytest.mark.parametrize("deg", [4, 40, 120])      # one launch, work queue, two-phase
@pytest.mark.parametrize("bad", ["A col high", "A col negative", "A row_ptr", "B col last", "B row_ptr end"])
@pytest.mark.parametrize("off", [0, 1])
def test_bad_index_is_caught_before_use(cb, deg, bad, off):
    n = 2001
    A, B = gen.er_exact(n, n, deg, 920), gen.er_exact(n, n, deg, 921)
    A, B = (M.with_values(gen.random_values(SR, M.nnz, 922 + k)) for k, M in enumerate((A, B)))
    dA, dB = operand(cb, A, off), operand(cb, B, off)
    ctx = cb.Context()
    want = oracle.spgemm(SR, A, B)
    target = dA if bad[0] == "A" else dB
    if "row_ptr" in bad:
        saved = target.row_ptr.clone()
        if "end" in bad:
            target.row_ptr[-1] += 1
        else:
            target.row_ptr[5] = target.row_ptr[7] + 1
    else:
        saved = target.col.clone()
        at = {"A col high": 4, "A col negative": A.nnz // 2, "B col last": B.nnz - 1}[bad]
        target.col[at] = -1 if "negative" in bad else n
    size = int(want[0][-1])
    out = cb.DeviceCSR(0, 0, torch.full((n + 1,), -7, dtype=torch.int64, device="cuda"),
                       torch.full((size,), -7, dtype=torch.int32, device="cuda"),
                       torch.full((size,), 77, dtype=torch.int32, device="cuda").view(torch.uint32))
    for buffers in (None, out):
        with pytest.raises(cb.CBError) as e:
            cb.spgemm(SR, dA, dB, ctx=ctx, out=buffers)
        assert e.value.code == CB_ERR_INDEX and ctx.error().startswith(bad[0] + ":")
    assert bool((out.col == -7).all()) and bool((out.row_ptr == -7).all())
    (target.row_ptr if "row_ptr" in bad else target.col).copy_(saved)
    compare_rows(SR, cb.spgemm(SR, dA, dB, ctx=ctx).to_host(), want)


@pytest.mark.parametrize("deg", [4, 40, 120])
def test_caller_struct_is_untouched(cb, deg):
    """A failed validation leaves every field of a caller-provided C as it was."""
    import ctypes
    n = 2001
    A = gen.er_exact(n, n, deg, 924)
    dA = operand(cb, A.with_values(gen.random_values(SR, A.nnz, 925)))
    dA.col[A.nnz - 1] = n
    rp, col = (torch.empty(k, dtype=t, device="cuda") for k, t in ((n + 1, torch.int64), (9, torch.int32)))
    sa, opts = dA.as_struct(), cb.make_opts(out_capacity=9)
    sc = cb.cb_csr(11, 12, 13, rp.data_ptr(), col.data_ptr(), col.data_ptr())
    ctx = cb.Context()
    rc = ctx.lib.cb_spgemm_ex(ctx.handle, 3, ctypes.byref(sa), ctypes.byref(sa), ctypes.byref(sc), ctypes.byref(opts))
    assert rc == CB_ERR_INDEX
    assert (sc.nrows, sc.ncols, sc.nnz) == (11, 12, 13)
    assert (sc.row_ptr, sc.col, sc.val) == (rp.data_ptr(), col.data_ptr(), col.data_ptr())

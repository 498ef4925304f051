"""(or,and) products: the values of C come from its pattern when no stored
value is false, and from the products otherwise; either way C equals the
oracle's.  Value arrays start at odd addresses, rows span several bitmap
spans, and a single false value (first, last, in A or in B) turns the path."""
import numpy as np
import pytest

import oracle
from paper_2106_14402_gb300 import gen
from parity import compare_rows
from test_gpu_parity import _tiered_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SR = "or_and_bool"


@pytest.fixture(scope="module")
def cb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_14402_gb300 import cb as _cb
    _cb.load()
    return _cb


def shifted(cb, M, by):
    d = cb.DeviceCSR.from_host(M, SR)
    v = torch.zeros(M.nnz + by, dtype=torch.uint8, device="cuda")
    v[by:] = d.val
    return cb.DeviceCSR(d.nrows, d.ncols, d.row_ptr, d.col, v[by:])


@pytest.mark.parametrize("false_at", [None, ("A", 0), ("A", -1), ("B", 0), ("B", -1)])
@pytest.mark.parametrize("ncols", [5000, 600000])
def test_true_and_false_values(cb, ncols, false_at):
    A, B = _tiered_inputs(SR, seed=910, ncols=ncols)
    A = A.with_values(np.full(A.nnz, 1, np.uint8))
    B = B.with_values(np.where(np.arange(B.nnz) % 2, 1, 255).astype(np.uint8))
    if false_at:
        (A if false_at[0] == "A" else B).val[false_at[1]] = 0
    want = oracle.spgemm(SR, A, B)
    for by in (0, 3):
        C = cb.spgemm(SR, shifted(cb, A, by), shifted(cb, B, 7 - by), check=True, fused=False)
        compare_rows(SR, C.to_host(), want)


@pytest.mark.parametrize("by", [1, 5, 15])
def test_unaligned_output_values(cb, by):
    P = gen.rmat(11, 16, *gen.RMAT_ABCD, seed=911)
    A = P.with_values(np.ones(P.nnz, np.uint8))
    want = oracle.spgemm(SR, A, A)
    n = int(want[0][-1])
    dA = cb.DeviceCSR.from_host(A, SR)
    val = torch.full((n + 32,), 77, dtype=torch.uint8, device="cuda")
    out = cb.DeviceCSR(0, 0, torch.empty(A.nrows + 1, dtype=torch.int64, device="cuda"),
                       torch.empty(n, dtype=torch.int32, device="cuda"), val[by:by + n])
    C = cb.spgemm(SR, dA, dA, out=out, fused=False)
    compare_rows(SR, C.to_host(), want)
    v = val.cpu().numpy()
    assert (v[:by] == 77).all() and (v[by + n:] == 77).all()


def test_column_batches(cb):
    P = gen.rmat(11, 16, *gen.RMAT_ABCD, seed=912)
    A = P.with_values(np.ones(P.nnz, np.uint8))
    want = oracle.spgemm(SR, A, A)
    dA = cb.DeviceCSR.from_host(A, SR)
    parts = []
    cb.spgemm_column_batches(SR, dA, dA, 8 * (A.nrows + 1) + 5 * int(want[0][-1]) // 3,
                             lambda b, lo, hi, Cb: parts.append(tuple(x.copy() for x in Cb.to_host())))
    assert len(parts) >= 3
    sizes = sum(np.diff(p[0]) for p in parts)
    assert np.array_equal(sizes, np.diff(want[0]))
    rows = [np.concatenate([p[1][p[0][r]:p[0][r + 1]] for p in parts]) for r in range(A.nrows)]
    assert np.array_equal(np.concatenate(rows), want[1])
    assert all((p[2] == 1).all() for p in parts)

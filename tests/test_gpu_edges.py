"""Sizes at which the tiled and tabled kernels change their course, against
the oracle: rank windows either side of a split-table boundary and of a bitmap
span, rows of the work-queue kernel either side of its staging, marking and
repeat limits, long rows of the row counting, and ragged row tiles of the
sizer kernels.  fp64 products are compared at parity.py's bound (its m is at
most 900 here); all other results bit for bit."""
import numpy as np
import pytest

import oracle
from oracle import mlp
from paper_2106_14402_gb300 import gen
from parity import compare_rows
from test_gpu_mlp import flat, forward_at_kernel_rounding, reference_inputs, setup_problem, unflat
from test_gpu_parity import _tiered_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SR = gen.SEMIRINGS


@pytest.fixture(scope="module")
def cb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_14402_gb300 import cb as _cb
    _cb.load()
    return _cb


def rows_reversed(M):
    """M with the entries of each row in descending order."""
    at = np.concatenate([np.arange(M.row_ptr[r + 1] - 1, M.row_ptr[r] - 1, -1) for r in range(M.nrows)])
    return gen.CSR(M.nrows, M.ncols, M.row_ptr, M.col[at], M.val[at])


def multiply(cb, sr, A, B, ctx=None, **kw):
    dA, dB = (cb.DeviceCSR.from_host(M, sr, operand=o) for M, o in ((A, "A"), (B, "B")))
    ctx = ctx or cb.context()
    return cb.spgemm(sr, dA, dB, ctx=ctx, **kw).to_host(), ctx.stats()


# rank windows: B rows cut by the split table (sorted) and by searching (not)
@pytest.mark.parametrize("ncols", [4095, 4096, 4097, 3 * 4096 + 1, (1 << 18) - 1, (1 << 18) + 1, (1 << 19) + 4097])
@pytest.mark.parametrize("sr", SR)
def test_rank_windows_at_boundaries(cb, sr, ncols):
    A, B = _tiered_inputs(sr, seed=930, ncols=ncols)
    want = oracle.spgemm(sr, A, B)
    assert np.diff(want[0]).max() > 2500
    for b in (B, rows_reversed(B)):
        compare_rows(sr, multiply(cb, sr, A, b, fused=False)[0], want)


@pytest.mark.parametrize("sr", ["min_plus_u32", "plus_times_i64"])
def test_rank_windows_of_column_batches(cb, sr):
    A, B = _tiered_inputs(sr, seed=931, ncols=300001)
    want = oracle.spgemm(sr, A, B)
    width = 4 + want[2].itemsize
    dA, dB = cb.DeviceCSR.from_host(A, sr), cb.DeviceCSR.from_host(B, sr)
    parts = []
    cb.spgemm_column_batches(sr, dA, dB, 8 * (A.nrows + 1) + width * int(want[0][-1]) // 3,
                             lambda b, lo, hi, C: parts.append(tuple(x.copy() for x in C.to_host())))
    assert len(parts) >= 3
    assert np.array_equal(sum(np.diff(p[0]) for p in parts), np.diff(want[0]))
    for k in (1, 2):
        got = [p[k][p[0][r]:p[0][r + 1]] for r in range(A.nrows) for p in parts]
        assert np.array_equal(np.concatenate(got), want[k])


def fixed_rows(lens, ncols, seed, sr, operand="A"):
    """Rows of the given lengths with random distinct columns, not sorted."""
    rng = np.random.default_rng(seed)
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    col = np.concatenate([rng.permutation(ncols)[:k] for k in lens]).astype(np.int32)
    return gen.CSR(len(lens), ncols, rp, col, gen.random_values(sr, int(rp[-1]), seed + 1))


# (A's row lengths, B's row lengths, B's columns): staging of 128 A entries;
# marked and unmarked rows (8 steps); empty groups of B rows; more than 256
# repeats; widths either side of the prefix's words per thread
QUEUE = [([127, 128, 129, 0, 1, 300], [12], 60000),
         ([60, 100], [31, 32, 33, 0, 0, 0, 0, 0, 0], 4097),
         ([60, 63], [63, 64, 65, 1], 16384),
         ([64, 33, 1], [64], 200),
         ([1, 1, 0], [4000, 4096, 3], 16385),
         ([200, 130], [0, 0, 0, 0, 20], 65536),
         ([70, 5], [40, 33], 65535)]


@pytest.mark.parametrize("case", range(len(QUEUE)))
@pytest.mark.parametrize("sr", SR)
def test_queue_rows_at_limits(cb, sr, case):
    la, lb, ncols = QUEUE[case]
    n = 800
    A = fixed_rows([la[i % len(la)] for i in range(1500)], n, 940 + case, sr)
    B = fixed_rows([lb[i % len(lb)] for i in range(n)], ncols, 960 + case, sr)
    got, st = multiply(cb, sr, A, B)
    assert oracle.row_stats(A, B)[0].max() <= 4096
    assert st["kernels"] == 6, st["kernels"]
    compare_rows(sr, got, oracle.spgemm(sr, A, B))


@pytest.mark.parametrize("m, step", [(7, 1), (100000, 1000)])
def test_row_counting_of_long_rows(cb, m, step):
    """Rows around the CTA-wide limit; the second size has more long rows than
    a CTA keeps aside."""
    i = torch.arange(m, device="cuda")
    lens = torch.where(i % step == 0, torch.tensor([1023, 1024, 1025, 3000, 0, 1, 33], device="cuda")[i // step % 7], 1025)
    rp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(lens, 0)
    n = 4096
    col = (torch.arange(int(rp[-1]), device="cuda") * 5 % n).to(torch.int32)
    blen = torch.arange(n, device="cuda") % 3
    brp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    brp[1:] = torch.cumsum(blen, 0)
    one = lambda k: torch.ones(k, dtype=torch.uint8, device="cuda")
    A = cb.DeviceCSR(m, n, rp, col, one(col.numel()))
    B = cb.DeviceCSR(n, 64, brp, torch.zeros(int(brp[-1]), dtype=torch.int32, device="cuda"), one(int(brp[-1])))
    F = cb.row_features(A, B).cpu().numpy().astype(np.int64)
    ends = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), torch.cumsum(blen[col.long()], 0)])
    assert np.array_equal(F[:, 0], lens.cpu().numpy())
    assert np.array_equal(F[:, 1], (ends[rp[1:]] - ends[rp[:-1]]).cpu().numpy())


# sizer: a row's logit does not depend on the tile that holds it
@pytest.mark.parametrize("m", [1, 31, 32, 33, 63, 64, 65, 127, 129, 255, 256, 257])
def test_sizer_row_tiles(cb, m):
    A, F, nnz, norm, p = setup_problem(2)
    model = cb.MLP(flat(p).astype(np.float32), norm)
    feat = torch.tensor(F, dtype=torch.float32, device="cuda")
    z_all, pred_all = model.predict(feat, ncols=A.ncols)
    z, pred = model.predict(feat[:m].contiguous(), ncols=A.ncols)
    assert torch.equal(z, z_all[:m]) and torch.equal(pred, pred_all[:m])
    g, loss = model.grad(feat[:m].contiguous(), torch.tensor(nnz[:m], dtype=torch.int64, device="cuda"), tau=0.9)
    g = unflat(g.cpu().numpy().astype(np.float64))
    q, X = reference_inputs(F[:m], norm, p)
    zr, cache = forward_at_kernel_rounding(q, X)
    L, dz = mlp.loss_and_dz(zr, F[:m, 1], nnz[:m], 0.9)
    want = mlp.backward(q, cache, dz)
    Xa, h1, _, h2, _ = cache
    gabs = mlp.backward({k: np.abs(v) for k, v in q.items()}, (np.abs(Xa), h1, h1, h2, h2), np.abs(dz))
    # one bf16 unit of one row's activation (test_gpu_mlp.py's bound): with few
    # rows that row may be all of the entry's sum, which the bound covers
    for k in want:
        assert (np.abs(g[k] - want[k]) <= 2.0 ** -8 * gabs[k] + 1e-7).all(), k


@pytest.mark.parametrize("bad", [-1, 700])
def test_spmspv_queued_validation(cb, bad):
    sr = "min_plus_u32"
    A = gen.random_csr(500, 700, 0.05, seed=970, semiring=sr)
    dA = cb.DeviceCSR.from_host(A, sr)
    xi = torch.arange(0, 500, 3, dtype=torch.int32, device="cuda")
    xv = torch.arange(xi.numel(), dtype=torch.int32, device="cuda").view(torch.uint32)
    ctx = cb.Context()
    want = [t.view(torch.int32).cpu() for t in cb.spmspv(sr, dA, xi, xv, ctx=ctx)]
    saved = dA.col[9].clone()
    dA.col[9] = bad
    with pytest.raises(cb.CBError) as e:
        cb.spmspv(sr, dA, xi, xv, ctx=ctx)
    assert e.value.code == 4
    dA.col[9] = saved
    got = [t.view(torch.int32).cpu() for t in cb.spmspv(sr, dA, xi, xv, ctx=ctx)]
    assert all(torch.equal(a, b) for a, b in zip(got, want))

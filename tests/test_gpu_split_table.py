"""The split table of sorted B rows: distances between its boundaries beyond
the smallest, and products for which it is not built, which then hold no
memory for it either."""
import gc

import numpy as np
import pytest

import oracle
from paper_2106_14402_gb300 import gen
from parity import compare_rows

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def cb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_14402_gb300 import cb as _cb
    _cb.load()
    return _cb


def operands(sr, n, ncols, spread, seed):
    """40 rows of A that name 30 of B's n rows each; those hold 600 columns
    below `spread`, many of them at multiples of 2^12 and on either side."""
    rng = np.random.default_rng(seed)
    used = np.unique(np.concatenate([rng.integers(0, n, 200), [0, n - 1]]))
    at = np.concatenate([[x - 1, x, x + 1] for x in range(4096, spread, 4096)] + [[0, spread - 1]])
    at = at[at < spread]
    rows = []
    for _ in used:
        c = np.concatenate([rng.choice(at, min(at.size // 2, 200), replace=False), rng.integers(0, spread, 800)])
        rows.append(np.sort(rng.permutation(np.unique(c))[:600]))
    lens = np.zeros(n, np.int64)
    lens[used] = [r.size for r in rows]
    rp = np.concatenate([[0], np.cumsum(lens)])
    B = gen.CSR(n, ncols, rp, np.concatenate(rows).astype(np.int32), gen.random_values(sr, int(rp[-1]), seed + 1))
    acol = np.concatenate([np.sort(rng.choice(used, 30, replace=False)) for _ in range(40)]).astype(np.int32)
    A = gen.CSR(40, n, np.arange(41, dtype=np.int64) * 30, acol, gen.random_values(sr, acol.size, seed + 2))
    return A, B


def free_bytes():
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


# B's rows, columns, highest column in use: boundaries 2^14 columns apart; a
# table that would be too large at any distance; rows of one window each
@pytest.mark.parametrize("sr", ["plus_times_i64", "min_plus_u32"])
@pytest.mark.parametrize("n, ncols, spread", [(1 << 19, 1 << 20, 1 << 20), (40_000_000, 1 << 20, 1 << 20),
                                              (1 << 19, 1 << 18, 1 << 18)])
def test_table_shapes(cb, sr, n, ncols, spread):
    A, B = operands(sr, n, ncols, spread, 990)
    want = oracle.spgemm(sr, A, B)
    assert np.diff(want[0]).min() > 4096
    dA, dB = cb.DeviceCSR.from_host(A, sr), cb.DeviceCSR.from_host(B, sr)
    cb.spgemm(sr, dA, dB, ctx=cb.Context())    # modules loaded
    before = free_bytes()
    ctx = cb.Context()
    C = cb.spgemm(sr, dA, dB, ctx=ctx)
    compare_rows(sr, C.to_host(), want)
    del C
    ctx.trim()
    # workspaces without a table, the 8-byte windows' slices among them (three
    # CTAs an SM, 16384 entries of 8 bytes, a quarter to spare)
    assert before - free_bytes() <= 64 * MB + 3 * 152 * 16384 * 8 * 5 // 4


def test_rows_beyond_32_bit_positions(cb):
    """A row of more than 2^31 entries (2048 of each column): no table, whose
    positions in a row are 32-bit."""
    n, each = (1 << 20) + 1, 2048
    nnz = n * each
    assert nnz > 1 << 31
    col = torch.arange(n, dtype=torch.int32, device="cuda")
    val = (col % 1000 + 1).repeat_interleave(each)
    val.view(n, each)[:, -1] -= 1              # the smallest of each column comes last
    B = cb.DeviceCSR(1, n, torch.tensor([0, nnz], device="cuda"), col.repeat_interleave(each), val.view(torch.uint32))
    A = cb.DeviceCSR(2, 1, torch.tensor([0, 1, 2], device="cuda"), torch.zeros(2, dtype=torch.int32, device="cuda"),
                     torch.tensor([5, 7], dtype=torch.int32, device="cuda").view(torch.uint32))
    C = cb.spgemm("min_plus_u32", A, B, ctx=cb.Context())
    assert C.row_ptr.tolist() == [0, n, 2 * n]
    assert torch.equal(C.col, torch.cat([col, col]))
    assert torch.equal(C.val.view(torch.int32), torch.cat([col % 1000 + 5, col % 1000 + 7]))

"""A row of A whose first 512 entries name 2^31 products or more, beyond the
32-bit offsets of the product loop: whole rows and slices of them, sorted and
not, and three more entries within the offsets.  Sums and minima of duplicates
in closed form; integers, so equal bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_14402_gb300 import cb as _cb
    _cb.load()
    return _cb


# columns: one rank window, or two (an 8-byte window holds 16384 entries, a
# 4-byte one about 15000); sorted slices are longer so that one window's part
# still takes 2^22 entries of each of the 512 rows
@pytest.mark.parametrize("sr, ncols, length, ordered", [("min_plus_u32", 8192, 1 << 22, False),
                                                        ("plus_times_i64", 8192, 1 << 22, True),
                                                        ("min_plus_u32", 24000, 1 << 22, False),
                                                        ("plus_times_i64", 24000, 6_300_000, True)])
def test_chunks_beyond_32_bit_offsets(cb, sr, ncols, length, ordered):
    dt = cb.SEMIRING[sr][1]
    kind = torch.int32 if dt == torch.uint32 else torch.int64
    col = torch.arange(length, device="cuda") % ncols
    if ordered:
        col = col.sort().values
    b = (torch.arange(length, device="cuda") * 7919 % 1009 + 1).to(kind)
    a = (torch.arange(515, device="cuda") * 31 % 101 + 2).to(kind)
    A = cb.DeviceCSR(1, 1, torch.tensor([0, 515], device="cuda"), torch.zeros(515, dtype=torch.int32, device="cuda"),
                     a.view(dt))
    B = cb.DeviceCSR(1, ncols, torch.tensor([0, length], device="cuda"), col.to(torch.int32), b.view(dt))
    C = cb.spgemm(sr, A, B, ctx=cb.Context())
    if sr == "min_plus_u32":
        want = torch.full((ncols,), 1 << 30, dtype=kind, device="cuda").scatter_reduce(0, col, b, "amin") + a.min()
    else:
        want = torch.zeros(ncols, dtype=kind, device="cuda").index_add(0, col, b) * a.sum()
    assert C.row_ptr.tolist() == [0, ncols]
    assert torch.equal(C.col, torch.arange(ncols, dtype=torch.int32, device="cuda"))
    assert torch.equal(C.val.view(kind), want)

"""Order-preserving selection at the edges of its scanner: one scanner chunk is 128 tiles, so
row counts just below, at and above 1 and 2 chunks of each tile shape, a last tile of one
row, and a column of many chunks; all, none, one and about a third of the rows selected."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

I32_MIN, I32_MAX = -(1 << 31), (1 << 31) - 1


@pytest.fixture(scope="module")
def crys():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2003_01178_gb300 import _build
    _build.build()
    import paper_2003_01178_gb300 as crys
    crys.crys_device_errors(clear=True)
    yield crys
    assert crys.crys_device_errors(clear=True) == 0
    crys.crys_set_tile(crys.OP_SELECT, 0)


@pytest.mark.parametrize("variant", range(4))
@pytest.mark.parametrize("tiles", [1, 2, 127, 128, 129, 256, 257, 5000])
def test_ordered_select_at_chunk_edges(crys, variant, tiles):
    threads, items = crys.crys_tile_variants(crys.OP_SELECT)[variant]
    crys.crys_set_tile(crys.OP_SELECT, variant)
    for n in (tiles * threads * items - 3, tiles * threads * items, tiles * threads * items + 1):
        g = torch.Generator(device="cuda")
        g.manual_seed(n)
        x = torch.randint(0, 1 << 20, (n,), dtype=torch.int32, device="cuda", generator=g)
        x[n - 1] = -5                                   # the one row of the last range
        for lo, hi in [(I32_MIN, I32_MAX), (1 << 20, I32_MAX), (0, (1 << 20) // 3), (-5, -5)]:
            got = crys.select(x, lo, hi, order_preserving=True)
            assert torch.equal(got, x[(x >= lo) & (x <= hi)]), (n, lo, hi)
    crys.crys_set_tile(crys.OP_SELECT, 0)


@pytest.mark.parametrize("n", [1, 2, 5, 31, 33, 4095, 4097, 32_767, 32_769, 65_535, 65_536, 65_537, 100_003, 131_071, 131_072, 131_073])
@pytest.mark.parametrize("ordered", [False, True])
def test_select_of_one_cluster(crys, n, ordered):
    # one cluster of 8 blocks selects up to 131072 rows, 65536 without an order to keep (and keeps
    # it all the same)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x = torch.randint(I32_MIN, I32_MAX, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
    for lo, hi in [(I32_MIN, I32_MAX), (0, I32_MAX), (-(1 << 28), 1 << 20), (int(x[n // 2]), int(x[n // 2])), (1, 0)]:
        got = crys.select(x, lo, hi, order_preserving=ordered)
        ref = x[(x >= lo) & (x <= hi)]
        if n <= 65_536 or ordered:
            assert torch.equal(got, ref), (lo, hi)
        else:
            assert torch.equal(got.sort().values, ref.sort().values), (lo, hi)

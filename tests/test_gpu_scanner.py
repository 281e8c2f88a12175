"""The scanner blocks of the ordered selection and of the sort's passes at few tiles and at the
edges of their chunks (128 tiles of a selection, 16 of a pass).  Columns this short normally
take one launch of their own; a request for a stall at tile 0, which stalls nothing,
sends them through the tiles."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

I32_MIN, I32_MAX = -(1 << 31), (1 << 31) - 1
BOUND = 2_000_000_000


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
@pytest.mark.parametrize("tiles", [1, 2, 3, 127, 128, 129, 256])
def test_select_tiles(crys, variant, tiles):
    threads, items = crys.crys_tile_variants(crys.OP_SELECT)[variant]
    crys.crys_set_tile(crys.OP_SELECT, variant)
    for n in (tiles * threads * items - 3, tiles * threads * items, tiles * threads * items + 1):
        g = torch.Generator(device="cuda")
        g.manual_seed(n)
        x = torch.randint(0, 1 << 20, (n,), dtype=torch.int32, device="cuda", generator=g)
        x[n - 1] = -5
        for lo, hi in [(I32_MIN, I32_MAX), (1 << 20, I32_MAX), (0, (1 << 20) // 3), (-5, -5)]:
            crys.crys_debug_stall(crys.OP_SELECT, 0, BOUND)
            got = crys.select(x, lo, hi, order_preserving=True)
            assert torch.equal(got, x[(x >= lo) & (x <= hi)]), (n, lo, hi)
    crys.crys_set_tile(crys.OP_SELECT, 0)


def _keys(kind, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(n + len(kind))
    if kind == "bits":
        return torch.randint(I32_MIN, I32_MAX, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
    if kind == "dense":
        return torch.randperm(n, device="cuda", generator=g).to(torch.int32) - n // 2
    if kind == "few":
        return torch.randint(-3, 4, (n,), dtype=torch.int32, device="cuda", generator=g)
    if kind == "equal":
        return torch.full((n,), -7, dtype=torch.int32, device="cuda")
    # most rows in one narrow range, a bucket too large for a block: four digits
    k = torch.randint(0, 300, (n,), dtype=torch.int32, device="cuda", generator=g)
    k[n // 3] = I32_MIN
    k[n // 2] = I32_MAX
    k[:n // 8] *= 7_000_001
    return k


@pytest.mark.parametrize("kind", ["bits", "dense", "few", "equal", "clustered"])
@pytest.mark.parametrize("n", [4993, 8191, 8193, 65_535, 65_536, 65_537, 131_073, 300_001, (1 << 20) - 1, 1 << 20])
def test_sort_passes(crys, n, kind):
    # up to 2^20 rows the general steps: 256 buckets after one pass, or the digits
    keys = _keys(kind, n)
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    rk, order = torch.sort(keys, stable=True)
    for _ in range(3):
        crys.crys_debug_stall(crys.OP_SORT, 0, BOUND)
        ko, vo = crys.sort(keys, vals)
        assert torch.equal(ko, rk) and torch.equal(vo, order.to(torch.int32))


@pytest.mark.parametrize("variant", range(4))
@pytest.mark.parametrize("kind", ["bits", "few", "clustered"])
@pytest.mark.parametrize("n", [(1 << 20) + 1, 3_000_017])
def test_sort_shapes(crys, n, kind, variant):
    # every tile shape by buckets (but the one that leaves no room for the counts) and by digits
    keys = _keys(kind, n)
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    rk, order = torch.sort(keys, stable=True)
    crys.crys_set_tile(crys.OP_SORT, variant)
    try:
        ko, vo = crys.sort(keys, vals)
    finally:
        crys.crys_set_tile(crys.OP_SORT, 0)
    assert torch.equal(ko, rk) and torch.equal(vo, order.to(torch.int32))

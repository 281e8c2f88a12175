"""Sorts over key sets that decide their buckets: row counts at the edges of one block
(4992 rows), one partition pass (2^20 rows) and the tiles; narrow, offset and full key
ranges, ranges with far outliers that a sample misses, repeated keys that crowd the bins of
a bucket, and one key value only.  The result is checked against torch's stable sort:
exactly for the stable sort, keys and key-value pairs for the unstable one."""
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


def _keys(kind, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(n * 7 + len(kind))

    def uni(lo, hi):
        return torch.randint(lo, hi + 1, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
    if kind == "bits":
        return uni(I32_MIN, I32_MAX)
    if kind == "dense":
        return torch.randperm(n, device="cuda", generator=g).to(torch.int32)
    if kind == "offset":                       # a narrow range that crosses zero
        return uni(-n, n // 3)
    if kind == "top":                          # up to the largest key
        return uni(I32_MAX - 5 * n, I32_MAX)
    if kind == "repeats":                      # about 64 rows per key: crowded bins
        return uni(0, max(1, n // 64))
    if kind == "wide_repeats":                 # the same, keys far apart
        return uni(0, max(1, n // 64)) * 1021
    if kind == "few":
        return uni(-3, 3)
    if kind == "equal":
        return torch.full((n,), -7, dtype=torch.int32, device="cuda")
    k = uni(0, n)                              # outliers
    k[n // 2] = I32_MAX
    k[n // 3] = I32_MIN
    return k


KINDS = ["bits", "dense", "offset", "top", "repeats", "wide_repeats", "few", "equal", "outliers"]
SIZES = [2, 33, 383, 4991, 4992, 4993, 6145, 70_001, (1 << 20) - 1, (1 << 20) + 1, 3_000_017]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", SIZES)
def test_msb_sort_ranges(crys, n, kind):
    keys = _keys(kind, n)
    vals = torch.randint(I32_MIN, I32_MAX, (n,), dtype=torch.int64, device="cuda").to(torch.int32)
    ko, vo = crys.sort_msb(keys, vals)
    rk, order = torch.sort(keys, stable=True)
    assert torch.equal(ko, rk)
    pair = (ko.long() << 32) | (vo.long() & 0xFFFFFFFF)
    ref = (rk.long() << 32) | (vals[order].long() & 0xFFFFFFFF)
    assert torch.equal(pair.sort().values, ref.sort().values)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", SIZES)
def test_stable_sort_ranges(crys, n, kind):
    keys = _keys(kind, n)
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    ko, vo = crys.sort(keys, vals)
    rk, order = torch.sort(keys, stable=True)
    assert torch.equal(ko, rk) and torch.equal(vo, order.to(torch.int32))


def test_msb_sort_unaligned_columns(crys):
    # the MSB sort takes columns at any element: every offset of a 16-byte group
    for off in range(4):
        for n in (1, 2, 3, 5, 4990, 100_003):
            base = _keys("bits", n + 8)
            vals = torch.arange(n + 8, dtype=torch.int32, device="cuda")
            k, v = base[off:off + n], vals[3 - off:3 - off + n]
            ko, vo = crys.sort_msb(k, v)
            rk, order = torch.sort(k, stable=True)
            assert torch.equal(ko, rk) and torch.equal(k[(vo - (3 - off)).long()], rk)


# keys that differ in few bytes (the stable sort goes by digits), and the same with rare keys
# outside the sample that differ in the others
@pytest.mark.parametrize("rare", [False, True])
@pytest.mark.parametrize("mask", [0x000000FF, 0x00FF00FF, 0x7FFF00FF, -0x10000, -0xFF0001, 0x00FFFFFF])
@pytest.mark.parametrize("n", [(1 << 20) + 1, 3_000_017])
def test_sorts_of_keys_with_few_bytes(crys, n, mask, rare):
    keys = _keys("bits", n) & mask
    if rare:
        keys[n // 7 + 5] = -2
        keys[n // 5 + 77] = I32_MAX - 255
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    rk, order = torch.sort(keys, stable=True)
    ko, vo = crys.sort(keys, vals)
    assert torch.equal(ko, rk) and torch.equal(vo, order.to(torch.int32))
    ko, vo = crys.sort_msb(keys, vals)
    assert torch.equal(ko, rk) and torch.equal(keys[vo.long()], rk)
    assert torch.equal(vo.sort().values, vals)

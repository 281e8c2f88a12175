"""MSB sorts whose buckets hold somewhat more rows than a block (4992 rows): divided in two by a cut
of the bucket's key range where one fits, through global memory otherwise."""
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


def _buckets(sizes, kind, seed):
    """Keys of 1024 buckets of 2^22 values each, sizes[i] rows in bucket i (range ends included)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    width = 1 << 22
    bucket = torch.repeat_interleave(torch.arange(1024, device="cuda"), torch.tensor(sizes, device="cuda"))
    n = bucket.numel()
    if kind == "even":
        off = torch.randint(0, width, (n,), device="cuda", generator=g)
    elif kind == "ends":                     # the two ends of a bucket and little between
        off = torch.randint(0, 2, (n,), device="cuda", generator=g) * (width - 3) + torch.randint(0, 3, (n,), device="cuda", generator=g)
    elif kind == "lopsided":                 # most rows near the lower end: no cut fits for some
        off = (torch.rand(n, dtype=torch.float64, device="cuda", generator=g) ** 12 * width).long()
    else:                                    # one value each
        off = torch.full((n,), 77, device="cuda")
    k = (bucket * width + off - (1 << 31)).to(torch.int32)
    k[0], k[n - 1] = I32_MIN, I32_MAX
    return k[torch.randperm(n, device="cuda", generator=g)]


@pytest.mark.parametrize("off", [0, 1, 3])
@pytest.mark.parametrize("kind", ["even", "ends", "lopsided", "one value"])
@pytest.mark.parametrize("rows", [4991, 4992, 4993, 5200, 9983, 9984, 9985, 12_000])
def test_large_buckets(crys, rows, kind, off):
    # every eighth bucket of the given size among small ones
    keys = _buckets([rows if i % 8 == 3 else 2300 for i in range(1024)], kind, rows)
    n = keys.numel()
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    ko, vo = (torch.empty(n + 4, dtype=torch.int32, device="cuda")[off:off + n] for _ in range(2))
    tb = crys.crys_sort_msb(None, None, None, None, n, None, -1)
    temp = crys.scratch(tb, "cuda")
    crys.crys_sort_msb(keys, vals, ko, vo, n, temp, tb)
    rk = torch.sort(keys).values
    assert torch.equal(ko, rk) and torch.equal(keys[vo.long()], rk) and torch.equal(vo.sort().values, vals)


def test_more_rows_than_the_blocks_hold(crys):
    # 330M rows over all 32 bits: buckets of 5035 rows on average
    n = 330_000_000
    keys = torch.randint(I32_MIN, I32_MAX, (n,), dtype=torch.int32, device="cuda")
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    ko, vo = crys.sort_msb(keys, vals)
    assert bool((ko[1:] >= ko[:-1]).all()) and torch.equal(keys[vo.long()], ko)
    seen = torch.zeros(n, dtype=torch.bool, device="cuda")
    seen[vo.long()] = True
    assert bool(seen.all())

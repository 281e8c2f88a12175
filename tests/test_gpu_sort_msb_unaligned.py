"""The MSB sort into columns that start at any element: its one partition pass (up to 2^20 rows;
aligned outputs take one launch instead) and its two passes, over key sets for small and
large buckets, against torch's stable sort."""
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
    g.manual_seed(n * 3 + len(kind))
    if kind == "bits":
        return torch.randint(I32_MIN, I32_MAX, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
    if kind == "repeats":
        return torch.randint(0, max(1, n // 64), (n,), dtype=torch.int32, device="cuda", generator=g) * 1021
    k = torch.randint(0, 40, (n,), dtype=torch.int32, device="cuda", generator=g)
    k[n // 2] = I32_MAX                        # few values beside a far one: buckets beyond a block
    return k


@pytest.mark.parametrize("off_k,off_v", [(0, 1), (1, 0), (1, 3), (2, 2), (3, 1)])
@pytest.mark.parametrize("kind", ["bits", "repeats", "few"])
@pytest.mark.parametrize("n", [4993, 70_001, 262_145, (1 << 20) - 3, 1 << 20, (1 << 20) + 1, 2_500_013])
def test_unaligned_outputs(crys, n, kind, off_k, off_v):
    keys = _keys(kind, n)
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    pad = 777
    bk = torch.full((n + 8,), pad, dtype=torch.int32, device="cuda")
    bv = torch.full((n + 8,), pad, dtype=torch.int32, device="cuda")
    ko, vo = bk[off_k:off_k + n], bv[off_v:off_v + n]
    tb = crys.crys_sort_msb(None, None, None, None, n, None, -1)
    temp = crys.scratch(tb, "cuda")
    crys.crys_sort_msb(keys, vals, ko, vo, n, temp, tb)
    rk = torch.sort(keys).values
    assert torch.equal(ko, rk) and torch.equal(keys[vo.long()], rk) and torch.equal(vo.sort().values, vals)
    for b, off in ((bk, off_k), (bv, off_v)):          # nothing outside the columns is written
        assert bool((b[:off] == pad).all()) and bool((b[off + n:] == pad).all())

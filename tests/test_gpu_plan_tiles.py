"""The fused date-join query with the default tile shape, at the row counts around the line
below which it takes smaller tiles, and at the edges of both tiles; against torch."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

I32_MIN = -(1 << 31)
LINE = 3 << 23


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


@pytest.mark.parametrize("kind", ["direct", "hashed"])
@pytest.mark.parametrize("n", [1, 2047, 2049, 4097, LINE - 1, LINE, LINE + 1])
def test_default_tiles(crys, n, kind):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)

    def uni(lo, hi, rows=n):
        return torch.randint(lo, hi + 1, (rows,), dtype=torch.int32, device="cuda", generator=g)
    fact = [uni(0, 2555), uni(1, 50), uni(0, 10), uni(1, 100_000)]
    key = torch.randperm(2556, device="cuda", generator=g).to(torch.int32)
    year = uni(0, 6, 2556)
    ht = crys.HashTable.build(key, year, filters=[(year, 3, 3)], capacity=2556 if kind == "direct" else 8192,
                              **({"kind": crys.HASH_DIRECT} if kind == "direct" else {}))
    by_key = torch.zeros(2556, dtype=torch.int32, device="cuda")
    by_key[key.long()] = year
    total, count = (torch.full((1,), -1, dtype=torch.int64, device="cuda") for _ in range(2))
    plan = crys.make_plan([(1, I32_MIN, 24), (2, 1, 3)], [(0, ht, 0)], ("mul", 3, 2), total, count)
    crys.crys_set_tile(crys.OP_PLAN, 0)
    crys.crys_run_plan(crys.make_table(fact), plan)
    hit = (fact[1] <= 24) & (fact[2] >= 1) & (fact[2] <= 3) & (by_key[fact[0].long()] == 3)
    assert int(total) == int((fact[3][hit].long() * fact[2][hit].long()).sum())
    assert int(count) == int(hit.sum())

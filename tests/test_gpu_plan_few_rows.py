"""Queries over tables of few rows, at the edges of the library's own choice of tiles: up to 2048
rows per SM in tiles of 2048 rows, up to 4096 in tiles of 4096, up to 6144 in the smaller
ones again; one to three joins on direct and hashed tables, grouped."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

I32_MIN = -(1 << 31)


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


@pytest.mark.parametrize("direct", [True, False])
@pytest.mark.parametrize("joins", [1, 2, 3])
@pytest.mark.parametrize("rows", [1, 2049, "line-1", "line", "line+1", "line+4097", "2line", "2line+1", "3line", "3line+1"])
def test_plans_of_few_rows(crys, rows, joins, direct):
    line = torch.cuda.get_device_properties(0).multi_processor_count * 2048
    if isinstance(rows, int):
        n = rows
    else:
        times, _, more = rows.partition("line")
        n = int(times or 1) * line + int(more or 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(n + joins)

    def col(lo, hi, k=n):
        return torch.randint(lo, hi + 1, (k,), dtype=torch.int32, device="cuda", generator=g)
    sizes, cards = [2556, 1000, 30_000][:joins], [7, 5, 4][:joins]
    fact = [col(0, s - 1 + s // 4) for s in sizes] + [col(1, 50), col(1, 1000)]
    tables, codes = [], []
    for s, card in zip(sizes, cards):
        key, code = torch.randperm(s, device="cuda", generator=g).to(torch.int32), col(0, card - 1, s)
        by = torch.full((s + s // 4 + 1,), -1, dtype=torch.int64, device="cuda")
        by[key.long()] = code.long()
        codes.append(by)
        tables.append(crys.HashTable.build(key, code, capacity=s, kind=crys.HASH_DIRECT) if direct
                      else crys.HashTable.build(key, code))
    sums, counts = crys.run_plan(fact, [(joins, I32_MIN, 24)], [(j, tables[j], cards[j]) for j in range(joins)],
                                 ("mul", joins, joins + 1))
    live, gid = fact[joins] <= 24, torch.zeros(n, dtype=torch.int64, device="cuda")
    for j in range(joins):
        c = codes[j][fact[j].long()]
        live, gid = live & (c >= 0), gid * cards[j] + c
    val = fact[joins].long() * fact[joins + 1].long()
    groups = int(np.prod(cards))
    want = torch.zeros(groups, dtype=torch.int64, device="cuda").index_add_(0, gid[live], val[live])
    assert torch.equal(sums, want) and torch.equal(counts, torch.bincount(gid[live], minlength=groups))

"""A tile shape that was set is used for every size, and without one the library's own choices
give the same results: sorts of few rows (one launch, or the passes of the shape), ordered
selections of few rows (no scratch, or the tiles' status words), probes and queries around the
sizes where the own choice changes."""
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


def _uni(seed, n, lo, hi):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randint(lo, hi + 1, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)


@pytest.mark.parametrize("variant", [None, 0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 3, 100, 4095, 4992, 4993, 100_003, 1 << 20])
def test_sorts_of_few_rows(crys, n, variant):
    keys, vals = _uni(n, n, I32_MIN, I32_MAX), torch.arange(n, dtype=torch.int32, device="cuda")
    if variant is not None:
        crys.crys_set_tile(crys.OP_SORT, variant)
    for k in (keys, keys & 7):
        before = crys.crys_launch_count()
        ko, vo = crys.sort(k, vals)
        launches = crys.crys_launch_count() - before
        assert launches == 1 if variant is None else launches >= 5
        rk, order = torch.sort(k, stable=True)
        assert torch.equal(ko, rk) and torch.equal(vo, order.to(torch.int32))


@pytest.mark.parametrize("variant", [None, 0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 511, 513, 65_536, 100_003, 131_072])
def test_selections_of_few_rows(crys, n, variant):
    x = _uni(n, n, 0, 999)
    if variant is not None:
        crys.crys_set_tile(crys.OP_SELECT, variant)
    tb = crys.crys_select(None, n, 0, 0, None, None, 1, None, -1)
    temp = torch.full((tb,), 0xA5, dtype=torch.uint8, device="cuda")
    out, count = torch.empty_like(x), torch.zeros(1, dtype=torch.int64, device="cuda")
    crys.crys_select(x, n, 200, 700, out, count, 1, temp, tb)
    ref = x[(x >= 200) & (x <= 700)]
    assert int(count) == ref.numel() and torch.equal(out[:ref.numel()], ref)
    assert bool((temp == 0xA5).all()) == (variant is None)          # the tiles' words were used
    got = crys.select(x, 200, 700, order_preserving=False)
    assert torch.equal(got.sort().values, ref.sort().values)


@pytest.mark.parametrize("variant", [None, 0, 1])
@pytest.mark.parametrize("nb", [2048, 4096, 8192, 32_768, 65_536])
@pytest.mark.parametrize("n", [(1 << 25) - 1, 1 << 25])
def test_probes(crys, n, nb, variant):
    if variant is not None:
        crys.crys_set_tile(crys.OP_PROBE, variant)
    bv, fk, pay = _uni(1, nb, 1, 100), _uni(2, n, 0, nb + nb // 3), _uni(3, n, 1, 100)
    bk = torch.randperm(nb, device="cuda").to(torch.int32)
    total, matches = crys.probe_aggregate(fk, pay, crys.HashTable.build(bk, bv))
    value = torch.zeros(2 * nb, dtype=torch.int64, device="cuda")
    value[bk.long()] = bv.long()
    assert int(matches) == int((fk < nb).sum()) and int(total) == int((value[fk.long()] * pay).sum())


@pytest.mark.parametrize("variant", [None, 0, 1])
@pytest.mark.parametrize("n", [2049, 300_000, 400_000, (3 << 23) - 1, 3 << 23, (3 << 23) + 1])
def test_date_join_queries(crys, n, variant):
    if variant is not None:
        crys.crys_set_tile(crys.OP_PLAN, variant)
    fact = [_uni(1, n, 0, 2555), _uni(2, n, 1, 50), _uni(3, n, 0, 10), _uni(4, n, 1, 100_000)]
    key, year = torch.randperm(2556, device="cuda").to(torch.int32), _uni(5, 2556, 0, 6)
    ht = crys.HashTable.build(key, year, filters=[(year, 3, 3)], capacity=2556, kind=crys.HASH_DIRECT)
    sums, counts = crys.run_plan(fact, [(1, I32_MIN, 24), (2, 1, 3)], [(0, ht, 0)], ("mul", 3, 2))
    by_key = torch.zeros(2556, dtype=torch.int32, device="cuda")
    by_key[key.long()] = year
    hit = (fact[1] <= 24) & (fact[2] >= 1) & (fact[2] <= 3) & (by_key[fact[0].long()] == 3)
    assert int(sums) == int((fact[3][hit].long() * fact[2][hit].long()).sum()) and int(counts) == int(hit.sum())

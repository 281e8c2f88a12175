"""Stable sorts in turn on one scratch buffer that held other bytes before: the tiles of a pass
leave their status words clear for the next pass, so sorts of two, three and four passes, by
buckets and by digits, follow one another; and the same from a captured graph."""
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
    crys.crys_set_tile(crys.OP_SORT, 0)


def _keys(kind, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(n + len(kind))
    k = torch.randint(I32_MIN, I32_MAX, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
    if kind == "one byte":
        k = k & 0xFF00
    elif kind == "three bytes":
        k = k & 0xFFFFFF
    elif kind == "repeats":                      # about 40 rows per value: four digits
        k = k[torch.randint(0, n // 40, (n,), device="cuda", generator=g)]
    elif kind == "heavy":                        # found by the counts, not by the sample
        k[: n // 100] = 12_345
    return k


KINDS = ["bits", "three bytes", "repeats", "bits", "one byte", "heavy", "bits"]


@pytest.mark.parametrize("variant", range(4))
@pytest.mark.parametrize("n", [(1 << 20) + 1, 2_097_153, 5_000_011])
def test_one_scratch(crys, n, variant):
    crys.crys_set_tile(crys.OP_SORT, variant)
    tb = crys.crys_sort(None, None, None, None, n, None, -1)
    temp = crys.scratch(tb, "cuda")
    temp.fill_(0xA5)
    keys, vals = torch.empty(n, dtype=torch.int32, device="cuda"), torch.arange(n, dtype=torch.int32, device="cuda")
    ko, vo = torch.empty_like(keys), torch.empty_like(vals)
    for kind in KINDS:
        keys.copy_(_keys(kind, n))
        crys.crys_sort(keys, vals, ko, vo, n, temp, tb)
        rk, order = torch.sort(keys, stable=True)
        assert torch.equal(ko, rk) and torch.equal(vo, order.to(torch.int32)), kind
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        crys.crys_sort(keys, vals, ko, vo, n, temp, tb)
    for kind in KINDS:
        keys.copy_(_keys(kind, n))
        graph.replay()
        rk, order = torch.sort(keys, stable=True)
        assert torch.equal(ko, rk) and torch.equal(vo, order.to(torch.int32)), kind
    crys.crys_set_tile(crys.OP_SORT, 0)


def test_more_rows_than_the_buckets_take(crys):
    # above 2^28 rows every stable sort goes by digits
    n = (1 << 28) + 77
    keys = torch.randint(I32_MIN, I32_MAX, (n,), dtype=torch.int32, device="cuda")
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    ko, vo = crys.sort(keys, vals)
    assert bool((ko[1:] >= ko[:-1]).all()) and torch.equal(keys[vo.long()], ko)
    equal = ko[1:] == ko[:-1]
    assert bool((vo[1:][equal] > vo[:-1][equal]).all())
    seen = torch.zeros(n, dtype=torch.bool, device="cuda")
    seen[vo.long()] = True
    assert bool(seen.all())

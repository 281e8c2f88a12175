"""Sorts of one launch (4993 to 2^20 rows) at the edges of their blocks' shares, in the general
steps just above, over key sets for each of their ways: buckets, a bucket per value, and digits;
twice on the same scratch, and replayed from a captured graph."""
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
    g.manual_seed(n + len(kind))
    lo, hi = {"bits": (I32_MIN, I32_MAX), "values_256": (-100, 155), "values_257": (-100, 156),
              "crowded": (5, 5 + 300), "two_far": (0, 1)}[kind]
    k = torch.randint(lo, hi + 1, (n,), dtype=torch.int64, device="cuda", generator=g)
    k[0], k[n - 1] = lo, hi                       # the whole range
    if kind == "two_far":
        k = k * (1 << 32) - (1 << 31)
        k[k > I32_MAX] = I32_MAX
    if kind == "crowded":                         # far keys beside many equal ones: four digits
        k[n // 2] = I32_MIN
    return k.to(torch.int32)


SIZES = [4993, 5120, 155_648, 155_649, 758_783, 758_784, 758_785, (1 << 20) - 1, 1 << 20, (1 << 20) + 1]


@pytest.mark.parametrize("kind", ["bits", "values_256", "values_257", "crowded", "two_far"])
@pytest.mark.parametrize("n", SIZES)
def test_small_sorts(crys, n, kind):
    keys = _keys(kind, n)
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    rk, order = torch.sort(keys, stable=True)
    for _ in range(2):
        ko, vo = crys.sort(keys, vals)
        assert torch.equal(ko, rk) and torch.equal(vo, order.to(torch.int32))
    ko, vo = crys.sort_msb(keys, vals)
    assert torch.equal(ko, rk) and torch.equal(keys[vo.long()], rk)
    assert torch.equal(vo.sort().values, vals)


def test_small_sort_from_a_graph(crys):
    n = 100_003
    keys = _keys("bits", n)
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    ko, vo = torch.empty_like(keys), torch.empty_like(vals)
    tb = crys.crys_sort(None, None, None, None, n, None, -1)
    temp = crys.scratch(tb, "cuda")
    crys.crys_sort(keys, vals, ko, vo, n, temp, tb)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        crys.crys_sort(keys, vals, ko, vo, n, temp, tb)
    for seed in range(3):
        keys.copy_(_keys("bits", n).roll(seed * 17))
        graph.replay()
        rk, order = torch.sort(keys, stable=True)
        assert torch.equal(ko, rk) and torch.equal(vo, order.to(torch.int32))

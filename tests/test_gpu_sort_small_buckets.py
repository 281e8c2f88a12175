"""Sorts of one launch whose blocks sort several buckets one after the other through the same
shared memory (more than 2^18 rows: 256 buckets on a block per SM): values that differ in every
row, so that one taken from another bucket's copy shows; buckets of a few rows beside full ones."""
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


@pytest.mark.parametrize("kind", ["even", "steps"])
@pytest.mark.parametrize("n", [(1 << 18) + 1, 300_001, 500_003, 1 << 20])
def test_blocks_with_several_buckets(crys, n, kind):
    for seed in range(10):
        g = torch.Generator(device="cuda")
        g.manual_seed(n + seed)
        if kind == "even":
            keys = torch.randint(I32_MIN, I32_MAX, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
        else:                 # the buckets fill up from the first to the last one
            u = torch.rand(n, dtype=torch.float64, device="cuda", generator=g)
            keys = ((u ** 0.9) * ((1 << 32) - 1) - (1 << 31)).to(torch.int64).to(torch.int32)
        vals = torch.randperm(n, device="cuda", generator=g).to(torch.int32)
        rk, order = torch.sort(keys, stable=True)
        ko, vo = crys.sort(keys, vals)
        assert torch.equal(ko, rk) and torch.equal(vo, vals[order])
        ko, vo = crys.sort_msb(keys, vals)
        assert torch.equal(ko, rk)
        pair = (ko.long() << 32) | vo.long()
        assert torch.equal(pair.sort().values, ((rk.long() << 32) | vals[order].long()).sort().values)

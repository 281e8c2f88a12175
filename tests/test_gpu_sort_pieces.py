"""Sorts of columns made of pieces, each with a key range of its own, in shuffled order: the
smallest and largest keys lie together in a few places.  Against torch's stable sort; the MSB
sort must also not send a piece's rows to one bucket (a block sorts a bucket of a hundred
thousand rows in milliseconds)."""
import statistics

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


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


def _pieces(n, pieces, seed):
    """`pieces` runs of rows, run i random in the p(i)-th of `pieces` equal parts of the int32 range."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    part = torch.randperm(pieces, device="cuda", generator=g)
    width = (1 << 32) // pieces
    row = torch.arange(n, device="cuda")
    piece = torch.clamp(row // (n // pieces), max=pieces - 1)
    k = part[piece] * width - (1 << 31) + torch.randint(0, width, (n,), device="cuda", generator=g)
    return k.to(torch.int32)


@pytest.mark.parametrize("n,pieces", [(5000, 7), (70_001, 64), (1_048_579, 1000), (3_000_017, 1000), (20_000_003, 3000)])
def test_pieces(crys, n, pieces):
    for seed in range(3):
        keys = _pieces(n, pieces, seed)
        vals = torch.arange(n, dtype=torch.int32, device="cuda")
        rk, order = torch.sort(keys, stable=True)
        ko, vo = crys.sort(keys, vals)
        assert torch.equal(ko, rk) and torch.equal(vo, order.to(torch.int32))
        ko, vo = crys.sort_msb(keys, vals)
        assert torch.equal(ko, rk) and torch.equal(keys[vo.long()], rk) and torch.equal(vo.sort().values, vals)


def test_pieces_take_no_longer(crys):
    # 2^26 rows in 1000 pieces against the same keys shuffled: twice the time at most (a
    # missed piece takes more than four times)
    n = 1 << 26
    keys = _pieces(n, 1000, 5)
    times = []
    for k in (keys, keys[torch.randperm(n, device="cuda")]):
        vals = torch.arange(n, dtype=torch.int32, device="cuda")
        ko, vo = torch.empty_like(k), torch.empty_like(vals)
        tb = crys.crys_sort_msb(None, None, None, None, n, None, -1)
        temp = crys.scratch(tb, "cuda")
        ms = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            crys.crys_sort_msb(k, vals, ko, vo, n, temp, tb)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        times.append(statistics.median(ms))
    assert times[0] < 2.0 * times[1], times

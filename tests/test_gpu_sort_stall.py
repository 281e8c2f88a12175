"""A requested stall reaches sorts of every size: the first pass's wait runs out, the flag says so
and the next sort is exact; a request at tile 0 stalls nothing."""
import time

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
    crys.crys_device_errors(clear=True)


@pytest.mark.parametrize("n", [4200, 4992, 4993, 100_003])
def test_stalled_sorts(crys, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    keys = torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    rk, order = torch.sort(keys, stable=True)
    crys.crys_device_errors(clear=True)
    crys.crys_debug_stall(crys.OP_SORT, 1, 2_000_000)
    t0 = time.perf_counter()
    crys.sort(keys, vals)
    torch.cuda.synchronize()
    assert time.perf_counter() - t0 < 1.5
    assert crys.crys_device_errors(clear=True) == crys.DEV_TIMEOUT
    for first in (None, 0):
        if first is not None:
            crys.crys_debug_stall(crys.OP_SORT, first, 2_000_000_000)
        ko, vo = crys.sort(keys, vals)
        assert torch.equal(ko, rk) and torch.equal(vo, order.to(torch.int32))
    assert crys.crys_device_errors(clear=True) == 0

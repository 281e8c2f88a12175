"""Ordered selections and stable sorts that start while other work leaves room for a few of their
blocks only: those are the scanners, which wait for blocks that cannot start yet.  The bound of
their wait counts from when a tile has been handed to a block, so the call ends exact however
long the other work takes.

The other work is a sort whose first pass is stalled for a second on all but a few of the places
that the SMs have for such blocks; it gives up by its own bound."""
import time

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

I32_MAX = (1 << 31) - 1
HOLD, BOUND = 1_000_000_000, 100_000_000        # ns: the other work's stall, the call's own bound


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


def _bits(n, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)


@pytest.mark.parametrize("left", [1, 2, 4, 30])
@pytest.mark.parametrize("op", ["select", "sort"])
def test_beside_other_work(crys, op, left):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = 8192                                   # of a tile of the sort's default shape, three per SM
    tiles = 3 * sms - 8 - left + 1                # 8 scanners and all tiles but the stalled one hold a place
    held_n, n = tiles * rows, 4_000_003 if op == "select" else 4992
    held = [_bits(held_n, 1), torch.arange(held_n, dtype=torch.int32, device="cuda")]
    held += [torch.empty_like(t) for t in held]
    held_bytes = crys.crys_sort(None, None, None, None, held_n, None, -1)
    held_temp = crys.scratch(held_bytes, "cuda")
    x, vals = _bits(n, 2), torch.arange(n, dtype=torch.int32, device="cuda")
    out, vout, count = torch.empty_like(x), torch.empty_like(x), torch.zeros(1, dtype=torch.int64, device="cuda")
    if op == "select":
        tb = crys.crys_select(None, n, 0, 0, None, None, 1, None, -1)
    else:
        tb = crys.crys_sort(None, None, None, None, n, None, -1)
    temp = crys.scratch(tb, "cuda")

    def call(stream):
        if op == "select":
            crys.crys_select(x, n, 0, I32_MAX, out, count, 1, temp, tb, stream=stream)
        else:
            crys.crys_set_tile(crys.OP_SORT, 3)   # passes of 4096-row tiles, not one launch
            crys.crys_sort(x, vals, out, vout, n, temp, tb, stream=stream)
            crys.crys_reset_tile(crys.OP_SORT)
    crys.crys_sort(*held, held_n, held_temp, held_bytes)
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    call(second)
    torch.cuda.synchronize()
    out.zero_()
    vout.zero_()
    count.zero_()
    torch.cuda.synchronize()
    crys.crys_device_errors(clear=True)
    t0 = time.perf_counter()
    crys.crys_debug_stall(crys.OP_SORT, 1, HOLD)
    crys.crys_sort(*held, held_n, held_temp, held_bytes, stream=first)
    time.sleep(0.05)                              # its first pass holds its places by now
    crys.crys_debug_stall(crys.OP_SELECT if op == "select" else crys.OP_SORT, 0, BOUND)
    call(second)
    second.synchronize()
    elapsed = time.perf_counter() - t0
    torch.cuda.synchronize()
    assert crys.crys_device_errors(clear=True) == crys.DEV_TIMEOUT     # the stalled sort's
    if op == "select":
        ref = x[x >= 0]
        assert int(count) == ref.numel() and torch.equal(out[:ref.numel()], ref), elapsed
    else:
        rk, order = torch.sort(x, stable=True)
        assert torch.equal(out, rk) and torch.equal(vout, order.to(torch.int32)), elapsed

"""Selections of one cluster of blocks beside other work: on a stream of their own while another
stream keeps the SMs busy, so that the cluster's blocks start when room comes free.  Every
position and the count follow from counts that the blocks write to one another."""
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


@pytest.mark.parametrize("n", [7, 1000, 32_769, 65_536, 100_003, 131_072])
def test_small_selects_beside_other_work(crys, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    cols = [torch.randint(0, I32_MAX, (n,), dtype=torch.int32, device="cuda", generator=g) for _ in range(8)]
    his = [I32_MAX // 8 * (i + 1) for i in range(8)]
    refs = [x[x <= hi] for x, hi in zip(cols, his)]
    outs = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(40)]
    counts = torch.full((40,), -1, dtype=torch.int64, device="cuda")
    tb = crys.crys_select(None, n, 0, 0, None, None, 1, None, -1)
    temp = crys.scratch(tb, "cuda")
    busy = torch.rand(4096, 4096, device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    for _ in range(12):
        busy @ busy
    for i in range(40):
        crys.crys_select(cols[i % 8], n, I32_MIN, his[i % 8], outs[i], counts[i:i + 1], 1, temp, tb, stream=side)
    torch.cuda.synchronize()
    for i, (out, c) in enumerate(zip(outs, counts.tolist())):
        assert c == refs[i % 8].numel() and torch.equal(out[:c], refs[i % 8]), i


@pytest.mark.parametrize("off", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [3, 4, 5, 4099, 65_536, 131_072])
def test_small_selects_of_most_rows(crys, n, off):
    # everything selected, and all but rows at every place of a group of four; outputs that start
    # at any element
    x = torch.arange(n, dtype=torch.int32, device="cuda")
    for gap in (0, 5, 64, 1021):
        if gap:
            x[::gap] = -1
        ref = x[x >= 0]
        buf = torch.full((n + 8,), 777, dtype=torch.int32, device="cuda")
        count = torch.zeros(1, dtype=torch.int64, device="cuda")
        tb = crys.crys_select(None, n, 0, I32_MAX, None, None, 1, None, -1)
        temp = crys.scratch(tb, "cuda")
        crys.crys_select(x, n, 0, I32_MAX, buf[off:off + n], count, 1, temp, tb)
        c = int(count.item())
        assert c == ref.numel() and torch.equal(buf[off:off + c], ref)
        assert bool((buf[:off] == 777).all()) and bool((buf[off + c:] == 777).all())
        x = torch.arange(n, dtype=torch.int32, device="cuda")

"""The partitioned join around the line between its 4096-slot and 8192-slot tables (2304 rows of
a partition), with hits, misses and keys whose hashes lie next to one another."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MULT = 2654435769


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


@pytest.mark.parametrize("rows", [2303, 2304, 2305])
@pytest.mark.parametrize("spread", ["random", "adjacent"])
@pytest.mark.parametrize("others", [0, 200_000])
def test_partition_at_the_line(crys, orc, rows, spread, others):
    rng = np.random.default_rng(rows)
    inv = pow(MULT, -1, 1 << 32)
    low = rng.choice(1 << 16, size=rows, replace=False) if spread == "random" else np.arange(65_536 - rows, 65_536)
    h = (np.uint64(0xA5A5) << np.uint64(16)) | low.astype(np.uint64)     # one partition at any depth
    if others:
        o = np.unique(rng.integers(0, 1 << 32, size=others, dtype=np.uint64))
        h = np.concatenate([h, o[(o >> np.uint64(16)) != 0xA5A5]])
    bk = rng.permutation(((h * np.uint64(inv)) & np.uint64(0xFFFFFFFF)).astype(np.uint32).view(np.int32))
    bv = rng.integers(-100, 101, size=bk.size).astype(np.int32)
    n = 50_003
    fk = np.where(rng.random(n) < 0.6, bk[rng.integers(0, bk.size, size=n)],
                  rng.integers(-(1 << 31), 1 << 31, size=n).astype(np.int32)).astype(np.int32)
    pay = rng.integers(-(1 << 31), 1 << 31, size=n).astype(np.int32)
    s, m = crys.join_partitioned(*(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (bk, bv, fk, pay)))
    assert (int(s.item()), int(m.item())) == orc.join_sum(bk, bv, fk, pay)

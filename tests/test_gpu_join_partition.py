"""The partitioned join at the edges of its tables: build partitions just below and above the
4096-slot (3072 rows) and 8192-slot (6144 rows) shared-memory tables and the scratch table,
at every partitioning depth, probe tiles of one row and ragged ones, misses, the one key
whose hash is the empty marker, and repeated build keys."""
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


def _keys_of_hash(h):
    """Keys whose multiplicative hash is h (the hash is one-to-one on 32 bits)."""
    inv = pow(MULT, -1, 1 << 32)
    return ((h.astype(np.uint64) * np.uint64(inv)) & np.uint64(0xFFFFFFFF)).astype(np.uint32).view(np.int32)


def _check(crys, orc, bk, bv, fk, pay):
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (bk, bv, fk, pay)]
    s, m = crys.join_partitioned(*dev)
    assert (int(s.item()), int(m.item())) == orc.join_sum(bk, bv, fk, pay)


@pytest.mark.parametrize("rows", [1, 3071, 3072, 3073, 6143, 6144, 6145, 9000])
@pytest.mark.parametrize("others", [0, 100_000])
def test_partition_of_given_size(crys, orc, rows, others):
    # one partition of exactly `rows` build rows (hashes with the same top 16 bits cover any
    # depth), the other build keys spread over the rest
    rng = np.random.default_rng(rows + others)
    low = rng.choice(1 << 16, size=rows, replace=False)
    bk = _keys_of_hash((np.uint64(0x5A5A) << np.uint64(16)) | low.astype(np.uint64))
    if others:
        h = np.unique(rng.integers(0, 1 << 32, size=others, dtype=np.uint64))
        bk = np.concatenate([bk, _keys_of_hash(h[(h >> np.uint64(16)) != 0x5A5A])])
    bk = rng.permutation(bk)
    bv = rng.integers(-100, 101, size=bk.size).astype(np.int32)
    for n in (1, 5119, 5121, 70_001):
        fk = np.where(rng.random(n) < 0.7, bk[rng.integers(0, bk.size, size=n)],
                      rng.integers(-(1 << 31), 1 << 31, size=n).astype(np.int32)).astype(np.int32)
        pay = rng.integers(-(1 << 31), 1 << 31, size=n).astype(np.int32)
        _check(crys, orc, bk, bv, fk, pay)


@pytest.mark.parametrize("nb", [1, 2048, 2049, 100_000])
def test_key_whose_hash_is_the_empty_marker(crys, orc, nb):
    odd = _keys_of_hash(np.array([0xFFFFFFFF], dtype=np.uint64))[0]
    for there in (True, False):
        bk = np.arange(nb, dtype=np.int32)
        if there:
            bk[nb // 2] = odd
        bv = np.arange(1, nb + 1, dtype=np.int32)
        fk = np.concatenate([np.full(1000, odd, np.int32), np.arange(5000, dtype=np.int32)])
        pay = np.arange(fk.size, dtype=np.int32)
        _check(crys, orc, bk, bv, fk, pay)


@pytest.mark.parametrize("nb", [100, 5000, 200_000])
def test_repeated_build_key_is_flagged(crys, nb):
    bk = torch.arange(nb, dtype=torch.int32, device="cuda")
    bk[nb - 1] = 3
    fk = torch.arange(1000, dtype=torch.int32, device="cuda")
    crys.join_partitioned(bk, bk, fk, fk)
    assert crys.crys_device_errors(clear=True) == crys.DEV_DUP_KEY

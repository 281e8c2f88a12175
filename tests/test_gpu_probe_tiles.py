"""Probes with the default tile shape around the lines at which it takes larger tiles: tables
of 32 KB to 1 MB, 2^25 probes and one less; against torch."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nb", [2048, 2049, 32_768, 32_769])
@pytest.mark.parametrize("n", [4097, (1 << 25) - 1, 1 << 25])
def test_default_probe_tiles(n, nb):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2003_01178_gb300 import _build
    _build.build()
    import paper_2003_01178_gb300 as crys
    g = torch.Generator(device="cuda")
    g.manual_seed(n + nb)

    def uni(lo, hi, rows):
        return torch.randint(lo, hi + 1, (rows,), dtype=torch.int32, device="cuda", generator=g)
    key, val, fk, pay = torch.randperm(nb, device="cuda", generator=g).to(torch.int32), uni(1, 100, nb), uni(0, 2 * nb, n), uni(1, 100, n)
    crys.crys_set_tile(crys.OP_PROBE, 0)
    total, matches = crys.probe_aggregate(fk, pay, crys.HashTable.build(key, val))
    by_key = torch.zeros(2 * nb + 1, dtype=torch.int64, device="cuda")
    by_key[key.long()] = val.long()
    assert int(total) == int((by_key[fk.long()] * pay.long()).sum())
    assert int(matches) == int((fk < nb).sum())

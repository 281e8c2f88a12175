"""The tile shape that was set and the library's own choice (host state, no GPU needed)."""
import json

import pytest


@pytest.fixture(scope="module")
def crys():
    from paper_2003_01178_gb300 import _build
    _build.build()
    import paper_2003_01178_gb300 as crys
    yield crys
    for op in range(crys.NUM_OPS):
        crys.crys_reset_tile(op)


def test_set_and_reset(crys):
    for op in range(crys.NUM_OPS):
        crys.crys_reset_tile(op)
        assert not crys.crys_tile_is_set(op) and crys.crys_get_tile(op) == 0
        for v in (0, 3):
            crys.crys_set_tile(op, v)
            assert crys.crys_tile_is_set(op) and crys.crys_get_tile(op) == v
        for bad in (-1, 4, 99):
            assert crys.lib().crys_set_tile(op, bad) == crys.EINVAL
            assert crys.crys_get_tile(op) == 3
        crys.crys_reset_tile(op)
        assert not crys.crys_tile_is_set(op)
    for bad in (-1, crys.NUM_OPS):
        assert crys.lib().crys_reset_tile(bad) == crys.EINVAL and crys.lib().crys_tile_is_set(bad) == crys.EINVAL
        with pytest.raises(crys.CrystalError):
            crys.crys_tile_is_set(bad)


def test_tuner_keeps_what_was_set(crys, tmp_path, monkeypatch):
    from paper_2003_01178_gb300 import tuner
    monkeypatch.setattr(tuner, "_key", lambda: "test-device")
    path = str(tmp_path / "tiles.json")
    crys.crys_set_tile(crys.OP_PLAN, 0)
    tuner.save(path)
    assert json.load(open(path)) == {"test-device": {crys.OP_NAMES[crys.OP_PLAN]: list(crys.crys_tile_variants(crys.OP_PLAN)[0])}}
    crys.crys_reset_tile(crys.OP_PLAN)
    assert tuner.load(path)
    assert [op for op in range(crys.NUM_OPS) if crys.crys_tile_is_set(op)] == [crys.OP_PLAN]
    assert crys.crys_get_tile(crys.OP_PLAN) == 0


@pytest.mark.parametrize("own,variants,chosen", [(1.0, [1.0, 1.2, 0.99, 1.5], None), (1.0, [1.0, 0.9, 1.2, 1.5], 1),
                                                  (0.5, [1.0, 0.9, 1.2, 1.5], None)])
def test_tuner_prefers_the_own_choice(crys, monkeypatch, own, variants, chosen):
    from paper_2003_01178_gb300 import tuner
    op = crys.OP_SELECT

    def timed(launch, reps=5, warmup=2, stream=None):
        return variants[crys.crys_get_tile(op)] if crys.crys_tile_is_set(op) else own
    monkeypatch.setattr(tuner, "time_variant", timed)
    res = tuner.tune(op, lambda: None)
    assert res["best"] == variants.index(min(variants)) and res["set"] == (chosen is not None)
    assert crys.crys_tile_is_set(op) == (chosen is not None)
    if chosen is not None:
        assert crys.crys_get_tile(op) == chosen

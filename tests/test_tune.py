"""What the tuner times, on the CPU: the timings are a table here."""
import pytest

from paper_1008_2602_gb300 import tune
from paper_1008_2602_gb300 import workloads as W


@pytest.fixture()
def timed(tmp_path, monkeypatch):
    calls = []

    def batch(probs, precision, cfg, steps):
        calls.append(cfg)
        return 1.0 if (cfg["tile_x"], cfg["tile_y"], cfg["zseg"]) == (124, 4, tune.ZSEG_AUTO) else 2.0

    def single(prob, precision, cfg, steps):
        calls.append(cfg)
        return 1.0 if cfg.get("depth") == 1 else 3.0

    monkeypatch.setattr(tune, "CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(tune, "_time_batch", batch)
    monkeypatch.setattr(tune, "_time_single", single)
    return calls


def test_resident_boards_keep_the_tiled_defaults(timed, monkeypatch):
    monkeypatch.setattr(tune, "_resident", lambda probs, precision: True)
    p = W.box(20, 20, 20)
    assert tune.tune([p, p], steps=4) == dict(tune.DEFAULT, depth=1) and not timed
    assert tune.tune([p], steps=4) == dict(tune.DEFAULT, depth=1)
    assert [c["depth"] for c in timed] == [1, 2, 2]   # one board: the depths alone
    monkeypatch.setattr(tune, "_resident", lambda probs, precision: False)
    del timed[:]
    tune.tune([p, p], steps=4)   # tiled boards of the class do not take that entry
    assert timed


def test_the_library_s_own_segments_are_among_the_candidates(timed, monkeypatch):
    monkeypatch.setattr(tune, "_resident", lambda probs, precision: False)
    cfg = tune.tune([W.box(20, 20, 20)] * 2, steps=4)
    assert (cfg["tile_x"], cfg["tile_y"], cfg["zseg"]) == (124, 4, tune.ZSEG_AUTO)
    from paper_1008_2602_gb300 import capi
    assert tune.ZSEG_AUTO == capi.FDTD_ZSEG_AUTO
    n = len(timed)
    assert tune.tune([W.box(20, 20, 20)] * 2, steps=4) == cfg and len(timed) == n   # cached

"""The tuner's candidates: the library's own defaults and the shipped entry are
measured, relabel caps up to the rule's are searched, and measurements of
another solver do not override the shipped table.  The timer is replaced by a
host-side cost model."""
import json

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture()
def tune(monkeypatch, tmp_path):
    from paper_1803_01516_gb300 import build
    build.build()
    from paper_1803_01516_gb300 import autotune
    monkeypatch.setenv("GAZECUT_TUNE_CACHE", str(tmp_path / "cache.json"))
    return autotune


def _pairs(p):
    return [(torch.zeros(p.h, p.w, dtype=torch.uint8),) * 2]


@pytest.mark.parametrize("w,h,D", [(271, 144, 62), (400, 300, 16), (400, 300, 19), (100, 40, 8)])
def test_result_is_no_slower_than_the_defaults(tune, monkeypatch, w, h, D):
    from paper_1803_01516_gb300 import gazecut as gc
    p = gc.Params(w=w, h=h, D=D, tau=30, lam=10)
    s = tune.tuned_opts(p)
    shipped = (s.sweeps_per_relabel, s.local_iters, s.relabel_passes, s.tile_w, s.tile_h,
               s.tail_iters, s.cta_threads)
    for fastest in ((16, 8, 0, 0, 0, 0, 512), shipped):
        monkeypatch.setattr(tune, "_time_config",
                            lambda pp, pairs, cfg, reps=2: 1.0 if tuple(cfg) == fastest else 2.0)
        assert tuple(tune.tune(p, pairs=_pairs(p), save=False)["best"]) == fastest


def test_caps_follow_the_tile(tune, monkeypatch):
    """8x4-site tiles that need 32 relabel passes: 37.6 ms under a cap of 8,
    27.5 under 32 or the rule; 16x4 tiles 30 under any."""
    from paper_1803_01516_gb300 import gazecut as gc

    def ms(pp, pairs, cfg, reps=2):
        rp, shape = cfg[2], tuple(cfg[3:5])
        if shape == (8, 4):
            return 27.5 if rp in (0, 32) else 37.6
        return 30.0 if shape == (16, 4) else 50.0

    monkeypatch.setattr(tune, "_time_config", ms)
    p = gc.Params(w=271, h=144, D=62, tau=30, lam=10)
    e = tune.tune(p, pairs=_pairs(p), save=False)
    assert e["ms"] == 27.5 and e["best"][3:5] == [8, 4] and e["best"][2] in (0, 32)


def test_measurements_of_another_solver_are_not_used(tune, monkeypatch):
    from paper_1803_01516_gb300 import gazecut as gc
    p = gc.Params(w=384, h=288, D=16, tau=30, lam=10)
    shipped = tune.tuned_opts(p)
    stale = {"best": [64, 4, 4, 16, 8, 16, 512], "ms": 1.0, "all_ms": {"64,4,4,16,8,16,512": 1.0}}
    with open(tune.cache_path(), "w") as f:
        json.dump({tune.bucket(p): stale}, f)
    assert tune.tuned_opts(p) == shipped
    monkeypatch.setattr(tune, "_time_config",
                        lambda pp, pairs, cfg, reps=2: 1.0 if cfg[0] == 64 else 2.0)
    e = tune.tune(p, pairs=_pairs(p))               # replaces the stale entry
    assert tune.tuned_opts(p).sweeps_per_relabel == 64 == e["best"][0]

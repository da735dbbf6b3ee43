"""The autotuner's candidates for contexts whose own form is one CTA per instance
(without a GPU): the default, the only choice that gives that form, is among them, and
a cached choice of it reads back."""
from types import SimpleNamespace

from paper_2303_01471_gb300 import autotune


def sims(*edges_and_ctas):
    return [SimpleNamespace(shape=(e, e), batch=400, cluster_ctas=lambda c=c: c) for e, c in edges_and_ctas]


def test_own_form_is_a_candidate():
    subs = {tuple(c.as_dict()["sub"]) for c in autotune.candidates(sims((64, 1), (128, 1), (256, 8)))}
    assert subs == {(a, b, 8) for a in (0, 2, 4, 8) for b in (0, 4, 8)}
    subs = {tuple(c.as_dict()["sub"]) for c in autotune.candidates(sims((64, 4), (128, 1)))}
    assert subs == {(a, b, 0) for a in (2, 4, 8) for b in (0, 4, 8)}


def test_own_form_is_kept_when_fastest(tmp_path, monkeypatch):
    monkeypatch.setattr(autotune, "time_config", lambda s, cfg, T, dt, reps=2: 1.0 + cfg.sub_cluster[0] + cfg.min_blocks)
    monkeypatch.setattr(autotune, "cache_key", lambda s: "k")
    cache = str(tmp_path / "group.json")
    for cached in (False, True):
        res = autotune.tune_group(sims((64, 1)), cache_file=cache)
        assert res["cached"] == cached and res["config"].as_dict() == {"sub": [0, 0, 0], "min_blocks": 1, "clusters": 0}

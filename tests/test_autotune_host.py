"""The autotuner's cache on the host, with the timing replaced."""
import json

import pytest


@pytest.fixture(scope="module")
def autotune():
    import __graft_entry__ as g

    g.build()
    from paper_2205_05835_gb300 import autotune

    return autotune


P = {"dim": 3, "n": (64, 64, 64), "precision": "fp64", "rho_in": 10.0, "rho_out": 1.0}


def test_a_cache_of_other_settings_is_not_used(autotune, monkeypatch, tmp_path):
    """A choice stored under a key without the settings' version (when 4096 was the
    default) is timed anew; one stored now is found again."""
    timed = []
    monkeypatch.setattr(autotune, "_time_candidate",
                        lambda pf, p, c, steps, warm: timed.append(c) or 1.0)
    path = tmp_path / "tuned.json"
    old_key = json.dumps([3, [64, 64, 64], "fp64", "None", "None", 10.0, 0, 0, 0.0, 0.0, False])
    old = {"choice": {"mg_coarse_cells": 4096, "mg_pre": 1, "mg_post": 1}, "ms_per_step": {}}
    path.write_text(json.dumps({old_key: old}))
    autotune._cache.clear()
    r = autotune.tune(P, cache_path=str(path))
    assert not r["cached"] and len(timed) == len(autotune.CANDIDATES)
    assert r["choice"] == autotune.DEFAULT_SHAPE
    autotune._cache.clear()
    again = autotune.tune(P, cache_path=str(path))
    assert again["cached"] and again["choice"] == r["choice"]
    assert len(timed) == len(autotune.CANDIDATES)
    autotune._cache.clear()


@pytest.mark.parametrize("one", [True, False])
def test_candidates_that_are_the_same_are_timed_once(autotune, monkeypatch, one):
    """On a 2D grid solved in one launch mg_coarse_cells does nothing: one timing for
    each pair of sweep counts, and the library's rule among equals."""
    timed = []

    def fake(pf, p, c, steps, warm):
        timed.append(c)
        return 0.5 if c["mg_pre"] == 2 else 1.0
    monkeypatch.setattr(autotune, "_time_candidate", fake)
    monkeypatch.setattr(autotune, "_one_launch", lambda pf, p: one, raising=False)
    autotune._cache.clear()
    r = autotune.tune(dict(P, dim=2, n=(64, 64, 1)))
    sweeps = {(c["mg_pre"], c["mg_post"]) for c in autotune.CANDIDATES}
    assert len(timed) == (len(sweeps) if one else len(autotune.CANDIDATES))
    assert len(r["ms_per_step"]) == len(autotune.CANDIDATES)
    assert r["choice"] == {"mg_coarse_cells": 0, "mg_pre": 2, "mg_post": 2}
    autotune._cache.clear()

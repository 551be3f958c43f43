"""The autotune cache's key and the candidates it stands for."""
import json

import pytest

import paper_2311_05341_gb300 as dd
from synth import channel_freqs


def test_cache_entries_of_older_candidates_are_not_taken(tmp_path):
    """A file written when the candidates were the explicit shapes alone (its key
    names no version) pins none of today's plans to one of them."""
    pytest.importorskip("torch")
    from paper_2311_05341_gb300 import batch
    freqs = channel_freqs(1500.0, 300.0, 64)
    plan = dd.Plan(freqs, 1500.0, 64e-6, [(0.0, 6.4, 0.1, 1)], "u8", upload=False)
    n = 20000
    key = json.loads(batch.plan_signature(plan, n))
    old = json.dumps(key[:7]) + "|packed|tiles=" + json.dumps([4])
    cache = tmp_path / "tune.json"
    cache.write_text(json.dumps({old: [["pattern", 0]]}))
    tuner = batch.Autotuner(shapes=[4], cache_path=str(cache))  # one candidate: nothing is timed
    assert tuner.choose(plan, n, None, None) == [(4, -1)]
    assert len(json.loads(cache.read_text())) == 2


def test_the_automatic_shape_is_a_candidate():
    pytest.importorskip("torch")
    from paper_2311_05341_gb300 import batch
    freqs = channel_freqs(1500.0, 300.0, 600)
    plan = dd.Plan(freqs, 1500.0, 64e-6, [(0.0, 10.0, 0.05, 1)], "u8", upload=False)
    found = batch.tile_candidates(plan, 0)
    assert ("pattern", -1) in found and ("packed", -1) in found

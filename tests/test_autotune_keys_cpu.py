"""Which cached choices the launch-configuration tuner reads (no GPU): those of
the same shapes, kernels and size of batch.  The timed calls are replaced by a
table of times by placement."""
import json
import types

import numpy as np
import pytest
import torch

from paper_1101_5803_gb300 import autotune


def _batch(n):
    geom = types.SimpleNamespace(nx=128, ny=128, sx=48, sy=48, kpsf=11, subpix=1, reg=2)
    return ([types.SimpleNamespace(geom=geom)], torch.zeros((n, 7), dtype=torch.float64), np.zeros(n, np.int32),
            torch.ones((n, 16), dtype=torch.float64), np.full(n, 16, np.int32))


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    path = tmp_path / "tune.json"
    monkeypatch.setenv("MIRAGE_TUNE_CACHE", str(path))
    timed = []

    def fake(ctx, probs, lens, prob_idx, lam, nl, reps, **kw):
        timed.append(int(lens.shape[0]))
        return 50.0 if kw.get("place") == 4 and int(lens.shape[0]) >= 256 else 100.0
    monkeypatch.setattr(autotune, "_time", fake)
    return types.SimpleNamespace(precision=autotune.MIRAGE_FP32), path, timed


def test_small_batches_do_not_take_a_full_devices_placement(tuner):
    # placement 4 (all in the slab) is faster on 256 candidates, the automatic one on 4
    ctx, _, timed = tuner
    assert autotune.tune_config(ctx, *_batch(256))["place"] == 4
    timed.clear()
    assert autotune.tune_config(ctx, *_batch(4))["place"] == 0
    assert timed
    timed.clear()
    assert autotune.tune_config(ctx, *_batch(4))["place"] == 0 and not timed  # each from the cache now
    assert autotune.tune_config(ctx, *_batch(256))["place"] == 4 and not timed


def test_choices_of_other_kernels_are_timed_again(tuner):
    ctx, path, timed = tuner
    autotune.tune_config(ctx, *_batch(256))
    db = json.loads(path.read_text())
    key, entry = next(iter(db.items()))
    old = json.loads(key)
    del old["kernels"], old["items"]  # as entries were keyed before
    path.write_text(json.dumps({json.dumps(old): dict(entry, place=3)}))
    timed.clear()
    assert autotune.tune_config(ctx, *_batch(256))["place"] == 4 and timed

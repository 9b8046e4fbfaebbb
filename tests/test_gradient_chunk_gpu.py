"""The x-chunk of the FWI gradient's passes: one that the options name is the one
that runs, whatever was timed for the grid before (a single chunk over all planes
of a one-tile grid is one CTA's chain of planes: several times the time of the
chunks that are timed), and no chunk changes a bit of the gradient, the traces or
the misfit, with checkpoints and without, nor does switching the timing off."""
from __future__ import annotations

import numpy as np
import pytest

import paper_1912_00695_gb300 as fd
from harness import dt_for
from paper_1912_00695_gb300 import inputs

pytestmark = pytest.mark.gpu

INTERIOR, NBL, K, NT = (300, 8, 20), 4, 8, 60  # 308 x 16 x 28 points: one 32x16 tile


def _gradient(repeats=1, segment=0, **opts):
    rng = np.random.default_rng(3)
    vel = inputs.smooth_random_velocity(INTERIOR, NBL, rng, sigma=3.0)
    spec = inputs.ShotSpec(INTERIOR, NBL, K, vel, (150, 4, 5), 25.0, NT)
    dt = dt_for(spec)
    rec = np.stack([np.linspace(1.0, 290.0, 40), np.full(40, 3.25), np.full(40, 10.5)], axis=1)
    obs = rng.standard_normal((40, NT)).astype(np.float32)
    with fd.Shot(INTERIOR, K, inputs.H, dt, NBL, **opts) as shot:
        shot.set_model(spec.m)
        shot.inject(*spec.source, inputs.ricker(spec.f0, dt, NT))
        ms = []
        for _ in range(repeats):
            out = shot.fwi_gradient(rec, obs, segment=segment)
            ms.append(shot.last_forward_ms())
    return out, min(ms)


def test_a_forced_chunk_is_the_one_that_runs():
    _, timed = _gradient(repeats=4)
    _, forced = _gradient(repeats=4, x_block=308)
    print(f"GRADIENT CHUNK timed {timed / NT * 1e3:.1f} forced {forced / NT * 1e3:.1f} us a step")
    assert forced >= 3.0 * timed


@pytest.mark.parametrize("segment", [0, 7])
def test_no_chunk_changes_a_bit(segment, monkeypatch):
    want, _ = _gradient(segment=segment)
    assert np.abs(want[0]).max() > 0
    others = [_gradient(segment=segment, x_block=xb)[0] for xb in (1, 5, 308)]
    monkeypatch.setenv("FDGB_NO_TUNE", "1")
    others.append(_gradient(segment=segment)[0])
    for got in others:
        np.testing.assert_array_equal(got[0], want[0])
        np.testing.assert_array_equal(got[1], want[1])
        assert got[2] == want[2]

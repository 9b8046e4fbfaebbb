"""The schedule of a BF16 shot left to the library follows the grid and the
handle's own calls, never a timing or another shot: a short forward is the flow
schedule bit for bit, before and after an FP32 shot has timed the same grid, whole
and in parts; a forward long enough to time runs per-step launches on a small grid
and the flow on a large one, from its first step on. (The two schedules store BF16
levels at different power-of-two scales, and their fields part after a few hundred
steps on the small grid used here.)"""
from __future__ import annotations

import numpy as np
import pytest

import paper_1912_00695_gb300 as fd
from harness import dt_for
from paper_1912_00695_gb300 import inputs

pytestmark = pytest.mark.gpu

SMALL = ((86, 83, 79), 12, 10)    # 2.9 planes per item: below the line of 5
LARGE = ((140, 150, 160), 8, 10)  # 9.3 planes: above it


def _run(grid, calls, **opts):
    """Fields after the calls, (steps, "forward" or "flow") each, and the schedule of the last."""
    interior, k, nbl = grid
    rng = np.random.default_rng(k)
    vel = inputs.smooth_random_velocity(interior, nbl, rng, sigma=4.0)
    spec = inputs.ShotSpec(interior, nbl, k, vel, tuple(n // 2 for n in interior), 15.0, 300)
    dt = dt_for(spec)
    with fd.Shot(interior, k, inputs.H, dt, nbl, **opts) as shot:
        shot.set_model(spec.m)
        shot.inject(*spec.source, inputs.ricker(spec.f0, dt, spec.nt))
        for n, how in calls:
            if n == 0:
                shot.reset()
            else:
                (shot.forward_flow if how == "flow" else shot.forward)(n)
        return shot.wavefield(0), shot.wavefield(1), shot.schedule[1]


def _equal(got, want):
    for g, w in zip(got[:2], want[:2]):
        np.testing.assert_array_equal(g, w)


def test_short_forward_does_not_depend_on_other_shots():
    want = _run(SMALL, [(130, "flow")], storage="bf16")
    assert np.abs(want[0]).max() > 0
    before = _run(SMALL, [(130, "forward")], storage="bf16")
    _run(SMALL, [(300, "forward")])                  # an FP32 shot times the grid
    _run(SMALL, [(300, "flow")], storage="bf16")     # and a BF16 one its x-chunks
    for got in (before, _run(SMALL, [(130, "forward")], storage="bf16"),
                _run(SMALL, [(1, "forward"), (40, "forward"), (89, "forward")], storage="bf16"),
                _run(SMALL, [(300, "forward"), (0, "reset"), (130, "forward")], storage="bf16")):
        _equal(got, want)
        assert got[2] == 1


@pytest.mark.parametrize("grid,schedule", [(SMALL, 0), (LARGE, 1)])
def test_long_forward_keeps_one_schedule(grid, schedule):
    pinned = dict(kernel="tma") if schedule == 0 else {}
    want = _run(grid, [(300, "forward" if schedule == 0 else "flow")], storage="bf16", **pinned)
    for calls in ([(300, "forward")], [(200, "forward"), (100, "forward")]):
        got = _run(grid, calls, storage="bf16")
        _equal(got, want)
        assert got[2] == schedule

"""A first forward too short to time the schedules picks one by rule from the
grid (per-step launches on small grids, the flow schedule with an even x-chunk
on larger ones): on grids on both sides of the rule's line the fields equal the
per-step launches' bit for bit, for one call, split calls and a longer call
after a short one."""
from __future__ import annotations

import numpy as np
import pytest

import paper_1912_00695_gb300 as fd
from harness import dt_for
from paper_1912_00695_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,form,interior,nbl", [
    (4, "factored", (20, 24, 30), 6), (2, "expanded", (64, 64, 64), 10), (8, "factored", (110, 101, 97), 10),
    (16, "factored", (140, 120, 131), 8), (8, "expanded", (9, 150, 170), 4), (24, "factored", (150, 90, 70), 10),
])
def test_short_forward_equals_per_step(k, form, interior, nbl):
    rng = np.random.default_rng(k)
    spec = inputs.ShotSpec(interior, nbl, k, inputs.smooth_random_velocity(interior, nbl, rng, sigma=4.0),
                           tuple(n // 2 for n in interior), 25.0, 60)
    dt = dt_for(spec)
    wav = inputs.ricker(spec.f0, dt, spec.nt)

    def run(chunks, **opts):
        with fd.Shot(interior, k, inputs.H, dt, nbl, form=form, **opts) as shot:
            shot.set_model(spec.m)
            shot.inject(*spec.source, wav)
            for n in chunks:
                shot.forward(n)
            return shot.wavefield(0), shot.wavefield(1)

    want = run([31], kernel="tma")
    for chunks in ([31], [1, 30], [10, 10, 11]):
        for got, ref in zip(run(chunks), want):
            np.testing.assert_array_equal(got, ref)
    want = run([221], kernel="tma")
    for got, ref in zip(run([21, 200]), want):
        np.testing.assert_array_equal(got, ref)

"""Short first forwards of FP32 shots with receivers and with more than the four
fused sources, on grids on both sides of the schedule rule's line and in calls below
and above its 16 steps; and steps whose launches overlap the end of the stream's
previous kernel, on a stream of the caller's behind another stream's kernel and an
event. Fields and traces equal the per-step launches' bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import paper_1912_00695_gb300 as fd
from harness import dt_for
from paper_1912_00695_gb300 import inputs

pytestmark = pytest.mark.gpu


def _spec(k, interior, nbl=8):
    rng = np.random.default_rng(k)
    vel = inputs.smooth_random_velocity(interior, nbl, rng, sigma=4.0)
    return inputs.ShotSpec(interior, nbl, k, vel, tuple(n // 2 for n in interior), 25.0, 60)


@pytest.mark.parametrize("k,form,interior", [(4, "factored", (40, 44, 50)), (8, "expanded", (61, 33, 70)),
                                             (8, "factored", (150, 140, 160)), (2, "factored", (50, 40, 60))])
@pytest.mark.parametrize("receivers,sources", [(True, 1), (False, 5), (True, 6)])
def test_receivers_and_extra_sources(k, form, interior, receivers, sources):
    spec = _spec(k, interior)
    dt = dt_for(spec)
    rng = np.random.default_rng(sources)
    rec = rng.uniform(0.0, 1.0, (50, 3)) * (np.array(interior) - 2)
    at = [tuple(int(v) for v in rng.integers(0, interior)) for _ in range(sources - 1)]

    def run(calls, **opts):
        with fd.Shot(interior, k, inputs.H, dt, spec.nbl, form=form, **opts) as shot:
            shot.set_model(spec.m)
            for i, node in enumerate([spec.source] + at):
                shot.inject(*node, inputs.ricker(20.0 + i, dt, spec.nt))
            if receivers:
                shot.set_receivers(rec, 40)
            for n in calls:
                shot.forward(n)
            out = [shot.wavefield(0), shot.wavefield(1)]
            return out + ([shot.traces()] if receivers else [])

    want = run([36], kernel="tma")
    for calls in ([36], [7, 29], [20, 16]):
        for g, w in zip(run(calls), want):
            np.testing.assert_array_equal(g, w)


@pytest.mark.parametrize("k,calls", [(2, [40]), (2, [1, 6, 33]), (4, [40]), (4, [200])])
def test_overlapped_launches_behind_another_stream(k, calls):
    torch = pytest.importorskip("torch")
    spec = _spec(k, (46, 50, 60))
    dt = dt_for(spec)
    wav = inputs.ricker(25.0, dt, sum(calls))

    def run(behind, **opts):
        m = torch.from_numpy(spec.m).cuda()
        held = torch.zeros_like(m) if behind else m
        a, b = torch.cuda.Stream(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with fd.Shot(spec.interior, k, inputs.H, dt, spec.nbl, **opts) as shot:
            shot.set_stream(b.cuda_stream)
            if behind:
                # the model arrives late, from the other stream; the shot's stream waits for it
                with torch.cuda.stream(a):
                    torch.cuda._sleep(20_000_000)
                    held.copy_(m)
                b.wait_stream(a)
            shot.set_model_device(held.data_ptr())
            shot.inject(*spec.source, wav)
            for n in calls:
                if behind:
                    with torch.cuda.stream(a):
                        torch.cuda._sleep(2_000_000)
                    b.wait_stream(a)
                    with torch.cuda.stream(b):
                        held.mul_(1.0)  # a kernel right before the steps
                shot.forward(n)
            out = shot.wavefield(0), shot.wavefield(1)
            torch.cuda.synchronize()
            return out

    want = run(False, kernel="tma")
    assert np.abs(want[0]).max() > 0
    for _ in range(2):
        for g, w in zip(run(True), want):
            np.testing.assert_array_equal(g, w)

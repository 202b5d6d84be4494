"""Launches of the solve server's residents.

Alone a resident takes the launch tuned for its shape; residents that step
together keep the automatic one, whose chunks go by all their grids.
"""
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tune", [True, False])
def test_residents_together_keep_the_automatic_launch(monkeypatch, tune):
    from paper_1010_4135_gb300 import autotune, serve

    def tuned(sims, *a, **k):  # an explicit launch for every shape
        for s in sims:
            s.set_launch("tiled", 4, 0)
        return {}

    monkeypatch.setattr(autotune, "_tune", tuned)
    seen = []
    real = serve.S.step_batch

    def step_batch(sims, n):
        seen.append([s.launch for s in sims])
        return real(sims, n)

    monkeypatch.setattr(serve.S, "step_batch", step_batch)
    tr = workloads.serving_trace(seed=7, n=5, rate=200.0, grids=((16, 16, 16), (24, 16, 16), (32, 16, 8)),
                                 steps=(6000, 12000))  # long enough that requests overlap
    srv = serve.Server(max_batch=3, tick=16, prep_workers=5, tune=tune)
    done = srv.run(tr)
    assert len(done) == 5 and all(j.health == 0 for j in done)
    assert max(map(len, seen)) > 1 and min(map(len, seen)) == 1
    for launches in seen:
        want = ("tiled", 4, 0) if tune and len(launches) == 1 else ("tiled", 0, 0)
        assert launches == [want] * len(launches)

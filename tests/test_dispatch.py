"""Which kernels a call launches (see dispatch.py): the rules on sizes and parameters."""
import pytest

import dispatch as D
from paper_2102_01747_gb300 import workloads as W


@pytest.mark.parametrize("p", [2, 3])
@pytest.mark.parametrize("max_iter,unroll", [(1, 2), (2, 2), (3, 8), (11, 8)])
def test_julia_steps_per_escape_test_follow_the_cap(max_iter, unroll, p):
    s = dict(W.julia_256(), p=p, max_iter=max_iter)
    assert D.launches(s) == [("plain_kernel", (0, unroll, 0, 0, 0, 0))]


def _scenes():
    for w, h in ((64, 36), (256, 120), (256, 130), (640, 360)):
        bulb, julia = W.bulb_1080p(10, w, h), W.julia_256(w, h)
        for s in (bulb, dict(bulb, n=5), dict(bulb, algebraic=True), dict(bulb, normal_mode="analytic"), julia,
                  dict(julia, max_iter=2), dict(julia, normal_mode="analytic")):
            for spp in (1, 3, 4):
                t = dict(s, camera=dict(s["camera"], spp=spp))
                yield t
                yield W.phong(t)


def test_the_tuner_times_each_kernel_once(monkeypatch):
    from paper_2102_01747_gb300 import api, autotune

    start = dict(plain_block=128, plain_unroll=1, persist_block=64, persist_ctas_per_sm=0, refill_threshold=16,
                 persist_unroll=4, single_kernel=0, batch_kernel=2, tile_order=0, sample_lanes=1)
    state = dict(start)
    monkeypatch.setattr(autotune, "current", lambda: dict(state))
    monkeypatch.setattr(autotune, "apply", state.update)
    monkeypatch.setattr(autotune, "_time_single", lambda *a: 1.0)
    monkeypatch.setattr(api, "alloc_image", lambda scene: None)
    for s in _scenes():
        for kernel in (0, 2):
            state.update(start)
            trials = autotune.tune_single(s, start_kernel=kernel)["trials"]
            trials = [{k: v for k, v in t.items() if k != "ms"} for t in trials]
            base = trials[0]
            for knob in ("plain_unroll", "sample_lanes"):
                for v in autotune.SINGLE_SPACE[knob]:
                    cand = dict(base, **{knob: v})
                    differs = D.launches(s, tuning=cand, shapes=True) != D.launches(s, tuning=base, shapes=True)
                    assert (cand in trials[1:]) == differs, (s, knob, v)


def test_kernel_scenes_reach_every_forward_kernel():
    import kernel_scenes

    reached = set()
    for group in kernel_scenes.GROUPS.values():
        for name, scenes, batch, tuning, stats in group():
            want = dict(rgba8=True, depth=True, stats=stats)
            reached.update(D.launches(scenes if batch else scenes[0], batch, tuning, **want))
    probe = {("plain_kernel", (kind, 1, 2, 1, 1, 0)) for kind in (0, 1)}  # fr_work_probe's
    forward = {k for k in D.kernels() if k[0] not in ("backward_kernel", "ffma_probe_kernel")} - probe
    assert reached <= forward
    assert reached == forward, sorted(forward - reached)

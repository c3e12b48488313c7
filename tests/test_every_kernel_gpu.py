"""Every forward kernel of the library (kernel_scenes.py) against the lane state machine,
which marches every ray to the end of its interval, tests each orbit step's escape and
takes the Mandelbulb's general step: colours, depth, saved state, trap and counters bit
for bit."""
import functools
import json

import numpy as np
import pytest

import kernel_scenes

pytestmark = pytest.mark.gpu

OUTS = dict(rgba8=True, rgba=True, depth=True, saved=True, trap=True)


def _render(scenes, batch, tuning, stats):
    import torch
    from paper_2102_01747_gb300 import api, autotune

    old = autotune.current()
    autotune.apply(tuning)
    try:
        want = dict(OUTS, stats=stats)
        outs = api.render_batch(scenes, **want) if batch else [api.render(scenes[0], **want)]
        torch.cuda.synchronize()
    finally:
        autotune.apply(old)
    return [{k: v.cpu().numpy().view(np.uint8) for k, v in o.items()} for o in outs]


@functools.lru_cache(maxsize=None)
def _reference(scene: str):
    return _render([json.loads(scene)], False, dict(single_kernel=1, persist_unroll=4), True)[0]


@pytest.mark.parametrize("group", list(kernel_scenes.GROUPS))
def test_every_kernel(group):
    for name, scenes, batch, tuning, stats in kernel_scenes.GROUPS[group]():
        refs = [_reference(json.dumps(s)) for s in scenes]
        assert any(r["saved"].any() for r in refs), name  # something was hit
        for i, (got, ref) in enumerate(zip(_render(scenes, batch, tuning, stats), refs)):
            assert set(got) == set(OUTS) | ({"stats"} if stats else set())
            for k in got:
                assert np.array_equal(got[k], ref[k]), (name, i, tuning, stats, k)

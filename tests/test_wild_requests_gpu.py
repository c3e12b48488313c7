"""Mandelbulb requests whose iterates may overflow: through every kernel the bits of
the lane state machine, which always takes the general orbit step."""
import numpy as np
import pytest

from paper_2102_01747_gb300 import workloads as W

pytestmark = pytest.mark.gpu

OUTS = dict(rgba8=True, rgba=True, depth=True, saved=True, trap=True)


def tuned(**kw):
    import contextlib

    from paper_2102_01747_gb300 import autotune

    @contextlib.contextmanager
    def scope():
        old = autotune.current()
        autotune.apply(kw)
        try:
            yield
        finally:
            autotune.apply(old)

    return scope()


def general(scene):
    import torch
    from paper_2102_01747_gb300 import api

    with tuned(single_kernel=1):
        out = api.render(scene, **OUTS)
        torch.cuda.synchronize()
    return {k: v.cpu().numpy().view(np.uint32) for k, v in out.items()}


def same(out, ref, where):
    for k in ref:
        got = out[k].cpu().numpy().view(np.uint32)
        assert np.array_equal(got, ref[k]), (where, k, float(np.mean(got != ref[k])))


def wild_scene(n, i, w=61, h=45):
    s = W.bulb_1080p(7 * i, w, h)
    s.update(n=n, bailout=10.0 ** (22.0 / n), max_iter=4 + i % 7, algebraic=bool(i % 2),
             normal_mode=("tetra", "central", "analytic")[i % 3])
    s["camera"]["spp"] = (1, 1, 2, 3, 4)[i % 5]
    return W.phong(s) if i % 4 == 3 else s


@pytest.mark.parametrize("phong", [False, True])
@pytest.mark.parametrize("spp", [1, 4])
@pytest.mark.parametrize("batch_kernel", [0, 1, 2])
def test_batch_with_wild_requests(batch_kernel, spp, phong):
    import torch
    from paper_2102_01747_gb300 import api

    scenes = W.batch_mixed(3, 8, 5.0, 6.5) + [wild_scene(n, i) for i, n in enumerate((2, 4, 8, 11, 16))]
    for i, s in enumerate(scenes):
        if not phong:
            s["light"]["shading"] = "lambert"
        s["camera"]["spp"] = spp if i % 3 else 1
    if phong:
        scenes[0], scenes[1] = W.phong(scenes[0]), W.phong(scenes[1])
    refs = [general(s) for s in scenes]
    with tuned(batch_kernel=batch_kernel):
        outs = api.render_batch(scenes, **OUTS)
        torch.cuda.synchronize()
    for i, (o, r) in enumerate(zip(outs, refs)):
        same(o, r, i)


@pytest.mark.parametrize("normal_mode", ["tetra", "central", "analytic"])
@pytest.mark.parametrize("phong", [False, True])
@pytest.mark.parametrize("n", [2, 3, 8, 16])
def test_single_wild_requests(n, phong, normal_mode):
    import torch
    from paper_2102_01747_gb300 import api

    for i, (w, h) in enumerate(((61, 45), (258, 151))):  # spare lanes, one lane per pixel
        for spp in (1, 3, 4):
            s = W.bulb_1080p(9 * n, w, h)
            s.update(n=n, bailout=10.0 ** (22.0 / n), max_iter=5 + i, normal_mode=normal_mode, algebraic=spp == 3)
            s["camera"]["spp"] = spp
            s = W.phong(s) if phong else s
            ref = general(s)
            for kernel in (0, 2):
                with tuned(single_kernel=kernel):
                    out = api.render(s, **OUTS)
                    torch.cuda.synchronize()
                same(out, ref, (w, spp, kernel))



@pytest.mark.parametrize("n", range(2, 17))
def test_both_steps_on_either_side_of_the_limit(n):
    import torch
    from paper_2102_01747_gb300 import api

    limit = 1e19 ** (1.0 / n)
    for factor in (0.5, 0.9999, 1.0001):
        s = W.bulb_1080p(11 * n, 150, 110)
        s.update(n=n, bailout=limit * factor, max_iter=9, algebraic=factor == 0.5)
        s["camera"]["spp"] = 3  # one lane per pixel
        far = dict(s, plane=None, bailout=2.0, bound_radius=min((limit - 1.0) / 1.01 * factor, 990.0), max_step=50.0)
        for scene in (s, far, dict(s, algebraic=factor != 0.5)):
            ref = general(scene)
            out = api.render(scene, **OUTS)
            torch.cuda.synchronize()
            same(out, ref, (factor, scene["bound_radius"]))

"""The Mandelbulb's orbit step without special paths (bulb_step_tame) against
the general step: the counting kernels run the general one, so an image rendered
with the statistics counters must equal the image without them bit for bit.
Scenes cover every power, both ends of the accepted parameters (large bailouts
and radii, where iterates overflow and the general step serves both), points on
the polar axis and at the origin, and every output."""
import numpy as np
import pytest

from paper_2102_01747_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def both(scene, **kw):
    import torch
    from paper_2102_01747_gb300 import api

    a = api.render(scene, rgba=True, trap=True, saved=True, **kw)
    b = api.render(scene, rgba=True, trap=True, saved=True, stats=True, **kw)
    torch.cuda.synchronize()
    for k in a:
        x, y = (o[k].cpu().numpy().view(np.uint32) for o in (a, b))
        assert np.array_equal(x, y), (k, float(np.mean(x != y)))
    return a


@pytest.mark.parametrize("n", range(2, 17))
@pytest.mark.parametrize("phong", [False, True])
@pytest.mark.parametrize("algebraic", [False, True])
def test_every_power(n, phong, algebraic):
    s = W.bulb_1080p(7 * n, 131, 93)
    s.update(n=n, algebraic=algebraic, max_iter=6 + n, normal_mode=("tetra", "central", "analytic")[n % 3])
    s["camera"]["spp"] = (1, 2, 3, 4)[n % 4]
    both(W.phong(s) if phong else s)


@pytest.mark.parametrize("n", [2, 5, 8, 16])
@pytest.mark.parametrize("bailout", [0.3, 1.0, 300.0, 1e4, 1e10, 1e20])
def test_bailouts(n, bailout):
    s = W.bulb_1080p(3, 65, 47)
    s.update(n=n, bailout=bailout, max_iter=9)
    both(s)
    both(dict(s, algebraic=True))


@pytest.mark.parametrize("change", [dict(bound_radius=0.5), dict(bound_radius=50.0), dict(bound_radius=1e5),
                                    dict(normal_h=0.3), dict(normal_h=1e4), dict(eps=0.2), dict(max_iter=1),
                                    dict(max_steps=1), dict(max_steps=9), dict(max_iter=200, eps=1e-5)])
def test_edges_of_the_parameters(change):
    s = W.bulb_1080p(20, 65, 47)
    s.update(change)
    both(s)


def test_axis_and_origin():
    # odd sizes put a pixel's ray through the origin, along each axis
    for eye, up in (((0.0, 2.5, 0.0), (0.0, 0.0, 1.0)), ((0.0, 0.0, 2.5), (0.0, 1.0, 0.0)),
                    ((2.5, 0.0, 0.0), (0.0, 1.0, 0.0)), ((0.0, 0.0, 0.0), (0.0, 1.0, 0.0))):
        for n in (2, 3, 8):
            s = W.bulb_1080p(0, 33, 33)
            s.update(n=n, plane={"n": (0.0, 1.0, 0.0), "o": 0.0}, eps=1e-6)
            s["camera"].update(eye=eye, up=up, target=(0.0, 0.0, -1.0) if eye == (0.0, 0.0, 0.0) else (0.0, 0.0, 0.0))
            both(s)
            both(dict(s, algebraic=True))


def test_batch_with_an_overflowing_request():
    import torch
    from paper_2102_01747_gb300 import api

    scenes = W.batch_mixed(5, 6, 5.0, 6.0)
    scenes[1]["bailout"] = 1e9
    outs = api.render_batch(scenes)
    for s, o in zip(scenes, outs):
        one = api.render(s)
        torch.cuda.synchronize()
        assert torch.equal(o["rgba8"], one["rgba8"]) and torch.equal(o["depth"], one["depth"])

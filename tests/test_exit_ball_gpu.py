"""Marches that end once the ray has left the fractal's ball (exit_t) against
marches to the end of the interval: the counting kernels take every distance,
so an image rendered with the statistics counters must equal the image without
them bit for bit.  Scenes reach the rule's edges: balls close to the bounding
sphere, step caps that could run out on the way, eyes inside and outside, long
steps, sets that fill the ball."""
import numpy as np
import pytest

from paper_2102_01747_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def both(scene):
    import torch
    from paper_2102_01747_gb300 import api

    a = api.render(scene, rgba=True, saved=True)
    b = api.render(scene, rgba=True, saved=True, stats=True)
    torch.cuda.synchronize()
    for k in a:
        x, y = (o[k].cpu().numpy().view(np.uint32) for o in (a, b))
        assert np.array_equal(x, y), (k, float(np.mean(x != y)))


def julia(c, **kw):
    s = W.julia_256(97, 71)
    s["c"] = c
    s["light"]["shadows"] = True
    s.update(kw)
    return s


@pytest.mark.parametrize("p", [2, 3])
@pytest.mark.parametrize("c", [(0.0, 0.0, 0.0, 0.0), (0.25, 0.0, 0.0, 0.0), (-1.0, 0.0, 0.0, 0.0),
                               (-0.2, 0.6, 0.2, 0.0), (0.0, 0.0, 0.0, 0.8), (1.2, 0.0, 0.0, 0.0), (-1.9, 0.1, 0.0, 0.0)])
def test_julia_constants(p, c):
    both(julia(c, p=p))
    both(julia(c, p=p, slice_w=0.4, escape_r2=256.0))


@pytest.mark.parametrize("kind", ["julia", "bulb"])
@pytest.mark.parametrize("change", [dict(max_steps=k) for k in (1, 3, 8, 20, 40, 90)] +
                         [dict(max_step=v) for v in (0.01, 0.05, 5.0)] +
                         [dict(bound_radius=v) for v in (0.7, 1.16, 1.2, 1.3, 8.0, 15.0)] +
                         [dict(eps=v) for v in (1e-6, 0.02, 0.05, 0.2)] +
                         [dict(max_iter=v) for v in (1, 2, 3, 40)] +
                         [dict(escape_r2=v * v, bailout=v) for v in (0.5, 1.05, 1.3, 40.0)])
def test_edges_of_the_rule(kind, change):
    s = julia((-0.2, 0.6, 0.2, 0.0)) if kind == "julia" else W.bulb_1080p(17, 97, 71)
    s.update(change)
    both(s)


@pytest.mark.parametrize("eye", [(0.0, 0.0, 1.3), (0.3, 1.1, 0.2), (0.0, 0.01, 15.9), (0.0, 0.01, 400.0), (1.0, 0.8, -2.0)])
@pytest.mark.parametrize("kind", ["julia", "bulb"])
def test_eyes_and_mirror_rays(kind, eye):
    s = julia((-0.2, 0.6, 0.2, 0.0)) if kind == "julia" else W.bulb_1080p(0, 97, 71)
    s["camera"].update(eye=eye, fov_y_deg=100.0 if eye[2] < 15 else 12.0)
    both(s)
    both(W.phong(s))


def test_small_exponents():
    for n in (2, 3, 4, 16):
        s = W.bulb_1080p(40, 97, 71)
        s.update(n=n, bound_radius=2.5, plane=None)
        both(s)


@pytest.mark.parametrize("max_iter", [1, 2, 3, 4, 5, 6, 9, 11])
@pytest.mark.parametrize("p", [2, 3])
@pytest.mark.parametrize("size", [(97, 71), (412, 395)])
def test_julia_steps_per_escape_test(size, p, max_iter):
    # small images take four orbit steps per escape test, larger ones two, the counting kernels one
    s = W.resized(julia((-0.3, 0.5, 0.3, 0.1), p=p, max_iter=max_iter), *size)
    both(s)
    both(W.phong(dict(s, normal_mode="tetra")))

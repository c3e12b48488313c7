"""Mandelbulb requests whose iterates may overflow (large bailouts and radii: r^n up to
1e19 keeps |w|^2 finite) take the general orbit step.  Which kernels such calls launch: none that counts, and
none that a request beside them would not have."""
import pytest

import dispatch as D
from paper_2102_01747_gb300 import workloads as W

COUNT_ARG = {"plain_kernel": 2, "batch_plain_kernel": 1, "batch_refill_kernel": 1, "persist_kernel": 1}


def wild(w=64, h=48, **kw):
    return dict(W.bulb_1080p(10, w, h), bailout=1e4, **kw)


def mixed(spp=1, phong=False):
    scenes = W.batch_mixed(3, 6, 5.0, 6.0)
    scenes[3] = wild(24, 16)
    scenes[2]["camera"]["spp"] = spp
    if phong:
        scenes[0] = W.phong(scenes[0])
    return scenes


@pytest.mark.parametrize("phong", [False, True])
@pytest.mark.parametrize("spp", [1, 4])
@pytest.mark.parametrize("batch_kernel", [0, 1, 2])
def test_batch_with_a_wild_request(batch_kernel, spp, phong):
    scenes = mixed(spp, phong)
    tuning = dict(batch_kernel=batch_kernel, plain_unroll=1)
    (kernel,) = D.launches(scenes, batch=True, tuning=tuning)
    (without,) = D.launches([dict(s, bailout=2.0) for s in scenes], batch=True, tuning=tuning)
    assert kernel[1][COUNT_ARG[kernel[0]]] == 0
    # the lane state machine always takes the general step; the others hold both steps
    assert kernel == (without if batch_kernel == 0 else (without[0], without[1][:-1] + (5,)))
    # one step serves them all where most of the work is wild
    (kernel,) = D.launches([dict(s, n=8, bailout=1e4) for s in scenes], batch=True, tuning=tuning)
    assert kernel == (without if batch_kernel == 0 else (without[0], without[1][:-1] + (4,)))
    # counters are for requests that ask for them
    (counting,) = D.launches(scenes, batch=True, tuning=tuning, stats=True)
    assert counting[1][COUNT_ARG[counting[0]]] == 1


def test_only_the_launch_with_the_wild_request_changes():
    scenes = W.batch_mixed(3, 130, 5.0, 6.0)
    scenes[7].update(n=8, max_iter=100, bailout=1e4)  # costliest: in the first launch
    first, second, third = D.launches(scenes, batch=True)
    assert first[1][-1] == 5 and second == third and second[1][-1] == 1


@pytest.mark.parametrize("normal_mode", ["tetra", "analytic"])
@pytest.mark.parametrize("phong", [False, True])
@pytest.mark.parametrize("spp", [1, 4])
def test_single_wild_request(spp, phong, normal_mode):
    s = wild(640, 360, normal_mode=normal_mode)
    s["camera"]["spp"] = spp
    s = W.phong(s) if phong else s
    ban = int(normal_mode == "analytic")
    assert D.launches(s) == [("plain_kernel", (4, 2, 0, int(phong), ban, int(spp == 4)))]
    ((name, args),) = D.launches(s, stats=True)
    assert name == "plain_kernel" and args[2] == 1
    ((name, args),) = D.launches(s, tuning=dict(single_kernel=2, plain_unroll=1))
    assert name == "batch_plain_kernel" and args == (1, 0, int(phong), int(spp == 4), 4)


@pytest.mark.parametrize("n", range(2, 17))
def test_limit(n):
    limit = 1e19 ** (1.0 / n)
    for field, value in (("bailout", limit), ("bound_radius", (limit - 1.0) / 1.01)):
        for factor, general in ((0.999, False), (1.001, True)):
            s = dict(W.bulb_1080p(10, 640, 360), n=n, **{field: value * factor})
            ((name, args),) = D.launches(s)
            if field == "bound_radius" and n < 7:
                general = value * factor >= 1e3  # positions round too coarsely
            assert (args[0] == 4) == general, (field, factor)


def test_the_listings_bailout():
    # |w|^2 > 256 ends the listing's orbit: the step without special paths for every power but 16
    for n in range(2, 17):
        ((name, args),) = D.launches(dict(W.bulb_1080p(10, 640, 360), n=n, bailout=16.0))
        assert (args[0] == 4) == (n == 16)

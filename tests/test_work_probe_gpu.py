"""fr_work_probe: the rays of fr_image.stats and the distances and orbit iterations up to
the ball around the fractal, which the bench's rates and rooflines are counted in."""
import pytest

from paper_2102_01747_gb300 import workloads as W

pytestmark = pytest.mark.gpu

RAYS, DES, ORBIT = (0, 1, 6), (2, 3, 4, 7), 5


def both(scene):
    import torch
    import bench
    from paper_2102_01747_gb300 import api

    taken = bench.count_scenes(api, torch, [scene])[0]
    whole = bench.count_scenes(api, torch, [scene], to_end=True)[0]
    assert [taken[k] for k in RAYS] == [whole[k] for k in RAYS]
    assert taken[3] == whole[3]  # the hits, and with them the normals, are the same
    return taken, whole


@pytest.mark.parametrize("phong", [False, True])
@pytest.mark.parametrize("scene", [W.bulb_1080p(10, 320, 180), W.julia_256(160, 160),
                                   dict(W.bulb_1080p(4, 97, 71), normal_mode="analytic", algebraic=True, n=5),
                                   dict(W.julia_256(97, 71), p=3, normal_mode="analytic")])
def test_marches_end_at_the_ball(scene, phong):
    taken, whole = both(W.phong(scene) if phong else scene)
    assert 0 < taken[2] < whole[2] and 0 < taken[ORBIT] < whole[ORBIT]
    assert taken[4] <= whole[4] and taken[7] <= whole[7]


@pytest.mark.parametrize("change", [dict(bound_radius=20.0), dict(bound_radius=1.0), dict(eps=0.5), dict(max_steps=2)])
def test_without_a_ball_the_counts_are_the_same(change):
    for s in (W.bulb_1080p(10, 97, 71), W.julia_256(97, 71)):
        taken, whole = both(dict(s, **change))
        assert taken == whole


def test_rays_past_the_ball_take_no_distance():
    s = W.julia_256(64, 64)
    s["c"] = (0.0, 0.0, 0.0, 0.0)  # the unit ball
    s["camera"].update(target=(1.9, 0.0, 0.0), eye=(1.9, 0.0, 3.0), fov_y_deg=2.0)
    taken, whole = both(s)
    assert taken[2] == 0 and whole[2] > 0


def test_errors():
    import torch
    from paper_2102_01747_gb300 import _ffi as F
    from paper_2102_01747_gb300 import api

    c = torch.zeros(F.FR_NSTATS + 1, dtype=torch.int64, device="cuda")
    r = api.request_struct(W.julia_256(32, 32), {})
    assert F.fr_work_probe(r, None) == F.FR_EINVAL
    assert F.fr_work_probe(r, c.data_ptr() + 4) == F.FR_EINVAL
    assert F.load().fr_work_probe(None, c.data_ptr(), None) == F.FR_EINVAL
    bad = api.request_struct(dict(W.julia_256(32, 32), max_steps=0), {})
    assert F.fr_work_probe(bad, c.data_ptr()) == F.FR_EINVAL
    torch.cuda.synchronize()
    assert not c.any()

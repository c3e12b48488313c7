"""Calls that between them launch every forward kernel of the library (test_dispatch.py
counts them) at sizes where its tiles are ragged: (name, scenes, batch, tuning, stats)."""
import itertools

from paper_2102_01747_gb300 import workloads as W

# Mandelbulb images of 96, 442 and 918 tiles take 8, 4 and 2 lanes per pixel, of 1122 one;
# Julia images of 2432 tiles and less four steps per escape test
BULB_SIZES = ((61, 45), (101, 130), (201, 139), (261, 131))
JULIA_SIZES = ((97, 71), (413, 199))
WILD = 10.0 ** 22


def _bulb(size, n, normal="tetra", algebraic=False, spp=1, wild=False, phong=False):
    s = W.bulb_1080p(13 + n, *size)
    s.update(n=n, normal_mode=normal, algebraic=algebraic, max_iter=7)
    if wild:
        s["bailout"] = WILD ** (1.0 / n)
    s["camera"].update(spp=spp, seed=5, eye=(0.35, 0.8, 2.3))
    return W.phong(s) if phong else s


def _julia(size, p, normal="central", spp=1, phong=False):
    s = W.julia_256(*size)
    s.update(p=p, normal_mode=normal, plane={"n": (0.25, 0.15, 1.0), "o": 0.5})
    s["light"]["shadows"] = True
    s["camera"].update(spp=spp, seed=5)
    return W.phong(s) if phong else s


def _bulbs():
    """One-lane and spare-lane images of one and of several samples, every form of the step."""
    for n, algebraic, normal, phong in itertools.product((8, 5), (False, True), ("tetra", "analytic"), (False, True)):
        for size in BULB_SIZES if not phong else BULB_SIZES[-1:]:
            yield _bulb(size, n, normal, algebraic, phong=phong)
        yield _bulb(BULB_SIZES[0], n, normal, algebraic, 4, phong=phong)
        yield _bulb(BULB_SIZES[0], n, normal, algebraic, 3, phong=phong)
    for n, normal, phong, spp in itertools.product((8, 3), ("tetra", "analytic"), (False, True), (1, 2)):
        yield _bulb(BULB_SIZES[-1], n, normal, False, spp, True, phong)


def _julias():
    for p, normal, phong in itertools.product((2, 3), ("central", "analytic"), (False, True)):
        for size in JULIA_SIZES:
            yield _julia(size, p, normal, 1, phong)
        yield _julia(JULIA_SIZES[0], p, normal, 8, phong)


def singles(kind):
    for i, s in enumerate(_bulbs() if kind == "bulb" else _julias()):
        name = "%s%d_%dx%d_spp%d" % (kind, i, s["camera"]["width"], s["camera"]["height"], s["camera"]["spp"])
        for t in (dict(), dict(plain_unroll=4), dict(sample_lanes=0), dict(sample_lanes=0, plain_unroll=4),
                  dict(single_kernel=2), dict(single_kernel=2, plain_unroll=2)):
            yield name, [s], False, t, False
        yield name, [s], False, dict(), True
        yield name, [s], False, dict(single_kernel=2), True
    for i, s in enumerate((_bulb(BULB_SIZES[0], 8), _julia(JULIA_SIZES[0], 2)) if kind == "julia" else ()):
        for k, phong, stats in itertools.product((1, 2, 4, 8), (False, True), (False, True)):
            yield "lanes%d" % i, [W.phong(s) if phong else s], False, dict(single_kernel=1, persist_unroll=k), stats


def batches():
    for spp, phong, wild, stats in itertools.product((1, 4), (False, True), (0, 1, 2), (False, True)):
        small = (45, 29)
        scenes = [_julia(JULIA_SIZES[0], 2, spp=spp, phong=phong), _bulb(BULB_SIZES[0], 8, wild=wild == 2),
                  _bulb(small, 5, "analytic", wild=wild > 0), _julia(small, 3, "analytic"),
                  _bulb((70, 44), 3, algebraic=True, spp=spp, wild=wild == 2, phong=phong)]
        name = "batch_spp%d%s_wild%d" % (spp, "_phong" * phong, wild)
        for t in (dict(batch_kernel=2, plain_unroll=1), dict(batch_kernel=2, plain_unroll=2),
                  dict(batch_kernel=1, plain_unroll=1), dict(batch_kernel=1, plain_unroll=2),
                  *(dict(batch_kernel=0, persist_unroll=k) for k in (1, 2, 4, 8))):
            yield name, scenes, True, t, stats


GROUPS = {"bulb": lambda: singles("bulb"), "julia": lambda: singles("julia"), "batch": batches}

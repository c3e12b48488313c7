"""The ball that lets marches end early, on the host: its bound lies below every distance
estimate outside, and finding it costs a call little."""
import os
import subprocess
import tempfile
import time

from paper_2102_01747_gb300 import _ffi as F
from paper_2102_01747_gb300 import api
from paper_2102_01747_gb300 import build as B
from paper_2102_01747_gb300 import workloads as W

import dispatch as D

HERE = os.path.dirname(os.path.abspath(__file__))


def test_bound_below_the_distance_estimates():
    B.build()
    D.load()
    objs = [os.path.join(B.BUILD, os.path.basename(s)[:-3] + ".o") for s in B._sources()]
    objs = [o for o in objs if os.path.basename(o) != "fr_api.o"]  # the test includes it
    inc = os.path.join(os.path.dirname(os.path.dirname(B.nvcc())), "include")
    with tempfile.TemporaryDirectory() as d:
        obj, exe = os.path.join(d, "t.o"), os.path.join(d, "t")
        subprocess.run([B.nvcc(), "-O2", "-std=c++17", *B.ARCH, "-I", B.CSRC, "-c",
                        os.path.join(HERE, "exit_bound", "exit_bound.cu"), "-o", obj], check=True)
        subprocess.run(["g++", "-O1", "-std=c++17", "-I", inc, "-o", exe, obj,
                        os.path.join(HERE, "fake_cudart", "fake_cudart.cpp"), *objs], check=True)
        out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=300).stdout.split()
    points, balls, worst = int(out[0]), int(out[1]), float(out[2])
    assert points > 100000 and balls > 2000
    # the bound has a slack of 1e-4 per step; the estimate is rounded in double
    assert 1.0 <= worst < 1.1, worst


def _host_us(scene, n=64):
    """Host time per request of a batch call, best of many."""
    lib = D.load()
    arr = (F.fr_request * n)()
    for r in arr:
        r.kind = F.FR_KIND_JULIA if scene["kind"] == "julia" else F.FR_KIND_BULB
        prm, r.plane, r.camera, r.light = api.scene_structs(scene)
        setattr(r, "julia" if scene["kind"] == "julia" else "bulb", prm)
        r.out = D._fake(scene, rgba8=True)
    best = 1e9
    for _ in range(200):
        t = time.perf_counter()
        st = lib.fr_render_batch(arr, n, 1 << 20, 256, None)
        best = min(best, time.perf_counter() - t)
        assert st == F.FR_OK
    return best / n * 1e6


def test_host_time_of_finding_the_ball():
    # against the same requests in a bounding sphere too large for a ball; with a logarithm
    # per orbit step the Mandelbulb took 6 times as long
    for s in (W.julia_256(), W.bulb_1080p()):
        assert _host_us(s) < 5.0 * _host_us(dict(s, bound_radius=20.0))

"""Which kernels a call launches, found out without a GPU: libfr's objects linked
with a stand-in for the CUDA runtime (fake_cudart/) that records launches.

A kernel is (name, template arguments), e.g. ("plain_kernel", (3, 2, 0, 0, 0, 0))."""
import ctypes
import os
import re
import subprocess

from paper_2102_01747_gb300 import _ffi as F
from paper_2102_01747_gb300 import api
from paper_2102_01747_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
LIB = os.path.join(B.BUILD, "libfr_dispatch.so")

_lib = None


def load():
    global _lib
    if _lib is None:
        B.build()
        objs = [os.path.join(B.BUILD, os.path.basename(s)[:-3] + ".o") for s in B._sources()]
        if not all(os.path.exists(o) for o in objs):
            B.build(force=True)
        src = os.path.join(HERE, "fake_cudart", "fake_cudart.cpp")
        if not os.path.exists(LIB) or any(os.path.getmtime(p) > os.path.getmtime(LIB) for p in objs + [src]):
            inc = os.path.join(os.path.dirname(os.path.dirname(B.nvcc())), "include")
            tmp = LIB + ".tmp%d" % os.getpid()
            subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-fvisibility=hidden", "-I", inc, "-shared",
                            "-Wl,-Bsymbolic", "-o", tmp, src, *objs], check=True, capture_output=True, text=True)
            os.replace(tmp, LIB)
        lib = ctypes.CDLL(LIB, mode=os.RTLD_LOCAL | os.RTLD_NOW)
        for name, (res, args) in F.SIGNATURES.items():
            fn = getattr(lib, name)
            fn.restype, fn.argtypes = res, args
        lib.fake_launches.restype = lib.fake_kernels.restype = ctypes.c_char_p
        lib.fake_launches.argtypes = [ctypes.c_int]
        _lib = lib
    return _lib


def parse(mangled: str):
    """_ZN2fr12plain_kernelILi3ELi2ELb0E...EEv... -> ("plain_kernel", (3, 2, 0, ...))"""
    nested = mangled.startswith("_ZN")
    rest, name = mangled[3 if nested else 2:], ""
    while rest[0].isdigit():  # length-prefixed names, the last one the kernel's
        n = re.match(r"\d+", rest).group()
        name, rest = rest[len(n):len(n) + int(n)], rest[len(n) + int(n):]
        if not nested:
            break
    args = re.match(r"I((?:L[ib]\d+E)+)E", rest)
    return name, tuple(int(v) for v in re.findall(r"L[ib](\d+)E", args.group(1))) if args else ()


def kernels():
    """Every kernel the library holds."""
    return sorted({parse(k) for k in load().fake_kernels().decode().split()})


def _fake(scene, **want):
    """Output pointers that no one follows (a render's images, or a count's counters)."""
    img = F.fr_image()
    for name in ("rgba8", "rgba", "depth", "saved", "stats", "trap"):
        if want.get(name):
            setattr(img, name, 1 << 20)
    return img


def launches(scenes, batch=False, tuning=None, shapes=False, **want):
    """Kernels of one call on `scenes` (a scene, or a list of them for fr_render_batch) with
    the tuning's fields replaced by `tuning`: a list of (name, template arguments), with `shapes` also
    (..., CTAs, threads per CTA)."""
    lib = load()
    want = want or dict(rgba8=True, depth=True)
    keep = F.fr_tuning()
    assert lib.fr_get_tuning(ctypes.byref(keep)) == F.FR_OK
    t = F.fr_tuning(*[(tuning or {}).get(n, getattr(keep, n)) for n, _ in F.fr_tuning._fields_])
    assert lib.fr_set_tuning(ctypes.byref(t)) == F.FR_OK
    lib.fake_launches(1)
    try:
        if batch:
            arr = (F.fr_request * len(scenes))()
            for i, s in enumerate(scenes):
                r = arr[i]
                r.kind = F.FR_KIND_JULIA if s["kind"] == "julia" else F.FR_KIND_BULB
                prm, r.plane, r.camera, r.light = api.scene_structs(s)
                setattr(r, "julia" if s["kind"] == "julia" else "bulb", prm)
                r.out = _fake(s, **want)
            st = lib.fr_render_batch(arr, len(scenes), 1 << 20, lib.fr_batch_workspace_bytes(len(scenes)), None)
        else:
            s = scenes
            call = lib.fr_render_julia if s["kind"] == "julia" else lib.fr_render_mandelbulb
            st = call(*[ctypes.byref(v) for v in api.scene_structs(s)], ctypes.byref(_fake(s, **want)), None)
        assert st == F.FR_OK, lib.fr_last_error()
    finally:
        lib.fr_set_tuning(ctypes.byref(keep))
    lines = [line.split() for line in lib.fake_launches(1).decode().splitlines()]
    return [(*parse(k), int(g), int(b)) if shapes else parse(k) for k, g, b in lines]

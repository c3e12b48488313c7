"""The renders and gradients that this framework is timed on.

Every case goes through a public entry point (api.render, api.render_batch,
autograd.julia_render, autograd.bulb_render) the way an interactive viewer, an
animation, a render server or a fitting loop calls it: the scene is a dict, the
output buffers are allocated once and reused from frame to frame, the tuning is
the default one.  Scenes are those of the package's workloads module; a seed
moves the camera along its orbit and, for the Julia set, moves c, as successive
frames and requests do.

exact() renders the same scenes in double precision with plain torch.  It does
not for batches, whose images are those of the single renders: one by one they
would take too long.
"""
import copy
import math

import numpy as np
import torch

from paper_2102_01747_gb300 import api, autograd
from paper_2102_01747_gb300 import workloads as W

# Mean orbit iterations per camera sample that the scenes take (from counted
# renders) and the listings' operations per iteration.
ITERS = {"julia": 120.0, "bulb": 25.0}
OPS = {("julia", 2): 24.0, ("julia", 3): 28.0, "bulb": 29.0}


def listed():
    return [
        # the smallest calls: a 256 x 256 preview of the Julia set (bound by latency, not by the
        # number of rays) and a thumbnail of the Mandelbulb
        {"name": "julia_256", "kind": "julia", "width": 256, "height": 256},
        {"name": "bulb_160x90", "kind": "bulb", "width": 160, "height": 90},
        # one frame of an interactive view at full HD: Lambert with a shadow ray, the paper's
        # closest-hit model (Phong and a mirror ray), and the power without transcendental calls
        {"name": "bulb_1080p", "kind": "bulb", "width": 1920, "height": 1080},
        {"name": "bulb_1080p_phong", "kind": "bulb", "width": 1920, "height": 1080, "phong": True},
        {"name": "bulb_1080p_algebraic", "kind": "bulb", "width": 1920, "height": 1080, "algebraic": True},
        # odd sizes and the other options: another power with the analytic normal, float colours and
        # orbit traps (recolouring a render afterwards); the listing's cube with a cut plane
        {"name": "bulb_n5_1283x723", "kind": "bulb", "width": 1283, "height": 723, "power": 5,
         "normal": "analytic", "extras": True},
        {"name": "julia3_1001x667", "kind": "julia", "width": 1001, "height": 667, "power": 3,
         "normal": "tetra", "shadows": True, "cut": True, "extras": True},
        # large frames: 4K Julia with shadow rays, 4K Mandelbulb with four jittered samples
        {"name": "julia_4k", "kind": "julia", "width": 3840, "height": 2160, "shadows": True},
        {"name": "bulb_4k_spp4", "kind": "bulb", "width": 3840, "height": 2160, "spp": 4},
        # a render server's queue in one call: 64 requests with sides 128..2048, and 64 thumbnails
        {"name": "batch_mixed", "kind": "batch", "requests": 64, "min_log2": 7.0, "max_log2": 11.0},
        {"name": "batch_small", "kind": "batch", "requests": 64, "min_log2": 5.0, "max_log2": 8.0},
        # one step of fitting c, the cut plane and the light to a target image: forward and adjoint
        {"name": "grad_julia_512", "kind": "grad_julia", "width": 512, "height": 512},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["julia", "julia", "bulb", "bulb", "bulb", "batch", "batch", "grad_julia", "grad_bulb"])
    if kind == "batch":
        lo = rng.uniform(5.0, 8.0)
        return {"kind": "batch", "requests": _log(rng, 2, 64), "min_log2": round(lo, 3),
                "max_log2": round(rng.uniform(lo + 1.0, 10.5), 3)}
    if kind.startswith("grad"):
        return {"kind": kind, "width": _log(rng, 64, 1024), "height": _log(rng, 64, 1024),
                "normal": rng.choice(["central", "tetra", "analytic"])}
    case = {"kind": kind, "width": _log(rng, 64, 3840), "height": _log(rng, 48, 2160),
            "normal": rng.choice(["tetra", "central", "analytic"]), "shadows": rng.random() < 0.6,
            "cut": rng.random() < 0.6, "phong": rng.random() < 0.25, "extras": rng.random() < 0.25,
            "spp": rng.choice([1, 1, 1, 2, 3, 4, 8])}
    while case["width"] * case["height"] * case["spp"] > 30_000_000:
        case["spp"] = 1 if case["spp"] == 1 else case["spp"] - 1
    if kind == "julia":
        case["power"] = rng.choice([2, 2, 3])
    else:
        case["power"] = rng.choice([8, 8, 2, 3, 4, 5, 6, 7, 9, 10])
        case["algebraic"] = rng.random() < 0.25
    return case


def _scene(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    kind = case["kind"].replace("grad_", "")
    w, h = case["width"], case["height"]
    azimuth = float(rng.uniform(0.0, 360.0))
    if kind == "julia":
        s = W.julia_256(w, h)
        if case["kind"] == "grad_julia":
            s, _ = W.diff_julia(seed, w, h)
        else:
            s["c"] = tuple(float(v) for v in np.array(s["c"]) + 0.05 * rng.standard_normal(4))
            s["camera"].update(eye=W.orbit_eye(3.0, azimuth, 20.0, 1.0))
        s["p"] = case.get("power", 2)
        if s["p"] == 3:
            s["escape_r2"] = 256.0  # as in the listing
        if case.get("cut"):
            s["plane"] = {"n": (0.25, 0.15, 1.0), "o": 0.5}
        s["light"]["shadows"] = case.get("shadows", False)
    else:
        s = W.bulb_1080p(0, w, h)
        s["camera"].update(eye=W.orbit_eye(2.5, azimuth, 20.0, 1.0))
        s["n"] = case.get("power", 8)
        s["algebraic"] = case.get("algebraic", False)
        s["light"]["shadows"] = case.get("shadows", True)
        if not case.get("cut", True):
            s["plane"] = None
    s["normal_mode"] = case.get("normal", s["normal_mode"])
    if case.get("phong"):
        s = W.phong(s)
    s["camera"].update(spp=case.get("spp", 1), seed=seed & 0xFFFF)
    return s


def _batch_scenes(case, seed):
    # a queue of fixed image sizes whose scenes change
    sized = W.batch_mixed(W.BASE_SEED, case["requests"], case["min_log2"], case["max_log2"])
    scenes = W.batch_mixed(seed, case["requests"], case["min_log2"], case["max_log2"])
    return [W.resized(s, z["camera"]["width"], z["camera"]["height"]) for s, z in zip(scenes, sized)]


def prepare(case, seed):
    if case["kind"] == "batch":
        scenes = _batch_scenes(case, seed)
        sizes = [s["camera"]["width"] * s["camera"]["height"] for s in scenes]
        # one buffer for all images, as a server's output arena (sides are multiples of 8)
        rgba8 = torch.zeros(sum(sizes), dtype=torch.int32, device="cuda")
        depth = torch.zeros(sum(sizes), dtype=torch.float32, device="cuda")
        outs, at = [], 0
        for s, n in zip(scenes, sizes):
            shape = (s["camera"]["height"], s["camera"]["width"])
            outs.append({"rgba8": rgba8[at:at + n].view(shape), "depth": depth[at:at + n].view(shape)})
            at += n
        return {"scenes": scenes, "outs": outs, "ws": api.workspace(len(scenes)), "rgba8": rgba8, "depth": depth}
    scene = _scene(case, seed)
    if not case["kind"].startswith("grad"):
        extras = case.get("extras", False)
        return {"scene": scene, "out": api.alloc_image(scene, rgba=extras, trap=extras)}
    # a fitting step: the parameters of the step before, the image to be reached
    target = api.render(scene, rgba8=False, rgba=True, depth=True)
    leaf = lambda v: torch.tensor(v, requires_grad=True)  # noqa: E731
    moved = copy.deepcopy(scene)
    if case["kind"] == "grad_julia":
        _, moved["c"] = W.diff_julia(seed, case["width"], case["height"])
    params = {"plane_n": leaf([0.05 + v for v in moved["plane"]["n"]]), "plane_o": leaf([moved["plane"]["o"]]),
              "light": leaf([v + 0.1 * k for k, v in enumerate(moved["light"]["dir"])])}
    if case["kind"] == "grad_julia":
        params["c"] = leaf(list(moved["c"]))
    return {"scene": moved, "target": target, "params": params}


def _loss(rgba, depth, target):
    """L2 of the colours, and of the depths where both images show the surface."""
    both = depth.isfinite() & target["depth"].isfinite()
    off = torch.where(both, depth, 0.0) - torch.where(both, target["depth"], 0.0)
    return (rgba - target["rgba"]).square().sum() + off.square().sum()


def run(state):
    if "scenes" in state:
        api.render_batch(state["scenes"], state["outs"], state["ws"])
        return {"rgba8": state["rgba8"], "depth": state["depth"]}
    if "out" in state:
        return api.render(state["scene"], state["out"])
    p = state["params"]
    if "c" in p:
        rgba, depth = autograd.julia_render(state["scene"], p["c"], p["plane_n"], p["plane_o"], p["light"])
    else:
        rgba, depth = autograd.bulb_render(state["scene"], p["plane_n"], p["plane_o"], p["light"])
    loss = _loss(rgba, depth, state["target"])
    names = sorted(p)
    grads = torch.autograd.grad(loss, [p[k] for k in names])
    return {"rgba": rgba.detach(), "depth": depth.detach(), "grad": dict(zip(names, grads))}


def work(case):
    if case["kind"] == "batch":
        scenes = _batch_scenes(case, 0)
        ops = {"julia": OPS["julia", 2], "bulb": OPS["bulb"]}
        flops = sum(W.total_pixels([s]) * ITERS[s["kind"]] * ops[s["kind"]] for s in scenes)
        return {"bytes": 8.0 * W.total_pixels(scenes), "flops": flops}
    pixels = case["width"] * case["height"]
    kind = case["kind"].replace("grad_", "")
    ops = OPS["bulb"] if kind == "bulb" else OPS["julia", case.get("power", 2)]
    flops = pixels * case.get("spp", 1) * ITERS[kind] * ops
    if case["kind"].startswith("grad"):
        # colour, depth and hit written, the target and the cotangents written and read, the hit read
        return {"bytes": 112.0 * pixels, "flops": 1.5 * flops}
    return {"bytes": (40.0 if case.get("extras") else 8.0) * pixels, "flops": flops}


# ---------------------------------------------------------------- double precision
# The listings' arithmetic in float64 on whole images: rays that are done are
# taken out of the arrays between steps.

def _normalize(v):
    return v / v.norm(dim=-1, keepdim=True)


def _vec(v):
    return torch.tensor([float(x) for x in v], dtype=torch.float64, device="cuda")


def _julia_step(s, z, c):
    v2 = z[..., 1:].square().sum(-1)
    a = z[..., 0]
    if s["p"] == 2:
        head, f = a * a - v2, 2 * a
    else:
        head, f = a * (a * a - 3 * v2), 3 * a * a - v2
    return torch.cat([head[..., None], f[..., None] * z[..., 1:]], -1) + c


def _bulb_step(s, w, c):
    n = s["n"]
    r = w.norm(dim=-1)
    b = n * torch.acos((w[..., 1] / r).clamp(-1, 1))
    a = n * torch.atan2(w[..., 0], w[..., 2])
    p = torch.stack([b.sin() * a.sin(), b.cos(), b.sin() * a.cos()], -1) * (r ** n)[..., None]
    return torch.where((r > 0)[..., None], p, torch.zeros_like(p)) + c


def _julia_start(s, x):
    return torch.cat([x, torch.full_like(x[..., :1], s["slice_w"])], -1)


def _escape(s):
    return s["escape_r2"] if s["kind"] == "julia" else s["bailout"] ** 2


def _de(s, x):
    julia = s["kind"] == "julia"
    z = _julia_start(s, x) if julia else x
    c = _vec(s["c"]) if julia else x
    m, dz = z.square().sum(-1), torch.ones_like(x[..., 0])
    m_end, dz_end = torch.empty_like(m), torch.empty_like(m)
    at = torch.arange(len(x), device=x.device)
    for k in range(s["max_iter"]):
        if julia:
            dz = dz * s["p"] ** 2 * m ** (s["p"] - 1)
            z = _julia_step(s, z, c)
        else:
            dz = s["n"] * m ** (0.5 * (s["n"] - 1)) * dz + 1
            z = _bulb_step(s, z, c)
        m = z.square().sum(-1)
        m_end[at], dz_end[at] = m, dz
        on = (m <= _escape(s)).nonzero()[:, 0]
        if not len(on):
            break
        at, z, m, dz = at[on], z[on], m[on], dz[on]
        c = c if julia else c[on]
    if julia:
        return 0.25 * m_end.log() * (m_end / dz_end).sqrt()
    return 0.25 * m_end.log() * m_end.sqrt() / dz_end


def _interval(s, ro, rd):
    b = (ro * rd).sum(-1)
    disc = b * b - ((ro * ro).sum(-1) - s["bound_radius"] ** 2)
    ok = disc >= 0
    root = disc.clamp(min=0).sqrt()
    t0, t1 = (-b - root).clamp(min=s["eps"]), (-b + root).clamp(max=7000.0)
    face = torch.zeros_like(ok)
    if s["plane"]:
        n = _vec(s["plane"]["n"])
        a, bb = (ro * n).sum(-1) - s["plane"]["o"], (rd * n).sum(-1)
        ts = -a / bb
        t1 = torch.where(bb > 0, torch.minimum(t1, ts), t1)
        face = (bb < 0) & (ts > t0)
        t0 = torch.where(face, ts, t0)
        ok &= ~((bb == 0) & (a > 0))
    return ok & (t0 <= t1), t0, t1, face


def _march(s, ro, rd):
    """(hit, t, whether the hit is on the cut face) of rays that may miss the bounding sphere."""
    hit, t0, t1, face = _interval(s, ro, rd)
    t_end, first = t0.clone(), torch.zeros_like(hit)
    at = hit.nonzero()[:, 0]
    t, t1, ro, rd = t0[at], t1[at], ro[at], rd[at]
    for k in range(s["max_steps"]):
        if not len(at):
            break
        d = _de(s, ro + t[:, None] * rd)
        on = ~(d < s["eps"])
        t = torch.where(on, t + torch.where(d < s["max_step"], d, s["max_step"]), t)
        t_end[at] = t
        out = on & (t > t1)
        hit[at[out]] = False
        if k == 0:
            first[at[~on]] = True
        go = (on & ~out).nonzero()[:, 0]
        at, t, t1, ro, rd = at[go], t[go], t1[go], ro[go], rd[go]
    return hit, t_end, hit & first & face


def _taps(s):
    h = s["normal_h"] or (0.5773 * s["eps"] if s["normal_mode"] == "tetra" else 1e-4)
    if s["normal_mode"] == "tetra":
        e = _vec([1, -1, -1, -1, -1, 1, -1, 1, -1, 1, 1, 1]).view(4, 3)
        return [(h * v, h * v) for v in e]
    e = torch.eye(3, dtype=torch.float64, device="cuda")
    return [(sign * h * v, sign * v) for v in e for sign in (1, -1)]


def _gradient_direction(s, x, c):
    """J^T z_N of the orbit at x (the analytic normal's gradient), differentiable in x and c."""
    x = x if x.requires_grad else x.detach().requires_grad_()
    with torch.enable_grad():
        julia = s["kind"] == "julia"
        z = _julia_start(s, x) if julia else x
        on = torch.ones_like(x[..., 0], dtype=torch.bool)
        for _ in range(s["max_iter"]):
            z = torch.where(on[..., None], _julia_step(s, z, c) if julia else _bulb_step(s, z, x), z)
            on = on & (z.detach().square().sum(-1) <= _escape(s))
        half = 0.5 * z.square().sum(-1)
        return torch.autograd.grad(half.sum(), x, create_graph=True)[0]


def _normal(s, x, rd):
    if s["normal_mode"] == "analytic":
        c = _vec(s["c"]) if s["kind"] == "julia" else None
        g = torch.cat([_gradient_direction(s, p, c).detach() for p in x.split(1 << 21)]) if len(x) else x
    else:
        g = sum(w * _de(s, x + o)[:, None] for o, w in _taps(s))
    length = g.norm(dim=-1, keepdim=True)
    ok = (length > 0) & length.isfinite()
    return torch.where(ok, g / torch.where(ok, length, 1.0), -rd)


def _phong(s, n, d, vis):
    li = s["light"]
    L, albedo = _normalize(_vec(li["dir"])), _vec(li["albedo"])
    ndl = (n * L).sum(-1)
    k = li["k_ambient"] + li["k_diffuse"] * ndl.clamp(min=0) * vis
    rv = -((2 * ndl[:, None] * n - L) * d).sum(-1)
    spec = torch.where(ndl > 0, rv.clamp(min=0) ** li.get("shininess", 1.0), torch.zeros_like(rv))
    return albedo * k[:, None] + (li.get("k_specular", 0.0) * spec * vis)[:, None]


def _trace(s, ro, rd):
    """Colour (N, 4), depth (N) of camera rays."""
    li = s["light"]
    L, albedo, bg = _normalize(_vec(li["dir"])), _vec(li["albedo"]), _vec(li["background"])
    phong = li.get("shading") == "phong"
    flat = _normalize(_vec(s["plane"]["n"])) if s["plane"] else None

    def hits(ro, rd):
        hit, t, face = _march(s, ro, rd)
        at = hit.nonzero()[:, 0]
        x = ro[at] + t[at][:, None] * rd[at]
        face = face[at]
        n = torch.empty_like(x)
        n[face] = flat if flat is not None else 0.0
        n[~face] = _normal(s, x[~face], rd[at][~face])
        return at, x, n, t[at]

    at, x, n, t = hits(ro, rd)
    rgba, depth = bg.repeat(len(ro), 1), torch.full_like(ro[:, 0], math.inf)
    depth[at] = t
    vis = torch.ones_like(t)
    start = x + 4 * s["eps"] * n
    if li["shadows"]:
        vis = 1.0 - _march(s, start, L.expand_as(start).contiguous())[0].double()
    if phong:
        d = rd[at]
        rr = d - 2 * (n * d).sum(-1, keepdim=True) * n
        seen = bg[:3].repeat(len(x), 1)
        at2, _, n2, _ = hits(start, rr)
        seen[at2] = _phong(s, n2, rr[at2], torch.ones_like(n2[:, 0]))
        u = 1 - (-(n * d).sum(-1)).clamp(min=0)
        fresnel = albedo + (1 - albedo) * (u ** 5)[:, None]
        col = _phong(s, n, d, vis) + li["reflect_coef"] * fresnel * seen
    else:
        k = li["k_ambient"] + li["k_diffuse"] * (n * L).sum(-1).clamp(min=0) * vis
        col = albedo * k[:, None]
    rgba[at] = torch.cat([col, torch.ones_like(col[:, :1])], -1)
    return rgba, depth


def _rays(s, sample):
    cam = s["camera"]
    w, h, spp = cam["width"], cam["height"], cam["spp"]
    px = np.arange(w * h, dtype=np.uint64)
    sx = sy = 0.5
    if spp > 1:  # splitmix64 of (seed << 40) + pixel * spp + sample
        z = (np.uint64(cam["seed"]) << np.uint64(40)) + px * np.uint64(spp) + np.uint64(sample)
        z = z + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
        sx = torch.from_numpy((z >> np.uint64(40)).astype(np.float64) / 2 ** 24).cuda()
        sy = torch.from_numpy(((z >> np.uint64(16)) & np.uint64(0xFFFFFF)).astype(np.float64) / 2 ** 24).cuda()
    at = torch.arange(w * h, device="cuda")
    th = math.tan(math.radians(cam["fov_y_deg"]) / 2)
    ax = (2 * ((at % w).double() + sx) / w - 1) * th * w / h
    ay = (1 - 2 * ((at // w).double() + sy) / h) * th
    eye = _vec(cam["eye"])
    fwd = _normalize(_vec(cam["target"]) - eye)
    right = _normalize(torch.linalg.cross(fwd, _vec(cam["up"])))
    up = torch.linalg.cross(right, fwd)
    return eye.expand(w * h, 3), _normalize(fwd + ax[:, None] * right + ay[:, None] * up)


def _image(s):
    cam = s["camera"]
    rgba, depth = 0.0, None
    for k in range(cam["spp"]):
        c, d = _trace(s, *_rays(s, k))
        rgba = rgba + c
        depth = d if depth is None else torch.minimum(depth, d)
    return (rgba / cam["spp"]).view(cam["height"], cam["width"], 4), depth.view(cam["height"], cam["width"])


def _diff_de(s, x, c):
    """The Julia distance, differentiable in x and c (escape counts held fixed)."""
    z, dz = _julia_start(s, x), torch.ones_like(x[..., 0])
    m = z.square().sum(-1)
    on = torch.ones_like(dz, dtype=torch.bool)
    for _ in range(s["max_iter"]):
        dz = torch.where(on, dz * s["p"] ** 2 * m ** (s["p"] - 1), dz)
        z = torch.where(on[..., None], _julia_step(s, z, c), z)
        m = z.square().sum(-1)
        on = on & (m.detach() <= _escape(s))
    return 0.25 * m.log() * (m / dz).sqrt()


def _gradient(case, state):
    """The fitting step by implicit differentiation: at a surface hit the depth moves along the ray as
    the level set of the distance does, at a cut-face hit with the plane."""
    p = {k: v.detach().double().cuda().requires_grad_() for k, v in state["params"].items()}
    s = copy.deepcopy(state["scene"])
    s["plane"] = {"n": p["plane_n"].tolist(), "o": float(p["plane_o"].item())}
    s["light"]["dir"] = p["light"].tolist()
    s["c"] = p["c"].tolist() if "c" in p else s["c"]
    li = s["light"]
    ro, rd = _rays(s, 0)
    hit, t, face = _march(s, ro, rd)
    rgba, depth = _vec(li["background"]).repeat(len(ro), 1), torch.full_like(t, math.inf)
    cut = face.nonzero()[:, 0]
    at = (hit & ~face).nonzero()[:, 0]
    x0 = ro[at] + t[at][:, None] * rd[at]
    n0 = _normal(s, x0, rd[at])
    with torch.enable_grad():
        if "c" in p:
            xg = x0.clone().requires_grad_()
            (slope,) = torch.autograd.grad(_diff_de(s, xg, p["c"].detach()).sum(), xg)
            d0 = _diff_de(s, x0, p["c"])
            ts = t[at] - (d0 - d0.detach()) / (slope * rd[at]).sum(-1)
            x = ro[at] + ts[:, None] * rd[at]
            if s["normal_mode"] == "analytic":
                g = _gradient_direction(s, x, p["c"])
            else:
                g = sum(w * _diff_de(s, x + o, p["c"])[:, None] for o, w in _taps(s))
            n_surface = _normalize(g)
        else:
            ts, n_surface = t[at], n0
        tc = (p["plane_o"] - (ro[cut] * p["plane_n"]).sum(-1)) / (rd[cut] * p["plane_n"]).sum(-1)
        n = torch.cat([n_surface, _normalize(p["plane_n"]).expand(len(cut), 3)])
        every = torch.cat([at, cut])
        vis = torch.ones_like(t[every])
        if li["shadows"]:
            start = torch.cat([x0, ro[cut] + t[cut][:, None] * rd[cut]]) + 4 * s["eps"] * n.detach()
            vis = 1.0 - _march(s, start, _normalize(_vec(li["dir"])).expand_as(start).contiguous())[0].double()
        k = li["k_ambient"] + li["k_diffuse"] * (n * _normalize(p["light"])).sum(-1).clamp(min=0) * vis
        col = torch.cat([_vec(li["albedo"]) * k[:, None], torch.ones_like(k)[:, None]], -1)
        rgba = rgba.index_copy(0, every, col)
        depth = depth.index_copy(0, every, torch.cat([ts, tc]))
        h, w = s["camera"]["height"], s["camera"]["width"]
        rgba, depth = rgba.view(h, w, 4), depth.view(h, w)
        loss = _loss(rgba, depth, {k: v.double() for k, v in state["target"].items()})
        names = sorted(p)
        grads = torch.autograd.grad(loss, [p[k] for k in names])
    return {"rgba": rgba.detach(), "depth": depth.detach(), "grad": {k: g.cpu() for k, g in zip(names, grads)}}


def exact(case, seed):
    if case["kind"] == "batch":
        return None
    if case["kind"].startswith("grad"):
        return _gradient(case, prepare(case, seed))
    with torch.no_grad():
        rgba, depth = _image(_scene(case, seed))
    out = {"rgba8": None, "depth": depth}
    if case.get("extras"):
        out.update(rgba=rgba, trap=None)
    return out

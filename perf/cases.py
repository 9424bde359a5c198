"""The renders, training steps and queries that programs ask of this package, as measured cases.

A case names a scene recipe of paper_2605_27323_gb300.scenes with its size, and the call made on it.
listed() holds the fixed ones, draw() gives more of the same ranges, prepare() builds the scene and what
the program holds beside it, run() makes one call through the public API and returns all it computes, and
exact() computes the same in 64 bits where a brute-force evaluation takes seconds (the box renders and the
ray queries).
"""
import math

import numpy as np
import torch

import paper_2605_27323_gb300 as pt
from paper_2605_27323_gb300 import scenes


def listed():
    return [
        # The first frame of a preview or a thumbnail: few pixels, one sample, a scene of 36 triangles.  Only
        # launches and latency count.
        {"name": "preview_box", "call": "render", "scene": "box", "width": 61, "height": 47, "spp": 1, "depth": 4},
        # The tiny box at its configured size: 128 x 128, 16 samples, paths of up to 8 vertices.
        {"name": "box_128", "call": "render", "scene": "box", "width": 128, "height": 128, "spp": 16, "depth": 8},
        # The frame that the benchmark is quoted on: 1.15 M triangles, 1920 x 1080, 1 sample, depth 5.
        {"name": "frame_1080p", "call": "render", "scene": "spheres", "spheres": 200, "level": 4, "ground": 256,
         "width": 1920, "height": 1080, "spp": 1, "depth": 5},
        # The other integrator of the same benchmark step.
        {"name": "megakernel_1080p", "call": "render", "scene": "spheres", "spheres": 200, "level": 4, "ground": 256,
         "width": 1920, "height": 1080, "spp": 1, "depth": 5, "mode": "megakernel"},
        # Long paths with multiple importance sampling on a ragged image: the deep, sparse bounces.
        {"name": "deep_mis_ragged", "call": "render", "scene": "spheres", "spheres": 150, "level": 3, "ground": 128,
         "width": 1277, "height": 717, "spp": 2, "depth": 16, "mis": True},
        # A heightfield with small spheres on it, four samples, depth 8: the largest render.
        {"name": "terrain_1440p", "call": "render", "scene": "terrain", "grid": 640, "spheres": 800, "level": 2,
         "width": 2560, "height": 1440, "spp": 3, "depth": 8},
        # The benchmark's scene as a two-level scene: one sphere mesh placed 200 times.
        {"name": "instanced_1080p", "call": "render", "scene": "instanced", "spheres": 200, "level": 4, "ground": 256,
         "width": 1920, "height": 1080, "spp": 1, "depth": 5},
        # A viewer that refines its view: four frames of one sample added to running sums, Halton jitter.
        {"name": "progressive_720p", "call": "progressive", "scene": "spheres", "spheres": 60, "level": 3, "ground": 96,
         "width": 1280, "height": 720, "frames": 4, "spp": 1, "depth": 5, "halton": True},
        # A step of inverse rendering: image, then gradients of a loss by every albedo and emission.
        {"name": "train_512", "call": "train", "scene": "diff", "spheres": 100, "level": 3, "ground": 128,
         "width": 512, "height": 512, "spp": 16, "depth": 6},
        # The gradient pass alone at the benchmark's size, as its step times it.
        {"name": "backward_1080p", "call": "backward", "scene": "spheres", "spheres": 200, "level": 4, "ground": 256,
         "width": 1920, "height": 1080, "spp": 1, "depth": 5},
        # Many small views in one call: 12 scenes of 1 k to 60 k triangles.
        {"name": "batch_12", "call": "batch", "scene": "batch", "scenes": 12, "max_tris": 60000, "width": 256, "height": 192,
         "spp": 4, "depth": 5},
        # A program that asks for closest hits of its own rays (picking, ambient occlusion, baking).
        {"name": "query_1m", "call": "query", "scene": "spheres", "spheres": 30, "level": 3, "ground": 48, "rays": 1000003},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["render", "render", "render", "progressive", "train", "backward", "batch", "query"])
    if call == "query":
        return {"call": "query", "scene": "spheres", "spheres": rng.randint(1, 60), "level": rng.randint(1, 3),
                "ground": rng.randint(4, 96), "rays": _log_int(rng, 3, 2000000)}
    if call == "batch":
        return {"call": "batch", "scene": "batch", "scenes": rng.randint(2, 20), "max_tris": _log_int(rng, 2000, 80000),
                "width": _log_int(rng, 17, 512), "height": _log_int(rng, 17, 384), "spp": rng.choice([1, 3, 4, 8]),
                "depth": rng.randint(1, 8)}
    width = _log_int(rng, 33, 1920)
    height = max(1, int(width * rng.uniform(0.4, 1.0)))
    spp = rng.choice([1, 1, 2, 3, 4, 8, 16])
    while width * height * spp > 6000000:
        spp = max(1, spp // 2)
    case = {"call": call, "width": width, "height": height, "spp": spp, "depth": rng.choice([1, 2, 3, 5, 5, 6, 8, 12, 16])}
    kind = "diff" if call == "train" else rng.choice(["box", "spheres", "spheres", "terrain", "instanced"])
    case["scene"] = kind
    if kind == "terrain":
        case.update(grid=rng.randint(64, 500), spheres=rng.randint(1, 500), level=rng.randint(1, 2))
    elif kind != "box":
        case.update(spheres=rng.randint(2, 150), level=rng.randint(1, 3), ground=rng.randint(4, 256))
    if call == "progressive":
        case["frames"] = rng.randint(1, 4)
        case["spp"] = 1
    if call == "render":
        case["mode"] = rng.choice(["wavefront", "wavefront", "megakernel"])
    if call in ("render", "progressive"):
        case["mis"] = rng.random() < 0.3
        case["halton"] = rng.random() < 0.3
    return case


def _scene_arrays(case, seed):
    kind = case["scene"]
    size = {"width": case.get("width", 16), "height": case.get("height", 16)}
    if kind == "box":
        return scenes.box_scene(seed=seed, **size)
    if kind == "terrain":
        return scenes.terrain_scene(seed=seed, grid=case["grid"], n_spheres=case["spheres"], level=case["level"], n_lights=16,
                                    **size)
    recipe = dict(seed=seed, n_spheres=case["spheres"], level=case["level"], ground_quads=case["ground"], **size)
    if kind == "instanced":
        return scenes.instanced_spheres_scene(**recipe)
    return scenes.spheres_scene(n_materials=256 if kind == "diff" else None, **recipe)


def _options(case):
    kw = {"mode": case.get("mode", "wavefront"), "mis": bool(case.get("mis")), "rr_start": 3,
          "sampler": "halton" if case.get("halton") else "pcg"}
    if case["call"] == "train":
        kw["rr_fixed"] = 0.9
    return kw


def _rays(case, seed, extent=60.0):
    """Half of the rays leave points above the ground in every direction (occlusion, baking), half come from
    a camera position toward points on the ground (picking)."""
    n = case["rays"]
    rng = torch.Generator(device="cuda")
    rng.manual_seed(seed)
    u = torch.rand((n, 6), generator=rng, device="cuda", dtype=torch.float32)
    o = torch.stack([(u[:, 0] - 0.5) * 1.4 * extent, 0.01 + 5.0 * u[:, 1], (u[:, 2] - 0.5) * 1.4 * extent], 1)
    d = torch.randn((n, 3), generator=rng, device="cuda", dtype=torch.float32)
    to = torch.stack([(u[:, 3] - 0.5) * 1.4 * extent, 2.0 * u[:, 4], (u[:, 5] - 0.5) * 1.4 * extent], 1)
    eye = torch.tensor([0.0, 0.5 * extent, 0.95 * extent], device="cuda")
    picked = (torch.arange(n, device="cuda") >= n // 2)[:, None]
    o = torch.where(picked, eye, o)
    d = torch.where(picked, to - eye, d)
    return o.contiguous(), (d / d.norm(dim=1, keepdim=True)).contiguous()


def prepare(case, seed):
    call = case["call"]
    state = {"call": call, "case": case, "seed": seed}
    if call == "batch":
        specs = scenes.batch_scenes(seed=seed % 100000, n=case["scenes"], max_tris=case["max_tris"])
        state["scenes"] = [pt.Scene.from_dict(s) for s in specs]
        # views of the full size, of two thirds and of a third of it in turn; every other one takes one sample
        state["cams"] = [dict(s["camera"], width=case["width"] * (3 - k % 3) // 3, height=case["height"] * (3 - k % 3) // 3)
                         for k, s in enumerate(specs)]
        state["spps"] = [case["spp"] if k % 2 else 1 for k in range(len(specs))]
        return state
    sc = _scene_arrays(case, seed)
    state["scene"] = pt.Scene.from_dict(sc)
    state["cam"] = sc["camera"]
    state["kw"] = _options(case)
    if call == "query":
        state["rays"] = _rays(case, seed)
    if call == "progressive":
        state["sums"] = torch.zeros((case["height"], case["width"], 3), device="cuda")
    if call in ("train", "backward"):
        rng = torch.Generator(device="cuda")
        rng.manual_seed(seed)
        state["grad"] = torch.randn((case["height"], case["width"], 3), generator=rng, device="cuda") / (
            case["height"] * case["width"])
    if call == "train":
        alb, em = scenes.diff_target(sc, seed=seed)
        state["albedo"] = torch.from_numpy(alb).cuda().requires_grad_()
        state["emission"] = torch.from_numpy(em.astype(np.float32)).cuda().requires_grad_()
    return state


def run(state):
    case, call, seed = state["case"], state["call"], state["seed"]
    depth = case.get("depth", 0)
    if call == "render":
        return state["scene"].render(state["cam"], case["spp"], depth, seed, **state["kw"])
    if call == "progressive":
        img = None
        for k in range(case["frames"]):
            img = state["scene"].render_progressive(state["cam"], case["spp"], depth, seed, k * case["spp"], state["sums"],
                                                    out=img, **state["kw"])
        return {"image": img, "sums": state["sums"]}
    if call == "train":
        kw = {k: v for k, v in state["kw"].items() if k != "mode"}
        img = pt.render_differentiable(state["albedo"], state["emission"], state["scene"], state["cam"], case["spp"], depth,
                                       seed, **kw)
        ga, ge = torch.autograd.grad(img, [state["albedo"], state["emission"]], grad_outputs=state["grad"])
        return {"image": img, "grad_albedo": ga, "grad_emission": ge}
    if call == "backward":
        ga, ge = state["scene"].backward(state["cam"], case["spp"], depth, seed, state["grad"], **state["kw"])
        return {"grad_albedo": ga, "grad_emission": ge}
    if call == "batch":
        return pt.render_batch(state["scenes"], state["cams"], state["spps"], depth, seed)
    t, prim = state["scene"].trace_closest(*state["rays"])
    return {"t": t, "prim": prim}


def _triangles(case):
    kind = case["scene"]
    if kind == "box":
        return 36
    if kind == "batch":
        return case["scenes"] * min(case["max_tris"], 20000)
    if kind == "terrain":
        return 2 * (case["grid"] - 1) ** 2 + case["spheres"] * 20 * 4 ** case["level"] + 32
    return case["spheres"] * 20 * 4 ** case["level"] + 2 * case["ground"] ** 2 + 16


def work(case):
    """Bytes: each triangle (36 bytes) and each input once, each output once.  Operations: every ray descends
    a tree over the triangles once (two boxes of 18 operations a level) and tests two triangles (45 operations
    each), every vertex is shaded (about 250); paths have 1.7 vertices and 1.4 shadow rays on average where
    the depth allows it (measured on the procedural scenes), and a gradient pass shades twice."""
    tris = _triangles(case)
    stored = 20 * 4 ** case["level"] + 2 * case["ground"] ** 2 + 2 if case["scene"] == "instanced" else tris
    ray = 36.0 * math.log2(tris + 1) + 90.0
    if case["call"] == "query":
        return {"bytes": 36 * stored + case["rays"] * 32, "flops": case["rays"] * ray}
    pixels = case["width"] * case["height"] * case.get("scenes", 1)
    if case["call"] == "batch":
        pixels *= 14 / 27
    spp = (1 + case["spp"]) / 2 if case["call"] == "batch" else case["spp"]
    paths = pixels * spp * case.get("frames", 1)
    vertices = min(case["depth"], 1.7)
    shadows = min(case["depth"] - 1, 1.4)
    flops = paths * ((vertices + shadows) * ray + vertices * 250)
    nbytes = 36 * stored + 12 * pixels
    if case["call"] == "train":
        nbytes, flops = nbytes + 12 * pixels, flops * 2 + paths * vertices * 250
    elif case["call"] == "backward":
        flops += paths * vertices * 250
    elif case["call"] == "progressive":
        nbytes += 12 * pixels
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits, by brute force
def _hits(o, d, tri):
    """Closest hits of rays (n x 3, float64) among triangles (m x 3 x 3): t (inf on a miss) and the index, the
    lower one on equal t.  Two-sided, barycentric bounds inclusive, t > 0."""
    n, m = o.shape[0], tri.shape[0]
    t_best = torch.full((n,), math.inf, dtype=torch.float64, device=o.device)
    i_best = torch.full((n,), -1, dtype=torch.int64, device=o.device)
    step = max(1, (1 << 25) // max(n, 1))
    for m0 in range(0, m, step):
        a = tri[m0:m0 + step, 0]
        e1, e2 = tri[m0:m0 + step, 1] - a, tri[m0:m0 + step, 2] - a
        # Moller-Trumbore's scalar triple products, as products of per-ray and per-triangle vectors
        nrm = torch.linalg.cross(e1, e2)
        det = -(d @ nrm.T)
        on = o @ nrm.T - (a * nrm).sum(1)
        t = on / det
        oxd = torch.linalg.cross(o, d)
        u = (oxd @ e2.T - d @ torch.linalg.cross(e2, a).T) / det
        v = (d @ torch.linalg.cross(e1, a).T - oxd @ e1.T) / det
        ok = (det != 0) & (u >= 0) & (u <= 1) & (v >= 0) & (u + v <= 1) & (t > 0)
        t = torch.where(ok, t, math.inf)
        tm, im = t.min(dim=1)
        better = tm < t_best
        i_best = torch.where(better, im + m0, i_best)
        t_best = torch.where(better, tm, t_best)
    return t_best, i_best


def _pcg(v):
    s = (v * 747796405 + 2891336453) & 0xFFFFFFFF
    w = (((s >> ((s >> 28) + 4)) ^ s) * 277803737) & 0xFFFFFFFF
    return (w >> 22) ^ w


def _unit(a):
    return a / a.norm(dim=1, keepdim=True)


def _exact_box(case, seed):
    """Mean radiance per pixel of the box (Lambert surfaces, one two-triangle light, black environment):
    light sampling at every vertex, cosine-weighted continuation, roulette from bounce 3."""
    f8 = dict(dtype=torch.float64, device="cuda")
    sc = _scene_arrays(case, seed)
    V = torch.tensor(np.asarray(sc["verts"], np.float32).astype(np.float64), **f8)
    tri = V[torch.tensor(np.asarray(sc["tris"]).astype(np.int64), device="cuda")]
    mat = torch.tensor(np.asarray(sc["tri_mat"]).astype(np.int64), device="cuda")
    albedo = torch.tensor(np.asarray(sc["mat_albedo"]).astype(np.float64), **f8)
    emission = torch.tensor(np.asarray(sc["mat_emission"]).astype(np.float64), **f8)
    normal = _unit(torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]))
    lights = torch.nonzero(emission[mat] > 0).flatten()
    areas = 0.5 * torch.linalg.cross(tri[lights, 1] - tri[lights, 0], tri[lights, 2] - tri[lights, 0]).norm(dim=1)
    area, cdf = areas.sum(), torch.cumsum(areas, 0) / areas.sum()
    W, H, spp, depth = case["width"], case["height"], case["spp"], case["depth"]
    path = torch.arange(W * H * spp, device="cuda")
    pixel, sample = path // spp, path % spp
    key = _pcg(sample ^ _pcg(pixel ^ _pcg((seed & 0xFFFFFFFF) ^ _pcg(torch.tensor(seed >> 32, device="cuda")))))

    def u(k, b, dim):
        return (_pcg(k ^ _pcg(torch.tensor((b << 4) | dim, device="cuda"))) >> 8).double() * 2.0 ** -24

    cam = sc["camera"]
    eye, target, up = (torch.tensor(np.asarray(cam[k]).astype(np.float64), **f8) for k in ("eye", "target", "up"))
    w = (eye - target) / (eye - target).norm()
    right = torch.linalg.cross(up, w)
    right = right / right.norm()
    th = math.tan(math.radians(cam["vfov_deg"]) / 2)
    sx = ((pixel % W).double() + u(key, 0, 0)) / W * 2 - 1
    sy = 1 - ((pixel // W).double() + u(key, 0, 1)) / H * 2
    d = _unit(sx[:, None] * right * (th * W / H) + sy[:, None] * torch.linalg.cross(w, right) * th - w)
    o = eye.expand_as(d)
    # the tangent frame is built in a frame rotated about (1, 2, 3) by one radian
    ax = np.array([1.0, 2.0, 3.0]) / math.sqrt(14.0)
    K = np.array([[0, -ax[2], ax[1]], [ax[2], 0, -ax[0]], [-ax[1], ax[0], 0]])
    R = torch.tensor(np.eye(3) + math.sin(1.0) * K + (1 - math.cos(1.0)) * K @ K, **f8)
    L = torch.zeros((W * H * spp, 3), **f8)
    tp = torch.ones_like(L)
    alive = path
    for b in range(depth):
        t, i = _hits(o, d, tri)
        keep = i >= 0
        alive, o, d, tp, t, i = alive[keep], o[keep], d[keep], tp[keep], t[keep], i[keep]
        if not len(alive):
            break
        k = key[alive]
        x, ng, m = o + d * t[:, None], normal[i], mat[i]
        front = (d * ng).sum(1) < 0
        if b == 0:
            L[alive] += torch.where(front, emission[m], 0.0)[:, None] * tp
        if b + 1 == depth:
            break
        n = torch.where(front[:, None], ng, -ng)
        eps = 1e-4 * x.abs().amax(1).clamp(min=1.0)[:, None]
        j = torch.searchsorted(cdf, u(k, b, 2), right=True).clamp(max=len(lights) - 1)
        su, u4 = u(k, b, 3).sqrt(), u(k, b, 4)
        b0, b1 = 1 - su, u4 * su
        P = tri[lights[j]]
        y = P[:, 0] * b0[:, None] + P[:, 1] * b1[:, None] + P[:, 2] * (1 - b0 - b1)[:, None]
        nl, os_ = normal[lights[j]], x + n * eps
        dv = y - os_
        dist2 = (dv * dv).sum(1)
        wi = dv / dist2.sqrt()[:, None]
        cx, cl = (n * wi).sum(1), -(wi * nl).sum(1)
        ys = y + nl * 1e-4 * y.abs().amax(1).clamp(min=1.0)[:, None]
        sv = ys - os_
        sd = sv.norm(dim=1)
        ts, _ = _hits(os_, sv / sd[:, None], tri)
        seen = (cx > 0) & (cl > 0) & ~(ts < sd)
        g = torch.where(seen, cx * cl * area / dist2, 0.0) / math.pi * emission[mat[lights[j]]]
        L[alive] += tp * albedo[m] * g[:, None]
        r = n @ R.T
        s = torch.copysign(torch.ones_like(r[:, 2]), r[:, 2])
        a = -1.0 / (s + r[:, 2])
        c = r[:, 0] * r[:, 1] * a
        T = torch.stack([1 + s * r[:, 0] ** 2 * a, s * c, -s * r[:, 0]], 1) @ R
        B = torch.stack([c, s + r[:, 1] ** 2 * a, -r[:, 1]], 1) @ R
        u6, phi = u(k, b, 6), 2 * math.pi * u(k, b, 7)
        rr = u6.sqrt()
        d = T * (rr * phi.cos())[:, None] + B * (rr * phi.sin())[:, None] + n * (1 - u6).sqrt()[:, None]
        tp = tp * albedo[m]
        o = x + n * eps
        if b >= 3:
            q = tp.amax(1).clamp(0.05, 0.95)
            live = u(k, b, 8) < q
            tp = tp / q[:, None]
            alive, o, d, tp = alive[live], o[live], d[live], tp[live]
    return L.reshape(H, W, spp, 3).mean(2)


def exact(case, seed):
    if case["call"] == "render" and case["scene"] == "box" and not case.get("halton") and not case.get("mis"):
        if case["width"] * case["height"] * case["spp"] <= 2000000:
            return _exact_box(case, seed)
    if case["call"] == "query" and case["rays"] * _triangles(case) <= 5e10:
        sc = _scene_arrays(case, seed)
        V = torch.tensor(np.asarray(sc["verts"], np.float32).astype(np.float64), device="cuda")
        tri = V[torch.tensor(np.asarray(sc["tris"]).astype(np.int64), device="cuda")]
        o, d = _rays(case, seed)
        t = torch.cat([_hits(o[k:k + 65536].double(), d[k:k + 65536].double(), tri)[0] for k in range(0, len(o), 65536)])
        return {"t": t, "prim": None}
    return None

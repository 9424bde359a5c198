"""Pooled walks of the wavefront's dense trace launches (pt_pool.cuh): a warp hands queue slots to its lanes
one by one, so slots at the ends of chunks, chunks at the ends of the queues and launches with fewer or more
chunks than warps are where it could go wrong.  The regenerating megakernel steps the walks of its lanes' paths in
the same phases.  The megakernel in the paper's layout walks each ray to its end in one thread and takes no slot
from a pool; all compute the same FP32 operations, so radiance, signatures and ray counts must be equal bit for bit."""
import numpy as np
import pytest

from paper_2605_27323_gb300 import scenes

pytestmark = pytest.mark.gpu

# paths per launch: one, a chunk of 32 and its neighbours, about one and about two chunks per warp of a full grid
# (152 SMs x 5 blocks x 8 warps x 32 = 194560 slots), and a queue that is no multiple of anything
SIZES = [(1, 1, 1), (31, 1, 1), (32, 1, 1), (33, 1, 1), (311, 313, 1), (441, 441, 1), (4865, 40, 1), (487, 799, 1),
         (523, 397, 3)]


@pytest.fixture(scope="module")
def views():
    import torch

    import paper_2605_27323_gb300 as pt
    assert torch.cuda.is_available()
    soup = scenes.random_soup(n_tris=3000, seed=11, spread=1.0, size=0.25)
    out = {}
    for name, sc in (("soup", soup), ("spheres", scenes.spheres_scene(seed=5, n_spheres=40, level=2, ground_quads=32,
                                                                      extent=15.0)),
                     ("placed", scenes.instanced_spheres_scene(seed=5, n_spheres=40, level=2, ground_quads=32,
                                                               extent=15.0))):
        out[name] = (pt.Scene.from_dict(sc), sc.get("camera") or scenes.camera((0.2, 0.4, 4.0), (0, 0, 0)))
    return out


@pytest.mark.parametrize("scene", ["soup", "spheres", "placed"])
@pytest.mark.parametrize("width,height,spp", SIZES)
def test_pooled_walks_equal_one_ray_per_thread(views, scene, width, height, spp):
    import torch
    g, cam = views[scene]
    cam = dict(cam, width=width, height=height)
    a = g.render(cam, spp, 4, 3, path_L=True, sig=True, mode="wavefront")
    sa = g.stats()
    for static in (False, True):
        b = g.render(cam, spp, 4, 3, path_L=True, sig=True, mode="megakernel", mk_static=static)
        sb = g.stats()
        assert sa["status"] == 0 and sb["status"] == 0
        for k in ("img", "path_L", "sig"):
            assert torch.equal(a[k], b[k]), (k, static)
        assert (sa["extension_rays"], sa["shadow_rays"]) == (sb["extension_rays"], sb["shadow_rays"])


@pytest.mark.parametrize("width,height", [(33, 1), (441, 441), (487, 799)])
def test_pooled_replay_equals_the_separate_order(views, width, height):
    """The adjoint replay's pooled shadow walks mark vertex records; the separate order marks them in lockstep.
    Gradients are sums of float atomics: 1e-5 of the largest covers a reordering of 4e5 terms (sqrt(n) 2^-24)."""
    import torch
    g, cam = views["spheres"]
    cam = dict(cam, width=width, height=height)
    grad = torch.ones((height, width, 3), device="cuda") / (width * height)
    ga, ge = g.backward(cam, 1, 4, 3, grad)
    ha, he = g.backward(cam, 1, 4, 3, grad, separate_shadow=True)
    for x, y in ((ga, ha), (ge, he)):
        assert float((x - y).abs().max()) <= 1e-5 * max(float(y.abs().max()), 1e-30)
    assert np.isfinite(float(ga.sum()))


@pytest.fixture(scope="module")
def large():
    import paper_2605_27323_gb300 as pt
    sc = scenes.spheres_scene(seed=7, n_spheres=30, level=4, ground_quads=160, extent=12.0)
    g = pt.Scene.from_dict(sc)
    assert g.info()["n_nodes"] >= 1 << 14
    return g, sc["camera"]


@pytest.mark.parametrize("width,height,spp", [(33, 1, 1), (311, 313, 1), (441, 441, 1), (487, 799, 1), (523, 397, 3)])
def test_shared_last_walks_equal_one_ray_per_thread(large, width, height, spp):
    """Trees of 2^14 nodes and more: the last walks of a trace launch are shared among a warp's lanes (renders
    without signatures).  The hit of a shared walk is the smallest (t, original id), that of a walk in one lane."""
    import torch
    g, cam = large
    cam = dict(cam, width=width, height=height)
    a = g.render(cam, spp, 4, 3, path_L=True, mode="wavefront")
    sa = g.stats()
    b = g.render(cam, spp, 4, 3, path_L=True, mode="megakernel", mk_static=True)
    sb = g.stats()
    assert sa["status"] == 0 and sb["status"] == 0
    for k in ("img", "path_L"):
        assert torch.equal(a[k], b[k]), k
    assert (sa["extension_rays"], sa["shadow_rays"]) == (sb["extension_rays"], sb["shadow_rays"])
    grad = torch.ones((height, width, 3), device="cuda") / (width * height)
    ga, ge = g.backward(cam, spp, 4, 3, grad)
    ha, he = g.backward(cam, spp, 4, 3, grad, separate_shadow=True)
    for x, y in ((ga, ha), (ge, he)):
        assert float((x - y).abs().max()) <= 1e-5 * max(float(y.abs().max()), 1e-30)


def _query(g, rays, n):
    import ctypes as C

    import torch

    from paper_2605_27323_gb300 import capi
    t = torch.empty(n, device="cuda")
    prim = torch.empty(n, device="cuda", dtype=torch.int32)
    capi.check(capi.load().pt_trace_closest(g.h, C.c_void_p(rays), n, C.c_void_p(t.data_ptr()), C.c_void_p(prim.data_ptr()),
                                            C.c_void_p(torch.cuda.current_stream().cuda_stream)))
    return t, prim


@pytest.mark.parametrize("scene", ["soup", "placed", "large"])
@pytest.mark.parametrize("n", [1, 31, 33, 194559, 194561, 400003])
def test_pooled_queries(views, large, scene, n):
    """Closest-hit queries at the edges of a warp's runs and of the grid, with rays at float alignment only: each
    ray's hit is that of a query of a few rays (a run of its own warp), whatever its place."""
    import torch
    g = large[0] if scene == "large" else views[scene][0]
    o, d = scenes.random_rays(n, seed=n, spread=1.5)
    rays = torch.zeros(8 * n + 1, device="cuda")
    r = rays[1:].view(n, 8)
    r[:, 0:3] = torch.as_tensor(o * (1.0 if scene == "soup" else 4.0), dtype=torch.float32, device="cuda")
    r[:, 4:7] = torch.as_tensor(d, dtype=torch.float32, device="cuda")
    t, prim = _query(g, r.data_ptr(), n)
    at = sorted({0, n - 1, n // 2, n // 3, 7 * n // 8})
    for i in at:
        m = min(n - i, 5)
        few = r[i:i + m].clone()
        t1, p1 = _query(g, few.data_ptr(), m)
        assert torch.equal(t[i:i + m], t1) and torch.equal(prim[i:i + m], p1), i
    assert bool(((prim >= 0) == torch.isfinite(t)).all())


# the wavefront's records are added up four floats a load, the megakernel's as three floats
@pytest.mark.parametrize("spp", [1, 2, 3, 4, 5, 7, 8, 16, 17])
def test_samples_add_up_alike(views, spp):
    import torch
    g, cam = views["soup"]
    cam = dict(cam, width=37, height=23)
    a = g.render(cam, spp, 3, 4, mode="wavefront")
    b = g.render(cam, spp, 3, 4, mode="megakernel")
    assert torch.equal(a, b)

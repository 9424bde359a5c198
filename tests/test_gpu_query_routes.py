"""Closest-hit queries take one of three routes: one ray per thread (8 rays or fewer, 4 on trees with
shared ends, or no more rays than threads on a tree of fewer than 64 nodes), pooled walks, and pooled walks with shared
ends (trees of 2^14 nodes and more).  The hit must not depend on
the route: the smallest t, and among equal t the lowest original triangle id.  Scenes hold many copies of their
triangles -- more than a leaf takes, so that equal hits are met in different leaves and by different lanes -- and
triangles without area."""
import ctypes as C

import numpy as np
import pytest

from paper_2605_27323_gb300 import scenes

pytestmark = pytest.mark.gpu


def _copied(sc, every, copies, seed=3):
    """The scene with `copies` more of every `every`-th triangle (same vertices, later ids) and as many triangles
    without area (two corners or three in one point, or in a line)."""
    rng = np.random.default_rng(seed)
    tris, mat, verts = np.asarray(sc["tris"]), np.asarray(sc["tri_mat"]), np.asarray(sc["verts"], np.float32)
    pick = np.repeat(np.arange(0, len(tris), every), copies)
    flat = tris[rng.integers(0, len(tris), 3 * (len(tris) // every) + 3)].copy()
    flat[0::3, 1] = flat[0::3, 0]
    flat[1::3, 1] = flat[1::3, 2] = flat[1::3, 0]
    mid = len(verts) + np.arange(len(flat[2::3]))
    v = np.concatenate([verts, 0.5 * (verts[flat[2::3, 0]] + verts[flat[2::3, 1]])]).astype(np.float32)
    flat[2::3, 2] = mid
    extra = np.concatenate([tris[pick], flat])
    em = np.concatenate([mat[pick], np.zeros(len(flat), mat.dtype)])
    order = rng.permutation(len(extra))
    return dict(sc, verts=v, tris=np.concatenate([tris, extra[order]]).astype(np.uint32),
                tri_mat=np.concatenate([mat, em[order]]).astype(mat.dtype))


@pytest.fixture(scope="module")
def views():
    import torch

    import paper_2605_27323_gb300 as pt
    assert torch.cuda.is_available()
    tiny = scenes.spheres_scene(seed=5, n_spheres=1, level=0, ground_quads=2, extent=10.0)
    mid = scenes.spheres_scene(seed=5, n_spheres=6, level=2, ground_quads=8, extent=10.0)
    large = scenes.spheres_scene(seed=7, n_spheres=20, level=4, ground_quads=128, extent=10.0)
    out = {"tiny": (tiny, 0), "mid": (mid, 5), "large": (large, 50),
           "placed": (scenes.instanced_spheres_scene(seed=5, n_spheres=2, level=0, ground_quads=4, extent=10.0), 0)}
    made = {}
    for k, (sc, every) in out.items():
        sc = _copied(sc, every, 40) if every else sc
        g = pt.Scene.from_dict(sc)
        made[k] = (g, sc["camera"])
    n = {k: g.info()["n_nodes"] for k, (g, _) in made.items()}
    assert n["tiny"] < 64 <= n["mid"] < 1 << 14 <= n["large"] and n["placed"] < 64, n
    return made


def _query(g, rays):
    import torch

    from paper_2605_27323_gb300 import capi
    n = rays.shape[0]
    t = torch.full((n,), -1.0, device="cuda")
    prim = torch.full((n,), -2, device="cuda", dtype=torch.int32)
    capi.check(capi.load().pt_trace_closest(g.h, C.c_void_p(rays.data_ptr()), n, C.c_void_p(t.data_ptr()),
                                            C.c_void_p(prim.data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream)))
    return t, prim


def _rays(n, seed):
    import torch
    rng = np.random.default_rng(seed)
    o = np.stack([rng.uniform(-8, 8, n), rng.uniform(0.2, 6, n), rng.uniform(-8, 8, n)], 1)
    d = rng.normal(size=(n, 3))
    d[: n // 2, 1] = -np.abs(d[: n // 2, 1])
    r = np.zeros((n, 8), np.float32)
    r[:, 0:3] = o
    r[:, 4:7] = d / np.linalg.norm(d, axis=1, keepdims=True)
    return torch.from_numpy(r).cuda()


@pytest.mark.parametrize("scene", ["tiny", "mid", "large", "placed"])
def test_hits_do_not_depend_on_the_route(views, scene):
    import torch
    g = views[scene][0]
    rays = _rays(200003, 11)
    t, prim = _query(g, rays)                       # more rays than a grid has threads
    assert float((prim >= 0).float().mean()) > 0.3
    for k in list(range(0, 2000, 4)) + [199999]:    # 4 at a time: one ray per thread
        t1, p1 = _query(g, rays[k:k + 4].clone())
        assert torch.equal(t[k:k + 4], t1) and torch.equal(prim[k:k + 4], p1), k
    for n in (1, 2, 3, 4, 5, 7, 8, 9, 31, 32, 33, 255, 257, 4001, 100003, 194560, 194561):
        t1, p1 = _query(g, rays[:n].clone())
        assert torch.equal(t[:n], t1) and torch.equal(prim[:n], p1), n


def test_a_query_of_no_rays(views):
    g = views["mid"][0]
    t, prim = g.trace_closest(np.zeros((0, 3), np.float32), np.zeros((0, 3), np.float32))
    assert t.numel() == 0 and prim.numel() == 0


@pytest.mark.parametrize("scene,capacity", [("large", 0), ("large", 30011), ("mid", 7001), ("tiny", 1000)])
def test_renders_of_copied_triangles(views, scene, capacity):
    """One wave and several: the wavefront against one thread per path, among coincident triangles."""
    import torch
    g, cam = views[scene]
    cam = dict(cam, width=317, height=211)
    a = g.render(cam, 2, 5, 9, path_L=True, queue_capacity=capacity)
    b = g.render(cam, 2, 5, 9, path_L=True, mode="megakernel", mk_static=True)
    assert torch.equal(a["path_L"], b["path_L"]) and torch.equal(a["img"], b["img"])

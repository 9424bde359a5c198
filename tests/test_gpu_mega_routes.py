"""The regenerating megakernel on trees of fewer than 64 nodes: in lockstep up to two paths a thread, by pooled walks from
there on (152 SMs x 8 blocks x 128 threads x 2 = 311296 paths).  Both must equal one thread per path bit for bit."""
import pytest

from paper_2605_27323_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def views():
    import torch

    import paper_2605_27323_gb300 as pt
    assert torch.cuda.is_available()
    made = {}
    for k, sc in (("box", scenes.box_scene()),
                  ("tiny", scenes.spheres_scene(seed=5, n_spheres=1, level=0, ground_quads=2, extent=10.0)),
                  ("placed", scenes.instanced_spheres_scene(seed=5, n_spheres=2, level=0, ground_quads=4, extent=10.0))):
        g = pt.Scene.from_dict(sc)
        assert g.info()["n_nodes"] < 64
        made[k] = (g, sc["camera"])
    return made


@pytest.mark.parametrize("scene", ["box", "tiny", "placed"])
@pytest.mark.parametrize("mis", [False, True])
@pytest.mark.parametrize("width,height,spp", [(1, 1, 1), (33, 7, 3), (608, 512, 1), (608, 513, 1)])
def test_small_trees(views, scene, mis, width, height, spp):
    import torch
    g, cam = views[scene]
    cam = dict(cam, width=width, height=height)
    a = g.render(cam, spp, 5, 3, path_L=True, sig=True, mode="megakernel", mis=mis)
    sa = g.stats()
    b = g.render(cam, spp, 5, 3, path_L=True, sig=True, mode="megakernel", mk_static=True, mis=mis)
    sb = g.stats()
    for k in ("img", "path_L", "sig"):
        assert torch.equal(a[k], b[k]), k
    assert sa["status"] == 0 and (sa["extension_rays"], sa["shadow_rays"]) == (sb["extension_rays"], sb["shadow_rays"])
    assert torch.equal(g.render(cam, spp, 5, 3, mode="megakernel", mis=mis), a["img"])

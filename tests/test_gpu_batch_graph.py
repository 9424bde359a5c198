"""The captured bounce loop of batched rendering is kept between calls and replayed when a call has the same shape.
Whatever the launches in it read from their arguments has to be part of that shape, and whatever they read through an
address has to stay at that address: each image must equal its standalone render bit for bit, whichever call came
before."""
import pytest

from paper_2605_27323_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def scene():
    import torch

    import paper_2605_27323_gb300 as pt
    assert torch.cuda.is_available()
    sc = scenes.spheres_scene(seed=3, n_spheres=12, level=2, ground_quads=16, extent=10.0)
    return pt.Scene.from_dict(sc), sc["camera"]


@pytest.mark.parametrize("order", [(False, True, False), (True, False, True)])
def test_batches_of_one_shape_with_and_without_mis(scene, order):
    import torch

    import paper_2605_27323_gb300 as pt
    g, cam = scene
    cams = [dict(cam, width=61, height=37), dict(cam, width=40, height=30)]
    for mis in order:
        outs = pt.render_batch([g, g], cams, [2, 4], 5, 7, mis=mis)
        for o, c, spp in zip(outs, cams, [2, 4]):
            assert torch.equal(o, g.render(c, spp, 5, 7, mis=mis)), mis
    assert not torch.equal(g.render(cams[1], 4, 5, 7, mis=False), g.render(cams[1], 4, 5, 7, mis=True))


# the waves of the first view hold one segment, those of the others 4, 16 and 64 (32 bytes each): the tables that
# follow the segments move
@pytest.mark.parametrize("sizes", [(8, 16, 32, 64), (64, 32, 16, 8)])
def test_batches_of_one_shape_with_other_image_sizes(scene, sizes):
    import torch

    import paper_2605_27323_gb300 as pt
    g, cam = scene
    for k, size in enumerate(sizes):
        c = dict(cam, width=size, height=size)
        out, = pt.render_batch([g], [c], [1], 5, 100 + k, queue_capacity=64)
        assert torch.equal(out, g.render(c, 1, 5, 100 + k)), size

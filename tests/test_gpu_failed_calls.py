"""Statistics after a call that failed to get its workspace: the call traced nothing, and pt_get_stats must not report
the counts of the call before it."""
import pytest

from paper_2605_27323_gb300 import scenes

pytestmark = pytest.mark.gpu

# 2^32 - 2^20 paths of 180 bytes are 773 GB: no device holds them, so the allocation is refused at once
CAM = {"width": 1024, "height": 1024}
SPP = 4096


@pytest.fixture(scope="module")
def scene():
    import torch

    import paper_2605_27323_gb300 as pt
    assert torch.cuda.is_available()
    sc = scenes.box_scene(width=32, height=24)
    return pt.Scene.from_dict(sc), sc["camera"]


def _fails(call):
    from paper_2605_27323_gb300 import capi
    with pytest.raises(capi.PtError) as e:
        call()
    assert "cudaMalloc" in str(e.value)


@pytest.mark.parametrize("call", ["render", "progressive"])
def test_a_failed_render_reports_no_rays(scene, call):
    import torch
    g, cam = scene
    want = g.render(cam, 4, 5, 3)
    before = g.stats()
    assert before["extension_rays"] > 0 and before["shadow_rays"] > 0
    big = dict(cam, **CAM)
    if call == "render":
        _fails(lambda: g.render(big, SPP, 5, 3))
    else:
        sums = torch.zeros((CAM["height"], CAM["width"], 3), device="cuda")
        _fails(lambda: g.render_progressive(big, SPP, 5, 3, 0, sums))
    st = g.stats()
    assert st["extension_rays"] == 0 and st["shadow_rays"] == 0 and st["bounces"] == 0 and sum(st["group_walks"]) == 0
    # and the scene renders as before
    assert torch.equal(g.render(cam, 4, 5, 3), want)
    after = g.stats()
    assert (after["extension_rays"], after["shadow_rays"]) == (before["extension_rays"], before["shadow_rays"])

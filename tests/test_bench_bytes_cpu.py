"""Algorithmic bytes of bench.py's rooflines, in numbers: a camera ray's walk reads its direction (16 B) and writes its hit
(8 B); its shading reads those and writes radiance (16 B), the next ray (48 B) and the shadow ray (48 B).  Later bounces
read origin, throughput and radiance too."""
import bench


def test_bounce_0_is_charged_what_it_moves():
    st = {"active": [100, 60, 30], "shadow_rays": 120}
    extend = 100 * 24 + 90 * 40
    shade = 100 * 136 + 90 * 184
    assert bench.frame_bytes(st, 100, 50) == extend + shade + 120 * 80 + 100 * 16 + 100 * 16 + 50 * 12 == 49560


def test_camera_rays_alone():
    assert bench.frame_bytes({"active": [7], "shadow_rays": 0}, 7, 7) == 7 * (24 + 136 + 16 + 16 + 12)
    assert bench.frame_bytes({"active": [], "shadow_rays": 0}, 0, 0) == 0


def test_extend_stage():
    # forward and adjoint: 190 extension rays each, 100 of them camera rays; 120 shadow walks each
    assert bench.extend_stage_bytes(380, 200, 120, 120) == 200 * 24 + 180 * 40 + 120 * 80 + 120 * 40 == 26400

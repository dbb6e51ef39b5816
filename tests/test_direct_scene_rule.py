"""Which frames take the direct route for their small triangles: the lines, in
pixels of the framebuffer a triangle, of meshes and soups by the frame's size."""
import pytest

from paper_1404_6293_gb300 import _lib as L


@pytest.mark.parametrize("width,height,mesh,soup", [
    (160, 120, 4, 2), (320, 240, 4, 2), (362, 362, 4, 2),           # below 2^17 pixels
    (512, 256, 7, 3), (640, 400, 7, 3), (900, 600, 7, 3),
    (1024, 768, 10, 3), (1280, 720, 10, 3), (1920, 1080, 10, 3), (32767, 32767, 10, 3)])
def test_lines_by_frame_size(width, height, mesh, soup):
    rule = L.load().piko_raster_direct_scene
    px = width * height
    for line, v_of in ((mesh, lambda t: t // 2 + 100), (mesh, lambda t: 2 * t - 1), (soup, lambda t: 2 * t),
                       (soup, lambda t: 3 * t)):
        t = -(-px // line)  # the fewest triangles at that many pixels each
        assert rule(width, height, t, v_of(t)) == 1
        assert rule(width, height, t - 1, v_of(t - 1)) == 0


def test_no_triangles_or_vertices():
    rule = L.load().piko_raster_direct_scene
    assert rule(64, 64, 0, 100) == 0
    assert rule(64, 64, 100000, 0) == 0

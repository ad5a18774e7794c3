"""Fine meshes (cells below 2.5 eye pixels: a raster lane takes a triangle) in calls of at least
3,648 tiles, where a warp draws half tiles with four pixels per lane, and of at least 5,472, where it
draws whole ones: strips that share a resident round whose bins exceed a window, several rounds of views, one and several set-up blocks per view,
plain and persistent grids.  The reference is the inspection render, which takes a lane per pixel;
the arithmetic is the same, so the images are compared bit for bit."""
import math

import numpy as np
import pytest

import scene

pytestmark = pytest.mark.gpu


def _eyes(n, w, h, f):
    """n heads inside the cap rig; focal length f, in pixels."""
    poses = [scene.head_pose_eyes(scene.SplitMix64(50 + k), w, h, 90.0, yaw_range=(-0.1, 0.1), pitch_deg=6.0,
                                  stereo=False)[0].pose for k in range(n)]
    return [scene.Eye(p, np.array([f, f, 0.5 * w, 0.5 * h]), w, h) for p in poses]


# views, grid, disk scale, ovals, eyes (number, width, height, focal length): cells of 2.0 pixels
# (16 eyes of 4,096 tiles, 22 of 5,632) and 1.6 and 1.9 pixels (one eye of 3,933 or 6,688 tiles)
@pytest.mark.parametrize("views,grid,disk,oval,eyes", [
    (9, 129, 1.2, False, (16, 256, 250, 128.0)),
    (9, 65, 1.2, True, (16, 256, 250, 64.0)),
    (40, 65, 6.0, False, (16, 256, 250, 64.0)),
    (9, 257, 1.2, False, (1, 1100, 901, 240.0)),
    (40, 257, 6.0, True, (1, 1100, 901, 210.0)),
    (9, 129, 1.2, True, (22, 256, 250, 128.0)),
    (40, 65, 6.0, False, (22, 256, 250, 64.0)),
    (9, 257, 1.2, False, (1, 1400, 1203, 240.0)),
])
@pytest.mark.parametrize("tile", [(16, 16), (32, 8)])
@pytest.mark.parametrize("fmt", ["f32", "u8"])
def test_fine_meshes_in_whole_tiles_draw_the_inspection_image(fmt, tile, views, grid, disk, oval, eyes):
    torch = pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm
    from paper_1810_08860_gb300 import disks

    side = math.isqrt(views - 1) + 1
    lf = scene.build_light_field(scene.sphere_scene(3, 8, forward_cone_deg=35.0), scene.cap_grid_directions(side, 40.0)[:views],
                                 64, 64, 90.0, grid, disk_scale=disk)
    E = _eyes(*eyes)
    tiles = sum(-(-e.width // tile[0]) * -(-e.height // tile[1]) for e in E)
    assert tiles >= 3648 and 64 / (grid - 1) * E[0].intr[0] / lf.intr[0][0] < 2.5
    r = lfm.Renderer(0, tile=tile, max_eyes=len(E), tri_capacity=24 << 20)
    r.load_views(lf, tex_format=fmt)
    r.build_meshes(lf)
    if oval:
        r.set_disk_ovals(disks.oval_extents(lf))
    want = [r.render_inspect(e, max_records=views)["rgba"] for e in E]
    assert all(int((w[..., 3] > 0).sum()) > 1000 for w in want)
    for got in (r.render(E), r.render_batch(E)):
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    r.stats()  # no scratch ran out
    r.close()

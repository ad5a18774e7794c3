"""The raster's forms draw one image: a warp per tile or per strip, a lane per
pixel or per triangle (fine meshes), one or several windows of gathered
triangles, one or several rounds of views.  The reference is the inspection
render, whose coverage is held to the oracle elsewhere; the arithmetic of every
form is the same, so the images are compared bit for bit.

Grids whose triangle set-up takes one block per view (up to 65^2 vertices) and
several: coverage records against the oracle, and the triangle pool's limit."""
import math

import pytest

import scene
from tests.test_gpu_parity import _check_full_frame

pytestmark = pytest.mark.gpu

# views, image size, grid, disk scale, eye size, ovals.  Cells of about 0.6-2 px (fine) and up to 64 px;
# eyes that no tile divides, one pixel and one row; 40 wide disks: two rounds of views and several windows.
CASES = [
    (16, 96, 65, 1.2, (61, 47), False),
    (16, 96, 33, 1.2, (63, 49), False),
    (16, 64, 65, 1.2, (17, 3), True),
    (9, 64, 9, 1.2, (257, 255), False),
    (9, 64, 9, 1.2, (1, 1), False),
    (9, 64, 5, 1.2, (1100, 900), True),
    (40, 64, 33, 6.0, (90, 70), False),
    (40, 64, 33, 6.0, (24, 20), False),
    (200, 16, 33, 1.2, (90, 70), False),
    (9, 64, 70, 1.2, (75, 53), False),
    (9, 64, 70, 1.2, (311, 203), True),
]


@pytest.mark.parametrize("views,size,grid,disk,eye,oval", CASES)
@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 8)])
def test_every_form_draws_the_inspection_image(views, size, grid, disk, eye, oval, tile):
    torch = pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm
    from paper_1810_08860_gb300 import disks

    side = math.isqrt(views - 1) + 1
    lf = scene.build_light_field(scene.sphere_scene(3, 8, forward_cone_deg=35.0), scene.cap_grid_directions(side, 40.0)[:views],
                                 size, size, 90.0, grid, disk_scale=disk)
    e = scene.head_pose_eyes(scene.SplitMix64(11), eye[0], eye[1], 90.0, yaw_range=(-0.1, 0.1), pitch_deg=6.0, stereo=False)[0]
    r = lfm.Renderer(0, tile=tile)
    r.load_views(lf)
    r.build_meshes(lf)
    if oval:
        r.set_disk_ovals(disks.oval_extents(lf))
    want = r.render_inspect(e, max_records=views)["rgba"]
    assert eye == (1, 1) or int((want[..., 3] > 0).sum()) > 0
    assert torch.equal(r.render([e])[0], want)
    assert torch.equal(r.render_batch([e])[0], want)
    tiles = -(-eye[0] // tile[0]) * -(-eye[1] // tile[1])
    if views <= 32 and grid <= 33 and tiles <= 8192:  # lf_render_static's limits
        assert torch.equal(r.render_static(e), want)
    r.close()


# Four pixels per lane: 256-pixel tiles in eyes of at least 3648 tiles (whole tiles).
@pytest.mark.parametrize("fmt", ["f32", "u8", "bf16", "fp8"])
@pytest.mark.parametrize("tile", [(16, 16), (32, 8)])
@pytest.mark.parametrize("views,grid,disk,oval", [(9, 5, 1.2, True), (40, 17, 6.0, False)])
def test_wide_lanes_draw_the_inspection_image(fmt, tile, views, grid, disk, oval):
    torch = pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm
    from paper_1810_08860_gb300 import disks

    side = math.isqrt(views - 1) + 1
    lf = scene.build_light_field(scene.sphere_scene(3, 8, forward_cone_deg=35.0), scene.cap_grid_directions(side, 40.0)[:views],
                                 64, 64, 90.0, grid, disk_scale=disk)
    e = scene.head_pose_eyes(scene.SplitMix64(11), 1100, 901, 90.0, yaw_range=(-0.1, 0.1), pitch_deg=6.0, stereo=False)[0]
    r = lfm.Renderer(0, tile=tile)
    r.load_views(lf, tex_format=fmt)
    r.build_meshes(lf)
    if oval:
        r.set_disk_ovals(disks.oval_extents(lf))
    want = r.render_inspect(e, max_records=views)["rgba"]
    assert int((want[..., 3] > 0).sum()) > 0
    assert torch.equal(r.render([e])[0], want)
    assert torch.equal(r.render_batch([e, e])[1], want)
    r.close()


@pytest.mark.parametrize("n", [1, 2, 3, 5])
def test_eyes_by_value_and_by_copy_draw_the_same(n):
    """Up to two eyes travel with the launch, more through the pinned ring."""
    torch = pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm

    lf, _ = _cap(9, 64, 17)
    eyes = [scene.head_pose_eyes(scene.SplitMix64(20 + k), 40 + 9 * k, 31 + 5 * k, 90.0, yaw_range=(-0.1, 0.1), pitch_deg=6.0,
                                 stereo=False)[0] for k in range(n)]
    r = lfm.Renderer(0, max_eyes=8)
    r.load_views(lf)
    r.build_meshes(lf)
    want = [r.render_inspect(e, max_records=9)["rgba"] for e in eyes]
    for _ in range(6):  # more calls than the ring has slots, each with its own eyes
        eyes, want = eyes[1:] + eyes[:1], want[1:] + want[:1]
        for got in (r.render(eyes), r.render_batch(eyes)):
            assert all(torch.equal(a, b) for a, b in zip(got, want))
    # a captured call replays its own eyes after other calls
    side = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    out = [torch.zeros_like(w) for w in want]
    if n <= 2:
        r.render(eyes, out=out)
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=side):
            r.render(eyes, out=out)
        r.render([eyes[-1]])
        for o in out:
            o.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(out, want))
    r.close()


def _cap(views, size, grid, seed=3, eye=(75, 53)):
    side = math.isqrt(views - 1) + 1
    lf = scene.build_light_field(scene.sphere_scene(seed, 8, forward_cone_deg=35.0),
                                 scene.cap_grid_directions(side, 40.0)[:views], size, size, 90.0, grid)
    e = scene.head_pose_eyes(scene.SplitMix64(seed), eye[0], eye[1], 90.0, yaw_range=(-0.1, 0.1), pitch_deg=6.0, stereo=False)[0]
    return lf, e


@pytest.mark.parametrize("grid,mesh,eye", [(2, "f32", (75, 53)), (6, "f16", (75, 53)), (65, "f32", (75, 53)), (66, "f32", (75, 53)),
                                           (70, "f32", (75, 53)), (131, "f32", (75, 53)), (66, "f32", (311, 203))])
def test_grids_of_one_and_of_several_parts_cover_as_the_oracle(grid, mesh, eye):
    pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm

    lf, e = _cap(9, 64, grid, eye=eye)
    if mesh == "f16":  # depths that FP16 offsets hold exactly: the oracle sees the same mesh
        lf.depth = (lf.depth * 8).round().clip(8, 48) / 8
        lf.depth = lf.depth.astype("float32")
    r = lfm.Renderer(0)
    r.load_views(lf)
    r.build_meshes(lf, mesh_format=mesh)
    _check_full_frame(r, lf, e)
    r.close()


@pytest.mark.parametrize("grid", [33, 66])
def test_a_pool_that_is_too_small_is_reported_and_the_context_stays_usable(grid):
    torch = pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm

    lf, e = _cap(9, 64, grid)
    r = lfm.Renderer(0, tri_capacity=500)
    r.load_views(lf)
    r.build_meshes(lf)
    r.render([e])
    with pytest.raises(lfm.LFError, match="CAPACITY"):
        r.stats()
    r.close()
    r = lfm.Renderer(0)
    r.load_views(lf)
    r.build_meshes(lf)
    img = r.render([e])[0]
    n = r.stats()["triangles"]
    q = lfm.Renderer(0, tri_capacity=n)  # the records that a view keeps fit exactly
    q.load_views(lf)
    q.build_meshes(lf)
    assert torch.equal(q.render([e])[0], img) and q.stats()["triangles"] == n
    q.close()
    r.close()

"""The share of the image that a raster warp takes changes with the number of tiles near the
eye's axis: strips of a tile, half tiles, whole tiles.  Rows added far from the axis, where there
is nothing to see, must not change the time by more than their writing (1,488 tiles of background,
a few per cent; drawing whole tiles in every call of 3,648 tiles and more made it 1.46 times here)."""
import pytest

import scene
from tests.test_gpu_raster_fine_tiles import _eyes

pytestmark = pytest.mark.gpu


def test_rows_far_from_the_axis_cost_what_they_write():
    """2,512 and 4,000 tiles, as much to see in each."""
    torch = pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm

    lf = scene.build_light_field(scene.sphere_scene(3, 8, forward_cone_deg=35.0), scene.cap_grid_directions(4, 40.0),
                                 64, 64, 90.0, 17, disk_scale=1.2)
    r = lfm.Renderer(0)
    r.load_views(lf)
    r.build_meshes(lf)
    ms = []
    for h in (2500, 4000):
        E = _eyes(1, 250, h, 125.0)
        out = [torch.empty((e.height, e.width, 4), device="cuda") for e in E]
        best = float("inf")
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            r.render(E, out=out)
            torch.cuda.synchronize()
            a.record()
            for _ in range(30):
                r.render(E, out=out)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / 30)
        ms.append(best)
    r.stats()
    r.close()
    assert ms[1] < 1.25 * ms[0], ms


@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 8)])
@pytest.mark.parametrize("oval", [False, True])
@pytest.mark.parametrize("size", [(960, 960, 480.0), (976, 971, 480.0), (1190, 1203, 590.0), (250, 16000, 125.0)])
def test_halves_and_whole_tiles_draw_the_inspection_image(size, oval, tile):
    """Images of fewer than 3,648 tiles, of fewer than 5,472, of more, and of many far from the axis."""
    torch = pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm
    from paper_1810_08860_gb300 import disks

    lf = scene.build_light_field(scene.sphere_scene(3, 8, forward_cone_deg=35.0), scene.cap_grid_directions(7, 40.0)[:40],
                                 64, 64, 90.0, 17, disk_scale=6.0)
    E = _eyes(1, *size)
    r = lfm.Renderer(0, tile=tile)
    r.load_views(lf)
    r.build_meshes(lf)
    if oval:
        r.set_disk_ovals(disks.oval_extents(lf))
    want = r.render_inspect(E[0], max_records=1)["rgba"]
    assert int((want[..., 3] > 0).sum()) > 10000
    assert torch.equal(r.render(E)[0], want)
    assert torch.equal(r.render_batch(E)[0], want)
    r.close()

"""Small and large images in one call: what a raster warp takes of a tile (a strip, half, all of it)
is decided for each eye.  The images are the inspection images to the bit, and a small image beside a
large one, whose tiles hold the views and triangles of many, does not hold the call up."""
import math

import pytest

import scene
from tests.test_gpu_raster_fine_tiles import _eyes

pytestmark = pytest.mark.gpu


def _field(views, grid, disk):
    side = math.isqrt(views - 1) + 1
    return scene.build_light_field(scene.sphere_scene(3, 8, forward_cone_deg=35.0), scene.cap_grid_directions(side, 40.0)[:views],
                                   64, 64, 90.0, grid, disk_scale=disk)


# strips, halves and whole tiles side by side; first, last and only images of a form; odd sizes
@pytest.mark.parametrize("sizes", [(48, 1250), (1250, 48), (300, 1250, 31, 700), (200, 200, 1, 1600), (17, 1100)])
@pytest.mark.parametrize("views,grid,disk,oval", [(16, 33, 1.2, False), (40, 17, 6.0, True), (9, 70, 1.2, False)])
@pytest.mark.parametrize("tile,fmt", [((16, 16), "f32"), ((32, 8), "u8"), ((32, 8), "bf16"), ((16, 16), "fp8"), ((8, 8), "f32")])
def test_images_of_several_sizes_draw_the_inspection_images(sizes, views, grid, disk, oval, tile, fmt):
    torch = pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm
    from paper_1810_08860_gb300 import disks

    lf = _field(views, grid, disk)
    r = lfm.Renderer(0, tile=tile, max_eyes=4, tri_capacity=16 << 20)
    r.load_views(lf, tex_format=fmt)
    r.build_meshes(lf)
    if oval:
        r.set_disk_ovals(disks.oval_extents(lf))
    E = [_eyes(k + 1, w, max(1, w - 5), 0.45 * w)[k] for k, w in enumerate(sizes)]
    want = [r.render_inspect(e, max_records=1)["rgba"] for e in E]
    for got in (r.render(E), r.render_batch(E)):
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    r.close()


@pytest.mark.parametrize("form", ["render", "render_batch"])
@pytest.mark.parametrize("sizes", [(48, 1200), (1200, 48), (96, 1600)])
def test_a_small_image_does_not_hold_a_large_one_up(sizes, form):
    """In one call they take less than in two (0.7 of it measured; drawing whole tiles of both 1.2 to 2)."""
    torch = pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm

    lf = _field(16, 33, 1.2)
    r = lfm.Renderer(0, max_eyes=4)
    r.load_views(lf)
    r.build_meshes(lf)
    E = [_eyes(1, w, w, 0.45 * w)[0] for w in sizes]
    out = [torch.empty((e.height, e.width, 4), device="cuda") for e in E]

    def time(k):
        best = float("inf")
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            getattr(r, form)([E[i] for i in k], out=[out[i] for i in k])
            torch.cuda.synchronize()
            a.record()
            for _ in range(20):
                getattr(r, form)([E[i] for i in k], out=[out[i] for i in k])
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / 20)
        return best

    both, one, other = time([0, 1]), time([0]), time([1])
    r.close()
    assert both < one + other, (both, one, other)

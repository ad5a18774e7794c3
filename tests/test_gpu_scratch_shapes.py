"""Per-call scratch follows from the number of eyes and screen tiles, not from the images' shapes:
after one call, a call of as many tiles in another shape allocates nothing, so it can be captured."""
import pytest

import scene
from tests.test_gpu_raster_fine_tiles import _eyes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warm,shape", [((640, 320), (320, 640)), ((320, 640), (640, 320)), ((512, 512), (16, 16384)),
                                        ((512, 512), (16384, 16)), ((1, 32767), (32767, 1)), ((32767, 1), (1, 32767))])
@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 8)])
def test_another_shape_of_as_many_tiles_can_be_captured(warm, shape, tile):
    torch = pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm

    tiles = lambda s: -(-s[0] // tile[0]) * -(-s[1] // tile[1])  # noqa: E731
    if tiles(shape) > tiles(warm):
        warm = (warm[0], tile[1] * -(-tiles(shape) // -(-warm[0] // tile[0])))  # rows of tiles enough
    assert tiles(shape) <= tiles(warm) and max(warm) <= 32767
    lf = scene.build_light_field(scene.sphere_scene(3, 8, forward_cone_deg=35.0), scene.cap_grid_directions(3, 40.0),
                                 64, 64, 90.0, 17)
    r = lfm.Renderer(0, tile=tile)
    r.load_views(lf)
    r.build_meshes(lf)
    r.render(_eyes(1, *warm, 100.0))
    E = _eyes(1, *shape, 100.0)
    out = [torch.zeros((shape[1], shape[0], 4), device="cuda")]
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=torch.cuda.Stream()):
        r.render(E, out=out)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(r.render(E)[0], out[0])
    r.close()

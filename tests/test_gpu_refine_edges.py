"""The per-layer convolutions and the weight gradients at the edges of their tiles
(30 x 16 outputs, 32 x 8 positions, groups of four pixels per store), at one pixel
and one row, and with more tiles per block than its ring has stages, against the
FP64 oracle with the tolerances of test_gpu_refine.py."""
import numpy as np
import pytest

from oracle import refine
from tests.test_gpu_refine import _bf16_weights, _check_forward, _params, _smooth_image

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 1), (1, 1, 40), (2, 40, 1), (2, 7, 29), (1, 8, 30), (1, 9, 31), (1, 16, 32), (3, 17, 33), (1, 33, 61),
         (2, 15, 65), (4, 256, 256)]


def _renderer(params):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm

    r = lfm.Renderer(0)
    r.load_refiner(params(lfm))
    r.set_refine_kernel("layers")
    return r


@pytest.mark.parametrize("n,h,w", SIZES)
def test_layers_and_gradients_at_tile_edges(n, h, w):
    r = _renderer(lambda lfm: _params(lfm, 21))
    import torch

    params = r.get_refiner()["params"]
    rng = np.random.default_rng(h * 1000 + w)
    x = np.stack([_smooth_image(rng, h, w, invalid=0.1 if h * w > 100 else 0.0) for _ in range(n)])
    t = x.copy()
    t[..., :3] += (0.15 * np.sin(np.arange(w)[None, None, :, None] * 0.3 + np.arange(h)[None, :, None, None] * 0.2)
                   + 0.05).astype(np.float32)
    t *= x[..., 3:]
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t.astype(np.float32)).cuda()
    if h * w * n < 100000:
        _check_forward(r.refine(xd).cpu().numpy(), list(x), params)
    r.refine_gradients(xd, td)
    st = r.get_refiner()
    r.close()
    loss, g = refine.loss_and_grad(list(x.astype(np.float64)), list(t.astype(np.float64)), _bf16_weights(params))
    assert abs(st["loss"] - loss) <= 2e-2 * loss
    k = 0
    for name, shape in refine.SHAPES:
        m = int(np.prod(shape))
        a, b = st["grad"][k:k + m].astype(np.float64), g[k:k + m]
        k += m
        rel = np.linalg.norm(a - b) / np.linalg.norm(b)
        cos = float(a @ b / (np.linalg.norm(a) * np.linalg.norm(b)))
        assert rel < 5e-2 and cos > 0.998, (name, rel, cos)

"""The order of the weight gradients' sums is part of their result (the tensor core truncates as
it adds, and Adam turns a last bit into another BF16 weight some steps later), so gradients and
weights are held to the bits that the kernels before the present ones gave for the same inputs:
chains of accumulation, three per SM, that take every n-th chunk of 32 x 2 pixels row by row.
The digests are of those kernels, on a chip of 152 SMs."""
import hashlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# images, height, width: digests of the gradient of one call, and of the weights after four steps.
# One chunk; partial chunks and chains of one; several chunks per chain; every chain of the chip.
DIGESTS = {
    (1, 1, 1): ("ee9ce40e36b38c6f", "2b35162e3680fd06"),
    (2, 7, 29): ("1b22cd3d9379ffff", "dd6630f8d4312bad"),
    (3, 17, 33): ("c14dcec85c6407ee", "a51aa1e7cf769b91"),
    (2, 15, 65): ("dedcf09ce3cb6056", "5c40d5a02d5c6567"),
    (7, 100, 90): ("5359a6ac04208142", "7ca9d4d339dd93da"),
    (1, 517, 731): ("15e74ece6a496c21", "16b2c8f937896005"),
    (16, 256, 256): ("5b2d5ad2a3f84e71", "4c79b623fbb04f48"),
}


def _inputs(n, h, w):
    rng = np.random.default_rng(n * 1000000 + h * 1000 + w)
    x = (rng.integers(0, 256, (n, h, w, 4)) / 255.0).astype(np.float32)
    x[..., 3] = rng.integers(0, 20, (n, h, w)) > 0
    x[..., :3] *= x[..., 3:]
    t = x.copy()
    t[..., :3] = (x[..., :3] * np.float32(0.875) + np.float32(0.03125)) * x[..., 3:]
    return x, t


def _params(lfm):
    """Weights of the size of an initialisation, from integers: the same on every machine."""
    rng = np.random.default_rng(7)
    p = rng.integers(-255, 256, lfm.REFINE_N_PARAMS).astype(np.float32) / np.float32(1024)
    p[10144:] /= np.float32(16)
    return p


def _digest(a):
    return hashlib.sha256(np.ascontiguousarray(a).tobytes()).hexdigest()[:16]


@pytest.mark.parametrize("size", list(DIGESTS))
def test_gradients_and_weights_keep_their_bits(size):
    torch = pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm

    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the number of chains follows the number of SMs")
    x, t = (torch.from_numpy(a).cuda() for a in _inputs(*size))
    r = lfm.Renderer(0)
    r.load_refiner(_params(lfm))
    r.refine_gradients(x, t)
    grad = _digest(r.get_refiner()["grad"])
    for _ in range(4):
        r.refine_train_step(x, t, 1e-3)
    params = _digest(r.get_refiner()["params"])
    r.close()
    assert (grad, params) == DIGESTS[size]

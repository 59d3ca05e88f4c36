"""The surrogate's kernels at the edges of their ranges, against the FP64
oracle: one mode, modes up to the Nyquist frequency, odd mode counts, grid
sides between the powers of two.

Transforms: an output passes six contractions of at most 64 terms per layer,
each with FP32 rounding (2^-24 a term, adding as a random walk), so about
6 * 8 * 6e-8 = 3e-6 of its norm a layer; two layers and the gradient's second
pass give 1e-5 and 2e-5."""
import numpy as np
import pytest

from oracle import fno_oracle as F
from test_gpu_fno import env, make, rel  # noqa: F401 (env is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 2, 1, 1), (8, 2, 4, 1), (12, 4, 3, 1), (16, 2, 8, 2), (20, 4, 5, 1),
                                   (28, 2, 7, 2), (32, 2, 16, 1), (36, 4, 9, 1), (40, 2, 8, 1), (60, 2, 30, 1),
                                   (64, 2, 32, 1)])
def test_transforms_at_every_bound(env, shape):  # noqa: F811
    torch, S = env
    n, C, M, L = shape
    net, flat = make(env, shape)
    sh = F.Shape(n, C, M, L)
    rng = np.random.default_rng(n * M)
    x = rng.normal(size=(4, n, n, n)).astype(np.float32)
    xd = torch.from_numpy(x).cuda()
    y = torch.empty((3, n, n, n), device="cuda")
    dy = rng.normal(size=(3, n, n, n)).astype(np.float32)
    net.forward(xd, y)
    net.grad.zero_()
    net.backward(xd, torch.from_numpy(dy).cuda())
    torch.cuda.synchronize()
    y_o, cache = F.forward(flat, x, sh)
    assert rel(y.cpu().numpy(), y_o) < 1e-5
    go = F.unpack(F.backward(flat, cache, dy.astype(np.float64), sh), sh)
    gg = F.unpack(net.grad.cpu().numpy(), sh)
    for key in ("P", "p", "Q", "q"):
        assert rel(gg[key], go[key]) < 2e-5, key
    for key in ("W", "b", "R"):
        for l in range(L):
            assert rel(gg[key][l], go[key][l]) < 2e-5, (key, l)

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


@pytest.mark.parametrize("N,n,shift", [(256, 4, 0), (192, 12, 0), (80, 20, 0), (80, 20, 1), (96, 8, 0), (60, 10, 0)])
def test_upsampling_in_one_pass(env, N, n, shift):  # noqa: F811
    """Factors 4 to 64, quads of fine cells that straddle a change of taps
    (factor 12), sides that leave part of a CTA idle; an output off the
    16-byte boundary takes the three passes. 12 products a value: 1e-6."""
    torch, S = env
    y = torch.from_numpy(np.random.default_rng(N + n).normal(size=(3, n, n, n)).astype(np.float32)).cuda()
    scale = torch.tensor([1.7, 0.0, 0.0, 0.0], device="cuda")
    H = torch.zeros(3 * N ** 3 + 4, device="cuda")[shift:shift + 3 * N ** 3].view(3, N, N, N)
    S.upsample(y, N, n, scale, H, torch.cuda.current_stream())
    torch.cuda.synchronize()
    want = torch.from_numpy(F.upsample(y.cpu().numpy().astype(np.float64), N, float(scale[0]))).cuda()
    assert float((H.double() - want).norm() / want.norm()) < 1e-6


@pytest.mark.parametrize("N,n,shift", [(40, 10, 0), (36, 12, 0), (36, 12, 1), (30, 10, 0), (256, 4, 0), (16, 16, 0)])
def test_block_means(env, N, n, shift):  # noqa: F811
    """Wide and narrow loads, one to 64 cells a side: sums of up to 64^3 cells
    in threads' and rows' partial sums, 1e-6."""
    torch, S = env
    g = torch.Generator().manual_seed(N)
    a, b = ((torch.randn(2 * N ** 3 + 4, generator=g) + 1).cuda()[shift:shift + 2 * N ** 3].view(2, N, N, N) for _ in "ab")
    c = torch.empty((2, n, n, n), device="cuda")
    scale = torch.tensor([1.7, 0.0, 0.0, 0.0], device="cuda")
    f = N // n
    for fine2 in (None, b):
        S.coarsen(a, N, n, 2, c, scale, torch.cuda.current_stream(), fine2=fine2)
        torch.cuda.synchronize()
        v = a.double() if fine2 is None else 0.5 * (a.double() + b.double())
        want = v.view(2, n, f, n, f, n, f).mean(dim=(2, 4, 6)) / float(scale[0])
        assert float((c.double() - want).norm() / want.norm()) < 1e-6

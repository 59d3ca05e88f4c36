"""Weight and bias gradients of a channel mixing: a CTA sums a tile of 64
voxels by itself before it adds it to its other tiles, so that on any path a
value goes through 64 additions and one per tile, not 64 per tile.

The gradient is nonzero, and constant, on every 152nd tile alone, those of one
CTA: equal addends are the worst case of a chain, as their roundings add up
instead of averaging out. Bound: the additions on the path, 2^-24 each."""
import pytest

from test_gpu_fno import env  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a", [0.1, 0.3, 0.7, 1.1])
def test_sums_of_one_cta(env, a):  # noqa: F811
    torch, S = env
    n, C, CH, CTAS = 64, 32, 64, 152
    net = S.FNO(n, C, 2, 1, seed=0)
    # one layer that passes channel 0 through: W = 1, no spectral part, Q[0][0] = 1
    par = torch.zeros_like(net.params)
    W0 = 5 * C
    par[W0:W0 + C * C] = torch.eye(C, device="cuda").flatten()
    Q0 = net.count - 3 - 3 * C
    par[Q0] = 1.0
    net.load(par)
    xs = [0.37, 1.9, 0.011, 5.3]
    x = torch.empty(4, n, n, n, device="cuda")
    for c in range(4):
        x[c] = xs[c]
    y = torch.empty(3, n, n, n, device="cuda")
    dy = torch.zeros(3, n ** 3, device="cuda")
    tiles = dy.view(3, -1, CH)[0, ::CTAS]
    tiles.fill_(a)
    m = tiles.numel()
    net.forward(x, y)
    net.backward(x, dy.view(3, n, n, n))
    torch.cuda.synchronize()
    g = net.grad.double().cpu()
    av = float(dy.max())
    ntile = m // CH
    bias, weight = (2 + CH // 4 + ntile) * 2.0 ** -24, (CH + ntile) * 2.0 ** -24
    for k in (4 * C, W0 + C * C, net.count - 3):  # lift, layer, projection: the bias of channel 0
        assert abs(float(g[k]) / (m * av) - 1) <= bias
    for c in range(4):  # lift weights of channel 0
        assert abs(float(g[c]) / (m * av * float(x[c, 0, 0, 0])) - 1) <= weight

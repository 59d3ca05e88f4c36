"""Every tap of the gather's ball counts. The acceleration mesh is set so that
each tap of the ball about one cell adds about as much to the force as any
other (the inverse of its Gaussian weight at the cell's centre, times a random
value), and the cells just outside the ball would add more: a row that is
dropped, given to the wrong lane or cut one tap short or long then shows at the
level of one tap, 4e-5 of the sum or more, against a bound of 1e-5:

per term, in units of 2^-24, 5 roundings of the exponent times its size (at most
13.3), 12 for three expf, 6 for their normalisation, 3 products, and 66 fused
adds, 5 steps of a warp and 8 warps at most on its way: 167, 1e-5 of the sum
(all terms are positive)."""
import numpy as np
import pytest

import oracle
from paper_2312_02968_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BOUND = 167 * 2.0 ** -24


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2312_02968_gb300 import binding

    return binding


def gather_from(B, n, sigma, cell, off, mesh):
    """Deposit accumulator of the particles, and their force from `mesh` [3, n, n, n]."""
    N = len(cell)
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in
         (cell.astype(np.int32), off.astype(np.float32), np.zeros((N, 3), np.float32), np.ones(N, np.float32))]
    h = B.MondPM(n, 1, float(n), 1.0, 1.0, B.MU_DEEP, sigma, N)
    h.bind_particles(*t)
    h.deposit()
    acc, ka = h.get_deposit_acc()
    h.solve_field(1)
    h.sync()

    class Mesh:  # the handle's own acceleration mesh
        __cuda_array_interface__ = {"shape": (3, n, n, n), "typestr": "<f4", "version": 3,
                                    "data": (h.field_ptr(B.FIELD_ACC), False)}

    torch.as_tensor(Mesh(), device="cuda").copy_(torch.from_numpy(mesh))
    torch.cuda.synchronize()
    g = h.gather().cpu().numpy().astype(np.float64)
    h.close()
    return acc.cpu().numpy().view(np.uint64), ka, g


@pytest.mark.parametrize("N", [3, 40])  # listed one by one; worked on from the staged tile
@pytest.mark.parametrize("cell", [(13, 18, 15), (1, 30, 0)])  # inside; across the faces
@pytest.mark.parametrize("sigma", [0.75, 1.0, 1.1, 1.25, 1.4, 1.5, 1.75, 1.9, 2.0])  # reach 2 to 7
def test_every_tap_counts(B, sigma, cell, N):
    n = 32
    rng = np.random.default_rng([int(100 * sigma), N])
    r = int(4 * sigma) + 1  # past the ball on every side
    d = np.arange(-r, r + 1)
    d2 = d[:, None, None] ** 2 + d[None, :, None] ** 2 + d[None, None, :] ** 2
    value = np.exp(d2 / (2 * sigma ** 2)) * rng.uniform(0.5, 1.5, (3,) + d2.shape)
    mesh = np.zeros((3, n, n, n), np.float32)
    at = [(c + d) % n for c in cell]
    mesh[np.ix_(range(3), at[2], at[1], at[0])] = value
    off = rng.uniform(-0.5, 0.5, (N, 3)).astype(np.float32)
    cells = np.tile(np.array(cell, np.int32), (N, 1))
    _, _, g = gather_from(B, n, sigma, cells, off, mesh)
    want = oracle.gather(sigma, mesh.astype(np.float64), cells, off.astype(np.float64))
    assert np.all(np.abs(g / want - 1) <= BOUND)


@pytest.mark.parametrize("sigma", [1.0, 1.5, 2.0])
def test_a_list_longer_than_the_warps(B, sigma):
    """More listed particles than the grid has warps: two entries at a time."""
    n, N = 128, 6000
    p = W.uniform_random(n, N, seed=11)
    per_tile = np.unique(p["cell"] // 8, axis=0, return_counts=True)[1]
    assert per_tile.max() < 16  # all are listed
    rng = np.random.default_rng(12)
    mesh = rng.uniform(0.5, 1.5, (3, n, n, n)).astype(np.float32)
    acc, ka, g = gather_from(B, n, sigma, p["cell"], p["offset"], mesh)
    ref, ka_ref, _ = oracle.deposit_fixed(n, sigma, p["cell"], p["offset"], np.ones(N, np.float32))
    assert ka == ka_ref and np.array_equal(acc, ref)
    want = oracle.gather(sigma, mesh.astype(np.float64), p["cell"], p["offset"].astype(np.float64))
    assert np.all(np.abs(g / want - 1) <= BOUND)

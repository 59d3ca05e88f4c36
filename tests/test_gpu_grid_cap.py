"""A cap on the CTAs of a step changes no bit of it: systems whose particles
are all listed one by one (fewer than 16 a tile), in numbers around the CTAs
that the GPU holds, down to a cap of one CTA."""
import numpy as np
import pytest

from paper_2312_02968_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sigma", [1.0, 2.0])
@pytest.mark.parametrize("N", [40, 152, 153, 200, 304, 305])
def test_cap_and_listed_particles(N, sigma):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2312_02968_gb300 import binding as B

    n = 64
    p = W.uniform_random(n, N, seed=N)
    t = [torch.from_numpy(np.ascontiguousarray(p[k])).cuda() for k in ("cell", "offset", "vel", "mass")]
    torch.cuda.synchronize()
    h = B.MondPM(n, 1, float(n), 1.0, 1.0, B.MU_DEEP, sigma, N)
    h.bind_particles(*t)
    want = None
    for cap in (0, 152, 40, 1):
        h.set_option(B.OPT_GRID_CAP, cap)
        h.deposit()
        h.solve_field(1)
        acc, _ = h.get_deposit_acc()
        got = (acc, h.gather())
        torch.cuda.synchronize()
        want = want or got
        assert all(torch.equal(a, b) for a, b in zip(want, got)), cap
    assert torch.isfinite(want[1]).all() and want[1].abs().max() > 0
    h.close()

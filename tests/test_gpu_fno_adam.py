"""One Adam step with the bfloat16 copy of the parameters, against torch."""
import ctypes

import numpy as np
import pytest

from test_gpu_fno import env  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,shift,size", [(1, 0, 1.0), (3, 0, 1.0), (4, 0, 1.0), (1027, 0, 1.0), (1027, 1, 1.0),
                                              (2_500_001, 0, 1.0), (2_500_001, 3, 1.0), (70_000, 0, 1e25),
                                              (70_000, 0, 1e-22), (70_000, 0, np.inf)])
def test_adam_and_the_bfloat16_copy(env, count, shift, size):  # noqa: F811
    """Vectors of four and their remainder, arrays off the 16-byte boundary,
    gradients whose squares leave FP32. The norm is exact to FP64 rounding of
    a few thousand partial sums (1e-12); parameters to a few FP32 roundings;
    the copy is the cast of the parameters, bit for bit."""
    torch, S = env
    from paper_2312_02968_gb300.binding import lib

    gen = torch.Generator().manual_seed(count + shift)
    mk = lambda: torch.randn(count + shift, generator=gen).cuda()[shift:]
    p, g, m, v = mk(), mk(), mk(), mk().abs()
    if np.isinf(size):
        g[count // 2] = float("inf")
    else:
        g *= size
    pb = torch.zeros(count + shift, dtype=torch.bfloat16, device="cuda")[shift:]
    norm2 = torch.zeros(1, dtype=torch.float64, device="cuda")
    p0, m0, v0, g0 = (t.double().clone() for t in (p, m, v, g))
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib().mond_fno_adam_cast(count, ptr(p), ptr(g), ptr(m), ptr(v), 1e-2, 0.9, 0.99, 1e-6, 3, 2.5, ptr(norm2),
                                    ptr(pb), st) == 0
    torch.cuda.synchronize()
    assert float(g.abs().max()) == 0.0
    assert torch.equal(pb, p.to(torch.bfloat16))
    if np.isinf(size):
        assert torch.equal(p.double(), p0) and torch.equal(m.double(), m0) and torch.equal(v.double(), v0)
        return
    want = float((g0 * g0).sum())
    assert float(norm2) == pytest.approx(want, rel=1e-12)
    gi = g0 * min(1.0, 2.5 / want ** 0.5)
    mi = 0.9 * m0 + 0.1 * gi
    vi = 0.99 * v0 + 0.01 * gi * gi
    pi = p0 - 1e-2 * (mi / (1 - 0.9 ** 3)) / ((vi / (1 - 0.99 ** 3)).sqrt() + 1e-6)
    for a, b in ((p, pi), (m, mi), (v, vi)):
        assert torch.allclose(a.double(), b, rtol=1e-5, atol=1e-6)

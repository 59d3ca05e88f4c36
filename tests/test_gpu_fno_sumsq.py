"""The sum of squares that normalises the surrogate's loss, input and gradient,
against the exact sum (the squares are exact in FP64, math.fsum adds them
without rounding). Few values: FP64 throughout, at most the additions on a
value's way (four values and a remainder, five steps of a warp, its CTA's eight
warps, the CTAs), 2^-53 each. From 65536 on FP32 pairs, about 48 bits each."""
import ctypes
import math

import pytest

from test_gpu_fno import env  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spread", [0.0, 3.0])
@pytest.mark.parametrize("count", [1, 7, 64, 1000, 65535, 65536, 100003])
def test_sum_of_squares(env, count, spread):  # noqa: F811
    torch, S = env
    from paper_2312_02968_gb300.binding import lib

    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    ctas = (count + 1023) // 1024
    bound = (4 + 1 + 5 + 7 + ctas) * 2.0 ** -53 if count < 65536 else 2.0 ** -45
    for seed in range(8):
        x = torch.randn(count, generator=torch.Generator().manual_seed(seed))
        x = torch.exp(spread * x) if spread else x
        t = x.cuda()
        assert t.data_ptr() % 16 == 0
        y, dy = torch.zeros_like(t), torch.empty_like(t)
        acc = torch.zeros(2, dtype=torch.float64, device="cuda")
        assert lib().mond_fno_loss(count, ptr(y), ptr(t), ptr(dy), 1.0, ptr(acc), st) == 0
        torch.cuda.synchronize()
        assert abs(float(acc[1]) / math.fsum((x.double() ** 2).tolist()) - 1) <= bound

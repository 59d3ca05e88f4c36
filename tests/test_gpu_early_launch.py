"""Kernels that start before the one ahead of them has completed: results of a
chain run at one go, behind kernels of another library on the same stream, are
those of the same chain with a synchronisation after every call, bit for bit
(the solver has no unordered floating-point sum on this path)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16, 96, 128])
def test_chain_equals_synchronised_chain(n):
    import torch

    import __graft_entry__

    __graft_entry__.build()
    from paper_2312_02968_gb300 import binding as B

    st = torch.cuda.Stream()
    N = 5000
    g = torch.Generator().manual_seed(n)
    with torch.cuda.stream(st):
        src = torch.randint(n // 4, 3 * n // 4, (N, 3), generator=g, dtype=torch.int32).cuda()
        cell = torch.zeros_like(src)
        off = (torch.rand((N, 3), generator=g) - 0.5).cuda()
        vel = torch.zeros((N, 3), device="cuda")
        mass = (torch.rand(N, generator=g) / N).cuda()
        acc = torch.empty((3, n, n, n), device="cuda")
        big = torch.zeros(1 << 26, device="cuda")
        h = B.MondPM(n, 1, float(n), 1.0, 1.0, B.MU_DEEP, 1.0, N, stream=st)
        h.bind_particles(cell, off, vel, mass)

        def chain(sync):
            outs = []
            for shift in (0, 1, 2):
                big.add_(1.0)  # keeps the stream busy, so that the next kernels queue up behind
                torch.add(src, shift, out=cell)
                for call in (h.deposit, lambda: h.solve_field(3), lambda: h.get_field(B.FIELD_ACC, acc)):
                    call()
                    if sync:
                        h.sync()
                        st.synchronize()
                outs.append(acc.clone())
            st.synchronize()
            return [o.cpu().numpy() for o in outs]

        want = chain(True)
        for _ in range(3):
            for a, b in zip(want, chain(False)):
                assert np.isfinite(a).all() and np.abs(a).max() > 0
                assert np.array_equal(a, b)

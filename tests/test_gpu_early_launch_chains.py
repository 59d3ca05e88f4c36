"""Chains whose kernels start before the one ahead of them has completed, as
test_gpu_early_launch does it for single calls of the solver: the surrogate's
inference, captured steps and a batch. Here a call has many launches, so the
other side is a process that waits for the GPU after every one
(CUDA_LAUNCH_BLOCKING) and takes its steps directly. Bit for bit: no float is
added in no order on these paths."""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu

NETS = [(16, 8, 4, 3), (32, 32, 16, 2), (48, 32, 12, 2), (64, 32, 16, 4)]
SYSTEMS = [(48, 8000), (64, 20000), (96, 30000)]


def chains(blocked):
    import torch

    import __graft_entry__

    __graft_entry__.build()
    from paper_2312_02968_gb300 import binding as B
    from paper_2312_02968_gb300 import surrogate as S
    from paper_2312_02968_gb300 import workloads as W

    out = {}
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        big = torch.zeros(1 << 26, device="cuda")
        for i, shape in enumerate(NETS):
            n, N = shape[0], 4 * shape[0]
            net = S.FNO(*shape, seed=i, stream=st)
            net.params.mul_(3.0)
            net.cast()
            gen = torch.Generator().manual_seed(i)
            fine = torch.randn((4, N, N, N), generator=gen).cuda()
            x, y = torch.empty((4, n, n, n), device="cuda"), torch.empty((3, n, n, n), device="cuda")
            H, scale = torch.empty((3, N, N, N), device="cuda"), torch.full((4,), 0.7, device="cuda")
            st.synchronize()
            for rep in range(2):
                big.add_(1.0)  # the launches queue up behind this one
                fine.mul_(1.5)
                S.coarsen(fine, N, n, 4, x, scale, st)
                net.forward(x, y)
                S.upsample(y, N, n, scale, H, st)
                st.synchronize()
                out[f"y{i}{rep}"], out[f"H{i}{rep}"] = y.cpu().numpy().copy(), H[:, ::3].cpu().numpy().copy()
    for how in ("graph", "batch"):
        hs = []
        for i, (n, N) in enumerate(SYSTEMS):
            p = W.isothermal(n, 1.0, N, n / 32, 0.4 * n, seed=i)
            s = torch.cuda.Stream()
            t = [torch.from_numpy(np.ascontiguousarray(p[k])).cuda() for k in ("cell", "offset", "vel", "mass")]
            torch.cuda.synchronize()
            h = B.MondPM(n, 1, float(n), 1.0, 1.0, B.MU_DEEP, 1.0, N, stream=s)
            h.bind_particles(*t)
            if how == "graph" and not blocked:
                h.set_option(B.OPT_USE_GRAPH, 1)
            hs.append((h, t))
        if how == "batch" and not blocked:
            b = B.Batch([h for h, _ in hs])
            b.step(0.5, n_steps=3, n_iter=3)
            b.sync()
            b.close()
        else:
            for h, _ in hs:
                for _ in range(3):
                    h.step(0.5, 3, B.WARM_NONE)
            for h, _ in hs:
                h.sync()
        for i, (h, t) in enumerate(hs):
            for k, a in zip(("cell", "offset", "vel"), t):
                out[f"{how}{i}{k}"] = a.cpu().numpy()
            h.close()
    return out


def test_chains_equal_those_of_a_process_that_waits(tmp_path):
    path = str(tmp_path / "blocked.npz")
    subprocess.run([sys.executable, os.path.abspath(__file__), path], check=True, cwd=ROOT, timeout=600,
                   env=dict(os.environ, CUDA_LAUNCH_BLOCKING="1", PYTHONPATH=ROOT))
    want = np.load(path)
    got = chains(False)
    assert sorted(want.files) == sorted(got)
    for k in want.files:
        assert np.isfinite(want[k]).all() and np.abs(want[k]).max() > 0
        assert np.array_equal(want[k], got[k]), k


if __name__ == "__main__":
    np.savez(sys.argv[1], **chains(True))

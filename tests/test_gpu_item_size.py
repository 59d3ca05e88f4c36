"""Particles per work item: the option's value exactly, the default 1024 or
fewer as the number of particles asks; the autotuner times no size twice."""
import numpy as np
import pytest

from paper_2312_02968_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2312_02968_gb300 import binding

    return binding


def make(B, n, p):
    t = [torch.from_numpy(np.ascontiguousarray(p[k])).cuda() for k in ("cell", "offset", "vel", "mass")]
    torch.cuda.synchronize()
    h = B.MondPM(n, 1, float(n), 1.0, 1.0, B.MU_DEEP, 1.0, len(p["mass"]), stream=torch.cuda.Stream())
    h.bind_particles(*t)
    return h


@pytest.mark.parametrize("option,size", [(None, 64), (1024, 64), (256, 256), (512, 512), (4096, 4096)])
def test_items_have_the_size_asked_for(B, option, size):
    n = 32
    p = W.isothermal(n, 1.0, 30000, 2.0, 12.0, seed=5)  # a default item of this many particles holds 64
    h = make(B, n, p)
    if option:
        h.set_option(B.OPT_CHUNK, option)
    h.deposit()
    h.sync()
    c = p["cell"] // 8
    per_tile = np.bincount((c[:, 2] * 4 + c[:, 1]) * 4 + c[:, 0], minlength=64)
    whole = per_tile[per_tile >= 16]
    want = [int((whole // size).sum()), int((whole % size > 0).sum()), int(per_tile[per_tile < 16].sum())]
    assert want[0] > 0
    # the list's three counters, in the handle's small tables at the front of its workspace
    base = -h.workspace.data_ptr() % 256
    front = h.workspace[base:base + (1 << 16)].view(torch.int32).cpu().numpy()
    assert any(front[i:i + 3].tolist() == want for i in range(len(front) - 2))
    h.close()


def test_autotune_leaves_out_what_the_default_stands_for(B):
    n = 32
    rng = np.random.default_rng(2)
    timed = []
    for N in (30000, 400000):  # default items of 64 and of 512
        p = W.uniform_random(n, N, seed=int(rng.integers(1 << 30)))
        h = make(B, n, p)
        h.step(0.0, 1, 0)
        l0 = h.kernel_launches()
        h.step(0.0, 1, 0)
        per_step = h.kernel_launches() - l0
        h.set_option(B.OPT_PIPELINED, 0)
        l0 = h.kernel_launches()
        h.step(0.0, 1, 0)
        per_step += h.kernel_launches() - l0
        h.set_option(B.OPT_PIPELINED, 1)
        l0 = h.kernel_launches()
        B.autotune(h, 1, 1)
        timed.append((h.kernel_launches() - l0) / (2 * per_step))
        h.close()
    assert timed == [4.0, 3.0]

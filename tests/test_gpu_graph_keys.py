"""A captured step is replayed only for what it was captured from: after an
option that changes the launches, or a binding of other arrays under the same
cell array and particle count, a captured step and a batch give what direct
steps give, bit for bit."""
import numpy as np
import pytest

from paper_2312_02968_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N_SIDE, N = 64, 20000


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2312_02968_gb300 import binding

    return binding


def system(B):
    p = W.isothermal(N_SIDE, 1.0, N, 2.0, 25.0, seed=7)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        h = B.MondPM(N_SIDE, 1, float(N_SIDE), 1.0, 1.0, B.MU_DEEP, 1.0, N, stream=st)
        t = [torch.from_numpy(np.ascontiguousarray(p[k])).cuda() for k in ("cell", "offset", "vel", "mass")]
    torch.cuda.synchronize()
    h.bind_particles(*t)
    return h, t


class Direct:
    def __init__(self, B, h):
        self.h = h

    def step(self):
        self.h.step(0.5, 4, 0)
        self.h.sync()


class Graph(Direct):
    def __init__(self, B, h):
        super().__init__(B, h)
        h.set_option(B.OPT_USE_GRAPH, 1)


class InBatch(Direct):
    def __init__(self, B, h):
        super().__init__(B, h)
        self.b = B.Batch([h])

    def step(self):
        self.b.step(0.5, n_steps=1, n_iter=4)
        self.b.sync()


def run(B, how, change):
    h, t = system(B)
    d = how(B, h)
    d.step()
    t = change(B, h, t)
    d.step()
    torch.cuda.synchronize()
    out = [x.cpu().numpy().copy() for x in t[:3]]
    if how is InBatch:
        d.b.close()
    h.close()
    return out


def cycle_mean(B, h, t):
    h.set_option(B.OPT_CYCLE_MEAN, 1)
    return t


def no_fold(B, h, t):
    h.set_option(B.OPT_FOLD, 0)
    return t


def rebind(B, h, t):
    """The same cell array and count, other offsets, velocities and masses
    (larger by a power of two: another fixed-point scale). The old arrays are
    spoilt and kept alive, so that a step on them would show and do no harm."""
    new = [t[0], t[1].clone(), t[2].clone(), t[3] * 64.0]
    t[1].zero_()
    t[2].zero_()
    torch.cuda.synchronize()
    h.bind_particles(*new)
    h.spoilt = t
    return new


@pytest.mark.parametrize("how", [Graph, InBatch])
@pytest.mark.parametrize("change", [cycle_mean, no_fold, rebind])
def test_change_after_the_capture(B, how, change):
    want = run(B, Direct, change)
    got = run(B, how, change)
    plain = run(B, Direct, lambda B, h, t: t)
    assert not np.array_equal(want[2], plain[2])  # the change matters
    for a, b in zip(want, got):
        assert np.array_equal(a, b)

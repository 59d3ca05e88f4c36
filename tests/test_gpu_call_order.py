"""Calls out of order are refused before anything is launched: a solve of a
density set directly makes the fields but no binning, and a binning is good for
the particles it was made of, where they were."""
import numpy as np
import pytest

from paper_2312_02968_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N_SIDE = 32


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2312_02968_gb300 import binding

    return binding


def system(B, N=3000):
    p = W.isothermal(N_SIDE, 1.0, max(N, 1), 2.0, 12.0, seed=3)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        h = B.MondPM(N_SIDE, 1, float(N_SIDE), 1.0, 1.0, B.MU_DEEP, 1.0, max(N, 1), stream=st)
        t = [torch.from_numpy(np.ascontiguousarray(p[k][:N])).cuda() for k in ("cell", "offset", "vel", "mass")]
    torch.cuda.synchronize()
    h.bind_particles(*t)
    return h, t


def refused(B, call):
    with pytest.raises(B.MondError) as e:
        call()
    assert e.value.code == -8  # MOND_ESTATE


def set_and_solve(h):
    h.set_density(torch.rand((N_SIDE,) * 3, device="cuda"))
    torch.cuda.synchronize()
    h.solve_field(2)


def test_particle_calls_without_a_binning(B):
    h, t = system(B)
    set_and_solve(h)
    for call in (h.gather, lambda: h.half_kick(0.1), lambda: h.gather_push(0.1)):
        refused(B, call)
    h.deposit()
    set_and_solve(h)  # the binning of this deposit still holds
    assert torch.isfinite(h.gather()).all()
    h.gather_push(0.1)
    set_and_solve(h)  # the particles have moved
    refused(B, h.gather)
    h.deposit()
    h.bind_particles(*[x[:100].contiguous() for x in t])
    set_and_solve(h)  # other particles
    refused(B, h.gather)
    h.sync()
    h.close()


def test_no_particles_and_a_density(B):
    h, _ = system(B, 0)
    set_and_solve(h)
    h.half_kick(0.1)
    h.gather_push(0.1)  # (a push ends the solve's validity)
    h.sync()
    h.close()


@pytest.mark.parametrize("how", ["graph", "batch"])
def test_a_replay_ends_a_solve_as_a_step_does(B, how):
    h, t = system(B)
    if how == "graph":
        h.set_option(B.OPT_USE_GRAPH, 1)
        step = lambda: h.step(0.5, 2)
    else:
        b = B.Batch([h])
        step = lambda: (b.step(0.5, n_steps=1, n_iter=2), b.sync())
    step()  # captured and run
    h.deposit()
    h.solve_field(1)
    assert torch.isfinite(h.gather()).all()
    step()  # replayed: the particles have moved
    refused(B, h.gather)
    refused(B, lambda: h.solve_field(1))
    assert h.diagnostics()["n_iter_done"] == 2
    if how == "batch":
        b.step(0.5, n_steps=0, n_iter=3)  # captured, not run
        assert h.diagnostics()["n_iter_done"] == 2
        b.close()
    h.close()


def test_a_capture_that_fails_leaves_nothing_behind(B):
    # the workspace of a handle that has never binned holds whatever was there
    junk = torch.full((B.workspace_bytes(N_SIDE, 1, 1.0, 3000) + 256,), 0x5A, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    del junk
    h, t = system(B)
    h.set_option(B.OPT_USE_GRAPH, 1)
    h.set_option(B.OPT_CYCLE_MEAN, 1)
    h.set_option(B.OPT_PIPELINED, 0)
    refused(B, lambda: h.step(0.5, 2))  # the mean needs the other passes: after the deposit was captured
    refused(B, lambda: h.solve_field(2))  # no deposit has run
    h.set_option(B.OPT_PIPELINED, 1)
    h.step(0.5, 2)
    h.sync()
    h2, t2 = system(B)
    h2.set_option(B.OPT_CYCLE_MEAN, 1)
    h2.step(0.5, 2)
    h2.sync()
    for a, b in zip(t, t2):
        assert torch.equal(a, b)
    h.close()
    h2.close()

"""The deposit and the gather at the edges of their work lists and sums: tiles
just below and above the sparse limit, cells with more particles than one
register sum takes, masses of alternating binades and of shifts past 32 bits,
systems of a few particles, and kernel widths between the widest of a reach.

The deposit is an exact integer rule: equal to the oracle's. The gather reads
the solver's own mesh in FP32, so it is compared with the FP64 ball sum of that
mesh: at most 3 |ball| roundings of 2^-24, relative to the sum of the terms'
sizes (the forces on lone particles cancel inside the ball).
"""
import numpy as np
import pytest

import oracle
from paper_2312_02968_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def particles(kind, n, rng):
    if kind == "edges":  # tiles of 15, 16 and 17 particles, one of 1100, wrapping corners
        pos = []
        for i, k in enumerate((15, 16, 17, 1100)):
            pos.append(rng.uniform(-0.5, 7.49, (k, 3)) + np.array([8 * i, 8 * (i % 2), 0.0]))
        pos.append(rng.uniform(-0.5, 0.5, (9, 3)) + n - 1)
        p = np.concatenate(pos)
        mass = rng.uniform(0.5, 1.0, len(p)).astype(np.float32)
    elif kind == "pile":  # 700 particles in one cell and its neighbour, one binade
        p = np.concatenate([rng.uniform(-0.5, 0.49, (700, 3)), rng.uniform(-0.5, 0.49, (40, 3)) + [1, 0, 0]]) + 13.0
        mass = rng.uniform(0.5, 0.999, len(p)).astype(np.float32)
    elif kind == "binades":  # equal cells, masses spread over 40 binades: shifts on both sides of 32
        p = rng.uniform(-0.5, 3.49, (900, 3)) + 5.0
        mass = np.ldexp(rng.uniform(0.5, 1.0, len(p)), -rng.integers(0, 40, len(p))).astype(np.float32)
    else:  # a few
        p = rng.uniform(-0.5, n - 0.51, (3, 3))
        mass = np.array([1.0, 0.25, 3.0], np.float32)
    cell = np.floor(p + 0.5)
    off = (p - cell).astype(np.float32)
    cell = np.mod(cell.astype(np.int64), n).astype(np.int32)
    return {"cell": np.ascontiguousarray(cell), "offset": np.ascontiguousarray(off),
            "vel": np.zeros((len(p), 3), np.float32), "mass": mass}


@pytest.mark.parametrize("sigma", [0.75, 1.0, 1.1, 1.5, 1.75, 2.0])
@pytest.mark.parametrize("kind", ["edges", "pile", "binades", "few"])
def test_deposit_and_gather_at_the_edges_of_the_work_lists(kind, sigma):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_02968_gb300 import binding as B

    n = 32
    p = particles(kind, n, np.random.default_rng([int(100 * sigma), len(kind)]))
    t = [torch.from_numpy(p[k]).cuda() for k in ("cell", "offset", "vel", "mass")]
    h = B.MondPM(n, 1, float(n), 1.0, 1.0, B.MU_SIMPLE, sigma, len(p["mass"]))
    h.bind_particles(*t)
    h.deposit()
    acc, ka = h.get_deposit_acc()
    ref, ka_ref, _ = oracle.deposit_fixed(n, sigma, p["cell"], p["offset"], p["mass"])
    assert ka == ka_ref and np.array_equal(acc.cpu().numpy().view(np.uint64), ref)
    h.solve_field(1)
    mesh = h.get_field(B.FIELD_ACC).cpu().numpy().astype(np.float64)
    g = h.gather().cpu().numpy().astype(np.float64)
    want = oracle.gather(sigma, mesh, p["cell"], p["offset"].astype(np.float64))
    size = oracle.gather(sigma, np.abs(mesh), p["cell"], p["offset"].astype(np.float64))
    taps = sum(1 for i in np.ndindex(17, 17, 17) if sum((v - 8) ** 2 for v in i) < 16 * sigma ** 2)
    assert np.all(np.abs(g - want) <= 3 * taps * 2.0 ** -24 * size)
    h.close()

"""What the MOND particle-mesh framework is used for, as cases that can be timed and compared.

A case is one call, or one short chain of calls, of the package's public entry
points (``binding.MondPM``, ``binding.Batch``, ``surrogate``) on a system of a
given size. The kinds:

  step     one leapfrog step, mond_pm_step, replayed as a CUDA graph
  force    deposit, field solve and gather: the forces of one configuration
  solve    the field solve of a mesh density, read back with get_field
  deposit  binning and mass deposit alone, the integer accumulator read back
  gather   the forces at the particles from a solved mesh
  batch    several independent systems stepped as one CUDA graph
  infer    the surrogate: features of g_N, forward pass, upsampled guess of H
  train    one training step of the surrogate: forward, loss, backward, Adam

``exact`` restates each in plain torch, 64 bits: complex FFTs of which the real
part is kept, Gaussian sums over the ball of taps, the network through autograd.
"""
from __future__ import annotations

import math

import torch

from paper_2312_02968_gb300 import binding as B
from paper_2312_02968_gb300 import surrogate as S

MU = {"deep": B.MU_DEEP, "simple": B.MU_SIMPLE, "standard": B.MU_STANDARD, "newton": B.MU_NEWTON}
LR = 7e-4
CLIP = 5.0


def listed():
    return [
        # two equal masses on a circular orbit, zero-padded domain, widest kernel of the test systems
        dict(name="two_body_128", kind="step", n=64, pad=2, N=2, sigma=2.0, mu="simple", shape="binary", K=4, mean=False,
             warm=False),
        # the smallest system of an ensemble run: every launch counts
        dict(name="member_64", kind="force", n=64, pad=1, N=10007, sigma=1.0, mu="deep", shape="isothermal", K=4,
             mean=False),
        # a large, cold Plummer system of an ensemble run
        dict(name="member_192", kind="force", n=192, pad=1, N=400009, sigma=1.0, mu="standard", shape="plummer", K=4,
             mean=False),
        # the benchmark's step: a million particles of an isothermal sphere
        dict(name="isothermal_256", kind="step", n=256, pad=1, N=1000000, sigma=1.5, mu="deep", shape="isothermal", K=4,
             mean=True, warm=False),
        # the same system advanced with one iteration from the previous step's H
        dict(name="isothermal_256_warm", kind="step", n=256, pad=1, N=1000000, sigma=1.5, mu="deep", shape="isothermal",
             K=1, mean=False, warm=True),
        # a central mass with a ring of 1e5 particles on the largest mesh
        dict(name="ring_512", kind="step", n=512, pad=1, N=100001, sigma=1.0, mu="deep", shape="ring", K=4, mean=False,
             warm=False),
        # deposit and gather of the ten-million-particle mixtures of the learned warm start
        dict(name="mixture_deposit_256", kind="deposit", n=256, pad=1, N=10000000, sigma=1.0, mu="standard",
             shape="mixture"),
        dict(name="mixture_gather_256", kind="gather", n=256, pad=1, N=10000000, sigma=1.0, mu="standard",
             shape="mixture", K=4, mean=True),
        # the solve of a density given on a mesh whose side is not a power of two
        dict(name="density_96", kind="solve", n=96, pad=1, mu="simple", K=3, mean=False),
        # an ensemble: systems of uneven sides and particle counts, one graph per step
        dict(name="ensemble_8", kind="batch", sides="64,96,128,192,64,128,96,192", K=4,
             counts="10007,33331,250007,100003,500009,20011,150001,300007"),
        # the surrogate at its default network grid guesses H for a 256^3 solve
        dict(name="fno_infer_64", kind="infer", n=256, fno=64),
        # and is trained on the benchmark's network grid
        dict(name="fno_train_32", kind="train", fno=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "force", "force", "solve", "deposit", "gather", "batch", "infer", "train"])
    if kind == "infer":
        f = rng.choice([16, 24, 32, 48, 64])
        return dict(kind=kind, n=rng.choice([128, 192, 256] if f not in (24, 48) else [192, 384]), fno=f)
    if kind == "train":
        return dict(kind=kind, fno=rng.choice([32, 36, 40, 48, 56, 64]))
    if kind == "batch":
        m = rng.randint(2, 8)
        return dict(kind=kind, sides=",".join(str(rng.choice([64, 96, 128, 192])) for _ in range(m)),
                    counts=",".join(str(_log(rng, 1e4, 5e5)) for _ in range(m)), K=rng.choice([2, 3, 4]))
    mu = rng.choice(["deep", "simple", "standard"])
    if kind == "solve":
        return dict(kind=kind, n=rng.choice([32, 48, 64, 96, 128, 192, 256, 384]), pad=1, mu=mu, K=rng.randint(0, 4),
                    mean=False)
    n, pad = rng.choice([(32, 1), (48, 1), (64, 1), (96, 1), (128, 1), (192, 1), (256, 1), (384, 1), (48, 2), (64, 2),
                         (96, 2), (128, 2)])
    sigma = rng.choice([1.0, 1.0, 1.25, 1.5, 2.0])
    taps = 4.0 / 3.0 * math.pi * (4 * sigma) ** 3
    top = 2e9 / taps if kind in ("deposit", "gather") else 1e9 / taps
    c = dict(kind=kind, n=n, pad=pad, N=_log(rng, 1e3, min(1e7, top, 4.0 * n ** 3)), sigma=sigma, mu=mu,
             shape=rng.choice(["isothermal", "plummer", "mixture", "uniform"]))
    if kind != "deposit":
        K = rng.randint(1, 4)
        c.update(K=K, mean=K >= 3 and rng.random() < 0.5)
    if kind == "step":
        c["warm"] = rng.random() < 0.3
    return c


# --------------------------------------------------------------------- inputs
def _dev():
    return torch.device("cuda", torch.cuda.current_device())


_streams = {}


def _stream():
    """The stream a program drives its systems on (graphs need one that is not the default)."""
    d = _dev().index
    if d not in _streams:
        _streams[d] = torch.cuda.Stream()
    return _streams[d]


def _gen(seed, k=0):
    g = torch.Generator(device=_dev())
    g.manual_seed((int(seed) * 1000003 + k) & 0x7FFFFFFFFFFFFFFF)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=_dev(), dtype=torch.float64)


def _directions(g, N):
    u, ph = 2 * _rand(g, N) - 1, 2 * math.pi * _rand(g, N)
    w = torch.sqrt(1 - u * u)
    return torch.stack([w * torch.cos(ph), w * torch.sin(ph), u], 1)


def _particles(shape, n, nf, N, seed):
    """Positions (pixels from the domain's centre), velocities and masses, FP64."""
    g = _gen(seed)
    lim = 0.4 * n
    dev = _dev()
    vel = torch.zeros(N, 3, device=dev, dtype=torch.float64)
    mass = torch.full((N,), 1.0 / max(N, 1), device=dev, dtype=torch.float64)

    def cut(x, f):  # radii by inverse cumulative mass, those outside redrawn
        r = f(x)
        for _ in range(64):
            bad = ~(r <= lim)
            if not bool(bad.any()):
                break
            r = torch.where(bad, f(_rand(g, N)), r)
        return torch.clamp(r, max=lim)

    if shape == "binary":  # seed: the phase of the orbit
        ph = 2 * math.pi * float(_rand(g, 1).item())
        d = torch.tensor([math.cos(ph), math.sin(ph), 0.0], device=dev, dtype=torch.float64)
        t = torch.tensor([-math.sin(ph), math.cos(ph), 0.0], device=dev, dtype=torch.float64)
        v = math.sqrt((2.0 / 3.0) * 2.0 / (1.0 + math.sqrt(0.5)))
        pos = torch.stack([8.0 * d, -8.0 * d])
        return pos, torch.stack([0.5 * v * t, -0.5 * v * t]), torch.full((2,), 0.5, device=dev, dtype=torch.float64)
    if shape == "ring":  # a central mass 1, the rest a ring of mass 0.1 and radius 64 of 512 pixels, jittered by 1/4 px
        m = 0.1 / (N - 1)
        r = n / 8.0
        ang = 2 * math.pi * torch.arange(N - 1, device=dev, dtype=torch.float64) / (N - 1)
        v = math.sqrt((2.0 / 3.0) * math.sqrt(1.1) * (1.0 / (1.0 + math.sqrt(1 / 1.1)) + math.sqrt(1 / 1.1)))
        pos = torch.zeros(N, 3, device=dev, dtype=torch.float64)
        pos[1:] = torch.stack([r * torch.cos(ang), r * torch.sin(ang), 0 * ang], 1) + 0.5 * (_rand(g, N - 1, 3) - 0.5)
        vel[1:] = torch.stack([-v * torch.sin(ang), v * torch.cos(ang), 0 * ang], 1)
        mass = torch.full((N,), m, device=dev, dtype=torch.float64)
        mass[0] = 1.0
        return pos, vel, mass
    if shape == "isothermal":
        b = n / 32.0
        r = cut(_rand(g, N), lambda x: b * (1.0 / torch.sqrt(torch.clamp(x, min=1e-300)) - 1.0) ** (-2.0 / 3.0))
        vel = torch.randn(N, 3, generator=g, device=dev, dtype=torch.float64) * math.sqrt(2.0 / 9.0)
        return _directions(g, N) * r[:, None], vel, mass
    if shape == "plummer":
        a = n / 16.0
        r = cut(_rand(g, N), lambda x: a / torch.sqrt(torch.clamp(x, 1e-12, 1 - 1e-12) ** (-2.0 / 3.0) - 1.0))
        return _directions(g, N) * r[:, None], vel, mass
    if shape == "mixture":
        sp = _spheres(n, seed)
        which = torch.multinomial(sp["mass"], N, replacement=True, generator=g)
        a, kind = sp["radius"][which], sp["kind"][which]
        x = torch.clamp(_rand(g, N), 1e-12, 0.97)
        r = torch.where(kind == 0, a / torch.sqrt(x ** (-2.0 / 3.0) - 1.0), a * torch.sqrt(x) / (1.0 - torch.sqrt(x)))
        pos = sp["centre"][which] + _directions(g, N) * torch.clamp(r, max=lim)[:, None]
        return torch.clamp(pos, -(n / 2 - 8.0), n / 2 - 8.5), vel, mass * float(sp["mass"].sum())
    pos = (_rand(g, N, 3) - 0.5) * (n if nf == n else 0.9 * n)  # uniform, periodic when there is no padding
    return pos, 0.05 * torch.randn(N, 3, generator=g, device=dev, dtype=torch.float64), mass * (0.5 + _rand(g, N))


def _spheres(n, seed):
    """A mixture of 1-8 Plummer (kind 0) and Hernquist (kind 1) spheres."""
    g = _gen(seed, 7)
    K = 1 + int(torch.randint(0, 8, (1,), generator=g, device=_dev()).item())
    kind = torch.randint(0, 2, (K,), generator=g, device=_dev())
    mass = torch.exp(math.log(1e-2) * _rand(g, K))
    radius = (4.0 + 28.0 * _rand(g, K)) * (n / 256.0)
    reach = torch.clamp(0.4 * n - 3 * radius, min=0.0)
    return {"kind": kind, "mass": mass, "radius": radius, "centre": (2 * _rand(g, K, 3) - 1) * reach[:, None]}


def _mesh_radius(n, sp, j):
    c = torch.arange(n, device=_dev(), dtype=torch.float64) - n / 2
    d = [c - sp["centre"][j, a] for a in range(3)]
    x, y, z = d[0][None, None, :], d[1][None, :, None], d[2][:, None, None]
    return x, y, z, torch.sqrt(x * x + y * y + z * z)


def _mixture_rho(n, seed):
    """The density of a mixture on an n^3 mesh, FP32 [z][y][x]."""
    sp = _spheres(n, seed)
    rho = torch.zeros(n, n, n, device=_dev(), dtype=torch.float64)
    for j in range(len(sp["mass"])):
        _, _, _, r = _mesh_radius(n, sp, j)
        a, m = sp["radius"][j], sp["mass"][j]
        if int(sp["kind"][j]) == 0:
            rho += 3 * m / (4 * math.pi * a ** 3) * (1 + (r / a) ** 2) ** -2.5
        else:
            q = torch.clamp(r, min=0.5)
            rho += m * a / (2 * math.pi * q * (q + a) ** 3)
    return rho.float()


def _mixture_gn(n, seed):
    """The Newtonian field of a mixture of Plummer spheres on an n^3 mesh, FP32 [3][z][y][x]."""
    sp = _spheres(n, seed)
    g = torch.zeros(3, n, n, n, device=_dev(), dtype=torch.float64)
    for j in range(len(sp["mass"])):
        x, y, z, r = _mesh_radius(n, sp, j)
        f = -sp["mass"][j] / (r * r + sp["radius"][j] ** 2) ** 1.5
        for a, d in enumerate((x, y, z)):
            g[a] += f * d
    return g.float().contiguous()


def _tensors(case, seed):
    """The particle arrays a program hands over: cell, offset, velocity, mass."""
    nf = case["n"] * case["pad"]
    pos, vel, mass = _particles(case["shape"], case["n"], nf, case["N"], seed)
    p = pos + nf / 2
    cell = torch.floor(p + 0.5)
    off = (p - cell).float()
    return [torch.remainder(cell, nf).to(torch.int32).contiguous(), off.contiguous(), vel.float().contiguous(),
            mass.float().contiguous()]


def _system(case, seed):
    t = _tensors(case, seed)
    torch.cuda.synchronize()
    h = B.MondPM(case["n"], case["pad"], float(case["n"]), 1.0, 1.0, MU[case["mu"]], case["sigma"], case["N"],
                 stream=_stream())
    h.bind_particles(*t)
    if case.get("mean"):
        h.set_option(B.OPT_CYCLE_MEAN, 1)
    return h, t


def _members(case):
    sides, counts = ([int(v) for v in case[k].split(",")] for k in ("sides", "counts"))
    for i, (n, N) in enumerate(zip(sides, counts)):
        yield dict(n=n, pad=1, N=N, sigma=1.0, mu=("deep", "standard")[i % 2], shape=("isothermal", "plummer")[i % 2])


def _net(case, seed):
    """A network with parameters of its initial distribution, made from the seed."""
    n, C, M, L = case["fno"], 32, min(16, case["fno"] // 2), 4
    net = S.FNO(n, C, M, L, device=_dev(), stream=_stream())
    p = _params(n, C, M, L, seed)
    with torch.cuda.stream(net.stream):
        net.load(p)
    return net


def _params(n, C, M, L, seed):
    g = _gen(seed, 3)
    K = M * (2 * M) * (2 * M)

    def u(scale, *shape):
        return scale * (2 * torch.rand(*shape, generator=g, device=_dev()) - 1).reshape(-1)

    parts = [u(0.5, C, 4), u(0.1, C)]
    for _ in range(L):
        parts += [u(C ** -0.5, C, C), u(0.1, C), u(1.0 / C ** 2, K, C, C, 2)]
    parts += [u(C ** -0.5, 3, C), u(0.1, 3)]
    return torch.cat(parts)


def _pair(case, seed):
    """One training pair: smooth fields of the network's grid, x [4][n^3] and the target t [3][n^3]."""
    n = case["fno"]
    x = torch.cat([_mixture_gn(n, seed), torch.zeros(1, n, n, n, device=_dev())])
    x[:3] /= x[:3].double().square().mean().sqrt().float()
    x[3] = 0.25 * torch.log10(x[:3].double().norm(dim=0) + 1e-12).float()
    return x.contiguous(), (0.3 * torch.roll(x[:3], 1, 0) * torch.sqrt(x[:3].norm(dim=0))).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind}
    if kind == "batch":
        sms = torch.cuda.get_device_properties(_dev()).multi_processor_count
        st["systems"] = []
        for i, c in enumerate(_members(case)):
            h, t = _system(c, seed * 64 + i)
            h.set_option(B.OPT_GRID_CAP, sms)
            st["systems"].append((h, t))
        st["batch"] = B.Batch([h for h, _ in st["systems"]], stream=_stream())
    elif kind == "infer":
        n, f = case["n"], case["fno"]
        st["net"] = _net(case, seed)
        st["gN"] = _mixture_gn(n, seed)
        st["x"] = torch.empty(4, f, f, f, device=_dev())
        st["y"] = torch.empty(3, f, f, f, device=_dev())
        st["scale"] = torch.empty(4, device=_dev())
        st["H"] = torch.empty(3, n, n, n, device=_dev())
        st["scratch"] = torch.empty(int(B.lib().mond_fno_output_scratch_bytes(n, f)), dtype=torch.uint8, device=_dev())
    elif kind == "train":
        st["net"] = _net(case, seed)
        st["x"], st["t"] = _pair(case, seed)
        st["y"], st["dy"] = torch.empty_like(st["t"]), torch.empty_like(st["t"])
    elif kind == "solve":
        n = case["n"]
        st["rho"] = _mixture_rho(n, seed)
        st["h"] = B.MondPM(n, 1, float(n), 1.0, 1.0, MU[case["mu"]], 1.0, 1, stream=_stream())
        st["acc"] = torch.empty(3, n, n, n, device=_dev())
    else:
        st["h"], st["t"] = _system(case, seed)
        h = st["h"]
        if kind == "step":
            h.set_option(B.OPT_USE_GRAPH, 1)
        elif kind == "gather":
            h.deposit()
            h.solve_field(case["K"])
        if kind in ("force", "gather"):
            st["g"] = torch.empty(case["N"], 3, device=_dev())
    torch.cuda.synchronize()
    return st


# ----------------------------------------------------------------------- runs
def run(st):
    case, kind = st["case"], st["kind"]
    with torch.cuda.stream(_stream()):
        if kind == "step":
            h, (cell, off, vel, _) = st["h"], st["t"]
            h.step(0.25, case["K"], B.WARM_PREV if case["warm"] else B.WARM_NONE)
            return {"vel": vel, "pos": cell + off}
        if kind == "force":
            h = st["h"]
            h.deposit()
            h.solve_field(case["K"])
            return {"force": h.gather(st["g"])}
        if kind == "solve":
            h = st["h"]
            h.set_density(st["rho"])
            h.solve_field(case["K"])
            return {"acc": h.get_field(B.FIELD_ACC, st["acc"])}
        if kind == "deposit":
            h = st["h"]
            h.deposit()
            return {"acc": h.get_deposit_acc()[0]}
        if kind == "gather":
            return {"force": st["h"].gather(st["g"])}
        if kind == "batch":
            st["batch"].step(0.25, 1, case["K"])
            return [{"vel": vel, "pos": cell + off} for _, (cell, off, vel, _) in st["systems"]]
        net = st["net"]
        if kind == "infer":
            n, f, stream = case["n"], case["fno"], net.stream
            S.features(st["gN"], n, f, 1.0, st["x"], st["scale"], stream)
            net.forward(st["x"], st["y"])
            S.upsample(st["y"], n, f, st["scale"], st["H"], stream, st["scratch"])
            return {"y": st["y"], "H": st["H"]}
        net.forward(st["x"], st["y"])
        net.loss(st["y"], st["t"], st["dy"])
        net.backward(st["x"], st["dy"])
        net.adam(LR, clip=CLIP)
        return {"y": st["y"], "params": net.params, "m": net.m, "v": net.v}


# ----------------------------------------------------------------------- work
def _taps(sigma):
    r = int(4 * sigma) + 1
    return sum(1 for x in range(-r, r + 1) for y in range(-r, r + 1) for z in range(-r, r + 1)
               if x * x + y * y + z * z < 16 * sigma * sigma)


def _fft_flops(n, transforms):
    return transforms * 2.5 * n ** 3 * 3 * math.log2(n)


def _solve_flops(n, K, warm=False):
    """One real transform forward and one inverse for each of the three components on both sides of each projection."""
    return _fft_flops(n, 4 if K == 0 else 4 + 12 * (K - 1) + 6 + (9 if warm else 0))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        every = [work(dict(c, kind="step", K=case["K"], warm=False)) for c in _members(case)]
        return {k: sum(w[k] for w in every) for k in ("bytes", "flops")}
    if kind in ("infer", "train"):
        n = case["fno"]
        M = min(16, n // 2)
        P = 4 * 2 * 1024 * 4 * M ** 3
        fwd = 4 * (32 * 2 * _fft_flops(n, 1) + 8 * 1024 * 4 * M ** 3 + 2 * 1024 * n ** 3) + 2 * 32 * 7 * n ** 3
        if kind == "infer":
            return {"bytes": 2 * P + 4 * 6 * case["n"] ** 3 + 4 * 3 * n ** 3, "flops": fwd + 24 * 3 * case["n"] ** 3}
        # the bf16 weights read twice and made once; parameters and moments read and written
        return {"bytes": 2 * P + 24 * P + 4 * 10 * n ** 3, "flops": 3 * fwd + 12 * P}
    if kind == "solve":
        n3 = case["n"] ** 3
        return {"bytes": 4 * n3 + 12 * n3, "flops": _solve_flops(case["n"], case["K"])}
    nf, N = case["n"] * case["pad"], case["N"]
    T = _taps(case["sigma"])
    if kind == "deposit":
        return {"bytes": 28 * N + 8 * nf ** 3, "flops": 2.0 * T * N}
    if kind == "gather":
        return {"bytes": 24 * N + 12 * N + 12 * nf ** 3, "flops": 6.0 * T * N}
    b = 40 * N + (12 if kind == "force" else 48) * N
    return {"bytes": b, "flops": 8.0 * T * N + _solve_flops(nf, case["K"], case.get("warm", False))}


# ---------------------------------------------------------------------- exact
def _waves(n):
    f = torch.fft.fftfreq(n, 1.0 / n, device=_dev(), dtype=torch.float64)
    k = 2 * math.pi * f / n
    kx, ky, kz = k[None, None, :], k[None, :, None], k[:, None, None]
    k2 = kx * kx + ky * ky + kz * kz
    A = torch.where(k2 > 0, 1.0 / torch.where(k2 > 0, k2, torch.ones_like(k2)), torch.zeros_like(k2))
    return (kx, ky, kz), A


def _nu(mu, F):
    f = torch.where(F > 0, F, torch.ones_like(F))
    if mu == "deep":
        v = 1.0 / torch.sqrt(f)
    elif mu == "simple":
        v = 0.5 + torch.sqrt(0.25 + 1.0 / f)
    else:
        v = torch.sqrt(0.5 + 0.5 * torch.sqrt(1.0 + 4.0 / (f * f)))
    return torch.where(F > 0, v, torch.zeros_like(v))


def _mu(mu, x):
    return x if mu == "deep" else x / (1 + x) if mu == "simple" else x / torch.sqrt(1 + x * x)


def _grad(phi):
    """-grad of phi by periodic central differences, [3][z][y][x]."""
    return torch.stack([-(torch.roll(phi, -1, 2 - a) - torch.roll(phi, 1, 2 - a)) / 2 for a in range(3)])


def _solve64(rho, mu, K, mean):
    """The iteration on a unit-pixel periodic mesh: the acceleration mesh, FP64."""
    n = rho.shape[0]
    k, A = _waves(n)
    gN = _grad(torch.fft.ifftn(-4 * math.pi * A * torch.fft.fftn(rho)).real)
    if K == 0:
        return gN
    H, last = None, None
    for j in range(1, K + 1):
        F = gN if H is None else gN + H
        gM = F * _nu(mu, F.square().sum(0).sqrt())
        del F
        s = 0
        for a in range(3):
            s = s + k[a] * torch.fft.fftn(gM[a])
        s = s * A
        if j == K:
            if mean and last is not None:
                s = 0.5 * (s + last)
            return _grad(torch.fft.ifftn(1j * s).real)
        last = s if j == K - 1 else None
        gM = torch.stack([torch.fft.ifftn(k[a] * s).real for a in range(3)])
        H = gM * _mu(mu, gM.square().sum(0).sqrt()) - gN
        del gM
        h = [torch.fft.fftn(H[a]) for a in range(3)]
        s = (k[0] * h[0] + k[1] * h[1] + k[2] * h[2]) * A
        for a in range(3):
            H[a] = torch.fft.ifftn(h[a] - k[a] * s).real
        del h, s


def _ball(sigma):
    r = int(4 * sigma) + 1
    return r, [(x, y, z) for z in range(-r, r + 1) for y in range(-r, r + 1) for x in range(-r, r + 1)
               if x * x + y * y + z * z < 16 * sigma * sigma]


def _weights(off, sigma, r):
    u = torch.arange(-r, r + 1, device=_dev(), dtype=torch.float64)[:, None, None] - off.double()[None]
    return torch.exp(-u * u / (2 * sigma * sigma)) / (sigma * math.sqrt(2 * math.pi))  # [2r+1][N][3]


def _sums(sigma, nf, cell, off, use):
    """use(index of the tap's mesh cell, weight) for each tap of the ball, in blocks of particles."""
    r, ball = _ball(sigma)
    for b in range(0, cell.shape[0], 2000000):
        c, w = cell[b:b + 2000000].long(), _weights(off[b:b + 2000000], sigma, r)
        row = None
        for x, y, z in ball:
            if row != (y, z):
                row = (y, z)
                base = (torch.remainder(c[:, 2] + z, nf) * nf + torch.remainder(c[:, 1] + y, nf)) * nf
                wyz = w[y + r, :, 1] * w[z + r, :, 2]
            use(slice(b, b + c.shape[0]), base + torch.remainder(c[:, 0] + x, nf), wyz * w[x + r, :, 0])


def _force64(case, seed):
    cell, off, vel, mass = _tensors(case, seed)
    nf, sigma = case["n"] * case["pad"], case["sigma"]
    rho = torch.zeros(nf ** 3, device=_dev(), dtype=torch.float64)
    m = mass.double()
    _sums(sigma, nf, cell, off, lambda p, i, w: rho.index_add_(0, i, w * m[p]))
    acc = _solve64(rho.view(nf, nf, nf), case["mu"], case["K"], case.get("mean")).view(3, -1)
    acc = acc.t().contiguous()
    g = torch.zeros(case["N"], 3, device=_dev(), dtype=torch.float64)

    def add(p, i, w):
        g[p] += w[:, None] * acc[i]

    _sums(sigma, nf, cell, off, add)
    return g, cell, off, vel


def _step64(case, seed):
    g, cell, off, vel = _force64(case, seed)
    nf = case["n"] * case["pad"]
    v = vel.double() + 0.25 * g
    p = cell.double() + off.double() + 0.25 * v
    return {"vel": v, "pos": torch.remainder(p + 0.5, nf) - 0.5}


def _unpack64(flat, n, C, M, L):
    K, at, out = M * 4 * M * M, 0, []
    for shape in [(C, 4), (C,)] + [(C, C), (C,), (K, C, C, 2)] * L + [(3, C), (3,)]:
        size = math.prod(shape)
        out.append(flat[at:at + size].view(*shape))
        at += size
    return out


def _net64(parts, x, n, M, L):
    """The network of the parameters `parts`: FP64 torch."""
    def pw(W, b, v):
        return torch.einsum("oi,izyx->ozyx", W, v) + b.view(-1, 1, 1, 1)

    at = torch.cat([torch.arange(M), torch.arange(n - M, n)]).to(x.device)
    v = pw(parts[0], parts[1], x)
    for l in range(L):
        W, b, R = parts[2 + 3 * l:5 + 3 * l]
        s = torch.fft.fftn(v, dim=(1, 2, 3))[:, at][:, :, at][:, :, :, :M].reshape(v.shape[0], -1)
        t = torch.einsum("kjc,jk->ck", torch.view_as_complex(R), s).reshape(-1, 2 * M, 2 * M, M)
        t = torch.cat([t[..., :1], 2 * t[..., 1:]], -1)  # the conjugate half of a real field
        full = torch.zeros(v.shape[0], n, n, n, dtype=torch.complex128, device=x.device)
        full = full.index_put((torch.arange(v.shape[0], device=x.device)[:, None, None, None],
                               at[None, :, None, None], at[None, None, :, None],
                               torch.arange(M, device=x.device)[None, None, None, :]), t)
        z = pw(W, b, v) + torch.fft.ifftn(full, dim=(1, 2, 3)).real
        v = torch.nn.functional.gelu(z, approximate="tanh") if l + 1 < L else z
    return pw(parts[-2], parts[-1], v)


def _features64(gN, n):
    N = gN.shape[1]
    f = N // n
    g = gN.double().view(3, n, f, n, f, n, f).mean((2, 4, 6))
    s = g.square().mean().sqrt()
    return torch.cat([g / s, (0.25 * torch.log10(g.square().sum(0).sqrt() + 1e-12))[None]]), s


def _upsample64(y, N):
    """Periodic cubic convolution (Keys, a = -1/2), cell centred, one axis after another."""
    n = y.shape[1]
    u = (torch.arange(N, device=_dev(), dtype=torch.float64) + 0.5) * n / N - 0.5
    i0 = torch.floor(u)
    u = u - i0
    w = [((-u + 2) * u - 1) * u / 2, ((3 * u - 5) * u * u + 2) / 2, ((-3 * u + 4) * u + 1) * u / 2, (u - 1) * u * u / 2]
    M = torch.zeros(N, n, device=_dev(), dtype=torch.float64)
    for a in range(4):
        M[torch.arange(N, device=_dev()), torch.remainder(i0.long() + a - 1, n)] += w[a]
    for _ in range(3):
        y = torch.einsum("ab,cxyb->caxy", M, y)
    return y


def exact(case, seed):
    kind = case["kind"]
    if kind == "deposit":
        return None  # whole numbers
    if kind == "solve":
        return {"acc": _solve64(_mixture_rho(case["n"], seed).double(), case["mu"], case["K"], case["mean"])}
    if kind == "step":
        return _step64(case, seed)
    if kind in ("force", "gather"):
        return {"force": _force64(case, seed)[0]}
    if kind == "batch":
        return [_step64(dict(c, K=case["K"]), seed * 64 + i) for i, c in enumerate(_members(case))]
    n, C, M, L = case["fno"], 32, min(16, case["fno"] // 2), 4
    p = _params(n, C, M, L, seed)
    w = p.to(torch.bfloat16).double()
    if kind == "infer":
        x, s = _features64(_mixture_gn(case["n"], seed), n)
        y = _net64(_unpack64(w, n, C, M, L), x, n, M, L)
        return {"y": y, "H": s * _upsample64(y, case["n"])}
    x, t = (v.double() for v in _pair(case, seed))
    w.requires_grad_(True)
    y = _net64(_unpack64(w, n, C, M, L), x, n, M, L)
    ((y - t).square().sum() / t.square().sum()).backward()
    g = w.grad * min(1.0, CLIP / float(w.grad.norm()))
    m, v = 0.1 * g, 0.001 * g * g
    step = (m / (1 - 0.9)) / (torch.sqrt(v / (1 - 0.999)) + 1e-8)
    return {"y": y.detach(), "params": p.double() - LR * step, "m": m, "v": v}

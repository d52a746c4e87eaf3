"""Timed cases of the PIC-MCC library: what its users run, through its public entry points.

Each case names one kind of work and its sizes:

  streamer   steps of a coupled simulation (push, collisions, deposit, field solve, weight updates), Cartesian or
             axisymmetric; the outputs are the fixed-point charge grids and the field the next step reads
  exchange   one step of electrons that live in host memory (upload, step in a given field, download)
  swarm      Monte Carlo swarms in uniform fields with their transport coefficients and per-step moments
  poisson    one stateless field solve on a charge density
  query      transport data from the network: features, then the network
  train      Adam steps of the network

Sizes are those of the repository's workloads, tests and benchmark.  Particles come back in an order that no run
repeats, so the particle cases return the charge grids, which hold every particle exactly.  Where the field solve
adds its block sums in float64 in no fixed order (float64 and axisymmetric runs), the fixed-point grids differ in
their last bits from run to run; those cases return the charge density in float64 instead.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2110_14494_gb300 import picmcc as P

E_CHARGE, M_ELECTRON, EPS0 = 1.602176634e-19, 9.1093837015e-31, 8.8541878128e-12
N_GAS = 2.45e25            # 1 bar at 300 K
AMU = 1.66053906660e-27
RTOL = 1e-6                # every coupled run's residual target


# ------------------------------------------------------------------ cases

def listed() -> list[dict]:
    return [
        # the benchmark's streamer: 20 um cells, 20 kV/cm, float32, ten steps between two looks at the grids
        dict(name="streamer_128", kind="streamer", nx=128, ny=128, nz=128, axi=False, precision=32, n=1_000_000,
             photo=False, steps=10),
        # the full-size streamer: 10 mm gap at 15.6 kV, photoionization
        dict(name="streamer_full", kind="streamer", nx=256, ny=256, nz=512, axi=False, precision=32, n=1_000_000,
             photo=True, steps=2),
        # the paper's axisymmetric geometry: 10 mm by 10 mm on (r, z), weight updates every ten steps
        dict(name="streamer_axi", kind="streamer", nx=512, ny=1, nz=512, axi=True, precision=32, n=100_000,
             photo=True, steps=10),
        # the plain float64 path that float32 results are judged against, on a small box
        dict(name="streamer_64_f64", kind="streamer", nx=64, ny=64, nz=64, axi=False, precision=64, n=100_000,
             photo=False, steps=2),
        # host-resident electrons: a small, odd-sized box (the tests' grid), where latency and launches count
        dict(name="exchange_small", kind="exchange", nx=24, ny=20, nz=28, precision=32, n=5_000),
        # ... and a million of them on the benchmark's grid
        dict(name="exchange_1m", kind="exchange", nx=128, ny=128, nz=128, precision=32, n=1_000_000),
        # the surrogate's training data: 256 values of E/N at once
        dict(name="swarm_batch", kind="swarm", swarms=256, n0=10_000, precision=32, steps=60, batched=True),
        # the plain float64 swarm at 120 Td, resampled to about its initial size
        dict(name="swarm_f64", kind="swarm", swarms=1, n0=10_000, precision=64, steps=300, batched=False),
        # a field solve in float64 on an uneven box, to the accuracy the tests ask for
        dict(name="poisson_f64", kind="poisson", nx=64, ny=48, nz=80, precision=64, electrode=True, rtol=1e-10),
        # the float-pair solve of the benchmark's grid
        dict(name="poisson_pair_128", kind="poisson", nx=128, ny=128, nz=128, precision=32, electrode=True,
             rtol=RTOL),
        # transport data for every cell and face of a large fluid run
        dict(name="query_16m", kind="query", n=1 << 24),
        # fitting the network to 4096 swarms
        dict(name="train_4096", kind="train", n=4096, steps=100),
    ]


def _log(rng, lo: float, hi: float) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng) -> dict:
    kind = rng.choice(["streamer", "streamer", "streamer", "exchange", "swarm", "poisson", "poisson", "query", "train"])
    if kind == "streamer":
        n = int(_log(rng, 2e4, 1e6))
        if rng.random() < 0.3:
            return dict(kind=kind, nx=32 * rng.randint(2, 16), ny=1, nz=32 * rng.randint(2, 16), axi=True,
                        precision=rng.choice([32, 32, 64]), n=min(n, 100_000), photo=rng.random() < 0.5,
                        steps=rng.randint(1, 10))
        prec = rng.choice([32, 32, 32, 64])
        top = 10 if prec == 32 else 5
        nx, ny, nz = (16 * rng.randint(2, top) for _ in range(3))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, axi=False, precision=prec, n=n if prec == 32 else min(n, 100_000),
                    photo=rng.random() < 0.5, steps=rng.randint(1, 6) if prec == 32 else 1)
    if kind == "exchange":
        nx, ny, nz = (int(_log(rng, 6, 128)) for _ in range(3))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=rng.choice([32, 32, 64]), n=int(_log(rng, 33, 1e6)))
    if kind == "swarm":
        if rng.random() < 0.5:
            return dict(kind=kind, swarms=1, n0=int(_log(rng, 500, 20_000)), precision=rng.choice([32, 64]),
                        steps=rng.randint(40, 200), batched=False)
        return dict(kind=kind, swarms=int(_log(rng, 2, 256)), n0=int(_log(rng, 500, 10_000)),
                    precision=rng.choice([32, 32, 64]), steps=rng.randint(20, 50), batched=True)
    if kind == "poisson":
        if rng.random() < 0.3:  # odd sizes have a single level: small boxes
            nx, ny, nz = (rng.randrange(9, 24, 2) for _ in range(3))
        else:
            nx, ny, nz = (8 * rng.randint(2, 16) for _ in range(3))
        prec = rng.choice([32, 64])
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=prec, electrode=rng.random() < 0.7,
                    rtol=rng.choice([1e-6, 1e-8] if prec == 32 else [1e-6, 1e-10]))
    if kind == "query":
        return dict(kind=kind, n=int(_log(rng, 100, 1 << 24)))
    return dict(kind=kind, n=rng.choice([64 * rng.randint(1, 4), 256 * rng.randint(2, 32)]), steps=rng.randint(20, 200))


# ------------------------------------------------------------------ inputs

def _air() -> dict:
    """Seven-process N2/O2 gas (80:20) on 1000 log-spaced energies, analytic cross sections."""
    n_bins, lo, hi = 1000, 0.01, 1000.0
    eps = lo * np.power(hi / lo, np.arange(n_bins) / (n_bins - 1))

    def inelastic(scale, thr):
        x = np.maximum(eps / thr, 1.0)
        return scale * np.log(x) / x

    el = 1e-19 / np.sqrt(1.0 + eps / 10.0)
    sigma = np.stack([el, el, inelastic(2e-21, 6.2), inelastic(1.5e-20, 11.0), inelastic(6e-20, 15.6),
                      inelastic(7e-20, 12.06), 1.3e-22 * np.exp(-(eps - 6.5) ** 2 / (2 * 0.7 ** 2))])
    o2 = np.array([0, 1, 0, 0, 0, 1, 1])
    return dict(eps=eps, sigma=np.ascontiguousarray(sigma), kind=np.array([0, 0, 1, 1, 2, 2, 3], np.int32),
                threshold=np.array([0.0, 0.0, 6.2, 11.0, 15.6, 12.06, 0.0]),
                density=np.where(o2 == 1, 0.2, 0.8) * N_GAS,
                mass=np.where(o2 == 1, 31.9988, 28.0134) * AMU, species=o2.astype(np.int32), n_gas=N_GAS)


def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _streamer_geometry(c: dict) -> dict:
    """Cell size, voltage, needle and seed: the 128^3, full-size and axisymmetric workloads, scaled by the gap."""
    full = c["axi"] or c["nz"] >= 512
    dx = 10e-3 / 512 if full else 20e-6
    L = c["nz"] * dx
    length = 0.2 * L if full else 0.5e-3 / 2.56e-3 * L
    radius = max(0.02 * L if full else 0.1e-3 / 2.56e-3 * L, 2.1 * dx)
    return dict(dx=dx, L=L, v_top=(15.6e5 if full else 20e5) * L, length=length, radius=radius,
                seed_radius=min(1e-4, 0.1 * L))


def _needle(c: dict, q: dict) -> np.ndarray:
    """uint8 [nz][ny][nx]: cells whose centre lies in the rod hanging from the top plate or in its cap."""
    dx, L = q["dx"], q["L"]
    x = (np.arange(c["nx"]) + 0.5) * dx
    if c["axi"]:
        r2 = (x ** 2)[None, :]
    else:
        y = (np.arange(c["ny"]) + 0.5) * dx
        r2 = (x[None, :] - 0.5 * c["nx"] * dx) ** 2 + (y[:, None] - 0.5 * c["ny"] * dx) ** 2
    z = (np.arange(c["nz"]) + 0.5) * dx
    zcap = L - q["length"] + q["radius"]
    rod = (r2 <= q["radius"] ** 2)[None] & (z >= zcap)[:, None, None]
    cap = r2[None] + ((z - zcap) ** 2)[:, None, None] <= q["radius"] ** 2
    return (rod | cap).astype(np.uint8)


def _prepare_streamer(c: dict, seed: int) -> dict:
    q = _streamer_geometry(c)
    grid = dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], dx=q["dx"], origin=(0.0, 0.0, 0.0))
    extra = dict(photo_xi=0.075, photo_pq=4000.0) if c["photo"] else {}
    if c["axi"]:
        extra.update(geometry=1, weight_interval=10)
    cap = 20_000_000
    ctx = P.PicContext(_air(), grid, precision=c["precision"], capacity=int(1.6 * cap), seed=2110144940 + seed, dt=2e-12,
                       mask=_needle(c, q), n_ppc=75, w_min=1.0, growth_trigger=1.25, particle_cap=cap, boundary=1,
                       sort_interval=20, coupled=True, v_lo=0.0, v_hi=q["v_top"], v_mask=q["v_top"],
                       poisson_rtol=RTOL, poisson_max_cycles=200, adaptive_dt=True, **extra)
    n0 = 1e16 if c["axi"] else 1e19
    center = (0.0, 0.0, q["L"] - q["length"]) if c["axi"] else \
        (0.5 * c["nx"] * q["dx"], 0.5 * c["ny"] * q["dx"], q["L"] - q["length"])
    electrons = n0 * math.pi ** 1.5 * q["seed_radius"] ** 3
    ctx.seed_gaussian(n0, q["seed_radius"], center, max(electrons / c["n"], 1.0 if c["axi"] else 0.0))
    ctx.step(3)  # a running simulation: past the first solves, which start from no potential
    cells = c["nx"] * c["ny"] * c["nz"]
    rho = torch.empty(cells, dtype=torch.float64, device="cuda") if c["axi"] or c["precision"] == 64 else None
    return dict(ctx=ctx, rho=rho, q=[torch.empty(cells, dtype=torch.int64, device="cuda") for _ in range(3)],
                E=[torch.empty(cells, dtype=torch.float64, device="cuda") for _ in range(3)])


def _prepare_exchange(c: dict, seed: int) -> dict:
    dx, n = 2e-5, c["n"]
    shape = (c["nz"], c["ny"], c["nx"])
    grid = dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], dx=dx, origin=(1e-5, -2e-5, 0.0))
    real = torch.float32 if c["precision"] == 32 else torch.float64
    g = _gen(seed)
    # a field that varies smoothly over the box, around 80 Td
    ax = [(torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) / m for m in shape]
    field = []
    for _ in range(3):
        a = torch.rand(8, generator=g, device="cuda", dtype=torch.float64)
        f = 2e6 * torch.sin(2 * math.pi * ((1 + 2 * a[0]) * ax[0][:, None, None] + a[1])) \
            * torch.sin(2 * math.pi * ((1 + 2 * a[2]) * ax[1][None, :, None] + a[3])) \
            * torch.sin(2 * math.pi * ((1 + 2 * a[4]) * ax[2][None, None, :] + a[5])) + 1e6 * (a[6] - 0.5)
        field.append(f.to(torch.float32).contiguous())
    ctx = P.PicContext(_air(), grid, precision=c["precision"], capacity=4 * n + 4096, seed=7 + seed, dt=2e-12)
    ctx.set_field(*field)
    box = [m * dx for m in reversed(shape)]
    host = torch.empty((10, n), dtype=real).pin_memory()
    for d in range(3):
        lo = grid["origin"][d]
        u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 0.998 + 0.001
        host[d].copy_((lo + box[d] * u).to(real))
        host[3 + d].copy_((torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * 1e6).to(real))
        host[6 + d].zero_()
    host[9].copy_((1 + 99 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)).to(real))
    ids = torch.arange(n, dtype=torch.int64).pin_memory()
    back = torch.empty((10, 2 * n + 2048), dtype=real).pin_memory()
    back_ids = torch.empty(2 * n + 2048, dtype=torch.int64).pin_memory()
    cells = c["nx"] * c["ny"] * c["nz"]
    return dict(ctx=ctx, n=n, up=ctx.host_set([host[i] for i in range(10)] + [ids], n),
                down=ctx.host_set([back[i] for i in range(10)] + [back_ids], back_ids.numel()),
                q=[torch.empty(cells, dtype=torch.int64, device="cuda") for _ in range(3)])


def _prepare_swarm(c: dict, seed: int) -> dict:
    s = c["swarms"]
    EN = np.array([120.0]) if s == 1 else 10.0 * np.power(100.0, np.arange(s) / (s - 1))
    kw = dict(precision=c["precision"], n0=c["n0"], n_steps=c["steps"], dt=1e-12, kT_eV=1.0, seed=1 + 1000 * seed,
              want_moments=True, n_lo=c["n0"] // 2, n_hi=2 * c["n0"])
    if c["batched"]:  # resampling bounds of the training data; the launch shape that tuning gives for it
        kw.update(batched=True, n_lo=1000, n_hi=100_000, block=256, blocks_per_sm=3, warp_chunk=512, use_graph=1)
    return dict(gas=_air(), EN=EN, kw=kw)


def _poisson_inputs(c: dict, seed: int):
    shape = (c["nz"], c["ny"], c["nx"])
    h = 2.56e-3 / max(shape)
    g = _gen(seed)
    z, y, x = torch.meshgrid(*[(torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) / m for m in shape],
                             indexing="ij")
    at = 0.3 + 0.4 * torch.rand(3, generator=g, device="cuda", dtype=torch.float64)
    rho = torch.exp(-((x - at[0]) ** 2 + (y - at[1]) ** 2 + (z - at[2]) ** 2) / 0.02)
    rho += 0.1 * torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    mask = None
    if c["electrode"]:
        L = shape[0] * h
        q = dict(dx=h, L=L, length=0.2 * L, radius=max(0.04 * L, 1.5 * h))
        mask = torch.as_tensor(_needle(dict(c, axi=False), q)).cuda()
    v = 2e6 * shape[0] * h
    return h, v, (rho * (1e-2 * v * EPS0 / (0.02 * h * h * max(shape) ** 2))).contiguous(), mask


def _prepare_poisson(c: dict, seed: int) -> dict:
    h, v, rho, mask = _poisson_inputs(c, seed)
    return dict(grid=dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], dx=h), v=v, rho=rho, mask=mask, phi=torch.empty_like(rho),
                E=tuple(torch.empty(rho.shape, dtype=torch.float32, device="cuda") for _ in range(3)),
                rtol=c["rtol"], precision=c["precision"])


def _network(g: torch.Generator) -> torch.Tensor:
    """Glorot-uniform weights and small biases in the order W1, b1, W2, b2, W3, b3."""
    parts = []
    for out, inp in ((128, 2), (128, 128), (6, 128)):
        a = math.sqrt(6.0 / (out + inp))
        parts.append((2 * torch.rand(out * inp, generator=g, device="cuda", dtype=torch.float64) - 1) * a)
        parts.append(0.1 * torch.randn(out, generator=g, device="cuda", dtype=torch.float64))
    return torch.cat(parts).to(torch.float32)


X_MEAN, X_SCALE = (2.0, 0.2), (0.577, 0.0577)
Y_MEAN, Y_SCALE = (55.0, 57.0, 57.0, -50.0, -53.0, 1.7), (0.4, 0.3, 0.35, 4.0, 2.0, 0.9)


def _prepare_query(c: dict, seed: int) -> dict:
    g = _gen(seed)
    params = P.mlp_fold_standardization(_network(g), X_MEAN, X_SCALE, Y_MEAN, Y_SCALE)
    EN = 10.0 ** (1.0 + 2.0 * torch.rand(c["n"], generator=g, device="cuda", dtype=torch.float64))
    f = 0.1 + 0.2 * torch.rand(c["n"], generator=g, device="cuda", dtype=torch.float64)
    return dict(params=params, EN=EN, f=f)


def _training_set(c: dict, g: torch.Generator):
    x = math.sqrt(3.0) * (2 * torch.rand((c["n"], 2), generator=g, device="cuda", dtype=torch.float64) - 1)
    k = torch.arange(1, 7, device="cuda", dtype=torch.float64)
    t = torch.sin(0.4 * k * x[:, :1] + 0.3 * x[:, 1:]) + 0.2 * x[:, :1] * x[:, 1:]
    t += 0.01 * torch.randn((c["n"], 6), generator=g, device="cuda", dtype=torch.float64)
    return x.to(torch.float32).contiguous(), ((t - t.mean(0)) / t.std(0)).to(torch.float32).contiguous()


def _prepare_train(c: dict, seed: int) -> dict:
    g = _gen(seed)
    params = _network(g)
    x, t = _training_set(c, g)
    return dict(params=params, m=torch.zeros_like(params), v=torch.zeros_like(params), x=x, t=t, step=0, steps=c["steps"])


def prepare(case: dict, seed: int) -> dict:
    make = dict(streamer=_prepare_streamer, exchange=_prepare_exchange, swarm=_prepare_swarm, poisson=_prepare_poisson,
                query=_prepare_query, train=_prepare_train)[case["kind"]]
    return dict(make(case, seed), kind=case["kind"], steps=case.get("steps", 1))


# ------------------------------------------------------------------ passes

def run(s: dict):
    kind = s["kind"]
    if kind == "streamer":
        s["ctx"].step(s["steps"])
        if s["rho"] is not None:
            s["ctx"].deposit(rho=s["rho"])
            s["ctx"].get_field(*s["E"])
            return dict(rho=s["rho"], Ex=s["E"][0], Ey=s["E"][1], Ez=s["E"][2])
        s["ctx"].get_deposit(*s["q"])
        s["ctx"].get_field(*s["E"])
        return dict(q_e=s["q"][0], q_pos=s["q"][1], q_neg=s["q"][2], Ex=s["E"][0], Ey=s["E"][1], Ez=s["E"][2])
    if kind == "exchange":
        s["ctx"].upload(s["up"], s["n"])
        s["ctx"].step(1)
        n = s["ctx"].download(s["down"])
        s["ctx"].get_deposit(*s["q"])
        return dict(n=n, q_e=s["q"][0], q_pos=s["q"][1], q_neg=s["q"][2])
    if kind == "swarm":
        res, moments, counts = P.swarm_run(s["gas"], s["EN"], **s["kw"])
        return dict(results=res, moments=moments, counts=counts)
    if kind == "poisson":
        s["phi"].zero_()
        P.poisson_solve(s["grid"], s["rho"], s["phi"], mask=s["mask"], E=s["E"], v_hi=s["v"], v_mask=s["v"],
                        rtol=s["rtol"], max_cycles=1000, precision=s["precision"])
        return dict(phi=s["phi"], Ex=s["E"][0], Ey=s["E"][1], Ez=s["E"][2])
    if kind == "query":
        return P.mlp_forward(s["params"], P.mlp_features(s["EN"], s["f"]))
    loss = P.mlp_train(s["params"], s["m"], s["v"], s["step"], s["x"], s["t"], s["steps"])
    s["step"] += s["steps"]
    return dict(params=s["params"], m=s["m"], v=s["v"], loss=loss)


# ------------------------------------------------------------------ work

def work(case: dict) -> dict:
    kind = case["kind"]
    if kind in ("streamer", "exchange"):
        cells, R, n = case["nx"] * case["ny"] * case["nz"], case["precision"] // 8, case["n"]
        steps = case.get("steps", 1)
        # electrons read and written, three charge grids, the field; about 15 candidate collisions an electron
        grids = cells * (3 * 8 + 3 * R)
        flops = 15.0 * 100.0 * n * steps
        if kind == "streamer":  # and one field solve a step: the potential and the charge, a few V-cycles
            return dict(bytes=float(steps * (n * 2 * (10 * R + 8) + grids + cells * 24)),
                        flops=flops + 300.0 * cells * steps)
        return dict(bytes=float(n * 2 * (10 * R + 8) + grids), flops=flops)
    if kind == "swarm":
        updates = float(case["swarms"]) * case["n0"] * case["steps"]
        R = case["precision"] // 8
        return dict(bytes=updates * 2 * (7 * R + 8), flops=updates * 8 * 100.0)
    if kind == "poisson":
        cells = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=cells * (8.0 + 8.0 + 12.0 + (1.0 if case["electrode"] else 0.0)),
                    flops=cells * 150.0 * math.log10(1 / case["rtol"]))
    macs = 2 * 128 + 128 * 128 + 128 * 6
    if kind == "query":
        return dict(bytes=case["n"] * (16.0 + 24.0) + 4 * P.MLP_NPARAMS, flops=2.0 * macs * case["n"])
    return dict(bytes=case["steps"] * (case["n"] * 32.0 + 6 * 4 * P.MLP_NPARAMS),
                flops=6.0 * macs * case["n"] * case["steps"])


# ------------------------------------------------------------------ the same in 64 bits

def _exact_poisson(c: dict, seed: int):
    h, v, rho, mask = _poisson_inputs(c, seed)
    m = torch.zeros(rho.shape, dtype=torch.bool, device="cuda") if mask is None else mask.bool()
    free = (~m).double()

    def neighbours(u, lo, hi):
        s = torch.cat([u[:, :, :1], u[:, :, :-1]], 2) + torch.cat([u[:, :, 1:], u[:, :, -1:]], 2)
        s += torch.cat([u[:, :1], u[:, :-1]], 1) + torch.cat([u[:, 1:], u[:, -1:]], 1)
        s += torch.cat([2 * lo - u[:1], u[:-1]], 0) + torch.cat([u[1:], 2 * hi - u[-1:]], 0)
        return s

    # conjugate gradients on the unmasked cells, on corrections to a potential that has the boundary values
    phi = torch.where(m, torch.full_like(rho, v), torch.zeros_like(rho))
    for _ in range(2):  # the second pass starts from the residual of the first
        r = free * (h * h / EPS0 * rho + neighbours(phi, 0.0, v) - 6.0 * phi)
        d, p = torch.zeros_like(r), r.clone()
        rr = first = float((r * r).sum())
        for _ in range(6000):
            if not rr > first * 1e-26:
                break
            q = free * (6.0 * p - neighbours(p, 0.0, 0.0))
            a = rr / float((p * q).sum())
            d += a * p
            r -= a * q
            old, rr = rr, float((r * r).sum())
            p = r + rr / old * p
        phi = phi + d
    ext = lambda u, dim: (torch.cat([u.narrow(dim, 0, 1), u.narrow(dim, 0, u.shape[dim] - 1)], dim),
                          torch.cat([u.narrow(dim, 1, u.shape[dim] - 1), u.narrow(dim, u.shape[dim] - 1, 1)], dim))
    xm, xp = ext(phi, 2)
    ym, yp = ext(phi, 1)
    zm, zp = torch.cat([-phi[:1], phi[:-1]], 0), torch.cat([phi[1:], 2 * v - phi[-1:]], 0)
    k = -1.0 / (2.0 * h)
    return dict(phi=phi, Ex=k * (xp - xm), Ey=k * (yp - ym), Ez=k * (zp - zm))


def _split(params: torch.Tensor):
    shapes = ((128, 2), (128,), (128, 128), (128,), (6, 128), (6,))
    out, o = [], 0
    for sh in shapes:
        k = math.prod(sh)
        out.append(params[o:o + k].reshape(sh))
        o += k
    return out


def _forward(params: torch.Tensor, x: torch.Tensor):
    W1, b1, W2, b2, W3, b3 = _split(params)
    h1 = torch.tanh(x @ W1.T + b1)
    h2 = torch.tanh(h1 @ W2.T + b2)
    return h1, h2, h2 @ W3.T + b3


def _exact_query(c: dict, seed: int):
    g = _gen(seed)
    params = _network(g).double()
    EN = 10.0 ** (1.0 + 2.0 * torch.rand(c["n"], generator=g, device="cuda", dtype=torch.float64))
    f = 0.1 + 0.2 * torch.rand(c["n"], generator=g, device="cuda", dtype=torch.float64)
    pair = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")
    y = torch.empty((c["n"], 6), dtype=torch.float64, device="cuda")
    for o in range(0, c["n"], 1 << 20):
        x = torch.stack([torch.log10(EN[o:o + (1 << 20)]), f[o:o + (1 << 20)]], 1)
        y[o:o + (1 << 20)] = _forward(params, (x - pair(X_MEAN)) / pair(X_SCALE))[2] * pair(Y_SCALE) + pair(Y_MEAN)
    return y


def _exact_train(c: dict, seed: int):
    g = _gen(seed)
    params = _network(g).double()
    x, t = (a.double() for a in _training_set(c, g))
    m, v = torch.zeros_like(params), torch.zeros_like(params)
    b1, b2 = 0.9, 0.999
    for k in range(1, c["steps"] + 1):
        W1, _, W2, _, W3, _ = _split(params)
        h1, h2, y = _forward(params, x)
        dy = 2.0 * (y - t) / y.numel()
        loss = ((y - t) ** 2).mean()
        d2 = (dy @ W3) * (1 - h2 * h2)
        d1 = (d2 @ W2) * (1 - h1 * h1)
        grad = torch.cat([a.reshape(-1) for a in (d1.T @ x, d1.sum(0), d2.T @ h1, d2.sum(0), dy.T @ h2, dy.sum(0))])
        m = b1 * m + (1 - b1) * grad
        v = b2 * v + (1 - b2) * grad * grad
        params = params - 1e-3 * (m / (1 - b1 ** k)) / (torch.sqrt(v / (1 - b2 ** k)) + 1e-8)
    return dict(params=params, m=m, v=v, loss=loss.reshape(1))


def exact(case: dict, seed: int):
    """What run() returns, in 64 bits.  Particle simulations have none: their random walks end elsewhere after the
    first decision that a rounding turns, and their charge grids are whole numbers."""
    make = dict(poisson=_exact_poisson, query=_exact_query, train=_exact_train).get(case["kind"])
    return make(case, seed) if make else None

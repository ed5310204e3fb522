"""What a user of this framework has it do, as cases that can be timed and checked.

A case is one of five kinds, each a whole call sequence of a user's program over the public entry points
(``Simulation`` / the C ABI of include/grpic.h), with inputs already on the GPU:

  plasma  load the field and the particles, take ``steps`` timesteps, read particles and fields back
  vacuum  load a field, take ``steps`` timesteps without particles, read the fields back
  sweep   several contexts of different grids and holes reloaded and advanced together (grpic_batch_*)
  serve   a few runs submitted to a server, ticked until they are done, read back and released
  diag    the diagnostics of a loaded state: charge density, Gauss residual, contravariant field

Particles come back in no fixed order within a cell, so ``run`` puts them in the order of their ids
(removed ones are zero).  FP32-mixed state is handed on in FP32, which is how the library holds it; J of
such a run is scratch of the step and is not part of the state.

``exact`` restates the timestep in plain FP64 torch: metric and Christoffel terms from the closed forms of
the Kerr-Schild metric, time-centred field half-steps, RK4 in proper time, the zig-zag deposit with
Gauss-Legendre face areas.
"""
import ctypes
import math

import numpy as np
import torch

from paper_0904_0232_gb300 import grpic as G

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64

# ---- cases ---------------------------------------------------------------------------------------


def plasma_case(nx, ny, nz, ppc, steps, m, spin, precision="fp32_mixed", plasma="ion", quad=2, sort=1, tuned=False,
           B0=0.1, u_th=0.05, layers=False):
    return dict(kind="plasma", nx=nx, ny=ny, nz=nz, ppc=ppc, steps=steps, m=m, a=spin * m, c=1.0, dt=0.4,
                precision=precision, plasma=plasma, quad=quad, sort=sort, tuned=tuned, B0=B0, u_th=u_th,
                layers=layers)


def vacuum_case(nx, ny, nz, steps, m, spin, precision):
    return dict(kind="vacuum", nx=nx, ny=ny, nz=nz, steps=steps, m=m, a=spin * m, c=1.0, dt=0.4,
                precision=precision, quad=2, B0=0.1, layers=True)


def listed():
    return [
        # the Schwarzschild pair plasma of the tests: a small run, where each launch counts; both precisions
        dict(plasma_case(32, 32, 32, 2, 5, 2.0, 0.0, plasma="pairs", B0=0.05, u_th=0.1), name="pairs_32"),
        dict(plasma_case(32, 32, 32, 2, 5, 2.0, 0.0, "fp64", plasma="pairs", B0=0.05, u_th=0.1), name="pairs_32_fp64"),
        # the Kerr electron-ion plasma at an ordinary size with the default launch shapes
        dict(plasma_case(64, 64, 64, 8, 4, 2.0, 0.9), name="kerr_64"),
        # the same in FP64, which a user takes for convergence studies
        dict(plasma_case(64, 64, 64, 8, 1, 2.0, 0.9, "fp64"), name="kerr_64_fp64"),
        # an odd, elongated box, three Gauss nodes, sorted every other step, absorbing layers
        dict(plasma_case(75, 50, 91, 5, 4, 1.6, 0.7, quad=3, sort=2, layers=True), name="kerr_75x50x91_q3"),
        # the benchmark's workload with the shapes its autotuner picks: the largest run
        dict(plasma_case(128, 128, 128, 8, 8, 4.0, 0.9, sort=4, tuned=True), name="kerr_128"),
        # the application set-up: disk and corona pairs as four species on 64 x 64 x 128, c = 0.05
        dict(kind="plasma", nx=64, ny=64, nz=128, ppc=0, steps=4, m=2.0, a=1.9, c=0.05, dt=1.0,
             precision="fp32_mixed", plasma="disk", quad=2, sort=1, tuned=False, B0=30.0, u_th=0.05, layers=False,
             name="jet_64x64x128"),
        # field evolution around a hole without plasma (stability studies), both precisions
        dict(vacuum_case(192, 192, 192, 8, 4.0, 0.9, "fp32_mixed"), name="vacuum_192"),
        dict(vacuum_case(96, 96, 96, 4, 2.0, 0.9, "fp64"), name="vacuum_96_fp64"),
        # a parameter sweep advanced as one batch
        dict(kind="sweep", n=8, pick=1, gmin=32, gmax=64, ppc=4, steps=4, precision="fp32_mixed", name="sweep_8"),
        # a burst of light requests to a server
        dict(kind="serve", n=4, pick=1, gmin=24, gmax=48, ppc=4, steps=6, precision="fp32_mixed", name="serve_4"),
        # the checks a run does between steps
        dict(kind="diag", nx=96, ny=96, nz=96, ppc=8, m=3.0, a=2.7, c=1.0, dt=0.4, precision="fp32_mixed",
             plasma="ion", quad=2, B0=0.1, u_th=0.05, layers=False, name="diag_96"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plasma", "plasma", "plasma", "plasma64", "plasma64", "vacuum", "vacuum", "sweep", "serve",
                       "diag"])
    if kind in ("plasma", "plasma64", "diag"):
        nx, ny, nz = (_log_int(rng, 20, 120 if kind == "plasma" else 72) for _ in range(3))
        m = rng.uniform(0.0, 1.0) * min(nx, ny, nz) / 24.0
        spin = rng.uniform(0.0, 0.99)
        if kind == "diag":
            return dict(kind="diag", nx=nx, ny=ny, nz=nz, ppc=rng.randint(1, 16), m=m, a=spin * m, c=1.0, dt=0.4,
                        precision=rng.choice(["fp32_mixed", "fp64"]), plasma="pairs", quad=2, B0=0.1, u_th=0.05,
                        layers=False)
        cells = (nx - 3) * (ny - 3) * (nz - 3)
        if kind == "plasma":
            ppc = max(1, min(_log_int(rng, 1, 16), int(1.4e7 / cells)))
            tuned = rng.random() < 0.4
            return plasma_case(nx, ny, nz, ppc, rng.randint(1, 6), m, spin, plasma=rng.choice(["ion", "pairs"]),
                          quad=2 if tuned else rng.choice([1, 2, 2, 3]), sort=rng.choice([1, 2, 4]), tuned=tuned,
                          u_th=rng.uniform(0.03, 0.12), layers=rng.random() < 0.5)
        ppc = max(1, min(_log_int(rng, 1, 16), int(1.6e6 / cells)))
        return plasma_case(nx, ny, nz, ppc, rng.randint(1, 2), m, spin, "fp64", plasma=rng.choice(["ion", "pairs"]),
                      quad=rng.choice([1, 2, 2, 3]), sort=rng.choice([1, 2]), u_th=rng.uniform(0.03, 0.12),
                      layers=rng.random() < 0.5)
    if kind == "vacuum":
        prec = rng.choice(["fp32_mixed", "fp32_mixed", "fp64"])
        nx, ny, nz = (_log_int(rng, 24, 200 if prec != "fp64" else 100) for _ in range(3))
        return vacuum_case(nx, ny, nz, rng.randint(1, 8), rng.uniform(0.0, 1.0) * min(nx, ny, nz) / 24.0,
                      rng.uniform(0.0, 0.99), prec)
    if kind == "sweep":
        return dict(kind="sweep", n=rng.randint(2, 16), pick=rng.randint(2, 9999), gmin=rng.randint(20, 32),
                    gmax=rng.randint(33, 64), ppc=rng.randint(1, 5), steps=rng.choice([2, 4]),
                    precision=rng.choice(["fp32_mixed"] * 3 + ["fp64"]))
    return dict(kind="serve", n=rng.randint(1, 6), pick=rng.randint(2, 9999), gmin=rng.randint(16, 24),
                gmax=rng.randint(25, 56), ppc=rng.randint(1, 5), steps=rng.randint(1, 8), precision="fp32_mixed")


# ---- inputs --------------------------------------------------------------------------------------


def _gen(seed, stream=0):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + stream) % (1 << 62))


def _maxwell_juettner(g, n, theta):
    """(3, n) isotropic momenta in units of c, |u| ~ u^2 exp(-(gamma - 1) / theta)."""
    u = torch.linspace(0.0, math.sqrt((1.0 + 40.0 * theta) ** 2 - 1.0), 20001, dtype=F64)
    cdf = torch.cumsum(u * u * torch.exp(-(torch.sqrt(1.0 + u * u) - 1.0) / theta), 0)
    cdf, u = (cdf / cdf[-1]).to(DEV), u.to(DEV)
    r = torch.rand(n, generator=g, device=DEV, dtype=torch.float32).double()
    i = torch.searchsorted(cdf, r).clamp(1, u.numel() - 1)
    mag = u[i - 1] + (r - cdf[i - 1]) / (cdf[i] - cdf[i - 1]) * (u[i] - u[i - 1])
    d = torch.randn((3, n), generator=g, device=DEV, dtype=torch.float32)
    return (d / d.norm(dim=0, keepdim=True)).double() * mag


def _cells(c):
    k, j, i = torch.meshgrid(*(torch.arange(1, n - 2, device=DEV) for n in (c["nz"], c["ny"], c["nx"])), indexing="ij")
    return torch.stack([i.reshape(-1), j.reshape(-1), k.reshape(-1)])


def _centre(c):
    return torch.tensor([(c["nx"] - 1) / 2, (c["ny"] - 1) / 2, (c["nz"] - 1) / 2], dtype=F64, device=DEV)[:, None]


def _place(g, base):
    """Positions uniform in the given cells, on FP32 values."""
    f = torch.rand(base.shape, generator=g, device=DEV, dtype=torch.float32)
    x = (base.float() + f).double()
    return torch.minimum(x, base.double() + (1.0 - 2.0 ** -16))


def _species(c, seed):
    """One (q/m, macro charge, x4, u4, ids, umode) a species: covariant spatial u (the disk: contravariant)."""
    g = _gen(seed)
    out = []
    if c["plasma"] == "disk":
        return _disk(c, g)
    cells = _cells(c)
    if c["plasma"] == "pairs":
        qms, wp = (-1.0, 1.0), 0.1
        cells = cells[:, (cells + 0.5 - _centre(c)).norm(dim=0) >= 3.0 * c["m"] + 1.0]
    else:
        qms, wp = (-1.0, 0.05), 0.025
    x = _place(g, cells.repeat_interleave(c["ppc"], dim=1))
    n = x.shape[1]
    q = (wp / c["dt"]) ** 2 / (4.0 * math.pi * c["ppc"] * sum(abs(v) for v in qms))
    x4 = torch.cat([x, torch.zeros((1, n), dtype=F64, device=DEV)])
    ids = torch.arange(n, dtype=torch.int32, device=DEV)
    for s, qm in enumerate(qms):
        u = _maxwell_juettner(_gen(seed, 1 + s), n, (c["u_th"] / c["c"]) ** 2) * c["c"]
        u4 = torch.cat([u, torch.zeros((1, n), dtype=F64, device=DEV)])
        out.append((qm, math.copysign(q, qm), x4, u4, ids, 1))
    return out


def _disk(c, g):
    """Keplerian disk (0.8 M particles, R > 6 m, |z| < R / 8) and a hundredfold thinner free-falling corona."""
    cells, cen = _cells(c), _centre(c)
    X = cells + 0.5 - cen
    R = X.norm(dim=0)
    m, cc, qm = c["m"], c["c"], 1e-3
    r_plus = m + math.sqrt(m * m - c["a"] ** 2)
    disk = (R > 6.0 * m) & (X[2].abs() < R / 8.0)
    corona = ~disk & (R > r_plus + 1.0)
    dens = 400_000 / int(disk.sum())
    q = (0.025 / c["dt"]) ** 2 / (4.0 * math.pi * dens * 2.0 * qm)
    out = []
    for part, sel, lam in ((0, disk, dens), (1, corona, 0.01 * dens)):
        cl = cells[:, sel]
        more = torch.rand(cl.shape[1], generator=_gen(part), device=DEV) < lam - math.floor(lam)
        cnt = math.floor(lam) + more.long()
        x = _place(g, torch.repeat_interleave(cl, cnt, dim=1))
        n = x.shape[1]
        zero = torch.zeros((1, n), dtype=F64, device=DEV)
        d = x - cen
        u0 = torch.zeros((3, n), dtype=F64, device=DEV)
        if part == 0:
            v = cc * torch.sqrt(m / d.norm(dim=0))
            gv = v / torch.sqrt(1.0 - (v / cc) ** 2) / d[:2].norm(dim=0)
            u0[0], u0[1] = gv * d[1], -gv * d[0]
        for sign in (-1.0, 1.0):
            u = u0 + c["u_th"] * cc * torch.randn((3, n), generator=g, device=DEV, dtype=torch.float32).double()
            out.append((sign * qm, sign * q, torch.cat([x, zero]), torch.cat([u, zero]),
                        torch.arange(n, dtype=torch.int32, device=DEV), 2 if part == 0 else 1))
    return out


def _noise_field(c, seed):
    """A uniform B_z with a rough perturbation: (d, b), on FP32 values."""
    g = _gen(seed, 7)
    shape = (3, c["nz"], c["ny"], c["nx"])
    d = 0.01 * torch.randn(shape, generator=g, device=DEV, dtype=torch.float32)
    b = 0.01 * torch.randn(shape, generator=g, device=DEV, dtype=torch.float32)
    b[2] += c["B0"]
    return d.double(), b.double()


def _sweep_cases(c, seed):
    r = np.random.Generator(np.random.Philox(key=[c["pick"], 5]))
    out = []
    for i in range(c["n"]):
        n = int(r.integers(c["gmin"], c["gmax"] + 1))
        m = float(r.uniform(0.5, n / 24.0))
        ppc, spin = int(r.integers(1, c["ppc"] + 1)), float(r.uniform(0.0, 0.99))
        out.append(dict(plasma_case(n, n, n, ppc, c["steps"], m, spin, c["precision"], layers=True),
                        seed=int(seed) * 100 + i))
    return out


def _serve_requests(c, seed):
    r = np.random.Generator(np.random.Philox(key=[c["pick"], 6]))
    out = []
    for i in range(c["n"]):
        n = int(r.integers(c["gmin"], c["gmax"] + 1))
        m = float(r.uniform(0.5, n / 24.0))
        out.append(dict(n=n, m=m, a=float(r.uniform(0.0, 0.95)) * m, ppc=int(r.integers(1, c["ppc"] + 1)),
                        nsteps=int(r.integers(max(1, c["steps"] // 2), c["steps"] + 1)),
                        seed=int(seed) * 100 + i, precision=c["precision"], absorb_inner=0.3,
                        absorb_outer=0.2, absorb_width=4))
    return out


# ---- the framework's side ------------------------------------------------------------------------


def _simulation(c):
    layers = dict(absorb_inner=0.3, absorb_outer=0.2, absorb_width=4) if c["layers"] else {}
    sim = G.Simulation(c["nx"], c["ny"], c["nz"], c["m"], c["a"], c["c"], c["dt"], precision=c["precision"],
                       quad_order=c["quad"], sort_interval=c.get("sort", 1), **layers)
    if c.get("tuned"):
        sim.set_tuning(far_min_blocks=5, sort_interval=c["sort"], spread=16, area_table=1)
    return sim


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind}
    if kind == "vacuum":
        st["sim"], st["field"] = _simulation(case), _noise_field(case, seed)
    elif kind == "sweep":
        st["items"] = [(_simulation(k), k, _species(k, k["seed"])) for k in _sweep_cases(case, seed)]
        for item in st["items"]:
            _load(*item)
        st["batch"] = Batch([sim for sim, _, _ in st["items"]])
    elif kind == "serve":
        st["server"] = Server()
        st["requests"] = [G.make_request(**r) for r in _serve_requests(case, seed)]
    else:
        st["sim"], st["species"] = _simulation(case), _species(case, seed)
        if kind == "diag":
            _load(st["sim"], case, st["species"])
            st["sim"].set_fields(*_noise_field(case, seed))
    return st


class Batch:
    """A batch handle freed with the state that holds it."""

    def __init__(self, sims):
        self.sims = sims
        self.handle = G.grpic_batch_create([s.handle for s in sims])

    def __del__(self):
        if self.handle:
            G.grpic_batch_destroy(self.handle)
            self.handle = None


class Server:
    def __init__(self):
        self.handle = G.grpic_server_create(100 << 30, 64)

    def __del__(self):
        if self.handle:
            G.grpic_server_destroy(self.handle)
            self.handle = None


def _load(sim, c, species):
    sim.set_uniform_field(B=(0.0, 0.0, c["B0"]))
    for s, (qm, q, x4, u4, ids, umode) in enumerate(species):
        sim.load_particles(s, qm, q, x4, u4, ids, umode)


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def _fields(handle, shape, dtype):
    """d and b of a context, on the GPU."""
    d = torch.empty((3,) + tuple(shape), dtype=F64, device=DEV)
    b = torch.empty_like(d)
    G._check(handle, G.load_library().grpic_get_fields(handle, _ptr(d), _ptr(b), None, G.GRPIC_MEM_DEVICE),
             "grpic_get_fields")
    return d.to(dtype), b.to(dtype)


def _by_id(handle, s, n, dtype):
    """(8, n) positions and velocities of a species in the order of the ids."""
    x4, u4, ids = G.grpic_get_particles(handle, s, device=True)
    out = torch.zeros((8, n), dtype=dtype, device=DEV)
    at = ids.long()
    out[:4].index_copy_(1, at, x4.to(dtype))
    out[4:].index_copy_(1, at, u4.to(dtype))
    return out


def run(state):
    case, kind = state["case"], state["kind"]
    dtype = F64 if case["precision"] == "fp64" else torch.float32
    if kind == "plasma":
        sim = state["sim"]
        _load(sim, case, state["species"])
        sim.step(case["steps"])
        return {"particles": [_by_id(sim.handle, s, sp[4].numel(), dtype) for s, sp in enumerate(state["species"])],
                "fields": _fields(sim.handle, sim.shape, dtype)}
    if kind == "vacuum":
        sim = state["sim"]
        sim.set_fields(*state["field"])
        sim.step(case["steps"])
        return {"fields": _fields(sim.handle, sim.shape, dtype)}
    if kind == "sweep":
        for item in state["items"]:
            _load(*item)
        G.grpic_batch_step(state["batch"].handle, case["steps"])
        return [{"particles": torch.cat([_by_id(sim.handle, s, sp[4].numel(), dtype) for s, sp in enumerate(sps)], 1),
                 "fields": torch.cat(_fields(sim.handle, sim.shape, dtype))} for sim, _, sps in state["items"]]
    if kind == "serve":
        srv = state["server"].handle
        tickets = [G.grpic_submit(srv, r) for r in state["requests"]]
        left, out = set(range(len(tickets))), [None] * len(tickets)
        while left:
            G.grpic_server_tick(srv)
            for i in sorted(left):
                done, ctx = G.grpic_poll(srv, tickets[i])
                if done != G.GRPIC_RUN_DONE:
                    continue
                r = state["requests"][i]
                n, slots = r.cfg.nx, (r.cfg.nx - 3) ** 3 * r.ppc
                out[i] = {"particles": torch.cat([_by_id(ctx, s, slots, dtype) for s in range(r.nspecies)], 1),
                          "fields": torch.cat(_fields(ctx, (n, n, n), dtype))}
                G.grpic_server_release(srv, tickets[i])
                left.discard(i)
        return out
    sim = state["sim"]
    lib, h = G.load_library(), sim.handle
    rho, res = (torch.empty(sim.shape, dtype=F64, device=DEV) for _ in range(2))
    hc = torch.empty((3,) + sim.shape, dtype=F64, device=DEV)
    G._check(h, lib.grpic_charge_density(h, 1, _ptr(rho), G.GRPIC_MEM_DEVICE), "grpic_charge_density")
    worst = ctypes.c_double(0.0)
    G._check(h, lib.grpic_gauss_residual(h, _ptr(res), G.GRPIC_MEM_DEVICE, ctypes.byref(worst)), "grpic_gauss_residual")
    G._check(h, lib.grpic_get_fields_contra(h, None, _ptr(hc), G.GRPIC_MEM_DEVICE), "grpic_get_fields_contra")
    return {"rho": rho, "residual": res, "contra": hc.to(dtype), "worst": worst.value}


# ---- work ----------------------------------------------------------------------------------------

# operations of one particle-step by quadrature order, and of one field step per cell (the metric and the
# conversions at three edges in each B half-step, at three faces twice in the E step)
PUSH_FLOPS = {1: 3401, 2: 6641, 3: 12041}
FIELD_FLOPS = 2 * 300 + 2 * 300


def _run_work(cells, parts, steps, quad, precision):
    t = 8 if precision == "fp64" else 4
    # inputs and outputs of the call, and per step the state in and out: 8 values and an id of each particle,
    # 6 field values of each cell
    per_call = parts * (8 * 8 + 4) + cells * 6 * 8 + parts * 8 * t + cells * 6 * t
    return {"bytes": float(per_call + steps * 2 * (parts * (8 * t + 4) + cells * 6 * t)),
            "flops": float(steps * (parts * PUSH_FLOPS[quad] + cells * FIELD_FLOPS))}


def work(case):
    def sub(c):
        cells = c["nx"] * c["ny"] * c["nz"]
        if c["kind"] == "vacuum":
            parts = 0
        elif c["plasma"] == "disk":
            parts = 970_000
        else:
            parts = 2 * c["ppc"] * (c["nx"] - 3) * (c["ny"] - 3) * (c["nz"] - 3)
        if c["kind"] == "diag":
            t = 8 if c["precision"] == "fp64" else 4
            return {"bytes": float(parts * 4 * t + cells * (6 * t + 2 * 8 + 3 * t)),
                    "flops": float(2 * parts * 30 + cells * 300)}
        return _run_work(cells, parts, c["steps"], c["quad"], c["precision"])

    if case["kind"] in ("plasma", "vacuum", "diag"):
        return sub(case)
    # the grids and densities of a sweep or a burst are drawn: their means here
    n, ppc = 0.5 * (case["gmin"] + case["gmax"]), 0.5 * (1 + case["ppc"])
    w = _run_work(n ** 3, 2 * ppc * (n - 3) ** 3, case["steps"], 2, case["precision"])
    return {k: case["n"] * v for k, v in w.items()}


# ---- the same in plain FP64 torch ----------------------------------------------------------------

HALF = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (0, 1, 1), (1, 0, 1), (1, 1, 0)]  # d edges, b faces
GAUSS = {1: ([0.0], [2.0]), 2: ([-3 ** -0.5, 3 ** -0.5], [1.0, 1.0]),
         3: ([-0.6 ** 0.5, 0.0, 0.6 ** 0.5], [5 / 9, 8 / 9, 5 / 9])}


def _kerr(X, Y, Z, m, a):
    """r, D, f and k of the Kerr-Schild metric; f = 0 and k = (0, 0, 1) where r = 0."""
    p, q = X * X + Y * Y + Z * Z - a * a, a * a * Z * Z
    D = torch.sqrt(p * p + 4.0 * q)
    r2 = torch.where(p >= 0, 0.5 * (p + D), 2.0 * q / (D - p))
    flat = ~(r2 > 0)
    r = torch.sqrt(torch.where(flat, 1.0, r2))
    f = 2.0 * m * r ** 3 / (r ** 4 + q)
    k = [(r * X - a * Y) / (r * r + a * a), (r * Y + a * X) / (r * r + a * a), Z / r]
    f = torch.where(flat, 0.0, f)
    k = [torch.where(flat, 0.0, k[0]), torch.where(flat, 0.0, k[1]), torch.where(flat, 1.0, k[2])]
    return torch.where(flat, 0.0, r), torch.where(flat, 1.0, D), f, k


def _cross(u, v):
    return [u[1] * v[2] - u[2] * v[1], u[2] * v[0] - u[0] * v[2], u[0] * v[1] - u[1] * v[0]]


def _dot(u, v):
    return u[0] * v[0] + u[1] * v[1] + u[2] * v[2]


def _contra(f, k, b, d):
    """Contravariant (F^yz, F^zx, F^xy) from covariant b and contravariant d."""
    al = [b[i] - f * x for i, x in enumerate(_cross(d, k))]
    ka = _dot(k, al)
    return [(al[i] + f * ka * k[i]) / (1.0 + f) for i in range(3)]


class Exact:
    def __init__(self, c):
        self.c = c
        self.n = (c["nx"], c["ny"], c["nz"])
        self.cen = [(n - 1) / 2 for n in self.n]
        self.m, self.a, self.q = c["m"], c["a"], c["quad"]
        self.r_plus = self.m + math.sqrt(max(0.0, self.m ** 2 - self.a ** 2))
        self.r_exc = (0.5 if c["layers"] else 1.0) * self.r_plus
        ax = [torch.arange(n, dtype=F64, device=DEV) for n in self.n]
        z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
        inside = torch.ones_like(x, dtype=torch.bool)
        dist = torch.full_like(x, 1e9)
        for v, n in zip((x, y, z), self.n):
            inside &= (v >= 2) & (v <= n - 3)
            dist = torch.minimum(dist, torch.minimum(v - 2, n - 3 - v))
        self.loc = []
        for h in HALF:
            r, _, f, k = _kerr(x + 0.5 * h[0] - self.cen[0], y + 0.5 * h[1] - self.cen[1],
                               z + 0.5 * h[2] - self.cen[2], self.m, self.a)
            exc = (r < self.r_exc) | (r == 0)
            fe = torch.where(exc, 0.0, f)
            ke = [torch.where(exc, 0.0, k[0]), torch.where(exc, 0.0, k[1]), torch.where(exc, 1.0, k[2])]
            kap = None
            if c["layers"]:
                s = dist + 1.0
                kap = torch.where((s >= 1) & (s <= 4), 0.2 * ((5.0 - s) / 4.0) ** 2, 0.0)
                inner = 0.3 * (self.r_plus - r) / max(self.r_plus - self.r_exc, 1e-300)
                kap = torch.maximum(kap, torch.where((r >= self.r_exc) & (r < self.r_plus) & (r > 0), inner, 0.0))
            self.loc.append((fe, ke, inside & ~exc, kap))
        self.conv = torch.zeros_like(inside)
        self.conv[1:-1, 1:-1, 1:-1] = True
        shape = (3,) + tuple(x.shape)
        self.d, self.b, self.J = (torch.zeros(shape, dtype=F64, device=DEV) for _ in range(3))
        self.parts = []

    def uniform(self, B):
        h, z = [torch.full_like(self.d[0], v) for v in B], torch.zeros_like(self.d[0])
        for q in range(3):
            f, k = self.loc[3 + q][:2]
            v = _cross(k, h)
            low = [h[i] + f * x for i, x in enumerate(_cross(v, k))]
            self.d[q], self.b[q] = z, low[q]
        self.target()

    def target(self):
        self.td, self.tb = self.d.clone(), self.b.clone()

    # ---- fields
    def _to(self, field, s, t):
        """Component field on lattice s brought to lattice t: the mean of the nearest points."""
        for ax in range(3):
            if HALF[s][ax] != HALF[t][ax]:
                field = 0.5 * (field + torch.roll(field, -1 if HALF[t][ax] else 1, dims=2 - ax))
        return field

    def _at(self, d, b, t):
        return [self._to(d[i], i, t) for i in range(3)], [self._to(b[i], 3 + i, t) for i in range(3)]

    def _e(self, d, b):
        out = []
        for t in range(3):
            f, k = self.loc[t][:2]
            dd, bb = self._at(d, b, t)
            kxh = _cross(k, _contra(f, k, bb, dd))[t]
            e = f * kxh + (f - 1.0) * dd[t] - f * k[t] * _dot(k, dd)
            out.append(torch.where(self.conv, e, 0.0))
        return out

    def _h(self, d, b):
        out = []
        for q in range(3):
            f, k = self.loc[3 + q][:2]
            dd, bb = self._at(d, b, 3 + q)
            out.append(torch.where(self.conv, _contra(f, k, bb, dd)[q], 0.0))
        return out

    def _relax(self, v, t, loc, relax):
        kap = self.loc[loc][3]
        return v if kap is None or not relax else t + (1.0 - kap) * (v - t)

    def _b_step(self, base, src, coef, relax):
        e = self._e(self.d, src)
        diff = lambda v, ax: torch.roll(v, -1, dims=2 - ax) - v  # noqa: E731
        curl = [diff(e[2], 1) - diff(e[1], 2), diff(e[0], 2) - diff(e[2], 0), diff(e[1], 0) - diff(e[0], 1)]
        new = [self._relax(base[q] - coef * curl[q], self.tb[q], 3 + q, relax) for q in range(3)]
        return torch.stack([torch.where(self.loc[3 + q][2], new[q], base[q]) for q in range(3)])

    def _rhs(self, d):
        h = self._h(d, self.b)
        diff = lambda v, ax: v - torch.roll(v, 1, dims=2 - ax)  # noqa: E731
        div = [diff(h[2], 1) - diff(h[1], 2), diff(h[0], 2) - diff(h[2], 0), diff(h[1], 0) - diff(h[0], 1)]
        return [4.0 * math.pi / self.c["c"] * self.J[q] - div[q] for q in range(3)]

    def step(self):
        dx4 = self.c["c"] * self.c["dt"]
        old = self.b
        self.b = self._b_step(old, old, 0.5 * dx4, False)
        self.J.zero_()
        for p in self.parts:
            self._push(p)
        self.b = self._b_step(old, self.b, dx4, True)
        adv = [self.loc[q][2] for q in range(3)]
        rhs = self._rhs(self.d)
        mid = torch.stack([torch.where(adv[q], self.d[q] + 0.5 * dx4 * rhs[q], self.d[q]) for q in range(3)])
        rhs = self._rhs(mid)
        new = [self._relax(self.d[q] + dx4 * rhs[q], self.td[q], q, True) for q in range(3)]
        self.d = torch.stack([torch.where(adv[q], new[q], self.d[q]) for q in range(3)])

    # ---- particles
    def load(self, qm, qmacro, x4, u4, umode):
        x = [x4[i].clone() for i in range(4)]
        r, _, f, k = _kerr(*(x[i] - self.cen[i] for i in range(3)), self.m, self.a)
        ui = [u4[i].clone() for i in range(3)]
        ku, uu, c2 = _dot(k, ui), _dot(ui, ui), self.c["c"] ** 2
        if umode == 1:  # covariant u_i: the root of g^mn u_m u_n = -c^2 with u^4 > 0
            A, B, C = -1.0 - f, 2.0 * f * ku, uu - f * ku * ku + c2
            sq = torch.sqrt(B * B - 4.0 * A * C)
            r1, r2 = (-B + sq) / (2.0 * A), (-B - sq) / (2.0 * A)
            ul = torch.where(-r1 + f * (ku - r1) > 0, r1, r2)
            u = [ui[i] - f * k[i] * (ku - ul) for i in range(3)] + [-ul + f * (ku - ul)]
        else:  # contravariant u^i
            A, B, C = -1.0 + f, 2.0 * f * ku, uu + f * ku * ku + c2
            sq = torch.sqrt(B * B - 4.0 * A * C)
            u = ui + [torch.maximum((-B + sq) / (2.0 * A), (-B - sq) / (2.0 * A))]
        alive = (r > self.r_plus) if self.m > 0 else torch.ones_like(r, dtype=torch.bool)
        self.parts.append(dict(qm=qm, q=qmacro, x=x, u=u, alive=alive))

    def _gather(self, x):
        out = []
        for comp in range(6):
            F = (self.d[comp] if comp < 3 else self.b[comp - 3]).reshape(-1)
            i0, w = [], []
            for ax in range(3):
                s = x[ax] - 0.5 * HALF[comp][ax]
                a = torch.floor(s).clamp(0, self.n[ax] - 2)
                i0.append(a.long())
                w.append(s - a)
            base = (i0[2] * self.n[1] + i0[1]) * self.n[0] + i0[0]
            v = torch.zeros_like(x[0])
            for dz in range(2):
                for dy in range(2):
                    for dx in range(2):
                        W = ((w[0] if dx else 1 - w[0]) * (w[1] if dy else 1 - w[1])) * (w[2] if dz else 1 - w[2])
                        v += W * F[base + (dz * self.n[1] + dy) * self.n[0] + dx]
            out.append(v)
        return out[:3], out[3:]

    def _accel(self, x, u, qm):
        d, b = self._gather(x)
        X = [x[i] - self.cen[i] for i in range(3)]
        m, a = self.m, self.a
        r, D, f, k = _kerr(*X, m, a)
        flat = r == 0
        r = torch.where(flat, 1.0, r)
        h = _contra(f, k, b, d)
        s = _dot(k, u) + u[3]
        uc = [u[i] + f * s * k[i] for i in range(3)]
        u4 = f * s - u[3]
        lor = [qm * (v + d[i] * u4) for i, v in enumerate(_cross(uc, h))] + [-qm * _dot(d, uc)]
        # Gamma u u = g^ab (u.d g_bn u^n - 1/2 d_b g_mn u^m u^n) for g = eta + f k k
        rho2, sig = r * r + a * a, r ** 4 + (a * X[2]) ** 2
        gr = [X[0] * r / D, X[1] * r / D, X[2] * rho2 / (r * D)]
        fr = f * (3.0 / r - 4.0 * r ** 3 / sig)
        gf = [fr * gr[0], fr * gr[1], fr * gr[2] - 2.0 * a * a * X[2] * f / sig]
        jac = []
        for i in range(3):
            jac.append([(X[0] * gr[i] + (r if i == 0 else 0.0) - (a if i == 1 else 0.0) - 2 * r * gr[i] * k[0]) / rho2,
                        (X[1] * gr[i] + (r if i == 1 else 0.0) + (a if i == 0 else 0.0) - 2 * r * gr[i] * k[1]) / rho2,
                        ((1.0 if i == 2 else 0.0) - k[2] * gr[i]) / r])
        uf = _dot(u, gf)
        Dv = [_dot(u, [jac[0][j], jac[1][j], jac[2][j]]) for j in range(3)]
        Ev = [_dot(u, jac[j]) for j in range(3)]
        c1 = uf * s + f * _dot(u, Dv)
        w = [c1 * k[j] + f * s * (Dv[j] - Ev[j]) - 0.5 * s * s * gf[j] for j in range(3)]
        kw = _dot(k, w) - c1
        gam = [w[j] - f * k[j] * kw for j in range(3)] + [-c1 + f * kw]
        return [lor[j] - torch.where(flat, 0.0, gam[j]) for j in range(4)]

    def _area(self, K, xk, i0, i1, j0, j1):
        """AREA over [i0, i1] x [j0, j1] (axes K+1, K+2) in the plane x^K = xk."""
        gx, gw = GAUSS[self.q]
        total = torch.zeros_like(xk)
        for p in range(self.q):
            for t in range(self.q):
                pt = [None] * 3
                pt[K] = xk
                pt[(K + 1) % 3] = 0.5 * (i0 + i1) + 0.5 * (i1 - i0) * gx[p]
                pt[(K + 2) % 3] = 0.5 * (j0 + j1) + 0.5 * (j1 - j0) * gx[t]
                _, _, f, k = _kerr(*(pt[q] - self.cen[q] for q in range(3)), self.m, self.a)
                total += gw[p] * gw[t] * torch.sqrt(1.0 + f * (1.0 - k[K] ** 2))
        return 0.25 * total * (i1 - i0) * (j1 - j0)

    def _deposit(self, x0, dx, flux):
        dt = self.c["dt"]
        cell = [[], []]
        disp = [[], []]
        for ax in range(3):
            a = torch.floor(x0[ax]).clamp(0, self.n[ax] - 2)
            b = torch.floor(x0[ax] + dx[ax]).clamp(0, self.n[ax] - 2)
            s1 = torch.where(a == b, 0.5 * dx[ax], torch.maximum(a, b) - x0[ax])
            cell[0].append(a)
            cell[1].append(b)
            disp[0].append(s1)
            disp[1].append(dx[ax] - s1)
        stride = (1, self.n[0], self.n[0] * self.n[1])
        for seg in range(2):
            fr = []
            for ax in range(3):
                s = disp[0][ax] + 0.5 * disp[1][ax] if seg else 0.5 * disp[0][ax]
                fr.append((x0[ax] - cell[seg][ax]) + s)
            base = sum(cell[seg][ax].long() * stride[ax] for ax in range(3))
            for K in range(3):
                I, Jx = (K + 1) % 3, (K + 2) % 3
                ci, cj = cell[seg][I], cell[seg][Jx]
                pk, pi, pj = cell[seg][K] + fr[K], ci + fr[I], cj + fr[Jx]
                A = [self._area(K, pk, pi, ci + 1, pj, cj + 1), self._area(K, pk, ci, pi, pj, cj + 1),
                     self._area(K, pk, pi, ci + 1, cj, pj), self._area(K, pk, ci, pi, cj, pj)]
                tot = A[0] + A[1] + A[2] + A[3]
                J = self.J[K].view(-1)
                for v, off in zip(A, (0, stride[I], stride[Jx], stride[I] + stride[Jx])):
                    J.index_add_(0, base + off, flux * disp[seg][K] / dt * v / tot)

    def _push(self, p, chunk=1 << 21):
        where = torch.nonzero(p["alive"]).reshape(-1)
        for part in where.split(chunk):
            self._push_part(p, part)

    def _push_part(self, p, at):
        c, dt = self.c["c"], self.c["dt"]
        x0 = [v[at] for v in p["x"]]
        u0 = [v[at] for v in p["u"]]
        xs, us = x0[:3], u0
        sx = [torch.zeros_like(x0[0]) for _ in range(4)]
        su = [torch.zeros_like(x0[0]) for _ in range(4)]
        h = None
        for stage in range(4):
            acc = self._accel(xs, us, p["qm"])
            if stage == 0:
                w = us[3] / c
                arg = w * w + 2.0 * acc[3] * dt / c
                g = 0.5 * (w + torch.sqrt(arg.clamp(min=0.0)))
                h = dt / torch.where((arg >= 0) & (g > 0), g, w)
            wgt, frac = (1.0 if stage in (0, 3) else 2.0), (h if stage == 2 else 0.5 * h)
            for q in range(4):
                sx[q] = sx[q] + wgt * us[q]
                su[q] = su[q] + wgt * acc[q]
            xs, us = [x0[q] + frac * us[q] for q in range(3)], [u0[q] + frac * acc[q] for q in range(4)]
        dx = [h / 6.0 * v for v in sx]
        u1 = [u0[q] + h / 6.0 * su[q] for q in range(4)]
        x1 = [x0[q] + dx[q] for q in range(4)]
        self._deposit(x0, dx, p["q"] * (u0[3] + u1[3]) / (2.0 * c))
        ok = torch.ones_like(at, dtype=torch.bool)
        for q in range(3):
            ok &= (x1[q] >= 1) & (x1[q] <= self.n[q] - 2)
        if self.m > 0:
            ok &= _kerr(*(x1[q] - self.cen[q] for q in range(3)), self.m, self.a)[0] > self.r_plus
        for q in range(4):
            p["x"][q][at], p["u"][q][at] = x1[q], u1[q]
        p["alive"][at] = ok

    def particles(self, p):
        return torch.where(p["alive"], torch.stack(p["x"] + p["u"]), 0.0)


def _exact_plasma(c, species, B):
    e = Exact(c)
    e.uniform(B)
    for qm, q, x4, u4, _, umode in species:
        e.load(qm, q, x4, u4, umode)
    for _ in range(c["steps"]):
        e.step()
    return [e.particles(p) for p in e.parts], (e.d, e.b)


def _served_plasma(r, c):
    """The server's seeded plasma: SplitMix64 draws keyed by (seed, stream, counter)."""
    def mix(z):
        z = z + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))

    def uniform(stream, counter):
        key = mix(np.array([r["seed"]], np.uint64)) ^ mix(np.array([stream], np.uint64) + np.uint64(0x632BE59BD9B4E019))
        return (mix(key ^ counter) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53

    n, theta = r["n"], 0.1 ** 2
    w = n - 3
    t = np.arange(w ** 3 * r["ppc"], dtype=np.uint64)
    cell = (t // np.uint64(r["ppc"])).astype(np.int64)
    three = np.uint64(3) * t
    x = np.stack([1 + cell % w, 1 + (cell // w) % w, 1 + cell // (w * w)]).astype(np.float64)
    x += np.stack([uniform(0, three + np.uint64(i)) for i in range(3)])
    keep = ((x - 0.5 * (n - 1)) ** 2).sum(0) >= (2.5 * r["m"]) ** 2
    ug = np.sqrt((1.0 + 40.0 * theta) ** 2 - 1.0) * np.arange(20001) / 20000
    pdf = ug * ug * np.exp(-(np.sqrt(1.0 + ug * ug) - 1.0) / theta)
    cdf = np.concatenate([[0.0], np.cumsum(0.5 * (pdf[1:] + pdf[:-1]) * np.diff(ug))])
    cdf, prob = cdf / cdf[-1], np.arange(4096) / 4095
    at = np.clip(np.searchsorted(cdf, prob, side="left") - 1, 0, 19999)
    inv = ug[at] + (prob - cdf[at]) / np.maximum(cdf[at + 1] - cdf[at], 1e-300) * (ug[at + 1] - ug[at])
    q = (0.025 / 0.4) ** 2 / (4.0 * math.pi * r["ppc"] * 2.0)
    dev = lambda v: torch.from_numpy(v).to(DEV)  # noqa: E731
    out = []
    for s, qm in enumerate((-1.0, 1.0)):
        mag = np.interp(uniform(1 + s, three) * 4095, np.arange(4096), inv)
        ct, ph = 2.0 * uniform(1 + s, three + np.uint64(1)) - 1.0, 2.0 * math.pi * uniform(1 + s, three + np.uint64(2))
        sn = np.sqrt(np.maximum(0.0, 1.0 - ct * ct))
        u = np.stack([mag * sn * np.cos(ph), mag * sn * np.sin(ph), mag * ct, 0.0 * mag])
        x4 = np.concatenate([x, np.zeros((1, x.shape[1]))])
        out.append((qm, qm * q, dev(x4[:, keep]), dev(u[:, keep]), None, 1))
    return out, dev(np.nonzero(keep)[0]), x.shape[1]


def exact(case, seed):
    kind = case["kind"]
    if kind == "plasma":
        parts, fields = _exact_plasma(case, _species(case, seed), (0.0, 0.0, case["B0"]))
        return {"particles": parts, "fields": fields}
    if kind == "vacuum":
        e = Exact(case)
        e.d, e.b = _noise_field(case, seed)
        e.target()
        for _ in range(case["steps"]):
            e.step()
        return {"fields": (e.d, e.b)}
    if kind == "sweep":
        out = []
        for k in _sweep_cases(case, seed):
            parts, fields = _exact_plasma(k, _species(k, k["seed"]), (0.0, 0.0, k["B0"]))
            out.append({"particles": torch.cat(parts, 1), "fields": torch.cat(fields)})
        return out
    if kind == "serve":
        out = []
        for r in _serve_requests(case, seed):
            n = r["n"]
            c = dict(plasma_case(n, n, n, r["ppc"], r["nsteps"], r["m"], r["a"] / r["m"], layers=True), a=r["a"])
            species, ids, slots = _served_plasma(r, c)
            parts, fields = _exact_plasma(c, species, (0.0, 0.0, 0.05))
            whole = [torch.zeros((8, slots), dtype=F64, device=DEV).index_copy_(1, ids, p) for p in parts]
            out.append({"particles": torch.cat(whole, 1), "fields": torch.cat(fields)})
        return out
    e = Exact(case)
    e.d, e.b = _noise_field(case, seed)
    rho = [torch.zeros(e.d[0].numel(), dtype=F64, device=DEV) for _ in range(2)]
    for qm, q, x4, u4, _, umode in _species(case, seed):
        e.load(qm, q, x4, u4, umode)
        p = e.parts.pop()
        x = [v[p["alive"]] for v in p["x"]]
        i0 = [torch.floor(x[ax]).long() for ax in range(3)]
        w = [x[ax] - i0[ax] for ax in range(3)]
        base = (i0[2] * e.n[1] + i0[1]) * e.n[0] + i0[0]
        for dz in range(2):
            for dy in range(2):
                for dx in range(2):
                    W = q * (w[0] if dx else 1 - w[0]) * (w[1] if dy else 1 - w[1]) * (w[2] if dz else 1 - w[2])
                    at = base + (dz * e.n[1] + dy) * e.n[0] + dx
                    rho[0].index_add_(0, at, W * p["u"][3][p["alive"]] / case["c"])
                    rho[1].index_add_(0, at, W)
    div = torch.zeros_like(e.d[0])
    for ax in range(3):
        dim = 2 - ax
        diff = e.d[ax] - torch.roll(e.d[ax], 1, dims=dim)
        diff.index_fill_(dim, torch.zeros(1, dtype=torch.long, device=DEV), 0.0)
        div -= diff
    res = div - 4.0 * math.pi * rho[1].view_as(div)
    return {"rho": rho[0].view_as(div), "residual": res, "contra": torch.stack(e._h(e.d, e.b)),
            "worst": float(res[2:-2, 2:-2, 2:-2].abs().max())}

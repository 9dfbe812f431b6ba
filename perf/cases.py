"""The work a user of this library has it do, as timed cases, with a 64-bit reference of each.

listed() gives the fixed cases, draw() more of the same ranges.  prepare() makes what a
program holds before the call (seeded particles on the device or in pinned host memory, and
the simulation, ensemble or recorded adjoint it keeps); run() is one pass through the public
entry points of the binding; work() counts what the pass cannot do without; exact() computes
the same outputs in FP64 with plain torch operations.

Kinds of pass:
  bound     a simulation that steps the caller's tensors in place (Simulation.bound): `steps`
            steps; the outputs are the caller's own eight arrays, nothing is copied or waited for
  steps     a simulation that owns its particles: `steps` steps, then its particles are read
            back into device tensors, as between two outputs of a long run
  short     a whole short run from pinned host arrays: set-up, `steps` steps, the particles and
            B_z read back to pinned host arrays, clean-up
  ensemble  independent runs advanced by one captured graph, then every run's particles read
            back into device tensors
  gradient  autograd.magnetic_energy and its gradient with respect to the initial velocities:
            set-up, recorded forward run and reverse sweep
  reverse   the reverse sweep alone, on a forward run recorded once, as an optimiser or a
            sensitivity study calls it with one objective after another
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2410_18414_gb300 import autograd, pic

WEIBEL_L = 1.153896  # the periodic square of the Weibel set-up, in c/omega_pe
DIRK = {
    2: {"A": [[0.25, 0.0], [0.5, 0.25]], "b": [0.5, 0.5], "c": [0.25, 0.75]},
    3: {"A": [[1 / 6, 0.0, 0.0], [1 / 3, 1 / 6, 0.0], [1 / 3, 1 / 3, 1 / 6]],
        "b": [1 / 3, 1 / 3, 1 / 3], "c": [1 / 6, 0.5, 5 / 6]},
}
# electrons, and half as many ions of mass 25 at twice their weight: the mean charge cancels
SPECIES = ((-1.0, 1.0, 1.0), (1.0, 25.0, 2.0))
KEYS = ("x", "y", "px", "py", "vx", "vy", "vx_old", "vy_old")


def _case(name, kind, nx, ny, n, p, stepper, order, steps, fp32, **more):
    c = {"name": name, "kind": kind, "nx": nx, "ny": ny, "n": n, "p": p, "stepper": stepper,
         "order": order, "steps": steps, "fp32": fp32, "sort": 0, "vdim": 2, "species": False,
         "cloud": False, "v_drift": 0.5, "u_th": 0.01, "runs": 1, "every": 0, "mode": "replay"}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: one step of the drifting cloud of the test suite in FP64; launches
        # and their latency are all there is
        _case("cloud32_fp64_step", "bound", 32, 32, 16384, 2, "bdf", 1, 1, False, cloud=True,
              v_drift=0.1),
        # a small ragged run in the FP32 form, CDF-2, stepped on tensors a torch program owns
        _case("ragged48x32_fp32_step", "bound", 48, 32, 20011, 3, "cdf2", 2, 1, True),
        # an unsorted FP32 run of ordinary size with an odd particle count, quartic shapes
        _case("unsorted256x192_fp32_step", "bound", 256, 192, 1500001, 4, "bdf", 3, 1, True),
        # the library's main workload: 2^20 particles, cubic, BDF-2, FP32 form, sorted
        _case("weibel128_fp32", "steps", 128, 128, 1 << 20, 3, "bdf", 2, 32, True, sort=8),
        # the same in the plain FP64 form, stepped in place
        _case("weibel128_fp64", "bound", 128, 128, 1 << 20, 3, "bdf", 2, 1, False),
        # the largest run: 26 million particles, quartic, three-stage DIRK
        _case("weibel512_fp32", "steps", 512, 512, 26214400, 4, "dirk", 3, 8, True, sort=8,
              v_drift=0.6, u_th=0.02),
        # three velocity components (A_z, J_z), FP32 form, sorted
        _case("weibel128_3v_fp32", "steps", 128, 128, 1 << 20, 3, "bdf", 2, 16, True, sort=8,
              vdim=3),
        # electrons and ions on a rectangular grid, two-stage DIRK, FP32 form, sorted
        _case("ions192x96_fp32", "steps", 192, 96, 786431, 2, "dirk", 2, 16, True, sort=4,
              species=True, v_drift=0.3),
        # a parameter study: 16 independent runs on grids of 32^2 to 128^2 in one graph
        _case("ensemble16_fp32", "ensemble", 128, 128, 0, 3, "bdf", 2, 64, True, sort=8,
              runs=16),
        # a whole short run from host arrays and back
        _case("short_run96_fp32", "short", 96, 96, 400000, 3, "cdf2", 2, 20, True, sort=8),
        # the gradient of the final magnetic energy, whole, FP64 (a quarter million particles)
        _case("gradient128_fp64", "gradient", 128, 128, 262144, 3, "bdf", 2, 40, False,
              every=20),
        # one more reverse sweep of a recorded run, FP32 form
        _case("reverse64_fp32", "reverse", 64, 64, 65536, 3, "cdf2", 2, 40, True, every=10,
              mode="replay_lean"),
    ]


_SIDES = (16, 24, 32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 162, 192, 216, 256, 288, 384, 512)


def draw(rng):
    kind = rng.choice(("bound", "bound", "bound", "steps", "steps", "steps", "short", "ensemble",
                       "gradient", "reverse"))
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    nx, ny = rng.choice(_SIDES), rng.choice(_SIDES)
    p = rng.choice((2, 3, 3, 4))
    stepper, order = rng.choice((("bdf", 1), ("bdf", 2), ("bdf", 3), ("cdf2", 2),
                                 ("cdf2_semi", 2), ("cdf2_explicit", 2), ("dirk", 2),
                                 ("dirk", 3)))
    fp32 = rng.random() < 0.6
    more = {"v_drift": round(rng.uniform(0.3, 0.7), 3)}
    if kind == "bound":
        n, steps = log(4000, 4000000), rng.randint(1, 4)
    elif kind == "steps":
        n, steps = log(20000, 6000000), rng.randint(8, 32)
        more["sort"] = rng.choice((4, 8, 8, 16)) if fp32 or rng.random() < 0.5 else 0
        more["vdim"] = rng.choice((2, 2, 3))
        more["species"] = rng.random() < 0.25
    elif kind == "short":
        n, steps = log(10000, 2000000), rng.randint(10, 50)
        more["sort"] = 8 if fp32 else 0
    elif kind == "ensemble":
        nx = ny = 128
        n, steps, fp32 = 0, 48, True
        p, stepper, order = 3, "bdf", 2
        more.update(runs=rng.randint(2, 24), sort=rng.choice((4, 8)))
    else:
        n, steps = log(4000, 262144), rng.randint(5, 40)
        nx, ny = min(nx, 144), min(ny, 144)
        more.update(every=rng.randint(3, 20), mode=rng.choice(("replay", "replay_lean",
                                                               "recompute")))
        if kind == "gradient":
            more["mode"] = "replay"
    # no drawn case costs more than the largest listed one
    n = min(n, (60000000 if fp32 else 12000000) // steps)
    c = _case("", kind, nx, ny, n, p, stepper, order, steps, fp32, **more)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs ----

def _parts(case, seed):
    """The runs of a case: (nx, ny, n, v_drift, seed) each.  An ensemble's runs are squares of
    32 to 128 cells with 16 to 64 particles per cell, drawn from the seed of the case's shape
    alone, so that its work is the same for every input seed."""
    if case["kind"] != "ensemble":
        return [(case["nx"], case["ny"], case["n"], case["v_drift"], seed)]
    out = []
    for r in range(case["runs"]):
        rng = np.random.Generator(np.random.PCG64(1000 + r))
        side = int(rng.choice([32, 48, 64, 96, 128]))
        ppc = int(rng.integers(16, 65))
        out.append((side, side, side * side * ppc, float(rng.uniform(0.3, 0.7)),
                    seed * 1009 + r))
    return out


def _particles(case, part):
    """Device FP64 tensors x, y, vx, vy (and vz, species) of one run."""
    nx, ny, n, v_drift, seed = part
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    f8 = {"dtype": torch.float64, "device": "cuda"}
    lx, ly = _lengths(case, nx, ny)
    odd = torch.arange(n, device="cuda") % 2
    out = {}
    if case["cloud"]:  # a drifting Gaussian cloud
        out["x"] = torch.remainder(0.5 + 0.1 * torch.randn(n, generator=g, **f8), lx)
        out["y"] = torch.remainder(0.5 + 0.1 * torch.randn(n, generator=g, **f8), ly)
        out["vx"] = v_drift + 0.01 * torch.randn(n, generator=g, **f8)
        out["vy"] = 0.01 * torch.randn(n, generator=g, **f8)
        return out
    # two counter-streaming beams along y, uniform positions, a Maxwellian in u = gamma v
    out["x"] = lx * torch.rand(n, generator=g, **f8)
    out["y"] = ly * torch.rand(n, generator=g, **f8)
    u_d = v_drift / math.sqrt(1.0 - v_drift * v_drift)
    u = [case["u_th"] * torch.randn(n, generator=g, **f8) for _ in range(case["vdim"])]
    u[1] += torch.where(odd == 0, u_d, -u_d).to(torch.float64)
    if case["species"]:  # every third particle is an ion, at rest but for a slower spread
        ion = torch.arange(n, device="cuda") % 3 == 0
        for k in range(case["vdim"]):
            u[k] = torch.where(ion, 0.2 * case["u_th"] * torch.randn(n, generator=g, **f8), u[k])
        out["species"] = ion.to(torch.int32)
    gamma = torch.sqrt(1.0 + sum(a * a for a in u))
    for k, name in enumerate(("vx", "vy", "vz")[:case["vdim"]]):
        out[name] = u[k] / gamma
    return out


def _lengths(case, nx, ny):
    if case["cloud"]:
        return 1.0, 1.0
    return WEIBEL_L, WEIBEL_L * ny / nx


def _dt(case, nx, ny):
    lx, _ = _lengths(case, nx, ny)
    return (0.5 if case["cloud"] else 0.4) * lx / nx


def _weight(case, part):
    lx, ly = _lengths(case, part[0], part[1])
    return lx * ly / max(part[2], 1)


def _species(case, part):
    if not case["species"]:
        return None
    w = _weight(case, part)
    return tuple((q, m, s * w) for q, m, s in SPECIES)


def _config(case, part):
    nx, ny = part[0], part[1]
    lx, ly = _lengths(case, nx, ny)
    return pic.make_config(
        nx, ny, lx, ly, _dt(case, nx, ny), p=case["p"], stepper=case["stepper"],
        bdf_order=case["order"], dirk=DIRK[case["order"]] if case["stepper"] == "dirk" else None,
        weight=_weight(case, part), precision=pic.FP32_FIX64 if case["fp32"] else pic.FP64,
        sort_interval=case["sort"], vdim=case["vdim"], species=_species(case, part))


def _bz_seed(case, part):
    """The objective of a reverse sweep: the amplitude of the lowest filamentation mode."""
    nx, ny = part[0], part[1]
    lx, ly = _lengths(case, nx, ny)
    x = torch.arange(nx, dtype=torch.float64, device="cuda") / nx
    area = (lx / nx) * (ly / ny)
    return (area * torch.cos(2.0 * math.pi * x))[:, None].expand(nx, ny).contiguous()


def _momentum_seeds(part):
    g = torch.Generator(device="cuda")
    g.manual_seed(part[4] + 77)
    return [torch.randn(part[2], generator=g, dtype=torch.float64, device="cuda") / part[2]
            for _ in range(2)]


def prepare(case, seed):
    parts = _parts(case, seed)
    part, kind = parts[0], case["kind"]
    if kind == "ensemble":
        sims, outs = [], []
        for q in parts:
            a = _particles(case, q)
            torch.cuda.synchronize()  # the runs' streams do not wait for the default one
            sims.append(pic.Simulation(_config(case, q), a["x"], a["y"], a["vx"], a["vy"],
                                       stream=_stream(sims)))
            outs.append(torch.empty((8, q[2]), dtype=torch.float64, device="cuda"))
        streams = list(_streams)
        ens = pic.Ensemble(sims, _main_stream().cuda_stream)
        return {"case": case, "ens": ens, "sims": sims, "outs": outs, "streams": streams}
    a = _particles(case, part)
    cfg = _config(case, part)
    if kind == "bound":
        t = torch.float32 if case["fp32"] else torch.float64
        arrays = {k: a[k].to(t) if k in a else torch.empty(part[2], dtype=t, device="cuda")
                  for k in KEYS}
        if case["fp32"]:  # rounding may carry a position onto the end of the period
            for k, length in (("x", cfg.lx), ("y", cfg.ly)):
                arrays[k] = torch.where(arrays[k] >= length, arrays[k] - length, arrays[k])
        sim = pic.Simulation.bound(cfg, arrays, stream=torch.cuda.current_stream().cuda_stream)
        return {"case": case, "sim": sim}
    if kind == "short":
        host = {k: v.cpu().pin_memory() for k, v in a.items()}
        out = {k: torch.empty(part[2], dtype=torch.float64).pin_memory() for k in KEYS}
        bz = torch.empty((part[0], part[1]), dtype=torch.float64).pin_memory()
        return {"case": case, "cfg": cfg, "host": host, "out": out, "bz": bz}
    if kind == "gradient":
        for k in ("vx", "vy"):
            a[k].requires_grad_(True)
        return {"case": case, "cfg": cfg, "a": a}
    sim = pic.Simulation(cfg, a["x"], a["y"], a["vx"], a["vy"],
                         stream=torch.cuda.current_stream().cuda_stream, vz=a.get("vz"),
                         species=a.get("species"))
    if kind == "reverse":
        adj = pic.Adjoint(sim, case["steps"], case["every"], mode=case["mode"])
        adj.forward()
        px, py = _momentum_seeds(part)
        return {"case": case, "sim": sim, "adj": adj, "bz": _bz_seed(case, part), "px": px,
                "py": py}
    out = {k: torch.empty(part[2], dtype=torch.float64, device="cuda") for k in KEYS}
    if case["vdim"] == 3:
        for k in ("pz", "vz", "vz_old"):
            out[k] = torch.empty(part[2], dtype=torch.float64, device="cuda")
    if case["species"]:
        out["species"] = torch.empty(part[2], dtype=torch.int32, device="cuda")
    return {"case": case, "sim": sim, "out": out}


_streams = []


def _stream(sims):
    while len(_streams) <= len(sims):
        _streams.append(torch.cuda.Stream())
    return _streams[len(sims)].cuda_stream


_main = []


def _main_stream():
    if not _main:
        _main.append(torch.cuda.Stream())
    return _main[0]


# -------------------------------------------------------------------- pass ----

def run(state):
    case = state["case"]
    kind, steps = case["kind"], case["steps"]
    if kind == "bound":
        sim = state["sim"]
        sim.step(steps)
        (vx, vy), (vx_old, vy_old) = sim.velocities()
        a = sim.arrays
        return [a["x"], a["y"], a["px"], a["py"], vx, vy, vx_old, vy_old]
    if kind == "steps":
        state["sim"].step(steps)
        return state["sim"].particles(state["out"])
    if kind == "ensemble":
        state["ens"].step(steps)
        for sim, out in zip(state["sims"], state["outs"]):
            sim.particles({k: out[i] for i, k in enumerate(KEYS)})
        return state["outs"]
    if kind == "short":
        h = state["host"]
        with pic.Simulation(state["cfg"], h["x"], h["y"], h["vx"], h["vy"]) as sim:
            sim.step(steps)
            sim.particles(state["out"])
            sim.field("bz", out=state["bz"])
        return [state["out"][k] for k in KEYS] + [state["bz"]]
    if kind == "gradient":
        a = state["a"]
        wb = autograd.magnetic_energy(state["cfg"], a["x"], a["y"], a["vx"], a["vy"], steps,
                                      checkpoint_every=case["every"], mode=case["mode"])
        gx, gy = torch.autograd.grad(wb, (a["vx"], a["vy"]))
        return [wb.detach(), gx, gy]
    g = state["adj"].backward(bz_bar=state["bz"], px_bar=state["px"], py_bar=state["py"])
    return [g["vx"], g["vy"], g["px"], g["py"]]


def work(case):
    size = 4 if case["fp32"] else 8
    v = 3 if case["vdim"] == 3 else 2
    p1, w = case["p"] + 1, {2: 10, 3: 19, 4: 39}[case["p"]]
    fields = 11 if v == 3 else 8
    flops_p = 4 + 2 * w + v * (1 + p1 + 2 * p1 * p1) + p1 * p1 + 2 * fields * p1 * p1 + 31
    total = {"bytes": 0.0, "flops": 0.0}
    for nx, ny, n, _, _ in _parts(case, 0):
        ng = nx * ny
        # a step reads x, y, P, v^n, v^{n-1} (P_z too) and writes x, y, P, v^{n+1}; the
        # stepper's levels of phi, A and rho are FP64 spectra, read once and written once
        values = (8 + 6) if v == 2 else (11 + 7)
        levels = {"bdf": 7 * case["order"] + 4, "dirk": 2 * 9}.get(case["stepper"], 2 * 8 + 2)
        step_bytes = values * size * n + (16 * levels + 8 * size) * ng
        step_flops = flops_p * n + 5 * 5 * ng * math.log2(ng)
        steps = case["steps"]
        more_bytes = 0
        if case["kind"] in ("steps", "ensemble"):
            more_bytes = (8 if v == 2 else 11) * n * (size + 8)
        elif case["kind"] == "short":
            more_bytes = 4 * 8 * n + 8 * n * (size + 8)
        if case["kind"] == "reverse":  # a reversed step: the records and the adjoint state
            step_bytes, step_flops, more_bytes = 20 * size * n, 2 * step_flops, 6 * 8 * n
        if case["kind"] == "gradient":
            step_bytes, step_flops, more_bytes = 34 * size * n, 3 * step_flops, 6 * 8 * n
        total["bytes"] += steps * step_bytes + more_bytes
        total["flops"] += steps * step_flops
    return total


# ------------------------------------------------------- 64-bit reference ----

def _weights(xi, p):
    """Nodes (unwrapped; base - k) and weights of the centred cardinal B-spline of degree p."""
    s = xi + 0.5 * (p + 1)
    base = torch.floor(s.detach())
    u = s - base
    v = [torch.ones_like(u)]
    for d in range(1, p + 1):
        v = [((u + k) * v[k] if k < d else 0.0) / d + ((d + 1 - u - k) * v[k - 1] if k else 0.0) / d
             for k in range(d + 1)]
    return base.to(torch.int64), v


def _stencil(c, x, y):
    ix, wx = _weights(x / (c["lx"] / c["nx"]), c["p"])
    iy, wy = _weights(y / (c["ly"] / c["ny"]), c["p"])
    for a in range(c["p"] + 1):
        row = torch.remainder(ix - a, c["nx"]) * c["ny"]
        for b in range(c["p"] + 1):
            yield row + torch.remainder(iy - b, c["ny"]), wx[a] * wy[b]


def _deposit(c, x, y, values):
    area = (c["lx"] / c["nx"]) * (c["ly"] / c["ny"])
    grid = torch.zeros((len(values), c["nx"] * c["ny"]), dtype=torch.float64, device=x.device)
    out = list(grid)
    for node, w in _stencil(c, x, y):
        for k, v in enumerate(values):
            out[k] = out[k].index_add(0, node, v * w) if torch.is_grad_enabled() else \
                out[k].index_add_(0, node, v * w)
    return [g.reshape(c["nx"], c["ny"]) / area for g in out]


def _gather(c, x, y, fields):
    table = torch.stack([f.reshape(-1) for f in fields], dim=1)
    out = 0.0
    for node, w in _stencil(c, x, y):
        out = out + w[:, None] * table[node]
    return out.unbind(1)


def _wave(nx, ny, lx, ly, device):
    def axis(n, length):
        m = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=device)
        m[n // 2] = 0.0  # the spectral derivative of the Nyquist mode is 0
        return 2.0 * math.pi / length * m
    kx, ky = axis(nx, lx)[:, None], axis(ny, ly)[None, :]
    return kx, ky, kx * kx + ky * ky


def _bdf(k):
    alpha = [0.0] * (k + 1)
    for j in range(1, k + 1):
        for i in range(j + 1):
            alpha[i] += (-1) ** i * math.comb(j, i) / j
    a = [v / alpha[0] for v in alpha]
    square = [sum(a[j] * a[d - j] for j in range(k + 1) if 0 <= d - j <= k)
              for d in range(2 * k + 1)]
    return a, square, 1.0 / alpha[0]


def _levels(c, start):
    """Histories of one wave field: every level at its value at t = 0, derivatives 0."""
    zero = torch.zeros_like(start)
    if c["stepper"] == "bdf":
        return [start] * (2 * c["order"])
    return [start, zero] if c["stepper"] == "dirk" else [start, start]


def _advance(c, K, hist, src):
    """New level and histories of (1/c^2) u_tt + K u = S, c = 1; src: (S^{n+1}, S^n, S^{n-1})."""
    dt = c["dt"]
    if c["stepper"] == "bdf":
        a, square, beta = _bdf(c["order"])
        g = (beta * dt) ** 2
        new = g * src[0]
        for d in range(1, len(square)):
            new = new - square[d] * hist[d - 1]
        new = new / (square[0] + g * K)
        return new, [new] + hist[:-1]
    if c["stepper"] == "dirk":
        t = DIRK[c["order"]]
        u, v = hist
        ku, kv = [], []
        for i in range(c["order"]):
            ub, vb = u, v
            for j in range(i):
                ub = ub + dt * t["A"][i][j] * ku[j]
                vb = vb + dt * t["A"][i][j] * kv[j]
            s = (1.0 - t["c"][i]) * src[1] + t["c"][i] * src[0]
            h = dt * t["A"][i][i]
            force = s - K * ub
            d = 1.0 + h * h * K
            ku.append((vb + h * force) / d)
            kv.append((force - h * K * vb) / d)
        un = u + dt * sum(b * k for b, k in zip(t["b"], ku))
        vn = v + dt * sum(b * k for b, k in zip(t["b"], kv))
        return un, [un, vn]
    u, old = hist
    th = 0.5 * dt * dt
    if c["stepper"] == "cdf2":
        new = (2.0 * u + th * (src[0] + src[2])) / (1.0 + th * K) - old
    elif c["stepper"] == "cdf2_semi":
        new = (2.0 * u + 2.0 * th * src[1]) / (1.0 + th * K) - old
    else:
        new = 2.0 * u - old + 2.0 * th * (src[1] - K * u)
    return new, [new, u]


def _start(c, x, y, v, q, m, qp):
    kx, ky, K = _wave(c["nx"], c["ny"], c["lx"], c["ly"], x.device)
    with torch.no_grad():
        rho = torch.fft.fft2(_deposit(c, x, y, [qp * torch.ones_like(x)])[0])
        rho = torch.where(K > 0.0, rho, torch.zeros_like(rho))
        phi = rho / torch.where(K > 0.0, K, torch.ones_like(K))
        e = [torch.fft.ifft2(-1j * k * phi).real for k in (kx, ky)]
        e = list(_gather(c, x, y, e)) + [torch.zeros_like(x)] * (len(v) - 2)
    gamma = 1.0 / torch.sqrt(1.0 - sum(a * a for a in v))
    vdote = sum(a * b for a, b in zip(v, e))
    coef = c["dt"] * q / (gamma * m)
    zero = torch.zeros_like(phi)
    return {"x": x, "y": y, "v": v, "vo": [a - coef * (b - a * vdote) for a, b in zip(v, e)],
            "P": [gamma * m * a for a in v], "phi": _levels(c, phi),
            "A": [_levels(c, zero) for _ in v], "rho": [rho] * max(2, c["order"]),
            "J": [[zero, zero] for _ in v]}


def _step(c, s, q, m, qp):
    dt = c["dt"]
    kx, ky, K = _wave(c["nx"], c["ny"], c["lx"], c["ly"], s["x"].device)
    wrap = lambda r, length: r - length * torch.floor(r.detach() / length)  # noqa: E731
    x, y = wrap(s["x"] + s["v"][0] * dt, c["lx"]), wrap(s["y"] + s["v"][1] * dt, c["ly"])
    J = [torch.fft.fft2(j) for j in _deposit(c, x, y, [qp * a for a in s["v"]])]
    div = 1j * kx * J[0] + 1j * ky * J[1]
    rho = s["rho"]
    if c["stepper"] == "bdf":
        a, _, beta = _bdf(c["order"])
        new = -beta * dt * div - sum(a[j] * rho[j - 1] for j in range(1, len(a)))
    elif c["stepper"] == "dirk":
        t = DIRK[c["order"]]
        div_n = 1j * kx * s["J"][0][0] + 1j * ky * s["J"][1][0]
        new = rho[0] - dt * sum(b * ((1.0 - e) * div_n + e * div)
                                for b, e in zip(t["b"], t["c"]))
    else:
        new = rho[0] - dt * div
    phi, h_phi = _advance(c, K, s["phi"], (new, rho[0], rho[1]))
    A, h_A = [], []
    for k in range(len(J)):
        u, h = _advance(c, K, s["A"][k], (J[k], s["J"][k][0], s["J"][k][1]))
        A.append(u)
        h_A.append(h)
    at = phi if c["stepper"] in ("bdf", "dirk") else 0.5 * (phi + s["phi"][0])
    spectra = [1j * kx * at, 1j * ky * at]
    for u in A:
        spectra += [u, 1j * kx * u, 1j * ky * u]
    f = _gather(c, x, y, [torch.fft.ifft2(g).real for g in spectra])
    vs = [2.0 * a - b for a, b in zip(s["v"], s["vo"])]
    P = list(s["P"])
    for d in range(2):
        P[d] = P[d] + q * dt * (-f[d] + sum(f[2 + 3 * k + 1 + d] * vs[k] for k in range(len(vs))))
    u = [P[k] - q * f[2 + 3 * k] for k in range(len(vs))]
    den = torch.sqrt(sum(a * a for a in u) + m * m)
    return {"x": x, "y": y, "v": [a / den for a in u], "vo": s["v"], "P": P, "phi": h_phi,
            "A": h_A, "rho": [new] + rho[:-1], "J": [[j, o[0]] for j, o in zip(J, s["J"])]}


def _constants(case, part, a):
    sp = _species(case, part)
    if sp is None:
        return -1.0, 1.0, -_weight(case, part)
    t = torch.tensor(sp, dtype=torch.float64, device="cuda")[a["species"].long()]
    return t[:, 0], t[:, 1], t[:, 0] * t[:, 2]


def _march(case, part, a):
    nx, ny = part[0], part[1]
    lx, ly = _lengths(case, nx, ny)
    c = {"nx": nx, "ny": ny, "lx": lx, "ly": ly, "dt": _dt(case, nx, ny), "p": case["p"],
         "stepper": case["stepper"], "order": case["order"]}
    q, m, qp = _constants(case, part, a)
    v = [a["vx"], a["vy"]] + ([a["vz"]] if case["vdim"] == 3 else [])
    s = _start(c, a["x"], a["y"], v, q, m, qp)
    for _ in range(case["steps"]):
        if torch.is_grad_enabled():
            s = checkpoint(_step, c, s, q, m, qp, use_reentrant=False)
        else:
            s = _step(c, s, q, m, qp)
    kx, ky, _ = _wave(nx, ny, lx, ly, "cuda")
    bz = torch.fft.ifft2(1j * kx * s["A"][1][0] - 1j * ky * s["A"][0][0]).real
    return s, bz, (lx / nx) * (ly / ny)


def _arrays(s):
    return [s["x"], s["y"], s["P"][0], s["P"][1], s["v"][0], s["v"][1], s["vo"][0], s["vo"][1]]


def exact(case, seed):
    parts = _parts(case, seed)
    part, kind = parts[0], case["kind"]
    a = _particles(case, part) if kind != "ensemble" else None
    if kind in ("gradient", "reverse"):
        if case["n"] * case["steps"] > 12000000:
            return None
        for k in ("vx", "vy"):
            a[k].requires_grad_(True)
        s, bz, area = _march(case, part, a)
        if kind == "gradient":
            wb = 0.5 * area * (bz * bz).sum()
            return [wb.detach(), *torch.autograd.grad(wb, (a["vx"], a["vy"]))]
        px, py = _momentum_seeds(part)
        obj = (_bz_seed(case, part) * bz).sum() + (px * s["P"][0]).sum() + (py * s["P"][1]).sum()
        gx, gy = torch.autograd.grad(obj, (a["vx"], a["vy"]))
        vx, vy = a["vx"].detach(), a["vy"].detach()
        # with P^0 = gamma m v^0 the independent variable: dv/dP = (I - v v^T) / gamma (m = c = 1)
        root, along = torch.sqrt(1.0 - vx * vx - vy * vy), vx * gx + vy * gy
        return [gx, gy, root * (gx - vx * along), root * (gy - vy * along)]
    with torch.no_grad():
        if kind == "ensemble":
            out = []
            for q in parts:
                out.append(torch.stack(_arrays(_march(case, q, _particles(case, q))[0])))
            return out
        s, bz, _ = _march(case, part, a)
        out = _arrays(s)
        if kind == "bound":
            return out
        if kind == "short":
            return out + [bz]
        out = dict(zip(KEYS, out))
        if case["vdim"] == 3:
            out.update(pz=s["P"][2], vz=s["v"][2], vz_old=s["vo"][2])
        if case["species"]:
            out["species"] = a["species"]
        return out

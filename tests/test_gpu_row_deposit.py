"""The row deposit (a warp's lanes on the words of one particle's stencil) where it can go
wrong: particle counts around a warp and a CTA, every particle in one cell (neighbours added
before their atomic) or anywhere (wrapping at every edge), the smallest and largest grid sides.

FP64: J against the same sums in extended precision (numpy.longdouble, at least 64 bits of
mantissa).  A contribution carries at most six roundings of 2^-62 in its two weights, one of
2^-63 in v, 2^-61 in v W_x and 2^-60 in the product, all in units of c: below 2^-58 in all, so
a node of n particles is within n 2^-57 c; the sum's conversion to FP64 and its scaling add
three roundings, 2^-51 |J| at most.  FP32: the int64 sums against oracle.fixed_point, bit for
bit (as in test_gpu_fixed_point)."""
import numpy as np
import pytest

from oracle import fixed_point as fx
from paper_2410_18414_gb300 import pic

pytestmark = pytest.mark.gpu


def _weights(xi, p):
    s = xi + np.longdouble(p + 1) / 2
    base = np.floor(s)
    u = s - base
    w = [np.ones_like(u)]
    for d in range(1, p + 1):
        w = [((u + k) * w[k] if k < d else 0) / d + ((d + 1 - u - k) * w[k - 1] if k else 0) / d
             for k in range(d + 1)]
    return base.astype(np.int64), w  # node base - k has weight w[k]


def _deposit(x, y, v, nx, ny, lx, ly, p):
    side = 62 - int(np.ceil(np.log2(max(nx, ny))))
    scale = np.longdouble(2) ** side
    xi = np.rint((x * (1.0 / (lx / nx))).astype(np.longdouble) * scale) / scale
    yj = np.rint((y * (1.0 / (ly / ny))).astype(np.longdouble) * scale) / scale
    ix, wx = _weights(xi, p)
    iy, wy = _weights(yj, p)
    out = np.zeros((nx, ny), dtype=np.longdouble)
    for a in range(p + 1):
        for b in range(p + 1):
            np.add.at(out, ((ix - a) % nx, (iy - b) % ny), v * wx[a] * wy[b])
    return out


@pytest.mark.parametrize("nx,ny,n,one_cell", [(8, 8, 1, False), (16, 12, 31, False),
                                              (16, 12, 33, True), (32, 8, 129, True),
                                              (8, 1024, 1000, False), (54, 36, 4099, False),
                                              # from 65,536 particles on: one index a stencil
                                              (8, 8, 65536, False), (54, 36, 65539, True)])
@pytest.mark.parametrize("p", [2, 3, 4])
def test_row_deposit(p, nx, ny, n, one_cell):
    rng = np.random.default_rng(1000 * p + n)
    lx, ly = 1.0, ny / nx
    dt = 0.3 * min(lx / nx, ly / ny)
    x, y = rng.uniform(0, lx, n), rng.uniform(0, ly, n)
    vx, vy = rng.uniform(-0.6, 0.6, n), rng.uniform(-0.6, 0.6, n)
    if one_cell:
        x, y = (2.4 + 0.1 * x) * lx / nx, (3.4 + 0.1 * y / ly) * ly / ny
        vx, vy = 0.1 * vx, 0.1 * vy
    weight = lx * ly / n
    area = (lx / nx) * (ly / ny)
    for precision in (pic.FP64, pic.FP32_FIX64):
        cfg = pic.make_config(nx, ny, lx, ly, dt, p=p, weight=weight, precision=precision)
        with pic.Simulation(cfg, x, y, vx, vy) as sim:
            sim.step(1)
            got, j = sim.particles(), (sim.field("jx"), sim.field("jy"))
        if precision == pic.FP64:
            for have, v in zip(j, (vx, vy)):
                want = -weight / area * _deposit(got["x"], got["y"], v, nx, ny, lx, ly, p)
                bound = weight / area * n * 2.0 ** -57 + 2.0 ** -51 * np.abs(want)
                assert np.all(np.abs(have - want) <= bound)
        else:
            scale = fx.current_scale(1.0, n)
            x1, y1, ix, iy = fx.move_deposit(x, y, vx, vy, dt, lx, ly, nx, ny, p, scale)
            assert np.array_equal(got["x"], x1.astype(np.float64))
            for have, q in zip(j, (ix, iy)):
                want = np.asarray(q, dtype=np.float64) * (1.0 / scale * (weight * -1.0 / area))
                assert np.array_equal(have, want)


def _gather(x, y, grid, lx, ly, p):
    nx, ny = grid.shape
    ix, wx = _weights((x * (1.0 / (lx / nx))).astype(np.longdouble), p)
    iy, wy = _weights((y * (1.0 / (ly / ny))).astype(np.longdouble), p)
    return sum(grid.astype(np.longdouble)[(ix - a) % nx, (iy - b) % ny] * wx[a] * wy[b]
               for a in range(p + 1) for b in range(p + 1))


@pytest.mark.parametrize("nx,ny,n", [(8, 8, 7), (8, 8, 8), (16, 12, 33), (8, 1024, 1025),
                                     (54, 36, 4099)])
@pytest.mark.parametrize("p", [2, 3, 4])
def test_row_gather_fp64(p, nx, ny, n):
    """The momentum update of one step from the mesh fields the library reports, against the
    gather in extended precision; counts on both sides of the fixed-point form's rule (n below
    nx ny / 8 takes the FP64 arithmetic).  A gathered value is within 2^-51 of the field's
    largest: at most 25 weights off by 2^-58, 2^-58 of the bound (up to twice the largest) for
    the fields' rounding and as much for the result's, 25 2^-60 of it for the dropped sum, and
    2^-53 from the conversion; FP64's own roundings are of that size too.  The force's three
    terms (|v*| < 3 c) and the update add 2^-53 of each."""
    rng = np.random.default_rng(77 * p + n)
    lx, ly = 1.0, ny / nx
    dt = 0.3 * min(lx / nx, ly / ny)
    x, y = rng.uniform(0, lx, n), rng.uniform(0, ly, n)
    vx, vy = rng.uniform(-0.6, 0.6, n), rng.uniform(-0.6, 0.6, n)
    cfg = pic.make_config(nx, ny, lx, ly, dt, p=p, weight=lx * ly / n)
    with pic.Simulation(cfg, x, y, vx, vy) as sim:
        sim.step(1)
        before = sim.particles()
        sim.step(1)
        after = sim.particles()
        names = ("dphidx", "dphidy", "daxdx", "daxdy", "daydx", "daydy")
        f = {k: sim.field(k) for k in names}
    g = {k: _gather(after["x"], after["y"], f[k], lx, ly, p) for k in names}
    vs = [2 * before[k].astype(np.longdouble) - before[k + "_old"] for k in ("vx", "vy")]
    for c, key in (("x", "px"), ("y", "py")):
        terms = (g["dphid" + c], g["daxd" + c] * vs[0], g["dayd" + c] * vs[1])
        want = before[key] - dt * (-terms[0] + terms[1] + terms[2])
        peak = sum(np.max(np.abs(f[k])) for k in ("dphid" + c, "daxd" + c, "dayd" + c))
        bound = dt * (3 * 2.0 ** -51 * peak + 2.0 ** -51 * sum(np.abs(t) for t in terms))
        assert np.all(np.abs(after[key] - want) <= bound + 2.0 ** -52 * np.abs(want))


@pytest.mark.parametrize("vdim", [2, 3])
@pytest.mark.parametrize("nx,ny,n", [(8, 8, 7), (8, 8, 8), (16, 12, 33), (54, 36, 1025)])
@pytest.mark.parametrize("p", [2, 3, 4])
def test_row_gather_fp64_species(p, nx, ny, n, vdim):
    """As test_row_gather_fp64 with a species table and, at vdim 3, the A_z fields: the
    momenta, with a fourth term of the force, and the velocities v = u / sqrt(u^2 + m^2) with
    u = P - q A (c = 1).  A gathered A is within 2^-51 of its peak and u adds 2^-51 of its two
    terms; |dv/du_c| <= 1 / m for each component, and the root and the quotient add less than
    2^-50 of v."""
    rng = np.random.default_rng(177 * p + n)
    lx, ly = 1.0, ny / nx
    dt = 0.3 * min(lx / nx, ly / ny)
    x, y = rng.uniform(0, lx, n), rng.uniform(0, ly, n)
    vx, vy, vz = (rng.uniform(-0.5, 0.5, n) for _ in range(3))
    sp = rng.integers(0, 2, n).astype(np.int32)
    w = lx * ly / n
    qs, ms = np.array([-1.0, 0.5])[sp], np.array([1.0, 4.0])[sp]
    cfg = pic.make_config(nx, ny, lx, ly, dt, p=p, vdim=vdim,
                          species=((-1.0, 1.0, w), (0.5, 4.0, 2 * w)))
    comps = ("x", "y", "z")[:vdim]
    with pic.Simulation(cfg, x, y, vx, vy, vz=vz if vdim == 3 else None, species=sp) as sim:
        sim.step(1)
        before = sim.particles()
        sim.step(1)
        after = sim.particles()
        f = {k: sim.field(k) for k in ["dphidx", "dphidy"] + [f"a{a}" for a in comps]
             + [f"da{a}d{c}" for a in comps for c in "xy"]}
    g = {k: _gather(after["x"], after["y"], f[k], lx, ly, p) for k in f}
    peak = {k: np.max(np.abs(f[k])) for k in f}
    vs = {a: 2 * before["v" + a].astype(np.longdouble) - before[f"v{a}_old"] for a in comps}
    for c in "xy":
        terms = [-g["dphid" + c]] + [g[f"da{a}d{c}"] * vs[a] for a in comps]
        want = before["p" + c] + qs * dt * sum(terms)
        peaks = peak["dphid" + c] + sum(peak[f"da{a}d{c}"] for a in comps)
        bound = np.abs(qs) * dt * (3 * 2.0 ** -51 * peaks
                                   + 2.0 ** -51 * sum(np.abs(t) for t in terms))
        assert np.all(np.abs(after["p" + c] - want) <= bound + 2.0 ** -52 * np.abs(want)), c
    u = {a: after["p" + a] - qs * g["a" + a] for a in comps}
    du = sum(np.abs(qs) * 2.0 ** -51 * peak["a" + a]
             + 2.0 ** -51 * (np.abs(after["p" + a]) + np.abs(qs * g["a" + a])) for a in comps)
    den = np.sqrt(sum(u[a] ** 2 for a in comps) + (ms * ms).astype(np.longdouble))
    for a in comps:
        want = u[a] / den
        assert np.all(np.abs(after["v" + a] - want) <= du / ms + 2.0 ** -50 * np.abs(want)), a


@pytest.mark.parametrize("n", [1, 31, 33, 129, 1000])
@pytest.mark.parametrize("p", [2, 3, 4])
def test_row_gather_fp32_is_the_sorted_gather(p, n):
    """The FP32 gather's lane pairs against the tiled gather of the sorted form: same bits."""
    rng = np.random.default_rng(7 * p + n)
    x, y = rng.uniform(0, 1.0, n), rng.uniform(0, 0.75, n)
    vx, vy = rng.uniform(-0.6, 0.6, n), rng.uniform(-0.6, 0.6, n)
    out = []
    for sort in (0, 1):
        cfg = pic.make_config(32, 24, 1.0, 0.75, 0.01, p=p, weight=0.75 / n,
                              precision=pic.FP32_FIX64, sort_interval=sort)
        with pic.Simulation(cfg, x, y, vx, vy) as sim:
            sim.step(3)
            out.append(sim.particles())
    for k in out[0]:
        assert np.array_equal(out[0][k], out[1][k]), k

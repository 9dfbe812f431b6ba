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
                                              (8, 1024, 1000, False), (54, 36, 4099, False)])
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

"""The rounding of the FP64 deposit's contributions: nearest, with no one-sided error, for the
current, J_z and both forms of the row deposit (below and from 65,536 particles on)."""
import numpy as np
import pytest

from paper_2410_18414_gb300 import pic
from test_gpu_row_deposit import _deposit

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pairs", [301, 33001])
@pytest.mark.parametrize("vdim", [2, 3])
@pytest.mark.parametrize("p", [2, 3, 4])
def test_opposite_velocities_cancel(p, vdim, pairs):
    """Two particles that meet at one place with velocities v and -v leave no current at all: the
    velocities (multiples of 2^-30), dt and the places (multiples of 2^-20) have so few bits that
    the moves are exact."""
    rng = np.random.default_rng(pairs + p)
    at = rng.integers(1 << 17, 7 << 17, (2, pairs)) * 2.0 ** -20
    v = rng.integers(-(1 << 17), 1 << 17, (3, pairs)) * 2.0 ** -30
    dt = 2.0 ** -10
    x, y = (np.concatenate([at[c] - v[c] * dt, at[c] + v[c] * dt]) for c in range(2))
    vx, vy, vz = (np.concatenate([a, -a]) for a in v)
    order = rng.permutation(2 * pairs)
    cfg = pic.make_config(24, 18, 1.0, 1.0, dt, p=p, weight=0.5 / pairs, vdim=vdim)
    with pic.Simulation(cfg, x[order], y[order], vx[order], vy[order],
                        vz=vz[order] if vdim == 3 else None) as sim:
        sim.step(1)
        for k in ("jx", "jy") + (("jz",) if vdim == 3 else ()):
            assert not np.any(sim.field(k)), k


@pytest.mark.parametrize("n", [4099, 65539])
@pytest.mark.parametrize("p", [2, 3, 4])
def test_no_mean_error_in_a_cold_current(p, n):
    """A current of 1e-6 c without drift, summed over the mesh, against extended precision: the
    errors of n (p+1)^2 contributions, at most 0.8 quanta (2^-60 c) each and of either sign, add
    up to less than six standard deviations; a node's FP64 value adds 2^-50 of itself."""
    rng = np.random.default_rng(n + p)
    x, y = rng.uniform(0, 1.0, n), rng.uniform(0, 1.0, n)
    vx, vy = 1e-6 * rng.standard_normal(n), 1e-6 * rng.standard_normal(n)
    cfg = pic.make_config(32, 32, 1.0, 1.0, 0.01, p=p, weight=1.0 / n)
    with pic.Simulation(cfg, x, y, vx, vy) as sim:
        sim.step(1)
        got, j = sim.particles(), (sim.field("jx"), sim.field("jy"))
    to_quanta = np.longdouble(2) ** 60 / (-np.longdouble(1.0 / n) * 32 * 32)
    for have, v in zip(j, (vx, vy)):
        want = _deposit(got["x"], got["y"], v, 32, 32, 1.0, 1.0, p) * np.longdouble(2) ** 60
        err = have.astype(np.longdouble) * to_quanta - want
        bound = 6 * 0.8 * np.sqrt(n) * (p + 1) + np.longdouble(2) ** -50 * np.sum(np.abs(want))
        assert abs(np.sum(err)) <= bound

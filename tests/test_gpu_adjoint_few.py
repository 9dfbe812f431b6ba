"""The FP64 adjoint of runs with few particles on the mesh, whose gathers stay in FP64 arithmetic
(fewer than nx ny / 8 particles), and of runs just above that rule, whose gathers run in fixed
point: both against the oracle's gradient, within the parity bound of test_gpu_adjoint (1e-11)."""
import numpy as np
import pytest

from oracle import adjoint as oadj
from oracle import pic as opic
from paper_2410_18414_gb300 import pic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["replay", "replay_lean"])
@pytest.mark.parametrize("n", [31, 95, 96, 129])
@pytest.mark.parametrize("p", [2, 3, 4])
def test_few_particles(p, n, mode):
    import torch
    rng = np.random.default_rng(10 * p + n)
    nx, ny, lx, ly = 32, 24, 1.0, 0.75
    x, y = rng.uniform(0, lx, n), rng.uniform(0, ly, n)
    vx, vy = rng.uniform(-0.5, 0.5, n), rng.uniform(-0.5, 0.5, n)
    w, dt = lx * ly / n, 0.4 * lx / nx
    cfg = pic.make_config(nx, ny, lx, ly, dt, p=p, stepper="bdf", bdf_order=2, weight=w)
    ocfg = opic.Config(nx=nx, ny=ny, lx=lx, ly=ly, dt=dt, p=p, stepper="bdf", bdf_order=2, w=w)
    pb = (rng.standard_normal(n), rng.standard_normal(n))
    want = oadj.gradient(oadj.record(ocfg, x, y, vx, vy, 5), px_bar=pb[0], py_bar=pb[1])
    with pic.Simulation(cfg, x, y, vx, vy) as sim:
        with pic.Adjoint(sim, 5, 2, mode=mode) as adj:
            adj.forward()
            got = adj.backward(px_bar=torch.tensor(pb[0], device="cuda"),
                               py_bar=torch.tensor(pb[1], device="cuda"))
    for key, ref in (("vx", want["v0"][0]), ("vy", want["v0"][1]), ("px", want["p0"][0]),
                     ("py", want["p0"][1])):
        have = got[key].cpu().numpy()
        assert np.linalg.norm(have - ref) <= 1e-11 * np.linalg.norm(ref), key

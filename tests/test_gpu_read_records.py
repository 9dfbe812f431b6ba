"""The read-back of sorted runs too large for one pass through L2, by records, against the
read-back to host memory, between steps that use the records' memory for the next sort."""
import numpy as np
import pytest

from paper_2410_18414_gb300 import pic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n", [(pic.FP32_FIX64, 2100003), (pic.FP64, 1050001)])
def test_read_back_by_records(precision, n):
    import torch
    rng = np.random.default_rng(5)
    x, y = rng.random(n), rng.random(n)
    vx, vy = 0.3 * rng.uniform(-1, 1, n), 0.3 * rng.uniform(-1, 1, n)
    cfg = pic.make_config(64, 64, 1.0, 1.0, 0.005, p=2, weight=1.0 / n, precision=precision,
                          sort_interval=2)
    with pic.Simulation(cfg, x, y, vx, vy) as sim:
        sim.step(3)
        host = sim.particles()
        device = {k: torch.empty(n, dtype=torch.float64, device="cuda") for k in host}
        sim.particles(device)
        sim.step(2)  # the records' memory is the sort's again
        after = sim.particles()
    with pic.Simulation(cfg, x, y, vx, vy) as sim:
        sim.step(5)
        straight = sim.particles()
    for k in host:
        assert np.array_equal(host[k], device[k].cpu().numpy()), k
        assert np.array_equal(after[k], straight[k]), k

"""A velocity above c that a caller writes into its bound FP64 arrays is reported, not deposited
as whatever its fixed-point product wraps to; speeds up to c are deposited as they are."""
import numpy as np
import pytest

from paper_2410_18414_gb300 import pic

pytestmark = pytest.mark.gpu


def _sim(n, p):
    import torch

    rng = np.random.default_rng(n)
    arrays = {k: torch.zeros(n, dtype=torch.float64, device="cuda") for k in pic.Simulation.BOUND_KEYS}
    for k, v in (("x", rng.uniform(0, 1, n)), ("y", rng.uniform(0, 1, n)),
                 ("vx", rng.uniform(-0.5, 0.5, n)), ("vy", rng.uniform(-0.5, 0.5, n))):
        arrays[k].copy_(torch.tensor(v))
    cfg = pic.make_config(16, 16, 1.0, 1.0, 0.01, p=p, weight=1.0 / n)
    return pic.Simulation.bound(cfg, arrays, stream=torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("p", [2, 3, 4])
@pytest.mark.parametrize("n", [100, 65600])
def test_speeds_above_c_are_reported(p, n):
    for speed in (1.9, -3.0, 1e30):
        with _sim(n, p) as sim:
            sim.arrays["vy"][n // 2] = speed
            with pytest.raises(pic.PicError, match="NONFINITE"):
                sim.step(1)
                sim.sync()


@pytest.mark.parametrize("p", [2, 3, 4])
def test_the_speed_of_light_is_deposited(p):
    """sum of J over the mesh is q weight sum of v / area (the weights add up to 1), within the
    rounding of 100 particles' contributions, 2^-55 c each."""
    with _sim(100, p) as sim:
        sim.arrays["vx"][:50] = 1.0
        sim.arrays["vx"][50:] = -1.0
        sim.arrays["vx"][7] = -1.0
        sim.step(1)
        total = np.sum(sim.field("jx"))
    assert abs(total - (-1.0 / 100 * 256) * -2.0) <= 256 * 2.0 ** -48

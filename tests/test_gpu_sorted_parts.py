"""Sorted runs whose particles crowd into few tiles: the CTAs of the binned pass are cut from the
tiles' own counts at each sort (several parts of one tile, none for an empty one), through a
checkpoint as well, and give the unsorted run's bits."""
import numpy as np
import pytest

from paper_2410_18414_gb300 import pic

pytestmark = pytest.mark.gpu


def _crowd(n, seed, share=0.9):
    """Most of the particles in a disc of two cells, the others anywhere (moving slowly, so
    that tiles fill and empty between the sorts)."""
    rng = np.random.default_rng(seed)
    inside = rng.random(n) < share
    x = np.where(inside, 0.4 + 0.03 * rng.standard_normal(n), rng.random(n)) % 1.0
    y = np.where(inside, 0.3 + 0.03 * rng.standard_normal(n), rng.random(n)) % 0.75
    v = [0.3 * rng.uniform(-1, 1, n) for _ in range(3)]
    return x, y, v


@pytest.mark.parametrize("vdim", [2, 3])
@pytest.mark.parametrize("p,n", [(2, 5000), (3, 30001), (4, 12000)])
def test_crowded_tiles_give_the_unsorted_bits(p, n, vdim):
    x, y, v = _crowd(n, 10 * p + vdim)
    z = {"vz": v[2]} if vdim == 3 else {}
    out = []
    for sort in (0, 2):
        cfg = pic.make_config(48, 36, 1.0, 0.75, 0.008, p=p, weight=0.75 / n, vdim=vdim,
                              precision=pic.FP32_FIX64, sort_interval=sort)
        with pic.Simulation(cfg, x, y, v[0], v[1], **z) as sim:
            sim.step(5)
            state = sim.save_state()
            sim.step(4)
            out.append(sim.particles())
        if sort:  # the parts are rebuilt from the loaded tile offsets
            with pic.Simulation(cfg, x, y, v[0], v[1], **z) as sim:
                sim.load_state(state)
                sim.step(4)
                out.append(sim.particles())
    for other in out[1:]:
        for k in out[0]:
            assert np.array_equal(out[0][k], other[k]), k

"""The row deposit's other forms: one component a node (J_z, the charge), where two or three
particles share a warp's pass, and the allocation-free FP64 sums, with particle counts on both
sides of 65,536 and around warps, on grids where many stencils wrap."""
import ctypes

import numpy as np
import pytest

from paper_2410_18414_gb300 import pic
from test_gpu_row_deposit import _deposit

pytestmark = pytest.mark.gpu

COUNTS = [1, 31, 33, 1003, 65535, 65571]


def _particles(n, seed, ly):
    rng = np.random.default_rng(seed)
    return (rng.uniform(0, 1.0, n), rng.uniform(0, ly, n), rng.uniform(-0.5, 0.5, n),
            rng.uniform(-0.5, 0.5, n))


@pytest.mark.parametrize("precision", [pic.FP64, pic.FP32_FIX64])
@pytest.mark.parametrize("n", COUNTS)
@pytest.mark.parametrize("p", [2, 3, 4])
def test_jz_is_jx_of_equal_velocities(p, n, precision):
    """With v_z = v_x every contribution to J_z is the integer that goes to J_x (which
    test_gpu_row_deposit compares with extended precision)."""
    x, y, vx, vy = _particles(n, n + p, 0.75)
    cfg = pic.make_config(24, 18, 1.0, 0.75, 0.3 / 24, p=p, weight=0.75 / n, precision=precision,
                          vdim=3)
    with pic.Simulation(cfg, x, y, vx, vy, vz=vx.copy()) as sim:
        sim.step(1)
        jx = sim.field("jx")
        assert np.any(jx) and np.array_equal(sim.field("jz"), jx)


@pytest.mark.parametrize("precision", [pic.FP64, pic.FP32_FIX64])
@pytest.mark.parametrize("n", COUNTS)
@pytest.mark.parametrize("p", [2, 3, 4])
def test_deposited_charge(p, n, precision):
    """rho of the naive update (without the modes whose wavenumbers are both 0, the Nyquist ones
    among them) against extended precision.  Positions in cells carry at most 24 2^-24 (FP32) a
    axis, the weights a few roundings more, the transforms there and back some ten of the largest
    value: below 100 roundings of it; one particle of 65,571 on 432 nodes is 2^-8 of a node at
    the least."""
    x, y, vx, vy = _particles(n, 2 * n + p, 0.75)
    nx, ny = 24, 18
    cfg = pic.make_config(nx, ny, 1.0, 0.75, 0.3 / nx, p=p, weight=0.75 / n, precision=precision,
                          charge=pic.CHARGE_DEPOSIT)
    with pic.Simulation(cfg, x, y, vx, vy) as sim:
        sim.step(1)
        got, rho = sim.particles(), sim.field("rho")
    want = _deposit(got["x"], got["y"], np.ones(n), nx, ny, 1.0, 0.75, p) * (-1.0 / n * nx * ny)
    spec = np.fft.fft2(want.astype(np.float64))
    spec[::nx // 2, ::ny // 2] = 0.0
    eps = 2.0 ** -53 if precision == pic.FP64 else 2.0 ** -24
    assert np.max(np.abs(rho - np.fft.ifft2(spec).real)) <= 100 * eps * np.max(np.abs(want))


@pytest.mark.parametrize("n", [33, 65571])
@pytest.mark.parametrize("p", [2, 3, 4])
def test_allocation_free_sums(p, n):
    """FP64 atomics against extended precision: each contribution rounds its two weights and two
    products (below 2^-50 of itself in all), its position differs from the reference's by 2^-58 of a
    cell (2^-57 in each weight), the sum of a node's n adds n 2^-53 of the magnitudes at most."""
    import torch

    lib = pic.load_library()
    fn = lib.pic_move_deposit_noalloc
    fn.argtypes = [ctypes.POINTER(pic.PicConfig), ctypes.c_int64] + [ctypes.c_void_p] * 7
    fn.restype = ctypes.c_int32
    nx, ny = 24, 18
    host = _particles(n, 3 * n + p, 0.75)
    cfg = pic.make_config(nx, ny, 1.0, 0.75, 0.3 / nx, p=p, weight=0.75 / n)
    dev = [torch.tensor(a, device="cuda") for a in host]
    j = [torch.full((nx, ny), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2)]
    st = fn(ctypes.byref(cfg), n, *[t.data_ptr() for t in dev], *[t.data_ptr() for t in j],
            torch.cuda.current_stream().cuda_stream)
    assert st == pic.PIC_OK
    x, y = (t.cpu().numpy() for t in dev[:2])
    for have, v in zip(j, host[2:]):
        factor = -1.0 / n * nx * ny
        want = _deposit(x, y, v, nx, ny, 1.0, 0.75, p) * factor
        size = _deposit(x, y, np.abs(v), nx, ny, 1.0, 0.75, p) * abs(factor)
        assert np.all(np.abs(have.cpu().numpy() - want) <= (2.0 ** -50 + n * 2.0 ** -53) * size
                      + n * 2.0 ** -56 * abs(factor))

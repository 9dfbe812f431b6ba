"""The kernel timers: the groups of a timed reverse sweep add up to about the time that the sweep
takes without them."""
import pytest

from paper_2410_18414_gb300 import pic, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [pic.FP32_FIX64, pic.FP64])
def test_reverse_groups_add_up(precision):
    """Three groups of each of 40 reversed BDF-2 steps.  An untimed step overlaps its kernels'
    starts, a few microseconds of about 122 (FP32 form) and 210 (FP64), and the sweep has work
    outside the groups: their sum is within 15% of the sweep."""
    import torch

    wl = workloads.weibel_adjoint_128(seed=5)
    cfg = pic.make_config(wl.nx, wl.ny, wl.lx, wl.ly, wl.dt, p=wl.p, stepper="bdf", bdf_order=2,
                          weight=wl.weight, precision=precision)
    dev = [torch.tensor(getattr(wl, k), device="cuda") for k in ("x", "y", "vx", "vy")]
    bz = torch.ones((wl.nx, wl.ny), dtype=torch.float64, device="cuda")
    steps = 40
    with pic.Simulation(cfg, *dev, stream=torch.cuda.current_stream().cuda_stream) as sim:
        with pic.Adjoint(sim, steps, steps) as adj:
            adj.forward()

            def sweep():
                ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                torch.cuda.synchronize()
                ev[0].record()
                adj.backward(bz_bar=bz)
                ev[1].record()
                torch.cuda.synchronize()
                return ev[0].elapsed_time(ev[1])

            sweep()
            tried = []
            for _ in range(12):  # until once: other programs on the GPU disturb either time
                plain = min(sweep() for _ in range(3))
                sim.set_kernel_timing(steps + 1)
                sweep()
                timers = [sim.kernel_time(k) for k in ("adj_push", "adj_field", "adj_deposit")]
                sim.set_kernel_timing(0)
                assert [n for _, n in timers] == [steps] * 3
                tried.append(sum(ms for ms, _ in timers) / plain)
                if 0.85 <= tried[-1] <= 1.15:
                    return
    raise AssertionError(tried)

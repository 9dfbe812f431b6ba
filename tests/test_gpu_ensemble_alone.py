"""Ensemble runs that were advanced alone, or given a saved state, between replays: their buffers
may then stand in another rotation than the one the graph was captured in.  The next replay gives
the bits of pic_step all the same."""
import numpy as np
import pytest

from paper_2410_18414_gb300 import pic, workloads

pytestmark = pytest.mark.gpu

# precision, sort interval, stepper, vdim
FORMS = [(pic.FP32_FIX64, 4, dict(stepper="bdf", bdf_order=2), 2),
         (pic.FP32_FIX64, 2, dict(stepper="cdf2"), 2),
         (pic.FP32_FIX64, 4, dict(stepper="bdf", bdf_order=1), 3),
         (pic.FP32_FIX64, 0, dict(stepper="bdf", bdf_order=3), 2),
         (pic.FP64, 2, dict(stepper="bdf", bdf_order=2), 3),
         (pic.FP64, 0, dict(stepper="cdf2"), 2)]


def _make(form):
    import torch

    precision, sort, kw, vdim = form
    wl = workloads.weibel(32, 24, 16, 0.4, 0.01, 77, 3)
    vz = np.random.default_rng(5).uniform(-0.1, 0.1, wl.n) if vdim == 3 else None
    cfg = pic.make_config(wl.nx, wl.ny, wl.lx, wl.ly, wl.dt, p=wl.p, weight=wl.weight,
                          precision=precision, sort_interval=sort, vdim=vdim, **kw)
    return pic.Simulation(cfg, wl.x, wl.y, wl.vx, wl.vy, vz=vz,
                          stream=torch.cuda.Stream().cuda_stream)


def _same(a, b):
    pa, pb = a.particles(), b.particles()
    assert a.step_count == b.step_count
    for k in pa:
        assert np.array_equal(pa[k], pb[k]), k
    for k in ("jx", "phi", "ay", "daxdy"):
        assert np.array_equal(a.field(k), b.field(k)), k


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("calls", [(1, 1), (2, 1), (1, 1, 1), (1, 1, 1, 1)])
def test_stepped_alone_by_whole_periods(form, calls):
    """Each call one or two periods; every call that follows another starts with the pending
    deposit of the one before."""
    import torch

    run, other, solo = _make(form), _make(form), _make(form)
    with pic.Ensemble([run, other], torch.cuda.Stream().cuda_stream) as ens:
        P = ens.period
        for k in calls:
            run.step(k * P)
            solo.step(k * P)
        for _ in range(2):
            ens.step(P)
            solo.step(P)
            _same(run, solo)
        run.step(1)
        solo.step(1)
        _same(run, solo)
    for s in (run, other, solo):
        s.close()


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("steps", [1, 3])
def test_state_loaded_after_an_odd_number_of_steps(form, steps):
    import torch

    run, solo = _make(form), _make(form)
    state = run.save_state()
    with pic.Ensemble([run], torch.cuda.Stream().cuda_stream) as ens:
        run.step(steps)
        run.load_state(state)
        ens.step(ens.period)
        solo.step(ens.period)
        _same(run, solo)
    run.close()
    solo.close()

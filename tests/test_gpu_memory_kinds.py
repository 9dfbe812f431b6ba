"""Particles and fields to and from every kind of memory: a kernel reads and writes this device's
memory and page-locked host memory in place, pageable memory takes copies.  Each gives the bits of
the pageable arrays, from the start of an allocation, inside it and up to its end."""
import numpy as np
import pytest

from paper_2410_18414_gb300 import pic

pytestmark = pytest.mark.gpu

KINDS = ("device", "pinned", "pinned inside")


def _array(kind, n, dtype="float64"):
    import torch

    t = getattr(torch, dtype)
    if kind == "device":
        return torch.full((n,), -7, dtype=t, device="cuda")
    if kind == "pinned":
        return torch.full((n,), -7, dtype=t).pin_memory()
    return torch.full((n + 3,), -7, dtype=t).pin_memory()[3:]


@pytest.mark.parametrize("precision,sort,vdim", [(pic.FP64, 0, 2), (pic.FP32_FIX64, 0, 2),
                                                 (pic.FP32_FIX64, 2, 2), (pic.FP64, 2, 3),
                                                 (pic.FP32_FIX64, 2, 3)])
@pytest.mark.parametrize("n", [1, 257, 5000])
def test_memory_kinds(n, precision, sort, vdim):
    import torch

    rng = np.random.default_rng(n + vdim)
    x, y = rng.uniform(0, 1.0, n), rng.uniform(0, 0.75, n)
    vx, vy, vz = (rng.uniform(-0.5, 0.5, n) for _ in range(3))
    cfg = pic.make_config(24, 18, 1.0, 0.75, 0.01, p=3, weight=0.75 / n, precision=precision,
                          sort_interval=sort, vdim=vdim)
    names = ("bz", "ax", "jx") + (("jz", "dazdx") if vdim == 3 else ())

    def run(arrays, out=None, fields=None):
        with pic.Simulation(cfg, *arrays[:4], vz=arrays[4] if vdim == 3 else None) as sim:
            sim.step(5)
            got = sim.particles(out) if out else sim.particles()
            return got, {k: sim.field(k, out=fields[k] if fields else None) for k in names}

    host = [x, y, vx, vy, vz]
    want, wantf = run(host)
    for kind in KINDS:
        arrays = [_array(kind, n) for _ in host]
        for a, b in zip(arrays, host):
            a.copy_(torch.from_numpy(b))
        out = {k: _array(kind, n) for k in want}
        fields = {k: _array(kind, 24 * 18) for k in names}
        run(arrays, out, fields)
        for k in want:
            assert np.array_equal(np.asarray(out[k].cpu()), want[k]), (kind, k)
        for k in names:
            assert np.array_equal(np.asarray(fields[k].cpu()).reshape(24, 18), wantf[k]), (kind, k)

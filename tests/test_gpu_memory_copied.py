"""Memory that no kernel may use in place (registered and managed memory, addresses that are not
a multiple of eight bytes, on the host and on the device) takes copies: the bits of the pageable
arrays, and nothing beside the arrays is written."""
import ctypes
import mmap

import numpy as np
import pytest

from paper_2410_18414_gb300 import pic

pytestmark = pytest.mark.gpu

N, NX, NY = 1003, 24, 18


@pytest.fixture(scope="module")
def cudart():
    for name in ("libcudart.so.13", "/usr/local/cuda/lib64/libcudart.so"):
        try:
            return ctypes.CDLL(name)
        except OSError:
            continue
    pytest.skip("no CUDA runtime library to allocate from")


class _Device:
    """`n` doubles of device memory that start 4 bytes past a multiple of eight."""

    def __init__(self, n):
        import torch

        self.raw = torch.zeros(8 * n + 16, dtype=torch.uint8, device="cuda")
        self.n, self.dtype = n, torch.float64

    def data_ptr(self):
        return self.raw.data_ptr() + 4

    def is_contiguous(self):
        return True

    def read(self):
        raw = self.raw.cpu().numpy()
        assert not np.any(raw[:4]) and not np.any(raw[4 + 8 * self.n:])
        return raw[4:4 + 8 * self.n].view(np.float64)


class _Pool:
    """Host arrays of one kind; close() gives the memory back."""

    def __init__(self, kind, cudart):
        self.kind, self.rt, self.keep = kind, cudart, []

    def array(self, n):
        if self.kind == "registered":
            m = mmap.mmap(-1, 8 * n)
            a = np.frombuffer(m, dtype=np.float64, count=n)
            assert self.rt.cudaHostRegister(ctypes.c_void_p(a.ctypes.data),
                                            ctypes.c_size_t(8 * n), 0) == 0
            self.keep.append((a, m))
            return a
        if self.kind == "managed":
            p = ctypes.c_void_p()
            assert self.rt.cudaMallocManaged(ctypes.byref(p), ctypes.c_size_t(8 * n), 1) == 0
            self.keep.append(p)
            return np.frombuffer((ctypes.c_char * (8 * n)).from_address(p.value), dtype=np.float64)
        import torch

        raw = torch.zeros(8 * n + 16, dtype=torch.uint8).pin_memory()
        self.keep.append(raw)
        return raw.numpy()[4:4 + 8 * n].view(np.float64)

    def close(self):
        import torch

        torch.cuda.synchronize()
        for k in self.keep:
            if self.kind == "registered":
                assert self.rt.cudaHostUnregister(ctypes.c_void_p(k[0].ctypes.data)) == 0
            elif self.kind == "managed":
                assert self.rt.cudaFree(k) == 0
            else:
                raw = k.numpy()
                assert not np.any(raw[:4]) and not np.any(raw[-12:])


def _case(precision, sort):
    rng = np.random.default_rng(9)
    x, y = rng.uniform(0, 1.0, N), rng.uniform(0, 0.75, N)
    vx, vy = rng.uniform(-0.5, 0.5, N), rng.uniform(-0.5, 0.5, N)
    return [x, y, vx, vy], pic.make_config(NX, NY, 1.0, 0.75, 0.01, p=3, weight=0.75 / N,
                                           precision=precision, sort_interval=sort)


def _run(cfg, arrays, out=None, bz=None):
    with pic.Simulation(cfg, *arrays) as sim:
        sim.step(5)
        return sim.particles(out) if out else sim.particles(), sim.field("bz", out=bz)


@pytest.mark.parametrize("precision,sort", [(pic.FP64, 0), (pic.FP32_FIX64, 0),
                                            (pic.FP32_FIX64, 2), (pic.FP64, 2)])
@pytest.mark.parametrize("kind", ["registered", "managed", "misaligned"])
def test_host_memory(cudart, kind, precision, sort):
    host, cfg = _case(precision, sort)
    want, want_bz = _run(cfg, host)
    pool = _Pool(kind, cudart)
    arrays = [pool.array(N) for _ in host]
    for a, b in zip(arrays, host):
        a[:] = b
    out = {k: pool.array(N) for k in want}
    bz = pool.array(NX * NY)
    _run(cfg, arrays, out, bz)
    for k in want:
        assert np.array_equal(out[k], want[k]), k
    assert np.array_equal(bz.reshape(NX, NY), want_bz)
    del arrays, out, bz
    pool.close()


@pytest.mark.parametrize("precision,sort", [(pic.FP64, 0), (pic.FP32_FIX64, 2)])
def test_device_memory_off_alignment(precision, sort):
    host, cfg = _case(precision, sort)
    want, want_bz = _run(cfg, host)
    out, bz = {k: _Device(N) for k in want}, _Device(NX * NY)
    _run(cfg, host, out, bz)
    for k in want:
        assert np.array_equal(out[k].read(), want[k]), k
    assert np.array_equal(bz.read().reshape(NX, NY), want_bz)

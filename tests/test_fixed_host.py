"""The integer arithmetic of the FP64 particle kernels (csrc/fixed.cuh), compiled for the CPU with
the signed-overflow sanitizer and compared with exact rational arithmetic."""
import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not (shutil.which("g++") and os.path.exists(nvcc)):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("fixed") / "fixed_host")
    cmd = ["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-fsanitize=undefined",
           "-fno-sanitize-recover=all",
           "-I", os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include"),
           "-I", os.path.join(ROOT, "include"),
           "-I", os.path.join(ROOT, "paper_2410_18414_gb300", "csrc"),
           os.path.join(ROOT, "tests", "fixed_host.cpp"), "-o", exe]
    subprocess.run(cmd, check=True, capture_output=True, text=True)

    def run(what, p, sh, data, *more):
        r = subprocess.run([exe, what, str(p), str(sh), *map(str, more)], input=data.tobytes(),
                           capture_output=True, timeout=300)
        assert r.returncode == 0, r.stderr.decode()[-2000:]
        return np.frombuffer(r.stdout, dtype=np.int64)

    return run


def spline(p, x, order=0):
    """The centred cardinal B-spline of degree p (or its derivative) at the rational x."""
    q = p - order
    total = sum((-1) ** k * math.comb(p + 1, k) * (x + Fraction(p + 1, 2) - k) ** q
                for k in range(p + 2) if x + Fraction(p + 1, 2) - k > 0)
    return Fraction(total) / math.factorial(q)


@pytest.mark.parametrize("p", [2, 3, 4])
def test_weights_and_derivatives(host, p):
    """Weights and derivatives in units of 2^-62 at offsets over the whole cell, its ends and the
    upper twentieth among them.  A multiply-high rounds down by less than one unit and a shift to
    units of 2^-60 (2^-58) by less than 4 (16) of them; the largest coefficients are 9 (12) and
    the sums of their magnitudes 16 (34), times 2/3 (16/24 in steps of 16): below 64 for the
    derivatives and 16 * 34 / 24 + 4 < 64 for the weights, whose last one takes the others'."""
    sh = 54
    rng = np.random.default_rng(p)
    u = np.concatenate([rng.integers(0, 1 << sh, 300), np.arange(4), (1 << sh) - 1 - np.arange(4),
                        rng.integers(int(0.94 * (1 << sh)), 1 << sh, 100)])
    X = (rng.integers(0, 256, u.size) << sh) + u
    out = host("shape", p, sh, X).reshape(-1, 2 * p + 3)
    for x, row in zip(X.tolist(), out.tolist()):
        xi = Fraction(x, 1 << sh)
        for a in range(p + 1):
            at = xi - (row[0] + a)
            assert abs(row[1 + a] - spline(p, at) * 2 ** 62) <= 64 * (p + 1)
            assert abs(row[2 + p + a] - spline(p, at, 1) * 2 ** 62) <= 64 * (p + 1)
        assert sum(row[1:p + 2]) == 2 ** 62 and sum(row[p + 2:]) == 0


@pytest.mark.parametrize("p", [2, 3, 4])
def test_deposit_rounding(host, p):
    """Contributions v W_x W_y (v in quarters of the quantum): nearest within what the rounding of
    the row factor (half of 1/8, times W_y <= 3/4) and the odd weight (t 2^-65 < 1/4, with t up
    to 2^63) add, -v the exact opposite of v, and no mean error: errors of at most 0.8 quanta
    average below 6 * 0.8 / sqrt(N)."""
    sh = 54
    rng = np.random.default_rng(40 + p)
    special = [0, 1, -1, 2, 3, 1 << 61, 1 << 62, 1 << 60, (1 << 62) - 1, 12345]
    v = np.concatenate([rng.integers(-(1 << 62), 1 << 62, 300), rng.integers(-(1 << 40), 1 << 40, 300),
                        rng.integers(-5000, 5000, 300), np.array(special)])
    X, Y = (rng.integers(0, 1 << 60, v.size) for _ in range(2))
    X[::7] &= ~np.int64((1 << (sh - 2)) - 1)  # on quarters of a cell: weights with few bits
    Y[::7] &= ~np.int64((1 << (sh - 2)) - 1)
    wx, wy = (host("shape", p, sh, c).reshape(-1, 2 * p + 3)[:, 1:p + 2].tolist() for c in (X, Y))
    n2 = (p + 1) ** 2
    plus = host("deposit", p, sh, np.stack([v, X, Y], 1)).reshape(-1, n2)
    minus = host("deposit", p, sh, np.stack([-v, X, Y], 1)).reshape(-1, n2)
    assert np.array_equal(minus, -plus)
    total = 0.0
    for k, vk in enumerate(v.tolist()):
        exact = [Fraction(vk * a * b, 1 << 126) for a in wx[k] for b in wy[k]]
        errs = [float(x - e) for x, e in zip(plus[k].tolist(), exact)]
        assert max(map(abs, errs)) <= 0.5 + 0.75 / 16 + 0.25
        total += sum(errs)
    assert abs(total) <= 6 * 0.8 * math.sqrt(v.size * n2)


def _weights(xi, p):
    """Nodes (base - k), weights and derivatives in extended precision."""
    s = xi.astype(np.longdouble) + np.longdouble(p + 1) / 2
    base = np.floor(s)
    u = s - base
    w = [np.ones_like(u)]
    for d in range(1, p + 1):
        low = w
        w = [((u + k) * w[k] if k < d else 0) / d + ((d + 1 - u - k) * w[k - 1] if k else 0) / d
             for k in range(d + 1)]
    dw = [(low[k] if k < p else 0) - (low[k - 1] if k else 0) for k in range(p + 1)]
    return base.astype(np.int64), w, dw


def _gather(f, x, y, p):
    """The value, its derivative along x and along y."""
    nx, ny = f.shape
    (ix, wx, dx), (iy, wy, dy) = _weights(x, p), _weights(y, p)
    v = {(a, b): f.astype(np.longdouble)[(ix - a) % nx, (iy - b) % ny]
         for a in range(p + 1) for b in range(p + 1)}
    return [sum(q[a] * r[b] * v[a, b] for a, b in v) for q, r in ((wx, wy), (dx, wy), (wx, dy))]


def _host_gather(host, f, x, y, p, sh):
    data = np.concatenate([[f.shape[0], f.shape[1], x.size], f.ravel(), x, y])
    out = host("gather", p, sh, data).view(np.float64).reshape(-1, 4).T
    return out[0], out[1:]  # the value with products of weights; value, d/dx, d/dy separably


@pytest.mark.parametrize("nx,ny", [(32, 32), (16, 1024)])
@pytest.mark.parametrize("p", [2, 3, 4])
def test_gather_beside_a_peak(host, p, nx, ny):
    """Rows where one node holds 1 and the others noise of 1e-17 (the size of a transform's error),
    gathered away from that node.  In units u = 2^-60 of the row's bound 2: the field's rounding,
    each row's sum and its shift add errors of variance 1/12 (the first and the derivatives' rows
    weighted, at most by 2), the others vanish with the fields: below 1 u rms and no mean."""
    rng = np.random.default_rng(p + ny)
    f = 1e-17 * rng.uniform(-1, 1, (nx, ny))
    f[5, 7] = 1.0
    n, sh = 2000, 52
    x, y = 5 + rng.uniform(-0.9, 0.9, n), rng.uniform(11.0, ny - 3.0, n)
    x, y = (np.rint(v * 2.0 ** 40) / 2.0 ** 40 for v in (x, y))
    want = _gather(f, x, y, p)
    two, sep = _host_gather(host, f, x, y, p, sh)
    u = 2.0 ** -59
    for have, ref in zip((two, *sep), (want[0], *want)):
        err = ((have - ref) / u).astype(np.float64)
        assert np.sqrt(np.mean(err ** 2)) <= 1.0
        assert abs(np.mean(err)) <= 6 / np.sqrt(n)


@pytest.mark.parametrize("p", [2, 3, 4])
def test_gather_of_uneven_rows(host, p):
    """Rows of very different size, zeros and powers of two among them: every result within its
    worst case.  In u (2^-60 of the stencil's largest row bound): half for each rounded field,
    row sum and shift, half a unit for each dropped product of low limbs, and (p+1)^2 weights off
    by 64 (p+1) 2^-62 at the very most (see test_weights_and_derivatives), a quarter of a unit
    of u each, doubled for derivatives; FP64's rounding of the result besides."""
    rng = np.random.default_rng(90 + p)
    nx, ny, n, sh = 24, 16, 1500, 57
    f = rng.standard_normal((nx, ny)) * 10.0 ** rng.integers(-25, 8, (nx, 1))
    f[3] = 0.0
    f[8] = 2.0 ** rng.integers(-40, 3, ny)
    x, y = rng.uniform(0, nx, n), rng.uniform(0, ny, n)
    x, y = (np.rint(v * 2.0 ** 45) / 2.0 ** 45 for v in (x, y))
    want = _gather(f, x, y, p)
    two, sep = _host_gather(host, f, x, y, p, sh)
    ix = _weights(x, p)[0]
    top = np.max([np.max(np.abs(f), axis=1)[(ix - a) % nx] for a in range(p + 1)], axis=0)
    u = 2.0 ** np.floor(np.log2(np.maximum(top, 1e-300)) + 1) * 2.0 ** -60
    worst = 2 * (0.5 + (p + 2) + 0.5 * (p + 1) ** 2 + 0.25 * (p + 1) ** 2 * 64 * (p + 1))
    for have, ref in zip((two, *sep), (want[0], *want)):
        assert np.all(np.abs(have - ref) <= worst * u + 2.0 ** -53 * np.abs(ref))

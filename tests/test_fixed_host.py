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

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

"""The float64 functions of the pair terms (csrc/f64math.cuh), compiled for the
host with seeds of the device's accuracy and checked against 40-digit
arithmetic.  Bounds in units of 2^-53 of the result: two roundings after a
correction of relative size 2^-20 (sqrt, 1 / sqrt, 1 / x: 2); an exact leading
part, a series of at most 2^-8 and three roundings (the logarithms: 3)."""
import os
import shutil
import struct
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2401_13708_gb300", "csrc")


def bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def number(h):
    return struct.unpack("<d", struct.pack("<Q", int(h, 16)))[0]


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("f64math") / "f64math_check")
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-I", CSRC, os.path.join(HERE, "f64math_check.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(xs):
        out = subprocess.run([exe], input="".join("%x\n" % bits(x) for x in xs), capture_output=True, text=True,
                             check=True).stdout
        return [[number(h) for h in line.split()] for line in out.splitlines()]
    return run


def test_errors_in_units_of_the_last_place(driver):
    getcontext().prec = 40
    rng = np.random.default_rng(3)
    xs = list(10.0 ** rng.uniform(-36, 33, 1500)) + list(10.0 ** rng.uniform(-3, 1, 1500))
    # table boundaries: 1 + g and x on and next to (1 + (j + 1/2) / 128) 2^k
    edges = [(1.0 + (j + 0.5) / 128.0) * 2.0 ** k for j in range(128) for k in (0, 1, 30)]
    xs += [e - 1.0 for e in edges] + [np.nextafter(e, 0.0) for e in edges] + [1.0 + 2.0 ** -k for k in range(1, 50)]
    xs = [float(x) for x in xs if x > 0.0]
    for x, (t, rs, rc, l1, lx) in zip(xs, driver(xs)):
        d = Decimal(x)
        want = {"sqrt": (t, d.sqrt(), 2), "rsqrt": (rs, 1 / d.sqrt(), 2), "reciprocal": (rc, 1 / d, 2),
                "log1p": (l1, (1 + d).ln() if x > 1e-12 else d - d * d / 2 + d * d * d / 3, 3), "log": (lx, d.ln(), 3)}
        for name, (got, ref, limit) in want.items():
            err = abs(Decimal(got) - ref) * 2 ** 53
            assert err <= limit * abs(ref), (name, x, got)

"""The quantised polar coordinates in float32 pairs (csrc/polar.cuh), compiled
for the host: wherever the pairs decide a coordinate they give the float64
definition's value, next to quantisation steps and octant lines too, and they
decide nearly always."""
import math
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2401_13708_gb300", "csrc")


def bits(x):
    return "%x" % struct.unpack("<Q", struct.pack("<d", float(x)))[0]


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("polar") / "polar_check")
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-I", CSRC,
                        os.path.join(HERE, "polar_check.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(x, y, lo, hi, area):
        text = "".join("%s %s %s %s %d\n" % (bits(a), bits(b), bits(lo), bits(hi), area) for a, b in zip(x, y))
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [[int(v) for v in line.split()] for line in out.splitlines()]
    return run


def quantise(u):
    return min(max(math.floor(u * 2.0 ** 29), 0), 2 ** 29 - 1)


@pytest.mark.parametrize("area", [0, 1])
@pytest.mark.parametrize("r0,r1", [(0.0, 0.05), (1e-3, 0.9), (0.76, 0.99999), (0.5, 0.50001)])
def test_decided_coordinates_are_the_definition(driver, r0, r1, area):
    rng = np.random.default_rng(5)
    n = 4000
    r = rng.uniform(r0, r1, n)
    phi = rng.uniform(0.0, 2.0 * math.pi, n)
    phi[:400] = math.pi / 4.0 * rng.integers(0, 8, 400) + rng.normal(0.0, 1e-12, 400)
    step = 2.0 * math.pi / 2.0 ** 29
    phi[400:800] = step * rng.integers(0, 2 ** 29, 400) + rng.normal(0.0, 1e-13, 400)
    x, y = r * np.cos(phi), r * np.sin(phi)
    x[-4:], y[-4:] = [0.0, 0.0, -r1, 1e-300], [0.0, -r1, 0.0, 1e-300]
    n2 = x * x + y * y
    c = (1.0 + n2) / (1.0 - n2) if area else np.sqrt(n2)
    lo, hi = float(c.min()), float(c.max())
    sure_a = sure_r = 0
    for i, (a, qa, b, qr) in enumerate(driver(x, y, lo, hi, area)):
        if a:
            p = math.atan2(y[i], x[i])
            assert qa == quantise((p + 2.0 * math.pi if p < 0 else p) / (2.0 * math.pi)), i
            sure_a += 1
        if b:
            assert qr == quantise((c[i] - lo) / (hi - lo)), i
            sure_r += 1
    assert sure_a > n - 900  # (all but those put on steps and lines)
    assert sure_r > n - 100 if hi - lo >= hi / 4.0 else sure_r == 0

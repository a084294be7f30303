"""csrc/polar.cuh and csrc/f64math.cuh as the device runs them (the host builds of
the other tests have other roundings to choose from, and other seeds): wherever
the float pairs decide a coordinate they give the float64 definition's value,
and they decide nearly always; the float64 functions keep the bounds of
test_f64math_host.py."""
import math
import os
import shutil
import struct
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2401_13708_gb300", "csrc")


def bits(x):
    return "%x" % struct.unpack("<Q", struct.pack("<d", float(x)))[0]


def compiled(folder, *flags):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not found")
    exe = str(folder / "device_math_check")
    r = subprocess.run([nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_103a,code=sm_103a", *flags, "-I", CSRC,
                        os.path.join(HERE, "device_math_check.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(mode, lines):
        out = subprocess.run([exe, mode], input="".join(lines), capture_output=True, text=True, check=True).stdout
        return [[int(v, 16) for v in line.split()] for line in out.splitlines()]
    return run


@pytest.fixture(scope="module")
def keys_build(tmp_path_factory):
    return compiled(tmp_path_factory.mktemp("keys"))


@pytest.fixture(scope="module")
def walk_build(tmp_path_factory):
    return compiled(tmp_path_factory.mktemp("walk"), "-ftz=true")  # (as traverse.cu)


def quantise(u):
    return min(max(math.floor(u * 2.0 ** 29), 0), 2 ** 29 - 1)


@pytest.mark.parametrize("area", [0, 1])
@pytest.mark.parametrize("r0,r1", [(0.0, 0.05), (1e-3, 0.9), (0.76, 0.99999), (0.5, 0.50001)])
def test_decided_coordinates_are_the_definition(keys_build, r0, r1, area):
    rng = np.random.default_rng(6)
    n = 20000
    r = rng.uniform(r0, r1, n)
    phi = rng.uniform(0.0, 2.0 * math.pi, n)
    phi[:400] = math.pi / 4.0 * rng.integers(0, 8, 400) + rng.normal(0.0, 1e-12, 400)
    phi[400:800] = 2.0 * math.pi / 2.0 ** 29 * rng.integers(0, 2 ** 29, 400) + rng.normal(0.0, 1e-13, 400)
    x, y = r * np.cos(phi), r * np.sin(phi)
    x[-4:], y[-4:] = [0.0, 0.0, -r1, 1e-300], [0.0, -r1, 0.0, 1e-300]
    n2 = x * x + y * y
    c = (1.0 + n2) / (1.0 - n2) if area else np.sqrt(n2)
    lo, hi = float(c.min()), float(c.max())
    sure_a = sure_r = 0
    lines = ["%s %s %s %s %x\n" % (bits(a), bits(b), bits(lo), bits(hi), area) for a, b in zip(x, y)]
    for i, (a, qa, b, qr, _) in enumerate(keys_build("polar", lines)):
        if a:
            p = math.atan2(y[i], x[i])
            assert qa == quantise((p + 2.0 * math.pi if p < 0 else p) / (2.0 * math.pi)), i
            sure_a += 1
        if b:
            assert qr == quantise((c[i] - lo) / (hi - lo)), i
            sure_r += 1
    assert sure_a > n - 1000  # (all but those put on steps and lines)
    assert sure_r > n - 100 if hi - lo >= hi / 4.0 else sure_r == 0


def test_float64_functions_in_units_of_the_last_place(walk_build):
    getcontext().prec = 40
    rng = np.random.default_rng(4)
    xs = list(10.0 ** rng.uniform(-36, 33, 1500)) + list(10.0 ** rng.uniform(-3, 1, 1500))
    edges = [(1.0 + (j + 0.5) / 128.0) * 2.0 ** k for j in range(128) for k in (0, 1, 30)]
    xs += [e - 1.0 for e in edges] + [np.nextafter(e, 0.0) for e in edges] + [1.0 + 2.0 ** -k for k in range(1, 50)]
    xs += [4e-300, 2.0 ** -127, 2.0 ** 126, np.nextafter(2.0 ** -127, 0.0), np.nextafter(2.0 ** 127, 0.0)]
    low = [5e-324, 1e-310, 2.0 ** 127, 2.0 ** 128, 1e300]  # (log alone: the library's outside its tables)
    xs = [float(x) for x in xs + low if x > 0.0]
    for k, (x, row) in enumerate(zip(xs, walk_build("math", ["%s\n" % bits(x) for x in xs]))):
        t, rs, rc, l1, lx = (struct.unpack("<d", struct.pack("<Q", v))[0] for v in row)
        d = Decimal(x)
        want = {"log": (lx, d.ln(), 3)}
        if k < len(xs) - len(low):
            want.update({"sqrt": (t, d.sqrt(), 2), "rsqrt": (rs, 1 / d.sqrt(), 2), "reciprocal": (rc, 1 / d, 2),
                         "log1p": (l1, (1 + d).ln() if x > 1e-12 else d - d * d / 2 + d * d * d / 3, 3)})
        for name, (got, ref, limit) in want.items():
            err = abs(Decimal(got) - ref) * 2 ** 53
            assert err <= limit * abs(ref), (name, x, got)

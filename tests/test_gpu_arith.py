"""The device arithmetic the marches are built from, against plain 64-bit numpy."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe():
    import torch
    from paper_1411_3246_gb300 import build
    assert torch.cuda.is_available()
    out = os.path.join(HERE, "_build", "device_arith.so")
    os.makedirs(os.path.dirname(out), exist_ok=True)
    flags = ["-O3", "-std=c++17", *build.ARCH, *build.EXTRA["march_mixed.cu"], "-Xcompiler", "-fPIC", "-shared"]
    subprocess.check_call(["nvcc", *flags, "-o", out, os.path.join(HERE, "device_arith.cu"), "-lcudart"])
    return C.CDLL(out)


def _call(fn, *arrays):
    assert fn(*[C.c_void_p(a.data_ptr()) for a in arrays]) == 0


@pytest.mark.parametrize("seed", range(4))
def test_float_float_sums_stay_normalised(probe, seed):
    """A sum's high part is the sum rounded to FP32 (the pair is normalised, so its low part holds 24 bits
    below it).  Error: a level's addition loses at most 2^-45 of the sum of the magnitudes; five levels."""
    import torch
    rng = np.random.default_rng(seed)
    x = np.exp(rng.uniform(-3, 3, 32)) * (1 if seed % 2 else rng.choice([-1.0, 1.0], 32))
    h = x.astype(np.float32)
    lo = (x - h).astype(np.float32)
    want = np.cumsum(h.astype(np.float64) + lo.astype(np.float64))
    size = np.cumsum(np.abs(x))
    dev = [torch.from_numpy(a.copy()).cuda() for a in (h, lo, h, lo)]
    _call(probe.probe_ff_scan, *dev)
    oh, ol = [d.cpu().numpy() for d in dev[2:]]
    assert np.array_equal(oh, (oh.astype(np.float64) + ol.astype(np.float64)).astype(np.float32))
    assert np.all(np.abs(oh.astype(np.float64) + ol.astype(np.float64) - want) <= 5 * 2.0 ** -45 * size)


def _fp64(probe, a, b):
    import torch
    out = torch.empty(6, a.size, dtype=torch.float64, device="cuda")
    da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    assert probe.probe_fp64(a.size, *[C.c_void_p(t.data_ptr()) for t in (da, db, out)]) == 0
    return out.cpu().numpy()


def _ulps(x, y):
    return np.abs(x - y) / np.spacing(np.abs(y))


# exponents of the operands: all that the functions take, the marches' own (Gamma and radii), next to the
# smallest square that the marches take as off the axis, around one
@pytest.mark.parametrize("lo,hi", [(-960, 1000), (-30, 30), (-964, -940), (0, 1)])
def test_fp64_reciprocal_and_root(probe, lo, hi):
    """Against the IEEE division and root: the reciprocal and the root are the rounded value or its
    neighbour; the root's reciprocal is within two ulp of 1/sqrt, and numpy's, from a rounded root, within
    one: three."""
    rng = np.random.default_rng(abs(hi))
    a = np.ldexp(rng.uniform(1, 2, 40000), rng.integers(lo, hi, 40000))
    a[:2000] = np.ldexp(1 + np.arange(-1000, 1000) * 2.0 ** -52, int(rng.integers(lo, hi)))  # around a power of two
    rcp, r, ir = _fp64(probe, a, np.ones_like(a))[:3]
    assert _ulps(rcp, 1 / a).max() <= 1
    assert (rcp != 1 / a).mean() <= 0.03  # beside a midpoint only: 2^-6 of the values
    assert _ulps(r, np.sqrt(a)).max() <= 1
    assert _ulps(ir, 1 / np.sqrt(a)).max() <= 3


def test_fp64_reciprocals_of_a_pair(probe):
    """Gamma in [1e-6, 1e6] and a radius from the smallest off the axis to 1e3: the product's rounding, its
    reciprocal's and the last product's, 3/2 2^-52 of the value in all: three ulp."""
    rng = np.random.default_rng(3)
    a, b = np.exp(rng.uniform(-13.8, 13.8, 40000)), 10.0 ** rng.uniform(-145, 3, 40000)
    ia, ib = _fp64(probe, a, b)[3:5]
    assert _ulps(ia, 1 / a).max() <= 3
    assert _ulps(ib, 1 / b).max() <= 3


def test_fp64_quotients_find_the_division_s_cells(probe):
    """Positions at and next to the nodes of boxes of 2 to 2,048 cells lie in the cell that the division
    gives; quotients of any numbers are the division's or its neighbour."""
    rng = np.random.default_rng(4)
    n = rng.integers(2, 2049, 60000)
    d = rng.choice([6.0, 8.0, 10.0, 12.0, 16.0, 25.0], n.size) / n
    x = rng.integers(0, n + 1) * d
    x = np.where(rng.random(n.size) < 0.3, np.nextafter(x, 100.0), np.where(rng.random(n.size) < 0.4, np.nextafter(x, 0.0), x))
    q = _fp64(probe, x, d)[5]
    assert np.array_equal(np.floor(q), np.floor(x / d))
    a, b = np.exp(rng.uniform(-20, 20, 40000)), np.exp(rng.uniform(-20, 20, 40000))
    q = _fp64(probe, a, b)[5]
    assert _ulps(q, a / b).max() <= 1 and (q != a / b).mean() <= 1e-4

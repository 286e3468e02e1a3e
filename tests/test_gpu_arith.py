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

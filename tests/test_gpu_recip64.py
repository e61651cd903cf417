"""recip64's device branch (hardware estimate and one third-order step) against
the division: within one unit in the last place wherever the estimate is a
normal number (its cubed error, 2^-60, and two roundings of the last multiply-
add), and the division's value where it is not (zeros, infinities, NaN, results
beyond the normal range)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reciprocal_on_the_device(tmp_path):
    import torch
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    so = str(tmp_path / "device_recip64.so")
    subprocess.run([nvcc, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared", "-cudart", "shared", "-Xcompiler", "-fPIC",
                    "-gencode", "arch=compute_103a,code=sm_103a", os.path.join(ROOT, "tests", "device_recip64.cu"), "-o", so],
                   check=True)
    L = ctypes.CDLL(so)
    L.device_recip64.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    rng = np.random.default_rng(1)
    near = 1.0 + rng.normal(size=400000) * 10.0 ** rng.uniform(-12, -0.5, size=400000)
    wide = rng.choice([-1.0, 1.0], size=400000) * 2.0 ** rng.uniform(-1073, 1023, size=400000)
    step = np.concatenate([np.nextafter(2.0 ** k, s * np.inf) for k in range(-4, 5) for s in (-1, 1)] * 1, axis=None)
    odd = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.0 ** -1022, 2.0 ** -1023, 2.0 ** 1022, 2.0 ** 1023,
                    np.finfo(np.float64).max, -np.finfo(np.float64).max, np.finfo(np.float64).tiny])
    x = np.concatenate([near, wide, step, odd])
    d = torch.tensor(x, device="cuda")
    o = torch.zeros_like(d)
    torch.cuda.synchronize()
    assert L.device_recip64(d.data_ptr(), o.data_ptr(), x.size) == 0
    got = o.cpu().numpy()
    with np.errstate(all="ignore"):
        want = 1.0 / x
    normal = np.isfinite(want) & (np.abs(want) >= np.finfo(np.float64).tiny)
    assert np.array_equal(got[~normal], want[~normal], equal_nan=True)
    ulp = np.spacing(np.abs(want[normal]))
    assert np.all(np.abs(got[normal] - want[normal]) <= ulp)
    assert np.array_equal(np.signbit(got[-14:-10]), np.signbit(want[-14:-10]))

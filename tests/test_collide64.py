"""The FP64 collisions with fewer FP64 instructions (lbm_collide64.cuh), built
for the host, against the FP64 oracle's node collision: BGK on every lattice
and the trimmed SMRT (tau_3 = tau_4 = 1) on D2Q9, over deviations of 1e-1 to
1e-6 of the weights and relaxation times near both ends of the usual range.
Bound: 1e-15 of the deviation scale per unit of population, i.e. a few units
in the last place of the largest intermediate value (an O(1) multiple of the
deviations), plus the oracle's own rounding of populations near w <= 4/9."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle as O

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "host_collide64.cu")
LATS = {0: O.D2Q9, 1: O.D3Q19, 2: O.D3Q27}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("collide64") / "host_collide64.so")
    subprocess.run([nvcc, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC", "-gencode",
                    "arch=compute_103a,code=sm_103a", SRC, "-o", out], check=True)
    L = ctypes.CDLL(out)
    P = ctypes.POINTER(ctypes.c_double)
    L.host_collide64.argtypes = [ctypes.c_int, ctypes.c_int, P, P, ctypes.c_double, P]
    return L


def _dp(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


# the kernel's velocities in its population order (include/lbm.h)
C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
C19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
       (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
C27 = C19 + [(1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1)]


@pytest.mark.parametrize("lat,trim", [(0, 0), (1, 0), (2, 0), (0, 1)])
@pytest.mark.parametrize("scale", [1e-1, 1e-3, 1e-6])
@pytest.mark.parametrize("tau", [0.51, 0.8, 1.5])
def test_fp64_forms_match_the_oracle(lib, lat, trim, scale, tau):
    D, Q, c, w, _ = O.lattice_tables(LATS[lat])
    vel = (C2, C19, C27)[lat]
    perm = [int(np.flatnonzero((c[:, :D] == np.array(v)).all(axis=1))[0]) for v in vel]
    rng = np.random.default_rng(7)
    p = O.make_params(LATS[lat], O.SMRT if trim else O.BGK, (2, 2, 2 if D == 3 else 1), tau=(1.0, 1.0, tau, 1.0, 1.0))
    worst = 0.0
    for _ in range(20):
        f = w * (1.0 + scale * rng.normal(size=Q))
        g = np.zeros(3)
        g[:D] = 0.01 * scale * rng.normal(size=D)
        fo, _ = O.collide_node(p, f, g[:D])
        din, dout = np.ascontiguousarray(f[perm] - w[perm]), np.zeros(Q)
        assert lib.host_collide64(lat, trim, _dp(din), _dp(g), tau, _dp(dout)) == 0
        worst = max(worst, float(np.abs(dout - (fo - w)[perm]).max()))
    assert worst <= 1e-15 * scale + 2.0 ** -53 * 4.0 / 9.0, worst

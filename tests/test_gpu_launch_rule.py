"""Where a new handle takes several steps per launch: never where single steps
were measured faster (2-byte storage, no mask, walls, ragged width or force per
node, and more than about 1e6 nodes).  Either way the state is that of single
steps, bit for bit."""
import numpy as np
import pytest

import lbm_workloads as W

pytestmark = pytest.mark.gpu

SMRT, TRIM = (1.0, 1.0, 0.63, 0.87, 1.1), (1.0, 1.0, 0.63, 1.0, 1.0)


# storage, shape, periodic, collision, tau, force, masked -> steps per launch
RULE = [
    ("F16", (1000, 1000), (1, 1, 1), "SMRT", TRIM, "none", False, 2), ("F16", (1008, 1000), (1, 1, 1), "SMRT", TRIM, "none", False, 1),
    ("BF16", (1280, 1280), (1, 1, 1), "BGK", (1.0, 1.0, 0.7, 1.0, 1.0), "uniform", False, 2),
    ("BF16", (1440, 1440), (1, 1, 1), "BGK", (1.0, 1.0, 0.7, 1.0, 1.0), "uniform", False, 1),
    ("F16", (1792, 1792), (1, 1, 1), "SMRT", TRIM, "rows", False, 1), ("F16", (1840, 1840), (1, 1, 1), "SMRT", TRIM, "rows", False, 2),
    ("F16", (1920, 1920), (1, 1, 1), "MRT_RAW", SMRT, "rows", False, 2), ("F16", (2304, 2304), (1, 1, 1), "MRT_RAW", SMRT, "rows", False, 1),
    ("F16", (2304, 2304), (1, 1, 1), "SMRT", TRIM, "none", False, 2), ("BF16", (2304, 2304), (1, 1, 1), "SMRT", SMRT, "none", False, 1),
    ("F16", (1280, 1280), (1, 0, 1), "SMRT", TRIM, "none", False, 2), ("F16", (1280, 1280), (0, 1, 1), "SMRT", TRIM, "none", False, 2),
    ("F16", (1281, 1280), (1, 1, 1), "SMRT", TRIM, "none", False, 2), ("F16", (1284, 1280), (1, 1, 1), "SMRT", TRIM, "none", False, 2),
    ("F16", (1280, 1280), (1, 1, 1), "SMRT", TRIM, "field", False, 2), ("F16", (1280, 1280), (1, 1, 1), "SMRT", TRIM, "none", True, 2),
    ("F32", (1280, 1280), (1, 1, 1), "SMRT", TRIM, "none", False, 2), ("F16", (384, 384), (1, 1, 1), "SMRT", TRIM, "none", False, 4),
]


@pytest.mark.parametrize("storage,shape,periodic,coll,tau,force,masked,steps", RULE)
def test_steps_per_launch_of_a_new_handle(storage, shape, periodic, coll, tau, force, masked, steps):
    import paper_2212_07494_gb300 as P
    nx, ny = shape
    g = {"none": None, "uniform": np.array([2e-5, -1e-5]), "rows": np.stack([1e-5 * np.sin(np.arange(ny)), np.zeros(ny)], 1),
         "field": 1e-5 * W.SplitMix64(9).normal(2 * nx * ny).reshape(2, 1, ny, nx)}[force]
    solid = W.random_solid((nx, ny, 1), 3, frac=0.05) if masked else None
    rng = np.random.default_rng(7)
    rho0, u0 = 1.0 + 0.01 * rng.normal(size=(1, ny, nx)), 0.03 * rng.normal(size=(2, 1, ny, nx))
    out = []
    for single in (False, True):
        gl = P.Lattice("D2Q9", coll, (nx, ny, 1), tau, storage, periodic, g=g, force_kind=force, solid=solid, rho0=rho0,
                       u0=u0)
        if single:
            gl.set_launch(64, 1)
        else:
            assert gl.launch_steps() == steps
        gl.step(11)
        out.append(gl.state()[0])
        gl.close()
    assert np.array_equal(*out)

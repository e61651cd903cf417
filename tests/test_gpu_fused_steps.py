"""Several steps per launch (k_step_tile) against one step per launch, bit for
bit: a new D2Q9 handle advances 2 or 4 steps per launch with the steps
between kept in shared memory, set_launch makes it one.  Sizes at the edges of
the tiles (one node more and less than a tile, odd widths, the narrowest
domain), walls and periodic faces on either axis, obstacles across tile edges,
every force kind and schedule, and step counts that leave every remainder.
The tolerance is zero: both run the same operations on the same values."""
import numpy as np
import pytest

import lbm_workloads as W

pytestmark = pytest.mark.gpu

TAU = {"BGK": (1.0, 1.0, 0.71, 1.0, 1.0), "SMRT": (1.0, 1.3, 0.63, 0.87, 1.1), "TRIM": (1.0, 1.3, 0.63, 1.0, 1.0),
       "SMRT_FNEQ": (1.0, 1.3, 0.63, 0.87, 1.1), "MRT_RAW": (1.0, 1.3, 0.63, 0.87, 1.1)}


def _pair(shape, periodic, storage, coll="TRIM", force="uniform", solid=None, seed=5):
    import paper_2212_07494_gb300 as P
    nx, ny = shape
    g = {"none": None, "uniform": np.array([2e-5, -1e-5]),
         "rows": np.stack([1e-5 * np.sin(np.arange(ny)), 1e-6 * np.cos(np.arange(ny))], 1),
         "field": 1e-5 * W.SplitMix64(9).normal(2 * nx * ny).reshape(2, 1, ny, nx)}[force]
    rho0, u0 = W.random_near_equilibrium("D2Q9", (nx, ny, 1), seed=seed, du=0.03)
    out = []
    for single in (False, True):
        gl = P.Lattice("D2Q9", "SMRT" if coll == "TRIM" else coll, (nx, ny, 1), TAU[coll], storage, periodic, g=g,
                       force_kind=force, solid=solid, rho0=rho0, u0=u0)
        if single:
            gl.set_launch(64, 1)
        out.append(gl)
    assert out[0].launch_steps() > 1 and out[1].launch_steps() == 1
    return out


def _same(a, b, n):
    a.step(n)
    b.step(n)
    sa, ta = a.state()
    sb, tb = b.state()
    assert ta == tb
    assert np.array_equal(sa, sb), n
    assert np.array_equal(a.moments()[1], b.moments()[1])


# 16 x 16 (four steps) and 32 x 8, 30 x 14 (two steps) tiles; 401 x 380 nodes take two steps per launch
SHAPES = [((5, 5), (1, 1, 1)), ((16, 16), (1, 1, 1)), ((17, 33), (1, 0, 1)), ((31, 15), (0, 1, 1)), ((64, 9), (0, 0, 1)),
          ((150, 37), (1, 0, 1)), ((401, 380), (1, 0, 1)), ((510, 300), (1, 1, 1))]


@pytest.mark.parametrize("storage", ["F32", "F16", "BF16"])
@pytest.mark.parametrize("shape,periodic", SHAPES)
@pytest.mark.parametrize("masked", [False, True])
def test_fused_steps_match_single_steps(storage, shape, periodic, masked):
    solid = W.random_solid(shape + (1,), 3, frac=0.1) if masked else None
    a, b = _pair(shape, periodic, storage, solid=solid)
    for n in (2, 3, 5, 71):
        _same(a, b, n)
    a.close()
    b.close()


@pytest.mark.parametrize("coll", ["BGK", "SMRT", "SMRT_FNEQ", "MRT_RAW"])
@pytest.mark.parametrize("force", ["none", "rows", "field"])
@pytest.mark.parametrize("shape", [(45, 39), (403, 377)])
def test_fused_steps_every_collision_and_force(coll, force, shape):
    a, b = _pair(shape, (1, 0, 1), "F32", coll, force)
    _same(a, b, 70)
    a.close()
    b.close()


@pytest.mark.parametrize("kind", ["uniform", "scale_uniform", "scale_rows", "scale_field"])
@pytest.mark.parametrize("shape", [(45, 39), (403, 377)])
def test_fused_steps_under_a_force_schedule(kind, shape):
    """Periods below, at and above the 64 steps whose forces are laid out at once (a per-node force of the larger
    domain is too large for that: one step per launch)."""
    force = kind.split("_")[-1]
    for period in (3, 64, 100):
        a, b = _pair(shape, (1, 0, 1), "F32", "TRIM", force)
        t = np.arange(period)
        for gl in (a, b):
            if kind == "uniform":
                gl.set_force_schedule(np.stack([1e-5 * np.cos(t), 1e-6 * np.sin(t)], 1))
            else:
                gl.set_force_scale_schedule(np.cos(0.1 * t))
        for n in (1, 6, 130):
            _same(a, b, n)
        for gl in (a, b):
            gl.set_force_schedule(None) if kind == "uniform" else gl.set_force_scale_schedule(None)
        _same(a, b, 5)
        a.close()
        b.close()


def test_autotune_keeps_the_state_and_a_valid_choice():
    a, b = _pair((300, 200), (1, 0, 1), "F32")
    a.step(10)
    b.step(10)
    before = a.state()[0]
    bx, npt, ms = a.autotune(trials=3)
    assert np.array_equal(a.state()[0], before) and ms > 0 and a.launch_steps() in (1, 4)
    _same(a, b, 9)
    a.close()
    b.close()


@pytest.mark.parametrize("coll", ["SMRT", "BGK", "SMRT_FNEQ", "MRT_RAW"])
@pytest.mark.parametrize("K", [1, 2, 3, 7])
def test_batch_pairs_of_steps_match_single_lattices(coll, K):
    """Two steps at a time between the checks of a batched run: channels one node around the 32 x 16 tiles, too narrow
    for pairs, with obstacles, and (SMRT) with and without the trimmed collision, over check intervals that leave
    every remainder."""
    import paper_2212_07494_gb300 as P
    chans = []
    for k, (nx, ny) in enumerate([(32, 16), (33, 17), (31, 15), (3, 9), (2, 3), (97, 40), (64, 33)]):
        tau = (1.0, 1.0, 0.6 + 0.1 * k) + ((1.0, 1.0) if k % 2 else (0.9, 1.2))
        ch = {"shape": (nx, ny, 1), "tau": tau, "periodic": (1, 0, 1), "g": [1e-5, 2e-6 * k]}
        if k in (1, 5):
            ch["solid"] = W.random_solid((nx, ny, 1), 40 + k, frac=0.1)
        chans.append(ch)
    b = P.Batch(chans, coll, "F32")
    b.set_handoff(0)
    for total, n in ((11, 11), (19, 8)):
        b.run_to_steady(0.0, K, max_steps=n)
        for i, ch in enumerate(chans):
            assert b.info(i)[0] == total
            gl = P.Lattice("D2Q9", coll, ch["shape"], ch["tau"], "F32", ch["periodic"], g=ch["g"], solid=ch.get("solid"))
            gl.set_launch(64, 1)
            gl.step(total)
            assert np.array_equal(b.populations(i), gl.populations()), (i, total)
            gl.close()
    b.close()

"""lbm_autotune, its cache and several steps per launch: a stored choice comes
back whole (shape and steps), an entry without the steps is not reused on a
handle that takes several, and the state is the same bits throughout."""
import json

import numpy as np
import pytest

import lbm_workloads as W

pytestmark = pytest.mark.gpu


def _lat(shape, storage="F32"):
    import paper_2212_07494_gb300 as P
    rho0, u0 = W.random_near_equilibrium("D2Q9", shape + (1,), seed=5, du=0.03)
    return P.Lattice("D2Q9", "SMRT", shape + (1,), (1.0, 1.0, 0.63, 1.0, 1.0), storage, (1, 1, 1), g=[2e-5, -1e-5], rho0=rho0,
                     u0=u0)


def test_steps_can_be_set_and_refused():
    import paper_2212_07494_gb300 as P
    for shape, k in (((96, 40), 4), ((400, 380), 2)):
        a, b = _lat(shape), _lat(shape)
        assert a.launch_steps() == k
        a.set_launch(64, 1)
        assert a.launch_steps() == 1
        a.set_launch_steps(k)
        assert a.launch_steps() == k and a.launch() == (64, 1, 0)
        for bad in (0, -1, 3, 6 - k):
            with pytest.raises(P.LbmError):
                a.set_launch_steps(bad)
        assert a.launch_steps() == k
        b.set_launch_steps(1)
        assert b.launch_steps() == 1
        a.step(71)
        b.step(71)
        assert np.array_equal(a.state()[0], b.state()[0])
        a.close()
        b.close()
    narrow = _lat((4, 40))
    with pytest.raises(P.LbmError):
        narrow.set_launch_steps(4)
    narrow.close()


@pytest.mark.parametrize("steps", [1, 4])
@pytest.mark.parametrize("default_shape", [True, False])
def test_cached_choice_comes_back_whole(tmp_path, steps, default_shape):
    from paper_2212_07494_gb300 import autotune as A
    path = str(tmp_path / "launch.json")
    a = _lat((96, 40))
    shape = a.launch() if default_shape else (32, 2, 0)
    A.store(path, A.signature(a), shape, 0.001, steps)
    assert a.autotune(cache=path) == shape + (0.001,)
    assert a.launch() == shape and a.launch_steps() == steps
    a.close()


def test_entry_without_steps_is_measured_again(tmp_path):
    from paper_2212_07494_gb300 import autotune as A
    path = str(tmp_path / "launch.json")
    a, b = _lat((96, 40)), _lat((96, 40), "F64")
    for gl in (a, b):
        A.store(path, A.signature(gl), (32, 1, 0), 123.0)
    assert a.autotune(trials=3, cache=path)[2] != 123.0          # takes several steps: ambiguous, measured and stored
    assert json.load(open(path))[A.signature(a)]["steps"] == a.launch_steps()
    assert b.autotune(trials=3, cache=path) == (32, 1, 0, 123.0)  # FP64 takes one step either way
    assert b.launch() == (32, 1, 0)
    a.close()
    b.close()

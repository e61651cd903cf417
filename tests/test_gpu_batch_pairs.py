"""Check intervals from which a batched run takes its steps in pairs (9 and
more): the channels, runs and reference of test_gpu_fused_steps, bit for bit,
with an odd and an even number of steps between the checks and none inside a
run; and runs that follow one another in either kernel."""
import numpy as np
import pytest

import test_gpu_fused_steps as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coll", ["SMRT", "BGK", "SMRT_FNEQ", "MRT_RAW"])
@pytest.mark.parametrize("K", [8, 9, 10, 20])
def test_pairs(coll, K):
    T.test_batch_pairs_of_steps_match_single_lattices(coll, K)


def test_intervals_in_turn():
    """Pairs move a channel's state to the other arena once per two steps: runs with and without them continue each other."""
    import paper_2212_07494_gb300 as P
    chans = [{"shape": (40 + 3 * k, 23, 1), "tau": (1.0, 1.0, 0.7, 0.9, 1.1), "periodic": (1, 0, 1), "g": [1e-5, 0.0]} for k in range(5)]
    a, b = P.Batch(chans, "SMRT", "F32"), P.Batch(chans, "SMRT", "F32")
    for x in (a, b):
        x.set_handoff(0)
    for K, n in ((20, 11), (1, 3), (9, 16), (2, 5), (50, 20)):
        a.run_to_steady(0.0, K, max_steps=n)
        b.run_to_steady(0.0, 1, max_steps=n)
        for i in range(5):
            assert np.array_equal(a.populations(i), b.populations(i)), (K, i)
    a.close()
    b.close()

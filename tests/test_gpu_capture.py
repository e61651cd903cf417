"""A caller's own stream capture of a handle's calls, replayed between direct
steps: the buffers in the graph are those the state lies in after any even
number of steps, however many steps a launch takes.  Domains that take four
and two steps per launch, walls, a schedule, obstacles; bit for bit against a
handle that is only stepped directly and one that takes one step per launch."""
import numpy as np
import pytest

import lbm_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["F32", "BF16"])
@pytest.mark.parametrize("shape", [(150, 37), (401, 380)])
@pytest.mark.parametrize("what", ["plain", "schedule", "solid"])
def test_replays_between_direct_steps(storage, shape, what):
    import torch
    import paper_2212_07494_gb300 as P
    nx, ny = shape
    stream = torch.cuda.Stream()
    solid = W.random_solid(shape + (1,), 3, frac=0.05) if what == "solid" else None
    rho0, u0 = W.random_near_equilibrium("D2Q9", (nx, ny, 1), seed=5, du=0.03)

    def make(**kw):
        gl = P.Lattice("D2Q9", "SMRT", (nx, ny, 1), (1.0, 1.0, 0.63, 1.0, 1.0), storage, (1, 0, 1), g=[2e-5, -1e-5],
                       force_kind="uniform", solid=solid, rho0=rho0, u0=u0, **kw)
        if what == "schedule":
            t = np.arange(37)
            gl.set_force_schedule(np.stack([1e-5 * np.cos(t), 1e-6 * np.sin(t)], 1))
        return gl

    a, b, c = make(torch_stream=stream), make(), make()
    c.set_launch(64, 1)
    assert a.launch_steps() > 1
    for o in (a, b, c):
        o.step(2)
    rho = torch.zeros(nx * ny, dtype=torch.float64, device="cuda")
    u = torch.zeros(2 * nx * ny, dtype=torch.float64, device="cuda")
    tot = torch.zeros(4, dtype=torch.float64, device="cuda")
    chk = torch.zeros(7, dtype=torch.float64, device="cuda")
    P.lbm_moments_device(a.h, rho.data_ptr(), u.data_ptr(), tot.data_ptr())
    a.check_device(chk.data_ptr())
    torch.cuda.synchronize()
    steps, moments, check = (torch.cuda.CUDAGraph() for _ in range(3))
    with torch.cuda.graph(steps, stream=stream):
        a.step(2)
    with torch.cuda.graph(moments, stream=stream):
        P.lbm_moments_device(a.h, rho.data_ptr(), u.data_ptr(), tot.data_ptr())
    with torch.cuda.graph(check, stream=stream):
        a.check_device(chk.data_ptr())
    for n in (100, 36, 2, 4, 6, 50, 130):
        a.step(n)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            steps.replay()
            moments.replay()
            check.replay()
        torch.cuda.synchronize()
        for o in (b, c):
            o.step(n + 2)
        sa, sb, sc = (o.state()[0] for o in (a, b, c))
        assert np.array_equal(sb, sc), n
        assert np.array_equal(sa, sb), n
        r, v, _ = b.moments()
        assert np.array_equal(rho.cpu().numpy(), np.asarray(r).ravel()), n
        assert np.array_equal(u.cpu().numpy(), np.asarray(v).ravel()), n
        assert chk[0].item() == tot[0].item() and chk[6].item() == 0.0
    for o in (a, b, c):
        o.close()


@pytest.mark.parametrize("shape", [(150, 37), (401, 380)])
def test_raw_state_of_solid_nodes(shape):
    """Steps never write solid nodes, so a buffer keeps there what an import or a restored checkpoint left in it: the raw
    state is the same bits with several steps per launch and with one only if both end in the same buffer."""
    import paper_2212_07494_gb300 as P
    solid = W.random_solid(shape + (1,), 3, frac=0.1)
    a, b = (P.Lattice("D2Q9", "SMRT", shape + (1,), (1.0, 1.0, 0.63, 1.0, 1.0), "F32", (1, 0, 1), g=[2e-5, 0.0], solid=solid)
            for _ in range(2))
    b.set_launch(64, 1)
    rng = np.random.default_rng(3)
    f = b.populations()
    f = f * (1.0 + 0.01 * rng.normal(size=f.shape))
    saved = None
    for n in (1, 2, 4, 3, 2, 66, 6, 5):
        for o in (a, b):
            if n == 4:
                o.set_populations(f)
            if n == 66:
                o.set_state(*saved)
            o.step(n)
        assert np.array_equal(a.state()[0], b.state()[0]), n
        if n == 3:
            saved = b.state()
    a.close()
    b.close()

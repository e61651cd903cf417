"""The work that users of this framework have it do, as measurable cases.

A case is one pass of a user's loop through the public entry points:

* ``lattice``: advance a flow (``Lattice.residual`` in the loops that watch the
  steady-state residual, ``Lattice.step`` in those that do not) and read its
  macroscopic fields into device tensors (``lbm_moments_device``);
* ``batch``: run a set of independent channels towards steady state in one
  launch (``Batch.run_to_steady``) and read every channel's fields;
* ``train``: a short epoch of the surrogate network (``UNet.train_step`` per
  minibatch) and its weights (``UNet.params``);
* ``predict``: the surrogate's prediction for one batch of channels
  (``UNet.forward``).

``exact`` computes the same outputs in 64 bits in plain torch, without this
repository's code: the lattice method from its statement (pull through index
tables, Hermite moments per axis, relaxation, reconstruction), the network as
a chain of float64 convolutions.  Storage rounding is left out of it.
"""
import functools
import math

import numpy as np
import torch

# ------------------------------------------------------------------- lattices
# population order of include/lbm.h
C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
C19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
       (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
       (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
C27 = C19 + [(1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1)]
VEL = {"D2Q9": C2, "D3Q19": C19, "D3Q27": C27}
BYTES = {"F64": 8, "F32": 4, "F16": 2, "BF16": 2}
# arithmetic operations of one collision (additions, multiplications and
# divisions as the method's transforms need them), per lattice
OPS = {"D2Q9": {"TRIM": 162, "SMRT": 210, "BGK": 304, "SMRT_FNEQ": 264, "MRT_RAW": 317},
       "D3Q19": {"TRIM": 444, "SMRT": 811, "BGK": 625, "SMRT_FNEQ": 1010, "MRT_RAW": 1047},
       "D3Q27": {"TRIM": 550, "SMRT": 873, "BGK": 889, "SMRT_FNEQ": 1072, "MRT_RAW": 1287}}


def _weights(lattice):
    if lattice == "D3Q19":
        return [(1 / 3, 1 / 18, 1 / 36)[sum(map(abs, c))] for c in C19]
    return [math.prod(2 / 3 if a == 0 else 1 / 6 for a in c) for c in VEL[lattice]]


# ---------------------------------------------------------------------- cases
# (cin, cout, ReLU, resolution divisor) of the network's 18 convolutions
NET = [(8, 32, 1, 1), (32, 32, 1, 1), (32, 64, 1, 2), (64, 64, 1, 2), (64, 128, 1, 4), (128, 128, 1, 4),
       (128, 256, 1, 8), (256, 256, 1, 8), (256, 128, 1, 4), (256, 128, 1, 4), (128, 128, 1, 4), (128, 64, 1, 2),
       (128, 64, 1, 2), (64, 64, 1, 2), (64, 32, 1, 1), (64, 32, 1, 1), (32, 32, 1, 1), (32, 3, 0, 1)]


def _lattice(name, lattice, collision, storage, nx, ny, nz, flow, steps, check, tau2, tau34=1.0, obstacles=0):
    return ({"name": name} if name else {}) | {"kind": "lattice", "lattice": lattice, "collision": collision, "storage": storage,
                                               "nx": nx, "ny": ny, "nz": nz, "flow": flow, "steps": steps, "check": check,
                                               "tau2": tau2, "tau34": tau34, "obstacles": obstacles}


def listed():
    return [
        # the analytic validation channel, the smallest domain a user runs, in the format that matches an FP64 reference
        _lattice("poiseuille_d2q9_bgk_f64_64x32", "D2Q9", "BGK", "F64", 64, 32, 1, "channel", 1000, False, 0.8),
        # the oscillating channel: a small domain whose force changes every step from a device-side schedule
        _lattice("womersley_d2q9_smrt_f64_50x200", "D2Q9", "SMRT", "F64", 50, 200, 1, "womersley", 600, False, 0.8),
        # one channel with cylinders relaxed to steady state, the residual watched (a surrogate's cold-start fallback)
        _lattice("obstacles_d2q9_smrt_f32_256x128", "D2Q9", "SMRT", "F32", 256, 128, 1, "channel", 1000, True, 0.7,
                 obstacles=4),
        # a medium channel of ragged width with general relaxation times and walls
        _lattice("channel_d2q9_smrt_f32_1001x517", "D2Q9", "SMRT", "F32", 1001, 517, 1, "channel", 200, False, 0.8,
                 tau34=1.1),
        # the double-precision run a reduced storage format is judged by
        _lattice("kolmogorov_d2q9_smrt_f64_512", "D2Q9", "SMRT", "F64", 512, 512, 1, "kolmogorov", 100, True, 0.6),
        # the headline flow: large periodic, FP32, residual and totals every 100 steps
        _lattice("kolmogorov_d2q9_smrt_f32_4096", "D2Q9", "SMRT", "F32", 4096, 4096, 1, "kolmogorov", 100, True, 0.6),
        # the same in 2-byte storage, which halves the traffic
        _lattice("kolmogorov_d2q9_smrt_f16_4096", "D2Q9", "SMRT", "F16", 4096, 4096, 1, "kolmogorov", 100, True, 0.6),
        # 3-D decaying turbulence on the full lattice
        _lattice("tgv_d3q27_smrt_f32_256", "D3Q27", "SMRT", "F32", 256, 256, 256, "tgv", 20, False, 0.50382),
        # a 3-D duct past obstacles on the small lattice, 2-byte storage
        _lattice("duct_d3q19_smrt_bf16_320x128x96", "D3Q19", "SMRT", "BF16", 320, 128, 96, "channel", 50, False, 0.7,
                 obstacles=12),
        # a parameter study: channels of uneven size and parameters towards steady state in one launch
        {"name": "batch_d2q9_smrt_f32_128", "kind": "batch", "channels": 128, "collision": "SMRT", "storage": "F32",
         "steps": 1000, "check_every": 500, "obstacles": 0},
        # training the surrogate that warm-starts such channels: four minibatches, then its weights
        {"name": "train_unet_128x256_b8", "kind": "train", "H": 128, "W": 256, "batch": 8, "minibatches": 4},
        # the surrogate's prediction for a batch of channels
        {"name": "predict_unet_128x256_b8", "kind": "predict", "H": 128, "W": 256, "batch": 8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice2", "lattice2", "lattice2", "lattice3", "lattice3", "batch", "train", "predict"])
    if kind in ("train", "predict"):
        # channel grids are multiples of 8; heights that divide or are divided by 128 are the usual ones
        H = rng.choice([32, 64, 64, 128, 128, 8 * rng.randint(4, 16)])
        c = {"kind": kind, "H": H, "W": 8 * _log_int(rng, 4, 32), "batch": rng.choice([1, 2, 4, 8, 8, rng.randint(1, 8)])}
        if kind == "train":
            c["minibatches"] = rng.randint(1, 4)
        return c
    if kind == "batch":
        steps = rng.randint(200, 500)
        return {"kind": "batch", "channels": _log_int(rng, 4, 128), "collision": rng.choice(["SMRT", "SMRT", "BGK", "SMRT_FNEQ"]),
                "storage": rng.choice(["F32", "F32", "F32", "F64"]), "steps": steps, "check_every": steps // 2 + 1,
                "obstacles": rng.choice([0, 0, 2])}
    collision = rng.choice(["SMRT", "SMRT", "SMRT", "BGK", "SMRT_FNEQ", "MRT_RAW"])
    storage = rng.choice(["F32", "F32", "F32", "F16", "BF16", "F64"])
    tau34 = rng.choice([1.0, 1.0, 1.0, round(rng.uniform(0.8, 1.3), 3)])
    if kind == "lattice2":
        nx, ny = _log_int(rng, 32, 4096), _log_int(rng, 16, 4096)
        if rng.random() < 0.5:
            nx = max(32, nx // 32 * 32)
        flow = rng.choice(["channel", "channel", "kolmogorov", "kolmogorov", "womersley", "field"])
        steps = max(20, min(1000, int(2e8 / (nx * ny)) if storage != "F64" else int(3e7 / (nx * ny))))
        obstacles = rng.choice([0, 0, 0, 4]) if flow == "channel" and min(nx, ny) >= 48 else 0
        return _lattice("", "D2Q9", collision, storage, nx, ny, 1, flow, steps, rng.random() < 0.4,
                        round(rng.uniform(0.55, 1.2), 3), tau34, obstacles)
    lattice = rng.choice(["D3Q19", "D3Q27"])
    n = _log_int(rng, 24, 224)
    nx, ny, nz = (max(8, int(n * rng.uniform(0.7, 1.4))) for _ in range(3))
    if rng.random() < 0.5:
        nx = max(8, nx // 8 * 8)
    flow = rng.choice(["tgv", "channel"])
    steps = max(5, min(200, int(6e7 / (nx * ny * nz)) if storage != "F64" else int(5e6 / (nx * ny * nz))))
    obstacles = rng.choice([0, 0, 6]) if flow == "channel" and min(nx, ny, nz) >= 32 else 0
    return _lattice("", lattice, collision, storage, nx, ny, nz, flow, steps, rng.random() < 0.4,
                    round(rng.uniform(0.55, 1.0), 3), tau34, obstacles)


# --------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _stream():
    """The one solver stream of the program."""
    return torch.cuda.Stream()


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _discs(rng, nx, ny, count, nz=0):
    """Solid cylinders (spheres in 3-D), a few cells clear of the walls; periodic in x."""
    r_hi = max(3.0, min(20.0, 0.15 * (min(ny, nz) if nz else ny)))
    x = np.arange(nx)
    solid = np.zeros((max(nz, 1), ny, nx), bool)
    for _ in range(count):
        r = rng.uniform(0.4 * r_hi, r_hi)
        dx = np.abs(x - rng.uniform(0, nx))
        d2 = (np.minimum(dx, nx - dx) ** 2)[None, None, :] + ((np.arange(ny) - rng.uniform(r + 2, ny - r - 3)) ** 2)[None, :, None]
        if nz:
            d2 = d2 + ((np.arange(nz) - rng.uniform(r + 2, nz - r - 3)) ** 2)[:, None, None]
        solid |= d2 <= r * r
    return solid.astype(np.uint8)


def _problem(c, seed):
    """The flow of a lattice case: periodic flags, force, mask and initial fields (host arrays, as lbm_create takes them)."""
    D = 2 if c["lattice"] == "D2Q9" else 3
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    shape = (nz, ny, nx)
    nu = (c["tau2"] - 0.5) / 3.0
    rng = np.random.default_rng(seed)
    noise = torch.randn((D,) + shape, generator=_gen(seed), device="cuda", dtype=torch.float64)
    p = {"D": D, "tau": (1.0, 1.0, c["tau2"], c["tau34"], c["tau34"]), "periodic": (1, 1, 1), "solid": None,
         "rho0": None, "schedule": None}
    if c["flow"] == "kolmogorov":
        # sinusoidal row force; the amplitude keeps the laminar speed below 0.05 on small domains
        k = 2.0 * math.pi / ny
        amp = min(1e-5, 0.05 * nu * k * k) * rng.uniform(0.8, 1.0)
        y = np.sin(k * np.arange(ny))
        p["force_kind"], p["g"] = "rows", np.stack([amp * y, np.zeros(ny)], 1)
        u0 = 1e-4 * noise
        u0[0] += torch.as_tensor(amp * y, device="cuda")[None, :, None]
    elif c["flow"] == "tgv":
        U0 = 0.05 * rng.uniform(0.8, 1.0)
        z, y, x = (2.0 * math.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n for n in shape)
        z, y, x = z[:, None, None], y[None, :, None], x[None, None, :]
        u0 = 1e-4 * noise
        u0[0] += U0 * torch.sin(x) * torch.cos(y) * torch.cos(z)
        u0[1] -= U0 * torch.cos(x) * torch.sin(y) * torch.cos(z)
        rho = 1.0 + 3.0 * (U0 * U0 / 16.0) * (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0)
        p["rho0"] = rho.cpu().numpy()
        p["force_kind"], p["g"] = "uniform", np.array([1e-6, 0.0, 0.0])
    elif c["flow"] == "field":
        # the forced Taylor-Green flow: a force of its own at every node
        U0 = 0.02 * rng.uniform(0.8, 1.0)
        kx, ky = 2.0 * math.pi / nx, 2.0 * math.pi / ny
        x, y = (torch.arange(n, device="cuda", dtype=torch.float64) for n in (nx, ny))
        x, y = x[None, None, :], y[None, :, None]
        one = torch.ones(shape, device="cuda", dtype=torch.float64)
        u0 = 1e-4 * noise
        u0[0] -= U0 * torch.cos(kx * x) * torch.sin(ky * y)
        u0[1] += U0 * torch.sin(kx * x) * torch.cos(ky * y)
        g = torch.stack([-0.5 * U0 * U0 * kx * torch.sin(2 * kx * x) * one, -0.5 * U0 * U0 * ky * torch.sin(2 * ky * y) * one])
        p["force_kind"], p["g"] = "field", g.cpu().numpy()
    else:
        # walls in y (and in z for a 3-D duct), driven along x to a laminar peak of at most 0.05
        p["periodic"] = (1, 0, 0 if D == 3 else 1)
        H = min(ny, nz) if D == 3 else ny
        gx = min(1e-5, 0.05 * 8.0 * nu / (H * H)) * rng.uniform(0.5, 1.0)
        p["force_kind"], p["g"] = "uniform", np.array([gx] + [0.0] * (D - 1))
        if c["obstacles"]:
            p["solid"] = _discs(rng, nx, ny, c["obstacles"], nz if D == 3 else 0)
        u0 = 1e-4 * noise
        if c["flow"] == "womersley":
            # oscillating pressure gradient, period 1200 steps, tabulated per step
            A = min(1e-4, 0.05 * 2.0 * math.pi / 1200)
            t = np.arange(1200)
            p["schedule"] = np.stack([-A * np.cos(2.0 * math.pi * t / 1200), np.zeros(1200)], 1)
            p["g"] = p["schedule"][0].copy()
    p["u0"] = u0.cpu().numpy()
    return p


def _channels(c, seed):
    """Channels of uneven size and parameters: periodic in x, walls in y."""
    rng = np.random.default_rng(seed)
    out = []
    # the sizes belong to the case, the parameters and masks to the seed: a pass costs the same for every seed
    sizes = np.random.default_rng(c["channels"])
    for _ in range(c["channels"]):
        nx, ny = int(sizes.integers(32, 513)), int(sizes.integers(16, 257))
        tau2 = rng.uniform(0.55, 1.5)
        gx = min(math.exp(rng.uniform(math.log(1e-7), math.log(1e-5))), 0.1 * 8.0 * (tau2 - 0.5) / 3.0 / (ny * ny))
        ch = {"shape": (nx, ny, 1), "tau": (1.0, 1.0, tau2, 1.0, 1.0), "periodic": (1, 0, 1), "g": [gx, 0.0]}
        if c["obstacles"] and ny >= 48:
            ch["solid"] = _discs(rng, nx, ny, c["obstacles"])
        out.append(ch)
    return out


def _net_params(seed):
    """He-normal weights, zero biases, in the canonical layout."""
    rng = np.random.default_rng(seed)
    out = []
    for cin, cout, relu, _ in NET:
        out.append(rng.normal(size=9 * cin * cout) * math.sqrt((2.0 if relu else 1.0) / (9 * cin)))
        out.append(np.zeros(cout))
    return np.concatenate(out).astype(np.float32)


def _net_data(c, seed):
    """Inputs, targets and fluid masks of the surrogate's training set: smooth per-node features of order one."""
    H, W = c["H"], c["W"]
    n = c["batch"] * c.get("minibatches", 1)
    g = _gen(seed)
    rand = lambda *s: torch.randn(s, generator=g, device="cuda", dtype=torch.float32)  # noqa: E731
    coarse = rand(n, 11, H // 8, W // 8)
    smooth = torch.nn.functional.interpolate(coarse, size=(H, W), mode="bilinear")
    X = (smooth[:, :8].permute(0, 2, 3, 1) + 0.1 * rand(n, H, W, 8)).contiguous()
    M = (X[..., 0] < 1.0).to(torch.float32).contiguous()
    X[..., 0] = 1.0 - M
    Y = (0.3 * smooth[:, 8:].permute(0, 2, 3, 1) * M[..., None]).contiguous()
    return X, Y, M


class _State:
    pass


def prepare(case, seed):
    import paper_2212_07494_gb300 as P
    s = _State()
    s.P, s.case = P, case
    if case["kind"] == "lattice":
        p = _problem(case, seed)
        shape = (case["nx"], case["ny"], case["nz"])
        s.solver = P.Lattice(case["lattice"], case["collision"], shape, p["tau"], case["storage"], p["periodic"], p["g"],
                             p["force_kind"], p["solid"], p["rho0"], p["u0"], torch_stream=_stream())
        if p["schedule"] is not None:
            s.solver.set_force_schedule(p["schedule"])
        s.rho = torch.empty(shape[::-1], dtype=torch.float64, device="cuda")
        s.u = torch.empty((p["D"],) + shape[::-1], dtype=torch.float64, device="cuda")
    elif case["kind"] == "batch":
        s.solver = P.Batch(_channels(case, seed), case["collision"], case["storage"], _stream().cuda_stream)
    else:
        s.X, s.Y, s.M = _net_data(case, seed)
        s.net = P.UNet(case["H"], case["W"], case["batch"], _stream().cuda_stream, cin=8, periodic_x=True)
        s.net.set_params(_net_params(seed))
        if case["kind"] == "train":
            b = case["batch"]
            s.scale = [1.0 / (3.0 * float(s.M[i * b:(i + 1) * b].sum())) for i in range(case["minibatches"])]
            s.loss = torch.zeros(case["minibatches"], dtype=torch.float64, device="cuda")
        else:
            s.y = torch.empty((case["batch"], case["H"], case["W"], 3), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    return s


def run(s):
    c = s.case
    if c["kind"] == "lattice":
        out = {"rho": s.rho, "u": s.u}
        if c["check"]:
            out["residual"] = s.solver.residual(c["steps"])
        else:
            s.solver.step(c["steps"])
        s.P.lbm_moments_device(s.solver.h, s.rho.data_ptr(), s.u.data_ptr(), None)
        return out
    if c["kind"] == "batch":
        _, steps, status, r = s.solver.run_to_steady(1e-9, c["check_every"], c["steps"])
        fields = [s.solver.moments(i) for i in range(s.solver.n)]
        return {"steps": steps, "status": status, "residual": r, "rho": np.concatenate([f[0].ravel() for f in fields]),
                "u": np.concatenate([f[1].ravel() for f in fields])}
    if c["kind"] == "train":
        b = c["batch"]
        for i in range(c["minibatches"]):
            x, y, m = (t[i * b:(i + 1) * b] for t in (s.X, s.Y, s.M))
            s.net.train_step(x.data_ptr(), y.data_ptr(), m.data_ptr(), b, s.scale[i], 1e-3, s.loss[i:].data_ptr())
        return {"loss": s.loss, "params": s.net.params()}
    s.net.forward(s.X.data_ptr(), s.y.data_ptr(), c["batch"])
    return {"y": s.y}


def work(case):
    """Bytes: the state (or the inputs and weights) read once and written once,
    and the outputs written once.  Flops: every node's collision at every
    step, every multiply-add of the convolutions."""
    if case["kind"] == "lattice":
        n = case["nx"] * case["ny"] * case["nz"]
        D, Q = (2, 9) if case["lattice"] == "D2Q9" else (3, len(VEL[case["lattice"]]))
        trim = case["collision"] == "SMRT" and case["tau34"] == 1.0
        ops = OPS[case["lattice"]]["TRIM" if trim else case["collision"]]
        force = n * D * BYTES["F64" if case["storage"] == "F64" else "F32"] if case["flow"] == "field" else 0
        return {"bytes": n * (2 * Q * BYTES[case["storage"]] + 8 * (1 + D) + (1 if case["obstacles"] else 0)) + force,
                "flops": float(n) * case["steps"] * ops}
    if case["kind"] == "batch":
        n = sum(ch["shape"][0] * ch["shape"][1] for ch in _channels(case | {"obstacles": 0}, 0))
        ops = OPS["D2Q9"]["TRIM" if case["collision"] == "SMRT" else case["collision"]]
        return {"bytes": n * (2 * 9 * BYTES[case["storage"]] + 24), "flops": float(n) * case["steps"] * ops}
    H, W, b = case["H"], case["W"], case["batch"]
    weights = sum(9 * ci * co + co for ci, co, _, _ in NET)
    fwd = sum(2.0 * (H // d) * (W // d) * 9 * ci * co for ci, co, _, d in NET)
    if case["kind"] == "predict":
        return {"bytes": b * H * W * 11 * 4 + weights * 4, "flops": b * fwd}
    # forward, input gradients (all layers but the first) and weight gradients
    k = case["minibatches"]
    return {"bytes": k * (b * H * W * 12 * 4 + weights * 4 * 6), "flops": k * b * (3.0 * fwd - 2.0 * H * W * 9 * 8 * 32)}


# ---------------------------------------------------------------- exact values
class _Exact:
    """The method in 64 bits on a flat list of nodes; state (Q, N): deviations
    of the post-collision populations, pulled through an index table."""

    def __init__(self, lattice, collision, index, tau, rho0, u0, g):
        # index (Q, N): flat entry of the (Q, N) state that population i of a node pulls; tau: 3 values or (N,) tensors
        # (orders 2, 3, 4); rho0 (N,), u0 (D, N), g (D, N) or (D, 1)
        self.lat, self.coll, self.index = lattice, collision, index
        self.c = VEL[lattice]
        self.D, self.Q = len(self.c[0]), len(self.c)
        self.om = [1.0 / t for t in tau]
        self.pos = [sum((c[a] + 1) * 3 ** a for a in range(self.D)) for c in self.c]
        self.order = [sum((m // 3 ** a) % 3 for a in range(self.D)) for m in range(3 ** self.D)]
        self.g = g
        target = self._initial(rho0 - 1.0, u0)
        # the state whose pull gives `target`: entry index[i, n] holds target[i, n]
        self.f = torch.zeros_like(target)
        self.f.view(-1)[index.view(-1)] = target.view(-1)

    def _axis(self, G, a):
        s = 3 ** a
        v = G.view(3 ** (self.D - 1 - a), 3, s, -1)
        return v[:, 0], v[:, 1], v[:, 2]

    def _project(self, G):
        for a in range(self.D):
            m, z, p = self._axis(G, a)
            s, d = p + m, p - m
            m.copy_(s + z)
            p.copy_((2.0 * s - z) / 3.0)
            z.copy_(d)

    def _shift(self, G, u):
        for a in range(self.D):
            a0, a1, a2 = self._axis(G, a)
            a2 += u[a] * (2.0 * a1 + u[a] * a0)
            a1 += u[a] * a0

    def _retained(self, m):
        d = [(m // 3 ** a) % 3 for a in range(self.D)]
        if self.lat == "D3Q19":
            return sum(d) <= 2 or (sum(d) == 3 and max(d) == 2)
        return self.D == 2 or sum(d) <= 4

    def _reconstruct(self, G):
        w = (1 / 6, 2 / 3, 1 / 6) if self.lat != "D3Q19" else (1.0, 1.0, 1.0)
        for a in range(self.D):
            t0, t1, t2 = self._axis(G, a)
            lo, mid, hi = t0 - 3.0 * t1 + 3.0 * t2, t0 - 1.5 * t2, t0 + 3.0 * t1 + 3.0 * t2
            t0.copy_(w[0] * lo)
            t1.copy_(w[1] * mid)
            t2.copy_(w[2] * hi)
        out = torch.stack([G[p] for p in self.pos])
        if self.lat == "D3Q19":
            out *= torch.tensor(_weights(self.lat), dtype=out.dtype, device=out.device)[:, None]
        return out

    def _grid(self, f):
        G = torch.zeros((3 ** self.D, f.shape[1]), dtype=f.dtype, device=f.device)
        G[self.pos] = f
        return G

    def _back(self, G, drho):
        for m in range(3 ** self.D):
            if not self._retained(m):
                G[m] = 0.0
        G[0] = drho
        return self._reconstruct(G)

    def _guo(self, drho, u, om):
        """Second-order equilibrium deviation and force term of every population."""
        rho = 1.0 + drho
        uu, gu = sum(v * v for v in u), sum(a * b for a, b in zip(self.g, u))
        for c, w in zip(self.c, _weights(self.lat)):
            cu, cg = sum(k * v for k, v in zip(c, u)), sum(k * v for k, v in zip(c, self.g))
            yield w * (drho + rho * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu)), w * rho * (3.0 * (cg - gu) + 9.0 * cu * cg)

    def _initial(self, drho, u):
        if self.coll == "BGK":
            return torch.stack([e - 0.5 * F for e, F in self._guo(drho, u, None)])
        G = torch.zeros((3 ** self.D, drho.shape[0]), dtype=drho.dtype, device=drho.device)
        G[0] = 1.0 + drho
        for a in range(self.D):
            G[3 ** a] = -0.5 * (1.0 + drho) * self.g[a]
        self._shift(G, u)
        return self._back(G, drho)

    def pull(self):
        return self.f.view(-1)[self.index.view(-1)].view(self.Q, -1)

    def macro(self, f):
        c = torch.tensor(self.c, dtype=f.dtype, device=f.device).T
        drho = f.sum(0)
        return drho, c @ f / (1.0 + drho) + 0.5 * self.g

    def _order2(self, G, om):
        for m, n in enumerate(self.order):
            if n == 2:
                G[m] *= 1.0 - om

    def step(self):
        f = self.pull()
        om2, om3, om4 = self.om
        if self.coll == "BGK":
            drho, u = self.macro(f)
            for i, (e, F) in enumerate(self._guo(drho, u, om2)):
                f[i] += om2 * (e - f[i]) + (1.0 - 0.5 * om2) * F
            self.f = f
            return
        G = self._grid(f)
        self._project(G)
        drho = G[0].clone()
        rho = 1.0 + drho
        u = torch.stack([G[3 ** a] / rho + 0.5 * self.g[a] for a in range(self.D)])
        G[0] = rho
        self._shift(G, -u)
        M = range(3 ** self.D)
        dig = [[(m // 3 ** a) % 3 for a in range(self.D)] for m in M]
        if self.coll == "MRT_RAW":
            G[0] = 0.0
            for a in range(self.D):
                G[3 ** a] = -0.5 * rho * self.g[a]
            for m in M:
                if self.order[m] >= 4:
                    G[m] = 0.0
            self._shift(G, u)
            for m in M:
                n = self.order[m]
                if n == 0 or n > 4:
                    G[m] = 0.0
                    continue
                eq = rho * math.prod(u[a] ** dig[m][a] for a in range(self.D))
                F = sum(dig[m][a] * rho * self.g[a] * math.prod(u[b] ** (dig[m][b] - (a == b)) for b in range(self.D))
                        for a in range(self.D) if dig[m][a])
                om = (None, 1.0, om2, om3, om4)[n]
                G[m] = eq + 0.5 * F if n == 1 else eq + (1.0 - om) * G[m] + (1.0 - 0.5 * om) * F
            self.f = self._back(G, drho)
            return
        F3, d3 = {}, {}
        if self.coll == "SMRT_FNEQ":
            for m in M:
                if self.order[m] == 3:
                    F3[m] = sum(dig[m][a] * self.g[a] * (1.0 - 0.5 * om2) * G[m - 3 ** a] for a in range(self.D) if dig[m][a])
                    d3[m] = (1.0 - 0.5 * om3) * (G[m] + 0.5 * F3[m])
        for m in M:
            n = self.order[m]
            if n == 2:
                G[m] *= 1.0 - om2
            elif n == 3:
                G[m] = (1.0 - om3) * G[m] + ((1.0 - 0.5 * om3) * F3[m] if F3 else 0.0)
            elif n == 4:
                F4 = sum(dig[m][a] * self.g[a] * d3[m - 3 ** a] for a in range(self.D) if dig[m][a]) if d3 else 0.0
                G[m] = (1.0 - om4) * G[m] + (1.0 - 0.5 * om4) * F4
            elif n > 4:
                G[m] = 0.0
        G[0] = rho
        for a in range(self.D):
            G[3 ** a] = 0.5 * rho * self.g[a]
        self._shift(G, u)
        self.f = self._back(G, drho)


def _pull_index(lattice, shape, periodic, solid, base=0, total=None):
    """(Q, N) flat entries pulled by the nodes of one domain (z, y, x), its first node `base` of `total`: the neighbour at
    x - c, or the node's own opposite population across a wall or a solid node."""
    c = VEL[lattice]
    D = len(c[0])
    nz, ny, nx = shape
    N = nx * ny * nz
    total = N if total is None else total
    z, y, x = torch.meshgrid(*(torch.arange(n, device="cuda") for n in shape), indexing="ij")
    own = ((z * ny + y) * nx + x).reshape(-1)
    mask = None if solid is None else torch.as_tensor(solid, device="cuda").reshape(-1).bool()
    opp = [c.index(tuple(-k for k in v)) for v in c]
    out = torch.empty((len(c), N), dtype=torch.int64, device="cuda")
    for i, v in enumerate(c):
        at, wall = [], torch.zeros(N, dtype=torch.bool, device="cuda")
        for a, (q, n) in enumerate(((x, nx), (y, ny), (z, nz))):
            t = q.reshape(-1) - (v[a] if a < D else 0)
            if not periodic[a]:
                wall |= (t < 0) | (t >= n)
            at.append(t % n)
        src = (at[2] * ny + at[1]) * nx + at[0]
        if mask is not None:
            # links into solid nodes bounce back; the solid nodes themselves keep their own entries
            wall = wall | mask[src]
            out[i] = torch.where(mask, i * total + base + own, torch.where(wall, opp[i] * total + base + own, i * total + base + src))
        else:
            out[i] = torch.where(wall, opp[i] * total + base + own, i * total + base + src)
    return out


def _residual(u, before, K):
    return float(torch.sqrt(((u - before) ** 2).sum()) / (K * torch.sqrt((u ** 2).sum())))


def exact(case, seed):
    if case["kind"] == "lattice":
        p = _problem(case, seed)
        shape = (case["nz"], case["ny"], case["nx"])
        N = math.prod(shape)
        if N * case["steps"] * len(VEL[case["lattice"]]) > 4e10:
            return None
        dev = functools.partial(torch.as_tensor, dtype=torch.float64, device="cuda")
        g = dev(p["g"])
        if p["force_kind"] == "rows":
            g = g.T[:, None, :, None].expand((p["D"],) + shape)
        g = g.reshape(p["D"], -1)
        rho0 = torch.ones(N, dtype=torch.float64, device="cuda") if p["rho0"] is None else dev(p["rho0"]).reshape(-1)
        e = _Exact(case["lattice"], case["collision"], _pull_index(case["lattice"], shape, p["periodic"], p["solid"]),
                   p["tau"][2:], rho0, dev(p["u0"]).reshape(p["D"], -1), g)
        fluid = torch.ones(N, dtype=torch.bool, device="cuda") if p["solid"] is None else dev(p["solid"]).reshape(-1) == 0
        table = None if p["schedule"] is None else dev(p["schedule"])
        before = e.macro(e.pull())[1] * fluid
        for t in range(case["steps"]):
            if table is not None:
                e.g = table[t % len(table)][:, None]
            e.step()
        if table is not None:
            e.g = table[case["steps"] % len(table)][:, None]
        drho, u = e.macro(e.pull())
        u = u * fluid
        out = {"rho": (1.0 + drho * fluid).view(shape), "u": u.view((p["D"],) + shape)}
        if case["check"]:
            out["residual"] = _residual(u, before, case["steps"])
        return out
    if case["kind"] == "batch":
        chans = _channels(case, seed)
        n = [ch["shape"][0] * ch["shape"][1] for ch in chans]
        at = np.concatenate([[0], np.cumsum(n)])
        total = int(at[-1])
        index = torch.cat([_pull_index("D2Q9", ch["shape"][::-1], ch["periodic"], ch.get("solid"), int(b), total)
                           for ch, b in zip(chans, at)], 1)
        per_node = lambda v: torch.repeat_interleave(torch.tensor(v, dtype=torch.float64, device="cuda"), torch.tensor(n, device="cuda"))  # noqa: E731
        one = torch.ones(total, dtype=torch.float64, device="cuda")
        g = torch.stack([per_node([ch["g"][0] for ch in chans]), 0.0 * one])
        fluid = torch.cat([torch.ones(k, device="cuda") if ch.get("solid") is None else 1.0 - torch.as_tensor(ch["solid"], device="cuda").reshape(-1).float()
                           for ch, k in zip(chans, n)]).double()
        e = _Exact("D2Q9", case["collision"], index, (per_node([ch["tau"][2] for ch in chans]), one, one), one,
                   torch.zeros((2, total), dtype=torch.float64, device="cuda"), g)
        u0 = e.macro(e.pull())[1] * fluid
        r = None
        for t in range(case["steps"]):
            # the residual over the last check interval, taken at the multiples of it that a step follows
            if t and t % case["check_every"] == 0:
                u = e.macro(e.pull())[1] * fluid
                r = np.array([_residual(u[:, a:b], u0[:, a:b], case["check_every"]) for a, b in zip(at[:-1], at[1:])])
                u0 = u
            e.step()
        drho, u = e.macro(e.pull())
        u = u * fluid
        return {"steps": None, "status": None, "residual": r, "rho": (1.0 + drho * fluid).cpu().numpy(),
                "u": torch.cat([u[:, a:b].reshape(-1) for a, b in zip(at[:-1], at[1:])]).cpu().numpy()}
    return _exact_net(case, seed)


def _unpack(p):
    """Canonical layout -> [(weight (co, ci, 3, 3), bias)]."""
    out, o = [], 0
    for ci, co, _, _ in NET:
        w = p[o:o + 9 * ci * co].view(co, 3, 3, ci).permute(0, 3, 1, 2)
        out.append((w, p[o + 9 * ci * co:o + 9 * ci * co + co]))
        o += 9 * ci * co + co
    return out


def _net_forward(p, x):
    """The surrogate on (n, c, H, W): convolutions periodic along x, zero-padded along y."""
    F = torch.nn.functional
    w = iter(_unpack(p))
    relu = iter(NET)

    def conv(v):
        k, b = next(w)
        v = F.pad(F.pad(v, (1, 1, 0, 0), mode="circular"), (0, 0, 1, 1))
        # one matrix product per tap
        H, W = v.shape[2] - 2, v.shape[3] - 2
        out = b[None, :, None, None]
        for dy in range(3):
            for dx in range(3):
                out = out + torch.einsum("oc,nchw->nohw", k[:, :, dy, dx], v[:, :, dy:dy + H, dx:dx + W])
        return out.relu() if next(relu)[2] else out

    pool = lambda v: F.avg_pool2d(v, 2)  # noqa: E731
    up = lambda v: v.repeat_interleave(2, 2).repeat_interleave(2, 3)  # noqa: E731
    e1 = conv(conv(x))
    e2 = conv(conv(pool(e1)))
    e3 = conv(conv(pool(e2)))
    v = conv(conv(pool(e3)))
    for skip in (e3, e2, e1):
        v = conv(conv(torch.cat([conv(up(v)), skip], 1)))
    return conv(v)


def _exact_net(case, seed):
    X, Y, M = _net_data(case, seed)
    X, Y, M = X.double().permute(0, 3, 1, 2), Y.double().permute(0, 3, 1, 2), M.double()
    p = torch.as_tensor(_net_params(seed), dtype=torch.float64, device="cuda")
    b = case["batch"]
    if case["kind"] == "predict":
        with torch.no_grad():
            return {"y": torch.cat([_net_forward(p, X[i:i + 1]) for i in range(b)]).permute(0, 2, 3, 1).contiguous()}
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    losses = []
    for k in range(case["minibatches"]):
        q = p.clone().requires_grad_(True)
        at = range(k * b, (k + 1) * b)
        scale = 1.0 / (3.0 * float(M[k * b:(k + 1) * b].sum()))
        loss, grad = 0.0, torch.zeros_like(p)
        for i in at:
            l = (M[i, None] * (_net_forward(q, X[i:i + 1])[0] - Y[i]) ** 2).sum() * scale
            grad += torch.autograd.grad(l, q)[0]
            loss += float(l.detach())
        losses.append(loss)
        m = 0.9 * m + 0.1 * grad
        v = 0.999 * v + 0.001 * grad * grad
        p = p - 1e-3 * (m / (1.0 - 0.9 ** (k + 1))) / (torch.sqrt(v / (1.0 - 0.999 ** (k + 1))) + 1e-8)
    return {"loss": torch.tensor(losses, dtype=torch.float64), "params": p.cpu().numpy()}

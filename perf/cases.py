"""Performance cases of the coupled lattice-Boltzmann phase-field library.

Each case is one call sequence of a user's program through the public entry
points: a simulation handle stepped and read out (2D and 3D, FP32 and 16-bit
storage, all boundary kinds, obstacles, both flow collisions), a batched sweep,
the U-Net surrogate's inference and gradient, and the block propagator.  The
sizes are those of the repository's workloads (128^2, 1024^2, 256^3, sweeps of
256..768 and 32..128, 512^2 networks) and grids of the paper's convergence
study (775 x 650 .. 2480 x 2080).

listed() gives the fixed cases, draw(rng) one more of the same ranges,
prepare(case, seed) the state a program holds before the call, run(state) one
pass with its outputs, work(case) the bytes and operations a pass cannot do
without, exact(case, seed) the outputs in 64 bits from plain torch and numpy.
"""
import math

import numpy as np
import torch

import paper_2206_02145_gb300 as lbpf

STORAGE = {"fp32": lbpf.FP32, "fp16": lbpf.FP16_SHIFTED, "bf16": lbpf.BF16_SHIFTED}
# boundaries: a periodic box with a flow through it; inflow at x = 0, outflow at
# x = nx - 1, the rest periodic; channel: periodic x, walls in y (and z), driven
# by a body force
BOUNDS = {"periodic": (0, 0, 0), "inflow": (1, 0, 0), "channel": (0, 2, 2)}
TAU_PHI, TAU_U, TAU_F, W0, DRAG = 0.8, 0.8, 0.6, 2.0, 2.757
U_CHANNEL = 0.01  # largest velocity of the channels' initial flow


def _grid(dim, nx, ny, nz, bounds, flow, storage, steps, fold=5, chm=False, baffle=False):
    return {"kind": "grid", "dim": dim, "nx": nx, "ny": ny, "nz": nz, "bounds": bounds,
            "flow": flow, "storage": storage, "steps": steps, "fold": fold, "chm": chm,
            "baffle": baffle}


def _batch(count, lo, hi, sweep, flow, storage, steps):
    return {"kind": "batch", "count": count, "lo": lo, "hi": hi, "sweep": sweep, "flow": flow,
            "storage": storage, "steps": steps}


def listed():
    cases = {
        # the smallest grid, phase field and solute only: a run of a few
        # thousand steps looked at every 50 (launch latency counts)
        "2d_128_no_flow": _grid(2, 128, 128, 1, "periodic", False, "fp32", 50, fold=4),
        # the benchmark's grid: crystal in an inflow, FP32
        "2d_1024_inflow": _grid(2, 1024, 1024, 1, "inflow", True, "fp32", 200),
        # the same with 16-bit storage
        "2d_1024_inflow_fp16": _grid(2, 1024, 1024, 1, "inflow", True, "fp16", 200),
        # a ragged grid of the paper's study, a baffle of solid nodes in front
        # of the inlet, the flow colliding by the central Hermite MRT
        "2d_775x650_baffle_chm": _grid(2, 775, 650, 1, "inflow", True, "fp32", 100, chm=True,
                                       baffle=True),
        # the study's finest grid: the largest 2D state
        "2d_2480x2080_inflow": _grid(2, 2480, 2080, 1, "inflow", True, "fp32", 50),
        # the 3D workload
        "3d_256_inflow": _grid(3, 256, 256, 256, "inflow", True, "fp32", 24, fold=0),
        # a ragged closed 3D channel with 16-bit storage
        "3d_203x150x134_channel_fp16": _grid(3, 203, 150, 134, "channel", True, "fp16", 64,
                                             fold=0),
        # a parametric sweep of uneven grids, advanced together in 16-bit storage
        "batch_32_of_256_768_fp16": _batch(32, 256, 768, 4, True, "fp16", 64),
        # a sweep of small grids
        "batch_30_of_32_128": _batch(30, 32, 128, 5, True, "fp32", 256),
        # the surrogate: inference on a whole domain
        "unet_forward_512": {"kind": "forward", "batch": 1, "height": 512, "width": 512,
                             "levels": 4},
        # the surrogate's training direction: loss and gradients of a minibatch of bands
        "unet_grad_8x256x512": {"kind": "grad", "batch": 8, "height": 256, "width": 512,
                                "levels": 4},
        # the block propagator: eight 50-step blocks, one judged by the LB
        "propagate_512": {"kind": "propagate", "height": 512, "width": 512, "block": 50,
                          "blocks": 8},
    }
    return [dict(c, name=k) for k, c in cases.items()]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["2d", "2d", "2d", "3d", "3d", "batch", "net"])
    storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
    if kind == "2d":
        nx, ny = log(96, 2480), log(96, 2080)
        flow = rng.random() < 0.8
        bounds = rng.choice(["inflow", "inflow", "periodic", "channel"]) if flow else "periodic"
        steps = max(10, min(200, int(2.0e8 / (nx * ny))))
        return _grid(2, nx, ny, 1, bounds, flow, storage, steps, fold=rng.choice([4, 5, 6]),
                     chm=flow and rng.random() < 0.25, baffle=flow and rng.random() < 0.25)
    if kind == "3d":
        nx, ny, nz = log(40, 256), log(40, 256), log(40, 256)
        bounds = rng.choice(["inflow", "inflow", "periodic", "channel"])
        steps = max(8, min(128, int(3.2e8 / (nx * ny * nz))))
        return _grid(3, nx, ny, nz, bounds, True, storage, steps, fold=0,
                     baffle=rng.random() < 0.2)
    if kind == "batch":
        lo = log(32, 256)
        hi = min(768, int(lo * rng.uniform(1.5, 3.0)))
        most = max(8, min(32, int(1.6e7 / (lo + hi) ** 2)))
        return _batch(rng.randint(8, most), lo, hi, rng.randint(0, 9999), True, storage, 64)
    levels = rng.choice([3, 4])
    width = 64 * 2 ** (levels - 1) * rng.choice([1, 1, 2])
    height = 2 ** (levels - 1) * rng.randint(16, 64)
    if rng.random() < 0.5:
        return {"kind": "forward", "batch": rng.randint(1, 3), "height": height, "width": width,
                "levels": levels}
    height = height // 2 // 8 * 8
    return {"kind": "grad", "batch": rng.randint(1, max(1, min(8, 2 ** 20 // (height * width)))),
            "height": height, "width": width, "levels": levels}


# ---- inputs -----------------------------------------------------------------------------
def _body(ny):
    """The body force that sustains U_CHANNEL between walls ny apart (2D)."""
    return 8.0 * (TAU_F - 0.5) / 3.0 * U_CHANNEL / ny ** 2, 0.0, 0.0


def _noise(seed, n):
    """The library's seeded noise in [-1, 1): SplitMix64 of seed ^ (index x golden ratio)."""
    z = np.arange(n, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ np.uint64(seed)) + np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    z = (z ^ (z >> np.uint64(31))) >> np.uint64(11)
    return torch.from_numpy(z.astype(np.float64) * 2.0 ** -52 - 1.0).cuda()


def _initial(p, crystal):
    """Initial phi and ux in 64 bits: a round crystal with a tanh interface and
    noise; the inflow's velocity, a uniform flow through a periodic box or a
    channel's parabola between its walls."""
    dim = p["dim"]
    shape = (p["ny"], p["nx"]) if dim == 2 else (p["nz"], p["ny"], p["nx"])
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") for n in shape]
    pos = torch.meshgrid(*ax, indexing="ij")[::-1]  # x, y[, z]
    r2 = sum((x - crystal[k]) ** 2 for x, k in zip(pos, ("cx", "cy", "cz")))
    phi = torch.tanh((crystal["radius"] - r2.sqrt()) / (math.sqrt(2.0) * W0))
    phi += crystal["noise_amp"] * _noise(crystal["seed"], phi.numel()).view(shape)
    ux = torch.full_like(phi, p["u_inlet"])
    if p["flow"] and p["bc"][0] == 0:
        ux += U_CHANNEL
        for x, n, bc in zip(pos[1:], shape[::-1][1:], p["bc"][1:]):
            if bc == 2:
                ux *= 4.0 * (x + 0.5) * (n - 0.5 - x) / n ** 2
    return phi, ux


def _start(sim, p, crystal):
    if p["flow"] and p["bc"][0] == 0:
        phi, ux = (x.cpu().numpy() for x in _initial(p, crystal))
        sim.init_fields(phi, np.full_like(phi, crystal["u0"]), ux=ux)
    else:
        sim.init_seed(**crystal)


def _problem(case, seed):
    """Model parameters and crystal seed of a grid case."""
    r = np.random.default_rng([seed, 11])
    dim, flow = case["dim"], case["flow"]
    size = (case["nx"], case["ny"], case["nz"])
    u_in = float(r.uniform(0.004, 0.012)) if flow and case["bounds"] == "inflow" else 0.0
    u0 = float(r.uniform(0.25, 0.45))
    p = dict(dim=dim, nx=size[0], ny=size[1], nz=size[2],
             bc=BOUNDS[case["bounds"]][:dim] + (0,) * (3 - dim),
             flow=int(flow), storage=STORAGE[case["storage"]], fold=case["fold"],
             tau_phi0=TAU_PHI, tau_u_liquid=TAU_U, tau_f=TAU_F, w0=W0, h_drag=DRAG,
             eps_aniso=float(r.uniform(0.02, 0.05)),
             theta0=float(r.uniform(0.0, 1.0)) if dim == 2 else 0.0,
             u_inlet=u_in, u0_inlet=u0 if case["bounds"] == "inflow" else 0.0,
             body_force=_body(size[1]) if flow and case["bounds"] == "channel" else (0.0,) * 3,
             collision=lbpf.COLL_CHM if case["chm"] else lbpf.COLL_BGK)
    least = min(size[:dim])
    crystal = dict(cx=(0.3 if case["bounds"] == "inflow" else 0.5) * size[0], cy=size[1] / 2.0,
                   cz=size[2] / 2.0 if dim == 3 else 0.0,
                   radius=float(min(r.uniform(8.0, 24.0), least / 5.0)), u0=u0, noise_amp=0.01,
                   seed=int(r.integers(1, 1 << 40)))
    return p, crystal


def _solid(case):
    """A baffle 4 nodes thick across the middle third at x = 0.15 nx, or None."""
    if not case["baffle"]:
        return None
    nx, ny = case["nx"], case["ny"]
    m = np.zeros((ny, nx) if case["dim"] == 2 else (case["nz"], ny, nx), bool)
    x0 = max(2, int(0.15 * nx))
    m[..., ny // 3: 2 * ny // 3, x0:x0 + 4] = True
    return m


def _sweep(case, seed):
    """(params, crystal seeds) of every instance of a batch: grids from the
    sweep's number, physics from the seed."""
    g = np.random.default_rng(case["sweep"])
    r = np.random.default_rng([seed, 12])
    ps, ss = [], []
    for _ in range(case["count"]):
        n = int(g.integers(case["lo"], case["hi"] + 1))
        u0 = float(r.uniform(0.1, 0.6))
        ps.append(dict(dim=2, nx=n, ny=n, flow=int(case["flow"]), bc=(1, 0, 0),
                       storage=STORAGE[case["storage"]], fold=int(r.choice([4, 5])),
                       tau_phi0=TAU_PHI, tau_u_liquid=TAU_U, tau_f=TAU_F, w0=W0, h_drag=DRAG,
                       eps_aniso=float(r.uniform(0.02, 0.06)),
                       u_inlet=float(r.uniform(0.0, 0.02)) if case["flow"] else 0.0,
                       u0_inlet=u0))
        ss.append((0.3 * n, 0.5 * n, 0.0, float(r.uniform(4.0, min(24.0, n / 5.0))), u0, 0.01,
                   int(r.integers(1, 1 << 40))))
    return ps, ss


def _net_layers(case):
    """(input channels, padded input channels, output channels) of every 3x3
    convolution in the order of the network's parameter vector."""
    C = [32 << i for i in range(case["levels"])]
    L = case["levels"]
    enc_a = [(4 if i == 0 else C[i - 1], 16 if i == 0 else C[i - 1], C[i]) for i in range(L)]
    enc_b = [(c, c, c) for c in C]
    up = [(C[i + 1], C[i + 1], C[i]) for i in range(L - 1)]
    dec_a = [(2 * C[i], 2 * C[i], C[i]) for i in range(L - 1)]
    dec_b = [(C[i], C[i], C[i]) for i in range(L - 1)]
    return enc_a, enc_b, up, dec_a, dec_b


def _net_weights(case, seed, head=1.0):
    """A parameter vector: per layer [3][3][out][in] weights and the biases,
    then the 1x1 head."""
    r = np.random.default_rng([seed, 13])
    out = []
    for group in _net_layers(case):
        for real, cin, cout in group:
            b = math.sqrt(6.0 / (9 * real))
            w = np.zeros((9, cout, cin), np.float32)
            w[:, :, :real] = r.uniform(-b, b, (9, cout, real))
            out += [w.reshape(-1), r.uniform(-0.05, 0.05, cout).astype(np.float32)]
    b = math.sqrt(6.0 / 32) * head
    out += [r.uniform(-b, b, 4 * 32).astype(np.float32),
            r.uniform(-0.01, 0.01, 4).astype(np.float32)]
    return np.concatenate(out)


def _net_fields(case, seed):
    """Normalised fields (phi, U, ux, uy) of crystals in channels and, as a
    target, the scaled change near their interfaces: FP32 NHWC on the GPU."""
    B, H, W = case["batch"], case["height"], case["width"]
    r = np.random.default_rng([seed, 14])
    g = torch.Generator(device="cuda").manual_seed(int(r.integers(1, 1 << 40)))
    y = torch.arange(H, device="cuda", dtype=torch.float32)[:, None]
    x = torch.arange(W, device="cuda", dtype=torch.float32)[None, :]
    X = torch.empty(B, H, W, 4, device="cuda")
    T = torch.empty_like(X)
    for b in range(B):
        d = float(r.uniform(8.0, 30.0)) - torch.hypot(x - W // 2, y - H // 2)
        noise = torch.rand(H, W, 4, generator=g, device="cuda") - 0.5
        X[b, ..., 0] = torch.tanh(d / (math.sqrt(2.0) * W0)) + 0.02 * noise[..., 0]
        X[b, ..., 1] = (float(r.uniform(0.25, 0.45)) - 0.3) / 0.2 - 0.5 * torch.exp(
            -(d / 20.0) ** 2) + 0.02 * noise[..., 1]
        X[b, ..., 2] = float(r.uniform(0.0, 1.0)) * 4.0 * (y + 0.5) * (H - 0.5 - y) / H ** 2 \
            + 0.02 * noise[..., 2]
        X[b, ..., 3] = 0.05 * noise[..., 3]
        band = torch.exp(-(d / 3.0) ** 2)
        for c, a in enumerate((1.0, -0.6, 0.2, 0.2)):
            T[b, ..., c] = a * band * (1.0 + 0.1 * noise[..., c])
    return X, T


class _Grid:
    def __init__(self, case, seed):
        p, s = _problem(case, seed)
        self.sim = lbpf.Sim(stream=lbpf.current_stream(), **p)
        _start(self.sim, p, s)
        solid = _solid(case)
        if solid is not None:
            self.sim.set_solid(solid)
        self.steps = case["steps"]
        names = ("phi", "U") + (("rho", "ux", "uy") + (("uz",) if case["dim"] == 3 else ())
                                if case["flow"] else ())
        self.mask = sum(1 << lbpf.FIELD_NAMES.index(k) for k in names)
        self.out = torch.empty(len(names), *self.sim.shape, pin_memory=True)
        self.fields = {k: self.out[i] for i, k in enumerate(names)}

    def run(self):
        self.sim.step(self.steps)
        lbpf.lbpf_read_fields(self.sim.h, self.mask, self.out.data_ptr(), self.out.nbytes, 0)
        return self.fields


class _Sweep:
    def __init__(self, case, seed):
        ps, ss = _sweep(case, seed)
        self.batch = lbpf.Batch(ps, ss, stream=lbpf.current_stream())
        self.steps = case["steps"]
        self.kids = [self.batch.instance(i) for i in range(case["count"])]
        self.out = [[torch.empty(k, s.nodes, pin_memory=True) for k in (3, 2)] for s in self.kids]

    def run(self):
        self.batch.step(self.steps)
        for s, (scalars, velocity) in zip(self.kids, self.out):
            for mask, o in ((lbpf.FIELD_PHI | lbpf.FIELD_U | lbpf.FIELD_RHO, scalars),
                            (lbpf.FIELD_UX | lbpf.FIELD_UY, velocity)):
                lbpf.lbpf_read_fields(s.h, mask, o.data_ptr(), o.nbytes, 0)
        return self.out


class _Net:
    def __init__(self, case, seed):
        self.grad = case["kind"] == "grad"
        self.net = lbpf.UNet(levels=case["levels"], batch=case["batch"], height=case["height"],
                             width=case["width"], stream=lbpf.current_stream())
        self.net.set_weights(_net_weights(case, seed))
        self.x, self.t = _net_fields(case, seed)
        self.y = torch.empty_like(self.x)

    def run(self):
        if self.grad:
            loss = self.net.grad(self.x, self.t)
            return {"loss": np.float32(loss), "grads": self.net.grads()}
        self.net.forward(self.x, self.y)
        return self.y


class _Propagator:
    def __init__(self, case, seed):
        H, W = case["height"], case["width"]
        r = np.random.default_rng([seed, 15])
        u0 = float(r.uniform(0.25, 0.45))
        p = dict(dim=2, nx=W, ny=H, flow=1, bc=(0, 2, 0), fold=int(r.choice([4, 5])),
                 eps_aniso=float(r.uniform(0.02, 0.05)), u_inlet=0.0, body_force=_body(H))
        self.sim = lbpf.Sim(stream=lbpf.current_stream(), **p)
        _start(self.sim, p, dict(cx=W // 2, cy=H // 2, cz=0.0,
                                 radius=float(r.uniform(8.0, 16.0)), u0=u0, noise_amp=0.01,
                                 seed=int(r.integers(1, 1 << 40))))
        self.sim.step(200)
        shape = {"levels": 4, "batch": 1, "height": H, "width": W}
        self.net = lbpf.UNet(height=H, width=W, stream=lbpf.current_stream())
        # a network whose predicted changes are small, as a trained one's are
        self.net.set_weights(_net_weights(shape, seed, head=0.01))
        self.cfg = lbpf.surrogate_cfg(steps_per_block=case["block"], judge_every=8)
        self.blocks = case["blocks"]
        names = ("phi", "U", "rho", "ux", "uy")
        self.mask = sum(1 << lbpf.FIELD_NAMES.index(k) for k in names)
        self.out = torch.empty(len(names), H, W, pin_memory=True)
        self.fields = {k: self.out[i] for i, k in enumerate(names)}

    def run(self):
        rep = lbpf.lbpf_surrogate_advance(self.sim, self.net, self.cfg, self.blocks)
        lbpf.lbpf_read_fields(self.sim.h, self.mask, self.out.data_ptr(), self.out.nbytes, 0)
        return {"fields": self.fields,
                "blocks": [rep["blocks"], rep["surrogate_blocks"], rep["judged_blocks"],
                           rep["fallback_blocks"]]}


def prepare(case, seed):
    kinds = {"grid": _Grid, "batch": _Sweep, "forward": _Net, "grad": _Net,
             "propagate": _Propagator}
    return kinds[case["kind"]](case, seed)


def run(state):
    return state.run()


# ---- bytes and operations of a pass ------------------------------------------------------
def _lb_work(dim, nodes, flow, storage, steps):
    """Per node and step: every population and phi(t - 1) read once and written
    once (with 16-bit storage also the node's reference of g)."""
    q = {(2, True): 27, (2, False): 18, (3, True): 33, (3, False): 14}[dim, flow]
    e = 4 if storage == "fp32" else 2
    per = 2 * q * e + 8 + (6 if e == 2 else 0)
    flops = {(2, True): 400, (2, False): 220, (3, True): 750, (3, False): 260}[dim, flow]
    return nodes * per * steps, nodes * flops * steps


def _net_flops(case):
    px, total = case["batch"] * case["height"] * case["width"], 0
    enc_a, enc_b, up, dec_a, dec_b = _net_layers(case)
    for group in (enc_a, enc_b, up, dec_a, dec_b):
        for i, (real, _, cout) in enumerate(group):
            total += 18 * real * cout * (px >> (2 * i))
    return total + 2 * 4 * 32 * px


def work(case):
    k = case["kind"]
    if k == "grid":
        n = case["nx"] * case["ny"] * case["nz"]
        b, f = _lb_work(case["dim"], n, case["flow"], case["storage"], case["steps"])
        fields = (2 + (1 + case["dim"] if case["flow"] else 0)) * 4 * n
        return {"bytes": b + fields, "flops": f}
    if k == "batch":
        g = np.random.default_rng(case["sweep"])
        n = sum(int(g.integers(case["lo"], case["hi"] + 1)) ** 2 for _ in range(case["count"]))
        b, f = _lb_work(2, n, case["flow"], case["storage"], case["steps"])
        return {"bytes": b + 20 * n, "flops": f}
    px = case.get("batch", 1) * case["height"] * case["width"]
    if k == "propagate":
        net = dict(case, batch=1, levels=4)
        judged = -(-case["blocks"] // 8)
        b, f = _lb_work(2, px, True, "fp32", case["block"] * judged)
        each = px * (27 * 4 * 2 + 8)  # the state read and written by a predicted block
        return {"bytes": b + (case["blocks"] - judged) * each + 20 * px,
                "flops": f + (case["blocks"] + 1) * _net_flops(net)}
    params = sum(9 * cin * cout + cout for g in _net_layers(case) for _, cin, cout in g) + 132
    if k == "forward":
        return {"bytes": 32 * px + 2 * params, "flops": _net_flops(case)}
    return {"bytes": 32 * px + 6 * params, "flops": 3 * _net_flops(case)}


# ---- the same in 64 bits, plain torch -----------------------------------------------------
_C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_C7 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
_C19 = _C7 + [c for d in ((0, 1), (0, 2), (1, 2)) for s, t in ((1, 1), (-1, -1), (1, -1), (-1, 1))
              for c in [tuple(s if i == d[0] else t if i == d[1] else 0 for i in range(3))]]


class _Lattice:
    def __init__(self, c, w, cs2):
        self.c, self.cs2 = c, cs2
        self.opp = [c.index(tuple(-v for v in d)) for d in c]
        view = (len(c),) + (1,) * len(c[0])
        self.w = torch.tensor(w, dtype=torch.float64, device="cuda").view(view)
        self.e = [torch.tensor([d[k] for d in c], dtype=torch.float64, device="cuda").view(view)
                  for k in range(len(c[0]))]

    def dot(self, v):
        """c_a . v for every direction: [q, ...]."""
        return sum(e * x for e, x in zip(self.e, v))


def _lattices(dim):
    if dim == 2:
        l9 = _Lattice(_C2, [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, 1 / 3)
        return l9, l9
    return (_Lattice(_C19, [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, 1 / 3),
            _Lattice(_C7, [1 / 4] + [1 / 8] * 6, 1 / 4))


class _Exact:
    """The coupled step (Eqs. 3-23 of the paper) on FP64 torch arrays [z,] y, x;
    populations stream by pulling from one-node padded arrays."""

    def __init__(self, p, crystal, solid=None):
        self.p, self.dim = p, p["dim"]
        self.lf, self.lg = _lattices(self.dim)
        self.shape = (p["nz"], p["ny"], p["nx"])[3 - self.dim:] if self.dim == 3 else (
            p["ny"], p["nx"])
        self.flow, self.bc = bool(p["flow"]), p["bc"]
        self.solid = None if solid is None else torch.from_numpy(solid).cuda()
        cs2 = self.lg.cs2
        self.tau0 = W0 * W0 / (cs2 * (TAU_PHI - 0.5))
        self.tpc = W0 * W0 / (cs2 * self.tau0)
        self.lam = cs2 * (TAU_U - 0.5) * self.tau0 / (0.6267 * W0 * W0)
        self.kdrag = DRAG * TAU_F / (4.0 * W0 * W0) if self.flow else 0.0
        self.body = p["body_force"]
        phi, ux = _initial(p, crystal)
        U = torch.full_like(phi, crystal["u0"])
        mask = 0.5 * (1.0 - phi.clamp(-1.0, 1.0)) if self.flow else torch.zeros_like(phi)
        u = [mask * ux if k == 0 else torch.zeros_like(phi) for k in range(self.dim)]
        self.f = self._feq(torch.ones_like(phi), u) if self.flow else None
        self.g = self.lg.w * U * (1.0 + self.lg.dot(u) / cs2)
        self.h = self.lg.w * phi
        self.prev = phi

    def _feq(self, rho, u):
        cu = self.lf.dot(u)
        uu = sum(x * x for x in u)
        return self.lf.w * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu)

    def _pad(self, a, left=None):
        """One node around a [..., (z,) y, x]: periodic wrap or nearest node;
        `left` replaces the ghost column at x = -1 of an inflow."""
        for k in range(self.dim):
            d = a.dim() - 1 - k
            n = a.shape[d]
            lo, hi = a.narrow(d, 0, 1), a.narrow(d, n - 1, 1)
            if self.bc[k] == 0:
                lo, hi = hi, lo
            elif k == 0 and self.bc[0] == 1 and left is not None:
                lo = left.expand(lo.shape)
            a = torch.cat([lo, a, hi], d)
        return a

    def _shift(self, padded, c, sign):
        """The values at x + sign c of a padded array."""
        for k in range(self.dim):
            d = padded.dim() - 1 - k
            padded = padded.narrow(d, 1 + sign * c[k], padded.shape[d] - 2)
        return padded

    def _behind_wall(self, c):
        """Nodes whose source x - c lies behind a wall or in a solid node."""
        b = torch.zeros(self.shape, dtype=torch.bool, device="cuda")
        for k in range(self.dim):
            if self.bc[k] == 2 and c[k]:
                d = self.dim - 1 - k
                b.narrow(d, 0 if c[k] > 0 else self.shape[d] - 1, 1).fill_(True)
        if self.solid is not None:
            # the copies beyond an inflow, outflow or wall are no solid nodes
            s = self._shift(self._pad(self.solid), c, -1)
            b |= s
        return b

    def _stream(self, lat, post, ghost):
        padded = self._pad(post, ghost)
        new = []
        for a, c in enumerate(lat.c):
            v = self._shift(padded[a], c, -1)
            if any(c) and (self.solid is not None or 2 in self.bc[:self.dim]):
                v = torch.where(self._behind(lat, a), post[lat.opp[a]], v)
            new.append(v)
        return torch.stack(new)

    def _behind(self, lat, a):
        cache = self.__dict__.setdefault("_walls", {})
        if lat.c[a] not in cache:
            cache[lat.c[a]] = self._behind_wall(lat.c[a])
        return cache[lat.c[a]]

    def _gradient(self, phi):
        P = self._pad(phi)
        S = None if self.solid is None else self._pad(self.solid)
        lat = self.lf
        grad = [0.0] * self.dim
        for a, c in enumerate(lat.c):
            if not any(c):
                continue
            v = self._shift(P, c, 1)
            if S is not None:
                alt = phi
                for k in reversed(range(self.dim)):
                    if c[k]:
                        one = tuple(c[k] if i == k else 0 for i in range(self.dim))
                        alt = torch.where(self._shift(S, one, 1), alt, self._shift(P, one, 1))
                v = torch.where(self._shift(S, c, 1), alt, v)
            for k in range(self.dim):
                if c[k]:
                    grad[k] = grad[k] + 3.0 * float(lat.w[a].flatten()[0]) * c[k] * v
        return grad

    def _anisotropy(self, grad):
        """a_s (Eq. 3) and N (Eq. 21); 1 and 0 where the gradient vanishes."""
        eps, k = self.p["eps_aniso"], self.p["fold"]
        g2 = sum(x * x for x in grad)
        flat = ~(g2 > 1e-12)
        norm = torch.where(flat, 1.0, g2).sqrt()
        n = [-x / norm for x in grad]
        if self.dim == 2:
            t = k * (torch.atan2(n[1], n[0]) - self.p["theta0"])
            a = 1.0 + eps * torch.cos(t)
            amp = k * eps * a * torch.sin(t)
            N = [amp * grad[1], -amp * grad[0]]
        else:
            S = sum(x ** 4 for x in n)
            a = 1.0 - 3.0 * eps + 4.0 * eps * S
            N = [16.0 * eps * a * norm * x * (S - x * x) for x in n]
        return torch.where(flat, 1.0, a), [torch.where(flat, 0.0, x) for x in N]

    def _moments(self):
        phi, U = self.h.sum(0), self.g.sum(0)
        if not self.flow:
            one, zero = torch.ones_like(phi), torch.zeros_like(phi)
            return phi, U, one, [zero] * self.dim, [zero] * self.dim
        rho = self.f.sum(0)
        ph = phi.clamp(-1.0, 1.0)
        K = self.kdrag * (1.0 + ph) ** 2 * (1.0 - ph)
        u = [((e * self.f).sum(0) + 0.5 * b) / (rho + 0.5 * K)
             for e, b in zip(self.lf.e, self.body)]
        return phi, U, rho, u, [b - K * x for x, b in zip(u, self.body)]

    def _chm(self, rho, us, F):
        """Central Hermite moments about u*, relaxed by order, and back by
        solving the q x q system of every node."""
        lat, d = self.lf, self.dim
        orders = [o for o in np.ndindex(*(3,) * d) if sum(v > 0 for v in o) <= 2]
        wf = 1.0 / TAU_F
        n = rho.numel()
        f = self.f.reshape(len(lat.c), n).T
        post = torch.empty_like(f)
        step = max(1, 60_000_000 // len(orders) ** 2)
        for i in range(0, n, step):
            s = slice(i, min(n, i + step))
            H = []  # per axis: the polynomials of c_a - u* at every node, [3, nodes, q]
            for k in range(d):
                X = lat.e[k].flatten()[None, :] - us[k].reshape(-1)[s][:, None]
                H.append((torch.ones_like(X), X, X * X - 1.0 / 3.0))
            M = torch.stack([math.prod(H[k][o[k]] for k in range(d)) for o in orders], 1)
            m = (M @ f[s][:, :, None])[:, :, 0]
            new = torch.zeros_like(m)
            at = {o: j for j, o in enumerate(orders)}
            new[:, at[(0,) * d]] = m[:, at[(0,) * d]]
            diag = [at[tuple(2 if i == k else 0 for i in range(d))] for k in range(d)]
            mean = m[:, diag].sum(1) / d
            for o, j in at.items():
                if sum(o) == 1:
                    k = o.index(1)
                    new[:, j] = (1.0 - wf) * m[:, j] + (1.0 - 0.5 * wf) * F[k].reshape(-1)[s]
                elif sum(o) == 2 and max(o) == 2:  # trace at rate 1, the rest at 1 / tau_f
                    new[:, j] = (1.0 - wf) * (m[:, j] - mean)
                elif sum(o) == 2:
                    new[:, j] = (1.0 - wf) * m[:, j]
            post[s] = torch.linalg.solve(M, new[:, :, None])[:, :, 0]
        return post.T.reshape(self.f.shape)

    def step(self):
        lf, lg = self.lf, self.lg
        phi, U, rho, u, F = self._moments()
        mask = 0.5 * (1.0 - phi.clamp(-1.0, 1.0))
        us = [mask * x for x in u]
        wU = 1.0 / (0.5 + (TAU_U - 0.5) * mask)
        a, N = self._anisotropy(self._gradient(phi))
        a2 = a * a
        wphi = 1.0 / (a2 * self.tpc + 0.5)
        Q = (phi - phi ** 3 + self.lam * U * (1.0 - phi * phi) ** 2) / self.tau0
        g = (1.0 - wU) * self.g + lg.w * (wU * U * (1.0 + lg.dot(us) / lg.cs2) -
                                          (phi - self.prev))
        h = (1.0 - wphi) * self.h + lg.w * (wphi * (phi - self.tpc * lg.dot(N)) + Q)
        f = None
        if self.flow:
            if self.p["collision"] == lbpf.COLL_CHM:
                f = self._chm(rho, us, F)
            else:
                cu, cF = lf.dot(us), lf.dot(F)
                uF = sum(x * y for x, y in zip(us, F))
                f = self.f + (self._feq(rho, us) - self.f) / TAU_F + (1.0 - 0.5 / TAU_F) * lf.w * (
                    cF * (3.0 + 9.0 * cu) - 3.0 * uF)
        old = (self.f, self.g, self.h)
        # the inflow ghost: rho = 1, u_in, U_in, phi = -1, a_s = 1
        one = torch.ones((1,) * self.dim, dtype=torch.float64, device="cuda")
        uin = [one * (self.p["u_inlet"] if self.flow and k == 0 else 0.0) for k in range(self.dim)]
        if self.flow:
            self.f = self._stream(lf, f, self._feq(one, uin))
        self.g = self._stream(lg, g, lg.w * self.p["u0_inlet"] * (1.0 + lg.dot(uin) / lg.cs2))
        # Eq. 19: a_s of the source, the old value of the destination
        src = self._stream(lg, h / a2, -lg.w)
        keep = self._stream(lg, (1.0 - 1.0 / a2).expand(h.shape), 0.0 * lg.w)
        self.h = src + keep * self.h
        if self.solid is not None:  # solid nodes keep their state
            if self.flow:
                self.f = torch.where(self.solid, old[0], self.f)
            self.g = torch.where(self.solid, old[1], self.g)
            self.h = torch.where(self.solid, old[2], self.h)
        self.prev = phi

    def fields(self):
        phi, U, rho, u, _ = self._moments()
        return dict(zip(("phi", "U", "rho", "ux", "uy", "uz"), [phi, U, rho] + u))


def _exact_grid(case, seed):
    p, s = _problem(case, seed)
    nodes = case["nx"] * case["ny"] * case["nz"]
    if case["chm"] and nodes * case["steps"] > (1.0e8 if case["dim"] == 2 else 1.0e7):
        return None  # a linear system per node and step
    e = _Exact(p, s, _solid(case))
    for _ in range(case["steps"]):
        e.step()
    f = e.fields()
    names = ("phi", "U") + (("rho", "ux", "uy", "uz")[:1 + case["dim"]] if case["flow"] else ())
    return {k: f[k].cpu() for k in names}


def _exact_batch(case, seed):
    out = []
    for p, s in zip(*_sweep(case, seed)):
        e = _Exact(dict(p, nz=1, theta0=0.0, collision=lbpf.COLL_BGK, body_force=(0.0,) * 3),
                   dict(zip(("cx", "cy", "cz", "radius", "u0", "noise_amp", "seed"), s)))
        for _ in range(case["steps"]):
            e.step()
        f = e.fields()
        out.append([torch.stack([f[k].reshape(-1) for k in names]).cpu()
                    for names in (("phi", "U", "rho"), ("ux", "uy"))])
    return out


def _exact_net(case, seed):
    import torch.nn.functional as fn

    flat = torch.from_numpy(_net_weights(case, seed)).cuda()
    flat = flat.double().requires_grad_(case["kind"] == "grad")
    groups, at = [], 0
    for group in _net_layers(case):
        layers = []
        for _, cin, cout in group:
            w = flat[at:at + 9 * cin * cout].view(3, 3, cout, cin)
            at += 9 * cin * cout
            layers.append((w.permute(2, 3, 0, 1), flat[at:at + cout]))
            at += cout
        groups.append(layers)
    head = flat[at:at + 128].view(4, 32, 1, 1), flat[at + 128:at + 132]
    enc_a, enc_b, up, dec_a, dec_b = groups

    def conv(x, wb):
        return fn.relu(fn.conv2d(x, wb[0][:, :x.shape[1]], wb[1], padding=1))

    X, T = _net_fields(case, seed)
    d, skips = X.double().permute(0, 3, 1, 2), []
    for i in range(case["levels"]):
        d = conv(conv(d, enc_a[i]), enc_b[i])
        if i < case["levels"] - 1:
            skips.append(d)
            d = fn.avg_pool2d(d, 2)
    for i in reversed(range(case["levels"] - 1)):
        d = conv(fn.interpolate(d, scale_factor=2, mode="nearest"), up[i])
        d = conv(conv(torch.cat([d, skips[i]], 1), dec_a[i]), dec_b[i])
    y = fn.conv2d(d, *head).permute(0, 2, 3, 1)
    if case["kind"] == "forward":
        return y.contiguous()
    loss = ((y - T.double()) ** 2).mean()
    loss.backward()
    return {"loss": np.float64(loss.item()), "grads": flat.grad.cpu()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "propagate":
        return None  # predictions are accepted or rejected on the way
    with torch.set_grad_enabled(kind == "grad"):
        if kind == "grid":
            return _exact_grid(case, seed)
        if kind == "batch":
            return _exact_batch(case, seed)
        return _exact_net(case, seed)

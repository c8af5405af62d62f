"""The work this framework is used for, as measurable cases.

Every solver case is one sampling interval of a running simulation: a number
of time steps, then the macroscopic fields read into the caller's device
tensors, the call pattern of a program that monitors or post-processes a run.
Surrogate cases are one inference or one training call.  Sizes are those of
the benchmark, the tests and the surrogate's data generation, or ragged ones
between them.

A case's "kind" names the workload:
  laplace     periodic 2D droplet (the small, launch-bound run)
  channel     2D droplet channel, velocity inlet and convective outlet
  obstacle    2D channel with a solid obstacle and Eq. 12 wetting
  ensemble    a batch of uneven 2D T-junction devices stepped together
  laplace3    periodic 3D droplet
  coflow3     3D co-flow device (tube, nozzle, both open faces)
  duct3       3D droplet in a walled duct, both open faces
  predict     surrogate ensemble inference
  train       surrogate ensemble training (Adam)
"""
import math

import numpy as np
import torch

from paper_2512_12934_gb300 import lbm
from paper_2512_12934_gb300 import workloads as W

STORE_BYTES = {"fp32": 4, "fp16store": 2, "fp64": 8}


def listed():
    return [
        # the smallest grid of the Laplace study (a droplet of 20 nodes' radius in a 100 x 100 box): hundreds of
        # these are run for one surface-tension fit; a step is a few microseconds, so launches and latency count
        {"name": "laplace_100x100", "kind": "laplace", "nx": 100, "ny": 100, "precision": "fp32", "steps": 100},
        # the headline channel of the benchmark: both open faces, walls with adhesion, a state that fits L2
        {"name": "channel_1024x128", "kind": "channel", "nx": 1024, "ny": 128, "precision": "fp32", "steps": 100},
        # the same physics on a grid far larger than L2: memory-bound stepping
        {"name": "channel_4096x2048", "kind": "channel", "nx": 4096, "ny": 2048, "precision": "fp32", "steps": 50},
        # half-precision storage, chosen to halve memory and traffic on large grids; ragged extents
        {"name": "channel_4001x1022_fp16", "kind": "channel", "nx": 4001, "ny": 1022, "precision": "fp16store",
         "steps": 20},
        # the double-precision diagnostic runs: obstacle geometry with phase-dependent wetting
        {"name": "obstacle_640x320_fp64", "kind": "obstacle", "nx": 640, "ny": 320, "precision": "fp64", "steps": 50},
        # a parameter study: uneven T-junction devices in one batch, every member's fields sampled
        {"name": "ensemble_24_tjunctions", "kind": "ensemble", "members": 24, "wc_lo": 24, "wc_hi": 72, "steps": 100},
        # the small 3D run (static droplet, 32^3): a step is a handful of short launches
        {"name": "laplace3_32", "kind": "laplace3", "n": 32, "precision": "fp32", "steps": 50},
        # the co-flow droplet generator at the benchmark's size: the large 3D run
        {"name": "coflow3_512x96x96", "kind": "coflow3", "nx": 512, "nc": 96, "precision": "fp32", "steps": 50},
        # 3D droplet migration with half-precision storage (a half-size copy of the paper's 500 x 100 x 100 duct)
        {"name": "duct3_250x50x50_fp16", "kind": "duct3", "nx": 250, "ny": 50, "nz": 50, "precision": "fp16store",
         "steps": 20},
        # a parameter sweep through the surrogate on device buffers (the benchmark's 65,536 points)
        {"name": "predict_65536", "kind": "predict", "n": 65536, "members": 5, "host": False},
        # the surrogate's answer to a handful of queries, host arrays in and out
        {"name": "predict_host_221", "kind": "predict", "n": 221, "members": 5, "host": True},
        # fitting the ensemble to a data set of the size the solver runs give, in the minibatches of Surrogate.fit
        {"name": "train_894_b64", "kind": "train", "n": 894, "batch": 64, "epochs": 2, "members": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["laplace", "channel", "channel16", "obstacle", "ensemble", "laplace3", "coflow3", "duct3",
                       "predict", "predict_host", "train"])
    if kind == "laplace":
        return {"kind": kind, "nx": _log_int(rng, 64, 1024), "ny": _log_int(rng, 64, 1024), "precision": "fp32",
                "steps": 100}
    if kind == "channel":
        return {"kind": kind, "nx": _log_int(rng, 900, 4096), "ny": _log_int(rng, 48, 2000), "precision": "fp32",
                "steps": 50}
    if kind == "channel16":
        return {"kind": "channel", "nx": rng.randint(2048, 4096), "ny": _log_int(rng, 512, 1024),
                "precision": "fp16store", "steps": 20}
    if kind == "obstacle":
        return {"kind": kind, "nx": _log_int(rng, 480, 960), "ny": _log_int(rng, 160, 320), "precision": "fp64",
                "steps": 50}
    if kind == "ensemble":
        lo = rng.randint(16, 48)
        return {"kind": kind, "members": _log_int(rng, 12, 32), "wc_lo": lo, "wc_hi": lo + rng.randint(8, 24),
                "steps": 100}
    if kind == "laplace3":
        return {"kind": kind, "n": _log_int(rng, 24, 96), "precision": "fp32", "steps": 50}
    if kind == "coflow3":
        return {"kind": kind, "nx": _log_int(rng, 192, 512), "nc": _log_int(rng, 48, 96), "precision": "fp32",
                "steps": 50}
    if kind == "duct3":
        return {"kind": kind, "nx": _log_int(rng, 200, 320), "ny": _log_int(rng, 32, 64), "nz": _log_int(rng, 32, 64),
                "precision": rng.choice(["fp32", "fp16store"]), "steps": 20}
    if kind in ("predict", "predict_host"):
        host = kind == "predict_host"
        return {"kind": "predict", "n": _log_int(rng, 16, 4096) if host else _log_int(rng, 512, 65536),
                "members": rng.randint(3, 8), "host": host}
    n = _log_int(rng, 256, 4096)
    return {"kind": "train", "n": n, "batch": _log_int(rng, 32, n), "epochs": 2, "members": rng.randint(3, 8)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _ensemble(case, rng):
    """T-junction devices with channel widths spread evenly over [wc_lo,
    wc_hi]; parameters from the box the surrogate's data generation samples
    (stable for a whole run)."""
    out = []
    for j in range(case["members"]):
        wc = case["wc_lo"] + (case["wc_hi"] - case["wc_lo"]) * j // max(1, case["members"] - 1)
        wd = max(4, int(round(rng.uniform(0.5, 1.0) * wc)))
        q = math.exp(rng.uniform(math.log(0.25), math.log(0.7)))
        m = math.exp(rng.uniform(math.log(0.4), math.log(2.5)))
        out.append(W.tjunction(Wc=wc, Wd=wd, q_ratio=q, M=m, G12=1.4, Gw=(0.3, -0.3), u_c=rng.uniform(0.005, 0.012),
                               front=wc // 2))
    return out


def _workload(case, seed):
    """The simulation of a single-solver case: geometry, parameters and
    initial fields.  The inflow is slow enough that no interface reaches the
    outlet while a case is being timed (a droplet there ends the run: the
    method's outlet does not carry it)."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "laplace":
        m = min(case["nx"], case["ny"])
        return W.laplace(nx=case["nx"], ny=case["ny"], R=m * rng.uniform(0.18, 0.25), G12=1.4, seed=seed)
    if kind == "channel":
        nx, ny = case["nx"], case["ny"]
        half = case["precision"] == "fp16store"
        return W.channel(nx=nx, ny=ny, R=min(0.23 * ny, 0.1 * nx) * rng.uniform(0.8, 1.0),
                         xc=nx * rng.uniform(0.19, 0.21), yc=ny * rng.uniform(0.48, 0.52),
                         u_max=(0.05 if half else 0.005) * rng.uniform(0.9, 1.0), seed=seed, noise=1e-4)
    if kind == "obstacle":
        nx, ny = case["nx"], case["ny"]
        x0, y0 = int(0.4 * nx), int(0.44 * ny)
        w = W.channel_obstacle(nx=nx, ny=ny, R=0.09 * ny * rng.uniform(0.8, 1.1), xc=0.15 * nx, yc=0.5 * ny,
                               obstacle=(x0, x0 + max(4, nx // 16), y0, y0 + int(0.37 * ny)),
                               u_max=0.005 * rng.uniform(0.8, 1.0), seed=seed)
        return w
    if kind == "laplace3":
        return W.laplace3(n=case["n"], R=case["n"] * rng.uniform(0.22, 0.28), G12=1.2, seed=seed)
    if kind == "coflow3":
        nc = case["nc"]
        return W.coflow3(nx=case["nx"], ny=nc, nz=nc, r_in=max(4, nc // 8), wall=2, r_out=nc // 2 - 2,
                         nozzle=max(8, case["nx"] * 3 // 32), q_ratio=rng.uniform(0.4, 0.6), M=rng.uniform(0.2, 0.5),
                         u_c=0.01 * rng.uniform(0.9, 1.0))
    if kind == "duct3":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        return W.duct3(nx=nx, ny=ny, nz=nz, R=0.2 * min(ny, nz) * rng.uniform(0.9, 1.1), xc=0.2 * nx,
                       u_max=0.02 * rng.uniform(0.9, 1.0), G12=1.2)
    raise ValueError("unknown kind %r" % kind)


def _net(case, seed):
    """A network ensemble's parameters: weights uniform in +-1/sqrt(fan_in),
    output biases 1 (the surrogate's targets are divided by their means)."""
    rng = np.random.default_rng(seed)

    def layer(fan_out, fan_in, bias, scale=1.0):
        b = scale / math.sqrt(fan_in)
        return [rng.uniform(-b, b, size=fan_out * fan_in), np.full(fan_out, bias) + rng.uniform(-0.02, 0.02, fan_out)]

    flat = [np.concatenate(layer(128, 4, 0.0) + layer(128, 128, 0.0) + layer(128, 128, 0.0) + layer(2, 128, 1.0))
            for _ in range(case["members"])]
    x = rng.standard_normal((case["n"], 4))
    return np.stack(flat).astype(np.float32), x.astype(np.float32), rng


def _labels(x, rng):
    """Smooth targets around 1 with a little scatter, as normalised droplet
    size and period are."""
    q, m = np.tanh(0.5 * x[:, 1]), np.tanh(0.5 * x[:, 2])
    t = np.stack([1.0 + 0.3 * q - 0.1 * m + 0.05 * x[:, 3], 1.0 - 0.4 * q + 0.1 * np.tanh(x[:, 0])], axis=1)
    return (t + rng.normal(0.0, 0.01, t.shape)).astype(np.float32)


LEARNING_RATE = 1e-4  # refining a fitted ensemble on new labels


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("predict", "train"):
        flat, x, rng = _net(case, seed)
        net = lbm.MLP(case["members"], seed=seed)
        net.set_params(flat)
        st = {"case": case, "net": net, "x": x}
        if kind == "train":
            st["t"] = _labels(x, rng)
        elif not case["host"]:
            st["x"] = torch.from_numpy(x).cuda()
            st["mean"] = torch.empty(case["n"], 2, device="cuda")
            st["spread"] = torch.empty(case["n"], device="cuda")
        return st
    if kind == "ensemble":
        ws, precision = _ensemble(case, np.random.default_rng(seed)), "fp32"
    else:
        ws, precision = [_workload(case, seed)], case["precision"]
    members = [lbm.Solver(w.cfg, w.solid, w.rho, w.u, precision=precision) for w in ws]
    return {"case": case, "members": members, "batch": lbm.Batch(members) if kind == "ensemble" else None,
            "rho": [torch.empty(2, *s.shape, device="cuda") for s in members],
            "u": [torch.empty(s.dim, *s.shape, device="cuda") for s in members]}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    case = state["case"]
    if case["kind"] == "predict":
        if case["host"]:
            return state["net"].predict(state["x"])
        state["net"].predict_device(state["x"].data_ptr(), case["n"], state["mean"].data_ptr(),
                                    state["spread"].data_ptr())
        return state["mean"], state["spread"]
    if case["kind"] == "train":
        state["net"].train(state["x"], state["t"], epochs=case["epochs"], batch=case["batch"], lr=LEARNING_RATE,
                           shuffle_seed=7)
        return state["net"].params()
    if state["batch"] is not None:
        state["batch"].step(case["steps"])
        state["batch"].sync()
    else:
        state["members"][0].step(case["steps"])
    for s, rho, u in zip(state["members"], state["rho"], state["u"]):
        s.macros_f32(rho.data_ptr(), u.data_ptr(), device=True)
    return {"rho": state["rho"], "u": state["u"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _geometry(case):
    """(nodes, fluid nodes) of a solver case."""
    kind = case["kind"]
    if kind == "ensemble":
        ws = _ensemble(case, np.random.default_rng(0))  # side-channel widths follow the seed: a typical draw
        return sum(w.nodes for w in ws), sum(w.fluid_nodes for w in ws)
    if kind == "laplace":
        return (case["nx"] * case["ny"],) * 2
    if kind == "laplace3":
        return (case["n"] ** 3,) * 2
    if kind == "channel":
        return case["nx"] * case["ny"], case["nx"] * (case["ny"] - 2)
    w = _workload(case, 0)
    return w.nodes, w.fluid_nodes


def work(case):
    kind = case["kind"]
    per_sample = 2 * (4 * 128 + 2 * 128 * 128 + 128 * 2)  # multiply-adds of one member's forward pass, as flops
    params = 33922
    if kind == "predict":
        return {"bytes": 4.0 * (case["n"] * 7 + case["members"] * params),
                "flops": float(per_sample) * case["members"] * case["n"]}
    if kind == "train":
        steps = case["epochs"] * (case["n"] // case["batch"])
        return {"bytes": 4.0 * (steps * case["batch"] * 6 + 2 * case["members"] * params),
                "flops": 3.0 * per_sample * case["members"] * case["batch"] * steps}
    nodes, fluid = _geometry(case)
    three = kind in ("laplace3", "coflow3", "duct3")
    precision = case.get("precision", "fp32")
    planes = 38 if three else 18
    # every population is read and written once per step, the fields are written once per pass; the collision,
    # the interaction stencil and the forces take about 30 (2D) and 45 (3D) operations per population
    return {"bytes": float(case["steps"]) * 2 * planes * STORE_BYTES[precision] * fluid + 4.0 * nodes * (5 if three else 4),
            "flops": float(case["steps"]) * planes * (45 if three else 30) * fluid}


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _lattice(dim):
    if dim == 2:
        return [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
    e = [(0, 0, 0)]
    for a in range(3):
        for s in (1, -1):
            e.append(tuple(s if b == a else 0 for b in range(3)))
    for a, b in ((0, 1), (0, 2), (1, 2)):
        for sb in (1, -1):
            for sa in (1, -1):
                v = [0, 0, 0]
                v[a], v[b] = sa, sb
                e.append(tuple(v))
    return e


def _moments(e, dim):
    """Rows of the orthogonal moment basis of the collision operator."""
    rows = []
    for v in e:
        e2 = sum(c * c for c in v)
        if dim == 2:
            x, y = v
            rows.append([1, 3 * e2 - 4, (9 * e2 * e2 - 21 * e2 + 8) / 2, x, (3 * e2 - 5) * x, y, (3 * e2 - 5) * y,
                         x * x - y * y, x * y])
        else:
            x, y, z = v
            q, p = 5 * e2 - 9, 3 * e2 - 5
            rows.append([1, 19 * e2 - 30, (21 * e2 * e2 - 53 * e2 + 24) / 2, x, q * x, y, q * y, z, q * z,
                         3 * x * x - e2, p * (3 * x * x - e2), y * y - z * z, p * (y * y - z * z), x * y, y * z, x * z,
                         (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z])
    return np.array(rows, dtype=np.float64).T


def _rates(cfg, k, dim):
    snu = 1.0 / (3.0 * cfg["nu"][k] + 0.5)
    eps = 1.0 / (3.0 * max(cfg["nu"]) + 0.5) if cfg["s_eps_mode"] else snu
    se, sq = (cfg["s_e"] if cfg["s_e"] > 0 else snu), cfg["s_q"]
    if dim == 2:
        return [1, se, eps, 1, sq, 1, sq, snu, snu]
    return [1, se, eps, 1, sq, 1, sq, 1, sq, snu, eps, snu, eps, snu, snu, snu, sq, sq, sq]


class _Reference:
    """The two-component step in double precision: whole-array operations on
    fields laid out as the solver's ([z][y][x] in 3D, [y][x] in 2D)."""

    SIDES = ("xmin", "xmax", "ymin", "ymax", "zmin", "zmax")

    def __init__(self, w):
        cfg = w.cfg
        self.cfg, self.dim = cfg, 3 if cfg.get("lattice") == "d3q19" else 2
        dim, dev = self.dim, {"dtype": torch.float64, "device": "cuda"}
        self.dev = dev
        self.ext = [cfg["nx"], cfg["ny"]] + ([cfg["nz"]] if dim == 3 else [])
        self.shape = tuple(reversed(self.ext))
        self.N = int(np.prod(self.shape))
        self.periodic = [bool(p) for p in cfg["periodic"]][:dim]
        self.e = _lattice(dim)
        self.Q = len(self.e)
        norm = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36} if dim == 2 else {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
        self.w = [norm[sum(c * c for c in v)] for v in self.e]
        self.opp = [self.e.index(tuple(-c for c in v)) for v in self.e]
        self.et = torch.tensor(self.e, **dev).T.contiguous()             # [dim][Q]
        T = _moments(self.e, dim)
        self.T = torch.tensor(T, **dev)
        self.Ti = torch.tensor(T.T / (T * T).sum(axis=1), **dev)
        self.s = [torch.tensor(_rates(cfg, k, dim), **dev)[:, None] for k in range(2)]
        shells = ({1: 4 / 21, 2: 4 / 45, 4: 1 / 60, 5: 2 / 315, 8: 1 / 5040} if dim == 2 else
                  {1: 4 / 45, 2: 1 / 21, 3: 2 / 105, 4: 5 / 504, 5: 1 / 315, 6: 1 / 630, 8: 1 / 5040})
        reach = np.stack(np.meshgrid(*[range(-2, 3)] * dim, indexing="ij"), -1).reshape(-1, dim)
        self.taps = [(tuple(int(c) for c in v), shells[int((v * v).sum())]) for v in reach
                     if int((v * v).sum()) in shells]
        self.faces = cfg["faces"]
        open_sides = {f["side"] for f in self.faces}
        # padded index of each axis for the interaction stencil: periodic wrap, mirror across an open side, solid
        # (index 0 with the valid flag off) beyond a closed one
        self.pad = []
        for a, n in enumerate(self.ext):
            i = torch.arange(-2, n + 2, device="cuda")
            ok = (i >= 0) & (i < n)
            if self.periodic[a]:
                i, ok = i % n, torch.ones_like(ok)
            else:
                if self.SIDES[2 * a] in open_sides:
                    ok, i = ok | (i < 0), torch.where(i < 0, -1 - i, i)
                if self.SIDES[2 * a + 1] in open_sides:
                    ok, i = ok | (i >= n), torch.where(i >= n, 2 * n - 1 - i, i)
                i = torch.where(ok, i, torch.zeros_like(i))
            self.pad.append((i, ok))
        solid = torch.zeros(self.shape, dtype=torch.bool, device="cuda")
        if w.solid is not None:
            solid = torch.from_numpy(np.ascontiguousarray(w.solid)).cuda().reshape(self.shape) != 0
        self.solid, self.fluid = solid, ~solid
        # blocked pulls: the source x - e is solid or beyond a non-periodic side
        self.blocked = []
        for v in self.e:
            b = self._shift(solid, v).clone()
            for a in range(dim):
                if v[a] and not self.periodic[a]:
                    b.select(dim - 1 - a, 0 if v[a] > 0 else self.ext[a] - 1).fill_(True)
            self.blocked.append(b)
        s_pad = self._padded(solid.double(), outside=1.0)
        self.adh = self._gradient(s_pad)
        # face nodes, their inward neighbours and the inflow there
        self.face_data = []
        strides = [1, self.ext[0]] + ([self.ext[0] * self.ext[1]] if dim == 3 else [])
        flat_solid = solid.reshape(-1)
        for f in self.faces:
            side = self.SIDES.index(f["side"])
            a, sign = side // 2, 1 if side & 1 else -1
            tang = [b for b in range(dim) if b != a]
            lo = [f["lo"]] if dim == 2 else list(f["lo"])
            hi = [f["hi"]] if dim == 2 else list(f["hi"])
            base = strides[a] * (self.ext[a] - 1 if side & 1 else 0)
            idx = torch.full((1,), base, device="cuda", dtype=torch.int64)
            for b, l, h in zip(tang, lo, hi):  # the first tangential axis varies fastest
                r = torch.arange(l, h + 1, device="cuda") * strides[b]
                idx = (r[:, None] + idx[None, :]).reshape(-1) if b != tang[0] else (idx[:, None] + r[None, :]).reshape(-1)
            keep = ~flat_solid[idx]
            d = {"kind": f["kind"], "axis": a, "sign": sign, "node": idx[keep], "nbr": (idx - sign * strides[a])[keep],
                 "unknown": [i for i, v in enumerate(self.e) if sign * v[a] < 0], "alpha": f.get("alpha", 1),
                 "chi": f.get("chi", 1)}
            if f["kind"] == "inlet":
                d["speed"] = torch.tensor(np.asarray(f["profile"], dtype=np.float64).reshape(-1), **dev)[keep]
                rp = f.get("rho_profile")
                rin = (np.asarray(rp, dtype=np.float64).reshape(2, -1) if rp is not None else
                       np.repeat(np.asarray(f["rho_in"], dtype=np.float64)[:, None], idx.numel(), axis=1))
                d["rho"] = torch.tensor(rin, **dev)[:, keep]
            self.face_data.append(d)
        self.G12, self.Gw, self.body = cfg["G12"], cfg["Gw"], cfg["body"]
        self.wet = cfg.get("wetting_delta", 0.0)
        rho = torch.from_numpy(np.ascontiguousarray(w.rho)).to(**dev).reshape(2, -1)
        u = torch.from_numpy(np.ascontiguousarray(w.u)).to(**dev).reshape(dim, -1)
        fl = self.fluid.reshape(-1)
        self.f = torch.stack([self._feq(rho[k], u) for k in range(2)]) * fl  # [2][Q][N]
        self.post = [self.f[:, :, d["node"]].clone() for d in self.face_data]
        self.F = torch.zeros(2, dim, self.N, **dev)
        self.lam, self.chi = 0.0, 1.0
        self.rho, self.u = rho * fl, u * fl

    def _shift(self, x, v):
        """x[r - v], wrapped on every axis."""
        sh = [(v[a], x.dim() - 1 - a) for a in range(self.dim) if v[a]]
        return torch.roll(x, [s for s, _ in sh], [d for _, d in sh]) if sh else x

    def _padded(self, x, outside=0.0):
        ok = None
        for a in range(self.dim):
            i, v = self.pad[a]
            x = x.index_select(x.dim() - 1 - a, i)
            v = v.reshape([-1 if b == a else 1 for b in reversed(range(self.dim))])
            ok = v if ok is None else ok & v
        return torch.where(ok, x, torch.full_like(x, outside)) if not bool(ok.all()) else x

    def _gradient(self, p):
        """sum over the interaction stencil of w(e) p(x + e) e, per axis."""
        g = [torch.zeros(self.shape, **self.dev) for _ in range(self.dim)]
        for v, wt in self.taps:
            cut = p
            for a in range(self.dim):
                cut = cut.narrow(self.dim - 1 - a, 2 + v[a], self.ext[a])
            for a in range(self.dim):
                if v[a]:
                    g[a].add_(cut, alpha=wt * v[a])
        return torch.stack([x.reshape(-1) for x in g])

    def _feq(self, rho, u):
        uu = (u * u).sum(0)
        out = []
        for i, v in enumerate(self.e):
            eu = sum(v[a] * u[a] for a in range(self.dim) if v[a]) if i else torch.zeros_like(uu)
            out.append(self.w[i] * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu))
        return torch.stack(out)

    def _open_faces(self, f):
        for n, d in enumerate(self.face_data):
            a, node, nbr = d["axis"], d["node"], d["nbr"]
            g, here = f[:, :, nbr], f[:, :, node]
            if d["kind"] == "inlet":
                r2 = g.sum(1)
                j = torch.einsum("aq,kqn->an", self.et, g) + 0.5 * self.F[:, :, nbr].sum(0)
                u2 = j / r2.sum(0)
                uin = torch.zeros(self.dim, node.numel(), **self.dev)
                uin[a] = -d["sign"] * d["speed"]
                for k in range(2):
                    new = self._feq(d["rho"][k], uin) + g[k] - self._feq(r2[k], u2)
                    for i in d["unknown"]:
                        here[k, i] = new[i]
                    if d["alpha"]:
                        miss = d["rho"][k] * uin - (self.et @ here[k] + 0.5 * self.F[k][:, node])
                        for i in d["unknown"]:
                            for b in range(self.dim):
                                if self.e[i][b]:
                                    den = sum(self.w[q] * self.e[q][b] ** 2 for q in d["unknown"])
                                    here[k, i] += self.w[i] * self.e[i][b] * miss[b] / den
            else:
                for i in d["unknown"]:
                    here[:, i] = (self.post[n][:, i] + self.lam * g[:, i]) / (1.0 + self.lam)
                self.post[n] = here.clone()
            f[:, :, node] = here

    def step(self):
        dim, fl = self.dim, self.fluid.reshape(-1)
        old = self.f.reshape(2, self.Q, *self.shape)
        f = torch.empty_like(old)
        for i, v in enumerate(self.e):
            f[:, i] = torch.where(self.blocked[i], old[:, self.opp[i]], self._shift(old[:, i], v))
        f = f.reshape(2, self.Q, -1)
        f *= fl
        del old
        self._open_faces(f)
        rho = f.sum(1)
        rt = torch.where(fl, rho.sum(0), torch.ones_like(rho[0]))
        grad = [self._gradient(self._padded(rho[k].reshape(self.shape))) for k in range(2)]
        gw = list(self.Gw)
        if self.wet > 0.0:
            re = (rho[0] - rho[1]) / rt
            one = torch.where(re > self.wet, torch.full_like(re, gw[0]), torch.where(
                re > 0, gw[0] * re / self.wet, torch.where(re > -self.wet, -gw[1] * re / self.wet,
                                                           torch.full_like(re, gw[1]))))
            gw = [one, one]
        body = torch.tensor(self.body[:dim], **self.dev)[:, None]
        F = torch.stack([-self.G12 * rho[k] * grad[1 - k] - gw[k] * rho[k] * self.adh + body * (rho[k] / rt)
                         for k in range(2)])
        del grad
        u = torch.stack([sum((self.et[a][:, None] * f[k]).sum(0) + 0.5 * F[k, a] for k in range(2)) / rt
                         for a in range(dim)])
        qin = qout = mean = 0.0
        have_in = have_out = False
        for d in self.face_data:
            a, n = d["axis"], d["nbr"] if d["kind"] == "outlet" else d["node"]
            if d["kind"] == "inlet":
                have_in = True
                qin = qin + (rho[:, n].sum(0) * (-d["sign"]) * u[a][n]).sum().item()
            else:
                have_out = True
                un = d["sign"] * u[a][n]
                qout, mean = (rho[:, n].sum(0) * un).sum().item(), un.mean().item()
                if d["chi"]:
                    u[a][d["node"]] = self.chi * u[a][n]
        u *= fl
        for k in range(2):
            eq = self._feq(rho[k], u)
            uF = (u * F[k]).sum(0)
            fb = torch.stack([self.w[i] * (sum((3.0 * v[a]) * F[k, a] for a in range(dim)) - 3.0 * uF +
                                           9.0 * sum(v[a] * u[a] for a in range(dim)) *
                                           sum(v[a] * F[k, a] for a in range(dim))) for i, v in enumerate(self.e)])
            m = -self.s[k] * (self.T @ (f[k] - eq))
            m += (1.0 - 0.5 * self.s[k]) * (self.T @ fb)
            del eq, fb
            f[k] += self.Ti @ m
        self.f, self.F, self.rho, self.u = f * fl, F * fl, rho, u
        if have_out:
            self.lam = max(mean, 0.0)
            self.chi = qin / qout if have_in and abs(qout) >= 1e-14 else 1.0


def _exact_fields(w, steps):
    r = _Reference(w)
    for _ in range(steps):
        r.step()
    return r.rho.reshape(2, *r.shape), r.u.reshape(r.dim, *r.shape)


def _split(flat):
    """One member's parameters as (W1, b1, W2, b2, W3, b3, W4, b4)."""
    out, at = [], 0
    for rows, cols in ((128, 4), (128, 128), (128, 128), (2, 128)):
        out.append(flat[at:at + rows * cols].reshape(rows, cols))
        at += rows * cols
        out.append(flat[at:at + rows])
        at += rows
    return out


def _forward(p, x):
    h = x
    for l in range(3):
        h = torch.nn.functional.gelu(h @ p[2 * l].T + p[2 * l + 1])
    return h @ p[6].T + p[7]


def _shuffles(n, seed, epochs):
    """The documented epoch order: a splitmix64 Fisher-Yates shuffle of
    0..n-1, the generator continuing from epoch to epoch."""
    s, mask = seed, (1 << 64) - 1
    for _ in range(epochs):
        p = list(range(n))
        for i in range(n - 1, 0, -1):
            s = (s + 0x9E3779B97F4A7C15) & mask
            z = s
            z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
            j = (z ^ (z >> 31)) % (i + 1)
            p[i], p[j] = p[j], p[i]
        yield p


def _exact_net(case, seed):
    flat, x, rng = _net(case, seed)
    x64 = torch.from_numpy(x).double().cuda()
    params = torch.from_numpy(flat).double().cuda()
    if case["kind"] == "predict":
        y = torch.stack([_forward(_split(p), x64) for p in params])
        mean = y.mean(0)
        spread = (((y - mean) ** 2).mean(0).sqrt() / mean.abs().clamp(min=1e-30)).amax(1)
        return mean, spread
    t64 = torch.from_numpy(_labels(x, rng)).double().cuda()
    n, batch = case["n"], min(case["batch"], case["n"])
    m, v, count = torch.zeros_like(params), torch.zeros_like(params), 0
    for order in _shuffles(n, 7, case["epochs"]):
        order = torch.tensor(order, device="cuda")
        for b0 in range(0, n - batch + 1, batch):
            rows = order[b0:b0 + batch]
            p = params.clone().requires_grad_(True)
            loss = sum(((_forward(_split(q), x64[rows]) - t64[rows]) ** 2).mean() for q in p)
            g, = torch.autograd.grad(loss, p)
            count += 1
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            params = params - LEARNING_RATE * (m / (1 - 0.9 ** count)) / ((v / (1 - 0.999 ** count)).sqrt() + 1e-8)
    return params


def exact(case, seed):
    if case["kind"] in ("predict", "train"):
        return _exact_net(case, seed)
    if case["kind"] == "ensemble":
        ws = _ensemble(case, np.random.default_rng(seed))
    else:
        ws = [_workload(case, seed)]
    fields = [_exact_fields(w, case["steps"]) for w in ws]
    return {"rho": [r for r, _ in fields], "u": [u for _, u in fields]}

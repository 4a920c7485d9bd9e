"""The work that programs using this library have it do, as measurable cases.

Four kinds, each through the public entry points (lbm.Lattice, the batch
calls of include/lbm.h, lbm.Surrogate):

  lattice  fields in, `steps` fused time steps, macroscopic fields out
  batch    the same for many independent periodic boxes in one handle
  forward  one jump of the learned surrogate on (rho, u_x, u_y, T)
  train    one Adam step of the surrogate, the updated parameters out
  grad     loss and gradients of the surrogate without an update

The lattice's read-out widens every field to float64 whatever the storage; a
program that stores its populations in 32 or 16 bits keeps the fields in
that type, so run() hands them back in the working precision of the case.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2106_01557_gb300 import lbm

DTYPE = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.float16, "bf16s": torch.bfloat16}
SIZE = {"f64": 8, "f32": 4, "f16s": 2, "bf16s": 2}
LAYOUTS = ("slab", "droplets", "boiling", "open")
HOT_LEN = 32
# g relaxation rates of the temperature sweep (the benchmark's batch)
SWEEP = {"sig_eps": 1.4, "sig_p": 1.8}
CH, BLOCKS = 64, 6


def listed():
    return [
        # the plain method's reference run: a liquid slab on a small periodic
        # box in double precision (oracle comparisons, conservation checks)
        {"name": "slab_128_f64", "kind": "lattice", "layout": "slab", "nx": 128, "ny": 128, "precision": "f64", "steps": 100},
        # the same box in single precision: the smallest steps, where launches and latency count
        {"name": "slab_128_f32", "kind": "lattice", "layout": "slab", "nx": 128, "ny": 128, "precision": "f32", "steps": 400},
        # static droplets for Laplace's law: a state that stays in the L2 cache
        {"name": "droplets_512_f32", "kind": "lattice", "layout": "droplets", "nx": 512, "ny": 512, "precision": "f32", "steps": 400},
        # the headline: heated-wall boiling between bounce-back walls, FP32
        {"name": "boiling_4096x1024_f32", "kind": "lattice", "layout": "boiling", "nx": 4096, "ny": 1024, "precision": "f32", "steps": 200},
        # the same with FP16 shifted storage and stochastic rounding (its default)
        {"name": "boiling_4096x1024_f16s", "kind": "lattice", "layout": "boiling", "nx": 4096, "ny": 1024, "precision": "f16s", "steps": 200},
        # a mid-size lattice of odd sides in the other 16-bit format
        {"name": "boiling_1363x777_bf16s", "kind": "lattice", "layout": "boiling", "nx": 1363, "ny": 777, "precision": "bf16s", "steps": 200},
        # a droplet evaporating in a box open and heated on all four sides (the D^2 law, the droplet pair)
        {"name": "open_512_f32", "kind": "lattice", "layout": "open", "nx": 512, "ny": 512, "precision": "f32", "steps": 200},
        # the coexistence sweep: 256 uneven boxes at their own temperatures, FP16 storage
        {"name": "batch_256_f16s", "kind": "batch", "cases": 256, "lo": 64, "hi": 512, "multiple": 8, "plan": 4, "precision": "f16s", "steps": 300},
        # training data of the surrogate: 40 equal boxes, K = 50 steps between two snapshots
        {"name": "batch_40x256_f32", "kind": "batch", "cases": 40, "lo": 256, "hi": 256, "multiple": 8, "plan": 10, "precision": "f32", "steps": 50},
        # one jump of the rollout at its full size
        {"name": "forward_1x1024x1024", "kind": "forward", "n": 1, "h": 1024, "w": 1024},
        # one training step on a minibatch of eight 256 x 256 pairs
        {"name": "train_8x256x256", "kind": "train", "n": 8, "h": 256, "w": 256},
        # gradients of a few small images whose width is no multiple of the 128-pixel strips
        {"name": "grad_3x100x208", "kind": "grad", "n": 3, "h": 100, "w": 208},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice"] * 5 + ["batch"] * 2 + ["forward", "train", "grad"])
    if kind == "lattice":
        precision = rng.choice(["f64", "f32", "f32", "f16s", "bf16s"])
        layout = rng.choice(LAYOUTS)
        hi = 512 if precision == "f64" else 4096
        nx, ny = _log_int(rng, 64, hi), _log_int(rng, 64, hi)
        while nx * ny > (1 << 22):
            nx, ny = (nx + 1) // 2, ny
        # the read-out interval: about 20 steps (a verification) to 400, no
        # more work than the largest listed case
        most = max(20, min(400, (200 << 22) // (nx * ny), (200 << 15) // (nx * ny) * 16 if precision == "f64" else 400))
        return {"kind": kind, "layout": layout, "nx": nx, "ny": ny, "precision": precision,
                "steps": _log_int(rng, 20, most)}
    if kind == "batch":
        lo = _log_int(rng, 48, 128)
        hi = min(512, lo * rng.randint(1, 6))
        return {"kind": kind, "cases": _log_int(rng, 2, 128), "lo": lo, "hi": hi, "multiple": rng.choice([1, 8]),
                "plan": rng.randrange(1000), "precision": rng.choice(["f32", "f16s", "bf16s"]), "steps": _log_int(rng, 20, 300)}
    n, h, w = _log_int(rng, 1, 8), _log_int(rng, 16, 512), 16 * _log_int(rng, 1, 32)
    if kind == "forward":
        n, h, w = _log_int(rng, 1, 4), _log_int(rng, 16, 1024), 16 * _log_int(rng, 1, 64)
    while n * h * w > ((1 << 20) if kind == "forward" else (1 << 19)):
        h = (h + 1) // 2
    return {"kind": kind, "n": n, "h": h, "w": w}


# ---------------------------------------------------------------------------
# Thermodynamics of the Carnahan-Starling fluid the inputs are built from
# (a = R = 1, b = 4: the default constants)
# ---------------------------------------------------------------------------
K_EOS, K_INT, VARPI = 0.479820, 2.294922, 1.0 / 6.0
TC = 0.1872945669467330 / 0.4963880577294099 / 4.0


def _p(r, T):
    return r * T * (1 + r + r * r - r**3) / (1 - r) ** 3 - r * r


def _dp(r, T):
    return T * (1 + 4 * r + 4 * r * r - 4 * r**3 + r**4) / (1 - r) ** 4 - 2 * r


def _mu(r, T):
    return T * (math.log(r) + (4 * r - 3 * r * r) / (1 - r) ** 2 + r * (4 - 2 * r) / (1 - r) ** 3) - 2 * r


def _bisect(fn, lo, hi):
    up = fn(lo) > 0
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        if (fn(mid) > 0) == up:
            lo = mid
        else:
            hi = mid
    return 0.5 * (lo + hi)


_COEX = {}


def _coexistence(Tr):
    """(rho_v, rho_l, p_s) at reduced temperature Tr: equal pressure and chemical potential."""
    if Tr in _COEX:
        return _COEX[Tr]
    T = Tr * TC
    low = min((k / 4000.0 for k in range(1, 4000)), key=lambda r: _dp(r, T))
    s1, s2 = _bisect(lambda r: _dp(r, T), 1e-9, low), _bisect(lambda r: _dp(r, T), low, 0.9999)

    def liquid(ps):
        hi = s2
        while _p(hi, T) < ps:
            hi += 0.5 * (1 - hi)
        return _bisect(lambda r: _p(r, T) - ps, s2, hi)

    lo = _bisect(lambda r: _p(r, T) - _p(s2, T), 1e-9, s1) if _p(s2, T) > 0 else 1e-9
    rv = _bisect(lambda r: _mu(liquid(_p(r, T)), T) - _mu(r, T), lo * (1 + 1e-12), s1 * (1 - 1e-12))
    _COEX[Tr] = rv, liquid(_p(rv, T)), _p(rv, T)
    return _COEX[Tr]


def _scales(Tr):
    rv, rl, ps = _coexistence(Tr)
    cs2 = K_INT**2 * K_EOS * (_dp(rl, Tr * TC) + 2 * rl)
    return {"T0": Tr * TC, "rho_v": rv, "rho_l": rl, "p_s": ps, "cs2": cs2, "c": math.sqrt(3 * cs2)}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _fields(layout, nx, ny, s, seed, gen, radius=None):
    """(rho, u_x, u_y, T) on the GPU: the layout's phases with tanh edges of
    width 4, a smooth flow and seeded noise, so that every term acts."""
    rng = np.random.default_rng(seed)
    y, x = torch.meshgrid(torch.arange(ny, dtype=torch.float64, device="cuda"),
                          torch.arange(nx, dtype=torch.float64, device="cuda"), indexing="ij")
    if layout == "slab":
        liq = 0.5 * (torch.tanh(0.5 * (x - nx / 4)) - torch.tanh(0.5 * (x - 3 * nx / 4)))
    elif layout == "boiling":
        liq = 0.5 * (1 - torch.tanh(0.5 * (y - 0.75 * ny)))
    else:
        m = min(nx, ny)
        if layout == "open" or radius is not None:
            drops = [(nx / 2, ny / 2, radius or m / 8)]
        else:
            drops = [(rng.uniform(0, nx), rng.uniform(0, ny), rng.uniform(0.04, 0.12) * m) for _ in range(8)]
        liq = torch.zeros_like(x)
        for cx, cy, r in drops:
            dx, dy = (x - cx).abs() % nx, (y - cy).abs() % ny
            dx, dy = torch.minimum(dx, nx - dx), torch.minimum(dy, ny - dy)
            liq = torch.maximum(liq, 0.5 * (1 - torch.tanh(0.5 * ((dx * dx + dy * dy).sqrt() - r))))

    def noise():
        return 2 * torch.rand((ny, nx), dtype=torch.float64, device="cuda", generator=gen) - 1

    a, b = rng.uniform(0, 2 * math.pi, 2)
    rho = (s["rho_v"] + (s["rho_l"] - s["rho_v"]) * liq) * (1 + 0.005 * noise())
    ux = 0.004 * s["c"] * (torch.sin(2 * math.pi * y / ny + a) + 0.2 * noise())
    uy = 0.004 * s["c"] * (torch.sin(2 * math.pi * x / nx + b) + 0.2 * noise())
    T = s["T0"] * (1 + 0.005 * noise())
    return torch.stack([rho, ux, uy, T])


def _options(case, seed):
    """Boundary options of a lattice case."""
    if case["layout"] == "boiling":
        return {"walls": 1, "accel_y": -1e-5, "Tr_bottom": 0.8, "Tr_hot": 0.95, "hot_len": HOT_LEN,
                "hot_x0": int(np.random.default_rng(seed).integers(0, case["nx"] - HOT_LEN + 1))}
    if case["layout"] == "open":
        return {"walls": 1, "open_sides": 15, "Tr_open": 0.85}
    return {}


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _plan(case):
    """(nx, ny, radius, reduced temperature) of every box of a batch: sides log-uniform, one droplet each."""
    rng = np.random.default_rng(case["plan"])
    m, out = case["multiple"], []
    for _ in range(case["cases"]):
        side = [int(min(max(round(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]))) / m) * m, case["lo"]), case["hi"]))
                for _ in range(2)]
        out.append((*side, float(rng.uniform(8, 0.3 * min(side))), round(float(rng.uniform(0.7, 0.95)), 2)))
    return out


def _batch_fields(case, seed):
    gen = _generator(seed)
    return [_fields("droplets", nx, ny, _scales(tr), seed, gen, radius=r) for nx, ny, r, tr in _plan(case)]


def _weights(seed):
    """[(9, cout, cin) weights, biases] of lift, 2 x BLOCKS block layers and projection."""
    rng = np.random.default_rng(seed + 77)
    shapes = [(4, CH, 1.0)] + [(CH, CH, 1.0 if k % 2 == 0 else 0.1) for k in range(2 * BLOCKS)] + [(CH, 4, 0.1)]
    return [((rng.standard_normal((9, co, ci)) * s * math.sqrt(2 / (9 * ci))).astype(np.float32),
             (0.01 * rng.standard_normal(co)).astype(np.float32)) for ci, co, s in shapes]


def _norm():
    s = _scales(0.8)
    return [s["rho_v"], 0.0, 0.0, s["T0"]], [s["rho_l"] - s["rho_v"], 0.01 * s["c"], 0.01 * s["c"], 0.1 * TC]


def _images(case, seed):
    """Droplet fields and, for training, the fields after a small smooth change."""
    gen = _generator(seed)
    x = torch.stack([_fields("droplets", case["w"], case["h"], _scales(0.8), seed + 1000 * k, gen) for k in range(case["n"])], 1).contiguous()
    scale = torch.tensor(_norm()[1], dtype=torch.float64, device="cuda").view(4, 1, 1, 1)
    t = x + 0.02 * scale * torch.randn(x.shape, dtype=torch.float64, device="cuda", generator=gen)
    return x, t


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        s = _scales(0.8)
        fields = _fields(case["layout"], case["nx"], case["ny"], s, seed, _generator(seed))
        lat = lbm.Lattice(lbm.default_config(case["nx"], case["ny"], precision=case["precision"], **_options(case, seed)))
        out = torch.empty_like(fields)
        return {"kind": kind, "lat": lat, "steps": case["steps"], "fields": fields, "out": out,
                "views": dict(zip(("rho", "ux", "uy", "T"), out)), "dtype": DTYPE[case["precision"]]}
    if kind == "batch":
        b = lbm.Batch([lbm.default_config(nx, ny, precision=case["precision"], Tr0=tr, **SWEEP) for nx, ny, _, tr in _plan(case)])
        fields = _batch_fields(case, seed)
        out = torch.empty(sum(f.numel() for f in fields), dtype=torch.float64, device="cuda")
        at = np.cumsum([0] + [f.numel() for f in fields])
        return {"kind": kind, "batch": b, "steps": case["steps"], "fields": fields, "out": out,
                "views": [out[a:a + f.numel()].view(f.shape) for a, f in zip(at, fields)], "dtype": DTYPE[case["precision"]]}
    off, scale = _norm()
    sur = lbm.Surrogate(off, scale, K=50, channels=CH, blocks=BLOCKS)
    sur.set_params(np.concatenate([a.reshape(-1) for wb in _weights(seed) for a in wb]))
    x, t = _images(case, seed)
    return {"kind": kind, "sur": sur, "x": x, "t": t, "out": torch.empty_like(x)}


_DP = ctypes.POINTER(ctypes.c_double)


def _ptrs(planes):
    return [ctypes.cast(ctypes.c_void_p(p.data_ptr()), _DP) for p in planes]


def run(state):
    kind = state["kind"]
    if kind == "lattice":
        lat = state["lat"]
        lat.set_fields(*state["fields"])
        lat.step(state["steps"])
        lat.moments(out=state["views"])
        return {"fields": state["out"].to(state["dtype"])}
    if kind == "batch":
        # the batch's fields live on the GPU: the C calls take device pointers
        b = state["batch"]
        torch.cuda.current_stream().synchronize()
        for i, f in enumerate(state["fields"]):
            lbm._check(b.lib.lbm_batch_set_fields(b.h, i, *_ptrs(f), 1))
        b.step(state["steps"])
        for i, f in enumerate(state["views"]):
            lbm._check(b.lib.lbm_batch_moments(b.h, i, *_ptrs(f), 1))
        return {"fields": state["out"].to(state["dtype"])}
    if kind == "forward":
        return {"fields": state["sur"].forward(state["x"], state["out"])}
    if kind == "train":
        loss = state["sur"].train_step(state["x"], state["t"], 1e-4)
        return {"loss": np.float32(loss), "params": state["sur"].get_params()}
    loss, grads = state["sur"].loss_grad(state["x"], state["t"])
    return {"loss": np.float32(loss), "grads": grads}


# floating-point operations of one node update, counted over its formulas:
# two moment transforms and their inverses, pair force, EOS, both collisions
NODE_FLOPS = 450


def work(case):
    kind = case["kind"]
    if kind in ("lattice", "batch"):
        nodes = case["nx"] * case["ny"] if kind == "lattice" else sum(nx * ny for nx, ny, _, _ in _plan(case))
        # 18 populations read and written per step, four fields in and out
        return {"bytes": nodes * (case["steps"] * 36 * SIZE[case["precision"]] + 64), "flops": nodes * case["steps"] * NODE_FLOPS}
    P = case["n"] * case["h"] * case["w"]
    nw = 9 * (8 * CH + 2 * BLOCKS * CH * CH)
    if kind == "forward":
        return {"bytes": 64 * P + 4 * nw, "flops": 2 * nw * P}
    return {"bytes": 64 * P + (24 if kind == "train" else 8) * nw, "flops": 6 * nw * P}


# ---------------------------------------------------------------------------
# The same in 64 bits with plain torch
# ---------------------------------------------------------------------------
EX, EY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
M = [[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
     [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1],
     [0, 0, 1, 0, -1, 1, 1, -1, -1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
     [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]]


class _Model:
    """One lattice of the double-distribution model in float64: default
    constants (s_p = s_eps = sigma_e = 1, gamma = (-2, 2), tau_j 0.25 / 2.5,
    c_v = 1.5 R, C_ref = rho_v c_v) at reduced temperature Tr."""

    def __init__(self, Tr, opt, sig_eps=1.0, sig_p=1.0):
        s = _scales(Tr)
        self.s, self.opt, self.sig_eps, self.sig_p = s, opt, sig_eps, sig_p
        self.c, self.dt = s["c"], 1 / s["c"]
        self.G2 = K_INT**2 * 2 * K_EOS
        self.a = self.G2 / 2
        self.cv = 1.5
        self.Cref = s["rho_v"] * self.cv
        self.beta = -2 / (1 - VARPI)
        kS = 1 - VARPI
        self.hS, self.bS, self.kS = 6 * VARPI * (1 - VARPI) / (1 - 3 * VARPI), (1 - VARPI) / (1 - 3 * VARPI), kS
        self.sq, self.se = 1 / (1 / 6 + 0.5), 1 / (0.5 / (kS + 1) + 0.5)
        self.M = torch.tensor(M, dtype=torch.float64, device="cuda")
        self.Mi = torch.linalg.inv(self.M.cpu()).cuda()
        self.walls, self.open = opt.get("walls", 0), opt.get("open_sides", 0)
        self.T_open = opt.get("Tr_open", 0.0) * TC
        if self.open:
            hi = next((k / 4000.0 for k in range(1, 4000) if _dp(k / 4000.0, self.T_open) < 0), 0.9999)
            hi = _bisect(lambda r: _dp(r, self.T_open), 1e-9, hi)
            self.rho_open = _bisect(lambda r: _p(r, self.T_open) - s["p_s"], 1e-12, hi)

    def mul(self, A, v):
        return (A @ v.reshape(9, -1)).view_as(v)

    def pad(self, v, edge_x, edge_y):
        """v with one more node on each side; edge_x, edge_y(row or column of v, side) where not periodic."""
        v = torch.cat([edge_x(0), v, edge_x(-1)], 1) if edge_x else torch.cat([v[:, -1:], v, v[:, :1]], 1)
        return torch.cat([edge_y(v, 0), v, edge_y(v, -1)], 0) if edge_y else torch.cat([v[-1:], v, v[:1]], 0)

    def force(self, rho):
        """Pair force over c and grad rho."""
        if self.open:
            full = lambda n, m: torch.full((n, m), self.rho_open, dtype=rho.dtype, device=rho.device)  # noqa: E731
            r = self.pad(rho, lambda k: full(rho.shape[0], 1), lambda v, k: full(1, v.shape[1]))
        elif self.walls:
            r = self.pad(rho, None, lambda v, k: v[:1] if k == 0 else v[-1:])
        else:
            r = self.pad(rho, None, None)
        ny, nx = rho.shape
        gx, gy = torch.zeros_like(rho), torch.zeros_like(rho)
        for i in range(1, 9):
            n = r[1 + EY[i]:1 + EY[i] + ny, 1 + EX[i]:1 + EX[i] + nx] * (1 / 3 if i <= 4 else 1 / 12)
            gx += n * EX[i]
            gy += n * EY[i]
        k = self.G2 / self.c
        ax, ay = self.opt.get("accel_x", 0.0) / self.c, self.opt.get("accel_y", 0.0) / self.c
        return rho * (k * gx + ax), rho * (k * gy + ay), gx, gy

    def p_be(self, rho, T):
        return K_EOS * (rho * T * (1 + rho + rho * rho - rho**3) / (1 - rho) ** 3 - rho * rho) + self.a * rho * rho

    def equilibria(self, rho, ux, uy, T, rek):
        pbe = self.p_be(rho, T)
        eta, rhk, u2 = pbe / self.s["cs2"] - rho, rek + pbe, ux * ux + uy * uy
        jx, jy, CT, z = rho * ux, rho * uy, self.Cref * T, torch.zeros_like(rho)
        meq = torch.stack([rho, -2 * rho + 2 * eta + 3 * rho * u2, rho + self.beta * eta - 3 * rho * u2,
                           jx, -jx, jy, -jy, jx * ux - jy * uy, jx * uy])
        neq = torch.stack([rek, -4 * rek + 2 * CT, 4 * rek - 2 * CT, rhk * ux, -rhk * ux, rhk * uy, -rhk * uy, z, z])
        return meq, neq

    def sources(self, Fx, Fy, ux, uy, q):
        FU, z = Fx * ux + Fy * uy, torch.zeros_like(q)
        Fm = torch.stack([z, 6 * FU, -6 * FU, Fx, -Fx, Fy, -Fy, 2 * (Fx * ux - Fy * uy), Fx * uy + Fy * ux])
        qm = torch.stack([q, -2 * q, 2 * q, q * ux, -q * ux, q * uy, -q * uy, z, z])
        return Fm, qm

    def init(self, rho, vx, vy, T):
        Fx, Fy, _, _ = self.force(rho)
        ux, uy = vx / self.c, vy / self.c
        q = self.c**2 * (Fx * ux + Fy * uy)
        rek = rho * self.cv * T + 0.5 * rho * (vx * vx + vy * vy)
        meq, neq = self.equilibria(rho, ux, uy, T, rek)
        Fm, qm = self.sources(Fx, Fy, ux, uy, q)
        return self.mul(self.Mi, meq - 0.5 * self.dt * Fm), self.mul(self.Mi, neq - 0.5 * self.dt * qm)

    def macro(self, m, n0):
        rho = m[0]
        Fx, Fy, gx, gy = self.force(rho)
        ux, uy = (m[3] + 0.5 * self.dt * Fx) / rho, (m[5] + 0.5 * self.dt * Fy) / rho
        q = self.c**2 * (Fx * ux + Fy * uy)
        rek = n0 + 0.5 * self.dt * q
        T = (rek / rho - 0.5 * self.c**2 * (ux * ux + uy * uy)) / self.cv
        return rho, Fx, Fy, gx, gy, ux, uy, q, rek, T

    def step(self, f, g):
        dt, c2, s = self.dt, self.c**2, self.s
        m, n = self.mul(self.M, f), self.mul(self.M, g)
        rho, Fx, Fy, gx, gy, ux, uy, q, rek, T = self.macro(m, n[0])
        meq, neq = self.equilibria(rho, ux, uy, T, rek)
        Fm, qm = self.sources(Fx, Fy, ux, uy, q)
        qc = self.G2 * dt * dt / 12
        w = m - meq + 0.5 * dt * Fm
        w[1] -= 6 * qc * (gx * gx + gy * gy)
        w[2] += 6 * qc * (gx * gx + gy * gy)
        w[7] -= qc * (gx * gx - gy * gy)
        w[8] -= qc * gx * gy
        we, wp, sq = self.se / 2 - 1, -0.5, self.sq
        mb = m + dt * Fm
        mb[1] -= self.se * w[1] + self.kS * we * w[2] + self.hS * sq * we * (ux * w[4] + uy * w[6])
        mb[2] -= w[2]
        mb[4] -= sq * w[4]
        mb[6] -= sq * w[6]
        mb[7] -= w[7] + 2 * self.bS * sq * wp * (ux * w[4] - uy * w[6])
        mb[8] -= w[8] + self.bS * sq * wp * (uy * w[4] + ux * w[6])
        d = 0.5 * (m + mb) - meq
        z = n - neq + 0.5 * dt * qm
        wl = ((rho - s["rho_v"]) / (s["rho_l"] - s["rho_v"])).clamp(0, 1)
        sj = 1 / (0.25 + 2.25 * wl + 0.5)
        wj = sj * (0.5 * sj - 1)
        yx = c2 * (ux * d[1] / 3 + ux * d[7] + 2 * uy * d[8])
        yy = c2 * (uy * d[1] / 3 - uy * d[7] + 2 * ux * d[8])
        nb = n + dt * qm
        nb[1] -= z[1]
        nb[2] -= self.sig_eps * z[2]
        nb[3] += yx - sj * z[3] - wj * z[4]
        nb[4] -= yx + sj * z[4]
        nb[5] += yy - sj * z[5] - wj * z[6]
        nb[6] -= yy + sj * z[6]
        nb[7] -= self.sig_p * z[7]
        nb[8] -= self.sig_p * z[8]
        fb, gb = self.mul(self.Mi, mb), self.mul(self.Mi, nb)
        fo = go = None
        if self.open:
            # beyond the open sides: the nearest node's populations with their equilibrium moved to the open state
            r0, T0 = torch.full_like(rho, self.rho_open), torch.full_like(rho, self.T_open)
            moved = []
            for r, t in ((rho, T), (r0, T0)):
                moved.append(self.equilibria(r, ux, uy, t, r * self.cv * t + 0.5 * c2 * r * (ux * ux + uy * uy)))
            fo, go = (b + self.mul(self.Mi, moved[1][k] - moved[0][k]) for k, b in ((0, fb), (1, gb)))
        return self.stream(fb, fo), self.walls_g(rho, gb, self.stream(gb, go))

    def stream(self, b, o):
        ny, nx = b.shape[1:]
        out = torch.empty_like(b)
        for i in range(9):
            if o is not None:
                q = o[i]
                ext = torch.cat([q[:, :1], q, q[:, -1:]], 1)
                v = self.pad(b[i], lambda k: q[:, :1] if k == 0 else q[:, -1:], lambda v, k: ext[:1] if k == 0 else ext[-1:])
            else:
                v = self.pad(b[i], None, None)
            out[i] = v[1 - EY[i]:1 - EY[i] + ny, 1 - EX[i]:1 - EX[i] + nx]
        if self.walls and o is None:
            for i, k in ((4, 2), (7, 5), (8, 6)):
                out[k][0] = b[i][0]
                out[i][-1] = b[k][-1]
        return out

    def walls_g(self, rho, b, out):
        if not self.walls or self.open:
            return out
        nx = rho.shape[1]
        x = torch.arange(nx, device="cuda")
        Tw = torch.full((nx,), self.opt["Tr_bottom"] * TC, dtype=torch.float64, device="cuda")
        Tw[(x - self.opt["hot_x0"]) % nx < self.opt["hot_len"]] = self.opt["Tr_hot"] * TC
        for i, k in ((4, 2), (7, 5), (8, 6)):
            t = torch.roll(Tw, -EX[i])
            E, CT = rho[0] * self.cv * t, self.Cref * t
            n1, n2 = -4 * E + 2 * CT, 4 * E - 2 * CT
            ge = E / 9 - n1 / 36 - 2 * n2 / 36 if i == 4 else E / 9 + 2 * n1 / 36 + n2 / 36
            out[k][0] = 2 * ge - b[i][0]
        return out

    def fields(self, f, g):
        rho, _, _, _, _, ux, uy, _, _, T = self.macro(self.mul(self.M, f), g.sum(0))
        return torch.stack([rho, ux * self.c, uy * self.c, T])


def _advance(model, fields, steps):
    f, g = model.init(*fields)
    for _ in range(steps):
        f, g = model.step(f, g)
    return model.fields(f, g)


def _conv(x, w, b):
    """3 x 3 periodic convolution, x (N, H, W, cin), tap 3 (dy + 1) + dx + 1 reads pixel (y + dy, x + dx)."""
    out = b.expand(*x.shape[:3], -1)
    for t in range(9):
        out = out + torch.roll(x, (1 - t // 3, 1 - t % 3), (1, 2)) @ w[t].T
    return out


def _network(x, weights):
    h = _conv(x, *weights[0])
    for k in range(BLOCKS):
        h = h + _conv(_conv(h.relu(), *weights[1 + 2 * k]).relu(), *weights[2 + 2 * k])
    y = x + _conv(h.relu(), *weights[-1])
    shift = (y[..., :1] - x[..., :1]).mean((1, 2), keepdim=True)
    return torch.cat([y[..., :1] - shift, y[..., 1:]], -1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        fields = _fields(case["layout"], case["nx"], case["ny"], _scales(0.8), seed, _generator(seed))
        return {"fields": _advance(_Model(0.8, _options(case, seed)), fields, case["steps"])}
    if kind == "batch":
        if case["cases"] * case["steps"] > 2500:
            return None  # small boxes one after another would take minutes
        out = []
        for f, (_, _, _, tr) in zip(_batch_fields(case, seed), _plan(case)):
            out.append(_advance(_Model(tr, {}, sig_eps=SWEEP["sig_eps"], sig_p=SWEEP["sig_p"]), f, case["steps"]).reshape(-1))
        return {"fields": torch.cat(out)}
    off, scale = (torch.tensor(v, dtype=torch.float64, device="cuda") for v in _norm())
    x, t = (((v.permute(1, 2, 3, 0) - off) / scale).contiguous() for v in _images(case, seed))
    weights = [[torch.tensor(a, dtype=torch.float64, device="cuda") for a in wb] for wb in _weights(seed)]
    if kind == "forward":
        with torch.no_grad():
            y = _network(x, weights)
        return {"fields": (off + y * scale).permute(3, 0, 1, 2).contiguous()}
    flat = [a.requires_grad_() for wb in weights for a in wb]
    loss = (_network(x, weights) - t).square().mean()
    grads = torch.autograd.grad(loss, flat)
    if kind == "grad":
        return {"loss": loss.detach(), "grads": torch.cat([v.reshape(-1) for v in grads])}
    # the first Adam step: lr g / (|g| + eps)
    new = torch.cat([(a.detach() - 1e-4 * v / (v.abs() + 1e-8)).reshape(-1) for a, v in zip(flat, grads)])
    return {"loss": loss.detach(), "params": new}

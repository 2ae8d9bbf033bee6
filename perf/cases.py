"""Cases that time this framework the way a program uses it: through the
public classes of ``paper_1806_10247_gb300.lbm`` and ``.surrogate``.

One pass advances a lattice (or a batch of lattices) by a number of time steps
and reads its macroscopic fields, or trains the warm-start network for one
iteration.  A lattice lives on between passes, as it does in a program's time
loop.  Fields of FP64 lattices come back as the library writes them (FP64);
those of the reduced-precision storages as single-precision snapshots, which
is what such a run keeps.

``exact`` restates the method in plain 64-bit torch: the cascaded
central-moment collision with Strang-split force or source on D2Q9, D3Q27,
D3Q15 and D2Q5, streaming with periodic wrap or halfway bounce-back, and the
network's training iteration.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1806_10247_gb300 import lbm, surrogate
from paper_1806_10247_gb300 import workloads as W

STORAGE = {"fp64": lbm.FP64, "fp32": lbm.FP32_DEV, "fp16": lbm.FP16_DEV, "bf16": lbm.BF16_DEV}
ELEM = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
Q = {"d2q9": 9, "d3q27": 27, "d2q5": 5, "d3q15": 15}
# floating-point operations of one node's step (a multiply-add counts two)
FLOPS = {"d2q9": 98, "d3q27": 325, "d2q5": 55, "d3q15": 280}


# ------------------------------------------------------------------- cases ---

def listed():
    return [
        # The channel of the convergence study: 99 nodes, stepped 100 at a time
        # between convergence checks.  The smallest call: latency counts.
        {"name": "poiseuille_fp64", "kind": "channel", "nx": 3, "ny": 33, "storage": "fp64", "steps": 100,
         "check": True},
        # The paper's D3Q15 duct (3 x 45 x 45), 50 steps at a time.
        {"name": "duct15_fp64", "kind": "duct15", "nx": 3, "n": 45, "steps": 50},
        # The scalar refinement sweep (32^2 .. 512^2) as one batch.
        {"name": "scalar_sweep_fp64", "kind": "scalar_sweep", "largest": 512, "storage": "fp64", "steps": 20},
        # A plane channel of ordinary size in FP64, and a large one in FP32.
        {"name": "channel_fp64", "kind": "channel", "nx": 2048, "ny": 1024, "storage": "fp64", "steps": 10,
         "check": False},
        {"name": "channel_fp32", "kind": "channel", "nx": 8192, "ny": 4096, "storage": "fp32", "steps": 10,
         "check": False},
        # A large scalar field in 16 bits at a per-node reference, rounded
        # stochastically: the 16-bit form that keeps second order.
        {"name": "scalar_fp16", "kind": "scalar", "nx": 8192, "ny": 8192, "storage": "fp16", "reference": 16,
         "stochastic": True, "steps": 16},
        # The parameter sweep of many small lattices of uneven size: channels
        # and scalars, one launch per step and kind under a CUDA graph.
        {"name": "batched_sweep_fp32", "kind": "sweep", "count": 192, "sizes": 10247, "storage": "fp32",
         "steps": 20},
        # Kolmogorov flow in 3D: the FP64 reference run, single precision on a
        # grid far larger than L2, and plain 16-bit storage.
        {"name": "kolmogorov_fp64", "kind": "kolmogorov", "nx": 256, "ny": 256, "nz": 256, "storage": "fp64",
         "steps": 4},
        {"name": "kolmogorov_fp32", "kind": "kolmogorov", "nx": 384, "ny": 384, "nz": 384, "storage": "fp32",
         "steps": 8},
        {"name": "kolmogorov_fp16", "kind": "kolmogorov", "nx": 256, "ny": 256, "nz": 256, "storage": "fp16",
         "steps": 8},
        # Duct sections iterated to a residual (training fields and warm
        # starts): 100 steps of a small batch, then every field on the host.
        {"name": "duct_sections_fp64", "kind": "sections", "n": 128, "count": 8, "storage": "fp64", "steps": 100},
        # One training iteration of the warm-start network at 128^2 sections.
        {"name": "surrogate_train", "kind": "train", "n": 128, "batch": 32},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["channel", "channel", "scalar", "scalar", "kolmogorov", "kolmogorov", "duct15", "sections",
                       "sweep", "scalar_sweep", "train"])
    storage = rng.choice(["fp64", "fp32", "fp16", "bf16"])
    if kind == "channel":
        # from a few nodes to 4096 x 4096, of any aspect
        nx, ny = _log_int(rng, 3, 4096), _log_int(rng, 9, 4096)
        return {"kind": kind, "nx": nx, "ny": ny, "storage": storage, "steps": rng.randint(5, 60 if nx * ny < 65536
                else 12), "check": rng.random() < 0.3}
    if kind == "scalar":
        nx, ny = _log_int(rng, 32, 6000), _log_int(rng, 32, 6000)
        c = {"kind": kind, "nx": nx, "ny": ny, "storage": storage, "reference": 0, "stochastic": False,
             "steps": rng.randint(5, 16)}
        if ELEM[storage] == 2 and rng.random() < 0.5:
            c["reference"], c["stochastic"] = rng.randint(4, 16), rng.random() < 0.7
        return c
    if kind == "kolmogorov":
        s = [_log_int(rng, 12, 288) for _ in range(3)]
        return {"kind": kind, "nx": s[0], "ny": s[1], "nz": s[2], "storage": storage, "steps": rng.randint(2, 8)}
    if kind == "duct15":
        return {"kind": kind, "nx": rng.choice([1, 3, 5, 32]), "n": rng.randint(9, 128), "steps": rng.randint(5, 60)}
    if kind == "sections":
        return {"kind": kind, "n": rng.randint(24, 128), "count": rng.randint(2, 12),
                "storage": rng.choice(["fp64", "fp64", "fp32"]), "steps": rng.randint(20, 100)}
    if kind == "sweep":
        return {"kind": kind, "count": _log_int(rng, 4, 160), "sizes": rng.randrange(1 << 20), "storage":
                rng.choice(["fp64", "fp32", "fp32"]), "steps": 2 * rng.randint(3, 10)}
    if kind == "scalar_sweep":
        return {"kind": kind, "largest": rng.choice([64, 128, 256, 512, 1024]),
                "storage": rng.choice(["fp64", "fp32"]), "steps": rng.randint(5, 30)}
    return {"kind": kind, "n": rng.randint(24, 128), "batch": rng.randint(1, 32)}


# ------------------------------------------------------------------ inputs ---

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _noise(seed, shape, amp):
    return (amp * torch.randn(shape, dtype=torch.float64, device="cuda", generator=_gen(seed))).cpu().numpy()


ONE, ZERO = np.array([1.0]), np.array([0.0])


def _channel_workload(nx, ny, rng, u0):
    tau = float(rng.uniform(0.55, 1.5))
    nu = (tau - 0.5) / 3.0
    # the centre line stays below Mach 0.3, as in the parameter sweep
    F = min(float(10.0 ** rng.uniform(-7.0, -5.0)), 0.17 * 8.0 * nu / (ny * ny))
    return W.Workload(name="channel", lattice=W.D2Q9, shape=(nx, ny, 1), wall=(0, 1, 0), omega=W.d2q9_omega(tau),
                      rho0=1.0, u0=u0, tables=[(np.array([F]), ONE, ONE), (ZERO, ONE, ONE)])


def _scalar_workload(nx, ny, rng, phi0):
    A = float(10.0 ** rng.uniform(-5.0, -3.0))
    x, y = np.arange(nx, dtype=np.float64), np.arange(ny, dtype=np.float64)
    tau = float(rng.uniform(0.53, 0.8))
    return W.Workload(name="scalar", lattice=W.D2Q5, shape=(nx, ny, 1), wall=(0, 0, 0), omega=W.d2q5_omega(tau),
                      rho0=phi0, u0=(0.01, 0.01, 0.0),
                      tables=[(A * np.sin(2.0 * np.pi * x / nx), np.sin(2.0 * np.pi * y / ny), ONE)])


def _workloads(case, seed):
    """The lattices of a case, made from the seed: a list of groups that are
    stepped together."""
    rng = np.random.default_rng([seed, 11])
    kind = case["kind"]
    if kind == "channel":
        nx, ny = case["nx"], case["ny"]
        return [[_channel_workload(nx, ny, rng, _noise(seed, (2, nx * ny), 1e-3))]]
    if kind == "scalar":
        nx, ny = case["nx"], case["ny"]
        return [[_scalar_workload(nx, ny, rng, 1.0 + _noise(seed, (nx * ny,), 1e-2))]]
    if kind == "scalar_sweep":
        sizes, n = [], 32
        while n <= case["largest"]:
            sizes.append(n)
            n *= 2
        ws = []
        for k, c in enumerate(W.cde_sweep_params(seed=seed, sizes=tuple(sizes))):
            w = W.cde_workload(c)
            w.envelope = None
            w.rho0 = 1.0 + _noise(seed + k, (c.N * c.N,), 1e-3)
            ws.append(w)
        return [ws]
    if kind == "sweep":
        channels, scalars = W.batched_sweep(count=case["count"], seed=case["sizes"])
        for w in channels + scalars:  # each amplitude between half and all of the sweep's own
            px, py, pz = w.tables[0]
            w.tables[0] = (px * rng.uniform(0.5, 1.0), py, pz)
        return [channels, scalars]
    if kind == "kolmogorov":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        py = 1e-5 * np.sin(2.0 * np.pi * np.arange(ny) / ny)
        w = W.Workload(name="kolmogorov", lattice=W.D3Q27, shape=(nx, ny, nz), wall=(0, 0, 0),
                       omega=W.d3q27_omega(W.tau_from_nu(0.02)), rho0=1.0, u0=_noise(seed, (3, nx * ny * nz), 1e-4),
                       tables=[(ONE, py, ONE), (ZERO, ONE, ONE), (ZERO, ONE, ONE)])
        return [[w]]
    if kind == "duct15":
        w = W.duct15(n=case["n"], nx=case["nx"], F0=float(10.0 ** rng.uniform(-7.0, -6.0)))
        w.u0 = _noise(seed, (3, w.nodes), 1e-3)
        return [[w]]
    if kind == "sections":
        ws = []
        for k, (F0, nu) in enumerate(surrogate.draw_params(case["count"], case["n"], seed)):
            w = surrogate.section(case["n"], F0, nu)
            w.u0 = _noise(seed + k, (3, w.nodes), 1e-3)
            ws.append(w)
        return [ws]
    raise ValueError(kind)


def _training_pairs(case, seed):
    """Minibatch of duct sections: features and a field of the steady flow's
    shape (a few modes of the section, scaled as the targets are)."""
    n, batch = case["n"], case["batch"]
    rng = np.random.default_rng([seed, 12])
    X = np.stack([surrogate.features(n, float(rng.uniform(0.01, 0.1))) for _ in range(batch)]).astype(np.float32)
    y = (np.arange(n) + 0.5) / n
    modes = [np.sin((k + 1) * np.pi * y) for k in range(3)]
    Y = np.empty((batch, 1, 1, n, n), dtype=np.float32)
    for s in range(batch):
        c = rng.uniform(-0.01, 0.01, (3, 3))
        c[0, 0] = rng.uniform(0.05, 0.09)
        Y[s, 0, 0] = sum(c[i, j] * np.outer(modes[i], modes[j]) for i in range(3) for j in range(3))
    return torch.tensor(X, device="cuda"), torch.tensor(Y, device="cuda")


# ----------------------------------------------------------------- measure ---

def _lattice(w, case):
    """What lbm.from_workload sets up, for a start with both phi and u."""
    storage = STORAGE[case.get("storage", "fp64")]
    L = lbm.from_workload(w, storage=storage)
    if case.get("reference"):
        L.set_local_reference(case["reference"])
    if case.get("stochastic"):
        L.set_stochastic_rounding(True, seed=10247)
    return L


def prepare(case, seed):
    if case["kind"] == "train":
        X, Y = _training_pairs(case, seed)
        return {"case": case, "net": surrogate.ConvNet(seed=seed), "X": X, "Y": Y}
    groups = _workloads(case, seed)
    s = {"case": case, "groups": []}
    for ws in groups:
        lats = [_lattice(w, case) for w in ws]
        nodes = sum(w.nodes for w in ws)
        dim = lats[0].dim
        g = {"lats": lats, "batch": None,
             "rho": torch.empty(nodes, dtype=torch.float64, device="cuda"),
             "u": None if ws[0].lattice == W.D2Q5 else torch.empty(dim * nodes, dtype=torch.float64, device="cuda")}
        if case["kind"] in ("sweep", "scalar_sweep", "sections"):
            g["batch"] = lbm.Batch(lats)
            if case["kind"] == "sweep":
                g["batch"].autotune(5)
                g["batch"].set_graph(case["steps"])
        s["groups"].append(g)
    if case.get("check"):
        s["groups"][0]["lats"][0].reduce()
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "train":
        loss, grads = s["net"].loss_and_grads(s["X"], s["Y"])
        s["net"].adam_step(grads)
        return {"loss": loss, "grads": grads, "weights": s["net"].W, "biases": s["net"].B}
    out = []
    n = case["steps"]
    single = case.get("storage", "fp64") != "fp64"
    for g in s["groups"]:
        if g["batch"] is not None:
            g["batch"].step(n)
        else:
            g["lats"][0].step(n)
    for g in s["groups"]:
        if case["kind"] == "sections":
            out.append(g["batch"].moments_packed())  # on the host, as the residual check takes them
            continue
        if g["batch"] is not None:
            g["batch"].moments_packed_into(g["rho"].data_ptr(), None if g["u"] is None else g["u"].data_ptr(), where=1)
        else:
            g["lats"][0].moments(out=(g["rho"], g["u"]), where=1)
        rho, u = g["rho"], g["u"]
        out.append((rho.float(), None if u is None else u.float()) if single else (rho, u))
    if case.get("check"):
        return {"fields": out, "sums": s["groups"][0]["lats"][0].reduce()}
    return out


def _sizes(case):
    """(lattice, nodes) of every lattice of a case."""
    kind = case["kind"]
    if kind == "channel":
        return [("d2q9", case["nx"] * case["ny"])]
    if kind == "scalar":
        return [("d2q5", case["nx"] * case["ny"])]
    if kind == "kolmogorov":
        return [("d3q27", case["nx"] * case["ny"] * case["nz"])]
    if kind == "duct15":
        return [("d3q15", case["nx"] * case["n"] ** 2)]
    if kind == "sections":
        return [("d3q27", case["n"] ** 2)] * case["count"]
    if kind == "scalar_sweep":
        return [("d2q5", 4 ** k) for k in range(5, 12) if 2 ** k <= case["largest"]]
    groups = W.batched_sweep(count=case["count"], seed=case["sizes"])
    return [(q, w.nodes) for q, ws in zip(("d2q9", "d2q5"), groups) for w in ws]


def work(case):
    """The state read once and written once, the fields written; the
    arithmetic of every step.  Training: each activation and its gradient
    written and read once, three products per layer."""
    if case["kind"] == "train":
        pix = case["batch"] * case["n"] ** 2
        layers = surrogate.DEFAULT_LAYERS
        macs = sum(ci * co * k[0] * k[1] * k[2] for ci, co, k, _, _ in layers)
        channels = sum(co for _, co, _, _, _ in layers)
        return {"bytes": pix * 4 * (layers[0][0] + 1 + 4 * channels), "flops": pix * 6 * macs}
    elem = ELEM[case.get("storage", "fp64")]
    out = 8 if case["kind"] == "sections" or elem == 8 else 4
    byts = flops = 0
    for lat, nodes in _sizes(case):
        fields = {"d2q9": 3, "d2q5": 1}.get(lat, 4)
        byts += nodes * (2 * Q[lat] * elem + fields * out)
        flops += nodes * FLOPS[lat] * case["steps"]
    return {"bytes": byts, "flops": flops}


# ------------------------------------------------------------------- exact ---

def _field(t, shape):
    """A separable table triple as a [nz, ny, nx] tensor (broadcastable)."""
    px, py, pz = (torch.tensor(np.asarray(v), dtype=torch.float64, device="cuda") for v in t)
    return (px.view(1, 1, -1) * py.view(1, -1, 1)) * pz.view(-1, 1, 1)


def _start(w):
    nx, ny, nz = w.shape
    shape = (nz, ny, nx)
    rho = torch.as_tensor(w.rho0, dtype=torch.float64, device="cuda")
    rho = rho.expand(shape).clone() if rho.dim() == 0 else rho.view(shape)
    u = torch.as_tensor(np.asarray(w.u0), dtype=torch.float64, device="cuda")
    u = [v.expand(shape) if v.dim() == 0 else v.view(shape) for v in u]
    return rho, u


def _pull(fp, vel, wall):
    """f_a(x) = fp_a(x - e_a), or the opposite population of the same node
    where x - e_a lies beyond a wall."""
    opp = [vel.index(tuple(-c for c in e)) for e in vel]
    out = []
    for a, e in enumerate(vel):
        v = torch.roll(fp[a], shifts=(e[2], e[1], e[0]), dims=(0, 1, 2))
        for d in range(3):
            if wall[d] and e[d] != 0:
                at = [slice(None)] * 3
                at[2 - d] = 0 if e[d] == 1 else v.shape[2 - d] - 1
                v[tuple(at)] = fp[opp[a]][tuple(at)]
        out.append(v)
    return out


def _maxwell(e, u):
    s = 1.0 / 3.0 + u * u
    return 1.0 - s if e == 0 else 0.5 * (s + e * u)


class _Product:
    """D2Q9 and D3Q27 as a product lattice: moments of order 0, 1, 2 per axis."""

    def __init__(self, w):
        self.dim = 2 if w.lattice == W.D2Q9 else 3
        rng3 = (-1, 0, 1)
        self.vel = [(x, y, z) for z in (rng3 if self.dim == 3 else (0,)) for y in rng3 for x in rng3]
        om = w.omega
        if self.dim == 2:  # trace, difference, off-diagonal
            self.wb, self.wd, self.ws = om[3], om[4], om[5]
            assert om[6] == om[7] == om[8] == 1.0
        else:
            self.wb, self.wd, self.ws = om[1], om[2], om[2]
            assert om[3] == om[4] == om[5] == om[6] == 1.0

    def equilibrium(self, rho, u):
        out = []
        for e in self.vel:
            v = rho.clone()
            for d in range(self.dim):
                v = v * _maxwell(e[d], u[d])
            out.append(v)
        return out

    def first(self, f):
        rho = sum(f)
        return rho, [sum(e[d] * f[a] for a, e in enumerate(self.vel) if e[d]) for d in range(self.dim)]

    def lines(self, d):
        st = 3 ** d
        return [(p, p + st, p + 2 * st) for p in range(len(self.vel)) if (p // st) % 3 == 0]

    def collide(self, f, F):
        m, dim = list(f), self.dim
        for d in range(dim):
            for p, q, r in self.lines(d):
                lo, mid, hi = m[p], m[q], m[r]
                m[p], m[q], m[r] = lo + mid + hi, hi - lo, hi + lo
        ax = [3 ** d for d in range(dim)]
        for d in range(dim):
            m[ax[d]] = m[ax[d]] + 0.5 * F[d]
        rho = m[0]
        u = [m[ax[d]] / rho for d in range(dim)]
        k = list(m)
        for d in range(dim):
            for p, q, r in self.lines(d):
                k2 = k[r] - 2.0 * u[d] * k[q] + u[d] * u[d] * k[p]
                k1 = k[q] - u[d] * k[p]
                k[q], k[r] = k1, k2
        second = [k[2 * a] for a in ax]
        T = sum(second)
        T1 = T + self.wb * (dim / 3.0 * rho - T)
        zero = torch.zeros_like(rho)
        c = [zero] * len(m)
        c[0] = rho
        for d in range(dim):
            c[2 * ax[d]] = T1 / dim + (1.0 - self.wd) * (second[d] - T / dim)
            for d2 in range(d + 1, dim):
                c[ax[d] + ax[d2]] = (1.0 - self.ws) * k[ax[d] + ax[d2]]
                c[2 * ax[d] + 2 * ax[d2]] = rho / 9.0
        if dim == 3:
            c[26] = rho / 27.0
        for d in range(dim):
            for p, q, r in self.lines(d):
                m2 = c[r] + 2.0 * u[d] * c[q] + u[d] * u[d] * c[p]
                m1 = c[q] + u[d] * c[p]
                c[q], c[r] = m1, m2
        # post-collision half step along e_d: sum e_d^2 = 6 (D2Q9), 18 (D3Q27)
        for d in range(dim):
            g = F[d] / (6.0 if dim == 2 else 18.0)
            c[ax[d]] = c[ax[d]] + 0.5 * F[d]
            others = [ax[j] for j in range(dim) if j != d]
            for o in others:
                c[ax[d] + 2 * o] = c[ax[d] + 2 * o] + (4.0 if dim == 2 else 12.0) * g
            if dim == 3:
                c[ax[d] + 2 * sum(others)] = c[ax[d] + 2 * sum(others)] + 8.0 * g
        for d in range(dim):
            for p, q, r in self.lines(d):
                c[p], c[q], c[r] = 0.5 * (c[r] - c[q]), c[p] - c[r], 0.5 * (c[r] + c[q])
        return c


class _D3Q15:
    """D3Q15 with the paper's fifteen monomials; every rate but the shear one is 1."""

    MONO = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (2, 0, 0), (0, 2, 0),
            (0, 0, 2), (1, 2, 0), (2, 1, 0), (2, 0, 1), (1, 1, 1), (2, 2, 0)]

    def __init__(self, w):
        self.dim = 3
        self.ws = w.omega[2]
        assert w.omega[1] == w.omega[3] == w.omega[4] == 1.0
        self.vel = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)] + \
            [(x, y, z) for z in (1, -1) for y in (1, -1) for x in (1, -1)]
        M = np.array([[float(x ** a * y ** b * z ** c) for x, y, z in self.vel] for a, b, c in self.MONO])
        self.M, self.Minv = M, np.linalg.inv(M)

    @staticmethod
    def _apply(A, v):
        out = []
        for row in A:
            acc = torch.zeros_like(v[0])
            for x, t in zip(row, v):
                if abs(x) > 1e-14:
                    acc = acc + x * t
            out.append(acc)
        return out

    def _shift(self, m, u, sign):
        """Moments about sign * u from moments about 0 (binomials per axis)."""
        at = {e: i for i, e in enumerate(self.MONO)}
        out = []
        for e in self.MONO:
            acc = torch.zeros_like(m[0])
            for i in range(e[0] + 1):
                for j in range(e[1] + 1):
                    for l in range(e[2] + 1):
                        cf = math.comb(e[0], i) * math.comb(e[1], j) * math.comb(e[2], l)
                        acc = acc + cf * (sign * u[0]) ** (e[0] - i) * (sign * u[1]) ** (e[1] - j) * \
                            (sign * u[2]) ** (e[2] - l) * m[at[(i, j, l)]]
            out.append(acc)
        return out

    def _from_central(self, rho, u, second, fourth):
        c = [torch.zeros_like(rho) for _ in self.MONO]
        c[0], c[14] = rho, fourth
        for i, v in zip((7, 8, 9, 4, 5, 6), second):
            c[i] = v
        return self._shift(c, u, 1.0)

    def equilibrium(self, rho, u):
        t, z = rho / 3.0, torch.zeros_like(rho)
        return self._apply(self.Minv, self._from_central(rho, u, (t, t, t, z, z, z), rho / 9.0))

    def first(self, f):
        m = self._apply(self.M[:4], f)
        return m[0], m[1:4]

    def collide(self, f, F):
        m = self._apply(self.M, f)
        j = m[1:4]
        for d in range(3):
            m[1 + d] = m[1 + d] + 0.5 * F[d]
        rho = m[0]
        u = [m[1 + d] / rho for d in range(3)]
        k = self._shift(m, u, -1.0)
        T = k[7] + k[8] + k[9]
        dev = [(1.0 - self.ws) * (k[i] - T / 3.0) + rho / 3.0 for i in (7, 8, 9)]
        off = [(1.0 - self.ws) * k[i] for i in (4, 5, 6)]
        c = self._from_central(rho, u, dev + off, dev[0] * dev[1] / rho)
        g = [F[d] / 10.0 for d in range(3)]
        for d in range(3):
            c[1 + d] = j[d] + 10.0 * g[d]
        for i, d in ((10, 0), (11, 1), (12, 2)):
            c[i] = c[i] + 8.0 * g[d]
        return self._apply(self.Minv, c)


class _D2Q5:
    def __init__(self, w):
        self.vel = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0)]
        self.om, self.ua = w.omega, (float(w.u0[0]), float(w.u0[1]))

    def equilibrium(self, phi, u):
        t = 1.0 / 3.0
        ux, uy = self.ua
        c = [t - ux * ux - uy * uy, 0.5 * (t + ux * ux + ux), 0.5 * (t + uy * uy + uy), 0.5 * (t + ux * ux - ux),
             0.5 * (t + uy * uy - uy)]
        return [v * phi for v in c]

    def collide(self, g, S):
        ux, uy = self.ua
        om = self.om
        kx, ky, xx, yy = g[1] - g[3], g[2] - g[4], g[1] + g[3], g[2] + g[4]
        phi = g[0] + xx + yy + 0.5 * S
        # central moments about the advecting velocity and their relaxation
        cx, cy = kx - ux * phi, ky - uy * phi
        cxx = xx - 2.0 * ux * kx + ux * ux * phi
        cyy = yy - 2.0 * uy * ky + uy * uy * phi
        T, D = cxx + cyy, cxx - cyy
        cx1, cy1 = (1.0 - om[1]) * cx, (1.0 - om[2]) * cy
        T1, D1 = T + om[3] * (2.0 / 3.0 * phi - T), (1.0 - om[4]) * D
        # back; the zeroth moment of the change is 0 before the source's share
        kx1, ky1 = cx1 + ux * phi, cy1 + uy * phi
        xx1 = 0.5 * (T1 + D1) + 2.0 * ux * kx1 - ux * ux * phi
        yy1 = 0.5 * (T1 - D1) + 2.0 * uy * ky1 - uy * uy * phi
        h = S / 5.0
        return [g[0] + (xx + yy) - (xx1 + yy1) + h, 0.5 * (xx1 + kx1) + h, 0.5 * (yy1 + ky1) + h,
                0.5 * (xx1 - kx1) + h, 0.5 * (yy1 - ky1) + h]


def _exact_lattice(w, steps):
    """rho and u (or phi) of a lattice after `steps` steps, as the library lays
    them out, and the state before the last fields (for the change)."""
    rho, u = _start(w)
    scalar = w.lattice == W.D2Q5
    L = _D2Q5(w) if scalar else (_D3Q15(w) if w.lattice == W.D3Q15 else _Product(w))
    F = [_field(t, w.shape) for t in w.tables]
    f = L.equilibrium(rho, u)
    if scalar:
        for _ in range(steps):
            f = _pull(L.collide(f, F[0]), L.vel, w.wall)
        return (sum(f) + 0.5 * F[0]).reshape(-1), None, None
    for _ in range(steps):
        f = _pull(L.collide(f, F), L.vel, w.wall)
    rho, j = L.first(f)
    u = torch.stack([((j[d] + 0.5 * F[d]) / rho).reshape(-1) for d in range(L.dim)])
    total = [float(rho.sum())] + [float(v.sum()) for v in j] + [0.0] * (3 - L.dim)
    return rho.reshape(-1), u.reshape(-1), total


def _exact_train(case, seed):
    """One training iteration in 64 bits, with the network's BF16 weights."""
    X, Y = _training_pairs(case, seed)
    net = surrogate.ConvNet(seed=seed)
    w = [t.to(torch.bfloat16).double().requires_grad_(True) for t in net.W]
    b = [t.double().requires_grad_(True) for t in net.B]
    h = X[:, :, 0].double()
    for li, (ci, co, k, dil, act) in enumerate(net.layers):
        ph, pw = dil[1] * (k[1] // 2), dil[2] * (k[2] // 2)
        p = torch.nn.functional.pad(h, (pw, pw, ph, ph))
        H, V = h.shape[2:]
        y = b[li].view(1, co, 1, 1)
        for r in range(k[1]):
            for c in range(k[2]):
                part = p[:, :, r * dil[1]:r * dil[1] + H, c * dil[2]:c * dil[2] + V]
                y = y + torch.einsum("oi,nihw->nohw", w[li][:, :, 0, r, c], part)
        h = torch.tanh(y) if act == "tanh" else y
    loss = ((h - Y[:, :, 0].double()) ** 2).mean()
    loss.backward()
    grads = [(x.grad, y.grad) for x, y in zip(w, b)]
    lr, eps = 2e-3, 1e-8
    step = [[t.double() - lr * g / (g.abs() + eps) for t, g in zip(ts, gs)]  # the first Adam step
            for ts, gs in ((net.W, [g[0] for g in grads]), (net.B, [g[1] for g in grads]))]
    return {"loss": float(loss), "grads": grads, "weights": step[0], "biases": step[1]}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    out, sums = [], None
    for ws in _workloads(case, seed):
        got = [_exact_lattice(w, case["steps"]) for w in ws]
        rho = torch.cat([g[0] for g in got])
        u = None if got[0][1] is None else torch.cat([g[1] for g in got])
        sums = got[0][2]
        out.append((rho, u))
    if case.get("check"):
        return {"fields": out, "sums": None}
    return out

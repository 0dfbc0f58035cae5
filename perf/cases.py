"""The measured calls of the framework: what its users have it do, over the sizes, meshes,
precisions and options they use.

A case is a dict of plain values; ``prepare`` makes the inputs on the GPU from the seed (the
mesh, the state, the step's dt, the solver or the network), ``run`` makes one call through the
public entry points, ``exact`` restates the same call in 64-bit torch, from the same inputs."""
import math

import numpy as np
import torch

from paper_2411_14631_gb300 import abi, hydro, poisson
from paper_2411_14631_gb300 import workloads as W

DEV = "cuda:0"
GAMMA = {"sod": W.SOD_GAMMA, "turb": W.TURB_GAMMA, "plummer": W.PLUMMER_GAMMA, "sedov": W.SEDOV_GAMMA}
RIEMANN = {"hllc": abi.RIEMANN_HLLC, "exact": abi.RIEMANN_EXACT}
LIMITER = {"minmod": abi.LIMITER_MINMOD, "mc": abi.LIMITER_MC}
CFL, RHO_FLOOR, P_FLOOR = 0.8, 1e-10, 1e-20
BYTES_PER_CELL = 80          # FP64 state read and written once, five variables
FLOPS_PER_CELL = 500         # prim, slopes, predictor, three Riemann solves, update


def listed():
    return [
        # the smallest run, a shock tube on 32^3 cells, default precision, stepped by replayed
        # graphs: launches and latency count
        {"name": "sod32_fp64", "kind": "sim", "field": "sod", "level": 5, "prec": 64, "riemann": "hllc", "bc": 1},
        # the benchmark: a turbulent periodic box of 256^3 cells, FP32 reconstruction and fluxes
        {"name": "box256_fp32", "kind": "box", "field": "turb", "mach": 2.0, "level": 8, "prec": 32, "riemann": "hllc",
         "limiter": "minmod", "bc": 0},
        # the plain FP64 path (the default of Params) on an ordinary box
        {"name": "box128_fp64", "kind": "box", "field": "turb", "mach": 2.0, "level": 7, "prec": 64, "riemann": "hllc",
         "limiter": "minmod", "bc": 0},
        # the exact Riemann solver, FP32, on an ordinary box with open boundaries
        {"name": "box128_exact_fp32", "kind": "box", "field": "turb", "mach": 2.0, "level": 7, "prec": 32,
         "riemann": "exact", "limiter": "minmod", "bc": 1},
        # clumps on an adaptive mesh, five levels, one time step for all levels
        {"name": "amr_fp32", "kind": "amr", "base": 7, "lmax": 11, "clumps": 64, "thr": 1.0, "prec": 32,
         "riemann": "hllc", "limiter": "minmod", "bc": 0},
        # a smaller adaptive mesh in FP64, open boundaries
        {"name": "amr_fp64", "kind": "amr", "base": 5, "lmax": 9, "clumps": 24, "thr": 1.0, "prec": 64,
         "riemann": "hllc", "limiter": "minmod", "bc": 1},
        # sub-cycled levels: one step of the coarsest level, many launches on small levels
        {"name": "subcycled_fp32", "kind": "sub", "base": 6, "lmax": 9, "clumps": 32, "thr": 1.0, "prec": 32,
         "bc": 0},
        # blast waves in independent boxes of uneven size, one launch per step, a dt per box
        {"name": "sedov_batch_fp32", "kind": "batch", "boxes": 24, "lo": 32, "hi": 160, "mult": 16, "prec": 32,
         "riemann": "hllc"},
        # a Poisson solve to its tolerance on an uneven box
        {"name": "poisson_solve", "kind": "poisson", "nx": 180, "ny": 141, "nz": 117, "precond": 1},
        # the Riemann surrogate over a level's faces, on the tensor cores
        {"name": "mlp_infer", "kind": "infer", "n": 3200017, "tc": 1},
        # one training step of the surrogate on its ordinary batch
        {"name": "mlp_train", "kind": "train", "n": 4096},
        # refinement between steps: the new mesh and the state on it
        {"name": "amr_refine", "kind": "refine", "base": 6, "lmax": 10, "clumps": 48, "thr": 1.0, "bc": 0},
    ]


def draw(rng):
    kind = rng.choice(("box", "box", "amr", "amr", "sub", "batch", "batch", "poisson", "infer", "train", "refine"))
    if kind == "box":
        prec, riemann = rng.choice((32, 64)), rng.choice(("hllc", "hllc", "exact"))
        top = 8 if prec == 32 and riemann == "hllc" else 7 if prec == 32 else 6 if riemann == "exact" else 7
        return {"kind": "box", "field": "turb", "mach": round(rng.uniform(0.3, 4.0), 2), "level": rng.randint(4, top),
                "prec": prec, "riemann": riemann, "limiter": rng.choice(("minmod", "minmod", "mc")) if prec == 32 else "minmod",
                "bc": rng.randint(0, 1)}
    mesh = {"base": rng.randint(4, 6), "clumps": rng.randint(6, 48), "thr": rng.choice((1.0, 1.7, 3.3)),
            "bc": rng.randint(0, 1)}
    mesh["lmax"] = mesh["base"] + rng.randint(1, 4)
    if kind == "amr":
        prec = rng.choice((32, 64))
        return {"kind": "amr", "prec": prec, "riemann": rng.choice(("hllc", "hllc", "exact")) if prec == 32 else "hllc",
                "limiter": rng.choice(("minmod", "minmod", "mc")), **mesh}
    if kind == "sub":
        return {"kind": "sub", "prec": 32, **mesh}
    if kind == "refine":
        return {"kind": "refine", **mesh}
    if kind == "batch":
        prec = rng.choice((32, 32, 64))
        return {"kind": "batch", "boxes": int(round(math.exp(rng.uniform(0.0, math.log(32.0))))),
                "lo": 16 if rng.random() < 0.5 else 32, "hi": rng.choice((48, 80, 96, 112) if prec == 32 else (48, 64)),
                "mult": rng.choice((4, 16, 16)), "prec": prec, "riemann": "hllc"}
    if kind == "poisson":
        return {"kind": "poisson", **{k: int(round(math.exp(rng.uniform(math.log(9.0), math.log(190.0)))))
                                      for k in ("nx", "ny", "nz")}, "precond": rng.choice((1, 1, 0))}
    if kind == "infer":
        return {"kind": "infer", "n": int(round(math.exp(rng.uniform(math.log(65.0), math.log(6e6))))),
                "tc": rng.choice((1, 1, 0))}
    return {"kind": "train", "n": int(round(math.exp(rng.uniform(math.log(100.0), math.log(65536.0)))))}


# ---- inputs ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _grf(n, g):
    """Unit-variance periodic Gaussian random field with P(k) ~ k^-4."""
    f = torch.fft.rfftn(torch.randn(n, n, n, generator=g, device=DEV, dtype=torch.float64))
    k = torch.fft.fftfreq(n, device=DEV, dtype=torch.float64) * n
    kz = torch.fft.rfftfreq(n, device=DEV, dtype=torch.float64) * n
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kz[None, None, :] ** 2
    k2[0, 0, 0] = math.inf
    d = torch.fft.irfftn(f / k2, s=(n, n, n))
    return (d - d.mean()) / d.std()


def _cells(tree):
    """(level, X, Y, Z) of every cell, cell coordinates at its own level."""
    t = tree.tables()
    c = torch.arange(8, device=DEV)
    xyz = [(2 * t[a].long()[:, None] + ((c >> d) & 1)).reshape(-1) for d, a in enumerate(("ix", "iy", "iz"))]
    return t["lvl"].long().repeat_interleave(8), xyz


def _turb(tree, level, mach, seed):
    g, n = _gen(seed), 1 << level
    lvl, xyz = _cells(tree)
    # a cell above the finest level takes the field at its lower corner; the restriction
    # replaces it
    i, j, k = (x << (level - lvl) for x in xyz)
    flat = (i * n + j) * n + k
    rho = torch.exp(_grf(n, g) - 0.5)
    v = torch.stack([_grf(n, g) for _ in range(3)])
    v *= mach / torch.sqrt((v * v).sum(0).mean())
    return torch.stack([rho.reshape(-1)[flat]] + [v[d].reshape(-1)[flat] for d in range(3)] + [rho.reshape(-1)[flat]])


def _sod(tree, seed):
    lvl, xyz = _cells(tree)
    g = _gen(seed)
    left = (xyz[0] + 0.5) * torch.exp2(-lvl.double()) < 0.5
    w = torch.zeros(5, tree.ncell, device=DEV, dtype=torch.float64)
    # Toro's test 1 with the seed's own strength
    s = 1.0 + 0.2 * float(_rand(g, 1))
    w[0] = torch.where(left, s, 0.125)
    w[4] = torch.where(left, s, 0.1)
    return w


def _plummer(tree, case, seed):
    """Clumps on a unit background, their places given by the case (so is the mesh); the
    smooth velocity field they move in and the temperature are the seed's."""
    g = _gen(seed)
    cen = _rand(_gen(7919 * case["clumps"] + case["base"]), case["clumps"], 3)
    ph = _rand(g, 4, 3) * 2 * math.pi
    a2 = (0.64 * 2.0 ** -case["base"]) ** 2
    lvl, xyz = _cells(tree)
    h = torch.exp2(-lvl.double())
    x = [(p + 0.5) * h for p in xyz]
    rho = torch.ones_like(h)
    for c in cen:
        r2 = 0.0
        for d in range(3):
            e = x[d] - c[d]
            r2 = r2 + (e - torch.round(e)) ** 2
        q = 1.0 / (1.0 + r2 / a2)
        rho += 1e4 * q * q * torch.sqrt(q)
    w = torch.empty(5, tree.ncell, device=DEV, dtype=torch.float64)
    w[0] = rho

    def waves(d):
        return sum(torch.sin(2 * math.pi * (k + 1) * x[(d + k) % 3] + ph[d, k]) for k in range(3))
    for d in range(3):
        w[1 + d] = 0.4 * waves(d)
    w[4] = rho * torch.exp(0.1 * waves(3))
    return w


def _params(case):
    field = "plummer" if case["kind"] in ("amr", "sub", "refine") else case.get("field", "sedov")
    return hydro.Params(GAMMA[field], cfl=CFL, rho_floor=RHO_FLOOR, p_floor=P_FLOOR,
                        riemann=RIEMANN[case.get("riemann", "hllc")], limiter=LIMITER[case.get("limiter", "minmod")],
                        precision=abi.PREC_FP32 if case.get("prec", 64) == 32 else abi.PREC_FP64)


def _mesh(case, seed, short=0):
    """The adaptive mesh grown a level at a time around the clumps, and the state on it."""
    prm = _params(case)
    base = case["base"]
    tree = hydro.Octree(W.uniform_tree(base), base, (case["bc"],) * 6, device=DEV)
    u = None
    for _ in range(case["lmax"] - base + 1 - short):
        if u is not None:
            tree, u = tree.refine(u, case["thr"] * 8.0 ** -base, case["lmax"])
        u = torch.empty((5, tree.ncell), dtype=torch.float64, device=DEV)
        hydro.hydro_init_from_prim(tree, prm, _plummer(tree, case, seed), u)
    return tree, prm, u


def _buffers(tree, prm, u):
    dt = torch.zeros(max(1, tree.n_inst), dtype=torch.float64, device=DEV)
    hydro.hydro_courant(tree, prm, u, dt)
    return {"tree": tree, "prm": prm, "u": u, "u_new": torch.zeros_like(u), "dt": dt, "dt_next": torch.zeros_like(dt),
            "reg": torch.zeros(max(1, tree.flux_reg_bytes() // 8), dtype=torch.float64, device=DEV)}


def _sizes(case, seed):
    choices = np.arange(case["lo"], case["hi"] + 1, case["mult"])
    n = np.random.default_rng(case["boxes"] * 1000 + case["hi"]).choice(choices, size=case["boxes"]).astype(np.int32)
    return n


def _blasts(tree, seed):
    """A blast wave at its own age in every box: a dense shell, hot inside, moving out."""
    g, parts = _gen(seed), []
    c = torch.arange(8, device=DEV)
    for n in (int(s) for s in tree.sizes):
        o = torch.arange((n // 2) ** 3, device=DEV)
        m = n // 2
        x = [((2 * q[:, None] + ((c >> d) & 1)).reshape(-1) + 0.5) / n - 0.5
             for d, q in enumerate((o % m, (o // m) % m, o // (m * m)))]
        r = torch.sqrt(x[0] ** 2 + x[1] ** 2 + x[2] ** 2)
        R = 0.12 + 0.3 * _rand(g, 1)
        shell = torch.exp(-((r - R) / 0.03) ** 2)
        inside = torch.sigmoid((R - r) / 0.01)
        w = torch.empty(5, r.numel(), device=DEV, dtype=torch.float64)
        w[0] = 1.0 + 3.0 * shell - 0.9 * inside * (1 - shell)
        for d in range(3):
            w[1 + d] = 0.6 * R ** -1.5 * inside * x[d] / R
        w[4] = 1e-5 + 0.15 * R ** -3 * (inside + shell)
        parts.append(w)
    return torch.cat(parts, 1)


def _theta(g):
    th = []
    for o, i in ((64, 7), (64, 64), (64, 64), (2, 64)):
        th += [torch.randn(o * i, generator=g, device=DEV) / math.sqrt(i),
               0.1 * torch.randn(o, generator=g, device=DEV)]
    return torch.cat(th)


def _features(g, n):
    """Normalised face problems: x = [0, -du, log pL/pref, log rhoR/rhoL, du, log pR/pref, gamma]."""
    x = torch.zeros(n, 8, device=DEV)
    d = 0.3 * torch.randn(n, 3, generator=g, device=DEV)
    x[:, 1], x[:, 4] = -d[:, 0], d[:, 0]
    x[:, 2], x[:, 5] = d[:, 1].clamp(max=0), (-d[:, 1]).clamp(max=0)
    x[:, 3] = d[:, 2]
    x[:, 6] = 5.0 / 3.0
    return x


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("box", "sim"):
        lev = case["level"]
        tree = hydro.Octree(W.uniform_tree(lev), lev, (case["bc"],) * 6, device=DEV)
        prm = _params(case)
        w = _sod(tree, seed) if case["field"] == "sod" else _turb(tree, lev, case["mach"], seed)
        u = torch.empty_like(w)
        hydro.hydro_init_from_prim(tree, prm, w, u)
        if kind == "sim":
            return {"kind": kind, "sim": hydro.Simulation(tree, prm, u0=u).use_graph()}
        return {"kind": kind, **_buffers(tree, prm, u)}
    if kind == "amr":
        return {"kind": kind, **_buffers(*_mesh(case, seed))}
    if kind == "sub":
        tree, prm, u = _mesh(case, seed)
        return {"kind": kind, "sim": hydro.SubcycledSimulation(tree, prm, u0=u)}
    if kind == "refine":
        tree, prm, u = _mesh(case, seed, short=1)
        return {"kind": kind, "tree": tree, "u": u, "thr": case["thr"] * 8.0 ** -case["base"], "lmax": case["lmax"]}
    if kind == "batch":
        tree = hydro.Octree.boxes(_sizes(case, seed), device=DEV)
        prm = _params(case)
        u = torch.empty((5, tree.ncell), dtype=torch.float64, device=DEV)
        hydro.hydro_init_from_prim(tree, prm, _blasts(tree, seed), u)
        return {"kind": kind, **_buffers(tree, prm, u)}
    if kind == "poisson":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        g = _gen(seed)
        k, j, i = torch.meshgrid(*(torch.arange(n, device=DEV, dtype=torch.float64) for n in (nz, ny, nx)),
                                 indexing="ij")
        rho, s = torch.ones_like(i), float(max(nx, ny, nz))
        for c in _rand(g, 24, 3):
            r2 = ((i + 0.5 - c[0] * nx) ** 2 + (j + 0.5 - c[1] * ny) ** 2 + (k + 0.5 - c[2] * nz) ** 2) / (s * s)
            q = 1.0 / (1.0 + r2 / 2.5e-5)
            rho += torch.where(r2 < 0.01, 1e4 * q * q * torch.sqrt(q), 0.0)
        b = (-4.0 * math.pi / (s * s) * (rho - rho.mean())).reshape(-1).contiguous()
        return {"kind": kind, "b": b, "solver": poisson.PPCG((nx, ny, nz), precond=case["precond"], max_iter=2000)}
    g = _gen(seed)
    net = hydro.Surrogate(theta=_theta(g).cpu().numpy(), device=DEV)
    x = _features(g, case["n"])
    if kind == "infer":
        return {"kind": kind, "net": net, "x": x, "tc": case["tc"]}
    # in the middle of a training run: the moments of the steps before
    net.m.copy_(1e-3 * torch.randn(net.m.shape, generator=g, device=DEV))
    net.v.copy_(1e-5 * (0.5 + torch.rand(net.v.shape, generator=g, device=DEV)))
    net.t = 1000
    y = 0.3 * torch.tanh(torch.stack([x[:, 2] + x[:, 5] - x[:, 4], x[:, 2] - x[:, 5]], 1))
    scratch = torch.empty(int(abi.lib().mlp_scratch_bytes(case["n"])) // 4 + 1, dtype=torch.float32, device=DEV)
    return {"kind": kind, "net": net, "x": x, "y": y, "scratch": scratch,
            "loss": torch.zeros(1, dtype=torch.float32, device=DEV)}


def run(s):
    kind = s["kind"]
    if kind in ("box", "amr", "batch"):
        hydro.hydro_step(s["tree"], s["prm"], s["u"], s["u_new"], s["reg"], s["dt"], s["dt_next"])
        return {"u": s["u_new"], "dt": s["dt_next"]}
    if kind in ("sim", "sub"):
        s["sim"].step()
        return {"u": s["sim"].u, "dt": s["sim"].dt}
    if kind == "refine":
        tree, u = s["tree"].refine(s["u"], s["thr"], s["lmax"])
        return {"u": u, **tree.tables()}
    if kind == "poisson":
        x, eps, info = s["solver"].solve(s["b"])
        return {"x": x, "eps": info.eps}
    net = s["net"]
    if kind == "infer":
        if not s["tc"]:
            return {"y": net.forward(s["x"])}
        y = torch.empty((s["x"].shape[0], 2), dtype=torch.float32, device=s["x"].device)
        hydro.mlp_forward_tc(net.packed, s["x"], y)
        return {"y": y}
    net.t += 1
    hydro.mlp_train_step(net.theta, net.m, net.v, net.packed, s["x"], s["y"], 1e-3, net.t, s["loss"], s["scratch"])
    return {"theta": net.theta, "m": net.m, "v": net.v, "loss": s["loss"]}


def work(case):
    kind = case["kind"]
    if kind in ("box", "sim"):
        cells = 8 ** case["level"]
    elif kind == "batch":
        cells = int((_sizes(case, 0).astype(np.int64) ** 3).sum())
    elif kind == "amr":
        cells = _mesh(case, 0)[0].leaf_cells()
    elif kind == "sub":
        t = _mesh(case, 0)[0].tables()                       # a level's leaves once per step of that level
        leaf = t["lvl"].long().repeat_interleave(8)[t["son"] < 0]
        cells = int((2.0 ** (leaf - case["base"]).double()).sum())
    elif kind == "refine":
        s = prepare(case, 0)
        new, _ = s["tree"].refine(s["u"], s["thr"], s["lmax"])
        # the state and the tables of the old mesh read, those of the new mesh written
        tables = sum(t.numel() * t.element_size() for t in new.tables().values())
        return {"bytes": 40 * (s["tree"].ncell + new.ncell) + tables + 40 * s["tree"].noct, "flops": 0}
    elif kind == "poisson":
        s = prepare(case, 0)
        it = s["solver"].solve(s["b"])[2].iters
        # eight vectors read and written each iteration (six without a preconditioner)
        return {"bytes": (128 if case["precond"] else 96) * s["b"].numel() * it,
                "flops": (46 if case["precond"] else 28) * s["b"].numel() * it}
    else:
        n, p = case["n"], 2 * (7 * 64 + 2 * 64 * 64 + 64 * 2)
        if kind == "infer":
            return {"bytes": 40 * n, "flops": p * n}
        return {"bytes": 40 * n + 24 * 8962, "flops": 3 * p * n}
    return {"bytes": BYTES_PER_CELL * cells, "flops": FLOPS_PER_CELL * cells}


# ---- the same calls in 64 bits ---------------------------------------------------------
class _Scheme:
    """MUSCL-Hancock on an octree, or on boxes, in FP64 torch: every oct with its two-cell
    halo as a 6^3 block.  Written from the scheme's statement in include/amrhydro.h."""

    def __init__(self, case, tree, gamma):
        self.g, self.case = gamma, case
        self.batch = tree.n_inst > 0
        self.lmin, self.lmax = tree.levelmin, tree.levelmax
        self.bc = case.get("bc", 1)
        if self.batch:                       # boxes: octs in lexicographic order, nothing refined
            self.sizes = [int(n) for n in tree.sizes]
            self.off_box = [0] + np.cumsum((np.array(self.sizes, dtype=np.int64) // 2) ** 3).tolist()
            self.son = torch.full((tree.ncell,), -1, device=DEV)
            o = [(torch.arange((n // 2) ** 3, device=DEV), n // 2) for n in self.sizes]
            self.ijk = torch.cat([torch.stack([i % m, (i // m) % m, i // (m * m)], 1) for i, m in o])
            return
        t = tree.tables()
        self.lvl, self.ijk = t["lvl"].long(), torch.stack([t[a].long() for a in ("ix", "iy", "iz")], 1)
        self.son = t["son"].long()
        self.off = [int(v) for v in tree.lvl_off]
        self.keys = {}
        for l in range(1, self.lmax + 1):
            k, order = torch.sort(self._code(self.ijk[self.off[l]:self.off[l + 1]]))
            self.keys[l] = (k, order + self.off[l])

    @staticmethod
    def _code(x):
        return (x[..., 0] << 42) | (x[..., 1] << 21) | x[..., 2]

    def _wrap(self, x, n):
        return x % n if self.bc == 0 else x.clamp(0, n - 1)

    def find(self, l, x):
        """Oct of level l at oct coordinates x (wrapped or clamped), -1 if there is none."""
        k, order = self.keys[l]
        c = self._code(self._wrap(x, 1 << (l - 1)))
        p = torch.searchsorted(k, c).clamp(max=k.numel() - 1)
        return torch.where(k[p] == c, order[p], -1)

    @staticmethod
    def _cell(x):
        return (x[..., 0] & 1) + 2 * (x[..., 1] & 1) + 4 * (x[..., 2] & 1)

    def children(self, U, l, x):
        """Interpolated children [m, 5, 8] of the level-l cells at cell coordinates x [m, 3]."""
        n = 1 << l
        x = self._wrap(x, n)
        me = U[:, self.find(l, x >> 1) * 8 + self._cell(x)].T
        out = me[:, :, None].repeat(1, 1, 8)
        c = torch.arange(8, device=U.device)
        for d in range(3):
            v = []
            for s in (-1, 1):
                y = x.clone()
                y[:, d] += s
                y = self._wrap(y, n)
                o = self.find(l, y >> 1)
                up = y >> 1                                   # the coarser leaf that holds it
                coarse = self.find(l - 1, up >> 1) * 8 + self._cell(up) if l > 1 else torch.zeros_like(o)
                v.append(U[:, torch.where(o >= 0, o * 8 + self._cell(y), coarse)].T)
            m = self.minmod(me - v[0], v[1] - me)
            out += 0.25 * m[:, :, None] * torch.where((c >> d) & 1 == 1, 1.0, -1.0)
        return out

    def block(self, U, l, o):
        """States [n, 5, 6, 6, 6] (z, y, x) around octs o of level l (batch: of box l), refined
        flags of the same cells, and which of the 27 neighbour octs are coarse leaves."""
        nb = torch.arange(27, device=U.device)
        step = torch.stack([nb % 3, (nb // 3) % 3, nb // 9], 1) - 1
        y = self.ijk[o][:, None, :] + step
        if self.batch:
            m = self.sizes[l] // 2
            w = y.clamp(0, m - 1)
            oct_ = self.off_box[l] + w[..., 0] + m * (w[..., 1] + m * w[..., 2])
            n = 2 * m
        else:
            oct_ = self.find(l, y)
            n = 1 << l
        cells = oct_.clamp(min=0)[..., None] * 8 + torch.arange(8, device=U.device)
        V = U[:, cells].permute(1, 0, 2, 3).contiguous()        # [n, 5, 27, 8]
        ref = (self.son[cells] >= 0) & (oct_ >= 0)[..., None]
        gone = oct_ < 0
        if bool(gone.any()):
            a, b = torch.nonzero(gone, as_tuple=True)
            V[a, :, b] = self.children(U, l - 1, y[a, b])
        V = V.reshape(-1, 5, 3, 3, 3, 2, 2, 2).permute(0, 1, 2, 5, 3, 6, 4, 7).reshape(-1, 5, 6, 6, 6)
        ref = ref.reshape(-1, 3, 3, 3, 2, 2, 2).permute(0, 1, 4, 2, 5, 3, 6).reshape(-1, 6, 6, 6)
        if self.bc == 1 or self.batch:                          # zero gradient beyond the box
            for d, ax in enumerate((4, 3, 2)):
                at = (2 * self.ijk[o][:, d, None] + torch.arange(-2, 4, device=U.device)).clamp(0, n - 1)
                at = at - 2 * self.ijk[o][:, d, None] + 2
                shape = [-1, 1, 1, 1, 1]
                shape[ax] = 6
                V = torch.gather(V, ax, at.reshape(shape).expand_as(V))
                ref = torch.gather(ref, ax - 1, at.reshape(shape)[:, 0].expand_as(ref))
            out = (y < 0) | (y >= n // 2)
            gone = gone & ~out.any(-1)
        return V, ref, gone, oct_, y

    @staticmethod
    def minmod(a, b):
        return torch.where(a * b > 0, torch.where(a.abs() < b.abs(), a, b), 0.0)

    def slope(self, a, b):
        """Slopes of the reconstruction (the ghost interpolation is MinMod in any case)."""
        if self.case.get("limiter", "minmod") == "minmod":
            return self.minmod(a, b)
        m = torch.minimum(2 * torch.minimum(a.abs(), b.abs()), 0.5 * (a + b).abs())
        return torch.where(a * b > 0, torch.copysign(m, a), 0.0)

    def prim(self, U, ax=1):
        r, mx, my, mz, E = U.unbind(ax)
        r = r.clamp(min=RHO_FLOOR)
        u, v, w = mx / r, my / r, mz / r
        p = ((self.g - 1) * (E - 0.5 * r * (u * u + v * v + w * w))).clamp(min=P_FLOOR)
        return torch.stack([r, u, v, w, p], ax)

    def flux(self, L, R):
        """Face-normal flux [n, 5, ...] of states with the normal velocity in slot 1."""
        g = self.g
        rL, uL, _, _, pL = L.unbind(1)
        rR, uR, _, _, pR = R.unbind(1)
        cL, cR = torch.sqrt(g * pL / rL), torch.sqrt(g * pR / rR)

        def phys(w):
            r, u, v, q, p = w.unbind(1)
            E = p / (g - 1) + 0.5 * r * (u * u + v * v + q * q)
            return (torch.stack([r * u, r * u * u + p, r * u * v, r * u * q, u * (E + p)], 1),
                    torch.stack([r, r * u, r * v, r * q, E], 1))
        if self.case.get("riemann", "hllc") == "exact":
            return phys(self.star(L, R, cL, cR))[0]
        SL, SR = torch.minimum(uL - cL, uR - cR), torch.maximum(uL + cL, uR + cR)
        Ss = (pR - pL + rL * uL * (SL - uL) - rR * uR * (SR - uR)) / (rL * (SL - uL) - rR * (SR - uR))
        out = None
        for w, S in ((L, SL), (R, SR)):
            F, U = phys(w)
            r, u, v, q, p = w.unbind(1)
            f = r * (S - u) / (S - Ss)
            star = F + S[:, None] * (torch.stack([f, f * Ss, f * v, f * q, f * (
                U[:, 4] / r + (Ss - u) * (Ss + p / (r * (S - u))))], 1) - U)
            if out is None:
                out = torch.where((SL >= 0)[:, None], F, star)
            else:
                right = torch.where((SR > 0)[:, None], star, F)
                out = torch.where(((SL >= 0) | (Ss >= 0))[:, None], out, right)
        return out

    def star(self, L, R, cL, cR):
        """The exact solution at x/t = 0 (Newton on the pressure function)."""
        g = self.g
        rL, uL, _, _, pL = L.unbind(1)
        rR, uR, _, _, pR = R.unbind(1)

        def side(p, r, pk, c):
            A, B = 2 / ((g + 1) * r), (g - 1) / (g + 1) * pk
            q = torch.sqrt(A / (p + B))
            e = (p / pk).clamp(min=1e-300)
            shock = p > pk
            return (torch.where(shock, (p - pk) * q, 2 * c / (g - 1) * (e ** ((g - 1) / (2 * g)) - 1)),
                    torch.where(shock, q * (1 - 0.5 * (p - pk) / (B + p)), e ** (-(g + 1) / (2 * g)) / (r * c)))
        z = (g - 1) / (2 * g)                                    # start: the two-rarefaction solution
        p = ((cL + cR - 0.5 * (g - 1) * (uR - uL)) / (cL * pL ** -z + cR * pR ** -z)).clamp(min=1e-60) ** (1 / z)
        for _ in range(20):
            (fL, dL), (fR, dR) = side(p, rL, pL, cL), side(p, rR, pR, cR)
            p = (p - (fL + fR + uR - uL) / (dL + dR)).clamp(min=1e-300)
        fL, fR = side(p, rL, pL, cL)[0], side(p, rR, pR, cR)[0]
        us = 0.5 * (uL + uR) + 0.5 * (fR - fL)
        left = us >= 0
        sg = torch.where(left, 1.0, -1.0)                        # mirror the right side onto the left
        r, u, pk, c, v = (torch.where(left, a, b) for a, b in ((rL, rR), (uL, uR), (pL, pR), (cL, cR), (us, us)))
        u, v = sg * u, sg * v
        x, g6 = p / pk, (g - 1) / (g + 1)
        S = u - c * torch.sqrt((g + 1) / (2 * g) * x + (g - 1) / (2 * g))
        head, tail = u - c, v - c * x ** ((g - 1) / (2 * g))
        fan = 2 / (g + 1) * (c + 0.5 * (g - 1) * u)
        e = (fan / c).clamp(min=1e-300)
        shock = p > pk
        out = torch.where(shock, S >= 0, head >= 0)
        infan = ~shock & ~out & (tail >= 0)
        ro = torch.where(shock, r * (x + g6) / (x * g6 + 1), r * x ** (1 / g))
        ro = torch.where(out, r, torch.where(infan, r * e ** (2 / (g - 1)), ro))
        uo = torch.where(out, u, torch.where(infan, fan, v))
        po = torch.where(out, pk, torch.where(infan, pk * e ** (2 * g / (g - 1)), p))
        tr = torch.where(left[:, None], L[:, 2:4], R[:, 2:4])
        return torch.stack([ro, sg * uo, tr[:, 0], tr[:, 1], po], 1)

    def octs(self, V, lam):
        """Fluxes (x, y, z) [n, 5, ...] through the faces of the inner 2^3 cells of each block."""
        Wp = self.prim(V)
        C = Wp[:, :, 1:5, 1:5, 1:5]
        D = []
        for ax in (4, 3, 2):
            lo, hi = [slice(1, 5)] * 3, [slice(1, 5)] * 3
            lo[ax - 2], hi[ax - 2] = slice(0, 4), slice(2, 6)
            D.append(self.slope(C - Wp[(slice(None), slice(None), *lo)], Wp[(slice(None), slice(None), *hi)] - C))
        r, u, v, w, p = C.unbind(1)
        h = 0.5 * lam
        div = D[0][:, 1] + D[1][:, 2] + D[2][:, 3]

        def adv(k):
            return u * D[0][:, k] + v * D[1][:, k] + w * D[2][:, k]
        P = torch.stack([r - h * (adv(0) + r * div), u - h * (adv(1) + D[0][:, 4] / r),
                         v - h * (adv(2) + D[1][:, 4] / r), w - h * (adv(3) + D[2][:, 4] / r),
                         p - h * (adv(4) + self.g * p * div)], 1)
        F = []
        for d, ax in enumerate((4, 3, 2)):
            a, b = [slice(1, 3)] * 3, [slice(1, 3)] * 3
            a[ax - 2], b[ax - 2] = slice(0, 3), slice(1, 4)
            a, b = (slice(None), slice(None), *a), (slice(None), slice(None), *b)
            perm = [0, d + 1] + [1 + k for k in range(3) if k != d] + [4]
            L, R = (P + 0.5 * D[d])[a][:, perm], (P - 0.5 * D[d])[b][:, perm]
            for q in (L, R):
                q[:, 0].clamp_(min=RHO_FLOOR)
                q[:, 4].clamp_(min=P_FLOOR)
            f = self.flux(L, R)
            back = torch.empty_like(f)
            back[:, perm] = f
            F.append(back)
        return F

    def advance(self, U, N, l, dt, chunk=100000):
        """The leaves of level l (batch: box l) into N; returns the coarse cells next to the
        level with the corrections they are due: (cells, sign * flux sum / 4)."""
        lo, hi = (self.off_box[l], self.off_box[l + 1]) if self.batch else (self.off[l], self.off[l + 1])
        lam = dt * (self.sizes[l] if self.batch else 2.0 ** l)
        due = []
        for s in range(lo, hi, chunk):
            o = torch.arange(s, min(hi, s + chunk), device=U.device)
            V, ref, gone, oct_, y = self.block(U, l, o)
            F = self.octs(V, lam)
            dU = 0.0
            for d, ax in enumerate((4, 3, 2)):
                for side in (0, 1):
                    sl = [slice(2, 4)] * 3
                    sl[ax - 2] = slice(1, 3) if side == 0 else slice(3, 5)
                    keep = ~ref[(slice(None), *sl)][:, None]
                    f = F[d].narrow(ax, side, 2)
                    dU = dU + (1 - 2 * side) * torch.where(keep, f, 0.0)
                    k = 13 + (2 * side - 1) * 3 ** d
                    at = torch.nonzero(gone[:, k]).reshape(-1)
                    if at.numel():
                        q = self._wrap(y[at, k], 1 << (l - 1))
                        cell = self.find(l - 1, q >> 1) * 8 + self._cell(q)
                        due.append((cell, (2 * side - 1) * 0.25 * F[d].narrow(ax, 2 * side, 1)[at].sum((2, 3, 4))))
            cells = (o[:, None] * 8 + torch.arange(8, device=U.device)).reshape(-1)
            leaf = self.son[cells] < 0
            new = U[:, cells] + lam * dU.reshape(-1, 5, 8).permute(1, 0, 2).reshape(5, -1)
            N[:, cells[leaf]] = new[:, leaf]
        return due

    @staticmethod
    def reflux(N, due, lam):
        for cell, f in due:
            N.index_add_(1, cell, (lam * f).T.contiguous())

    def restrict(self, N, l):
        c = torch.arange(self.off[l] * 8, self.off[l + 1] * 8, device=N.device)
        c = c[self.son[c] >= 0]
        if c.numel():
            N[:, c] = N[:, self.son[c][:, None] * 8 + torch.arange(8, device=N.device)].mean(2)

    def speed(self, U):
        """cfl / sum_d(|u_d| + c) of every cell."""
        Wp = self.prim(U, 0)
        return CFL / (Wp[1:4].abs().sum(0) + 3 * torch.sqrt(self.g * Wp[4] / Wp[0]))

    def step(self, U, dt):
        N = U.clone()
        if self.batch:
            for b in range(len(self.sizes)):
                self.advance(U, N, b, dt[b])
            v = self.speed(N)
            return N, torch.stack([v[8 * self.off_box[b]:8 * self.off_box[b + 1]].min() / n
                                   for b, n in enumerate(self.sizes)])
        due = {l: self.advance(U, N, l, dt[0]) for l in range(self.lmin, self.lmax + 1)}
        for l in range(self.lmax, 0, -1):
            if l > self.lmin:
                self.reflux(N, due[l], dt[0] * 2.0 ** (l - 1))
            if l < self.lmax:
                self.restrict(N, l)
        for l in range(self.lmax - 1, 0, -1):
            self.restrict(N, l)
        leaf = self.son < 0
        h = torch.exp2(-self.lvl.double()).repeat_interleave(8)
        return N, (self.speed(N) * h)[leaf].min().reshape(1)

    def subcycle(self, U):
        U = U.clone()
        N = U.clone()
        leaf = self.son < 0
        base = self.lmin
        dt0 = (self.speed(U) * 2.0 ** -base)[leaf].min()

        def go(c):
            dt = dt0 * 2.0 ** (base - c)
            due = self.advance(U, N, c, dt)
            mine = torch.arange(self.off[c] * 8, self.off[c + 1] * 8, device=U.device)
            if c < self.lmax:
                lam = 0.5 * dt * 2.0 ** c
                fine = go(c + 1)
                m = mine[leaf[mine]]
                U[:, m] = 0.5 * (U[:, m] + N[:, m])
                for A in (U, N):
                    self.reflux(A, fine, lam)
                    self.restrict(A, c)
                fine = go(c + 1)
                self.reflux(N, fine, lam)
                self.restrict(N, c)
            U[:, mine] = N[:, mine]
            return due
        go(base)
        for l in range(base - 1, 0, -1):
            self.restrict(U, l)
        return U, dt0.reshape(1)


def _pcg(b, shape, precond, iters):
    """Textbook preconditioned CG from zero, `iters` iterations; x and Eq. 3's last value."""
    nx, ny, nz = shape
    b = b.reshape(nz, ny, nx)

    def near(v):
        q = torch.nn.functional.pad(v, (1, 1, 1, 1, 1, 1))
        return (q[1:-1, 1:-1, :-2] + q[1:-1, 1:-1, 2:] + q[1:-1, :-2, 1:-1] + q[1:-1, 2:, 1:-1] +
                q[:-2, 1:-1, 1:-1] + q[2:, 1:-1, 1:-1])

    def minv(v):
        return 13.0 / 12.0 * v + near(v) / 6.0 if precond else v
    x, r = torch.zeros_like(b), b.clone()
    u = minv(r)
    p, gam = u.clone(), (r * u).sum()
    g0 = gam
    for _ in range(iters):
        s = 6.0 * p - near(p)
        a = gam / (p * s).sum()
        x += a * p
        r -= a * s
        u = minv(r)
        new = (r * u).sum()
        p = u + (new / gam) * p
        gam = new
    return x.reshape(-1), float(torch.sqrt(gam / g0))


def _net(theta, x):
    t, o, a = theta, 0, x[:, :7]
    for k, (m, n) in enumerate(((64, 7), (64, 64), (64, 64), (2, 64))):
        a = a @ t[o:o + m * n].reshape(m, n).T + t[o + m * n:o + m * n + m]
        o += m * n + m
        a = a * torch.sigmoid(a) if k < 3 else a
    return a


def exact(case, seed):
    kind = case["kind"]
    if kind == "refine":
        return None              # a mesh of whole numbers, and the state copied or interpolated onto it
    s = prepare(case, seed)
    if kind in ("box", "amr", "batch", "sim", "sub"):
        h = s["sim"] if kind in ("sim", "sub") else None
        tree, prm, u = (h.tree, h.prm, h.u) if h else (s["tree"], s["prm"], s["u"])
        S = _Scheme(case, tree, float(prm.c.gamma))
        if kind == "sub":
            u, dt = S.subcycle(u)
        else:
            u, dt = S.step(u, h.dt if h else s["dt"])
        return {"u": u, "dt": dt}
    if kind == "poisson":
        shape = (case["nx"], case["ny"], case["nz"])
        it = s["solver"].solve(s["b"])[2].iters             # as many iterations as the tolerance takes
        x, eps = _pcg(s["b"], shape, case["precond"], it)
        return {"x": x, "eps": eps}
    theta = s["net"].theta.double()
    if kind == "infer":
        return {"y": _net(theta, s["x"].double())}
    th = theta.clone().requires_grad_(True)
    loss = ((_net(th, s["x"].double()) - s["y"].double()) ** 2).sum() / case["n"]
    (g,) = torch.autograd.grad(loss, th)
    t = s["net"].t + 1
    m = 0.9 * s["net"].m.double() + 0.1 * g
    v = 0.999 * s["net"].v.double() + 0.001 * g * g
    new = theta - 1e-3 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return {"theta": new, "m": m, "v": v, "loss": loss.detach().reshape(1)}

"""The work this library is measured on: its public calls over their range of
block sizes, wavelets, schemes, precisions and tree sizes.

A case names an operation, a forest of octrees and the options of the call:
  step     one RK3 step with a constant velocity          Grid.step
  vel      one RK3 step with three velocity fields        Grid.step_vel
  loop     time step from the fields, RK3 step, mass      Grid.dt, step_vel, mass
  ghost    padded blocks of one field                     Grid.ghost_fill
  crit     block norms of one field                       Grid.criterion
  adapt    the tree follows a moved feature and back      Grid.field_set, adapt
Trees: nested balls of refinement (as the benchmark's fixed workloads), a
batch of uneven one-tree grids, a slab that meets the domain's faces, or, for
adapt, the tree the call itself builds around the feature.
"""
import functools

import numpy as np
import torch

from paper_2112_07537_gb300 import mrgb

SCHEME = {"cons3": 0, "cons5": 1, "wenoz5": 2}


def listed():
    def c(name, op, **kw):
        base = {"name": name, "op": op, "tree": "balls", "nt": "1,1,1", "len": 1.0, "nb": 24, "base": 3,
                "radii": "", "lmax": 0, "wav": "6.2", "prec": "f32", "scheme": "wenoz5", "diff": 0, "shell": 3}
        base.update(kw)
        return base

    return [
        # the tiny two-level start configuration (15 leaves): latency of a step
        c("step-tiny-f64", "step", tree="corner", nt="2,2,2", len=0.5, nb=16, base=0, wav="4.0", prec="f64"),
        # a small velocity-field run, one launch's worth of leaves per kernel
        c("vel-tiny-f32", "vel", nt="2,2,2", len=0.5, nb=16, base=0, radii="0.3,0.16", wav="4.2", scheme="cons5"),
        # advection-diffusion on an uneven forest with the cheapest scheme and wavelet, blocks off the tuned sizes
        c("step-diff-f32", "step", nt="3,2,2", len=0.5, nb=20, base=1, radii="0.35,0.2,0.1", wav="2.2",
          scheme="cons3", diff=2),
        # the adaptive solver's step on a small grid (47 M points): three velocity fields
        c("vel-small-f32", "vel", radii="0.3,0.2"),
        # the largest fixed grid of the benchmark (586 M points), constant velocity
        c("step-large-f32", "step", radii="0.35,0.25,0.17,0.11,0.06"),
        # the plain double-precision form of the solver's step
        c("vel-f64", "vel", radii="0.2,0.12", prec="f64"),
        # 64 uneven one-tree grids advanced together: what a time loop calls between adaptations
        c("loop-batch-f32", "loop", tree="batch", nt="4,4,4", nb=16, base=1, radii="0.4,0.25", wav="4.2"),
        # physical boundaries on every face, refinement meeting them
        c("step-bounded-f32", "step", tree="slab", nt="4,4,4", len=0.25, nb=16, base=0, wav="4.2"),
        # the wavelet kernels alone (2 080 leaves): stencil ghosts of a field with a front
        c("ghost-f32", "ghost", radii="0.25,0.14"),
        # ... and its block norms, the decision every adaptation starts from
        c("crit-f32", "crit", radii="0.25,0.14"),
        # remeshing of a production-sized grid after its front moved (scalar and three velocity fields)
        c("adapt-front-f32", "adapt", tree="front", base=2, lmax=5),
        # remeshing of a small double-precision run
        c("adapt-front-f64", "adapt", tree="front", nb=16, base=2, lmax=4, wav="4.2", prec="f64"),
    ]


def draw(rng):
    while True:
        op = rng.choice(["step", "step", "vel", "vel", "loop", "ghost", "crit", "adapt"])
        case = {"op": op, "tree": "balls", "nt": "1,1,1", "len": 1.0, "nb": rng.choice([8, 12, 16, 20, 24]), "base": 2,
                "radii": "", "lmax": 0, "wav": rng.choice(["2.0", "2.2", "4.0", "4.2", "6.0", "6.2", "6.2"]),
                "prec": rng.choice(["f32", "f32", "f32", "f64"]),
                "scheme": rng.choice(["wenoz5", "wenoz5", "cons5", "cons3"]),
                "diff": rng.choice([0, 0, 0, 2, 4]) if op in ("step", "vel") else 0, "shell": 3}
        N, Nt = wavelet(case)
        if internal_shell(N, Nt, 3, case["nb"]) > case["nb"] // 2:
            continue
        if op in ("crit", "adapt") and adapt_shell(N, Nt) > case["nb"] // 2:
            continue
        if op == "ghost":
            case["shell"] = rng.randint(1, internal_shell(N, Nt, 3, case["nb"]))
        if op == "adapt":
            case.update(tree="front", lmax=rng.choice([3, 4, 4, 5] if case["prec"] == "f32" else [3, 4]),
                        base=rng.choice([1, 2]))
            return case
        kind = rng.random()
        if kind < 0.12:
            case.update(tree="batch", nt=rng.choice(["2,2,2", "4,4,4", "3,5,1"]), base=1,
                        radii="%.3f,%.3f" % (rng.uniform(0.15, 0.45), rng.uniform(0.05, 0.25)))
        elif kind < 0.2 and op in ("step", "ghost"):
            # physical boundaries: wavelets up to fourth order (sixth-order extrapolation loses FP32 digits)
            if N == 6:
                continue
            case.update(tree="slab", nt="4,4,4", len=0.25, base=0)
        else:
            r, radii = rng.uniform(0.1, 0.4), []
            for _ in range(rng.randint(1, 4)):
                radii.append("%.3f" % r)
                r *= rng.uniform(0.45, 0.75)
            case.update(nt=rng.choice(["1,1,1", "1,1,1", "2,2,2", "3,2,1"]), radii=",".join(radii),
                        base=rng.choice([1, 2, 2, 3]))
        most = 8e6 if case["tree"] == "slab" else 6e7 if case["prec"] == "f64" else 4e8
        if len(tree(case)[0]) * case["nb"] ** 3 <= most:
            return case


# ------------------------------------------------------------------- trees
def wavelet(case):
    return tuple(int(v) for v in case["wav"].split("."))


def forest(case):
    return tuple(int(v) for v in case["nt"].split(","))


def uniform(nt, level):
    z, y, x = np.meshgrid(*[np.arange(nt[d] << level) for d in (2, 1, 0)], indexing="ij")
    anc = np.stack([x.ravel(), y.ravel(), z.ravel()], 1).astype(np.int64)
    return np.full(len(anc), level, np.int64), anc


def split(lev, anc, hit):
    kids = np.array([[c & 1, (c >> 1) & 1, c >> 2] for c in range(8)])
    return (np.concatenate([lev[~hit], np.repeat(lev[hit] + 1, 8)]),
            np.concatenate([anc[~hit], (2 * anc[hit][:, None] + kids).reshape(-1, 3)]))


def level_map(nt, lev, anc, M):
    D = np.zeros([nt[d] << M for d in (2, 1, 0)], np.int8)
    for L in np.unique(lev):
        V, s, a = np.zeros([nt[d] << L for d in (2, 1, 0)], np.int8), 1 << (M - L), anc[lev == L]
        V[a[:, 2], a[:, 1], a[:, 0]] = L + 1
        D = np.maximum(D, V.repeat(s, 0).repeat(s, 1).repeat(s, 2))
    return D - 1


def balanced(nt, lev, anc):
    """2:1 balance over faces, edges and corners (periodic forest)."""
    while True:
        M = int(lev.max())
        D = level_map(nt, lev, anc, M)
        for ax in range(3):
            D = np.maximum(D, np.maximum(np.roll(D, 1, ax), np.roll(D, -1, ax)))
        need = np.zeros(len(lev), bool)
        for L in np.unique(lev):
            s, i = 1 << (M - L), np.nonzero(lev == L)[0]
            B = D.reshape(D.shape[0] // s, s, D.shape[1] // s, s, -1, s).max((1, 3, 5))
            need[i] = B[anc[i, 2], anc[i, 1], anc[i, 0]] > L + 1
        if not need.any():
            return lev, anc
        lev, anc = split(lev, anc, need)


def balls(nt, length, base, radii, centre):
    """Uniform at base; every block of level base + k meeting the ball radii[k] refined; balanced."""
    lev, anc = uniform(nt, base)
    ext = np.array(nt) * length
    for k, r in enumerate(radii):
        size = length / (1 << lev)
        d = np.abs((anc + 0.5) * size[:, None] - np.array(centre))
        d = np.maximum(np.minimum(d, ext - d) - 0.5 * size[:, None], 0)
        lev, anc = balanced(nt, *split(lev, anc, (np.sqrt((d ** 2).sum(1)) <= r) & (lev == base + k)))
    return lev, anc


@functools.lru_cache(maxsize=8)
def build_tree(kind, nt, length, base, radii):
    if kind == "corner":  # the first tree of the forest refined once
        lev, anc = uniform(nt, base)
        lev, anc = split(lev, anc, (anc == 0).all(1))
    elif kind == "slab":  # refinement on the x = 0 face and the x = 0, z = 0 edge
        lev, anc = uniform(nt, base)
        lev, anc = split(lev, anc, (anc[:, 0] <= 1) & (anc[:, 1] >= 1) & (anc[:, 1] <= 2))
        lev, anc = balanced(nt, *split(lev, anc, (lev == 1) & (anc == (0, 2, 0)).all(1)))
    elif kind == "batch":  # every tree its own periodic grid, refined by its own balls
        rng, ls, as_ = np.random.default_rng(11), [], []
        for k in range(nt[0] * nt[1] * nt[2]):
            l, a = balls((1, 1, 1), length, base, [r * rng.uniform(0.5, 1.2) for r in radii], rng.uniform(0, 1, 3))
            t = np.array([k % nt[0], (k // nt[0]) % nt[1], k // (nt[0] * nt[1])])
            ls.append(l)
            as_.append(a + t * (1 << l)[:, None])
        lev, anc = np.concatenate(ls), np.concatenate(as_)
    elif kind == "front":
        lev, anc = uniform(nt, base)
    else:
        lev, anc = balls(nt, length, base, radii, 0.5 * np.array(nt) * length)
    return morton_sorted(lev, anc)


def morton_sorted(lev, anc):
    a = anc << (lev.max() - lev)[:, None]
    key = np.zeros(len(lev), np.int64)
    for bit in range(19):
        for d in range(3):
            key |= ((a[:, d] >> bit) & 1) << (3 * bit + d)
    o = np.argsort(key, kind="stable")
    return lev[o], anc[o]


def tree(case):
    radii = tuple(float(r) for r in case["radii"].split(",") if r)
    return build_tree(case["tree"], forest(case), case["len"], case["base"], radii)


# ------------------------------------------------------------------ inputs
def device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def coords(case, lev, anc):
    """x, y, z of every point, [leaf, z, y, x] (broadcastable), in tree-local units for a batch."""
    lev, anc = (torch.as_tensor(v, device=device()) for v in (lev, anc))
    if case["tree"] == "batch":
        anc = anc & ((1 << lev) - 1)[:, None]
    h = case["len"] / (case["nb"] * (1 << lev).double())
    i = torch.arange(case["nb"], device=device())
    g = [(anc[:, d, None] * case["nb"] + i) * h[:, None] for d in range(3)]
    return g[0][:, None, None, :], g[1][:, None, :, None], g[2][:, :, None, None]


def dtype(case):
    return torch.float32 if case["prec"] == "f32" else torch.float64


def inputs(case, seed):
    """Seeded field values [leaf, z, y, x], the velocity and the time step."""
    rng = np.random.default_rng([seed, 7])
    lev, anc = tree(case)
    x = coords(case, lev, anc)
    ext = [(1 if case["tree"] == "batch" else n) * case["len"] for n in forest(case)]
    nb, dt_ = case["nb"], dtype(case)
    phi = torch.empty((len(lev), nb, nb, nb), dtype=dt_, device=device())
    c = 0.5 * np.array(ext) + rng.uniform(-0.03, 0.03, 3) * min(ext)
    sigma = min(ext) * rng.uniform(0.07, 0.09)
    two_pi = 2 * np.pi
    modes = [(rng.integers(-4, 5, 3), rng.uniform(0, two_pi)) for _ in range(6)] if case["op"] in ("ghost", "crit") else []
    for b in range(0, len(lev), 512):
        xb = [v[b:b + 512] for v in x]
        r2 = 0
        for d in range(3):
            e = xb[d] - c[d]
            r2 = r2 + (e - ext[d] * torch.round(e / ext[d])) ** 2
        f = torch.exp(-r2 / sigma ** 2)
        if modes:  # smooth modes and a front on a sphere
            f = 0.5 * torch.tanh((3 * sigma - r2.sqrt()) / (0.25 * sigma))
            for k, th in modes:
                a = sum(two_pi * float(k[d]) / ext[d] * xb[d] for d in range(3))
                f = f + torch.cos(a + th) / (1.0 + float((k ** 2).sum()))
        phi[b:b + 512] = f.to(dt_)
    out = {"phi": phi}
    hmin = case["len"] / (nb * 2.0 ** lev.max())
    if case["op"] in ("vel", "loop"):
        ph = rng.uniform(0, two_pi)
        X, Y, Z = (two_pi * x[d] / ext[d] for d in range(3))
        out["vel"] = [(torch.sin(X + ph) * torch.cos(Y) * torch.cos(Z)).to(dt_),
                      (-torch.cos(X + ph) * torch.sin(Y) * torch.cos(Z)).to(dt_),
                      (0.3 * torch.sin(X) * torch.cos(Y + ph) + 0 * Z).to(dt_)]
        umax = 2.3
    else:
        u = rng.normal(size=3)
        u = u / np.linalg.norm(u)
        out["u"] = tuple(float(v) for v in u)
        umax = float(np.abs(u).sum())
    out["dt"] = 0.5 * hmin / umax
    if case["diff"]:
        out["nu"] = 0.02 * hmin
        out["dt"] = 0.3 * hmin / umax
    return out


def front_fields(case, seed):
    """A front on a sphere at two radii (tanh-sphere parameters, periodic) and the velocity scale."""
    rng = np.random.default_rng([seed, 7])
    # the centre moves by whole blocks of the coarsest level: every seed's tree has as many leaves
    c = [v + k / (1 << case["base"]) for v, k in zip((0.513, 0.478, 0.491), rng.integers(0, 1 << case["base"], 3).tolist())]
    width = 6.0 / (case["nb"] << case["lmax"])  # six points of the finest level
    r = 0.304
    return [c + [r, width], c + [r + 0.4 / (1 << case["lmax"]), width]], rng.uniform(0.5, 1.0)


EPS = (1e-3, 1e-5)  # refine, coarsen


def prepare(case, seed):
    N, Nt = wavelet(case)
    lev, anc = tree(case)
    prec = mrgb.F32 if case["prec"] == "f32" else mrgb.F64
    op, nb = case["op"], case["nb"]
    kw = dict(precision=prec, device="cuda", independent_trees=case["tree"] == "batch",
              bounded=(1, 1, 1) if case["tree"] == "slab" else (0, 0, 0))
    if op == "adapt":
        lmax = case["lmax"]
        cap = max(512, int(16 * 8 ** (lmax - 3) * 8 if lmax < 4 else 3.2 * 4 ** (lmax - 4) * 900))
        g = mrgb.Grid(forest(case), case["len"], nb, case["base"], lmax, N, Nt, lev, anc, nfields=4, capacity=cap, **kw)
        fronts, scale = front_fields(case, seed)
        for _ in range(lmax + 2):  # the initial grid: sample, refine, until nothing refines
            g.field_set(0, mrgb.INIT_TANH_SPHERE, fronts[0])
            if g.adapt_iter(0, *EPS, flags=mrgb.ADAPT_REFINE) == 0:
                break
        g.field_set(0, mrgb.INIT_TANH_SPHERE, fronts[0])
        for d in range(3):
            g.field_set(1 + d, mrgb.INIT_TAYLOR_GREEN, [d, scale, 0.3])
        g.adapt(0, *EPS)
        return {"g": g, "op": op, "fronts": fronts}
    x = inputs(case, seed)
    vel = "vel" in x
    g = mrgb.Grid(forest(case), case["len"], nb, 0, int(lev.max()), N, Nt, lev, anc, nfields=4 if vel else 1,
                  velocity=vel, fixed_tree=op not in ("crit",), **kw)
    g.field_copy_in(0, x["phi"])
    for d in range(3 if vel else 0):
        g.field_copy_in(1 + d, x["vel"][d].contiguous())
    if case["diff"]:
        g.set_diffusion(x["nu"], case["diff"])
    s = {"g": g, "op": op, "phi": g.field_view(0), "dt": x["dt"], "u": x.get("u"), "scheme": SCHEME[case["scheme"]]}
    if op == "ghost":
        s["shell"], W = case["shell"], nb + 2 * case["shell"]
        s["pad"] = torch.empty((len(lev), W, W, W), dtype=dtype(case), device="cuda")
    if op == "crit":
        s["norms"] = torch.empty(len(lev), dtype=torch.float64, device="cuda")
    return s


def run(state):
    g, op = state["g"], state["op"]
    if op == "step":
        g.step(0, state["dt"], state["u"], state["scheme"])
        return state["phi"]
    if op == "vel":
        g.step_vel(0, state["dt"], (1, 2, 3), state["scheme"])
        return state["phi"]
    if op == "loop":
        dt = g.dt(0.5, vel_fids=(1, 2, 3))
        g.step_vel(0, dt, (1, 2, 3), state["scheme"])
        return {"phi": state["phi"], "dt": dt, "mass": g.mass(0)}
    if op == "ghost":
        return {"pad": g.ghost_fill(0, state["shell"], state["pad"]), "phi": state["phi"]}
    if op == "crit":
        return {"norms": g.criterion(0, state["norms"]), "phi": state["phi"]}
    for k in (1, 0):  # the front moves and the tree follows it, then back
        g.field_set(0, mrgb.INIT_TANH_SPHERE, state["fronts"][k])
        g.adapt(0, *EPS)
    lev, anc, _ = g.leaves()
    return {"lev": lev, "anc": anc, "fields": [g.field_view(f) for f in range(4)]}


def work(case):
    N, Nt = wavelet(case)
    es, nb = (4 if case["prec"] == "f32" else 8), case["nb"]
    if case["op"] == "adapt":
        # blocks within one of the front on the finest level; every field read and written by each adaptation
        n = int(1.13 * 4 ** case["lmax"] * 3.5 * 1.3)
        pts = n * nb ** 3
        return {"bytes": float(2 * 4 * 2 * es * pts), "flops": float(2 * 2 * 3 * 4 * N * pts)}
    n = len(tree(case)[0])
    pts = n * nb ** 3
    if case["op"] == "ghost":
        W = nb + 2 * case["shell"]
        return {"bytes": float(es * (pts + n * W ** 3)), "flops": float(n * (W ** 3 - nb ** 3) * 2 * N)}
    if case["op"] == "crit":
        return {"bytes": float(es * pts + 8 * n), "flops": float(3 * 2 * N * pts)}
    flops = {"wenoz5": 235, "cons5": 60, "cons3": 35}[case["scheme"]] + {0: 0, 2: 14, 4: 30}[case["diff"]]
    fields = 2 + (3 if case["op"] in ("vel", "loop") else 0)
    return {"bytes": float(fields * es * pts), "flops": float(3 * flops * pts)}


# --------------------------------------------------------- the same in 64 bits
H = {(2, 2): {0: 3 / 4, 1: 1 / 4, 2: -1 / 8}, (4, 2): {0: 23 / 32, 1: 1 / 4, 2: -1 / 8, 4: 1 / 64},
     (6, 2): {0: 181 / 256, 1: 1 / 4, 2: -125 / 1024, 4: 11 / 512, 6: -3 / 1024}}
PREDICT = {2: {1: 1 / 2}, 4: {1: 9 / 16, 3: -1 / 16}, 6: {1: 75 / 128, 3: -25 / 256, 5: 3 / 256}}


def adapt_shell(N, Nt):
    h, g, ef = (N if Nt else 0), N - 1, (N - 1 if Nt else N - 2)
    reach = [p + (g if p & 1 else h) for p in range(ef + 1)] + [p + (g if (p + 1) & 1 else h) for p in range(ef + 2)]
    return max(reach + [N // 2, h])


def internal_shell(N, Nt, G, nb):
    h = N if Nt else 0
    return max(G, h, N - 1, 2 * G + h - nb)


def tap(f, ax, table, at, centre):
    """sum_t table[|t|] f[at + t] along axis ax (at: positions), f's centre weight replaced by `centre`."""
    s = None if centre == 0 else centre * f.index_select(ax, at)
    for t, w in table.items():
        if t:
            v = w * (f.index_select(ax, at - t) + f.index_select(ax, at + t))
            s = v if s is None else s + v
    return s


class Forest:
    """Leaves in Morton order with the block-wise reconstruction in 64-bit torch."""

    def __init__(self, case, lev, anc):
        self.nt, self.nb, self.len = forest(case), case["nb"], case["len"]
        self.N, self.Nt = wavelet(case)
        self.batch, self.bounded = case["tree"] == "batch", case["tree"] == "slab"
        dev = device()
        self.lev, self.anc = (torch.as_tensor(np.asarray(v, np.int64), device=dev) for v in (lev, anc))
        self.M = int(lev.max())
        m = torch.zeros([self.nt[d] << self.M for d in (2, 1, 0)], dtype=torch.int64, device=dev)
        for L in np.unique(lev):
            i = torch.nonzero(self.lev == int(L))[:, 0]
            s, a = 1 << (self.M - int(L)), self.anc[i]
            V = torch.full([self.nt[d] << int(L) for d in (2, 1, 0)], -1, dtype=torch.int64, device=dev)
            V[a[:, 2], a[:, 1], a[:, 0]] = i
            V = V.repeat_interleave(s, 0).repeat_interleave(s, 1).repeat_interleave(s, 2)
            m = torch.where(V >= 0, V, m)
        self.map = m
        self.ef = self.N - 1 if self.Nt else self.N - 2

    def owners(self, ids, L, lo, hi):
        """Owner leaf of the level-L points [lo, hi)^3 around the leaves ids (all such that their first point
        is a point of level L), and the wrapped coordinates per axis."""
        p = torch.arange(lo, hi, device=self.map.device)
        g = []
        for d in range(3):
            a = self.anc[ids, d] * self.nb
            sh = L - self.lev[ids]
            a = torch.where(sh >= 0, a << sh.clamp(min=0), a >> (-sh).clamp(min=0))
            P = (1 if self.batch else self.nt[d]) * self.nb << L
            T = (self.anc[ids, d] >> self.lev[ids])[:, None] * P if self.batch else 0
            g.append(T + (a[:, None] + p - T) % P)
        c = [(v << (self.M - L)) // self.nb for v in g]
        return self.map[c[2][:, :, None, None], c[1][:, None, :, None], c[0][:, None, None, :]], g

    def read(self, f, o, g, L):
        """Values that the owners o hold at level-L points g (the coincident point of a finer owner)."""
        Lo, idx = self.lev[o], 0
        for d in (2, 1, 0):
            v = g[d].reshape([len(o)] + [-1 if k == 2 - d else 1 for k in range(3)])
            q = torch.where(Lo >= L, v << (Lo - L).clamp(min=0), v >> (L - Lo).clamp(min=0)) - self.anc[o, d] * self.nb
            idx = idx * self.nb + q.clamp(0, self.nb - 1)
        return f.reshape(-1)[o * self.nb ** 3 + idx]

    def beyond(self, P, ids, lo, n, L):
        """Polynomial values beyond the domain's faces from the N nearest points inside (axis by axis)."""
        if not self.bounded:
            return P
        N, W = self.N, P.shape[1]
        for d in range(3):
            ax = 3 - d
            for side in (0, 1):
                hit = self.anc[ids, d] == (0 if side == 0 else (self.nt[d] << L) - 1)
                pos = list(range(0, -lo)) if side == 0 else list(range(n - lo, W))
                nodes = [k - lo for k in (range(N) if side == 0 else range(n - N, n))]
                if not hit.any() or not pos:
                    continue
                w = torch.tensor([[float(np.prod([(p - b) / (a - b) for b in nodes if b != a])) for a in nodes]
                                  for p in pos], dtype=P.dtype, device=P.device)
                v = torch.tensordot(P[hit].index_select(ax, torch.tensor(nodes, device=P.device)).movedim(ax, 3), w.T, 1)
                P[hit] = P[hit].index_copy(ax, torch.tensor(pos, device=P.device), v.movedim(3, ax))
        return P

    def bands(self, cm):
        """[leaf, nb, nb, nb]: points of the substitution band for the coarser directions cm [leaf, 27]."""
        nb, i = self.nb, torch.arange(self.nb, device=cm.device)
        side = {-1: i < self.ef + 1, 0: i >= 0, 1: i >= nb - self.ef}
        out = torch.zeros((len(cm), nb, nb, nb), dtype=torch.bool, device=cm.device)
        for m in range(27):
            if m != 13 and cm[:, m].any():
                x, y, z = side[m % 3 - 1], side[m // 3 % 3 - 1], side[m // 9 - 1]
                out |= cm[:, m, None, None, None] & (z[:, None, None] & y[None, :, None] & x)
        return out

    def refine(self, T, lo, hi, qlo):
        """Zero-detail refinement of coarse values T (first point qlo) at the fine points [lo, hi)^3."""
        for ax in (1, 2, 3):
            c = torch.arange(lo, hi, device=T.device)
            even = T.index_select(ax, torch.div(c, 2, rounding_mode="floor") - qlo)
            odd = 0
            for t, w in PREDICT[self.N].items():
                for o in (-t, t):
                    odd = odd + w * T.index_select(ax, torch.div(c + o, 2, rounding_mode="floor") - qlo)
            T = torch.where((c & 1 == 1).reshape([-1 if k == ax else 1 for k in range(4)]), odd, even)
        return T

    def fill(self, f, G):
        """Padded blocks (shell G) of the field f and the field with its bands substituted."""
        nb, N, n, hb = self.nb, self.N, len(self.lev), self.nb // 2
        Gi = internal_shell(N, self.Nt, G, nb)
        W = nb + 2 * Gi
        P = torch.empty((n, W, W, W), dtype=torch.float64, device=f.device)
        C = torch.empty((n, hb, hb, hb), dtype=torch.float64, device=f.device)
        qlo = -(Gi + N) // 2 - 1
        qhi = (nb + Gi + N) // 2 + 1
        chunks = []
        for L in torch.unique(self.lev).tolist():
            chunks += [(L, ids) for ids in torch.nonzero(self.lev == L)[:, 0].split(max(1, int(2.5e7) // W ** 3))]
        for L, ids in chunks:
            o, g = self.owners(ids, L, -Gi, nb + Gi)
            A = self.read(f, o, g, L)
            at = [Gi - 1, Gi, Gi + nb]
            near = torch.stack([self.lev[o[:, at[m // 9], at[m // 3 % 3], at[m % 3]]] < L for m in range(27)], 1)
            if self.bounded:
                for m in range(27):
                    for d, s in enumerate((m % 3 - 1, m // 3 % 3 - 1, m // 9 - 1)):
                        if s:
                            near[:, m] &= self.anc[ids, d] != (0 if s < 0 else (self.nt[d] << L) - 1)
            if near.any():
                oq, gq = self.owners(ids, L - 1, qlo, qhi)
                T = self.beyond(self.read(f, oq, gq, L - 1), ids, qlo, hb, L)
                A = torch.where(self.lev[o] < L, self.refine(T, -Gi, nb + Gi, qlo), A)
            A = self.beyond(A, ids, -Gi, nb, L)
            if near.any():
                band, i = self.bands(near), torch.arange(nb, device=f.device)
                deg = (i & 1)[:, None, None] + (i & 1)[None, :, None] + (i & 1)
                for k in (1, 2, 3):
                    B = A
                    for ax in (1, 2, 3):  # the detail along every odd dimension
                        c = torch.arange(W, device=f.device).clamp(N - 1, W - N)
                        D = tap(B, ax, {t: -w for t, w in PREDICT[N].items()}, c, 1.0)
                        odd = ((torch.arange(W, device=f.device) - Gi) & 1 == 1)
                        B = torch.where(odd.reshape([-1 if j == ax else 1 for j in range(4)]), D, B)
                    s = slice(Gi, Gi + nb)
                    A[:, s, s, s] = torch.where(band & (deg == k), A[:, s, s, s] - B[:, s, s, s], A[:, s, s, s])
            P[ids] = A
            B, c = A, Gi + 2 * torch.arange(hb, device=f.device)
            for ax in (1, 2, 3):
                B = tap(B, ax, H[(N, 2)], c, H[(N, 2)][0]) if self.Nt else B.index_select(ax, c)
            C[ids] = B
        for L, ids in chunks:
            o, g = self.owners(ids, L, -Gi, nb + Gi)
            fine, idx = self.lev[o] > L, 0
            if fine.any():
                for d in (2, 1, 0):
                    v = g[d].reshape([len(o)] + [-1 if k == 2 - d else 1 for k in range(3)])
                    idx = idx * hb + torch.div(v * 2 - self.anc[o, d] * nb, 2, rounding_mode="floor").clamp(0, hb - 1)
                P[ids] = torch.where(fine, C.reshape(-1)[o * hb ** 3 + idx], P[ids])
            P[ids] = self.beyond(P[ids], ids, -Gi, nb, L)
        s, e = slice(Gi, Gi + nb), slice(Gi - G, Gi + nb + G)
        return P[:, e, e, e], P[:, s, s, s].clone()

    def norms(self, f):
        G = adapt_shell(self.N, self.Nt)
        P, new = self.fill(f, G)
        r = torch.arange(-self.ef, self.nb + self.ef + 1, device=f.device)
        odd = r & 1 == 1
        c = (r + G).clamp(0, P.shape[1] - 1)
        out = []
        for B in P.split(256):
            for ax in (1, 2, 3):
                pad = [0, 0] * (3 - ax) + [self.N, self.N]
                Q = torch.nn.functional.pad(B, pad)
                D = tap(Q, ax, {t: -w for t, w in PREDICT[self.N].items()}, c + self.N, 1.0)
                S = tap(Q, ax, H[(self.N, 2)], c + self.N, H[(self.N, 2)][0]) if self.Nt else B.index_select(ax, c)
                B = torch.where(odd.reshape([-1 if j == ax else 1 for j in range(4)]), D, S)
            some = odd[:, None, None] | odd[None, :, None] | odd
            out.append(torch.where(some, B.abs(), torch.zeros_like(B)).amax((1, 2, 3)))
        return torch.cat(out), new


def flux(scheme, f, left):
    a, b, c, d, e = (torch.where(left, f[k], f[5 - k]) for k in range(5))
    if scheme == "cons3":
        return (-0.5 * b + 1.5 * c) / 3 + 2 * (0.5 * c + 0.5 * d) / 3
    s = [a / 3 - 7 * b / 6 + 11 * c / 6, -b / 6 + 5 * c / 6 + d / 3, c / 3 + 5 * d / 6 - e / 6]
    if scheme == "cons5":
        return 0.1 * s[0] + 0.6 * s[1] + 0.3 * s[2]
    t = [a - 4 * b + 3 * c, d - b, -3 * c + 4 * d - e]
    u = [a - 2 * b + c, b - 2 * c + d, c - 2 * d + e]
    be = [0.25 * t[k] ** 2 + 13 / 12 * u[k] ** 2 for k in range(3)]
    tau = (be[0] - be[2]).abs()
    w = [g * (1 + (tau / (be[k] + 1e-30)).clamp(max=1e15) ** 2) for k, g in enumerate((0.1, 0.6, 0.3))]
    return (w[0] * s[0] + w[1] * s[1] + w[2] * s[2]) / (w[0] + w[1] + w[2])


def step64(case, T, phi, vel, u, dt, nu):
    """One RK3-TVD step: ghosts, conservative upwind fluxes (and Laplacian), stage."""
    nb, y, un = case["nb"], phi, None
    vp = [T.fill(T.fill(v, 3)[1], 3)[0] for v in vel] if vel else None
    h = T.len / (nb * (1 << T.lev).double())[:, None, None, None]
    for stage in range(3):
        P, sub = T.fill(y, 3)
        un = sub if stage == 0 else un
        y = torch.empty_like(sub)
        for b in range(0, len(P), 256):
            k, r = slice(b, b + 256), 0
            Pb, hb = P[k], h[k]
            for d in range(3):
                ax = 3 - d
                if not vel and u[d] == 0:
                    continue
                v = vp[d][k] if vel else torch.full_like(Pb, u[d])
                line, vl = (X.narrow(1, 0 if ax == 1 else 3, nb + 6 if ax == 1 else nb)
                            .narrow(2, 0 if ax == 2 else 3, nb + 6 if ax == 2 else nb)
                            .narrow(3, 0 if ax == 3 else 3, nb + 6 if ax == 3 else nb) for X in (v * Pb, v))
                F = flux(case["scheme"], [line.narrow(ax, m, nb + 1) for m in range(6)],
                         vl.narrow(ax, 2, nb + 1) + vl.narrow(ax, 3, nb + 1) >= 0)
                r = r - (F.narrow(ax, 1, nb) - F.narrow(ax, 0, nb)) / hb
            for d in range(3 if case["diff"] else 0):
                at = [slice(3, 3 + nb)] * 3
                p = [Pb[(slice(None), *[slice(3 + m, 3 + m + nb) if j == d else at[j] for j in range(3)])] for m in range(-2, 3)]
                lap = p[1] - 2 * p[2] + p[3] if case["diff"] == 2 else (16 * (p[1] + p[3]) - p[0] - p[4] - 30 * p[2]) / 12
                r = r + nu * lap / hb ** 2
            v = sub[k] + dt * r
            y[k] = v if stage == 0 else 0.75 * un[k] + 0.25 * v if stage == 1 else un[k] / 3 + 2 * v / 3
    return y


def exact(case, seed):
    lev, anc = tree(case)
    nb = case["nb"]
    # the remeshing loop and the largest grids take longer than this is worth
    if case["op"] == "adapt" or len(lev) * nb ** 3 > 6e7:
        return None
    T, x = Forest(case, lev, anc), inputs(case, seed)
    phi = x["phi"].double()
    if case["op"] == "ghost":
        pad, sub = T.fill(phi, case["shell"])
        return {"pad": pad.contiguous(), "phi": sub}
    if case["op"] == "crit":
        n, sub = T.norms(phi)
        return {"norms": n, "phi": sub}
    vel = [v.double().expand(phi.shape).contiguous() for v in x["vel"]] if "vel" in x else None
    dt = x["dt"]
    if case["op"] == "loop":
        umax = float((vel[0].abs() + vel[1].abs() + vel[2].abs()).max())
        dt = 0.5 * (case["len"] / (nb * 2.0 ** int(lev.max()))) / umax
    y = step64(case, T, phi, vel, x.get("u"), dt, x.get("nu"))
    if case["op"] == "loop":
        h = case["len"] / (nb * (1 << T.lev).double())
        return {"phi": y, "dt": dt, "mass": float((y.sum((1, 2, 3)) * h ** 3).sum())}
    return y

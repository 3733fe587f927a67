"""What a user of this library waits for: force steps and integrator runs through the public entry points.

Every case is one pass of a call (or of the four phase calls) of `paper_0912_1786_gb300.evol` on device
arrays, over the particle sets of `paper_0912_1786_gb300.workloads`.  A pass starts from the same state each
time: the starting guesses of the lengths (and, for the integrators, positions, velocities and internal
energies) are restored by device copies first, since the calls update them in place.

`exact` evaluates the same method in FP64 with torch alone: the oct-tree of cubes, the length equations by
bisection, the opening criterion, the far and pair terms and the leapfrog, on the same inputs.
"""
import math

import numpy as np
import torch

from paper_0912_1786_gb300 import evol as E
from paper_0912_1786_gb300 import workloads as W
from paper_0912_1786_gb300.device import DeviceSet

GRAV_OUT = ["ax", "ay", "az", "pot", "ups", "X"]
GAS_OUT = ["rho", "P", "c", "omega", "zeta", "dudt"]
STATE_KEYS = ["x", "y", "z", "vx", "vy", "vz", "u", "h", "eps"]
# the global step's criteria (Sect. 4.2), as a run of the gas sphere takes them
CRITERIA = dict(eta_acc=0.1, eta_courant=0.1, eta_u=0.1, dt_min=0.0, dt_max=0.01)
KDK_DT = 1e-4                      # the fixed step of the shock-tube run
JITTER = 0.25                      # of a lattice spacing: as irregular as the glass of the paper's tube
VARIANTS = dict(visc_form=1, balsara=1, variable_alpha=1, conduction=1)


# ---- the cases --------------------------------------------------------------------------------------

def listed():
    return [
        # a small test problem, or one of the many short steps of a parameter study: launches and latency
        {"name": "gas_sphere_1000", "kind": "gas_sphere", "n": 1000, "leaf": 8, "group": 0},
        # the adiabatic collapse test at its usual small size
        {"name": "gas_sphere_4096", "kind": "gas_sphere", "n": 4096, "leaf": 8, "group": 0},
        # the four phase calls one after the other (tree, density, gravity, SPH forces), as a program
        # with its own integrator uses them; an odd size
        {"name": "phases_30011", "kind": "phases", "n": 30011, "leaf": 8, "group": 0},
        # a small galaxy (halo + gas) with the default cost parameters; ragged sizes
        {"name": "halo_gas_49k", "kind": "halo_gas", "n_dm": 32771, "n_gas": 16381, "leaf": 8, "group": 0},
        # the production force step: halo + gas at the autotuned leaf and group sizes
        {"name": "halo_gas_3m", "kind": "halo_gas", "n_dm": 1 << 21, "n_gas": 1 << 20, "leaf": 24, "group": 16},
        # the mixed-precision form, for energy-conservation studies
        {"name": "halo_gas_mixed_393k", "kind": "halo_gas", "n_dm": 1 << 18, "n_gas": 1 << 17, "leaf": 24, "group": 16,
         "mixed": True},
        # every dissipation variant on, moving gas
        {"name": "halo_gas_dissipation_393k", "kind": "halo_gas", "n_dm": 1 << 18, "n_gas": 1 << 17, "leaf": 24,
         "group": 16, "dissipation": True},
        # collisionless N-body: gravity alone with adaptive softening
        {"name": "plummer_1m", "kind": "plummer", "n": 1 << 20, "theta": 0.6, "leaf": 16, "group": 16},
        # SPH alone in a slab periodic on two axes: a run of fixed leapfrog steps (the 3-D shock tube)
        {"name": "shock_tube_kdk_1m", "kind": "shock_tube", "a": 55, "b": 35, "steps": 4, "leaf": 32, "group": 16},
        # many independent systems in one call
        {"name": "ensemble_64", "kind": "ensemble", "systems": 64, "log2_min": 10.0, "log2_max": 17.0, "layout": 5,
         "leaf": 16, "group": 16},
        # cosmological box: periodic gravity by Ewald summation
        {"name": "periodic_box_262k", "kind": "periodic_box", "n": 1 << 18, "leaf": 8, "group": 0},
        # the global-time-step integrator: criteria, predicted lengths and velocities, a few steps a call
        {"name": "run_131k", "kind": "run", "n": 131071, "steps": 4, "leaf": 16, "group": 8},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["gas_sphere", "gas_sphere", "phases", "halo_gas", "halo_gas", "plummer", "shock_tube",
                       "ensemble", "periodic_box", "run"])
    c = {"kind": kind, "leaf": rng.choice([8, 8, 16, 24, 32]), "group": rng.choice([0, 0, 8, 16])}
    if kind == "gas_sphere":
        c["n"] = size(700, 1 << 20)
    elif kind == "phases":
        c["n"] = size(1000, 1 << 18)
    elif kind == "halo_gas":
        form = rng.choice(["plain", "plain", "mixed", "dissipation"])
        c["n_dm"] = size(1 << 13, 1 << 21 if form == "plain" else 1 << 19)
        c["n_gas"] = max(1000, int(c["n_dm"] * rng.uniform(0.25, 0.5)))
        if form != "plain":
            c[form] = True
    elif kind == "plummer":
        c["n"] = size(2000, 1 << 20)
        c["theta"] = rng.choice([0.4, 0.5, 0.6, 0.8])
    elif kind == "shock_tube":
        c["a"] = rng.randint(11, 52)
        c["b"] = max(7, int(round(c["a"] * 35 / 55)))
        c["steps"] = rng.randint(1, 4)
    elif kind == "ensemble":
        c["systems"] = rng.randint(2, 64)
        c["log2_min"], c["log2_max"], c["layout"] = 10.0, rng.uniform(12.0, 16.5), rng.randrange(1 << 16)
    elif kind == "periodic_box":
        c["n"] = size(2000, 1 << 18)
    else:
        c["n"] = size(1000, 1 << 17)
        c["steps"] = rng.randint(1, 4)
    return c


def _counts(case):
    """(particles, gas particles) of a case."""
    k = case["kind"]
    if k == "halo_gas":
        return case["n_dm"] + case["n_gas"], case["n_gas"]
    if k == "shock_tube":
        n = 5 * case["a"] ** 3 + 5 * case["b"] ** 3
        return n, n
    if k == "ensemble":
        n = int(_system_sizes(case).sum())
        return n, n
    return case["n"], 0 if k in ("plummer", "periodic_box") else case["n"]


def _system_sizes(case):
    r = np.random.default_rng(case["layout"])
    return np.floor(2.0 ** r.uniform(case["log2_min"], case["log2_max"], case["systems"])).astype(np.int64)


def work(case):
    n, ng = _counts(case)
    k = case["kind"]
    grav = k != "shock_tube"
    theta = case.get("theta", 0.6 if k == "plummer" else 0.5)
    # inputs and outputs of one force step, 4 bytes each (shock_tube: ax ay az; gas: h u and its outputs)
    per, per_gas = (8 + len(GRAV_OUT) + 1 if grav else 7 + 3), (2 + len(GAS_OUT) + 1)
    evaluations = case.get("steps", 0) + 1
    # interactions per particle, fitted to the counts of the listed sets, and their operations: far node 53,
    # Newtonian pair 19, softened pair 89, SPH pair 85
    log2 = math.log2(max(n / case.get("systems", 1), 600.0))
    far = {"halo_gas": 680 + 86 * log2, "plummer": 73 * log2 * (0.6 / theta) ** 2.2, "periodic_box": 71 * log2,
           "shock_tube": 0.0}.get(k, 88 * (log2 - 8.2))
    flops = n * (far * 53 + 250 * 19 + 50 * 89) if grav else 0.0
    flops += ng * 50 * 85
    # the length equations: three sweeps over the neighbours (about 12 operations each)
    flops += (n * (1 if grav else 0) + ng) * 3 * 60 * 12
    return {"bytes": 4.0 * evaluations * (n * per + ng * per_gas), "flops": float(evaluations * flops)}


# ---- a user's program -------------------------------------------------------------------------------

def _params(case, **kw):
    return W.Params(leaf_size=case["leaf"], length_group=case["group"], **kw)


def _workload(case, seed):
    k = case["kind"]
    if k in ("gas_sphere", "phases"):
        return W.evrard_sphere(case["n"], seed=seed, sigma_v=0.1, params=_params(case))
    if k == "run":
        return W.hot_core(W.evrard_sphere(case["n"], seed=seed, sigma_v=0.05, params=_params(case)), factor=3.0)
    if k == "halo_gas":
        w = W.hernquist_gas(case["n_dm"], case["n_gas"], seed=seed, params=_params(case))
        if case.get("dissipation"):
            w = W.with_dissipation(w, seed=seed + 1, sigma_v=0.1, **VARIANTS)
        return w
    if k == "plummer":
        return W.plummer(case["n"], seed=seed, theta=case["theta"],
                         params=_params(case, theta=case["theta"], n_nei_grav=32.0, sph=0))
    if k == "shock_tube":
        a, b = case["a"], case["b"]
        return W.shock_tube(seed=seed, left=(5 * a, a, a), right=(5 * b, b, b), jitter=JITTER,
                            params=_params(case, gravity=0, adaptive_softening=0, periodic_mask=0b110,
                                           periodic_hi=(1.0, 0.1, 0.1)))
    if k == "ensemble":
        sizes = _system_sizes(case)
        parts = [W.evrard_sphere(int(s), seed=seed + 1009 * i, params=_params(case)) for i, s in enumerate(sizes)]
        cat = {f: np.concatenate([getattr(w, f) for w in parts]) for f in parts[0].arrays()}
        off = np.concatenate([[0], np.cumsum(sizes)])
        return W.Workload("ensemble", **cat, n_gas=int(off[-1]), params=parts[0].params, sys_offsets=off)
    return W.periodic_box(case["n"], seed=seed,
                          params=_params(case, sph=0, n_nei_grav=32.0, periodic_mask=7))


class Program:
    """A context, the particles' device arrays and the outputs, held as a user's program holds them."""

    def __init__(self, case, seed):
        w = _workload(case, seed)
        self.case = case
        self.gravity, self.gas = bool(w.params.gravity), w.n_gas > 0 and bool(w.params.sph)
        names = (GRAV_OUT if self.gravity else ["ax", "ay", "az"]) + (GAS_OUT if self.gas else [])
        if case.get("dissipation"):
            names = names + ["dalpha", "dalpha_u"]
        self.ds = DeviceSet(w, outputs=names,
                            precision=E.EVOL_FP32_MIXED if case.get("mixed") else E.EVOL_FP32_PLAIN)
        self.offsets = None if w.sys_offsets is None else [int(v) for v in w.sys_offsets]
        self.lengths = (["h"] if self.gas else []) + (["eps"] if self.gravity else [])
        self.start = ({q: self.ds.inp[q].clone() for q in STATE_KEYS if q in self.ds.inp}
                      if "steps" in case else {q: self.ds.inp[q].clone() for q in self.lengths})
        self.integrator = E.make_integrator(**CRITERIA)
        self.ctx = E.evol_create(w.n, torch.cuda.current_stream().cuda_stream)

    def __del__(self):
        if getattr(self, "ctx", None) is not None:
            E.evol_destroy(self.ctx)
            self.ctx = None


def prepare(case, seed):
    return Program(case, seed)


def run(s):
    ds, kind = s.ds, s.case["kind"]
    for q, t in s.start.items():
        ds.inp[q].copy_(t)
    args = (s.ctx, ds.particles, ds.params)
    out = dict(ds.out)
    if kind == "phases":
        E.evol_build_tree(*args)
        E.evol_sph_density(*args, ds.outputs)
        E.evol_gravity(*args, ds.outputs)
        E.evol_sph_forces(*args, ds.outputs)
    elif kind == "ensemble":
        E.evol_step_batched(s.ctx, s.offsets, ds.particles, ds.params, ds.outputs)
    elif kind == "shock_tube":
        E.evol_kdk(*args, ds.outputs, KDK_DT, s.case["steps"])
    elif kind == "run":
        out["time"], out["dt"] = E.evol_run(*args, s.integrator, ds.outputs, s.case["steps"], 0.0)
    else:
        E.evol_step(*args, ds.outputs)
    keys = [q for q in STATE_KEYS if q in s.start] if "steps" in s.case else s.lengths
    out.update({"in_" + q: ds.inp[q] for q in keys if not (q == "eps" and not s.gravity)})
    return out


# ---- the same in FP64 (torch alone) -----------------------------------------------------------------

LEVELS = 21
CHUNK = 1 << 15                    # particles walked together


def _wrap(d, length):
    return d - length * torch.round(d / length) if length else d


def _spread(q):
    q = (q | (q << 32)) & 0x1F00000000FFFF
    q = (q | (q << 16)) & 0x1F0000FF0000FF
    q = (q | (q << 8)) & 0x100F00F00F00F00F
    q = (q | (q << 4)) & 0x10C30C30C30C30C3
    return (q | (q << 2)) & 0x1249249249249249


def _segments(values, counts):
    """Sums of consecutive runs of `values` with the given lengths."""
    return torch.segment_reduce(values, "sum", lengths=counts, unsafe=True, initial=0.0)


def _expand(owner, first, count):
    """For rows (owner, first, count): every index first .. first + count - 1 with its row's owner."""
    rows = torch.repeat_interleave(torch.arange(len(count), device=count.device), count)
    start = torch.cumsum(count, 0) - count
    return owner[rows], first[rows] + torch.arange(len(rows), device=rows.device) - start[rows]


class Tree:
    """Cubes split while they hold more than `leaf` particles, level by level; particles in key order."""

    def __init__(self, pos, m, gas, leaf):
        lo = pos.min(0).values
        ext = float((pos.max(0).values - lo).max())
        fr, ex = math.frexp(ext * (1.0 + 2.0 ** -20))
        self.side = (math.ldexp(1.0, ex - 1) if fr == 0.5 else math.ldexp(1.0, ex)) if ext > 0 else 1.0
        q = torch.floor((pos - lo) * (2.0 ** LEVELS / self.side)).clamp(0, 2 ** LEVELS - 1).long()
        key = (_spread(q[:, 0]) << 2) | (_spread(q[:, 1]) << 1) | _spread(q[:, 2])
        key, self.perm = torch.sort(key, stable=True)
        self.pos, self.m, self.gas = pos[self.perm], m[self.perm], gas[self.perm]
        dev, n = pos.device, len(m)
        beg, end = torch.zeros(1, dtype=torch.long, device=dev), torch.full((1,), n, device=dev)
        inside = torch.zeros(n, dtype=torch.long, device=dev)        # this level's node of each particle, -1: none
        cols = {f: [] for f in ("beg", "end", "child", "nch", "M", "com", "Q", "delta", "side", "mid", "half", "gas")}
        total = 0
        self.level = []                                                # (particles of the level, their node ids)
        for lev in range(LEVELS + 1):
            k = len(beg)
            at = torch.nonzero(inside >= 0).flatten()
            nid, p, mm = inside[at], self.pos[at], self.m[at]
            self.level.append((at, nid + total))
            M = torch.zeros(k, dtype=torch.double, device=dev).index_add_(0, nid, mm)
            com = torch.zeros(k, 3, dtype=torch.double, device=dev).index_add_(0, nid, mm[:, None] * p) / M[:, None]
            d = p - com[nid]
            d2 = (d * d).sum(1)
            terms = [3 * d[:, 0] ** 2 - d2, 3 * d[:, 1] ** 2 - d2, 3 * d[:, 2] ** 2 - d2, 3 * d[:, 0] * d[:, 1],
                     3 * d[:, 0] * d[:, 2], 3 * d[:, 1] * d[:, 2]]
            Q = torch.zeros(k, 6, dtype=torch.double, device=dev).index_add_(0, nid, mm[:, None] * torch.stack(terms, 1))
            e3 = nid[:, None].expand(-1, 3)
            bmin = torch.full((k, 3), math.inf, dtype=torch.double, device=dev).scatter_reduce_(0, e3, p, "amin")
            bmax = torch.full((k, 3), -math.inf, dtype=torch.double, device=dev).scatter_reduce_(0, e3, p, "amax")
            s = math.ldexp(self.side, -lev)
            cell = torch.floor((self.pos[beg] - lo) * (2.0 ** LEVELS / self.side)).clamp(0, 2 ** LEVELS - 1).long() >> (LEVELS - lev)
            delta = (com - (lo + (cell.double() + 0.5) * s)).norm(dim=1)
            split = (end - beg > leaf) & (lev < LEVELS)
            nch, child = torch.zeros_like(beg), torch.zeros_like(beg)
            if bool(split.any()):
                inside = torch.where((inside >= 0) & split[inside.clamp(min=0)], inside, -1)
                octant = key >> (3 * (LEVELS - lev - 1))
                first = inside >= 0
                first[1:] &= (octant[1:] != octant[:-1]) | (inside[1:] != inside[:-1])
                b2 = torch.nonzero(first).flatten()
                par = inside[b2]
                e2 = torch.minimum(torch.cat([b2[1:], torch.full((1,), n, device=dev)]), end[par])
                nch = torch.bincount(par, minlength=k)
                child = torch.cumsum(nch, 0) - nch + total + k
                inside = torch.where(inside >= 0, torch.cumsum(first.long(), 0) - 1, -1)
            for f, v in (("beg", beg), ("end", end), ("child", child), ("nch", nch), ("M", M), ("com", com), ("Q", Q),
                         ("delta", delta), ("side", torch.full_like(M, s)), ("mid", 0.5 * (bmin + bmax)),
                         ("half", 0.5 * (bmax - bmin)),
                         ("gas", torch.zeros(k, device=dev).index_add_(0, nid, self.gas[at].float()) > 0)):
                cols[f].append(v)
            total += k
            if not bool(split.any()):
                break
            beg, end = b2, e2
        for f, v in cols.items():
            setattr(self, "n_" + f, torch.cat(v))

    def node_max(self, values, of):
        out = torch.full((len(self.n_M),), -1.0, dtype=torch.double, device=values.device)
        for at, ids in self.level:
            keep = of[at]
            out.scatter_reduce_(0, ids[keep], values[at[keep]], "amax")
        return out


class Exact:
    """One force step in FP64 on the particles of a workload (positions etc. may change between steps)."""

    def __init__(self, w, mask=0, length=(0.0, 0.0, 0.0)):
        self.p, self.n, self.ng = w.params, w.n, w.n_gas
        self.len = [float(np.float32(v)) if (mask >> a) & 1 else 0.0 for a, v in enumerate(length)]
        self.ewald = _ewald_table() if mask == 7 and w.params.gravity else None

    def boxdist2(self, t, i, node):
        d = torch.stack([(_wrap(t.pos[i, a] - t.n_mid[node, a], self.len[a]).abs() - t.n_half[node, a]).clamp(min=0)
                         for a in range(3)], 1)
        return (d * d).sum(1)

    def vector(self, a, b):
        return torch.stack([_wrap(a[:, k] - b[:, k], self.len[k]) for k in range(3)], 1)

    def neighbours(self, t, i, R, gas_only):
        """(row, j, r): every j within R of particle i (rows ascending)."""
        row, node = torch.arange(len(i), device=i.device), torch.zeros_like(i)
        rows, js = [], []
        while len(row):
            keep = self.boxdist2(t, i[row], node) < R[row] ** 2
            if gas_only:
                keep &= t.n_gas[node]
            row, node = row[keep], node[keep]
            leaf = t.n_nch[node] == 0
            a, b = _expand(row[leaf], t.n_beg[node[leaf]], (t.n_end - t.n_beg)[node[leaf]])
            r = self.vector(t.pos[i[a]], t.pos[b]).norm(dim=1)
            keep = r < R[a]
            if gas_only:
                keep &= t.gas[b]
            rows.append(a[keep])
            js.append(b[keep])
            row, node = _expand(row[~leaf], t.n_child[node[~leaf]], t.n_nch[node[~leaf]])
        row, j = torch.cat(rows), torch.cat(js)
        row, o = torch.sort(row, stable=True)
        j = j[o]
        return row, j, self.vector(t.pos[i[row]], t.pos[j]).norm(dim=1)

    def solve(self, t, guess, nnei, gas_only, v=None):
        """Roots of L^3 n(L) = eta^3; the kernel sums there, and div v and |curl v| where v is given."""
        eta3 = 3.0 * nnei / (32.0 * math.pi)
        out = torch.zeros(8, len(t.m), dtype=torch.double, device=guess.device)
        todo = torch.nonzero(t.gas).flatten() if gas_only else torch.arange(len(t.m), device=guess.device)
        R = 2.6 * guess
        while len(todo):
            again = []
            for c0 in range(0, len(todo), CHUNK):
                i = todo[c0:c0 + CHUNK]
                row, j, r = self.neighbours(t, i, R[i], gas_only)
                cnt = torch.bincount(row, minlength=len(i))

                def f(L):
                    return _segments(_w(r / L[row]), cnt) / math.pi - eta3

                lo, hi = torch.zeros_like(R[i]), 0.5 * R[i]
                ok = f(hi) >= 0
                again.append(i[~ok])
                for _ in range(48):
                    mid = 0.5 * (lo + hi)
                    up = f(mid) >= 0
                    hi, lo = torch.where(up, mid, hi), torch.where(up, lo, mid)
                L = 0.5 * (lo + hi)
                u = r / L[row]
                w, uw, mj = _w(u), u * _dw(u), t.m[j]
                Sw, Suw = _segments(w, cnt), _segments(uw, cnt)
                vals = [L, -Suw / (3 * Sw)]
                if gas_only:
                    Smw, Smuw = _segments(mj * w, cnt), _segments(mj * uw, cnt)
                    vals += [Smw / (math.pi * L ** 3), (3 * Smw + Smuw) / (3 * Sw)]
                else:
                    vals += [-math.pi * L ** 2 * _segments(mj * _dphideps(u), cnt) / (3 * Sw), torch.zeros_like(L)]
                if v is not None:
                    d = self.vector(t.pos[i[row]], t.pos[j])
                    dv = v[i[row]] - v[j]
                    g = torch.where(r > 0, _dw(u) / r.clamp(min=1e-300), torch.zeros_like(r))
                    vals.append(3 * _segments((dv * d).sum(1) * g, cnt) / (L * Suw))
                    cr = torch.linalg.cross(dv, d, dim=1) * g[:, None]
                    vals.append(3 * torch.stack([_segments(cr[:, a].contiguous(), cnt) for a in range(3)], 1).norm(dim=1)
                                / (L * Suw.abs()))
                for k, x in enumerate(vals):
                    out[k, i[ok]] = x[ok]
            todo = torch.cat(again)
            R[todo] *= 1.5
        return out

    def __call__(self, pos, v, m, u, guess_h, guess_e, alpha=None, alpha_u=None, flow=False):
        p, n, ng, dev = self.p, self.n, self.ng, pos.device
        isgas = torch.arange(n, device=dev) < ng
        t = Tree(pos, m, isgas, p.leaf_size)
        o = t.perm
        srt = lambda x: x[o]
        S = {"v": srt(v), "u": srt(u)}
        res = {}
        if p.gravity:
            e = self.solve(t, srt(guess_e), p.n_nei_grav, False, S["v"] if flow else None)
            S.update(eps=e[0], ups=e[1], X=e[2])
            t.emax = t.node_max(2 * e[0], torch.ones_like(t.gas))
            res.update(in_eps=e[0], ups=e[1], X=e[2], divv_e=e[4])
        diss = p.visc_form or p.balsara or p.variable_alpha or p.conduction
        if ng and p.sph:
            hs = self.solve(t, srt(guess_h), p.n_nei_sph, True, S["v"] if flow or diss else None)
            P, c = (p.gamma - 1) * hs[2] * S["u"], torch.sqrt(p.gamma * (p.gamma - 1) * S["u"])
            S.update(h=hs[0], omega=hs[1], rho=hs[2], zeta=hs[3], divv=hs[4], P=P, c=c)
            S["Prho2"] = torch.where(t.gas, P / hs[2].clamp(min=1e-300) ** 2, torch.zeros_like(P))
            S["zo"] = torch.where(t.gas, hs[3] / hs[1], torch.zeros_like(P))
            t.hmax = t.node_max(2 * hs[0], t.gas)
            if diss:
                den = hs[4].abs() + hs[5] + p.balsara_eta * c / hs[0].clamp(min=1e-300)
                S.update(f=torch.where(den > 0, hs[4].abs() / den, torch.zeros_like(den)), alpha=srt(alpha),
                         alpha_u=srt(alpha_u))
            res.update(in_h=hs[0], omega=hs[1], rho=hs[2], zeta=hs[3], P=P, c=c, divv_h=hs[4])
        acc = torch.zeros(n, 8, dtype=torch.double, device=dev)      # a, pot, du/dt, max mu, max v_sig, lap u
        for c0 in range(0, n, CHUNK):
            i = torch.arange(c0, min(n, c0 + CHUNK), device=dev)
            self.forces(t, S, i, acc, bool(diss))
        if p.gravity:
            acc[:, 3] += p.G * t.m * -1.4 / S["eps"]
            if self.ewald is not None:
                acc[:, 3] += p.G * t.m * self.ewald[0, 0, 0, 3] / self.len[0]
        res.update(ax=acc[:, 0], ay=acc[:, 1], az=acc[:, 2], pot=acc[:, 3], dudt=acc[:, 4], mumax=acc[:, 5])
        if diss and ng:
            rate = torch.maximum(acc[:, 6], 2 * S["c"]) / (p.alpha_tau * S["h"])
            res["dalpha"] = -(S["alpha"] - p.alpha_min) * rate + p.alpha_source * S["f"] * (-S["divv"]).clamp(min=0)
            res["dalpha_u"] = -(S["alpha_u"] - p.alpha_u_min) * rate + S["h"] * acc[:, 7].abs() / torch.sqrt(S["u"])
        back = torch.empty_like(o)
        back[o] = torch.arange(n, device=dev)
        gas_len = {"in_h", "omega", "rho", "zeta", "P", "c", "dudt", "dalpha", "dalpha_u", "divv_h", "mumax"}
        return {k: x[back][:ng] if k in gas_len else x[back] for k, x in res.items()}

    def forces(self, t, S, i, acc, diss):
        p = self.p
        row, node = torch.arange(len(i), device=i.device), torch.zeros_like(i)

        def runs(row):                 # length of each particle's run of the ascending rows
            return torch.searchsorted(row, torch.arange(len(i) + 1, device=i.device)).diff()

        def add(col, runs, val):
            acc[i[0]:i[0] + len(i), col] += _segments(val.contiguous(), runs)

        near = []
        while len(row):
            ii = i[row]
            R = torch.zeros(len(row), dtype=torch.double, device=i.device)
            if p.gravity:
                R = torch.maximum(2 * S["eps"][ii], t.emax[node])
            if "h" in S:
                both = t.gas[ii] & t.n_gas[node]
                R = torch.where(both, torch.maximum(R, torch.maximum(2 * S["h"][ii], t.hmax[node])), R)
            far = self.boxdist2(t, ii, node) > R * R
            if p.gravity:
                dv = self.vector(t.pos[ii], t.n_com[node]) if self.ewald is not None else t.pos[ii] - t.n_com[node]
                far &= dv.norm(dim=1) > t.n_side[node] / p.theta + t.n_delta[node]
                if self.ewald is not None:
                    far &= t.n_side[node] <= 0.125 * self.len[0]
                d, k, r = dv[far], node[far], runs(row[far])
                q, M = t.n_Q[k], t.n_M[k]
                Qd = torch.stack([q[:, 0] * d[:, 0] + q[:, 3] * d[:, 1] + q[:, 4] * d[:, 2],
                                  q[:, 3] * d[:, 0] + q[:, 1] * d[:, 1] + q[:, 5] * d[:, 2],
                                  q[:, 4] * d[:, 0] + q[:, 5] * d[:, 1] + q[:, 2] * d[:, 2]], 1)
                dQd, di = (d * Qd).sum(1), 1 / d.norm(dim=1)
                a = (-M * di ** 3 - 2.5 * dQd * di ** 7)[:, None] * d + Qd * (di ** 5)[:, None]
                pot = -M * di - 0.5 * dQd * di ** 5
                if self.ewald is not None:
                    fe, ge = self.replicas(d)
                    a, pot = a + M[:, None] * fe, pot + M * ge
                for c in range(3):
                    add(c, r, p.G * a[:, c])
                add(3, r, p.G * pot)
            opened = ~far
            row, node = row[opened], node[opened]
            leaf = t.n_nch[node] == 0
            near.append((row[leaf], node[leaf]))
            row, node = _expand(row[~leaf], t.n_child[node[~leaf]], t.n_nch[node[~leaf]])
        row, node = torch.cat([a for a, _ in near]), torch.cat([b for _, b in near])
        row, o = torch.sort(row, stable=True)
        node = node[o]
        for part in range(0, len(row), 1 << 21):
            a, j = _expand(row[part:part + (1 << 21)], t.n_beg[node[part:part + (1 << 21)]],
                           (t.n_end - t.n_beg)[node[part:part + (1 << 21)]])
            keep = i[a] != j
            self.pairs(t, S, i, a[keep], j[keep], acc, runs, add, diss)

    def pairs(self, t, S, i, row, j, acc, runs, add, diss):
        p, ii = self.p, i[row]
        d = self.vector(t.pos[ii], t.pos[j])
        r2 = (d * d).sum(1)
        if p.gravity:
            r, mj, ei, ej = r2.sqrt(), t.m[j], S["eps"][ii], S["eps"][j]
            rs = r.clamp(min=1e-300)
            fg = -0.5 * mj * (_dphi(r / ei) / ei ** 2 + _dphi(r / ej) / ej ** 2)
            fg = fg - 0.5 / math.pi * (S["X"][ii] / S["ups"][ii] * _dw(r / ei) / ei ** 4 +
                                       mj / t.m[ii] * S["X"][j] / S["ups"][j] * _dw(r / ej) / ej ** 4)
            fg = torch.where(r > 0, fg / rs, torch.zeros_like(r))
            pot = mj * _phi(r / ei) / ei
            a = fg[:, None] * d
            if self.ewald is not None:
                fe, ge = self.replicas(d)
                a, pot = a + mj[:, None] * fe, pot + mj * ge
            seg = runs(row)
            for c in range(3):
                add(c, seg, p.G * a[:, c])
            add(3, seg, p.G * pot)
        if "h" not in S:
            return
        hit = t.gas[ii] & t.gas[j] & (r2 > 0) & (r2 < 4 * torch.maximum(S["h"][ii], S["h"][j]) ** 2)
        row, j, d = row[hit], j[hit], d[hit]
        ii, r = i[row], r2[hit].sqrt()
        hi, hj, mj, mi = S["h"][ii], S["h"][j], t.m[j], t.m[ii]
        gi, gj = _tc(r / hi) / (math.pi * hi ** 4), _tc(r / hj) / (math.pi * hj ** 4)
        fi, fj = 1 + S["zo"][ii] / mj, 1 + S["zo"][j] / mi
        vr = ((S["v"][ii] - S["v"][j]) * d).sum(1)
        cb, rb, hb = 0.5 * (S["c"][ii] + S["c"][j]), 0.5 * (S["rho"][ii] + S["rho"][j]), 0.5 * (hi + hj)
        mu = torch.where(vr < 0, hb * vr / (r * r + 0.01 * hb * hb), torch.zeros_like(vr))
        w = vr / r
        vsig = 2 * cb - w.clamp(max=0)
        al = 0.5 * (S["alpha"][ii] + S["alpha"][j]) if diss and p.variable_alpha else p.alpha
        visc = -al * vsig * w.clamp(max=0) / rb if p.visc_form else (-al * cb * mu + p.beta * mu * mu) / rb
        if p.balsara:
            visc = visc * 0.5 * (S["f"][ii] + S["f"][j])
        gbar, own = 0.5 * (gi * fi + gj * fj), S["Prho2"][ii] * fi * gi
        s = -mj * (own + S["Prho2"][j] * fj * gj + visc * gbar) / r
        seg = runs(row)
        for c in range(3):
            add(c, seg, s * d[:, c])
        heat = mj * (own + 0.5 * visc * gbar) * vr / r
        top = acc[i[0]:i[0] + len(i)]
        if p.conduction:
            du = S["u"][ii] - S["u"][j]
            heat = heat - mj * 0.5 * (S["alpha_u"][ii] + S["alpha_u"][j]) * vsig * du / rb * gbar.abs()
            add(7, seg, 2 * mj * du / S["rho"][j] * gbar.abs() / r)
        add(4, seg, heat)
        top[:, 5] = top[:, 5].scatter_reduce(0, row, mu.abs(), "amax")
        top[:, 6] = top[:, 6].scatter_reduce(0, row, vsig, "amax")

    def replicas(self, d):
        """The tabulated periodic correction (trilinear on the octant's grid), f and g for unit mass."""
        L, N = self.len[0], 64
        u = d.abs() / L * (2 * N)
        k = u.floor().clamp(0, N - 1).long()
        x = u - k
        out = torch.zeros(len(d), 4, dtype=torch.double, device=d.device)
        for c in range(8):
            o = [(c >> 2) & 1, (c >> 1) & 1, c & 1]
            wgt = torch.ones(len(d), dtype=torch.double, device=d.device)
            for a in range(3):
                wgt = wgt * (x[:, a] if o[a] else 1 - x[:, a])
            out += wgt[:, None] * self.ewald[k[:, 0] + o[0], k[:, 1] + o[1], k[:, 2] + o[2]]
        return torch.where(d < 0, -out[:, :3], out[:, :3]) / L ** 2, out[:, 3] / L


def _ewald_table():
    """(f, g) of the periodic correction (the series of Sect. 4.3, |n|, |h| < 5, omega = 2) for a unit cube."""
    g = torch.arange(65, dtype=torch.double, device="cuda") / 128.0
    x = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    w, sp = 2.0, math.sqrt(math.pi)
    F, G = torch.zeros_like(x), torch.full((len(x),), math.pi / w ** 2, dtype=torch.double, device="cuda")
    for a in range(-4, 5):
        for b in range(-4, 5):
            for c in range(-4, 5):
                n2 = a * a + b * b + c * c
                if n2 >= 25:
                    continue
                k = torch.tensor([a, b, c], dtype=torch.double, device="cuda")
                d = x - k
                r = d.norm(dim=1)
                z = w * r
                if n2 == 0:
                    rs = r.clamp(min=1e-300)
                    k3 = torch.where(z < 1e-3, 4 / (3 * sp) * w ** 3 * (1 - 0.6 * z * z),
                                     (torch.erf(z) - 2 * z / sp * torch.exp(-z * z)) / rs ** 3)
                    F += d * k3[:, None]
                    G += torch.where(z < 1e-3, 2 * w / sp * (1 - z * z / 3), torch.erf(z) / rs)
                else:
                    F -= d * ((torch.erfc(z) + 2 * z / sp * torch.exp(-z * z)) / r ** 3)[:, None]
                    G -= torch.erfc(z) / r
                    e, ph = math.exp(-(math.pi / w) ** 2 * n2), 2 * math.pi * (x @ k)
                    F -= (2 * e / n2 * torch.sin(ph))[:, None] * k
                    G -= e / (math.pi * n2) * torch.cos(ph)
    return torch.cat([F, G[:, None]], 1).reshape(65, 65, 65, 4)


# the kernel functions of r/L (Eqs. spline, softforce, softphi, dphidh and the Thomas-Couchman gradient)
def _w(u):
    return 0.25 * (2 - u).clamp(min=0) ** 3 - (1 - u).clamp(min=0) ** 3


def _dw(u):
    return -0.75 * (2 - u).clamp(min=0) ** 2 + 3 * (1 - u).clamp(min=0) ** 2


def _tc(u):
    return torch.where(u < 2 / 3, -torch.ones_like(u), _dw(u))


def _outer(u):
    return u.clamp(min=0.5)


def _dphi(u):
    o = _outer(u)
    return torch.where(u < 1, 4 / 3 * u - 1.2 * u ** 3 + 0.5 * u ** 4,
                       torch.where(u < 2, 8 / 3 * u - 3 * u ** 2 + 1.2 * u ** 3 - u ** 4 / 6 - 1 / (15 * o ** 2),
                                   1 / o ** 2))


def _phi(u):
    o = _outer(u)
    return torch.where(u < 1, 2 / 3 * u ** 2 - 0.3 * u ** 4 + 0.1 * u ** 5 - 1.4,
                       torch.where(u < 2, 4 / 3 * u ** 2 - u ** 3 + 0.3 * u ** 4 - u ** 5 / 30 - 1.6 + 1 / (15 * o),
                                   -1 / o))


def _dphideps(u):
    return torch.where(u < 1, -2 * u ** 2 + 1.5 * u ** 4 - 0.6 * u ** 5 + 1.4,
                       torch.where(u < 2, -4 * u ** 2 + 4 * u ** 3 - 1.5 * u ** 4 + 0.2 * u ** 5 + 1.6,
                                   torch.zeros_like(u)))


def exact(case, seed):
    n, ng = _counts(case)
    evaluations = case.get("steps", 0) + 1
    if n * evaluations > (6_000_000 if case["kind"] == "shock_tube" else 2_000_000):
        return None                # over the time that a reference may take
    w = _workload(case, seed)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda").double()
    keep = (["ax", "ay", "az", "pot", "ups", "X", "in_eps"] if w.params.gravity else ["ax", "ay", "az"])
    if ng:
        keep = keep + GAS_OUT + ["in_h"]
    if case.get("dissipation"):
        keep = keep + ["dalpha", "dalpha_u"]
    if case["kind"] == "ensemble":
        parts, off = [], w.sys_offsets
        for a, b in zip(off[:-1], off[1:]):
            one = W.Workload("system", **{f: x[a:b] for f, x in w.arrays().items()}, n_gas=int(b - a), params=w.params)
            parts.append(_evaluate(Exact(one), one, dev))
        return {k: torch.cat([x[k] for x in parts]) for k in keep}
    p = w.params
    ex = Exact(w, p.periodic_mask, [h - l for l, h in zip(p.periodic_lo, p.periodic_hi)])
    if "steps" not in case:
        r = _evaluate(ex, w, dev)
        return {k: r[k] for k in keep}
    return _leapfrog(case, ex, w, dev, keep)


def _evaluate(ex, w, dev):
    pad = lambda a: None if a is None else torch.nn.functional.pad(dev(a), (0, w.n - len(a)))
    return ex(torch.stack([dev(w.x), dev(w.y), dev(w.z)], 1), torch.stack([dev(w.vx), dev(w.vy), dev(w.vz)], 1),
              dev(w.m), dev(w.u), dev(w.h), dev(w.eps), pad(w.alpha), pad(w.alpha_u))


def _leapfrog(case, ex, w, dev, keep):
    """Kick-drift-kick: the fixed step of evol_kdk, or evol_run's criteria with predicted v and u."""
    p = w.params
    X, V = torch.stack([dev(w.x), dev(w.y), dev(w.z)], 1), torch.stack([dev(w.vx), dev(w.vy), dev(w.vz)], 1)
    m, U, h, eps = dev(w.m), dev(w.u), dev(w.h), dev(w.eps)
    ranged = case["kind"] == "run"
    time, dt = 0.0, float(np.float32(KDK_DT))
    r = ex(X, V, m, U, h, eps, flow=ranged)
    for _ in range(case["steps"]):
        A, D = torch.stack([r["ax"], r["ay"], r["az"]], 1), r["dudt"]
        if ranged:
            c = {k: float(np.float32(v)) for k, v in CRITERIA.items()}
            L = torch.minimum(r["in_eps"], r["in_h"])
            crit = [c["eta_acc"] * torch.sqrt(L / A.norm(dim=1)), c["eta_u"] * (U / D).abs(),
                    c["eta_courant"] * r["in_h"] / (r["in_h"] * r["divv_h"].abs() + r["c"] +
                                                     1.2 * (p.alpha * r["c"] + p.beta * r["mumax"]))]
            dt = min([c["dt_max"]] + [float(x.min()) for x in crit])
            time += dt
        V, U = V + 0.5 * dt * A, U + 0.5 * dt * D
        X = X + dt * V
        for a in range(3):
            if ex.len[a]:
                X[:, a] = torch.remainder(X[:, a], ex.len[a])
        h, eps = r["in_h"], r.get("in_eps", eps)
        r = ex(X, V + 0.5 * dt * A, m, U + 0.5 * dt * D, h, eps, flow=True) if ranged else ex(X, V, m, U, h, eps)
        V, U = V + 0.5 * dt * torch.stack([r["ax"], r["ay"], r["az"]], 1), U + 0.5 * dt * r["dudt"]
    out = {k: r[k] for k in keep}
    out.update({"in_" + k: X[:, a] for a, k in enumerate("xyz")} | {"in_v" + k: V[:, a] for a, k in enumerate("xyz")})
    out["in_u"] = U
    if ranged:
        out["time"], out["dt"] = time, dt
    return out

"""Performance cases of the batched hyperdynamics path.

Each case is one call pattern of a program that uses this package: advance a
batch of AFM replicas and read the observables (`md`), quench it for the
transition test of Sec. 2.3 (`quench`), one whole round of stepped sliding
(`cycle`: move the sliders, advance, quench, read), or build a neighbour list
on the caller's own device buffers (`lists`).  Models and sizes are those of
the package's workloads (`model.WORKLOADS`), of the paper's own models
(`model.paper2d`, `model.paper3d`) and of the tests.

Inputs.  A user starts such a run from an equilibrated state around a basin
minimum r_O, with the bias band taken from a pre-run (5% and 50% quantiles of
the slope).  Both come from the plain FP64 torch code below, once per model
(it is kept for the process): every replica of a case then gets that state
plus a small displacement, its own Maxwell-Boltzmann velocities, slider
position and noise key, all drawn from the seed.

Outputs.  All observables of every replica, and the whole state of the last
one, which stepped sliding carries into its next interval.  The split form
computes its forces in FP32: what follows from them (velocities, energies,
slopes, quenched positions) is returned in FP32, which is how far it is
meant to be good; positions, clocks and everything of the FP64 form stay
FP64, counters are whole numbers.
"""
import math

import numpy as np
import torch

from paper_0909_5215_gb300 import hd
from paper_0909_5215_gb300 import model as M

DT, RC, SKIN = 0.005, 2.5, 0.3
OBS = {name: k for k, name in enumerate(hd.OBS_FIELDS)}


# ---------------------------------------------------------------- the cases
def _md(name, model, n_rep, prec, driver, steps, **kw):
    c = dict(kind="md", model=model, n_rep=n_rep, prec=prec, driver=driver, block=0, steps=steps, kT=0.1, bias=1,
             chain=0, state=1)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the paper's 113-atom model at 8 slider positions, FP64: the inner loop of stepped sliding,
        # a few steps and the observables (20 MD steps between samples of F_R)
        _md("sliding_2d_8x113_f64", "paper2d", 8, 0, "persistent", 20, kT=0.05, state=0),
        # one 421-atom replica, plain FP64 MD without bias, as the plain 2-D workload runs it
        _md("md_2d_1x421_f64", "afm2d", 1, 0, "persistent", 100, block=64, kT=0.05, bias=0, cols=48, tip=37),
        # 16 slider positions of the 421-atom model, split form, bias on
        _md("md_2d_16x421_split", "afm2d", 16, 1, "persistent", 100, block=64, kT=0.05, cols=48, tip=37),
        # one round of stepped sliding of the same batch: sliders, steps, transition quench, observables
        _md("cycle_2d_16x421_split", "afm2d", 16, 1, "persistent", 25, block=64, kT=0.05, cols=48, tip=37,
            kind="cycle", iters=64),
        # the paper's bonded 1,983-atom model with its Nose-Hoover chain, on the default driver
        _md("md_3d_8x1983_chain_split", "paper3d", 8, 1, "kernels", 50, chain=3),
        # the default 3-D workload: 64 slider positions of 14,272 atoms, split form, bias on
        _md("md_3d_64x14272_split", "afm3d", 64, 1, "kernels", 40, nx=24, ny=24, nz=6, radius=6.0),
        # the transition test's FIRE quench of that batch, with a budget of iterations
        _md("quench_3d_64x14272_split", "afm3d", 64, 1, "kernels", 0, nx=24, ny=24, nz=6, radius=6.0,
            kind="quench", iters=64),
        # the plain FP64 form of the 3-D model
        _md("md_3d_4x14272_f64", "afm3d", 4, 0, "kernels", 20, nx=24, ny=24, nz=6, radius=6.0),
        # replicas of uneven size, 2-D and 3-D, each at its own temperature, in one batch
        _md("md_mixed_24_split", "mixed", 24, 1, "kernels", 40, pick=4),
        # the large 3-D model: 167,612 atoms a replica
        _md("md_3d_8x167612_split", "afm3d", 8, 1, "kernels", 20, nx=64, ny=64, nz=10, radius=12.0),
        # the list build on caller-owned device buffers, one 3-D replica
        dict(name="lists_14272", kind="lists", model="afm3d", nx=24, ny=24, nz=6, radius=6.0, maxnb=112),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def tip(nx, ny):      # the tip stays clear of its periodic images
        return round(rng.uniform(2.5, min(7.0, 0.6 * min(nx, ny))), 2)

    prec = 1 if rng.random() < 0.7 else 0
    kT = round(rng.uniform(0.05, 0.15), 4)
    kind = rng.choice(["md", "md", "md", "quench", "cycle", "lists"])
    fam = rng.choice(["2d", "2d", "3d", "3d", "3d", "paper2d", "paper3d", "mixed"])
    if kind == "lists":
        nx = log(5, 48)
        ny = nx if rng.random() < 0.5 else log(5, 48)
        return dict(kind="lists", model="afm3d", nx=nx, ny=ny, nz=rng.randint(3, 6), radius=tip(nx, ny),
                    maxnb=rng.choice([112, 128]))
    kw = dict(kind=kind, kT=kT, bias=1 if rng.random() < 0.8 else 0)
    steps, iters = log(10, 40), log(16, 64)
    if fam == "2d":
        kw.update(cols=log(16, 480), tip=rng.choice([13, 37, 60]))
        n_rep, model, big = log(1, 32), "afm2d", 0
    elif fam == "3d":
        nx = log(5, 36)
        ny = nx if rng.random() < 0.75 else log(5, 36)
        kw.update(nx=nx, ny=ny, nz=rng.randint(3, 7), radius=tip(nx, ny))
        atoms = 4 * kw["nx"] * kw["ny"] * kw["nz"] + 500
        n_rep, model = log(1, max(1, min(64, (400000 if prec else 40000) // atoms))), "afm3d"
        big = atoms * n_rep > 40000
    elif fam == "mixed":
        n_rep, model, big = rng.randint(2, 20) if prec else 2, "mixed", 1
        kw["pick"] = rng.randint(1, 1000)
    else:
        n_rep, model, big = log(1, 32), fam, 0
        if rng.random() < 0.4 and kind == "md":
            kw["chain"] = rng.choice([1, 3])
    driver = "kernels" if big or rng.random() < 0.5 else "persistent"
    block = rng.choice([0, 64]) if driver == "persistent" else rng.choice([0, 64, 256])
    if kind != "md":
        kw["iters"] = iters
    return _md("", model, n_rep, prec, driver, 0 if kind == "quench" else steps, block=block, **kw)


# ---------------------------------------------------------------- inputs
_bases = {}


def _base(case, kT):
    """(replica at r_O with its box and roles, equilibrated positions, sigma_L, sigma_U) of one model."""
    m = case["model"]
    key = (m, kT) + tuple(case.get(k) for k in ("cols", "tip", "nx", "ny", "nz", "radius"))
    if key not in _bases:
        if m == "afm2d":
            rep = M.afm2d(n_cols=case["cols"], n_tip=case["tip"], eps=M.PAPER_EPS_2D, kT=kT)
        elif m == "afm3d":
            rep = M.afm3d(nx=case["nx"], ny=case["ny"], nz=case["nz"], tip_radius=case["radius"],
                          eps=M.PAPER_EPS_3D, kT=kT)
        else:
            rep = (M.paper2d if m == "paper2d" else M.paper3d)(kT=kT)
        if len(_bases) >= 40:
            _bases.clear()
        _bases[key] = (rep,) + _equilibrate(rep)
    return _bases[key]


def _mixed(case):
    """Sizes of the uneven batch: up to six models, 2-D and 3-D in turn, log-uniform, with their temperatures."""
    rng = np.random.default_rng(case["pick"])
    out = []
    for k in range(min(6, case["n_rep"])):
        kT = round(float(rng.uniform(0.05, 0.15)), 2)
        u = float(rng.random())
        if k % 2 == 0:
            out.append((dict(model="afm2d", cols=max(8, int((400 * 10 ** u - 37) / 8)), tip=37), kT))
        else:
            side = max(5, int(round(math.sqrt((5000 * 8 ** u - 448) / 24.0))))
            out.append((dict(model="afm3d", nx=side, ny=side, nz=6, radius=6.0), kT))
    return [out[k % len(out)] for k in range(case["n_rep"])]


def _replicas(case, seed):
    models = _mixed(case) if case["model"] == "mixed" else [(case, case["kT"])] * case["n_rep"]
    reps = []
    for k, (m, kT) in enumerate(models):
        base, x, lo, hi = _base(m, kT)
        rng = np.random.default_rng([seed, k])
        r = base.copy()
        mob = r.role == M.ROLE_MOBILE
        d = r.dim
        r.pos_ref = base.pos.copy()
        r.pos = x.copy()
        r.pos[:, :d] += mob[:, None] * rng.normal(0.0, 0.01, size=(r.n, d))
        r.vel = np.zeros_like(r.pos)
        r.vel[:, :d] = mob[:, None] * rng.normal(0.0, math.sqrt(kT), size=(r.n, d))
        r.slider = base.slider + np.array([0.02 * (k + rng.random()), 0.0])
        r.rep_id = k
        r.kT = kT
        if case["bias"]:
            r.dvmax, r.sig_lo, r.sig_hi = 4.0 * kT, lo, hi
        if case["chain"]:
            r.nhc_len, r.nhc_tau = case["chain"], 0.5
        reps.append(r)
    return reps, M.Params(dt=DT, rc=RC, skin=SKIN, bias_on=case["bias"], seed=20250909 + 7 * seed, prec=case["prec"])


def _sliders(reps):
    return np.array([[r.slider[0] + 0.01, r.slider[1]] for r in reps])


def prepare(case, seed):
    if case["kind"] == "lists":
        base, x, _, _ = _base(case, 0.1)
        rng = np.random.default_rng([seed, 0])
        pos = x + (base.role == M.ROLE_MOBILE)[:, None] * rng.normal(0.0, 0.02, size=x.shape)
        dev = torch.device("cuda:0")
        return dict(case=case, n=base.n, box=base.box, periodic=base.periodic,
                    pos=torch.from_numpy(pos).to(dev),
                    nbr=torch.empty((base.n, case["maxnb"]), dtype=torch.int32, device=dev),
                    nnb=torch.empty(base.n, dtype=torch.int32, device=dev))
    reps, params = _replicas(case, seed)
    driver = hd.HD_DRIVER_PERSISTENT if case["driver"] == "persistent" else hd.HD_DRIVER_KERNELS
    return dict(case=case, sliders=_sliders(reps), batch=hd.Batch(reps, params, driver=driver, block=case["block"]))


# ---------------------------------------------------------------- one pass
_WHOLE = ("step", "n_rebuild", "n_dv_zero", "n_dv_band", "n_dv_max")
_CLOCK = ("t_md", "x_S")
_PAIRS = ("t_h", "V", "K", "dV", "sigma", "d", "F_R", "x_T", "y_T", "z_T", "G")


def _observed(ob, prec):
    real = np.float32 if prec else np.float64
    out = {k: ob[:, OBS[k]].astype(np.int64) for k in _WHOLE}
    out.update({k: ob[:, OBS[k]].copy() for k in _CLOCK})
    out.update({k: ob[:, OBS[k]].astype(real) for k in _PAIRS})
    return out


def run(state):
    case = state["case"]
    if case["kind"] == "lists":
        st = hd.hd_nlist_static(state["pos"].data_ptr(), state["n"], state["box"], state["periodic"], RC + SKIN,
                                case["maxnb"], state["nbr"].data_ptr(), state["nnb"].data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
        if st != hd.HD_OK:
            raise hd.HdError(st, "hd_nlist_static")
        return state["nbr"], state["nnb"]
    b = state["batch"]
    real = np.float32 if case["prec"] else np.float64
    last = b.n_rep - 1
    if case["kind"] == "quench":
        flags = b.quench(method=1, ftol=1e-3, max_iter=case["iters"], step_size=0.005, theta=0.5, adopt=0)
        ob = b.obs()
        return dict(flags=flags, iters=ob[:, OBS["q_iter"]].astype(np.int64),
                    moved=ob[:, OBS["q_disp"]].astype(real), positions=b.qpos(last).astype(real))
    if case["kind"] == "cycle":
        b.set_slider(state["sliders"])
    b.step(case["steps"])
    out = {}
    if case["kind"] == "cycle":
        out["flags"] = b.quench(method=1, ftol=1e-3, max_iter=case["iters"], step_size=0.005, theta=0.5, adopt=1)
    out["obs"] = _observed(b.obs(), case["prec"])
    if case["state"]:
        out["positions"] = b.positions(last)
        out["velocities"] = b.velocities(last).astype(real)
    return out


# ---------------------------------------------------------------- what a pass cannot do without
def _pairs(dim):
    """Unique pairs an atom has within rc, and list entries within rc + skin (each pair twice)."""
    return (27.0, 76.0) if dim == 3 else (8.0, 20.0)


def work(case):
    """Per step and atom: the state read and written once (position and velocity, r_O, type and role), every
    unique pair's index once; per unique pair the Lennard-Jones force and, with the bias, its Hessian-vector term."""
    if case["kind"] == "lists":
        n = _atoms(case)
        return {"bytes": n * (24.0 + 4.0 * case["maxnb"] + 4.0), "flops": n * 76.0 * 8.0}
    models = [m for m, _ in _mixed(case)] if case["model"] == "mixed" else [case] * case["n_rep"]
    byt = flo = 0.0
    for m in models:
        n, (pairs, entries) = _atoms(m), _pairs(2 if m["model"] in ("afm2d", "paper2d") else 3)
        if case["steps"]:
            byt += case["steps"] * n * (2 * 24 + 2 * 24 + 2 + 2 * entries + (24 if case["bias"] else 0))
            flo += case["steps"] * n * (pairs * (75 if case["bias"] else 40) + 100)
        byt += case.get("iters", 0) * n * (2 * 24 + 2 * 12 + 2 + 2 * entries)
        flo += case.get("iters", 0) * n * (pairs * 40 + 40)
    return {"bytes": byt, "flops": flo}


def _atoms(m):
    if m["model"] == "afm2d":
        return 8 * m["cols"] + m["tip"]
    if m["model"] == "afm3d":
        return 4 * m["nx"] * m["ny"] * m["nz"] + int(2.0 * m["radius"] ** 3)
    return 113 if m["model"] == "paper2d" else 1983


# ---------------------------------------------------------------- the same in plain FP64 torch
class _Plain:
    """One replica in FP64 torch: LJ with shift (and bonds), the slope bias, BAOAB or the chain, FIRE."""

    def __init__(self, rep, bias, seed=0):
        t = lambda a, k=torch.float64: torch.as_tensor(np.ascontiguousarray(a), dtype=k, device="cuda")  # noqa: E731
        self.r, self.bias, self.seed = rep, bias, seed
        self.x, self.xo = t(rep.pos), t(rep.pos if rep.pos_ref is None else rep.pos_ref)
        self.v = t(np.zeros_like(rep.pos) if rep.vel is None else rep.vel)
        self.type, self.mob = t(rep.type, torch.long), t(rep.role == M.ROLE_MOBILE, torch.bool)
        self.rig = t(np.flatnonzero(rep.role == M.ROLE_RIGID), torch.long)
        self.move = self.mob[:, None] * t([1.0, 1.0, 1.0 if rep.dim == 3 else 0.0])
        self.L = t([rep.box[a] if rep.periodic[a] else 1e30 for a in range(3)])
        eps = np.array(rep.eps, dtype=float)
        if rep.bonds is not None:
            eps[1, 1] = 0.0
        self.eps, self.sig2 = t(eps), t(np.array(rep.sig) ** 2)
        s6 = (self.sig2 / RC ** 2) ** 3
        self.shift = 4 * self.eps * (s6 * s6 - s6)
        self.bonds = None
        if rep.bonds is not None:
            both = np.concatenate([rep.bonds, rep.bonds[:, ::-1]])
            both = both[np.argsort(both[:, 0], kind="stable")]
            deg = np.bincount(both[:, 0], minlength=rep.n)
            self.bonds = np.full((rep.n, max(1, deg.max())), -1)
            self.bonds[both[:, 0], np.arange(len(both)) - (np.cumsum(deg) - deg)[both[:, 0]]] = both[:, 1]
            self.bonds = t(self.bonds, torch.long)
        self.vb = torch.zeros(3, dtype=torch.float64, device="cuda")
        self.t_h = self.t_md = 0.0
        self.steps, self.ndv = 0, [0, 0, 0]
        self.xi, self.vchain = np.zeros(8), np.zeros(8)
        self.xs = float(rep.slider[0])
        self.xb = None

    def mi(self, d):
        return d - self.L * torch.round(d / self.L)

    def rows(self):
        """Padded rows of all pairs within RC + 0.5, rebuilt when an atom has moved 0.25."""
        x = self.x
        if self.xb is not None and float((x - self.xb).square().sum(1).max()) < 0.0625:
            return
        rl, n = RC + 0.5, len(x)
        lo = x.min(0).values - 1e-9
        ext = torch.where(self.L < 1e29, self.L, x.max(0).values - lo + 1e-6).cpu().numpy()
        nc = [max(1, int(e / rl)) for e in ext]
        nc = [c if c >= 3 or self.r.periodic[a] == 0 else 1 for a, c in enumerate(nc)]
        w = torch.tensor([e / c for e, c in zip(ext, nc)], dtype=torch.float64, device="cuda")
        frac = torch.where(self.L < 1e29, x - self.L * torch.floor(x / self.L), x - lo)
        top = torch.tensor(nc, device="cuda") - 1
        c3 = torch.minimum((frac / w).long().clamp(min=0), top)
        cell = (c3[:, 2] * nc[1] + c3[:, 1]) * nc[0] + c3[:, 0]
        order = torch.argsort(cell, stable=True)
        cnt = torch.bincount(cell, minlength=nc[0] * nc[1] * nc[2])
        cap = int(cnt.max())
        table = torch.full((len(cnt) + 1, cap), -1, dtype=torch.long, device="cuda")
        table[cell[order], torch.arange(n, device="cuda") - (cnt.cumsum(0) - cnt)[cell[order]]] = order
        near = []
        for dz in ((0,) if nc[2] == 1 else (-1, 0, 1)):
            for dy in ((0,) if nc[1] == 1 else (-1, 0, 1)):
                for dx in ((0,) if nc[0] == 1 else (-1, 0, 1)):
                    q, ok = [], torch.ones(n, dtype=torch.bool, device="cuda")
                    for a, s in enumerate((dx, dy, dz)):
                        v = c3[:, a] + s
                        if self.r.periodic[a]:
                            v = v % nc[a]
                        else:
                            ok &= (v >= 0) & (v < nc[a])
                        q.append(v)
                    near.append(torch.where(ok, (q[2] * nc[1] + q[1]) * nc[0] + q[0], len(cnt)))
        near = torch.stack(near, 1)
        parts, step = [], max(1, 40_000_000 // (near.shape[1] * cap))
        for i in range(0, n, step):
            j = table[near[i:i + step]].flatten(1)
            me = torch.arange(i, min(n, i + step), device="cuda")[:, None]
            hit = (j >= 0) & (j != me)
            hit &= self.mi(x[i:i + step, None] - x[j.clamp(min=0)]).square().sum(2) < rl * rl
            k = int(hit.sum(1).max())
            at = torch.argsort((~hit).to(torch.int8), dim=1, stable=True)[:, :k]
            parts.append(torch.where(hit.gather(1, at), j.gather(1, at), -1))
        k = max(p.shape[1] for p in parts)
        self.nb = torch.cat([torch.nn.functional.pad(p, (0, k - p.shape[1]), value=-1) for p in parts])
        self.xb = x.clone()

    def forces(self, hess):
        """LJ (and bond) force, per-atom energy, H (r - r_O)."""
        self.rows()
        x, dr = self.x, self.x - self.xo
        F, H, E = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x[:, 0])
        chunk = max(1, 24_000_000 // self.nb.shape[1])

        def add(s, j, ok, d, A, B, e):
            F[s] += torch.where(ok, -A, 0.0).unsqueeze(2).mul(d).sum(1)
            E[s] += torch.where(ok, 0.5 * e, 0.0).sum(1)
            if hess:
                u = dr[s, None] - dr[j]
                g = torch.where(ok, A, 0.0).unsqueeze(2) * u
                H[s] += (g + torch.where(ok, B * (d * u).sum(2), 0.0).unsqueeze(2) * d).sum(1)

        for i in range(0, len(x), chunk):
            s = slice(i, min(len(x), i + chunk))
            j = self.nb[s].clamp(min=0)
            d = self.mi(x[s, None] - x[j])
            r2 = d.square().sum(2)
            ok = (self.nb[s] >= 0) & (r2 < RC * RC)
            ti, tj = self.type[s, None].expand_as(j), self.type[j]
            eps, s6 = self.eps[ti, tj], (self.sig2[ti, tj] / r2) ** 3
            add(s, j, ok, d, -24 * eps * s6 * (2 * s6 - 1) / r2, 96 * eps * s6 * (7 * s6 - 2) / r2 ** 2,
                4 * eps * s6 * (s6 - 1) - self.shift[ti, tj])
        if self.bonds is not None:
            j, ok = self.bonds.clamp(min=0), self.bonds >= 0
            d = self.mi(x[:, None] - x[j])
            r = torch.where(ok, d.square().sum(2), 1.0).sqrt()
            A = self.r.k_bond * (r - self.r.r_bond) / r
            add(slice(0, len(x)), j, ok, d, A, (self.r.k_bond - A) / r ** 2,
                0.5 * self.r.k_bond * (r - self.r.r_bond) ** 2)
        return F, E, H, dr

    def load(self, xT):
        g = torch.zeros(3, dtype=torch.float64, device="cuda")
        g[0] = self.r.k_spring * (xT[0] - self.xs)
        if self.r.dim == 3:
            g[1] = self.r.k_spring * (xT[1] - float(self.r.slider[1]))
        g[self.r.dim - 1] = self.r.f_normal
        return g

    def evaluate(self, hess=True):
        r, rig = self.r, self.rig
        F, E, H, dr = self.forces(hess)
        nr = len(rig)
        xT = self.x[rig].mean(0)
        gs = self.load(xT)
        if hess:
            axes = [0] if r.dim == 2 else [0, 1]
            for a in axes:
                H[rig, a] += r.k_spring / nr * dr[rig, a]
        d = dr.square().sum().sqrt()
        G = -(F * dr).sum() + (gs * dr[rig].sum(0)).sum() / nr
        sig = G / d if float(d) > 0 else G * 0
        dV, dVp = 0.0, 0.0
        if self.bias:
            s, lo, hi, m = float(sig), r.sig_lo, r.sig_hi, r.m_exp
            if s >= hi:
                dV = r.dvmax
            elif s > lo:
                t = (s - hi) / (lo - hi)
                q = 1 - t ** m
                dV, dVp = r.dvmax * q * q, 2 * r.dvmax * q * (-m * t ** (m - 1)) / (lo - hi)
        fb = F[rig].sum(0) - gs
        tot = F
        if dVp != 0.0:
            tot = F - dVp * ((H - F) / d - sig * dr / d ** 2)
            fb = fb - dVp * ((H[rig].sum(0) - F[rig].sum(0) + gs) / d - sig * dr[rig].sum(0) / d ** 2)
        if r.dim == 2:
            fb[2] = 0.0
        ext = 0.5 * r.k_spring * (xT[0] - self.xs) ** 2 + r.f_normal * xT[r.dim - 1]
        if r.dim == 3:
            ext = ext + 0.5 * r.k_spring * (xT[1] - float(r.slider[1])) ** 2
        self.F, self.fb, self.dV = tot, fb, dV
        self.now = dict(V=E.sum() + ext, dV=dV, sigma=sig, d=d, F_R=r.k_spring * (self.xs - xT[0]), x_T=xT[0],
                        y_T=xT[1], z_T=xT[2], G=G)
        return self

    def chain_half(self, k2):
        """One half step of the Nose-Hoover chain (Martyna et al. 1996, one stage): the velocities' scale."""
        M_, kT, v = self.r.nhc_len, self.r.kT, self.vchain
        nf = self.r.dim * int(self.mob.sum())
        Q = [(nf if j == 0 else 1) * kT * self.r.nhc_tau ** 2 for j in range(M_)]
        g = lambda j: (k2 - nf * kT) / Q[0] if j == 0 else (Q[j - 1] * v[j - 1] ** 2 - kT) / Q[j]  # noqa: E731
        v[M_ - 1] += 0.25 * DT * g(M_ - 1)
        for j in range(M_ - 2, -1, -1):
            e = math.exp(-0.125 * DT * v[j + 1])
            v[j] = (v[j] * e + 0.25 * DT * g(j)) * e
        s = math.exp(-0.5 * DT * v[0])
        k2 *= s * s
        self.xi[:M_] += 0.5 * DT * v[:M_]
        for j in range(M_ - 1):
            e = math.exp(-0.125 * DT * v[j + 1])
            v[j] = (v[j] * e + 0.25 * DT * g(j)) * e
        v[M_ - 1] += 0.25 * DT * g(M_ - 1)
        return s

    def step(self, n):
        """n BAOAB steps (or steps of the chain) from an evaluated state."""
        r, rig, nr, h = self.r, self.rig, len(self.rig), DT
        c = math.exp(-r.gamma * h)
        s = math.sqrt((1 - c * c) * r.kT)
        for _ in range(n):
            self.t_h += h * math.exp(self.dV / r.kT)
            self.t_md += h
            self.ndv[0 if self.dV <= 0 else 2 if self.dV >= r.dvmax else 1] += 1
            if r.nhc_len:
                self.v = self.v * self.chain_half(float((self.v[self.mob] ** 2).sum()))
            self.v = self.v + 0.5 * h * self.F * self.move
            self.vb = self.vb + 0.5 * h * self.fb / nr
            self.x = self.x + 0.5 * h * self.v
            if not r.nhc_len:
                self.v = c * self.v + s * _noise(self.seed, self.steps, r.rep_id, len(self.x)) * self.move
            self.x = self.x + 0.5 * h * self.v
            self.x[rig] += h * self.vb
            self.steps += 1
            self.evaluate(bool(self.bias))
            self.v = self.v + 0.5 * h * self.F * self.move
            self.vb = self.vb + 0.5 * h * self.fb / nr
            if r.nhc_len:
                self.v = self.v * self.chain_half(float((self.v[self.mob] ** 2).sum()))
        K = 0.5 * self.v[self.mob].square().sum() + 0.5 * nr * self.vb.square().sum()
        self.now.update(K=K, t_h=self.t_h)
        v = self.v.clone()
        v[rig] = self.vb
        return v

    def fire(self, iters, dt0, ftol):
        """FIRE (Bitzek et al. 2006) on this state, the rigid layer as one body; (iterations, max |F|)."""
        rig, nr, dim = self.rig, len(self.rig), self.r.dim
        v, vb = torch.zeros_like(self.x), torch.zeros_like(self.vb)
        dt, alpha, npos = dt0, 0.1, 0
        for it in range(iters + 1):
            F, _, _, _ = self.forces(False)
            fb = F[rig].sum(0) - self.load(self.x[rig].mean(0))
            F = F * self.mob[:, None]
            fmax = float(torch.maximum(F.square().sum(1).max(), fb.square().sum()).sqrt())
            if fmax < ftol or it == iters:
                return it, fmax
            b = fb[:dim]
            p = float((F * v).sum() + (b * vb[:dim]).sum())
            vv = float(v.square().sum() + nr * vb[:dim].square().sum())
            ff = float(F.square().sum() + b.square().sum() / nr)
            if p > 0:
                mix = alpha * math.sqrt(vv / ff) if ff > 0 else 0.0
                v, vb = (1 - alpha) * v + mix * F, (1 - alpha) * vb + mix * fb / nr
                npos += 1
                if npos > 5:
                    dt, alpha = min(1.1 * dt, 10 * dt0), 0.99 * alpha
            else:
                v, vb, dt, alpha, npos = v * 0, vb * 0, 0.5 * dt, 0.1, 0
            v, vb = v + dt * F * self.move, vb + dt * fb / nr
            if dim == 2:
                vb[2] = 0.0
            self.x = self.x + dt * v
            self.x[rig] += dt * vb


def _noise(seed, step, rep_id, n):
    """The documented thermostat draws: Philox4x32-10 (Salmon et al. 2011) per atom, 52-bit uniforms, Box-Muller."""
    mask = 0xFFFFFFFF
    atom = torch.arange(n, dtype=torch.int64, device="cuda")

    def normals(call):
        c = [torch.full_like(atom, step & mask), atom, torch.full_like(atom, rep_id & mask),
             torch.full_like(atom, (call | ((step >> 32) << 8)) & mask)]
        k0, k1 = seed & mask, (seed >> 32) & mask
        for rnd in range(10):
            if rnd:
                k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
            hl = []
            for a, q in ((0xD2511F53, c[0]), (0xCD9E8D57, c[2])):
                p0, p1 = (a & 0xFFFF) * q, (a >> 16) * q
                hl.append(((p1 + (p0 >> 16)) >> 16, (((p1 & 0xFFFF) << 16) + p0) & mask))
            c = [hl[1][0] ^ c[1] ^ k0, hl[1][1], hl[0][0] ^ c[3] ^ k1, hl[0][1]]
        u = [((c[i] >> 6).double() * 2.0 ** 26 + (c[i + 1] >> 6).double() + 0.5) * 2.0 ** -52 for i in (0, 2)]
        rad = (-2 * torch.log(u[0])).sqrt()
        return rad * torch.cos(2 * math.pi * u[1]), rad * torch.sin(2 * math.pi * u[1])

    n0, n1 = normals(0)
    return torch.stack([n0, n1, normals(1)[0]], 1)


def _equilibrate(rep):
    """Relaxes the lattice to its r_O (kept as rep.pos), heats it, and takes the slope's band over a pre-run."""
    p = _Plain(rep, 0, 1)
    p.fire(150, 0.005, 1e-2)
    rep.pos = p.x.cpu().numpy()
    g = np.random.default_rng(1)
    start = rep.copy()
    mob = (rep.role == M.ROLE_MOBILE)[:, None]
    on = np.array([1.0, 1.0, 1.0 if rep.dim == 3 else 0.0])
    start.pos_ref = rep.pos
    start.pos = rep.pos + mob * on * g.normal(0.0, 0.05 * math.sqrt(rep.kT), size=rep.pos.shape)
    start.vel = mob * on * g.normal(0.0, math.sqrt(rep.kT), size=rep.pos.shape)
    p = _Plain(start, 0, 1).evaluate(False)
    p.step(150)
    sigma = []
    for _ in range(50):
        p.step(5)
        sigma.append(float(p.now["sigma"]))
    return p.x.cpu().numpy(), float(np.quantile(sigma, 0.05)), float(np.quantile(sigma, 0.5))


def _max_shift(p, x0):
    return float(p.mi(p.x - x0).square().sum(1).max().sqrt())


def exact(case, seed):
    if case["kind"] == "lists":
        return None
    reps, params = _replicas(case, seed)
    sliders = _sliders(reps)
    out, flags, moved = [], [], []
    for k, r in enumerate(reps):
        p = _Plain(r, case["bias"], params.seed)
        if case["kind"] == "cycle":
            p.xs = float(sliders[k, 0])
        if case["kind"] == "quench":
            p.fire(case["iters"], 0.005, 1e-3)
            moved.append(_max_shift(p, p.xo))
            continue
        p.evaluate(bool(case["bias"]))
        v = p.step(case["steps"])
        if case["kind"] == "cycle":
            # the quench changes the observables only where r_O moves: a converged, flagged replica
            q = _Plain(r, 0)
            q.x, q.xs = p.x.clone(), p.xs
            _, f = q.fire(case["iters"], 0.005, 1e-3)
            flags.append(int(_max_shift(q, p.xo) > 0.5))
            if f < 1e-3 and flags[-1]:
                p.xo = q.x
            kept = {name: p.now[name] for name in ("K", "t_h")}
            p.evaluate(bool(case["bias"]))
            p.now.update(kept)
        out.append((p, v))
    if case["kind"] == "quench":
        return dict(flags=None, iters=None, moved=np.array(moved), positions=p.x.cpu().numpy())
    res = {"flags": np.array(flags, dtype=np.int32)} if case["kind"] == "cycle" else {}
    obs = {k: None for k in _WHOLE}
    obs["t_md"], obs["x_S"] = np.array([p.t_md for p, _ in out]), np.array([p.xs for p, _ in out])
    for k in _PAIRS:
        obs[k] = np.array([float(p.now[k]) for p, _ in out])
    res["obs"] = obs
    if case["state"]:
        res["positions"], res["velocities"] = out[-1][0].x.cpu().numpy(), out[-1][1].cpu().numpy()
    return res

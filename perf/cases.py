"""The work a user of this package has it do, as timed cases.

Each case goes through the package's public entry points (the functions with
the C names, SoftStep, Ensemble, soft_kdk) on the seeded disks of
``paper_2007_15432_gb300.disks``.  ``listed()`` names twelve cases, ``draw``
gives more of the same ranges, ``prepare`` makes the inputs and the handle a
program keeps, ``run`` is one pass, ``work`` the bytes and operations a pass
cannot do without, and ``exact`` the same outputs in 64-bit torch, written
from the formulas, where that can be had.

Kinds:
  step      one soft step (SoftStep.step) of a disk that goes on from pass to
            pass, as an integration does
  force     tree, soft force, neighbour lists and clusters of one state
            (SoftStep.force): what a new state costs before it can be stepped
  hard      the first half of a step on a copy of a kept state: soft kick,
            Hermite integration of the clusters, Kepler drift of the rest
  ensemble  one soft step of many small disks batched in one context and
            replayed from the captured CUDA graph
  gradient  forward and reverse sweep of a differentiable rollout
  cutoffs   cut-off and search radii of a state
  direct    the soft force summed over all pairs
  energy    the total energy
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2007_15432_gb300 import adjoint as AD
from paper_2007_15432_gb300 import disks
from paper_2007_15432_gb300 import ensemble as EN
from paper_2007_15432_gb300 import p3t as P

XV = ("x", "y", "z", "vx", "vy", "vz")


# ---- the cases ---------------------------------------------------------------
def listed():
    return [
        # the smallest call: a thousand equal-mass bodies in plain FP64 with the
        # soft force summed directly (theta = 0) and collisions, the
        # configuration for small studies and for checking a set-up; launches
        # and latency count
        dict(name="step_narrow_1000_fp64", kind="step", disk="narrow", n=1000, fp64=True,
             theta=0.0, group=0, collisions=True),
        # the headline workload: a million bodies on 1-10 au with individual
        # cut-off radii over two decades, mixed precision, perfect accretion
        dict(name="step_wide_1000000_mixed", kind="step", disk="wide", n=1_000_000, fp64=False,
             theta=0.5, group=64, collisions=True),
        # the equal-mass ring at the size of the precision study, mixed
        dict(name="step_ring_100000_mixed", kind="step", disk="ring", n=100_000, fp64=False,
             theta=0.5, group=64, collisions=False),
        # a small wide disk of odd size: what one state's force costs when the
        # launches weigh as much as the pairs
        dict(name="force_wide_3001_mixed", kind="force", disk="wide", n=3001, fp64=False,
             theta=0.5, group=64),
        # the ring's force in plain FP64 (the other side of the precision study)
        dict(name="force_ring_100000_fp64", kind="force", disk="ring", n=100_000, fp64=True,
             theta=0.5, group=64),
        # the hard part where it is busy: the mass spectrum of the paper's
        # cut-off study, clusters of two to many members
        dict(name="hard_spectrum_377740", kind="hard", disk="spectrum", n=377_740, fp64=False,
             rcut0=3.0),
        # many small independent disks in one captured step
        dict(name="ensemble_256_disks", kind="ensemble", disks=256, fp64=False),
        # the differentiation workload: 32 soft steps, direct force, FP32 pairs
        dict(name="gradient_direct_10000", kind="gradient", form="direct", n=10_000, steps=32,
             checkpoint=8, fp64=False),
        # the same disk through the paper's own step: tree force, Hermite
        # clusters, FP64
        dict(name="gradient_tree_10000", kind="gradient", form="tree", n=10_000, steps=4,
             checkpoint=4, fp64=True),
        # radii of the mass-spectrum ring: after every collision, and at the start
        dict(name="cutoffs_spectrum_377740", kind="cutoffs", disk="spectrum", n=377_740, mode=0,
             noalloc=False),
        # the direct sum in FP64: checks of the tree, small systems
        dict(name="direct_narrow_8191_fp64", kind="direct", disk="narrow", n=8191, fp64=True),
        # the energy, the diagnostic every run prints
        dict(name="energy_ring_100000_mixed", kind="energy", disk="ring", n=100_000, fp64=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "force", "step", "force", "hard", "ensemble", "gradient", "cutoffs",
                       "direct", "energy"])
    disk = rng.choice(["narrow", "ring", "wide", "wide", "spectrum"])
    fp64 = rng.random() < 0.4
    if kind in ("step", "force"):
        n = _log_int(rng, 512, 8192 if disk == "narrow" else (100_000 if fp64 else 1_000_000))
        c = dict(kind=kind, disk=disk, n=n, fp64=fp64,
                 theta=0.0 if n <= 2000 and rng.random() < 0.5 else rng.choice([0.3, 0.5, 0.7]),
                 group=rng.choice([0, 16, 32, 64]))
        if kind == "step":
            c["collisions"] = disk == "narrow" or rng.random() < 0.5
        return c
    if kind == "hard":
        disk = rng.choice(["ring", "wide", "spectrum"])
        return dict(kind=kind, disk=disk, n=_log_int(rng, 1000, 377_740), fp64=fp64,
                    rcut0=rng.choice([1.0, 2.0, 3.0] if disk == "spectrum" else [2.0, 3.0]))
    if kind == "ensemble":
        return dict(kind=kind, disks=_log_int(rng, 4, 256), fp64=False)
    if kind == "gradient":
        if rng.random() < 0.5:
            return dict(kind=kind, form="direct", n=_log_int(rng, 500, 10_000),
                        steps=rng.randint(4, 32), checkpoint=8, fp64=False)
        return dict(kind=kind, form="tree", n=_log_int(rng, 500, 10_000), steps=rng.randint(1, 4),
                    checkpoint=rng.choice([2, 4]), fp64=True)
    if kind == "cutoffs":
        noalloc = rng.random() < 0.3
        return dict(kind=kind, disk="ring" if disk == "narrow" else disk,
                    n=_log_int(rng, 1000, 1_000_000), mode=rng.randint(0, 1 if noalloc else 2),
                    noalloc=noalloc)
    if kind == "direct":
        return dict(kind=kind, disk="narrow" if disk == "narrow" else "ring",
                    n=_log_int(rng, 500, 16_384), fp64=fp64)
    return dict(kind="energy", disk="ring" if disk == "narrow" else disk,
                n=_log_int(rng, 1000, 30_000 if fp64 else 100_000), fp64=fp64)


# ---- inputs ------------------------------------------------------------------
def _disk(case, seed):
    n, d = case["n"], case["disk"]
    if d == "narrow":
        return disks.equal_mass_narrow(n=n, seed=seed)
    if d == "ring":
        return disks.equal_mass_ring(n=n, seed=seed)
    if d == "wide":
        return disks.wide_power_law(n=n, seed=seed)
    return disks.mass_spectrum_ring(n=n, seed=seed)


def _params(case, **kw):
    return P.Params(precision=P.P3T_FP64 if case["fp64"] else P.P3T_MIXED, **kw)


class _Context:
    """A context that goes with the state that holds it."""

    def __init__(self, params):
        self.h = P.p3t_create(params)

    def __del__(self):
        P.p3t_destroy(self.h)


def _stepper(case, s, params, r_phys=None):
    st, buf = P.State.from_numpy_packed(s, r_phys=r_phys)
    ss = P.SoftStep(params, st, nb_cap=16 * len(s["m"]) + 1024)
    ss.init()
    ss.status()
    return ss, buf


def prepare(case, seed):
    kind = case["kind"]
    out = dict(case=case)
    if kind in ("step", "force"):
        s = _disk(case, seed)
        coll = bool(case.get("collisions"))
        prm = _params(case, theta=case["theta"], group_size=case["group"],
                      f_radius=1.0 if coll else 0.0)
        out["ss"], out["buf"] = _stepper(case, s, prm, disks.physical_radius(s["m"]) if coll else None)
    elif kind == "hard":
        s = _disk(case, seed)
        ss, buf = _stepper(case, s, _params(case, group_size=64, rcut0=case["rcut0"]))
        out.update(ss=ss, buf=buf, base=buf.clone())
    elif kind == "ensemble":
        # the ensemble's sizes and its two families of disks; the seed moves the
        # particles, not the sizes
        ds = []
        for d, n in enumerate(disks.ensemble_sizes(case["disks"])):
            n, sd = int(n), 1000 * seed + d
            ds.append(disks.wide_power_law(n=n, seed=sd, n_proto=0) if d % 2 else
                      disks.disk(n, 0.95, 1.05, 0.01, 0.005, 1e-6 / n, sd))
        prm = [_params(case, group_size=64) for _ in ds]
        ens = EN.Ensemble(ds, prm, batched=True)
        ens.init()
        ens.capture()
        out["ens"] = ens
    elif kind == "gradient":
        s = disks.adjoint_disk(case["n"], seed)
        dev = torch.device("cuda")
        x0 = torch.as_tensor(np.stack([s["x"], s["y"], s["z"]])).to(dev)
        v0 = torch.as_tensor(np.stack([s["vx"], s["vy"], s["vz"]])).to(dev)
        m = torch.as_tensor(s["m"]).to(dev)
        prm = _params(case, group_size=64)
        tree = case["form"] == "tree"
        ro, rs = AD.cutoffs(prm, x0, v0, m, with_search=True)
        runner = AD.SoftKDK(prm, case["n"], case["steps"], case["checkpoint"],
                            force="tree" if tree else "direct", hard="p3t" if tree else "kepler")
        # where the disk would be without the soft force, moved by seeded offsets
        T = case["steps"] * prm.dt_soft
        target, _ = _kepler(x0, v0, T)
        target += torch.as_tensor(disks.target_offsets(case["n"], seed + 1)).to(dev)
        out.update(runner=runner, x0=x0.requires_grad_(), v0=v0.requires_grad_(),
                   m=m.requires_grad_(), ro=ro, rs=rs if tree else None, target=target)
    elif kind == "cutoffs":
        prm = P.Params(cutoff_mode=case["mode"])
        out["st"] = P.State.from_numpy(_disk(case, seed))
        out["prm"] = prm
        if not case["noalloc"]:
            out["ctx"] = _Context(prm)
            P.p3t_reserve(out["ctx"].h, case["n"])
    else:
        prm = _params(case)
        out["st"] = P.State.from_numpy(_disk(case, seed))
        out["ctx"] = _Context(prm)
        P.p3t_reserve(out["ctx"].h, case["n"])
        P.p3t_cutoffs(out["ctx"].h, out["st"])
        out["acc"] = torch.zeros(3, case["n"], dtype=torch.float64, device="cuda")
        out["e"] = torch.zeros(4, dtype=torch.float64, device="cuda")
    return out


# ---- one pass ----------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        ss = state["ss"]
        ss.step()
        buf = state["buf"]
        if ss.n < buf.shape[1]:  # particles merged: the columns past the count are empty
            buf[:, ss.n:] = 0.0
        return dict(zip(P._KEYS, buf), counts=ss.counts)
    if kind == "force":
        ss = state["ss"]
        ss.force()
        return dict(acc=ss.acc, counts=ss.counts, nb_off=ss.nb_off, nb_idx=ss.nb_idx)
    if kind == "hard":
        ss = state["ss"]
        state["buf"].copy_(state["base"])
        P.p3t_kick(ss.ctx, ss.st, ss.acc, 0.5 * ss.params.dt_soft)
        P.p3t_hard_step(ss.ctx, ss.st, ss.cl, ss.params.dt_soft, ss.hsteps)
        return dict(xv=state["buf"][:6], steps=ss.hsteps)
    if kind == "ensemble":
        ens = state["ens"]
        ens.step_graph()
        return dict(ens.arrays)
    if kind == "gradient":
        x0, v0, m = state["x0"], state["v0"], state["m"]
        x0.grad = v0.grad = m.grad = None
        xn, vn = AD.soft_kdk(x0, v0, m, state["ro"], state["runner"], state["rs"])
        loss = ((xn - state["target"]) ** 2).sum()
        loss.backward()
        return dict(x=xn.detach(), v=vn.detach(), loss=loss.detach(), gx=x0.grad, gv=v0.grad,
                    gm=m.grad)
    if kind == "cutoffs":
        st = state["st"]
        if case["noalloc"]:
            P.p3t_cutoffs_noalloc(state["prm"], st)
        else:
            P.p3t_cutoffs(state["ctx"].h, st)
        return dict(r_out=st.r_out, r_search=st.r_search)
    if kind == "direct":
        P.p3t_soft_force_direct(state["ctx"].h, state["st"], state["acc"])
        return dict(acc=state["acc"])
    P.p3t_energy(state["ctx"].h, state["st"], state["e"])
    return dict(e=state["e"])


# ---- what a pass cannot do without -------------------------------------------
# operations: about 30 a changeover pair and 70 a monopole + quadrupole term
# (45 on the lists' mean), 55 a pair of the force's vector-Jacobian product,
# 150 a Kepler drift; bytes: every input array read once, every output written
# once
def _walk_terms(n, theta):
    """Interactions of one soft force: n (n - 1) pairs, or by the tree about 32
    log2 n a particle at theta = 0.5 (640 at a million), as theta^-1.5."""
    return min(n * (n - 1.0), n * 32.0 * math.log2(max(n, 2)) * (0.5 / theta) ** 1.5
               if theta > 0 else n * (n - 1.0))


def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        n = 5000.0 * case["disks"]
        terms = case["disks"] * _walk_terms(5000, 0.5)
        return dict(bytes=n * 8 * (9 + 6), flops=45 * terms + 150 * n)
    n = case["n"]
    if kind == "step":
        return dict(bytes=n * 8.0 * (9 + 6), flops=45 * _walk_terms(n, case["theta"]) + 150 * n)
    if kind == "force":
        return dict(bytes=n * 8.0 * (9 + 3 + 1), flops=45 * _walk_terms(n, case["theta"]))
    if kind == "hard":
        return dict(bytes=n * 8.0 * (9 + 3 + 6 + 6), flops=150.0 * n)
    if kind == "gradient":
        k = case["steps"]
        if case["form"] == "direct":
            return dict(bytes=n * 8.0 * (8 + 13), flops=n * (n - 1.0) * (30 * (k + 1) + 55 * (k + 1)))
        return dict(bytes=n * 8.0 * (9 + 13), flops=_walk_terms(n, 0.5) * (45 + 150) * (k + 1))
    if kind == "cutoffs":
        return dict(bytes=n * 8.0 * (7 + 2), flops=100.0 * n)
    if kind == "direct":
        return dict(bytes=n * 8.0 * (5 + 3), flops=30.0 * n * (n - 1.0))
    return dict(bytes=n * 8.0 * 7, flops=12.0 * n * (n - 1.0))


# ---- the same outputs in 64-bit torch ----------------------------------------
def _t(s):
    return {k: torch.as_tensor(np.asarray(s[k], dtype=np.float64)).cuda() for k in disks.KEYS}


def _kepler(x, v, dt):
    """The Kepler drift of every particle about a unit mass (bound orbits), by
    the difference of eccentric anomaly; differentiable in x and v."""
    r0 = (x * x).sum(0).sqrt()
    rv = (x * v).sum(0)
    a = 1.0 / (2.0 / r0 - (v * v).sum(0))
    n = a ** -1.5
    ec, es = 1.0 - r0 / a, rv / a.sqrt()

    def f(d):
        return d - ec * torch.sin(d) + es * (1.0 - torch.cos(d)) - n * dt

    def fp(d):
        return 1.0 - ec * torch.cos(d) + es * torch.sin(d)

    with torch.no_grad():
        d = n * dt
        for _ in range(20):
            d = d - f(d) / fp(d)
        slope = fp(d)
    d = d - f(d) / slope  # carries the derivative
    c1, s1 = 2.0 * torch.sin(0.5 * d) ** 2, torch.sin(d)
    fl = 1.0 - a / r0 * c1
    g = dt - (d - s1) / n
    xn = fl * x + g * v
    r = (xn * xn).sum(0).sqrt()
    vn = (-a.sqrt() / (r * r0) * s1) * x + (1.0 - a / r * c1) * v
    return xn, vn


def _pairs(xi, x, m, roi, ro, gamma=0.1):
    """Soft accelerations (3, k) of the targets xi from all sources."""
    d = xi[:, :, None] - x[:, None, :]
    r2 = (d * d).sum(0)
    far = r2 > 0
    r = torch.where(far, r2, torch.ones_like(r2)).sqrt()
    u = ((r / torch.maximum(roi[:, None], ro[None, :]) - gamma) / (1.0 - gamma)).clamp(0.0, 1.0)
    k = u ** 4 * (35.0 - 84.0 * u + 70.0 * u ** 2 - 20.0 * u ** 3)
    w = torch.where(far, m[None, :] * k / r ** 3, torch.zeros_like(r))
    return -(w[None] * d).sum(2)


def _soft(x, m, ro):
    n = x.shape[1]
    step = max(1, 40_000_000 // n)
    return torch.cat([_pairs(x[:, i:i + step], x, m, ro[i:i + step], ro)
                      for i in range(0, n, step)], 1)


def _soft_vjp(x, m, ro, lam):
    """Gradients of (lam . a).sum() with respect to x and m."""
    n = x.shape[1]
    step = max(1, 10_000_000 // n)
    gx, gm = torch.zeros_like(x), torch.zeros_like(m)
    for i in range(0, n, step):
        xg, mg = x.detach().requires_grad_(), m.detach().requires_grad_()
        a = _pairs(xg[:, i:i + step], xg, mg, ro[i:i + step], ro)
        dx, dm = torch.autograd.grad((a * lam[:, i:i + step]).sum(), (xg, mg))
        gx += dx
        gm += dm
    return gx, gm


def _radii(t, mode, dt=1.0 / 64.0):
    """Cut-off and search radii at the default parameters."""
    n = t["m"].numel()
    R2 = t["x"] ** 2 + t["y"] ** 2
    R = R2.sqrt()
    r = (R2 + t["z"] ** 2).sqrt()
    vk = r ** -0.5
    u2 = (t["vx"] + vk * t["y"] / R) ** 2 + (t["vy"] - vk * t["x"] / R) ** 2 + t["vz"] ** 2
    nb = max(1, min(1024, n // 1000))
    l, l0, l1 = R.log(), R.min().log(), R.max().log()
    b = ((l - l0) / (l1 - l0) * nb).floor().clamp(0, nb - 1).long()
    one = torch.ones_like(u2)
    vr = (torch.zeros(nb, dtype=u2.dtype, device=u2.device).index_add_(0, b, u2)
          / torch.zeros(nb, dtype=u2.dtype, device=u2.device).index_add_(0, b, one)).sqrt()[b]
    al = 2.0 / r - (t["vx"] ** 2 + t["vy"] ** 2 + t["vz"] ** 2)
    a = torch.where(al > 0, 1.0 / al, r)
    hill = 2.0 * (t["m"] / 3.0) ** (1.0 / 3.0) * a
    ro = torch.maximum(hill, 8.0 * vr * dt) if mode == 0 else hill
    rs = 1.1 * ro + 6.0 * vr * dt
    if mode == 2:
        ro, rs = ro.max().expand(n).clone(), rs.max().expand(n).clone()
    return ro, rs


def exact(case, seed):
    kind = case["kind"]
    if kind == "cutoffs":
        ro, rs = _radii(_t(_disk(case, seed)), case["mode"])
        return dict(r_out=ro, r_search=rs)
    if kind in ("direct", "energy") or (kind == "force" and case["n"] <= 131_072):
        t = _t(_disk(case, seed))
        x = torch.stack([t["x"], t["y"], t["z"]])
        if kind == "energy":
            n, m = case["n"], t["m"]
            ek = (0.5 * m * (t["vx"] ** 2 + t["vy"] ** 2 + t["vz"] ** 2)).sum()
            es = -(m / (x * x).sum(0).sqrt()).sum()
            ep = torch.zeros((), dtype=torch.float64, device="cuda")
            step = max(1, 40_000_000 // n)
            for i in range(0, n, step):
                d = x[:, i:i + step, None] - x[:, None, :]
                r2 = (d * d).sum(0)
                ep -= 0.5 * (m[i:i + step, None] * m[None, :]
                             * torch.where(r2 > 0, r2.rsqrt(), torch.zeros_like(r2))).sum()
            return dict(e=torch.stack([ek + es + ep, ek, es, ep]))
        ro, _ = _radii(t, 0)
        a = _soft(x, t["m"], ro)
        if kind == "direct":
            return dict(acc=a)
        # the tree's force is this one up to its opening angle; at theta = 0 it is this one
        return dict(acc=a, counts=None, nb_off=None, nb_idx=None)
    if kind == "gradient" and case["form"] == "direct":
        t = _t(disks.adjoint_disk(case["n"], seed))
        x, v = torch.stack([t[k] for k in XV[:3]]), torch.stack([t[k] for k in XV[3:]])
        m, dt = t["m"], 1.0 / 64.0
        ro, _ = _radii(t, 0)
        target, _ = _kepler(x, v, case["steps"] * dt)
        target += torch.as_tensor(disks.target_offsets(case["n"], seed + 1)).cuda()
        kept = []
        a = _soft(x, m, ro)
        for _ in range(case["steps"]):
            v = v + 0.5 * dt * a
            kept.append((x, v))
            x, v = _kepler(x, v, dt)
            a = _soft(x, m, ro)
            v = v + 0.5 * dt * a
        xn, vn = x, v
        lx, lv, gm = 2.0 * (xn - target), torch.zeros_like(vn), torch.zeros_like(m)
        h = 0.5 * dt
        for k in range(case["steps"], -1, -1):
            dx, dm = _soft_vjp(x, m, ro, lv)
            w = h if k in (0, case["steps"]) else dt
            lx, gm = lx + w * dx, gm + w * dm
            if k == 0:
                break
            x, v = kept[k - 1]
            xg, vg = x.detach().requires_grad_(), v.detach().requires_grad_()
            lx, lv = torch.autograd.grad(_kepler(xg, vg, dt), (xg, vg), (lx, lv))
        return dict(x=xn, v=vn, loss=((xn - target) ** 2).sum(), gx=lx, gv=lv, gm=gm)
    # whole steps, the hard part and the tree's gradient follow their own
    # decisions (block steps, lists): no value without them
    return None

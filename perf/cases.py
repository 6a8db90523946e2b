"""Performance cases of the Lennard-Jones framework.

Each case is one call sequence of a user's program through the public Python
entry points (``LJMD`` and the autograd functions), at sizes of the repository's
own workloads: fcc liquids from a few hundred to 16.4 million atoms, batches of
uneven replicas, the charged pair style, the 80:20 mixture with its gradients,
steepest descent, and a driver that holds the state on the host.

Kinds of case (``case["kind"]``):
  md         ``step(steps)``, the thermodynamic state, the whole state back
  batch      the same for many uneven boxes in one context
  force_grad force-matching loss at given positions, forward and backward
  traj_grad  the loss after ``steps`` velocity-Verlet steps, forward and backward
  relax      load positions, ``steps`` steepest-descent steps, state back
  coupled    host buffers -> one step -> host buffers
"""
import math

import numpy as np
import torch

import paper_2508_13523_gb300 as md
from paper_2508_13523_gb300.autograd import lj_forces, lj_trajectory_forces

RC, SKIN, DT = 2.5, 0.3, 0.005
LISTS = {"half": md.MD_LIST_HALF, "full": md.MD_LIST_FULL}
PRECISIONS = {"fp64": md.MD_PREC_FP64, "mixed": md.MD_PREC_MIXED}
# 80:20 A:B mixture (eps, sigma per type pair; rc = 2.5 sigma)
MIX_EPS = ((1.0, 1.5), (1.5, 0.5))
MIX_SIGMA = ((1.0, 0.8), (0.8, 0.88))
CHARGES = (0.5, -0.5)  # lj/cut/coul/cut: +-0.5 by fcc site


# ---- the cases ---------------------------------------------------------------

def _md(name, nx, ny, nz, precision, kind, steps, every=20, check_disp=False, coulomb=False):
    case = dict(kind="md", nx=nx, ny=ny, nz=nz, precision=precision, list=kind, steps=steps,
                every=every, check_disp=check_disp, coulomb=coulomb)
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest boxes: a unit test or a toy run, where launches, the
        # per-step displacement check and host calls are what counts
        _md("small_864_fp64_full", 6, 6, 6, "fp64", "full", 10, check_disp=True),
        # the standard 32,000-atom LJ melt over 100 steps, FP64 half list
        _md("melt_32k_fp64_half", 20, 20, 20, "fp64", "half", 100),
        # the 256,000-atom scaling point with a full list (each pair twice)
        _md("liquid_256k_fp64_full", 40, 40, 40, "fp64", "full", 20),
        # an odd, non-cubic box in mixed precision with a full list
        _md("slab_309k_mixed_full", 47, 31, 53, "mixed", "full", 20),
        # charged fluid: the second pair style, two types
        _md("charged_500k_fp64_half", 50, 50, 50, "fp64", "half", 20, coulomb=True),
        # the production size, FP64 half list
        _md("liquid_4m_fp64_half", 100, 100, 100, "fp64", "half", 20),
        # the largest scaling point, mixed precision half list
        _md("liquid_16m_mixed_half", 160, 160, 160, "mixed", "half", 20),
        # ensemble sampling: 512 uneven boxes of 108 to 32,000 atoms
        dict(name="replicas_512_fp64_half", kind="batch", replicas=512, lo=3, hi=20,
             sizes_seed=7, precision="fp64", list="half", steps=20, every=20),
        # force matching: per-type-pair (eps, sigma) and position gradients
        dict(name="force_grad_64k_fp64", kind="force_grad", nx=20, ny=25, nz=32,
             precision="fp64", list="half"),
        # backprop through 100 steps, a checkpoint every 10
        dict(name="traj_grad_64k_mixed", kind="traj_grad", nx=20, ny=25, nz=32,
             precision="mixed", list="half", steps=100, every=10),
        # relaxing a strained mixture before a run
        dict(name="relax_64k_fp64", kind="relax", nx=20, ny=25, nz=32, precision="fp64",
             list="full", steps=50, every=10),
        # another code holds the state in pinned host memory between steps
        dict(name="coupled_256k_fp64_half", kind="coupled", nx=40, ny=40, nz=40,
             precision="fp64", list="half"),
    ]


def _cells(rng, lo, hi):
    """Box edges in unit cells for about lo..hi atoms (log-uniform), not cubic."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    edge = (n / 4.0) ** (1.0 / 3.0)
    nx, ny = (max(3, round(edge * rng.uniform(0.8, 1.25))) for _ in range(2))
    return nx, ny, max(3, round(n / (4.0 * nx * ny)))


def draw(rng):
    kind = rng.choice(["md", "md", "md", "md", "batch", "force_grad", "traj_grad", "relax",
                       "coupled"])
    precision, lst = rng.choice(["fp64", "mixed"]), rng.choice(["half", "full"])
    if kind == "md":
        nx, ny, nz = _cells(rng, 500, 4.0e6)
        n = 4 * nx * ny * nz
        every = rng.choice([10, 20])
        steps = every * (rng.choice([2, 5]) if n < 100000 else 1)
        return _md(None, nx, ny, nz, precision, lst, steps, every,
                   check_disp=n < 200000 and rng.random() < 0.25,
                   coulomb=rng.random() < 0.25)
    if kind == "batch":
        lo = rng.randint(3, 6)
        return dict(kind=kind, replicas=rng.randint(16, 256), lo=lo, hi=lo + rng.randint(3, 12),
                    sizes_seed=rng.randint(1, 999), precision=precision, list=lst, steps=20,
                    every=20)
    nx, ny, nz = _cells(rng, 4000, 100000)
    case = dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, list=lst)
    if kind == "traj_grad":
        case.update(steps=rng.choice([20, 50]), every=10)
    if kind == "relax":
        case.update(steps=rng.choice([20, 50]), every=10)
    return case


# ---- inputs ------------------------------------------------------------------

def _density(case):
    return 1.2 if case["kind"] in ("force_grad", "traj_grad", "relax") else 0.8442


def _mixture(case):
    return case["kind"] in ("force_grad", "traj_grad", "relax")


def _replica_edges(case):
    """(replicas, 3) edges in unit cells."""
    if case["kind"] != "batch":
        return np.array([[case["nx"], case["ny"], case["nz"]]])
    n = np.random.RandomState(case["sizes_seed"]).randint(case["lo"], case["hi"] + 1,
                                                          case["replicas"])
    return np.repeat(n[:, None], 3, axis=1)


def _inputs(case, seed):
    """Positions (fcc with thermal displacements), velocities, types and boxes."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    a = (4.0 / _density(case)) ** (1.0 / 3.0)
    basis = torch.tensor([[0, 0, 0], [0.5, 0.5, 0], [0.5, 0, 0.5], [0, 0.5, 0.5]],
                         dtype=torch.float64, device=dev)
    edges = _replica_edges(case)
    parts = []
    for e in edges:
        g = torch.meshgrid(*[torch.arange(int(k), dtype=torch.float64, device=dev) for k in e],
                           indexing="ij")
        cells = torch.stack([c.reshape(-1) for c in g], 1)
        parts.append(((cells[:, None, :] + basis) * a).reshape(-1, 3))
    counts = [len(p) for p in parts]
    x = torch.cat(parts)
    n = len(x)
    spread = 0.1 if case["kind"] == "relax" else 0.05
    x = x + spread * torch.randn((n, 3), generator=gen, dtype=torch.float64,
                                 device=dev).clamp_(-2.5, 2.5)
    boxes = edges * a
    rep = torch.repeat_interleave(torch.arange(len(counts), device=dev),
                                  torch.tensor(counts, device=dev))
    temp = torch.ones(len(counts), dtype=torch.float64, device=dev)
    if case["kind"] == "batch":
        temp = 0.7 + 0.8 * torch.rand(len(counts), generator=gen, dtype=torch.float64, device=dev)
    v = torch.randn((n, 3), generator=gen, dtype=torch.float64, device=dev)
    v = v * temp.sqrt()[rep][:, None]
    mean = torch.zeros((len(counts), 3), dtype=torch.float64, device=dev).index_add_(0, rep, v)
    v = v - (mean / torch.tensor(counts, device=dev)[:, None])[rep]
    if _mixture(case):
        t = (torch.rand(n, generator=gen, device=dev) < 0.2).to(torch.int32)
    elif case.get("coulomb"):
        t = (torch.arange(n, device=dev) % 4 >= 2).to(torch.int32)
    else:
        t = torch.zeros(n, dtype=torch.int32, device=dev)
    return dict(x=x.contiguous(), v=v.contiguous(), t=t, rep=rep, boxes=boxes, counts=counts)


def _tables(case):
    """eps, sigma, rc per type pair and the number of types."""
    if _mixture(case):
        sigma = np.array(MIX_SIGMA)
        return np.array(MIX_EPS), sigma, 2.5 * sigma, 2
    nt = 2 if case.get("coulomb") else 1
    return np.ones((nt, nt)), np.ones((nt, nt)), np.full((nt, nt), RC), nt


def prepare(case, seed):
    s = _inputs(case, seed)
    eps, sigma, rc, nt = _tables(case)
    kw = {}
    if case["kind"] == "batch":
        kw["rep_offset"] = np.concatenate([[0], np.cumsum(s["counts"])])
    ctx = md.LJMD(s["x"], s["v"], s["t"], s["boxes"], eps, sigma, rc, np.ones(nt), skin=SKIN,
                  dt=DT, list_kind=LISTS[case["list"]], precision=PRECISIONS[case["precision"]],
                  rebuild_every=case.get("every", 20), threads_per_atom=0,
                  check_disp=case.get("check_disp", False), **kw)
    state = dict(kind=case["kind"], steps=case.get("steps"), every=case.get("every"), ctx=ctx)
    if case.get("coulomb"):
        ctx.set_coulomb(CHARGES, RC)
    if case["kind"] in ("force_grad", "traj_grad"):
        dev = s["x"].device
        te, ts = (torch.tensor(w, dtype=torch.float64, device=dev) for w in (eps, sigma))
        x, v = s["x"], s["v"]
        with torch.no_grad():  # the target: the same model at parameters 5 % larger
            if case["kind"] == "force_grad":
                target = lj_forces(x, 1.05 * te, 1.05 * ts, ctx)
            else:
                target = lj_trajectory_forces(x, v, 1.05 * te, 1.05 * ts, ctx, case["steps"],
                                              case["every"])
        state.update(x=x.requires_grad_(True), v=v.requires_grad_(True),
                     eps=te.requires_grad_(True), sigma=ts.requires_grad_(True), target=target)
    if case["kind"] == "relax":
        state.update(x=s["x"], v=torch.zeros_like(s["v"]))
    if case["kind"] == "coupled":
        state.update(x=torch.empty(s["x"].shape, dtype=torch.float64, pin_memory=True),
                     v=torch.empty(s["x"].shape, dtype=torch.float64, pin_memory=True))
        ctx.get_state_into(state["x"], state["v"], None, md.MD_MEM_HOST)
    return state


# ---- one pass ----------------------------------------------------------------

def run(state):
    ctx, kind = state["ctx"], state["kind"]
    if kind == "md":
        ctx.step(state["steps"])
        th = ctx.energy()
        x, v, f = ctx.get_state()
        return dict(x=x, v=v, f=f, energy=np.array([th.pe, th.ke, th.temperature]),
                    virial=th.virial)
    if kind == "batch":
        ctx.step(state["steps"])
        th = ctx.energy_replicas()
        x, v, f = ctx.get_state()
        return dict(x=x, v=v, f=f, thermo=th)
    if kind in ("force_grad", "traj_grad"):
        if kind == "force_grad":
            inputs = (state["x"], state["eps"], state["sigma"])
            f = lj_forces(*inputs, ctx)
        else:
            inputs = (state["x"], state["v"], state["eps"], state["sigma"])
            f = lj_trajectory_forces(*inputs, ctx, state["steps"], state["every"])
        loss = ((f - state["target"]) ** 2).sum()
        grads = torch.autograd.grad(loss, inputs)
        return dict(f=f.detach(), loss=loss.detach(), grads=list(grads))
    if kind == "relax":
        ctx.set_state(state["x"], state["v"])
        ctx.minimize(state["steps"], 0.01)
        x, _, f = ctx.get_state()
        return dict(x=x, f=f)
    # coupled
    ctx.set_state_from(state["x"], state["v"], md.MD_MEM_HOST | md.MD_MEM_KEEP_LIST)
    ctx.step(1)
    ctx.get_state_into(state["x"], state["v"], None, md.MD_MEM_HOST)
    return dict(x=state["x"], v=state["v"])


# ---- what a pass cannot do without --------------------------------------------

def work(case):
    """Bytes: the state in and the results out, once.  Operations: about 25 per
    pair inside the cutoff per force evaluation (70 with its derivative), each
    pair once."""
    n = float(4 * np.prod(_replica_edges(case), axis=1).sum())
    if _mixture(case):  # mean of (2.5 sigma_ab)^3 over 80:20 pairs
        rc3 = 2.5 ** 3 * (0.64 + 0.32 * 0.8 ** 3 + 0.04 * 0.88 ** 3)
    else:
        rc3 = RC ** 3
    pairs = n * 0.5 * 4.0 / 3.0 * math.pi * rc3 * _density(case)
    kind, steps = case["kind"], case.get("steps") or 1
    if kind == "force_grad":
        return {"bytes": n * (24 + 4 + 48), "flops": pairs * 95.0}
    if kind == "traj_grad":
        return {"bytes": n * (48 + 4 + 72), "flops": pairs * steps * 95.0}
    if kind == "relax":
        return {"bytes": n * (24 + 4 + 48), "flops": pairs * steps * 25.0}
    if kind == "coupled":
        return {"bytes": n * (48 + 4 + 48), "flops": pairs * 25.0}
    ops = 32.0 if case.get("coulomb") else 25.0
    return {"bytes": n * (48 + 4 + 72), "flops": pairs * (steps + 1) * ops}


# ---- the same answers in plain torch, 64 bits ----------------------------------

class _Exact:
    """Velocity Verlet, steepest descent and Eq. 1 with plain tensor operations;
    unordered pairs (i, j) within max rc + skin, listed when the framework's
    contract says that the list is built."""

    def __init__(self, case, s):
        self.case = case
        self.dev = s["x"].device
        self.rep, self.t = s["rep"], s["t"].long()
        self.boxes = torch.tensor(s["boxes"], dtype=torch.float64, device=self.dev)
        self.single = len(self.boxes) == 1
        self.L = self.boxes if self.single else self.boxes[self.rep]
        self.n = len(s["x"])
        eps, sigma, rc, self.nt = _tables(case)
        tab = lambda w: torch.tensor(w, dtype=torch.float64, device=self.dev)
        self.eps, self.sigma, self.rc2 = tab(eps), tab(sigma), tab(rc) ** 2
        self.rlist = float(rc.max()) + SKIN
        q = tab(CHARGES) if case.get("coulomb") else None
        self.qq = None if q is None else q[:, None] * q[None, :]

    def wrap(self, x):
        w = x - self.L * torch.floor(x / self.L)
        return torch.where(w == self.L, torch.zeros_like(w), w)

    def edge(self, i):
        return self.L if self.single else self.L[i]

    def pairs(self, x):
        nc = torch.floor(self.boxes / self.rlist * (1 - 1e-9)).long()
        nc = torch.where(nc < 3, torch.ones_like(nc), nc)  # (boxes, 3)
        size = nc.prod(1)
        base = torch.cumsum(size, 0) - size
        c3 = (x / self.L * nc[self.rep]).long().clamp_(min=0)
        c3 = torch.minimum(c3, nc[self.rep] - 1)
        cid = lambda c, m, b: b + (c[:, 0] * m[:, 1] + c[:, 1]) * m[:, 2] + c[:, 2]
        cell = cid(c3, nc[self.rep], base[self.rep])
        count = torch.bincount(cell, minlength=int(size.sum()))
        start = torch.cumsum(count, 0) - count
        order = torch.argsort(cell)
        out = []
        step = max(1000, int(4.0e7 / max(1.0, float(count[cell].double().mean()))))
        for lo in range(0, self.n, step):
            i = order[lo:lo + step]
            m, b, ci = nc[self.rep[i]], base[self.rep[i]], c3[i]
            for off in range(27):
                o = torch.tensor([off // 9 - 1, off // 3 % 3 - 1, off % 3 - 1], device=self.dev)
                ok = ((m > 1) | (o == 0)).all(1)
                q = cid((ci + o) % m, m, b)
                k = torch.where(ok, count[q], torch.zeros_like(q))
                end = torch.cumsum(k, 0)
                r = torch.repeat_interleave(torch.arange(len(i), device=self.dev), k)
                at = torch.arange(len(r), device=self.dev) - (end - k)[r] + start[q][r]
                ir, j = i[r], order[at]
                keep = ir < j
                ir, j = ir[keep], j[keep]
                d = x[j] - x[ir]
                L = self.edge(ir)
                d = d - L * torch.round(d / L)
                keep = (d * d).sum(1) < self.rlist ** 2
                out.append((ir[keep].int(), j[keep].int()))
        return torch.cat([p[0] for p in out]), torch.cat([p[1] for p in out])

    def _pair_terms(self, x, i, j, eps, sigma):
        """Separation, force factor and energy of each pair (zero outside rc)."""
        L = self.edge(i)
        d = x[j] - x[i]
        d = d - L * torch.round(d.detach() / L)
        r2 = (d * d).sum(1)
        ab = self.t[i] * self.nt + self.t[j]
        inside = r2.detach() < self.rc2.reshape(-1)[ab]
        s6 = (sigma.reshape(-1)[ab] ** 2 / r2) ** 3
        e = torch.where(inside, eps.reshape(-1)[ab], torch.zeros_like(r2))
        fpair = 24.0 * e * s6 * (2.0 * s6 - 1.0) / r2
        energy = 4.0 * e * s6 * (s6 - 1.0)
        if self.qq is not None:
            qr = torch.where(r2 < RC ** 2, self.qq.reshape(-1)[ab], torch.zeros_like(r2))
            qr = qr / r2.sqrt()
            fpair, energy = fpair + qr / r2, energy + qr
        return d, fpair, energy

    def forces(self, x, pairs, thermo=False):
        f = torch.zeros_like(x)
        nrep = len(self.boxes)
        pe = torch.zeros(nrep, dtype=torch.float64, device=self.dev)
        w = torch.zeros((nrep, 6), dtype=torch.float64, device=self.dev)
        for i, j in zip(*(torch.split(p, 20000000) for p in pairs)):
            d, fpair, energy = self._pair_terms(x, i, j, self.eps, self.sigma)
            g = fpair[:, None] * d
            f.index_add_(0, j, g)
            f.index_add_(0, i, -g)
            if thermo:
                r = self.rep[i]
                pe.index_add_(0, r, energy)
                w.index_add_(0, r, torch.cat([g * d, g[:, :1] * d[:, 1:2], g[:, :1] * d[:, 2:],
                                              g[:, 1:2] * d[:, 2:]], 1))
        return (f, pe, w) if thermo else f

    def forces_of(self, x, eps, sigma, pairs):
        """Differentiable forces; tables are used as (T + T^T) / 2."""
        i, j = pairs
        d, fpair, _ = self._pair_terms(x, i, j, 0.5 * (eps + eps.t()), 0.5 * (sigma + sigma.t()))
        g = fpair[:, None] * d
        return torch.zeros_like(x).index_add(0, j, g).index_add(0, i, -g)

    def run_md(self, x, v, steps, every, check):
        h = 0.5 * DT  # unit masses
        x = self.wrap(x)
        pairs, at = self.pairs(x), x
        f = self.forces(x, pairs)
        for s in range(steps):
            v = v + h * f
            x = x + DT * v
            moved = check and float(((x - at) ** 2).sum(1).max()) > (0.5 * SKIN) ** 2 * (1 - 1e-5)
            if (s + 1) % every == 0 or moved:
                x = self.wrap(x)
                pairs, at = self.pairs(x), x
            f = self.forces(x, pairs)
            v = v + h * f
        return x, v, pairs

    def traj_forces(self, x, v, eps, sigma, steps, every):
        from torch.utils.checkpoint import checkpoint
        h = 0.5 * DT
        f_at = lambda y, p: checkpoint(self.forces_of, y, eps, sigma, p, use_reentrant=False)
        x = x - self.L * torch.floor(x.detach() / self.L)
        pairs = self.pairs(x.detach())
        f = f_at(x, pairs)
        for s in range(steps):
            v = v + h * f
            x = x + DT * v
            if (s + 1) % every == 0:
                x = x - self.L * torch.floor(x.detach() / self.L)
                pairs = self.pairs(x.detach())
            f = f_at(x, pairs)
            v = v + h * f
        return f


def exact(case, seed):
    s = _inputs(case, seed)
    ref = _Exact(case, s)
    x, v, kind = s["x"], s["v"], case["kind"]
    if kind in ("md", "batch"):
        x, v, pairs = ref.run_md(x, v, case["steps"], case["every"],
                                 case.get("check_disp", False))
        f, pe, w = ref.forces(x, pairs, thermo=True)
        ke = torch.zeros_like(pe).index_add_(0, ref.rep, 0.5 * (v * v).sum(1))
        dof = 3.0 * torch.tensor(s["counts"], dtype=torch.float64, device=x.device) - 3.0
        if kind == "md":
            # where a displacement starts a rebuild, the step at which an atom
            # is wrapped is the framework's own choice
            return dict(x=None if case["check_disp"] else x, v=v, f=f,
                        energy=torch.stack([pe[0], ke[0], 2.0 * ke[0] / dof[0]]), virial=w[0])
        th = torch.cat([pe[:, None], ke[:, None], (pe + ke)[:, None], (2.0 * ke / dof)[:, None],
                        w], 1)
        return dict(x=x, v=v, f=f, thermo=th)
    if kind == "relax":
        x = ref.wrap(x)
        pairs = ref.pairs(x)
        for k in range(case["steps"]):
            if k > 0 and k % case["every"] == 0:
                x = ref.wrap(x)
                pairs = ref.pairs(x)
            f = ref.forces(x, pairs)
            x = x + (0.01 / f.norm(dim=1).max()) * f
        x = ref.wrap(x)
        return dict(x=x, f=ref.forces(x, ref.pairs(x)))
    if kind == "coupled":
        x, v, _ = ref.run_md(x, v, 1, 20, False)
        return dict(x=x, v=v)
    eps, sigma = ref.eps.requires_grad_(True), ref.sigma.requires_grad_(True)
    x, v = x.requires_grad_(True), v.requires_grad_(True)
    if kind == "force_grad":
        inputs = (x, eps, sigma)
        at = lambda e, g: ref.forces_of(x, e, g, pairs)
        pairs = ref.pairs(ref.wrap(x.detach()))
    else:
        inputs = (x, v, eps, sigma)
        at = lambda e, g: ref.traj_forces(x, v, e, g, case["steps"], case["every"])
    with torch.no_grad():
        target = at(1.05 * eps, 1.05 * sigma)
    f = at(eps, sigma)
    loss = ((f - target) ** 2).sum()
    grads = torch.autograd.grad(loss, inputs)
    return dict(f=f.detach(), loss=loss.detach(), grads=list(grads))

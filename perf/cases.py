"""Performance cases of the batched Hines solver, through its public entry points.

A case is one call (or one captured rollout) of `hines` / `rollout` on a seeded
synthetic population.  The populations are the ones of `inputs.WORKLOADS`
(branch counts, branch lengths, split probabilities, coefficient ranges) at
several cell counts: the smallest batch is latency and launches, the largest
streams far more than the caches hold.  To keep preparation quick the cells of
a class take their branch trees from a pool of `POOL` shapes, each cell with
its own branch lengths (network models instantiate a few reconstructed morphologies
many times).  The morphology belongs to the case, coefficients and right-hand
sides to the seed: a program plans once and solves with many values.

`op` of a case:
  solve       hines.solve, dtype f64 / f32, natural or solver layout
  comp        hines.solve_compensated (FP32 in, FP64 out), both layouts
  refine      hines.solve_refine with `steps` refinement steps
  cable       rollout.CableStepper: `steps` implicit-Euler steps in one CUDA
              graph, both layouts, with or without factor re-use
  rollout     rollout.CableRollout: loss of a rollout and its gradients
  autograd    rollout.HinesSolve forward and backward
  pipeline    hines.HostPipeline: the compensated solve from pinned host arrays
"""
from __future__ import annotations

import numpy as np
import torch

from paper_1810_12742_gb300 import hines as H
from paper_1810_12742_gb300 import inputs as I
from paper_1810_12742_gb300 import rollout as R

POOL = 24           # branch-tree shapes per cell class
DT, E = 0.025, -65.0

_W = I.WORKLOADS
# population -> (classes, share of the cells in each class)
POPULATIONS = {
    "binary31": (_W["fp64_small"].classes, (1.0,)),
    "uniform": (_W["fp64_uniform"].classes, (1.0,)),
    "small": (_W["uneven_mixed"].classes[:1], (1.0,)),
    "large": (_W["uneven_mixed"].classes[1:], (1.0,)),
    "uneven": (_W["uneven_mixed"].classes, _W["uneven_mixed"].class_frac),
    "adjoint": (_W["adjoint"].classes, (1.0,)),
}


def listed():
    return [
        # one time step's solve of a small circuit: launch and chain latency
        dict(name="f64_64_cells", op="solve", dtype="f64", layout="natural", pop="binary31", cells=64),
        # a handful of detailed reconstructions, each cut into subtrees and a top part
        dict(name="f64_37_large_cells", op="solve", dtype="f64", layout="natural", pop="large", cells=37),
        # a whole network of mid-size cells in FP64 (the uniform workload at its full size)
        dict(name="f64_uniform_16384", op="solve", dtype="f64", layout="natural", pop="uniform", cells=16384),
        # single precision, an odd number of simplified cells
        dict(name="f32_1001_small_cells", op="solve", dtype="f32", layout="natural", pop="small", cells=1001),
        # the mixed-morphology population, FP32 coefficients in, FP64 solution out
        dict(name="comp_uneven_1024", op="comp", layout="natural", pop="uneven", cells=1024),
        # the same solve for a simulation that keeps its arrays in the solver layout
        dict(name="comp_uneven_777_packed", op="comp", layout="solver", pop="uneven", cells=777),
        # FP32 elimination with two refinement steps
        dict(name="refine2_uneven_301", op="refine", steps=2, pop="uneven", cells=301),
        # simulation main loop, natural layout: matrix and right-hand side rebuilt every step
        dict(name="cable_uneven_512", op="cable", steps=10, theta=1, layout="natural", reuse=False, reroot=False,
             pop="uneven", cells=512),
        # simulation main loop of a mid-size network, solver layout of re-rooted cells, factor kept after the
        # first step; the state comes back to the natural layout
        dict(name="cable_uniform_500_reuse", op="cable", steps=40, theta=1, layout="solver", reuse=True, reroot=True,
             pop="uniform", cells=500),
        # parameter fitting: loss and gradients of a rollout with checkpoints
        dict(name="rollout_256", op="rollout", steps=40, every=20, theta=1, pop="adjoint", cells=256),
        # one differentiable solve inside a larger model
        dict(name="autograd_uniform_1000", op="autograd", pop="uniform", cells=1000),
        # the solve for a program whose arrays live in host memory
        dict(name="pipeline_uneven_256", op="pipeline", pieces=8, pop="uneven", cells=256),
    ]


# largest cell count of each population: the compartments of the largest listed case, or fewer
_MOST_CELLS = {"binary31": 65536, "uniform": 16384, "small": 16384, "large": 400, "uneven": 1400, "adjoint": 4096}


def _mean_compartments(case):
    classes, frac = POPULATIONS[case["pop"]]
    return case["cells"] * sum(f * (c.branches[0] + c.branches[1]) / 2 * (c.lengths[0] + c.lengths[1]) / 2
                               for c, f in zip(classes, frac))


def draw(rng):
    op = rng.choice(["solve", "solve", "comp", "comp", "refine", "cable", "cable", "rollout", "autograd", "pipeline"])
    pop = rng.choice(["adjoint", "uniform"] if op == "rollout" else list(POPULATIONS))
    # cells, log-uniform; iterated calls stop at smaller batches so that no
    # drawn case does more work than the largest listed one
    most = _MOST_CELLS[pop]
    if op in ("cable", "rollout", "refine", "autograd", "pipeline"):
        most = max(4, most // 8)
    if op == "rollout":
        most = min(most, 400)
    least = {"binary31": 32, "large": 2}.get(pop, 8)
    cells = int(round(least * (most / least) ** rng.random()))
    case = dict(op=op, pop=pop, cells=cells)
    if op == "solve":
        case.update(dtype=rng.choice(["f64", "f64", "f32"]), layout=rng.choice(["natural", "natural", "solver"]))
    elif op == "comp":
        case.update(layout=rng.choice(["natural", "solver"]))
    elif op == "refine":
        case.update(steps=rng.choice([1, 2, 3]))
    elif op == "cable":
        layout = rng.choice(["natural", "solver"])
        case.update(steps=rng.randint(4, 16), theta=rng.choice([1, 1, 0]), layout=layout,
                    reuse=rng.random() < 0.4, reroot=layout == "solver" and rng.random() < 0.5)
    elif op == "rollout":
        case.update(steps=rng.randint(12, 40), every=rng.choice([10, 20]), theta=rng.choice([1, 1, 0]))
    elif op == "pipeline":
        case.update(pieces=rng.choice([1, 4, 8, 16]))
    return case


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _morphology(case):
    """Cells in Hines order: per branch (parent branch, first compartment,
    length, level; branches of all cells in a row) and the batch's parent array."""
    classes, frac = POPULATIONS[case["pop"]]
    rng = np.random.default_rng(I.SEED_BASE)
    n = case["cells"]
    counts = [int(round(f * n)) for f in frac]
    counts[0] = n - sum(counts[1:])
    cls = rng.permutation(np.repeat(np.arange(len(classes)), counts))
    pools = []
    for k, c in enumerate(classes):
        pool = []
        for _ in range(min(POOL, counts[k])):
            nb = int(rng.integers(c.branches[0], c.branches[1] + 1))
            pool.append(I.grow_branch_tree(rng, nb, c.p_split, c.p_ternary, c.depth_cap))
        pools.append(pool)
    shape = [pools[k][int(j) % len(pools[k])] for k, j in zip(cls, rng.integers(0, POOL, n))]
    nb = np.array([s[0].size for s in shape], np.int64)
    boff = np.concatenate(([0], np.cumsum(nb)))
    bparent = np.concatenate([s[0] for s in shape]).astype(np.int64)
    level = np.concatenate([s[1] for s in shape])
    lo = np.repeat(np.array([classes[k].lengths[0] for k in cls]), nb)
    hi = np.repeat(np.array([classes[k].lengths[1] for k in cls]), nb)
    blen = rng.integers(lo, hi + 1)
    bfirst = np.concatenate(([0], np.cumsum(blen)))
    total = int(bfirst[-1])
    bfirst = bfirst[:-1]
    bpar = np.where(bparent >= 0, bparent + np.repeat(boff[:-1], nb), -1)
    plast = np.where(bpar >= 0, (bfirst + blen - 1)[np.maximum(bpar, 0)], -1)  # global parent compartment
    off = np.concatenate((bfirst[boff[:-1]], [total]))
    ncomp = np.diff(off).astype(np.int32)
    # inside a branch the parent is the compartment before; at its start, the parent branch's last one
    local = torch.arange(total, dtype=torch.int64, device="cuda")
    cell0 = torch.repeat_interleave(torch.as_tensor(off[:-1], device="cuda"),
                                    torch.as_tensor(np.diff(off), device="cuda"))
    parent = local - cell0 - 1
    first = torch.as_tensor(bfirst, device="cuda")
    pl = torch.as_tensor(plast, device="cuda")
    parent[first] = torch.where(pl >= 0, pl - cell0[first], torch.full_like(pl, -1))
    host_parent = parent.to(torch.int32).cpu().numpy()
    return dict(ncomp=ncomp, parent=host_parent, off=off, bfirst=first, blen=blen, bpar=bpar, plast=pl, level=level,
                n=total)


def _edge_sum(m, a):
    """sum of a over the edges at every compartment (edge i joins i and its parent); a fixed order of additions."""
    out = a.clone()
    inner = torch.ones(m["n"], dtype=torch.bool, device="cuda")  # compartments whose parent is the one before
    inner[m["bfirst"]] = False
    out[:-1] += torch.where(inner[1:], a[1:], torch.zeros_like(a[1:]))
    bpar = torch.as_tensor(m["bpar"], device="cuda")
    # children of one branch are neighbours in the branch order: rank among siblings
    k = torch.arange(bpar.numel(), device="cuda")
    start = torch.ones_like(bpar, dtype=torch.bool)
    start[1:] = bpar[1:] != bpar[:-1]
    rank = k - torch.cummax(torch.where(start, k, torch.zeros_like(k)), 0).values
    for r in range(8):
        pick = (rank == r) & (bpar >= 0)
        out[m["plast"][pick]] += a[m["bfirst"][pick]]
    assert int(rank[bpar >= 0].max() if bool((bpar >= 0).any()) else 0) < 8
    return out


def _coefficients(m, case, seed):
    """The workloads' distributions, drawn on the GPU: a, s, u, d, b and for time steps g, V0, target."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 977 + 13)

    def uniform(lo, hi, k=m["n"]):
        return torch.empty(k, dtype=torch.float64, device="cuda").uniform_(lo, hi, generator=gen)
    a = uniform(0.5, 2.0)
    a[torch.as_tensor(m["off"][:-1], device="cuda")] = 0.0
    c = dict(a=a, s=uniform(0.01, 0.1), u=-a)
    if case["op"] in ("cable", "rollout"):
        c.update(g=uniform(0.1, 1.0), V0=uniform(-80.0, -50.0), target=uniform(-70.0, -50.0, m["ncomp"].size))
    else:
        c.update(d=c["s"] + _edge_sum(m, a), b=uniform(-1.0, 1.0))
        if case["op"] in ("comp", "refine", "pipeline") or case.get("dtype") == "f32":
            for k in ("d", "u", "b"):
                c[k] = c[k].to(torch.float32)
    return c


def prepare(case, seed):
    m = _morphology(case)
    c = _coefficients(m, case, seed)
    op = case["op"]
    st = dict(op=op, case=case)
    if op == "pipeline":
        st["pipe"] = H.HostPipeline(m["ncomp"], m["parent"], pieces=case["pieces"])
        for k in ("d", "u", "b"):
            st[k] = c[k].cpu().pin_memory()
        st["x"] = torch.empty(m["n"], dtype=torch.float64).pin_memory()
        return st
    plan = st["plan"] = H.Plan(m["ncomp"], m["parent"], reroot=bool(case.get("reroot", False)))
    if op == "cable":
        st["V"] = c["V0"].clone()
        st["stepper"] = R.CableStepper(plan, c["s"], c["g"], c["u"], st["V"], DT, E, theta=case["theta"],
                                       steps=case["steps"], layout=case["layout"], reuse_factor=case["reuse"])
        st["keep"] = c  # the graph reads the caller's arrays
    elif op == "rollout":
        st.update(g=c["g"].requires_grad_(), a=c["a"].requires_grad_(), s=c["s"], V0=c["V0"], target=c["target"])
        R.rollout_graphs(plan, case["steps"], DT, E, case["theta"], case["every"])  # kept with the plan
    elif op == "autograd":
        st.update({k: c[k].requires_grad_() for k in ("d", "u", "b")})
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 5)
        st["xbar"] = torch.empty_like(c["b"]).uniform_(-1.0, 1.0, generator=gen)
    else:
        if case.get("layout") == "solver":
            for k in ("d", "u", "b"):
                c[k] = (H.pack_coupling if k == "u" else H.pack)(plan, c[k])
        st.update({k: c[k] for k in ("d", "u", "b")})
        st["x"] = torch.zeros(c["b"].numel(), dtype=c["b"].dtype if op == "solve" else torch.float64, device="cuda")
    return st


def run(st):
    op, case = st["op"], st["case"]
    if op == "solve":
        st["x"].copy_(st["b"])  # the solve is in place: this step's right-hand side goes into its array
        (H.solve_packed if case["layout"] == "solver" else H.solve)(st["plan"], st["d"], st["u"], st["x"])
        return _owned(st, st["x"])
    if op == "comp":
        f = H.solve_compensated_packed if case["layout"] == "solver" else H.solve_compensated
        return _owned(st, f(st["plan"], st["d"], st["u"], st["b"], st["x"]))
    if op == "refine":
        return H.solve_refine(st["plan"], st["d"], st["u"], st["b"], st["x"], steps=case["steps"])
    if op == "cable":
        st["stepper"].replay()
        return st["stepper"].fetch()
    if op == "rollout":
        loss = R.CableRollout.apply(st["g"], st["a"], st["plan"], st["s"], st["V0"], st["target"], case["steps"], DT, E,
                                    case["theta"], case["every"])
        gg, ga = torch.autograd.grad(loss, (st["g"], st["a"]))
        return {"loss": loss.detach(), "grad_g": gg, "grad_a": ga}
    if op == "autograd":
        x = R.HinesSolve.apply(st["plan"], st["d"], st["u"], st["b"])
        gd, gu, gb = torch.autograd.grad(x, (st["d"], st["u"], st["b"]), st["xbar"])
        return {"x": x.detach(), "grad_d": gd, "grad_u": gu, "grad_b": gb}
    if op == "pipeline":
        return st["pipe"].solve_compensated(st["d"], st["u"], st["b"], st["x"])
    raise ValueError(op)


def _owned(st, x):
    """Solver-layout outputs: the padding slots are unspecified, so the values come back without them."""
    if st["case"].get("layout") != "solver":
        return x
    return H.unpack(st["plan"], x)


def work(case):
    """One pass: each input read and each output written once (per time step where a pass makes several), and the
    operations of the elimination (quotient, two multiply-adds) and the substitution (a multiply-add, a multiply)."""
    n, op = _mean_compartments(case), case["op"]
    if op == "solve":
        w = 8 if case["dtype"] == "f64" else 4
        return {"bytes": 4 * w * n, "flops": 9 * n}
    if op in ("comp", "pipeline"):
        return {"bytes": 20 * n, "flops": 9 * n}
    if op == "refine":
        return {"bytes": 20 * n, "flops": (9 + 16 * case["steps"]) * n}
    if op == "cable":
        per = 9 if case["reuse"] else 16
        return {"bytes": 40 * n * case["steps"], "flops": per * n * case["steps"]}
    if op == "rollout":  # forward step; recomputed step, adjoint solve and gradient accumulation
        return {"bytes": (40 + 40 + 40 + 32) * n * case["steps"], "flops": (16 + 16 + 14 + 12) * n * case["steps"]}
    return {"bytes": (32 + 56) * n, "flops": (9 + 9 + 5) * n}  # autograd


# ----------------------------------------------------------------------------
# the same in 64 bits: plain torch, compartments of equal depth at once
# ----------------------------------------------------------------------------
class _Tree:
    def __init__(self, m):
        level, bpar, blen = m["level"], m["bpar"], m["blen"]
        d0 = np.zeros(level.size, np.int64)  # depth of each branch's first compartment
        order = np.argsort(level, kind="stable")
        cut = np.searchsorted(level[order], np.arange(int(level.max()) + 2))
        for k in range(1, int(level.max()) + 1):
            b = order[cut[k]:cut[k + 1]]
            d0[b] = d0[bpar[b]] + blen[bpar[b]]
        lens = torch.as_tensor(blen, device="cuda")
        depth = torch.repeat_interleave(torch.as_tensor(d0, device="cuda") - m["bfirst"], lens)
        depth += torch.arange(m["n"], device="cuda")
        self.perm = torch.sort(depth, stable=True).indices  # depth order -> natural
        counts = torch.bincount(depth).cpu().numpy()
        self.cut = np.concatenate(([0], np.cumsum(counts)))
        inv = torch.empty_like(self.perm)
        inv[self.perm] = torch.arange(m["n"], device="cuda")
        parent = torch.arange(m["n"], device="cuda") - 1
        parent[m["bfirst"]] = m["plast"]
        p = parent[self.perm]
        self.par = torch.where(p >= 0, inv[p.clamp(min=0)], torch.zeros_like(p))
        self.global_parent = parent
        self.roots = torch.as_tensor(m["off"][:-1], device="cuda")

    def factor(self, d, u):
        D, u = d[self.perm].clone(), u[self.perm]
        f = torch.zeros_like(D)
        for k in range(len(self.cut) - 2, 0, -1):
            a, b = self.cut[k], self.cut[k + 1]
            f[a:b] = u[a:b] / D[a:b]
            D.index_add_(0, self.par[a:b], -f[a:b] * u[a:b])
        return D, u, f

    def solve(self, fac, b):
        D, u, f = fac
        B = b[self.perm].clone()
        for k in range(len(self.cut) - 2, 0, -1):
            i, j = self.cut[k], self.cut[k + 1]
            B.index_add_(0, self.par[i:j], -f[i:j] * B[i:j])
        B /= D
        for k in range(1, len(self.cut) - 1):
            i, j = self.cut[k], self.cut[k + 1]
            B[i:j] -= f[i:j] * B[self.par[i:j]]
        x = torch.empty_like(B)
        x[self.perm] = B
        return x


def exact(case, seed):
    m = _morphology(case)
    op = case["op"]
    c = {k: v.double() for k, v in _coefficients(m, case, seed).items()}
    T = _Tree(m)
    if op == "autograd":
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 5)
        xbar = torch.empty_like(c["b"]).uniform_(-1.0, 1.0, generator=gen)
        fac = T.factor(c["d"], c["u"])
        x, lam = T.solve(fac, c["b"]), T.solve(fac, xbar)
        p = T.global_parent.clamp(min=0)
        gu = torch.where(T.global_parent >= 0, -(lam * x[p] + lam[p] * x), torch.zeros_like(x))
        return {"x": x, "grad_d": -lam * x, "grad_u": gu, "grad_b": lam}
    if op in ("cable", "rollout"):
        th, s, g, u = case["theta"], c["s"], c["g"], c["u"]
        d = s * (1 + th * DT * g) + _edge_sum(m, c["a"])
        fac = T.factor(d, u)

        def rhs(V):
            return s * V + s * DT * g * (E - (1 - th) * V)
        V = c["V0"]
        if op == "cable":
            for _ in range(case["steps"]):
                V = T.solve(fac, rhs(V))
            return V
        states = [V]
        loss = torch.zeros((), dtype=torch.float64, device="cuda")
        for _ in range(case["steps"]):
            states.append(T.solve(fac, rhs(states[-1])))
            loss = loss + (states[-1][T.roots] - c["target"]).square().sum()
        p = T.global_parent.clamp(min=0)
        inner = T.global_parent >= 0
        gg, ga, vbar = (torch.zeros_like(V) for _ in range(3))
        for k in range(case["steps"], 0, -1):
            vbar[T.roots] += 2 * (states[k][T.roots] - c["target"])
            lam = T.solve(fac, vbar)
            gg += lam * s * DT * (E - (1 - th) * states[k - 1]) - th * s * DT * lam * states[k]
            ga -= torch.where(inner, (lam - lam[p]) * (states[k] - states[k][p]), torch.zeros_like(lam))
            vbar = lam * s * (1 - (1 - th) * DT * g)
        return {"loss": loss, "grad_g": gg, "grad_a": ga}
    return T.solve(T.factor(c["d"], c["u"]), c["b"])

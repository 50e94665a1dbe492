"""What the solver is measured on: calls that a program makes through the package's public entry points, from the
smallest solve to the largest instance, the plain method, training steps through the adjoint, and the features.

Instances are the repository's own generators at its benchmark's and tests' sizes.  A case fixes the rows (a program
solves and trains on one instance set many times); the seed draws the costs and every per-slot vector.  Vectors of a program are indexed by (row, variable) in CSR order, so inputs
enter through ``from_csr`` (before the call) and results leave through ``to_csr`` (inside it).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import workloads
from paper_2205_11638_gb300 import solver
from paper_2205_11638_gb300.solver import DualIterate, LowerBound, NonParamUpdate, ParamTransform

SMOOTHING = (1.0, 10.0, 100.0)


def listed():
    return [
        # the smallest solve: one tile of BDDs, where a call is nothing but latency and launches
        dict(name="set_cover_24_solve", do="solve", rows="set_cover", n=24, m=16, kmin=3, kmax=8, iters=100),
        # independent set on 10,000 nodes, 40,000 two-variable rows, 200 iterations: state that stays on the chip
        dict(name="independent_set_10k_solve", do="solve", rows="independent_set", n=10_000, iters=200),
        # a training step on one graph-matching instance with quadratic terms: 20 unrolled iterations, a checkpoint
        # every 10, gradients of the predicted parameters
        dict(name="matching_200_train", do="train", rows="matching", L=200, pairs=20_000, iters=20, every=10),
        # 64 uneven instances in one arena, 50 iterations replayed from a CUDA graph: batched inference
        dict(name="batch_64_solve_graph", do="solve", rows="batch", num=64, iters=50, graph=True),
        # a training step on a batch of 16 uneven instances
        dict(name="batch_16_train", do="train", rows="batch", num=16, iters=20, every=10),
        # a mid-sized tracking instance with predicted (per-slot) damping and averaging weights
        dict(name="tracking_50x400_solve_per_slot", do="solve", rows="tracking", frames=50, dets=400, cand=4,
             iters=100, per_slot=True),
        # the largest solve: the benchmark's tracking instance, 6 million variables, 18 million (row, variable) pairs
        dict(name="tracking_500x2000_solve", do="solve", rows="tracking", frames=500, dets=2000, cand=4, iters=50),
        # a training step on a large tracking instance, the records of all its sweeps kept
        dict(name="tracking_200x2000_train", do="train", rows="tracking", frames=200, dets=2000, cand=4, iters=10,
             every=10),
        # assignment with rows of about 300 variables: the long subproblems
        dict(name="assignment_2000x300_solve", do="solve", rows="assignment", L=2000, cand=300, iters=50),
        # a training step on long rows
        dict(name="assignment_400x300_train", do="train", rows="assignment", L=400, cand=300, iters=10, every=10),
        # the feature pass of the parameter predictor: min-marginals, energies, smoothed dual for three factors
        dict(name="tracking_200x2000_features", do="features", rows="tracking", frames=200, dets=2000, cand=4),
        # long cardinality rows, a wide knapsack row and short rows of general integer coefficients
        dict(name="general_rows_solve", do="solve", rows="general", short=40, iters=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["solve", "solve", "train", "features"])
    rows = rng.choice(["set_cover", "independent_set", "matching", "batch", "tracking", "tracking", "assignment",
                       "general"])
    c = dict(do=do, rows=rows, structure=rng.randint(1, 1 << 20))
    if rows == "set_cover":
        n = _log(rng, 17, 20_000)
        kmin = rng.randint(2, 3)
        c.update(n=n, m=max(2, int(n * rng.uniform(0.4, 0.8))), kmin=kmin, kmax=rng.randint(kmin + 3, 12))
    elif rows == "independent_set":
        c.update(n=_log(rng, 300, 50_000))
    elif rows == "matching":
        L = _log(rng, 50, 300)
        c.update(L=L, pairs=int(L * rng.uniform(50, 110)))
    elif rows == "batch":
        c.update(num=_log(rng, 4, 24))
    elif rows == "tracking":
        c.update(frames=_log(rng, 4, 150), dets=_log(rng, 50, 2000), cand=rng.randint(2, 5))
    elif rows == "assignment":
        L = _log(rng, 100, 1500)
        c.update(L=L, cand=_log(rng, 10, min(300, L - 1)))
    else:
        c.update(short=_log(rng, 20, 400))
    long_rows = rows in ("assignment", "general")
    if do == "solve":
        c.update(iters=_log(rng, 10, 40 if long_rows else 100))
        if rng.random() < 0.4:
            c.update(per_slot=True)
        if rng.random() < 0.3:
            c.update(graph=True)
    elif do == "train":
        c.update(iters=rng.randint(3, 8 if long_rows else 20))
        c.update(every=rng.choice([c["iters"], max(1, c["iters"] // 2), 5]))
    return c


# -- the instances -------------------------------------------------------------

def _rows(c, seed):
    s, k = workloads.BASE_SEED + c.get("structure", 0), c["rows"]
    if k == "set_cover":
        p = workloads.set_cover(n=c["n"], m=c["m"], kmin=c["kmin"], kmax=c["kmax"], seed=s)
    elif k == "independent_set":
        p = workloads.independent_set(n=c["n"], seed=s)
    elif k == "matching":
        p = workloads.matching_quadratic(L=c["L"], R=c["L"], pairs=c["pairs"], seed=s)
    elif k == "batch":
        p = workloads.batched_mix(num=c["num"], seed=s)[0]
    elif k == "tracking":
        p = workloads.tracking(frames=c["frames"], dets=c["dets"], cand=c["cand"], seed=s)
    elif k == "assignment":
        p = workloads.assignment(L=c["L"], R=c["L"], cand=c["cand"], seed=s)
    else:
        p = workloads.long_rows_mix(seed=s, n_short=c["short"])
    # each cost keeps its sign and its kind's scale
    p["c"] = p["c"] * np.random.default_rng(int(seed)).uniform(0.5, 1.5, size=p["n"])
    return p


def _vectors(c, seed, nnz, device="cuda"):
    """The per-(row, variable) inputs a program holds, in CSR order: the parameter predictor's outputs for a training
    step or a per-slot solve, a perturbation of the initial state for the features."""
    g = torch.Generator("cpu").manual_seed(int(seed) * 3 + 1) if nnz < 1 << 16 else \
        torch.Generator(device).manual_seed(int(seed) * 3 + 1)
    z = [torch.randn(nnz, generator=g, device=g.device).to(device) for _ in range(3)]
    return dict(a=z[0], w=z[1], t=0.1 * z[2])


def prepare(case, seed):
    p = _rows(case, seed)
    A = solver.plan(p).bind()
    nnz = int(p["row_ptr"][-1])
    lam, M = A.init_lambda()
    s = dict(case=case, A=A, lam=lam, M=M)
    if case["do"] == "solve":
        if case.get("per_slot"):
            v = _vectors(case, seed, nnz)
            alpha, omega, _ = A.param_transform(A.from_csr(v["a"]), A.from_csr(v["w"]), A.zeros())
            s.update(alpha=alpha, omega=omega)
        if case.get("graph"):
            s["lb"] = torch.zeros(A.num_inst, dtype=torch.float64, device=A.device)
            s["graph"] = A.graph(lam, M, s.get("omega"), s.get("alpha"), iters=case["iters"], lb_out=s["lb"])
    else:
        v = _vectors(case, seed, nnz)
        if case["do"] == "train":
            s["hat"] = [A.from_csr(v[k]).requires_grad_() for k in ("a", "w", "t")]
        else:
            s["lam"] = lam + A.from_csr(v["t"])
            s["M"] = A.from_csr(0.1 * v["w"])
    return s


def run(state):
    case, A = state["case"], state["A"]
    if case["do"] == "solve":
        lam, M = state["lam"], state["M"]
        if case.get("graph"):
            state["graph"].replay()
            lb = state["lb"]
        else:
            lb = A.iterate(lam, M, state.get("omega"), state.get("alpha"), iters=case["iters"], lb=True)
        return dict(lam=A.to_csr(lam), M=A.to_csr(M), lb=lb)
    if case["do"] == "train":
        hat = state["hat"]
        alpha, omega, theta = ParamTransform.apply(*hat, A)
        lam = NonParamUpdate.apply(state["lam"], theta, A)
        lam, M = DualIterate.apply(lam, state["M"], omega, alpha, A, case["iters"], case["every"])
        lb = LowerBound.apply(lam, M, A)
        grads = torch.autograd.grad(-lb.sum(), hat)
        return dict(lam=A.to_csr(lam.detach()), M=A.to_csr(M.detach()), lb=lb.detach(),
                    **{"grad_" + k: A.to_csr(g) for k, g in zip(("alpha", "omega", "theta"), grads)})
    lam, M = state["lam"], state["M"]
    m0, m1 = A.min_marginals(lam)
    lb, energy = A.lower_bound(lam, M, energies=True)
    out = dict(m0=A.to_csr(m0), m1=A.to_csr(m1), lb=lb, energy=energy)
    for a in SMOOTHING:
        e, marginals = A.smoothed_dual(lam, a)
        out["smooth_%g" % a] = (e, A.to_csr(marginals))
    return out


# -- what a pass cannot do without ---------------------------------------------

def _counts(c):
    """Expected (variables, rows, (row, variable) pairs, BDD nodes) of a case's instance."""
    def amo(rows, k):  # rows of k variables whose BDD has two nodes a level after the root
        return np.array([0, rows, rows * k, rows * (2 * k - 1)], float)

    def is_(n):
        return amo(4 * n, 2) + [n, 0, 0, 0]

    def cover(n, m, k):
        return amo(m, k) + [n, 0, 0, 0]

    def match(L, pairs):
        return amo(2 * L, 10) + 2 * amo(pairs, 2) + amo(pairs, 3) + [10 * L + pairs, 0, 0, 0]
    k = c["rows"]
    if k == "independent_set":
        t = is_(c["n"])
    elif k == "set_cover":
        t = cover(c["n"], c["m"], (c["kmin"] + c["kmax"]) / 2)
    elif k == "matching":
        t = match(c["L"], c["pairs"])
    elif k == "batch":
        t = c["num"] / 3 * (is_(25_500) + cover(10_250, 5_125, 7.5) + match(175, 17_500))
    elif k == "tracking":
        d, q = c["frames"] * c["dets"], c["cand"]
        width = sum(min(h + 1, q + 2, 2 * q + 2 - h) for h in range(2 * q + 2))
        t = amo(2 * d, q) + [d * (2 + q), d, d * (2 * q + 2), d * width]
    elif k == "assignment":
        t = amo(2 * c["L"], c["cand"]) + [c["L"] * c["cand"], 0, 0, 0]
    else:
        t = np.array([700, 5 + c["short"], 1830 + 3.5 * c["short"], 21_000 + 12 * c["short"]], float)
    return [float(x) for x in t]


def work(case):
    n, m, nnz, nodes = _counts(case)
    rows_in = 8 * nnz + 8 * m + 8 * n          # the rows (variable, coefficient), their bounds, the costs
    sweep = 2 * nodes * 6                      # per arc: a path cost each way and the min-marginal, an add and a min each
    if case["do"] == "solve":
        per_slot = 8 * nnz if case.get("per_slot") else 0
        return dict(bytes=rows_in + per_slot + 16 * nnz, flops=2 * sweep * case["iters"])
    if case["do"] == "train":
        # in: lambda, M and the three predicted vectors; out: lambda, M and their gradients
        return dict(bytes=rows_in + 20 * nnz + 20 * nnz, flops=4 * sweep * case["iters"])
    k = len(SMOOTHING)
    return dict(bytes=rows_in + 8 * nnz + 8 * nnz + 4 * m + k * (4 * nnz + 4 * m), flops=(2 + 3 * k) * sweep)


# -- the same in 64 bits ---------------------------------------------------------
# Dense dynamic programs over partial sums (no BDDs): rows of similar length together, one tensor (rows, sums) per
# level.  A sum from which every completion is feasible (or none is) stays so, so sums are clamped to that window.

class _Bucket:
    def __init__(self, rows, rp, coef, sense, rhs, dev):
        order = np.argsort(-(rp[rows + 1] - rp[rows]), kind="stable")
        rows = rows[order]
        ln = rp[rows + 1] - rp[rows]
        self.rows = torch.as_tensor(rows, device=dev)
        kmax = int(ln.max())
        self.cnt = [int(np.searchsorted(-ln, -h, side="left")) for h in range(kmax + 1)]  # rows longer than h
        pos = rp[rows][:, None] + np.arange(kmax)
        inside = np.arange(kmax) < ln[:, None]
        a = np.where(inside, coef[np.minimum(pos, len(coef) - 1)], 0).astype(np.int64)
        P, N = np.maximum(a, 0).sum(1), np.minimum(a, 0).sum(1)
        s, b = sense[rows], rhs[rows].astype(np.int64)
        lo = np.maximum(N, np.where(s == 0, b - P, b - P - 1))
        hi = np.minimum(P, np.where(s == 1, b - N, b - N + 1))
        lo, hi = np.minimum(lo, 0), np.maximum(hi, 0)
        self.W = int((hi - lo).max()) + 1
        at = lo[:, None] + np.arange(self.W)
        ok = np.where(s[:, None] == 0, at <= b[:, None], np.where(s[:, None] == 1, at >= b[:, None], at == b[:, None]))
        ok &= at <= hi[:, None]
        self.term = torch.as_tensor(np.where(ok, 0.0, np.inf), device=dev)
        self.start = torch.as_tensor(-lo, device=dev)
        self.top = torch.as_tensor(hi - lo, device=dev)
        self.a = torch.as_tensor(a, device=dev)
        self.q = torch.as_tensor(rp[rows], device=dev)
        self.k = kmax
        self.ar = torch.arange(self.W, device=dev)

    def slots(self, h):
        return self.q[: self.cnt[h]] + h

    def to(self, h):
        c = self.cnt[h]
        return torch.minimum((self.ar + self.a[:c, h, None]).clamp(min=0), self.top[:c, None])

    def below(self, T, h):
        """The costs of level h + 1 for the rows that have a level h."""
        if h + 1 == self.k:
            return self.term[: self.cnt[h]]
        d = self.cnt[h + 1]
        return T[h + 1] if d == self.cnt[h] else torch.cat([T[h + 1], self.term[d: self.cnt[h]]])

    def costs(self, lam, join):
        """join(0-arc, 1-arc) costs of every level to the end of the row."""
        T = [None] * self.k
        for h in range(self.k - 1, -1, -1):
            B = self.below(T, h)
            T[h] = join(B, lam[self.slots(h)][:, None] + B.gather(1, self.to(h)))
        return T

    def root(self, T):
        c = self.cnt[0]
        return T[0].gather(1, self.start[:c, None])[:, 0]

    def first(self):
        R = torch.full((self.cnt[0], self.W), math.inf, dtype=torch.float64, device=self.term.device)
        return R.scatter(1, self.start[: self.cnt[0], None], 0.0)


class _Exact:
    def __init__(self, p, dev):
        rp, coef = np.asarray(p["row_ptr"]), np.asarray(p["coef"])
        ln = np.diff(rp)
        sense, rhs = np.asarray(p["sense"]), np.asarray(p["rhs"])
        # rows together by length, and apart those whose window of sums is much wider
        span = np.add.reduceat(np.abs(coef), rp[:-1]) + 1
        wide = np.minimum(span, np.where(sense == 2, span, np.minimum(np.abs(rhs) + 2, span)))
        key = np.ceil(np.log2(np.maximum(ln, 2))).astype(int) * 64 + np.ceil(np.log2(np.maximum(wide, 2))).astype(int)
        self.dev = dev
        self.buckets = [_Bucket(np.nonzero(key == k)[0], rp, coef, sense, rhs, dev) for k in np.unique(key)]
        self.col = torch.as_tensor(p["col"], dtype=torch.int64, device=dev)
        self.c = torch.as_tensor(p["c"], dtype=torch.float64, device=dev)
        self.n, self.m, self.nnz = int(p["n"]), len(ln), int(rp[-1])
        self.deg = torch.bincount(self.col, minlength=self.n).double()
        irp, ivp = p.get("inst_row_ptr"), p.get("inst_var_ptr")
        self.num = 1 if irp is None else len(irp) - 1
        irp, ivp = (np.array([0, self.m]), np.array([0, self.n])) if irp is None else (irp, ivp)
        inst = [np.repeat(np.arange(self.num), np.diff(x)) for x in (irp, ivp)]
        self.row_inst, self.var_inst = [torch.as_tensor(x, device=dev) for x in inst]
        q = torch.cat([b.slots(h) for b in self.buckets for h in range(b.k)])
        self.back = torch.empty_like(q)
        self.back[q] = torch.arange(len(q), device=dev)
        r = torch.cat([b.rows[: b.cnt[0]] for b in self.buckets])
        self.row_back = torch.empty_like(r)
        self.row_back[r] = torch.arange(len(r), device=dev)

    def init(self):
        lam = (self.c / self.deg.clamp(min=1))[self.col]
        return lam, torch.zeros_like(lam)

    def per_var(self, x):
        return torch.zeros(self.n, dtype=torch.float64, device=self.dev).index_add(0, self.col, x)

    def sweep(self, lam, M, omega, alpha, forward):
        add = alpha * self.per_var(M)[self.col]
        low = torch.minimum
        new = {}
        for b in self.buckets:
            if forward:
                T, R = b.costs(lam, low), b.first()
                for h in range(b.k):
                    c, q, to, B = b.cnt[h], b.slots(h), b.to(h), b.below(T, h)
                    R = R[:c]
                    d = lam[q] + (R + B.gather(1, to)).amin(1) - (R + B).amin(1)
                    m = omega[q] * d
                    ln = lam[q] - m + add[q]
                    new[id(b), h] = (ln, m)
                    far = torch.full_like(R, math.inf).scatter_reduce(1, to, R + ln[:, None], "amin")
                    R = low(R, far)
            else:
                R, Rs = b.first(), []
                for h in range(b.k):
                    R = R[: b.cnt[h]]
                    Rs.append(R)
                    far = torch.full_like(R, math.inf).scatter_reduce(1, b.to(h), R + lam[b.slots(h)][:, None], "amin")
                    R = low(R, far)
                T = [None] * b.k
                for h in range(b.k - 1, -1, -1):
                    q, B = b.slots(h), b.below(T, h)
                    H = B.gather(1, b.to(h))
                    m = omega[q] * (lam[q] + (Rs[h] + H).amin(1) - (Rs[h] + B).amin(1))
                    ln = lam[q] - m + add[q]
                    new[id(b), h] = (ln, m)
                    T[h] = low(B, ln[:, None] + H)
        order = [new[id(b), h] for b in self.buckets for h in range(b.k)]
        return tuple(torch.cat([x[i] for x in order])[self.back] for i in (0, 1))

    def iterate(self, lam, M, omega, alpha, iters):
        for _ in range(iters):
            lam, M = self.sweep(lam, M, omega, alpha, True)
            lam, M = self.sweep(lam, M, omega, alpha, False)
        return lam, M

    def energies(self, lam):
        return torch.cat([b.root(b.costs(lam, torch.minimum)) for b in self.buckets])[self.row_back]

    def bound(self, lam, M):
        E, S = self.energies(lam), self.per_var(M)
        v = torch.where(self.deg > 0, S.clamp(max=0), self.c.clamp(max=0))
        lb = torch.zeros(self.num, dtype=torch.float64, device=self.dev)
        return lb.index_add(0, self.row_inst, E).index_add(0, self.var_inst, v), E

    def min_marginals(self, lam):
        out = []
        for b in self.buckets:
            T, R = b.costs(lam, torch.minimum), b.first()
            for h in range(b.k):
                R, to, B = R[: b.cnt[h]], b.to(h), b.below(T, h)
                l = lam[b.slots(h)]
                out.append(((R + B).amin(1), l + (R + B.gather(1, to)).amin(1)))
                far = torch.full_like(R, math.inf).scatter_reduce(1, to, R + l[:, None], "amin")
                R = torch.minimum(R, far)
        return tuple(torch.cat([x[i] for x in out])[self.back] for i in (0, 1))

    def smoothed(self, lam, a):
        """(-a log sum over feasible x of exp(-<lam, x>/a) per row, P(x_i = 1) per slot)."""
        E, out = [], []
        w = lam / a
        for b in self.buckets:
            T = b.costs(w, lambda x, y: -torch.logaddexp(-x, -y))
            logz = -b.root(T)
            E.append(-a * logz)
            F = -b.first()  # log weights of the prefixes
            for h in range(b.k):
                c, to, B = b.cnt[h], b.to(h), b.below(T, h)
                F = F[:c]
                up = F - w[b.slots(h)][:, None]
                out.append(torch.exp(torch.logsumexp(up - B.gather(1, to), 1) - logz[:c]))
                far = torch.zeros_like(F).scatter_add(1, to, torch.exp(up))
                F = torch.logaddexp(F, torch.log(far))
        return torch.cat(E)[self.row_back], torch.cat(out)[self.back]


def exact(case, seed):
    dev = "cuda"
    n, m, nnz, nodes = _counts(case)
    if case["do"] == "train" and 2 * nodes * 2 * 8 * 24 * case["iters"] > 5e10:
        return None  # autograd through every sweep would not fit in time
    p = _rows(case, seed)
    X = _Exact(p, dev)
    v = _vectors(case, seed, X.nnz) if case["do"] != "solve" or case.get("per_slot") else None
    share = (1.0 / X.deg.clamp(min=1))[X.col]

    def transforms(a, w, t):
        top = torch.full((X.n,), -math.inf, dtype=torch.float64, device=dev).scatter_reduce(0, X.col, a.detach(), "amax")
        e = torch.exp(a - top[X.col])
        return e / X.per_var(e)[X.col], torch.sigmoid(w), t - X.per_var(t)[X.col] * share

    lam, M = X.init()
    if case["do"] == "solve":
        alpha, omega = share, torch.full_like(lam, 0.5)
        if v:
            alpha, omega, _ = transforms(*(v[k].double() for k in ("a", "w", "t")))
        with torch.no_grad():
            lam, M = X.iterate(lam, M, omega, alpha, case["iters"])
            return dict(lam=lam, M=M, lb=X.bound(lam, M)[0])
    if case["do"] == "train":
        hat = [v[k].double().requires_grad_() for k in ("a", "w", "t")]
        alpha, omega, theta = transforms(*hat)
        # the centred theta moves lambda as it is: its mean over a variable's rows is zero already
        lam, M = X.iterate(lam + theta - X.per_var(theta)[X.col] * share, M, omega, alpha, case["iters"])
        lb, _ = X.bound(lam, M)
        g = torch.autograd.grad(-lb.sum(), hat)
        return dict(lam=lam.detach(), M=M.detach(), lb=lb.detach(),
                    **{"grad_" + k: x for k, x in zip(("alpha", "omega", "theta"), g)})
    with torch.no_grad():
        lam = lam + v["t"].double()
        m0, m1 = X.min_marginals(lam)
        lb, E = X.bound(lam, 0.1 * v["w"].double())
        out = dict(m0=m0, m1=m1, lb=lb, energy=E)
        for a in SMOOTHING:
            out["smooth_%g" % a] = X.smoothed(lam, a)
        return out

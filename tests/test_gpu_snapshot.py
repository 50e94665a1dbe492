"""The averaging snapshot of dg_sweep: the one of the last dg_sum_M, or of the
last S reduction before a sweep inside another call, on every kind of row alike.
Calls that only evaluate (bound, seed, marginals) leave it alone.  All
comparisons are exact: the same kernels on the same inputs, or (doubled problem)
the general kernels on the same BDDs, which make the same additions."""
import numpy as np
import pytest
import torch

import workloads
from paper_2205_11638_gb300 import build, solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _all_kinds():
    """Short rows with and without coefficients beyond +-1, long rows of both
    kinds and a wide one, over common variables."""
    rng = np.random.default_rng(3)
    n = 300
    rows = [r for amax in (1, 3) for r in workloads.random_rows(400, kmax=6, n=n, amax=amax, seed=amax)
            if workloads._free_row(r)]
    for a, b in ((np.ones(260), 1), (np.ones(200), 9), (np.ones(180), 40), (2 * np.ones(260), 3)):
        rows.append((np.sort(rng.choice(n, size=len(a), replace=False)), a.astype(np.int64), workloads.LE, b))
    rows.append((np.arange(100, 130), np.arange(1, 31), workloads.LE, 200))
    return workloads.single_rows_problem(rows, n, rng.normal(size=n))


CASES = {
    "all_kinds": _all_kinds,
    "one_tile": lambda: workloads.single_rows_problem(
        [(np.array([0, 1, 2]), np.ones(3, np.int64), workloads.LE, 1),
         (np.array([1, 2, 3]), np.ones(3, np.int64), workloads.LE, 1)], 4, np.array([-1.0, 0.5, -2.0, 0.3])),
}


def _doubled(p):
    return dict(p, coef=(2 * p["coef"]).astype(np.int32), rhs=(2 * p["rhs"]).astype(np.int32))


def _state(X, p, mode):
    rng = np.random.default_rng(9)
    nnz = len(p["col"])
    e = np.exp(rng.normal(size=nnz))
    s = np.zeros(p["n"])
    np.add.at(s, p["col"], e)
    lam, M, other, om, al = [X.from_csr(x) for x in (rng.normal(size=nnz), rng.normal(size=nnz), rng.normal(size=nnz),
                                                     rng.uniform(0.1, 0.9, size=nnz), e / s[p["col"]])]
    return lam, M, other, (om if mode else None), (al if mode else None)


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("mode", [0, 1])
def test_evaluations_leave_the_snapshot(name, mode):
    p = CASES[name]()
    out = []
    for evaluate in (False, True):
        X = solver.plan(p).bind()
        lam, M, other, om, al = _state(X, p, mode)

        def between():
            if evaluate:
                X.lower_bound(lam, other)
                X.lb_seed(lam, other)
                X.min_marginals(lam)
                X.lower_bound_noalloc(lam, other)
        between()
        X.sweep(lam, M, forward=True, omega=om, alpha=al)  # no snapshot taken yet: zeros
        X.sum_M(M, alpha=al)
        between()
        X.sweep(lam, M, forward=True, omega=om, alpha=al)
        between()
        X.sweep(lam, M, forward=False, omega=om, alpha=al)
        X.iterate(lam, M, om, al, iters=2)
        between()
        X.sweep(lam, M, forward=True, omega=om, alpha=al)
        out.append((X.to_csr(lam), X.to_csr(M)))
    for a, b in zip(*out):
        assert torch.equal(a, b) and torch.isfinite(a).all()


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("mode", [0, 1])
def test_the_snapshot_a_call_leaves_is_the_same_on_every_kind_of_row(name, mode):
    p = CASES[name]()
    out = []
    for q in (p, _doubled(p)):
        X = solver.plan(q).bind()
        lam, M, other, om, al = _state(X, p, mode)
        zero = X.zeros()
        for call in (lambda: X.iterate(lam, M, om, al, iters=2, lb=True),
                     lambda: X.iterate(lam, M, om, al, iters=0, lb=True),
                     lambda: X.iterate(lam, M, om, al, iters=2, renorm_every=1),
                     lambda: X.iterate_checkpointed(lam, M, om, al, iters=3, ckpt_every=2),
                     lambda: X.backward(lam, M, om, al, 3, 2, zero, zero),
                     lambda: X.lower_bound(lam, other)):
            call()
            X.sweep(lam, M, forward=True, omega=om, alpha=al)
            X.sweep(lam, M, forward=False, omega=om, alpha=al, energy=True)
            lb = torch.zeros(X.num_inst, dtype=torch.float64, device=X.device)
            X.bound_from_energies(lb)
            out.append((X.to_csr(lam), X.to_csr(M), lb))
    half = len(out) // 2
    for x, y in zip(out[:half], out[half:]):
        for a, b in zip(x, y):
            assert torch.equal(a, b) and torch.isfinite(a).all()

"""Unit rows (coefficients +1 and -1), in tiles of one shape and, beyond a tile
lane, as long unit rows, against the kernels of the mixed tiles and of the
other long BDDs.  Doubling a row's coefficients and
right-hand side leaves its canonical BDD unchanged but makes it no unit row,
so the doubled problem runs the general kernels on the same BDDs.  Both do
the same FP32 additions along the same arcs and take exact minima, hence the
results have to be equal bit for bit (no tolerance)."""
import numpy as np
import pytest
import torch

import workloads
from paper_2205_11638_gb300 import build, solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _doubled(p):
    return dict(p, coef=(2 * p["coef"]).astype(np.int32), rhs=(2 * p["rhs"]).astype(np.int32))


def _random_unit_rows(seed, n=300, patterns=60):
    """Random sign patterns of 1..14 terms, every sense and right-hand side,
    each as 1, 31, 32, 33 or 70 rows over random variables."""
    rng = np.random.default_rng(seed)
    rows = []
    while len(rows) < patterns * 60:
        k = int(rng.integers(1, 15))
        a = rng.choice([-1, 1], size=k) if rng.random() < 0.6 else np.full(k, rng.choice([-1, 1]))
        sense = int(rng.integers(0, 3))
        b = int(rng.integers(np.minimum(a, 0).sum(), np.maximum(a, 0).sum() + 1))
        if not workloads._free_row((None, a, sense, b)):
            continue
        for _ in range(int(rng.choice([1, 31, 32, 33, 70]))):
            rows.append((np.sort(rng.choice(n, size=k, replace=False)), a, sense, b))
    rng.shuffle(rows)
    return workloads.single_rows_problem(rows, n, rng.normal(size=n))


def _long_unit_rows(seed, n=700):
    """Long rows of both layouts' limits: cardinality rows of several lengths,
    senses and widths (up to 32 states a level; one of 33, which stays with
    the general loops), clauses of random signs (two to four states, level
    types alternating), and short rows next to them."""
    rng = np.random.default_rng(seed)
    rows = []

    def add(a, sense, b, copies):
        for _ in range(copies):
            rows.append((np.sort(rng.choice(n, size=len(a), replace=False)), np.asarray(a, np.int64), sense, b))
    for k in (128, 130, 257, 300, 511):
        add(np.ones(k), workloads.LE, 1, 3)
        add(np.ones(k), workloads.GE, 1, 2)
        add(np.ones(k), workloads.EQ, 1, 2)
    for b in (2, 5, 12, 31, 32):
        add(np.ones(150 + b), workloads.LE, b, 2)
        add(np.ones(150 + b), workloads.EQ, b, 1)
        add(np.ones(140), workloads.GE, b, 1)
    for b in (1, 3):
        for copies in (1, 4):
            a = rng.choice([-1, 1], size=260)
            add(a, workloads.GE, b - int((a < 0).sum()), copies)
    for r in workloads.random_rows(200, kmax=6, n=n, amax=1, seed=seed + 1):
        if workloads._free_row(r):
            rows.append(r)
    return workloads.single_rows_problem(rows, n, rng.normal(size=n))


def _short_rows(seed, copies, more=(), n=400):
    """Every unit row of up to three variables that leaves some choice, `copies`
    rows each, and `more` rows of six."""
    rng = np.random.default_rng(seed)
    kinds = [(np.array(a), sense, b) for k in (1, 2, 3) for a in np.ndindex(*(2,) * k) for sense in range(3)
             for b in range(-k, k + 1) if workloads._free_row((None, 2 * np.array(a) - 1, sense, b))]
    rows = []
    for a, sense, b in kinds:
        var = rng.integers(0, n - len(a), size=copies)
        rows += [(v + np.arange(len(a)), 2 * a - 1, sense, b) for v in var]
    rows += [(np.sort(rng.choice(n, size=6, replace=False)), np.ones(6, np.int64), 0, b) for b in more]
    return workloads.single_rows_problem(rows, n, rng.normal(size=n))


CASES = {
    "independent_set": lambda: workloads.independent_set(n=500, seed=45),  # short tiles only
    "long_rows": lambda: _long_unit_rows(6),
    "assignment": lambda: workloads.assignment(L=50, R=300, cand=260, seed=44),
    "random_signs": lambda: _random_unit_rows(5),
    "tracking": lambda: workloads.tracking(frames=8, dets=150, seed=41),
    "matching": lambda: workloads.matching_quadratic(L=40, R=40, pairs=1500, seed=42),
    "set_cover": lambda: workloads.set_cover(n=400, m=300, kmin=2, kmax=12, seed=43),
    "one_row": lambda: workloads.single_rows_problem([(np.arange(3), np.ones(3, np.int64), 0, 1)], 3,
                                                     np.array([-1.0, 0.5, -2.0])),
}


def _pair(name):
    p = CASES[name]()
    return p, solver.plan(p).bind(), solver.plan(_doubled(p)).bind()


def _vectors(p, seed):
    rng = np.random.default_rng(seed)
    nnz = len(p["col"])
    e = np.exp(rng.normal(size=nnz))
    s = np.zeros(p["n"])
    np.add.at(s, p["col"], e)
    return [torch.as_tensor(x, dtype=torch.float32) for x in
            (rng.normal(size=nnz), 0.1 * rng.normal(size=nnz), rng.uniform(0.1, 0.9, size=nnz), e / s[p["col"]])]


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("mode", [0, 1])
def test_sweeps_equal_the_mixed_tiles(name, mode):
    p, A, B = _pair(name)
    v = _vectors(p, 7)
    out = []
    for X in (A, B):
        lam, M, om, al = [X.from_csr(x) for x in v]
        lb = X.iterate(lam, M, om if mode else None, al if mode else None, iters=5, lb=True)
        assert torch.equal(X.from_csr(X.to_csr(lam)), lam)  # padding stays 0
        out.append((X.to_csr(lam), X.to_csr(M), lb))
    for a, b in zip(*out):
        assert torch.equal(a, b) and torch.isfinite(a).all()


@pytest.mark.parametrize("name", sorted(CASES))
def test_scalar_damping_equals_the_mixed_tiles(name):
    p = CASES[name]()
    v = _vectors(p, 8)
    out = []
    for q in (p, _doubled(p)):
        X = solver.plan(q, omega=0.3).bind()
        lam, M = X.from_csr(v[0]), X.from_csr(v[1])
        X.iterate(lam, M, iters=3)
        out.append((X.to_csr(lam), X.to_csr(M)))
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("name", sorted(CASES))
def test_marginals_energies_and_minimisers_equal_the_mixed_tiles(name):
    p, A, B = _pair(name)
    v = _vectors(p, 9)
    # many equal costs: ties between paths follow the same rule
    tied = torch.round(v[0])
    for x in (v[0], tied):
        out = []
        for X in (A, B):
            lam, M = X.from_csr(x), X.from_csr(v[1])
            m0, m1 = X.min_marginals(lam)
            lb, E = X.lower_bound(lam, M, energies=True)
            gl, gM = X.lb_seed(lam, M)
            out.append([X.to_csr(m0), X.to_csr(m1), lb, E, X.to_csr(gl), X.to_csr(gM)])
        for a, b in zip(*out):
            assert torch.equal(a, b) and torch.isfinite(a).all()


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("tied", [False, True])
def test_gradients_equal_the_mixed_tiles(name, mode, tied):
    """Recording sweeps and adjoint: the same argmins (many equal path costs
    when tied), so the gradients differ by the rounding of sums alone: at most
    64 roundings per sweep on the way of a value, 6 sweeps, 2^-24 each, against
    the largest gradient."""
    p, A, B = _pair(name)
    v = _vectors(p, 10)
    lam0 = torch.round(v[0]) if tied else v[0]
    g = [torch.as_tensor(np.random.default_rng(s).normal(size=len(p["col"])), dtype=torch.float32) for s in (1, 2)]
    for iters, every in ((1, 1), (3, 2)):
        out = []
        for X in (A, B):
            lam, M, om, al = [X.from_csr(x) for x in (lam0, *v[1:])]
            gl, gM = [X.from_csr(x) for x in g]
            res = X.backward(lam, M, om if mode else None, al if mode else None, iters, every, gl, gM)
            w, _ = X.iterate_checkpointed(lam, M, om if mode else None, al if mode else None, iters, every)
            res2 = X.backward_checkpointed(om if mode else None, al if mode else None, iters, every, gl, gM, w)
            for a, b in zip(res, res2):
                assert torch.equal(X.to_csr(a), X.to_csr(b))
            out.append([X.to_csr(t) for t in (*res, lam, M)])
        for a, b in zip(out[0][:4], out[1][:4]):
            assert torch.isfinite(a).all()
            assert (a - b).abs().max() <= 64 * 6 * 2.0 ** -24 * b.abs().max().clamp(min=1e-30)
        for a, b in zip(out[0][4:], out[1][4:]):
            assert torch.equal(a, b)


@pytest.mark.parametrize("scale", [1.0, 30.0])
@pytest.mark.parametrize("name", sorted(CASES))
def test_smoothed_dual_against_float64(name, scale):
    """Energies and marginals of the smoothed subproblems on unit rows: the
    walk over sums of products (scale 1) and, with path costs beyond its range,
    the logarithmic one (scale 30), against the oracle.  Both make at most four
    roundings per level and state on a logarithm of size up to the row's costs:
    tolerance 4 levels 2^-24 relative to that size for E, absolute on the
    marginals (a logarithm's error is a factor's relative error)."""
    import oracle
    p = CASES[name]()
    O = oracle.Oracle(p)
    A = solver.plan(p).bind()
    lam = A.from_csr(scale * _vectors(p, 11)[0])
    lam_c = A.to_csr(lam).double().cpu().numpy()
    rp, absl = p["row_ptr"], np.abs(lam_c)
    for a in (1.0, 10.0):
        E, marg = A.smoothed_dual(lam, a)
        oE, om = O.smoothed(lam_c, a)
        size = np.add.reduceat(absl, rp[:-1]) / a + np.diff(rp)  # bound on the logarithms in a row
        tol = 4 * np.diff(rp) * 2.0 ** -24 * size + 1e-6
        assert torch.isfinite(E).all() and torch.isfinite(marg).all()
        assert (np.abs(E.double().cpu().numpy() - oE) <= a * tol).all()
        assert (np.abs(A.to_csr(marg).double().cpu().numpy() - om) <= np.repeat(tol, np.diff(rp))).all()


@pytest.mark.parametrize("mode", [0, 1])
def test_short_tiles_of_a_large_arena_equal_the_mixed_tiles(mode):
    """More than 8192 unit tiles, most of them short (one lane of the last of a
    shape): these are a launch of their own between the other unit tiles' and
    the mixed tiles'.  Plain sweeps, and recording ones through the gradients
    (tolerance as above: 64 roundings in each of 4 sweeps)."""
    p = _short_rows(4, 69 * 32 + 1, more=[1, 2, 3] * 50)
    out = []
    for q in (p, _doubled(p)):
        X = solver.plan(q).bind()
        lam, M, om, al = [X.from_csr(x) for x in _vectors(p, 12)]
        par = (om, al) if mode else (None, None)
        g = X.backward(lam, M, *par, 2, 1, *[X.from_csr(x) for x in _vectors(p, 13)[:2]])
        lb = X.iterate(lam, M, *par, iters=2, lb=True)
        out.append(([X.to_csr(lam), X.to_csr(M), lb], [X.to_csr(x) for x in g]))
    for a, b in zip(out[0][0], out[1][0]):
        assert torch.equal(a, b) and torch.isfinite(a).all()
    for a, b in zip(out[0][1], out[1][1]):
        assert (a - b).abs().max() <= 64 * 4 * 2.0 ** -24 * b.abs().max().clamp(min=1e-30)


def _packed_long_rows(num, seed, n=600):
    """Rows "sum of k = 12", k = 40 to 60: 13 states a level held by 16 lanes, one
    kind whatever the length, two BDDs to a warp from 1,216 of them on."""
    rng = np.random.default_rng(seed)
    rows = [(np.sort(rng.choice(n, size=int(k), replace=False)), np.ones(int(k), np.int64), workloads.EQ, 12)
            for k in rng.integers(40, 61, size=num)]
    return workloads.single_rows_problem(rows, n, rng.normal(size=n))


@pytest.mark.parametrize("mode", [0, 1])
def test_packed_segments_of_unequal_lengths(mode):
    """Two BDDs of different lengths to a warp, a segment of lanes each: sweeps
    bit for bit, gradients up to the rounding of sums (at most 64 roundings in
    each of 4 sweeps, as above)."""
    p = _packed_long_rows(1300, 14)
    v, g = _vectors(p, 15), _vectors(p, 16)[:2]
    out = []
    for q in (p, _doubled(p)):
        X = solver.plan(q).bind()
        assert X.plan.sizes.num_long_bdds == 1300
        lam, M, om, al = [X.from_csr(x) for x in v]
        par = (om, al) if mode else (None, None)
        res = X.backward(lam, M, *par, 2, 1, *[X.from_csr(x) for x in g])
        lb = X.iterate(lam, M, *par, iters=2, lb=True)
        out.append(([X.to_csr(x) for x in res], [X.to_csr(lam), X.to_csr(M), lb]))
    for a, b in zip(out[0][1], out[1][1]):
        assert torch.equal(a, b) and torch.isfinite(a).all()
    for a, b in zip(out[0][0], out[1][0]):
        assert torch.isfinite(a).all()
        assert (a - b).abs().max() <= 64 * 4 * 2.0 ** -24 * b.abs().max().clamp(min=1e-30)


def _two_footprints(seed, n=3000):
    """Unit rows alone in tiles of two footprints: 10,000 covering rows of 126
    variables, which fill the chip by themselves, and 2,000 of four."""
    rng = np.random.default_rng(seed)
    rows = [(rng.integers(0, n - 126) + np.arange(126), np.ones(126, np.int64), workloads.GE, 1) for _ in range(10000)]
    rows += [(rng.integers(0, n - 4) + np.arange(4), np.ones(4, np.int64), workloads.LE, 1) for _ in range(2000)]
    return workloads.single_rows_problem(rows, n, rng.normal(size=n))


def _mostly_short(seed, n=20000):
    """Unit rows alone, most of them of two and three variables: 8,320 tiles of
    these and 60 of six."""
    rng = np.random.default_rng(seed)
    rows = []
    for a, sense, b in (([1, 1], workloads.LE, 1), ([1, 1], workloads.GE, 1), ([1, 1, 1], workloads.LE, 1),
                        ([-1, -1, 1], workloads.LE, 0)):
        rows += [(v + np.arange(len(a)), np.array(a), sense, b) for v in rng.integers(0, n - 3, size=2080 * 32)]
    rows += [(v + np.arange(6), np.ones(6, np.int64), 0, 1) for v in rng.integers(0, n - 6, size=60 * 32)]
    return workloads.single_rows_problem(rows, n, rng.normal(size=n))


# instance, launch groups: one launch for tiles of many shapes, and where most
# are short; two on streams of their own
LAUNCHES = {
    "one": (lambda: workloads.tracking(frames=50, dets=400, seed=46), 1),
    "mostly_short": (lambda: _mostly_short(7), 1),
    "forked": (lambda: _two_footprints(8), 2),
}


@pytest.mark.parametrize("name", sorted(LAUNCHES))
@pytest.mark.parametrize("mode", [0, 1])
def test_launches_of_a_unit_arena(name, mode):
    """Every call's launches, chained or forked, against the doubled problem's:
    sweeps over many iterations, marginals, energies and minimisers bit for bit,
    gradients up to the rounding of sums (tolerance as above, 4 sweeps)."""
    make, groups = LAUNCHES[name]
    p = make()
    exact, grads = [], []
    for q in (p, _doubled(p)):
        X = solver.plan(q).bind()
        if q is p:
            assert X.plan.sizes.num_launch_groups == groups
            X.plan.validate()
        lam, M, om, al = [X.from_csr(x) for x in _vectors(p, 17)]
        par = (om, al) if mode else (None, None)
        grads.append([X.to_csr(x) for x in X.backward(lam, M, *par, 2, 2, *[X.from_csr(x) for x in _vectors(p, 18)[:2]])])
        l2, M2 = lam.clone(), M.clone()
        X.iterate_checkpointed(l2, M2, *par, iters=3, ckpt_every=3)
        m0, m1 = X.min_marginals(lam)
        lb0, E = X.lower_bound(lam, M, energies=True)
        gl, gM = X.lb_seed(lam, M)
        g = X.graph(lam, M, *par, iters=2)
        torch.cuda.synchronize()
        lb = X.iterate(lam, M, *par, iters=50, lb=True)
        g.replay()
        exact.append([X.to_csr(x) for x in (l2, M2, m0, m1, gl, gM, lam, M)] + [lb0, E, lb])
    for a, b in zip(*exact):
        assert torch.equal(a, b) and torch.isfinite(a).all()
    for a, b in zip(*grads):
        assert torch.isfinite(a).all()
        assert (a - b).abs().max() <= 64 * 4 * 2.0 ** -24 * b.abs().max().clamp(min=1e-30)


def _many_small_shapes(seed, n=60):
    """Clauses of every sign pattern of two to four variables and of eight of
    five, one to four rows each: a tile per pattern, 36 in all, more than a block
    has warps and few enough for the kernel that runs whole iterations of a small
    arena."""
    rng = np.random.default_rng(seed)
    signs = [2 * np.array(a) - 1 for k in (2, 3, 4) for a in np.ndindex(*(2,) * k)]
    signs += [2 * np.array(a) - 1 for a in list(np.ndindex(*(2,) * 5))[seed % 4::4]]
    rows = [(np.sort(rng.choice(n, size=len(a), replace=False)), a, workloads.GE, 1 - int((a < 0).sum()))
            for a in signs for _ in range(int(rng.integers(1, 5)))]
    return workloads.single_rows_problem(rows, n, rng.normal(size=n))


def _many_long_wide_rows(seed, num=1700, n=3000):
    """Rows "sum of k = 30", k = 990 to 1000: 31 states a level, so long and so
    many that their plain sweeps run in the general kernels (the other calls do
    not), and a few of another kind and short ones next to them."""
    rng = np.random.default_rng(seed)
    kinds = [(int(k), workloads.EQ, 30) for k in rng.integers(990, 1001, size=num)]
    kinds += [(300, workloads.LE, 1)] * 8 + [(3, workloads.GE, 1)] * 40
    rows = [(f + np.arange(k), np.ones(k, np.int64), s, b) for (k, s, b), f in
            zip(kinds, rng.integers(0, n - 1000, size=len(kinds)))]
    return workloads.single_rows_problem(rows, n, rng.normal(size=n))


@pytest.mark.parametrize("mode", [0, 1])
def test_long_unit_rows_swept_by_the_general_kernels(mode):
    """Plain sweeps against recording ones and against the doubled problem, bit
    for bit, with bounds and sweeps by hand in between."""
    p = _many_long_wide_rows(24)
    out = []
    for q in (p, _doubled(p)):
        X = solver.plan(q).bind()
        X.plan.validate()
        lam, M, om, al = [X.from_csr(x) for x in _vectors(p, 20)]
        par = (om, al) if mode else (None, None)
        l2, M2 = lam.clone(), M.clone()
        X.iterate_checkpointed(l2, M2, *par, iters=2, ckpt_every=1)
        lb = X.iterate(lam, M, *par, iters=2, lb=True)
        assert torch.equal(lam, l2) and torch.equal(M, M2)
        X.sum_M(M, alpha=par[1])
        X.sweep(lam, M, forward=True, omega=par[0], alpha=par[1], costs_out=True)
        X.sum_M(M, alpha=par[1])
        X.sweep(lam, M, forward=False, omega=par[0], alpha=par[1], costs_in=True, energy=True)
        lb2 = X.lower_bound(lam, M)
        out.append((X.to_csr(lam), X.to_csr(M), lb, lb2))
    for a, b in zip(*out):
        assert torch.equal(a, b) and torch.isfinite(a).all()


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("seed", [21, 22, 23])
def test_small_arena_of_many_shapes(seed, mode):
    p = _many_small_shapes(seed)
    out = []
    for q in (p, _doubled(p)):
        X = solver.plan(q).bind()
        lam, M, om, al = [X.from_csr(x) for x in _vectors(p, 19)]
        lb = X.iterate(lam, M, om if mode else None, al if mode else None, iters=100, lb=True)
        out.append((X.to_csr(lam), X.to_csr(M), lb))
        if q is p:
            assert X.plan.sizes.num_tiles > 32
    for a, b in zip(*out):
        assert torch.equal(a, b) and torch.isfinite(a).all()


def _lanes_rows(seed, n=400):
    """Long rows of several lengths of four kinds: two, six, 13 and 31 states."""
    rng = np.random.default_rng(seed)
    rows = []
    for b, lo, hi, num in ((1, 128, 170, 70), (5, 60, 80, 45), (12, 40, 60, 45), (30, 61, 75, 9)):
        rows += [(np.sort(rng.choice(n, size=int(k), replace=False)), np.ones(int(k), np.int64), workloads.EQ, b)
                 for k in rng.integers(lo, hi, size=num)]
    return workloads.single_rows_problem(rows, n, rng.normal(size=n))


@pytest.mark.parametrize("lanes", [1, 2, 8, 32])
@pytest.mark.parametrize("mode", [0, 1])
def test_long_unit_rows_at_any_packing(lanes, mode):
    """32 / lanes BDDs of unequal lengths to a warp (at most one per G lanes
    above eight states): all calls bit for bit, gradients up to the rounding of
    sums (tolerance as above, 4 sweeps)."""
    p = _lanes_rows(25)
    exact, grads = [], []
    for q in (p, _doubled(p)):
        X = solver.plan(q, long_lanes=lanes).bind()
        X.plan.validate()
        assert X.plan.sizes.num_tiles == 0
        lam, M, om, al = [X.from_csr(x) for x in _vectors(p, 26)]
        par = (om, al) if mode else (None, None)
        grads.append([X.to_csr(x) for x in X.backward(lam, M, *par, 2, 1, *[X.from_csr(x) for x in _vectors(p, 27)[:2]])])
        l2, M2 = lam.clone(), M.clone()
        X.iterate_checkpointed(l2, M2, *par, iters=3, ckpt_every=3)
        m0, m1 = X.min_marginals(lam)
        lb0, E = X.lower_bound(lam, M, energies=True)
        gl, gM = X.lb_seed(lam, M)
        lb = X.iterate(lam, M, *par, iters=3, lb=True)
        assert torch.equal(lam, l2) and torch.equal(M, M2)
        exact.append([X.to_csr(x) for x in (lam, M, m0, m1, gl, gM)] + [lb0, E, lb])
    for a, b in zip(*exact):
        assert torch.equal(a, b) and torch.isfinite(a).all()
    for a, b in zip(*grads):
        assert torch.isfinite(a).all()
        assert (a - b).abs().max() <= 64 * 4 * 2.0 ** -24 * b.abs().max().clamp(min=1e-30)


def test_workspace_of_long_unit_rows():
    """Their records (a word a level where a lane holds it) replace those of the
    general kernels (16 bytes for two states): no more memory for a training step
    than the doubled problem takes, and 5 % for partly filled tiles."""
    p = workloads.assignment(L=30, R=300, cand=260, seed=44)
    a, b = [solver.plan(q).bind().backward_workspace_bytes(10, 10) for q in (p, _doubled(p))]
    assert a <= 1.05 * b

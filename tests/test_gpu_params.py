"""GPU parity of the non-parametric update (eq. 2), the output transforms of
Alg. 3 and their adjoints against the FP64 oracle, and of one whole DOGE
round (transforms -> eq. 2 -> T iterations of Alg. 1 -> lower bound) end to
end through the autograd Functions.  Tolerances as for the solver: 1e-5
relative on values, 1e-4 absolute on O(1) gradients."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from paper_2205_11638_gb300 import build, solver
from paper_2205_11638_gb300.solver import DualIterate, LowerBound, NonParamUpdate, ParamTransform

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _np(t):
    return t.detach().double().cpu().numpy()


def _f32(x):
    return np.float32(x).astype(np.float64)


def test_nonparam_and_transforms_vs_oracle():
    prob = workloads.matching_quadratic(L=60, R=60, pairs=3000, seed=6)
    O = oracle.Oracle(prob)
    A = solver.plan(prob).bind()
    rng = np.random.default_rng(0)
    lam = _f32(rng.normal(size=O.num_slots))
    th, ah, wh = (_f32(rng.normal(size=O.num_slots) * 2) for _ in range(3))
    lam_g = A.from_csr(lam)
    A.nonparam_update(lam_g, A.from_csr(th))
    np.testing.assert_allclose(_np(A.to_csr(lam_g)), O.nonparam_update(lam, th), atol=1e-5)
    got = A.param_transform(A.from_csr(ah), A.from_csr(wh), A.from_csr(th))
    want = O.param_transform(ah, wh, th)
    for g, w in zip(got, want):
        np.testing.assert_allclose(_np(A.to_csr(g)), w, atol=1e-5, rtol=1e-5)
    ga, gw, gt = (_f32(rng.normal(size=O.num_slots)) for _ in range(3))
    gotb = A.param_transform_backward(got[0], got[1], A.from_csr(ga), A.from_csr(gw), A.from_csr(gt))
    wantb = O.param_transform_backward(want[0], want[1], ga, gw, gt)
    for g, w in zip(gotb, wantb):
        np.testing.assert_allclose(_np(A.to_csr(g)), w, atol=1e-5)
    g_th = A.nonparam_backward(A.from_csr(gt))
    np.testing.assert_allclose(_np(A.to_csr(g_th)), wantb[2], atol=1e-5)


def _tiny(seed, n=14, rows=12, kmax=6):
    good = []
    for r in workloads.random_rows(8 * rows, kmax=kmax, n=n, seed=seed):
        try:
            oracle.Oracle(workloads.single_rows_problem([r], n, np.zeros(n)))
            good.append(r)
        except oracle.OracleError:
            pass
        if len(good) == rows:
            break
    rng = np.random.default_rng(seed)
    return workloads.single_rows_problem(good, n, rng.normal(size=n))


@pytest.mark.parametrize("seed", [31, 32])
def test_doge_round_end_to_end_gradients(seed):
    """alpha-hat, omega-hat, theta-hat -> Alg. 3 transforms -> eq. 2 ->
    2 iterations of Alg. 1 -> lower bound; gradients of the bound with respect
    to the predictor outputs, GPU autograd chain vs the oracle's chain."""
    prob = _tiny(seed)
    O = oracle.Oracle(prob)
    A = solver.plan(prob).bind()
    rng = np.random.default_rng(seed)
    lam0, M0 = O.init_lambda()
    lam0 = _f32(lam0)
    ah, wh, th = (_f32(rng.normal(size=O.num_slots)) for _ in range(3))
    T = 2
    # oracle chain
    a, w, t = O.param_transform(ah, wh, th)
    lam1 = O.nonparam_update(lam0, t)
    lT, MT = O.iterate(lam1, M0, w, a, T)
    sl, sM = O.lb_seed(lT, MT)
    gl1, _, gw, ga = O.backward(lam1, M0, w, a, T, sl, sM)
    g_t = gl1 - (np.bincount(O.col, weights=gl1, minlength=O.n) / np.maximum(O.deg, 1))[O.col]
    want = O.param_transform_backward(a, w, ga, gw, g_t)
    # GPU chain through autograd
    leaves = [A.from_csr(x).requires_grad_(True) for x in (ah, wh, th)]
    a_g, w_g, t_g = ParamTransform.apply(*leaves, A)
    lam1_g = NonParamUpdate.apply(A.from_csr(lam0), t_g, A)
    lT_g, MT_g = DualIterate.apply(lam1_g, A.from_csr(M0), w_g, a_g, A, T, 1)
    lb = LowerBound.apply(lT_g, MT_g, A).sum()
    lb.backward()
    v = float(lb.detach())
    assert abs(v - O.lower_bound(lT, MT)) < 1e-4 * max(1.0, abs(v))
    for leaf, wv in zip(leaves, want):
        np.testing.assert_allclose(_np(A.to_csr(leaf.grad)), wv, atol=1e-4)


@pytest.mark.parametrize("a", [1.0, 10.0, 100.0])
def test_smoothed_dual_vs_oracle(a):
    """Smoothed-dual features for the three smoothing factors of the feature
    table, FP32 log-sum-exp on the GPU against the FP64 oracle."""
    prob = workloads.matching_quadratic(L=60, R=60, pairs=3000, seed=8)
    O = oracle.Oracle(prob)
    A = solver.plan(prob).bind()
    rng = np.random.default_rng(int(a))
    lam = _f32(rng.normal(size=O.num_slots) * 2)
    E, mg = A.smoothed_dual(A.from_csr(lam), a)
    oE, omg = O.smoothed(lam, a)
    np.testing.assert_allclose(_np(E), oE, rtol=1e-5, atol=1e-5 * a)
    np.testing.assert_allclose(_np(A.to_csr(mg)), omg, atol=1e-4)


@pytest.mark.parametrize("long_row", [0, 700])
def test_transforms_at_every_list_length(long_row):
    """Variables in 0, 1, 3, 4, 5, 31, 32, 33, 64 and 65 rows (the first four
    slots come from columns, more than 32 are a warp's), with and without a row
    of the long layout.  A softmax over d
    slots and a mean are d + 2 operations of O(1) values: below 70 * 2^-24 * 10
    = 4e-5 from FP64."""
    deg = [0, 1, 3, 4, 5, 31, 32, 33, 64, 65]
    n = len(deg) + 65 + long_row
    rows = [([i, len(deg) + j], [1, 1], 0, 1) for i, d in enumerate(deg) for j in range(d)]
    if long_row:
        rows.append((list(range(len(deg) + 65, n)), [1] * long_row, 0, 1))
    prob = dict(n=n, row_ptr=np.cumsum([0] + [len(r[0]) for r in rows]).astype(np.int64),
                col=np.concatenate([r[0] for r in rows]).astype(np.int32),
                coef=np.concatenate([r[1] for r in rows]).astype(np.int32),
                sense=np.array([r[2] for r in rows], np.int8), rhs=np.array([r[3] for r in rows], np.int64),
                c=np.zeros(n))
    O = oracle.Oracle(prob)
    A = solver.plan(prob).bind()
    rng = np.random.default_rng(5)
    lam, th, ah, wh, ga, gw, gt = (_f32(rng.normal(size=O.num_slots)) for _ in range(7))
    got = A.param_transform(A.from_csr(ah), A.from_csr(wh), A.from_csr(th))
    want = O.param_transform(ah, wh, th)
    back = A.param_transform_backward(got[0], got[1], A.from_csr(ga), A.from_csr(gw), A.from_csr(gt))
    want += O.param_transform_backward(want[0], want[1], ga, gw, gt)
    lam_g = A.from_csr(lam)
    A.nonparam_update(lam_g, A.from_csr(th))
    for g, w in zip((*got, *back, lam_g), (*want, O.nonparam_update(lam, th))):
        np.testing.assert_allclose(_np(A.to_csr(g)), w, atol=4e-5)


@pytest.mark.parametrize("shift", [0, 1, 2])
def test_transform_outputs_in_place_of_inputs(shift):
    """From C an output may take the place of an input: its own, or that of one
    transformed before it.  Compared with separate buffers, bit for bit."""
    from paper_2205_11638_gb300 import _lib
    prob = workloads.matching_quadratic(L=40, R=40, pairs=1500, seed=7)
    A = solver.plan(prob).bind()
    rng = np.random.default_rng(6)
    x = [A.from_csr(rng.normal(size=len(prob["col"]))) for _ in range(5)]
    want = A.param_transform(*x[:3])
    back = A.param_transform_backward(*x)
    st = torch.cuda.current_stream().cuda_stream
    t = [v.clone() for v in x[:3]]
    spare = [A.zeros() for _ in range(2)]
    # own input; omega over alpha-hat; theta over omega-hat as well
    out = [[t[0], t[1], t[2]], [spare[0], t[0], spare[1]], [spare[0], t[0], t[1]]][shift]
    rc = _lib.load().dg_param_transform(A._h, st, *[v.data_ptr() for v in (*t, *out)])
    assert rc == 0 and all(torch.equal(a, b) for a, b in zip(out, want))
    t = [v.clone() for v in x]
    out = [[t[2], t[3], t[4]], [spare[0], t[2], spare[1]], [spare[0], t[2], t[3]]][shift]
    rc = _lib.load().dg_param_transform_backward(A._h, st, *[v.data_ptr() for v in (*t, *out)])
    assert rc == 0 and all(torch.equal(a, b) for a, b in zip(out, back))

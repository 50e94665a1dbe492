"""dg_iterate_launches against the kernels a dg_iterate call really issues: the
kernel nodes of a graph captured from it."""
import ctypes

import numpy as np
import pytest
import torch

import workloads
from paper_2205_11638_gb300 import _lib, build, solver
from paper_2205_11638_gb300.solver import _ptr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _kernels(stream, call):
    """Kernel nodes of what `call` enqueues on the stream (captured, not run)."""
    cu = ctypes.CDLL("libcuda.so.1")
    st, graph, num = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert cu.cuStreamBeginCapture_v2(st, 1) == 0  # thread-local mode
    try:
        call()
    finally:
        assert cu.cuStreamEndCapture(st, ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(num)) == 0
    nodes = (ctypes.c_void_p * num.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(num)) == 0
    count, kind = 0, ctypes.c_int()
    for x in nodes:
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(x), ctypes.byref(kind)) == 0
        count += kind.value == 0  # CU_GRAPH_NODE_TYPE_KERNEL
    assert cu.cuGraphDestroy(graph) == 0
    return count


def _doubled(p):
    return dict(p, coef=(2 * p["coef"]).astype(np.int32), rhs=(2 * p["rhs"]).astype(np.int32))


CASES = {
    "small": lambda: workloads.set_cover(),
    "one_launch": lambda: workloads.tracking(frames=8, dets=150, seed=41),
    "mixed_tiles": lambda: _doubled(workloads.tracking(frames=8, dets=150, seed=41)),
    "batch": lambda: workloads.batched_mix(num=6, scale=0.1, seed=5)[0],
    "long_unit": lambda: workloads.assignment(L=20, R=300, cand=260, seed=44),
    "long_general": lambda: _doubled(workloads.assignment(L=20, R=300, cand=260, seed=44)),
    "every_kind": lambda: workloads.long_rows_mix(seed=3),
    "no_rows": lambda: workloads.single_rows_problem([], 7, np.arange(7.0) - 3),
}


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("name", sorted(CASES))
def test_launch_count(name, mode):
    p = CASES[name]()
    A = solver.plan(p).bind()
    lam, M = A.init_lambda()
    om, al = (torch.full_like(lam, 0.5), torch.full_like(lam, 0.1)) if mode and lam.numel() else (None, None)
    mode = 0 if om is None else 1
    lb = torch.zeros(A.num_inst, dtype=torch.float64, device=A.device)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    lib = _lib.load()
    for renorm in (0, 2):
        o = A._opts(renorm_every=renorm)
        for iters in (0, 1, 3):
            for want in (False, True):
                def call():
                    assert lib.dg_iterate(A._h, ctypes.c_void_p(stream.cuda_stream), _ptr(lam), _ptr(M), _ptr(om),
                                          _ptr(al), mode, iters, _ptr(lb) if want else None, ctypes.byref(o)) == 0
                told = lib.dg_iterate_launches(A._h, iters, int(want), ctypes.byref(o))
                assert told == _kernels(stream, call), (renorm, iters, want)


@pytest.mark.parametrize("n,launches", [(100, 1), (4000, 1), (8300, 9), (32000, 9)])
def test_one_launch_while_the_variables_are_few(n, launches):
    """A few rows over many variables: one block would spend its time summing
    over variables, so that from some 8,000 on the launches are separate."""
    rng = np.random.default_rng(n)
    rows = [(np.sort(rng.choice(n, size=3, replace=False)), np.ones(3, np.int64), workloads.GE, 1) for _ in range(20)]
    A = solver.plan(workloads.single_rows_problem(rows, n, rng.normal(size=n))).bind()
    assert A.iterate_launches(2) == launches


def test_bytes_of_an_iteration():
    """Rows of +1 and -1 move 20 bytes a pair and sweep and no node data, 4 bytes
    a pair and 20 a variable in a reduction (partly filled tiles add their ids
    and lambda, at most 8 bytes a slot); the doubled rows at least the child codes
    and path costs of their nodes on top."""
    p = workloads.tracking(frames=30, dets=400, seed=9)
    A, B = solver.plan(p).bind(), solver.plan(_doubled(p)).bind()
    pairs, n = len(p["col"]), p["n"]
    least = 2 * (20 * pairs + 4 * pairs + 20 * n)
    assert least <= A.stats.actual_bytes_per_iter <= least + 2 * 8 * (A.num_slots - pairs)
    assert B.stats.actual_bytes_per_iter >= 2 * (10 * int(B.plan.sizes.num_nodes) + 16 * pairs) + 2 * 8 * pairs
    L = solver.plan(workloads.assignment(L=20, R=300, cand=260, seed=44)).bind()
    assert L.stats.actual_bytes_per_iter < 2 * (28 * L.num_slots + 20 * L.n)

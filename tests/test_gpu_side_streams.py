"""A batch whose systems take several solver paths at once (Jacobi, the one-CTA and the cluster dense
reduction, band chases of three window classes) runs the paths side by side: each system's results
equal those of the system alone, for repeated runs and under graph replay."""

import numpy as np
import pytest

from paper_2005_03426_gb300 import mmf as M
from paper_2005_03426_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [(M.MMF_FP64, 1e-10), (M.MMF_MIXED, 1e-8)])
def test_mixed_batch_equals_each_alone(precision, tol):
    ctx = M.Context(0)
    ctx.set_option(M.MMF_OPT_BAND_MAX, 40)
    ctx.set_option(M.MMF_OPT_JACOBI_N_FP64 if precision == M.MMF_FP64 else M.MMF_OPT_JACOBI_N_MIXED, 30)
    rng = W.SplitMix64(11)
    # n = D prod (2 N + 1): 27 (Jacobi), 85 (one CTA: two modes, wide band), 315 (cluster), bands 5, 11, 31
    shapes = [(3, [4]), (5, [1, 8]), (7, [2, 4]), (3, [40]), (6, [20]), (16, [8]), (5, [1, 8]), (5, [6, 6])]
    ps = [W.random_multimode(rng, D, Ns) for D, Ns in shapes]
    nt = 6
    ts = np.stack([W.time_grid(p, nt) for p in ps])
    b = M.Batch(ctx, [M.System(ctx, p) for p in ps], precision, nt)
    b.set_times(0.0, ts)
    alone = []
    for i, p in enumerate(ps):
        s = M.Batch(ctx, [M.System(ctx, p)], precision, nt)
        s.set_times(0.0, ts[i:i + 1])
        s.run()
        assert (s.sync() == 0).all()
        alone.append(s.get(0))
    paths = {b.path(i) for i in range(b.count)}
    assert {q[0] for q in paths} >= {M.MMF_PATH_JACOBI, M.MMF_PATH_DENSE, M.MMF_PATH_BAND}
    for graph in (False, True):
        b.graph(graph)
        for _ in range(3):
            b.run()
            assert (b.sync() == 0).all()
            for i, (E, U, P) in enumerate(alone):
                e, u, pp = b.get(i)
                assert np.abs(e - E).max() <= 1e-12 * np.abs(E).max() * (1 if precision == M.MMF_FP64 else 1e3), i
                assert np.abs(u - U).max() <= tol and np.abs(pp - P).max() <= tol, i


@pytest.mark.parametrize("precision", [M.MMF_FP64, M.MMF_MIXED])
def test_whole_gpu_reduction_under_graph_replay(precision):
    """The whole-GPU reduction's launches depend on one another programmatically; captured in a graph
    and replayed they give what plain launches give (n at the edges of the 64-row groups and of the
    32-column panels)."""
    for D, N in [(1, 46), (3, 21), (1, 80)]:  # n = 93, 129, 161
        ctx = M.Context(0)
        ctx.set_option(M.MMF_OPT_LARGE_N, 90)
        ctx.set_option(M.MMF_OPT_BAND_MAX, 0)
        ctx.set_option(M.MMF_OPT_JACOBI_N_FP64 if precision == M.MMF_FP64 else M.MMF_OPT_JACOBI_N_MIXED, 4)
        s = M.System(ctx, W.random_multimode(W.SplitMix64(5), D, [N]))
        b = M.Batch(ctx, [s], precision, 0)
        b.run()
        assert (b.sync() == 0).all() and b.path(0)[0] == M.MMF_PATH_WHOLE_GPU
        E = b.get(0)[0].copy()
        s.build(M.MMF_FP64)
        ref = np.linalg.eigvalsh(s.hamiltonian())
        tol = (1e-12 if precision == M.MMF_FP64 else 1e-9) * np.abs(ref).max()
        assert np.abs(E - ref).max() <= tol
        b.graph(True)
        for _ in range(2):
            b.run()
            assert (b.sync() == 0).all()
            assert np.abs(b.get(0)[0] - E).max() <= tol


def test_one_system_calls_in_any_order():
    """U and Pbar of a one-system handle are computed by their own calls: any order gives the same."""
    ctx = M.Context(0)
    p = W.spin1_bichromatic(0.3, 0.2, N1=4, N2=3)
    t = W.time_grid(p, 5)
    ref = None
    for order in ("UP", "PU", "PUP", "UUP"):
        for precision in (M.MMF_FP64, M.MMF_MIXED):
            s = M.System(ctx, p)
            s.build(precision)
            s.diagonalise()
            got = {}
            for c in order:
                got[c] = s.time_evolution(t) if c == "U" else s.transition_avg()
            ref = ref or got
            assert np.abs(got["U"] - ref["U"]).max() <= 1e-8 and np.abs(got["P"] - ref["P"]).max() <= 1e-8
            s.diagonalise()  # new eigenpairs: Pbar again
            assert np.abs(s.transition_avg() - ref["P"]).max() <= 1e-8

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

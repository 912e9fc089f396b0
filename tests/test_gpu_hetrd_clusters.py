"""The dense Householder reduction (k_hetrd) over its cluster sizes: the largest cluster that one wave
holds for the batch (8, 6, 4, 2 or 1 CTAs per system), at dimensions on both sides of the tiles'
edges (32-row chunks, 64- and 128-row tasks, 32-column panels) and of the sizes from which larger
clusters are taken.  Quasienergies against LAPACK on the assembled matrix, to the library's bounds of
1e-12 ||H_F|| (FP64) and 1e-9 ||H_F|| (mixed)."""

import numpy as np
import pytest

from paper_2005_03426_gb300 import mmf as M
from paper_2005_03426_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {M.MMF_FP64: 1e-12, M.MMF_MIXED: 1e-9}


def _check(problems, precision, at, tc=1):
    ctx = M.Context(0)
    ctx.set_option(M.MMF_OPT_BAND_MAX, 0)
    ctx.set_option(M.MMF_OPT_JACOBI_N_FP64 if precision == M.MMF_FP64 else M.MMF_OPT_JACOBI_N_MIXED, 4)
    ctx.set_option(M.MMF_OPT_HETRD_TC, tc)
    systems = [M.System(ctx, p) for p in problems]
    b = M.Batch(ctx, systems, precision, 0)
    b.run()
    assert (b.sync() == 0).all()
    for i in at:
        assert b.path(i)[0] == M.MMF_PATH_DENSE
        systems[i].build(M.MMF_FP64)
        ref = np.linalg.eigvalsh(systems[i].hamiltonian())
        assert np.abs(b.get(i)[0] - ref).max() <= TOL[precision] * np.abs(ref).max(), i


# n = D (2 N + 1)
@pytest.mark.parametrize("precision", [M.MMF_FP64, M.MMF_MIXED])
@pytest.mark.parametrize("D,N", [(3, 1), (5, 6), (7, 4), (5, 25), (15, 8), (17, 7), (35, 5), (43, 4), (55, 3), (77, 2),
                                 (129, 1), (171, 1)])
def test_one_system(precision, D, N):
    _check([W.random_multimode(W.SplitMix64(D), D, [N])], precision, [0])


@pytest.mark.parametrize("precision,tc", [(M.MMF_FP64, 0), (M.MMF_MIXED, 0), (M.MMF_MIXED, 1)])
@pytest.mark.parametrize("count", [10, 20, 30, 60, 100])
def test_batches(precision, tc, count):
    rng = W.SplitMix64(count)
    shapes = [(43, 4), (5, 6), (35, 5)]  # n = 387, 65, 385 in turn
    _check([W.random_multimode(rng, *[(D, [N]) for D, N in shapes][i % 3]) for i in range(count)], precision,
           [0, 1, count - 1], tc)

"""The whole-GPU reduction's workspace: systems behind others of odd dimension in the same plan (the
sum of n^2 before them is odd), and the smallest systems it can be asked for, whose n^2 doubles are
fewer than the workspace takes.  Quasienergies against LAPACK on the assembled matrix, to the
library's bounds of 1e-12 ||H_F|| (FP64) and 1e-9 ||H_F|| (mixed); the eigenvectors by their residual
and orthogonality."""

import numpy as np
import pytest

from paper_2005_03426_gb300 import mmf as M
from paper_2005_03426_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {M.MMF_FP64: 1e-12, M.MMF_MIXED: 1e-9}
VEC = {M.MMF_FP64: 1e-10, M.MMF_MIXED: 1e-8}  # the library's bounds on U, which the eigenvectors carry


# n = D (2 N + 1); `large`: smallest n reduced by the whole GPU
@pytest.mark.parametrize("precision", [M.MMF_FP64, M.MMF_MIXED])
@pytest.mark.parametrize("large,shapes", [
    (90, [(3, 10), (3, 21)]),                        # 63, 129: one odd square before
    (90, [(5, 6), (8, 9), (7, 9), (4, 16), (3, 21)]),  # 65, 152, 133, 132, 129
    (5, [(1, 2)]), (5, [(2, 1)]), (5, [(1, 3)]), (5, [(1, 4), (1, 2)]), (5, [(1, 5), (3, 2)]),  # n = 5 .. 15
])
def test_matches_lapack(precision, large, shapes):
    ctx = M.Context(0)
    ctx.set_option(M.MMF_OPT_LARGE_N, large)
    ctx.set_option(M.MMF_OPT_BAND_MAX, 0)
    ctx.set_option(M.MMF_OPT_JACOBI_N_FP64 if precision == M.MMF_FP64 else M.MMF_OPT_JACOBI_N_MIXED, 4)
    rng = W.SplitMix64(large + len(shapes))
    systems = [M.System(ctx, W.random_multimode(rng, D, [N])) for D, N in shapes]
    b = M.Batch(ctx, systems, precision, 0)
    b.run()
    assert (b.sync() == 0).all()
    for i, s in enumerate(systems):
        assert b.path(i)[0] == (M.MMF_PATH_WHOLE_GPU if s.n >= large else M.MMF_PATH_DENSE)
        s.build(M.MMF_FP64)
        H = s.hamiltonian()
        ref = np.linalg.eigvalsh(H)
        nrm = np.abs(ref).max()
        E, Z = b.get(i)[0], b.eigenvectors(i)
        assert np.abs(E - ref).max() <= TOL[precision] * nrm, i
        assert np.abs(H @ Z - Z * E[None, :]).max() <= VEC[precision] * nrm, i
        assert np.abs(Z.conj().T @ Z - np.eye(s.n)).max() <= VEC[precision], i

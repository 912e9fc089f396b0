"""The one-CTA dense reduction (k_hetrd_small): dimensions at the edges of its 32-row groups and of its
range (n up to 103 in FP64, 152 in FP32, the next size taking the cluster kernel), a system alone and
in a batch of uneven ones.  Quasienergies against LAPACK on the assembled matrix, to the library's
bounds of 1e-12 ||H_F|| (FP64) and 1e-9 ||H_F|| (mixed); the back-transformed eigenvectors by their
residual and orthogonality."""

import numpy as np
import pytest

from paper_2005_03426_gb300 import mmf as M
from paper_2005_03426_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {M.MMF_FP64: 1e-12, M.MMF_MIXED: 1e-9}
VEC = {M.MMF_FP64: 1e-10, M.MMF_MIXED: 1e-8}  # the library's bounds on U, which the eigenvectors carry


@pytest.mark.parametrize("precision", [M.MMF_FP64, M.MMF_MIXED])
@pytest.mark.parametrize("shapes", [[(1, 2)], [(1, 15)], [(1, 16)], [(1, 51)], [(1, 52)], [(1, 75)], [(8, 9)], [(9, 8)],
                                    [(3, 1), (2, 20), (5, 6), (1, 47), (1, 48), (8, 9), (1, 51)]])
def test_matches_lapack(precision, shapes):
    ctx = M.Context(0)
    ctx.set_option(M.MMF_OPT_BAND_MAX, 0)
    ctx.set_option(M.MMF_OPT_JACOBI_N_FP64 if precision == M.MMF_FP64 else M.MMF_OPT_JACOBI_N_MIXED, 4)
    rng = W.SplitMix64(len(shapes) + shapes[0][1])
    systems = [M.System(ctx, W.random_multimode(rng, D, [N])) for D, N in shapes]  # n = D (2 N + 1)
    b = M.Batch(ctx, systems, precision, 0)
    b.run()
    assert (b.sync() == 0).all()
    for i, s in enumerate(systems):
        assert b.path(i)[0] == M.MMF_PATH_DENSE
        s.build(M.MMF_FP64)
        H = s.hamiltonian()
        ref = np.linalg.eigvalsh(H)
        nrm = np.abs(ref).max()
        E, Z = b.get(i)[0], b.eigenvectors(i)
        assert np.abs(E - ref).max() <= TOL[precision] * nrm, i
        # eigenvectors (the back-transform, k_bt_small)
        assert np.abs(H @ Z - Z * E[None, :]).max() <= VEC[precision] * nrm, i
        assert np.abs(Z.conj().T @ Z - np.eye(s.n)).max() <= VEC[precision], i

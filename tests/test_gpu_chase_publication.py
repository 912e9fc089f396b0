"""The band chase (k_sbr_chase) where a sweep's first rows are published ahead (narrow windows, whatever
the number of CTAs per system) and where they are not (wide windows with one or two CTAs per system):
batches large enough that a system gets one or two CTAs, at every window class.  Quasienergies against
LAPACK on the assembled matrix, to the library's bounds of 1e-12 ||H_F|| (FP64) and 1e-9 ||H_F||
(mixed); the eigenvectors (back-transform) by their residual and orthogonality."""

import numpy as np
import pytest

from paper_2005_03426_gb300 import mmf as M
from paper_2005_03426_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {M.MMF_FP64: 1e-12, M.MMF_MIXED: 1e-9}
VEC = {M.MMF_FP64: 1e-10, M.MMF_MIXED: 1e-8}  # the library's bounds on U, which the eigenvectors carry


# one mode, dense coupling: half-bandwidth 2 D - 1, n = D (2 N + 1)
@pytest.mark.parametrize("precision", [M.MMF_FP64, M.MMF_MIXED])
@pytest.mark.parametrize("D,N,count", [(2, 60, 200), (4, 35, 70), (4, 35, 200), (8, 17, 70), (8, 17, 200),
                                       (16, 8, 40), (16, 8, 170), (32, 5, 70), (32, 5, 160)])
def test_batches(precision, D, N, count):
    ctx = M.Context(0)
    ctx.set_option(M.MMF_OPT_BAND_MAX, 64)
    ctx.set_option(M.MMF_OPT_JACOBI_N_FP64 if precision == M.MMF_FP64 else M.MMF_OPT_JACOBI_N_MIXED, 4)
    rng = W.SplitMix64(100 * D + count)
    systems = [M.System(ctx, W.random_multimode(rng, D, [N - i % 2])) for i in range(count)]
    b = M.Batch(ctx, systems, precision, 0)
    b.run()
    assert (b.sync() == 0).all()
    for i in (0, 1, count // 2, count - 1):
        assert b.path(i) == (M.MMF_PATH_BAND, 2 * D - 1)
        systems[i].build(M.MMF_FP64)
        H = systems[i].hamiltonian()
        ref = np.linalg.eigvalsh(H)
        nrm = np.abs(ref).max()
        E, Z = b.get(i)[0], b.eigenvectors(i)
        assert np.abs(E - ref).max() <= TOL[precision] * nrm, i
        assert np.abs(H @ Z - Z * E[None, :]).max() <= VEC[precision] * nrm, i
        assert np.abs(Z.conj().T @ Z - np.eye(systems[i].n)).max() <= VEC[precision], i

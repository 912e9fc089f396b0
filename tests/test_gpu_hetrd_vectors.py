"""The dense Householder reduction (k_hetrd) at every cluster size (1, 2, 4, 6 and 8 CTAs per system, which
size is asserted): quasienergies, and the eigenvectors that come back through its stored reflectors
and scalars, by their residual and orthogonality.  Bounds: 1e-12 ||H_F|| (FP64) and 1e-9 ||H_F||
(mixed) for the quasienergies against LAPACK on the assembled matrix; 1e-10 and 1e-8, the library's
bounds on U, for the eigenvectors."""

import ctypes

import numpy as np
import pytest

from paper_2005_03426_gb300 import mmf as M
from paper_2005_03426_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {M.MMF_FP64: 1e-12, M.MMF_MIXED: 1e-9}
VEC = {M.MMF_FP64: 1e-10, M.MMF_MIXED: 1e-8}


# systems of n = D (2 N + 1), dealt over the batch in turn; the last dimension is a system's on its own
@pytest.mark.parametrize("precision,tc", [(M.MMF_FP64, 0), (M.MMF_MIXED, 0), (M.MMF_MIXED, 1)])
@pytest.mark.parametrize("ctas,count,shapes", [
    (8, 1, [(43, 4)]), (8, 9, [(43, 4), (35, 5), (31, 2)]),
    (6, 20, [(43, 4), (35, 5), (31, 2)]),
    (4, 1, [(37, 4)]), (4, 30, [(43, 4), (35, 5), (31, 2)]),
    (2, 1, [(31, 2)]), (2, 60, [(43, 4), (35, 5), (31, 2)]),
    (1, 160, [(43, 4), (31, 2), (17, 7)]),
])
def test_eigenvectors(precision, tc, ctas, count, shapes):
    ctx = M.Context(0)
    ctx.set_option(M.MMF_OPT_BAND_MAX, 0)
    ctx.set_option(M.MMF_OPT_HETRD_TC, tc)
    rng = W.SplitMix64(100 * ctas + count)
    systems = [M.System(ctx, W.random_multimode(rng, D, [N])) for D, N in (shapes * count)[:count]]
    got = ctypes.c_int()
    assert M.lib().mmf_selftest_hetrd_ctas(max(s.n for s in systems), count, precision, tc, ctypes.byref(got)) == 0
    assert got.value == ctas
    b = M.Batch(ctx, systems, precision, 0)
    b.run()
    assert (b.sync() == 0).all()
    for i in {0, min(1, count - 1), min(2, count - 1), count - 1}:
        assert b.path(i)[0] == M.MMF_PATH_DENSE
        systems[i].build(M.MMF_FP64)
        H = systems[i].hamiltonian()
        ref = np.linalg.eigvalsh(H)
        nrm = np.abs(ref).max()
        E, Z = b.get(i)[0], b.eigenvectors(i)
        assert np.abs(E - ref).max() <= TOL[precision] * nrm, i
        assert np.abs(H @ Z - Z * E[None, :]).max() <= VEC[precision] * nrm, i
        assert np.abs(Z.conj().T @ Z - np.eye(systems[i].n)).max() <= VEC[precision], i

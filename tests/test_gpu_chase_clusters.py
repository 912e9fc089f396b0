"""The band chase (k_sbr_chase) over its cluster sizes: one system takes the most CTAs its pipeline
can use (8 from these sizes on), larger batches 4, 2 and 1 per system; bands at both ends of every
window class, and dimensions one past a multiple of the band.  Quasienergies against LAPACK on the
assembled matrix, to the library's bounds of 1e-12 ||H_F|| (FP64) and 1e-9 ||H_F|| (mixed); the
eigenvectors (back-transform) by their residual and orthogonality."""

import numpy as np
import pytest

from paper_2005_03426_gb300 import mmf as M
from paper_2005_03426_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {M.MMF_FP64: 1e-12, M.MMF_MIXED: 1e-9}
VEC = {M.MMF_FP64: 1e-10, M.MMF_MIXED: 1e-8}  # the library's bounds on U, which the eigenvectors carry


def _check(problems, precision, at):
    ctx = M.Context(0)
    ctx.set_option(M.MMF_OPT_BAND_MAX, 64)
    systems = [M.System(ctx, p) for p in problems]
    b = M.Batch(ctx, systems, precision, 0)
    b.run()
    assert (b.sync() == 0).all()
    for i in at:
        assert b.path(i)[0] == M.MMF_PATH_BAND
        systems[i].build(M.MMF_FP64)
        H = systems[i].hamiltonian()
        ref = np.linalg.eigvalsh(H)
        nrm = np.abs(ref).max()
        E, Z = b.get(i)[0], b.eigenvectors(i)
        assert np.abs(E - ref).max() <= TOL[precision] * nrm, i
        # eigenvectors (the band back-transforms)
        assert np.abs(H @ Z - Z * E[None, :]).max() <= VEC[precision] * nrm, i
        assert np.abs(Z.conj().T @ Z - np.eye(systems[i].n)).max() <= VEC[precision], i


# one mode, dense coupling: half-bandwidth 2 D - 1, n = D (2 N + 1)
@pytest.mark.parametrize("precision", [M.MMF_FP64, M.MMF_MIXED])
@pytest.mark.parametrize("D,N", [(2, 130), (4, 65), (5, 52), (8, 64), (9, 29), (16, 16), (17, 15), (32, 8)])
def test_one_system_takes_the_largest_cluster(precision, D, N):
    _check([W.random_multimode(W.SplitMix64(D), D, [N])], precision, [0])


@pytest.mark.parametrize("precision", [M.MMF_FP64, M.MMF_MIXED])
@pytest.mark.parametrize("count", [24, 48, 100])
def test_batches_take_smaller_clusters(precision, count):
    rng = W.SplitMix64(count)
    _check([W.random_multimode(rng, 32, [4 + i % 2]) for i in range(count)], precision, [0, count // 2, count - 1])

"""Pbar of a one-system handle is kept until its eigenpairs are computed again: whether a call computes
it is read off the launch count."""

import numpy as np
import pytest

from paper_2005_03426_gb300 import mmf as M
from paper_2005_03426_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [M.MMF_FP64, M.MMF_MIXED])
def test_pbar_is_kept_until_new_eigenpairs(precision):
    count = M.lib().mmf_last_launch_count
    ctx = M.Context(0)
    p = W.spin1_bichromatic(0.3, 0.2, N1=4, N2=3)
    s = M.System(ctx, p)
    s.build(precision)
    s.diagonalise()
    ref = s.transition_avg()

    def launches(call):
        before = count()
        got = call()
        return count() - before, got

    def check(computed):
        k, P = launches(s.transition_avg)
        assert (k > 0) == computed
        assert np.abs(P - ref).max() <= 1e-8  # the library's bound on Pbar (mixed)

    check(False)
    s.time_evolution(W.time_grid(p, 3))  # another number of times: a new plan, with new eigenpairs
    check(True)
    check(False)
    s.time_evolution(W.time_grid(p, 3))  # the same plan and eigenpairs
    check(False)
    s.diagonalise()
    check(True)
    s.build(precision)
    s.diagonalise()
    check(True)
    check(False)

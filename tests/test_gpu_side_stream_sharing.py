"""The side streams on which a batch's solver paths run beside one another: plans of one stream share
them, so that their number does not grow with the plans (resident ones of a server included), and
plans that share them give what each gives alone; they have the priority of the stream they serve."""

import numpy as np
import pytest

from paper_2005_03426_gb300 import mmf as M
from paper_2005_03426_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NT = 4


def _context(stream=None):
    ctx = M.Context(0, stream=stream)
    ctx.set_option(M.MMF_OPT_BAND_MAX, 40)
    ctx.set_option(M.MMF_OPT_JACOBI_N_MIXED, 30)
    return ctx


def _problems(seed):
    # one-CTA and cluster dense reductions, chases of three window classes
    rng = W.SplitMix64(seed)
    return [W.random_multimode(rng, D, Ns) for D, Ns in [(5, [1, 8]), (7, [2, 4]), (3, [40]), (6, [20]), (16, [8])]]


def _batch(ctx, problems):
    b = M.Batch(ctx, [M.System(ctx, p) for p in problems], M.MMF_MIXED, NT)
    b.set_times(0.0, np.stack([W.time_grid(p, NT) for p in problems]))
    return b


def test_plans_of_one_stream_share_side_streams():
    ctx = _context()
    sets = [_problems(seed) for seed in range(6)]
    plans = [_batch(ctx, ps) for ps in sets]
    n = len(ctx.side_streams())
    assert 1 <= n <= 7
    for b in plans:  # all in flight before the first is waited for
        b.run()
    plans[0].graph(True)
    plans[0].run()
    for b, ps in zip(plans, sets):
        assert (b.sync() == 0).all()
        alone = _batch(_context(), ps)
        alone.run()
        assert (alone.sync() == 0).all()
        for i in range(b.count):
            for x, y, tol in zip(b.get(i), alone.get(i), (1e-9, 1e-8, 1e-8)):
                assert np.abs(x - y).max() <= tol * max(1.0, np.abs(y).max())
    assert len(ctx.side_streams()) == n


def test_resident_plans_of_a_server_share_side_streams():
    ctx = _context()
    slots, structures = 2, 6
    srv = M.Server(ctx, slots=slots, max_batch=5, precision=M.MMF_MIXED)
    for k in range(structures):
        # the same size class throughout, another structure each time: another resident plan
        ps = [W.random_multimode(W.SplitMix64(k), D, [N + k]) for D, N in [(9, 13), (17, 7), (40, 3)]]
        systems = [M.System(ctx, p) for p in ps]
        tickets = [srv.submit(s, W.time_grid(p, NT)) for s, p in zip(systems, ps)]
        for t in tickets:
            assert srv.wait(t, timeout_ms=120000)[3] == 0
    assert len(ctx.side_streams()) <= 7 * slots
    srv.close()
    assert ctx.side_streams() == []


def test_side_streams_have_the_priority_of_the_program_s_stream():
    torch = pytest.importorskip("torch")
    streams = [torch.cuda.Stream(priority=p) for p in torch.cuda.Stream.priority_range()]
    assert streams[0].priority != streams[1].priority
    for stream in streams:
        ctx = _context(stream.cuda_stream)
        b = _batch(ctx, _problems(1))
        b.run()
        assert (b.sync() == 0).all()
        got = [torch.cuda.ExternalStream(s).priority for s in ctx.side_streams()]
        assert got and set(got) == {stream.priority}

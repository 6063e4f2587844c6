"""lsas_run_frame and lsas_demodulate recorded into CUDA graphs, for batches
that a live call splits (one frame; 88 frames, which are cut into antenna
units; rows of N = 2048), on a plan that has split before the capture and on one
whose first call is the captured one.

The capture succeeds, replays give the live call's results bit for bit (both
run the same split), and live calls after it give what they gave on a plan that
was never captured.  Replays and live splits run on streams of their own with
inputs of their own and nothing between them, so that partial sums in a shared
place would meet.
"""

import numpy as np
import pytest

import synth
from synth.frames import FrameConfig

pytestmark = pytest.mark.gpu


def _frames(M, N, cp, F):
    import torch
    cfg = FrameConfig(M=M, N=N, cp=cp, S=6, Q=16, taps=4, decay_db=2.0, snr_db=25.0, fmt="sc16",
                      F=9, seed=5 + N)
    b = synth.generate(cfg)
    x = torch.from_numpy(np.ascontiguousarray(b.frames)).cuda()
    at = torch.arange(F, device="cuda") % 3
    return cfg, b, [x[3 * i:3 * i + 3][at].contiguous() for i in range(3)]


def _plan(cfg, b, F):
    import paper_1901_07499_gb300.lsas as L
    return L.Plan(cfg.M, cfg.N, cfg.cp, cfg.S, 0, 16, max_frames=F, pilot=b.pilot)


def _same(got, want):
    import torch
    return all(torch.equal(u, v) for u, v in zip(got, want))


@pytest.mark.parametrize("warm", [False, True], ids=["fresh", "after_a_split"])
@pytest.mark.parametrize("M,N,cp,F", [(64, 1024, 72, 1), (64, 1024, 72, 88), (32, 2048, 144, 3)])
def test_recorded_splits(M, N, cp, F, warm):
    import torch
    import paper_1901_07499_gb300.lsas as L
    cfg, b, x = _frames(M, N, cp, F)
    other = _plan(cfg, b, F)   # never captured
    want = [other.run_frame(x[i], want_eq=True) for i in range(3)]
    want_demod = [other.demodulate(x[i], want[i][0], want_eq=True) for i in range(3)]
    plan = _plan(cfg, b, F)
    assert plan.batch_split_shards(F) > 1
    if warm:
        assert _same(plan.run_frame(x[0], want_eq=True), want[0])
    torch.cuda.synchronize()
    outs, graphs = [], []
    for i in range(2):
        outs.append([plan.empty_H(F), plan.empty_bits(F), plan.empty_eq(F)])
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[i]):
            if i == 0:
                plan.run_frame(x[0], H=outs[0][0], bits=outs[0][1], eq=outs[0][2])
            else:
                plan.demodulate(x[1], want[1][0], bits=outs[1][1], eq=outs[1][2])
    streams = [torch.cuda.Stream() for _ in range(3)]
    for _ in range(5):
        for o in outs:
            for t in o:
                t.zero_()
        torch.cuda.synchronize()
        for i in range(2):
            with torch.cuda.stream(streams[i]):
                graphs[i].replay()
        with torch.cuda.stream(streams[2]):
            live = plan.run_frame(x[2], want_eq=True)
            live_demod = plan.demodulate(x[2], live[0], want_eq=True)
        torch.cuda.synchronize()
        assert plan.sync_status() == L.LSAS_OK
        assert _same(outs[0], want[0])
        assert _same(outs[1][1:], want_demod[1])
        assert _same(live, want[2]) and _same(live_demod, want_demod[2])
    del graphs
    plan.close()
    other.close()


def test_recorded_past_the_scratch_limit():
    """88 frames a call take about 13 MB of partial sums each: past 96 MiB the
    calls are recorded whole, with the unsplit call's results, and the earlier
    graphs keep theirs."""
    import torch
    import paper_1901_07499_gb300.lsas as L
    F = 88
    cfg, b, x = _frames(64, 1024, 72, F)
    plan = _plan(cfg, b, F)
    split = [t.clone() for t in plan.run_frame(x[0], want_eq=True)]
    plan.set_batch_split(0)
    whole = [t.clone() for t in plan.run_frame(x[0], want_eq=True)]
    plan.set_batch_split(1)
    assert not _same(split, whole)
    torch.cuda.synchronize()
    outs = [plan.empty_H(F), plan.empty_bits(F), plan.empty_eq(F)]
    graphs = []
    for _ in range(24):
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1]):
            plan.run_frame(x[0], H=outs[0], bits=outs[1], eq=outs[2])
    ran = []
    for g in graphs:
        for t in outs:
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        ran.append("split" if _same(outs, split) else "whole" if _same(outs, whole) else "other")
    first = ran.index("whole")
    assert first > 0 and ran == ["split"] * first + ["whole"] * (24 - first)
    assert plan.sync_status() == L.LSAS_OK
    del graphs
    plan.close()

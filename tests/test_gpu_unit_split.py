"""Batches whose frames after the last whole wave run as blocks of consecutive
antenna units (the two-symbol kernels): for frame counts from one to a wave,
antenna counts that are and are not whole units, every frame's H is the bytes
of the unsplit run, z within 1e-5 of its RMS (the antenna sums are ordered
differently: at most 256 terms, 256 * 2^-24 = 1.5e-5 in the worst case for terms
of one sign) and the bits the slicer's decision on that z; sampled frames meet
the oracle.  All frames are one frame repeated, so that a block's second
segment, another frame's antennas, would show.
"""

import numpy as np
import pytest

import oracle
import synth
from synth.frames import FrameConfig
from tests.parity_util import check_frame_outputs, oracle_run, unpack

pytestmark = pytest.mark.gpu

SHAPES = [(64, 1024, 72, 14, "sc16"), (20, 1024, 128, 5, "sc16"), (40, 512, 36, 8, "sc16"),
          (136, 256, 32, 4, "sc16"), (36, 2048, 144, 8, "sc16"), (18, 2048, 144, 5, "fc32"),
          (64, 2048, 144, 3, "fc32")]


@pytest.mark.parametrize("given", [False, True], ids=["estimate", "given"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "M%d_N%d_cp%d_S%d_%s" % s)
def test_unit_split(shape, given):
    import torch
    import paper_1901_07499_gb300.lsas as L
    M, N, cp, S, fmt = shape
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cfg = FrameConfig(M=M, N=N, cp=cp, S=S, Q=16, pilot_idx=1, taps=4, decay_db=2.0, snr_db=25.0,
                      fmt=fmt, F=2, seed=3 + M)
    b = synth.generate(cfg)
    most = sms + 130
    plan = L.Plan(M, N, cp, S, 1, 16, fmt=fmt, max_frames=most, pilot=b.pilot)
    two = torch.from_numpy(np.ascontiguousarray(b.frames)).cuda()
    ref = oracle_run(cfg, b)
    Hg = torch.from_numpy(ref.H.astype(np.complex64)).cuda()
    plan.set_batch_split(0)
    H0, bits0, eq0 = plan.run_frame(two, want_eq=True)
    if given:
        bits0, eq0 = plan.demodulate(two, Hg, want_eq=True)
    rms = float(eq0.abs().square().mean().sqrt())
    plan.set_batch_split(1)
    split = 0
    for F in (1, 2, 3, 7, 19, 44, 77, 88, 121, sms - 1, sms, sms + 5, sms + 76, most):
        idx = torch.arange(F, device="cuda") % 2
        x = two[idx].contiguous()
        split += plan.batch_split_shards(F) > 1
        if given:
            bits, eq = plan.demodulate(x, Hg[idx].contiguous(), want_eq=True)
        else:
            H, bits, eq = plan.run_frame(x, want_eq=True)
            assert torch.equal(H, H0[idx])
        assert plan.sync_status() == L.LSAS_OK
        assert float((eq - eq0[idx]).abs().max()) <= 1.5e-5 * rms * 4
        at = [0, F // 2, F - 1]
        z = eq[at].cpu().numpy()
        got = unpack(bits[at].cpu().numpy(), cfg.D, N, 4)
        want, _ = oracle.demap(z, 16, dtype=np.float32)
        assert np.array_equal(got, want)
        assert np.mean(bits.cpu().numpy() != bits0[idx].cpu().numpy()) <= 1e-4
    assert split > 0
    check_frame_outputs(cfg, ref, H0.cpu().numpy(), bits0.cpu().numpy(), eq0.cpu().numpy())
    plan.close()


def test_split_scratch_over_streams():
    """Splits of one plan on one stream, on others in turn and on a stream
    created after one was destroyed: each must wait for the previous split's
    combine, by stream order or by event.  Every call has inputs of its own and
    nothing synchronises in between."""
    import torch
    import paper_1901_07499_gb300.lsas as L
    cfg = FrameConfig(M=64, N=1024, cp=72, S=14, Q=16, taps=4, snr_db=25.0, fmt="sc16", F=6, seed=8)
    b = synth.generate(cfg)
    plan = L.Plan(cfg.M, cfg.N, cfg.cp, cfg.S, 0, 16, max_frames=2, pilot=b.pilot)
    assert plan.batch_split_shards(1) > 1
    x = torch.from_numpy(np.ascontiguousarray(b.frames)).cuda()
    want = [[t.clone() for t in plan.run_frame(x[i:i + 1], want_eq=True)] for i in range(6)]
    torch.cuda.synchronize()
    a, c = torch.cuda.Stream(), torch.cuda.Stream()
    order = [a, a, c, a, c, c] * 5
    outs = []
    for k, st in enumerate(order):
        with torch.cuda.stream(st):
            outs.append((k % 6, plan.run_frame(x[k % 6:k % 6 + 1], want_eq=True)))
    torch.cuda.synchronize()
    for _ in range(3):   # ids are not taken over by streams created later
        d = torch.cuda.Stream()
        with torch.cuda.stream(d):
            outs.append((1, plan.run_frame(x[1:2], want_eq=True)))
        outs.append((2, plan.run_frame(x[2:3], want_eq=True)))
        del d
    torch.cuda.synchronize()
    assert plan.sync_status() == L.LSAS_OK
    for i, got in outs:
        for u, v in zip(got, want[i]):
            assert torch.equal(u, v)
    plan.close()

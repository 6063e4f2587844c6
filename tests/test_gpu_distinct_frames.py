"""Batches of frames that all differ, through every way of dividing them: tail
frames as symbol parts and pairs cut over warps (the per-warp kernel), antenna
units and equal shards (the two-symbol kernels), each with the channel estimated
and given.  A block that reads another frame's or antenna's rows, however far
off, shows.

Frames: thirteen generated ones, their antennas rotated by one more position
each time round.  Every frame is also received alone and unsplit.  The per-warp
kernel's batches give those bytes.  Where antennas are split only the order of
their sums differs: H and, where z lies away from a boundary, the bits are the
same, and z differs by at most M * 2^-24 of the largest amplitude for the
numerator and as much for the energy; 1.5 times the RMS bounds the amplitudes
of 16-QAM with noise at 25 dB.  Sampled frames meet the oracle, the given channel's
with that channel.
"""

import numpy as np
import pytest

import oracle
import synth
from synth.frames import FrameConfig
from tests.parity_util import check_frame_outputs, unpack

pytestmark = pytest.mark.gpu

# M, N, cp, S, pilot_idx, fmt, frames after the last whole wave, whole waves
SHAPES = [
    (8, 64, 16, 15, 0, "fc32", 16, 0),       # pairs cut over warps, symbol parts
    (24, 256, 18, 14, 3, "sc16", 48, 1),     # parts behind a wave, shifted copies
    (11, 512, 36, 14, 0, "sc16", 7, 1),
    (3, 1024, 9, 14, 13, "sc16", 30, 0),
    (64, 1024, 72, 6, 0, "sc16", 88, 0),     # antenna units over two frames
    (64, 1024, 128, 4, 1, "sc16", 76, 1),    # behind a wave
    (40, 512, 36, 5, 2, "sc16", 121, 0),
    (36, 2048, 144, 4, 0, "sc16", 44, 0),
    (18, 2048, 144, 4, 3, "fc32", 19, 0),
    (64, 1024, 9, 4, 0, "sc16", 20, 0),      # unaligned rows: equal shards, per-warp kernel
]


def _frames(b, M, F):
    import torch
    base = torch.from_numpy(np.ascontiguousarray(b.frames)).cuda()
    return torch.cat([base[f % 13:f % 13 + 1].roll(f // 13, dims=1) for f in range(F)]).contiguous()


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "M%d_N%d_cp%d_S%d_p%d_%s_F%d+%dw" % s)
def test_every_frame_is_its_own(shape):
    import torch
    import paper_1901_07499_gb300.lsas as L
    M, N, cp, S, pi, fmt, tail, waves = shape
    F = tail + waves * torch.cuda.get_device_properties(0).multi_processor_count
    cfg = FrameConfig(M=M, N=N, cp=cp, S=S, Q=16, pilot_idx=pi, taps=3, decay_db=2.0, snr_db=25.0,
                      fmt=fmt, F=13, seed=29 + M + N)
    b = synth.generate(cfg)
    x = _frames(b, M, F)
    plan = L.Plan(M, N, cp, S, pi, 16, fmt=fmt, max_frames=F, pilot=b.pilot)
    plan.set_batch_split(0)
    alone = [[], [], [], [], []]
    for f in range(F):
        H, bits, eq = plan.run_frame(x[f:f + 1], want_eq=True)
        given = H * (1.0 + 0.01 * (f % 7))   # not the estimate
        for into, t in zip(alone, (H, bits, eq, *plan.demodulate(x[f:f + 1], given, want_eq=True))):
            into.append(t)
    H1, bits1, eq1, dbits1, deq1 = (torch.cat(t) for t in alone)
    scale = 1.0 + 0.01 * (torch.arange(F, device="cuda") % 7)
    given = H1 * scale[:, None, None].float()
    plan.set_batch_split(1)
    split = plan.batch_split_shards(F) > 1
    H, bits, eq = plan.run_frame(x, want_eq=True)
    dbits, deq = plan.demodulate(x, given, want_eq=True)
    assert plan.sync_status() == L.LSAS_OK
    assert torch.equal(H, H1)
    for z, z1, c, c1 in ((eq, eq1, bits, bits1), (deq, deq1, dbits, dbits1)):
        if not split:
            assert torch.equal(z, z1) and torch.equal(c, c1)
            continue
        rms = float(z1.abs().square().mean().sqrt())
        assert float((z - z1).abs().max()) <= 2 * M * 2.0**-24 * 1.5 * rms
        want, _ = oracle.demap(z.cpu().numpy(), 16, dtype=np.float32)
        assert np.array_equal(unpack(c.cpu().numpy(), cfg.D, N, 4), want)
    at = sorted({0, 5, F // 2, F - 1})
    sub = cfg.replace(F=len(at))
    xb = x[at].cpu().numpy()
    ref = oracle.receive(xb, N, cp, S, pi, 16, b.pilot)
    check_frame_outputs(sub, ref, H[at].cpu().numpy(), bits[at].cpu().numpy(), eq[at].cpu().numpy())
    Hg = given[at].cpu().numpy().astype(np.complex128)
    ref = oracle.receive(xb, N, cp, S, pi, 16, b.pilot, H_given=Hg)
    check_frame_outputs(sub, ref, None, dbits[at].cpu().numpy(), deq[at].cpu().numpy(), check_H=False)
    plan.close()

"""The per-warp kernel's ways of dividing a frame: antenna chunks on fewer
warps than the block has (pairs of chunk and data symbol cut evenly), frames
after the last whole wave as several blocks with a part of the data symbols
each, and rows that do not start on 16 bytes.

One frame repeated (a wave and a few more): every frame's H, z and bits are the
same bits whichever way it ran, and the oracle's within the bars of
parity_util.
"""

import numpy as np
import pytest

import synth
from synth.frames import FrameConfig
from tests.parity_util import check_frame_outputs, oracle_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import paper_1901_07499_gb300.lsas as lsas
    return lsas


# M, N, cp, S, pilot_idx, fmt: chunks of 32/(N/32) antennas
SHAPES = [
    (8, 64, 16, 15, 0, "fc32"),      # one chunk, half full
    (3, 64, 9, 2, 1, "sc16"),        # one data symbol
    (40, 64, 5, 64, 7, "sc16"),      # three chunks, 63 data symbols, rows at 4 mod 16
    (5, 128, 9, 14, 0, "sc16"),      # one chunk
    (24, 256, 18, 14, 3, "sc16"),    # six chunks, rows at 8 mod 16
    (28, 256, 18, 14, 0, "fc32"),    # seven chunks
    (24, 256, 17, 5, 0, "fc32"),     # rows at 8 mod 16, three blocks of fc32
    (64, 256, 19, 7, 2, "sc16"),     # as many pairs of chunks as warps
    (11, 512, 36, 14, 0, "sc16"),    # six chunks, the last half full
    (10, 512, 3, 3, 0, "sc16"),
    (5, 1024, 9, 14, 13, "sc16"),    # five antennas, several data-symbol groups
    (3, 1024, 128, 14, 0, "fc32"),
    (9, 1024, 11, 4, 0, "sc16"),     # one chunk more than warps
]


@pytest.mark.parametrize("extra", [0, 1, 5, 60])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "M%d_N%d_cp%d_S%d_p%d_%s" % s)
def test_every_division_gives_the_same_bits(L, shape, extra):
    import torch
    M, N, cp, S, pi, fmt = shape
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    F = extra if extra else sms
    F = F if extra != 5 else sms + 5
    cfg = FrameConfig(M=M, N=N, cp=cp, S=S, Q=4, pilot_idx=pi, taps=3, decay_db=2.0, snr_db=25.0,
                      fmt=fmt, F=1, seed=11 + M + N)
    b = synth.generate(cfg)
    plan = L.Plan(M, N, cp, S, pi, 4, fmt=fmt, max_frames=F, pilot=b.pilot)
    plan.set_batch_split(0)
    x = torch.from_numpy(np.ascontiguousarray(b.frames)).cuda().repeat(F, 1, 1, 1)
    H, bits, eq = plan.run_frame(x, want_eq=True)
    dbits, deq = plan.demodulate(x, H, want_eq=True)
    plan.sync()
    check_frame_outputs(cfg, oracle_run(cfg, b), H[:1].cpu().numpy(), bits[:1].cpu().numpy(),
                        eq[:1].cpu().numpy())
    assert torch.equal(dbits[:1].cpu(), bits[:1].cpu()) or shape[1] >= 1024
    for t in (H, bits, eq, dbits, deq):
        v = torch.view_as_real(t) if t.is_complex() else t
        assert bool((v == v[:1]).all())
    plan.close()


@pytest.mark.parametrize("cp", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_buffers_at_every_alignment(L, cp, offset):
    """Input buffers at every 4-byte offset, with prefixes shorter than the
    step back to a 16-byte boundary; nothing around the buffer is read into
    the results (the guard samples would change them)."""
    import torch
    cfg = FrameConfig(M=6, N=128, cp=cp, S=4, Q=4, taps=1, snr_db=25.0, fmt="sc16", F=2,
                      seed=cp + 10)
    b = synth.generate(cfg)
    plan = L.Plan(cfg.M, cfg.N, cp, cfg.S, 0, 4, max_frames=2, pilot=b.pilot)
    n = b.frames.size
    outs = []
    for guard in (0, 32767):
        buf = torch.full((n + 64,), guard, dtype=torch.int16, device="cuda")
        x = buf[32 + 2 * offset:32 + 2 * offset + n].view(2, cfg.M, cfg.T, 2)
        x.copy_(torch.from_numpy(b.frames))
        outs.append([t.cpu().numpy() for t in plan.run_frame(x, want_eq=True)])
    plan.sync()
    for u, v in zip(*outs):
        assert np.array_equal(u, v)
    check_frame_outputs(cfg, oracle_run(cfg, b), outs[0][0], outs[0][1], outs[0][2])
    plan.close()

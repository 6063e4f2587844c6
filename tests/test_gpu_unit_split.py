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

"""Which split the two-symbol kernels take for a batch under one wave of 152
blocks: equal shards where they fill it with as many steps a warp as antenna
units would (a block of units pays the group ends of two frames), units where
whole shards would leave the wave half empty or need a second one.  Figures:
lsas_plan_batch_split_shards, 2 for two shards a frame; units of five out of
eight make at most three blocks touch a frame.
"""

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,fmt,F,shards", [
    (48, 512, "sc16", 72, 2), (40, 1024, "sc16", 72, 2), (72, 1024, "sc16", 76, 2),
    (36, 2048, "sc16", 72, 2), (136, 256, "sc16", 72, 2), (36, 2048, "fc32", 76, 2),
    (64, 1024, "sc16", 88, 3), (64, 1024, "sc16", 1, 8), (64, 1024, "sc16", 151, 1)])
def test_shards(M, N, fmt, F, shards):
    import torch
    import paper_1901_07499_gb300.lsas as L
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms != 152:
        pytest.skip("figures for 152 SMs")
    plan = L.Plan(M, N, N // 8, 14, 0, 16, fmt=fmt, max_frames=2 * F)
    assert plan.batch_split_shards(F) == shards
    assert plan.batch_split_shards(F + sms) == shards
    plan.close()


@pytest.mark.parametrize("M,cp,F,shards", [(6, 109, 4, 2), (6, 109, 1, 2), (4, 33, 3, 2), (12, 1, 2, 4)])
def test_float_rows_off_16_bytes(M, cp, F, shards):
    """N = 2048 float rows that bulk copies cannot bring run on the
    warp-specialised kernel, whose pipeline takes two antennas: shards of two
    and three antennas are used and right."""
    import numpy as np
    import torch
    import synth
    import paper_1901_07499_gb300.lsas as L
    from synth.frames import FrameConfig
    from tests.parity_util import check_frame_outputs, oracle_run, to_torch_frames
    cfg = FrameConfig(M=M, N=2048, cp=cp, S=5, Q=16, pilot_idx=1, taps=3, decay_db=2.0, snr_db=25.0,
                      fmt="fc32", F=F, seed=cp)
    b = synth.generate(cfg)
    plan = L.Plan(M, 2048, cp, 5, 1, 16, fmt="fc32", max_frames=F, pilot=b.pilot)
    assert plan.batch_split_shards(F) == shards
    x, ref = to_torch_frames(b), oracle_run(cfg, b)
    H, bits, eq = plan.run_frame(x, want_eq=True)
    given = torch.from_numpy(ref.H.astype(np.complex64)).cuda()
    dbits, deq = plan.demodulate(x, given, want_eq=True)
    assert plan.sync_status() == L.LSAS_OK
    check_frame_outputs(cfg, ref, H.cpu().numpy(), bits.cpu().numpy(), eq.cpu().numpy())
    check_frame_outputs(cfg, ref, None, dbits.cpu().numpy(), deq.cpu().numpy(), check_H=False)
    plan.close()

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

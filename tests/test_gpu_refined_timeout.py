"""Failure detection in the learned receiver without a GPU fault: the
refinement's bounded wait for a tile's input rows runs out
(lsas_plan_set_fault(1): block 0 waits for 16 bytes that no copy delivers).

Twelve tiles a slot follow the one that gave up: no copy is issued into a buffer
whose last one was not waited for.  The call finishes, the refinement's status
word is LSAS_ERR_TIMEOUT (and the receiver's, whose first wait is held up too),
and the next call gives the bytes of a call before the fault.
"""

import time

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_input_wait_runs_out_and_recovers():
    import torch
    import paper_1901_07499_gb300.denoiser as D
    import paper_1901_07499_gb300.lsas as L
    cfg = synth.CONFIGS["scale"]
    b = synth.generate(cfg, frame_ids=range(2))
    F = 26   # 1664 rows, 14976 tiles: about 12 a slot on 304 blocks of four
    plan = L.Plan(cfg.M, cfg.N, cfg.cp, cfg.S, cfg.pilot_idx, cfg.Q, max_frames=F, pilot=b.pilot)
    x = torch.from_numpy(np.ascontiguousarray(b.frames)).cuda()[torch.arange(F, device="cuda") % 2]
    x = x.contiguous()
    dn = D.Denoiser(D.init_params(3))
    params, work = dn.bf16_params(), dn.work(F * cfg.M, cfg.N)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    want = [t.clone() for t in plan.run_frame_refined(x, params, work, status, want_eq=True)]
    assert plan.sync_status() == L.LSAS_OK and status.item() == 0
    assert L.lsas_plan_set_fault(plan.handle, 1) == L.LSAS_OK
    t0 = time.time()
    plan.run_frame_refined(x, params, work, status, want_eq=True)
    assert plan.sync_status() == L.LSAS_ERR_TIMEOUT
    assert status.item() == L.LSAS_ERR_TIMEOUT
    assert time.time() - t0 < 60.0
    assert L.lsas_plan_set_fault(plan.handle, 0) == L.LSAS_OK
    status.zero_()
    got = plan.run_frame_refined(x, params, work, status, want_eq=True)
    assert plan.sync_status() == L.LSAS_OK and status.item() == 0
    for u, v in zip(got, want):
        assert torch.equal(u, v)
    plan.close()

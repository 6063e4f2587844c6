"""Antenna shards of rows that do not start on 16 bytes: shards in the middle
and at either end of the antennas, prefixes shorter and longer than the step
back to a 16-byte boundary, at every 4-byte offset of the input.

Bars of the antenna split (partial sums and the combined outputs against the
oracle, H the unsharded call's bits, tests/test_gpu_shard.py); and what other
antennas hold changes no bit of a shard's outputs.
"""

import pytest

import synth
from synth.frames import FrameConfig
from tests.test_gpu_shard import check_split, make_plan

pytestmark = pytest.mark.gpu

BOUNDS = [(0, 1), (1, 6), (6, 11)]


def _cfg(N, cp, fmt):
    return FrameConfig(M=11, N=N, cp=cp, S=4, Q=16, pilot_idx=3, taps=2, decay_db=2.0, snr_db=25.0,
                       fmt=fmt, F=3, seed=cp + N)


@pytest.mark.parametrize("N,cp,fmt", [(64, 1, "sc16"), (128, 2, "sc16"), (128, 3, "sc16"),
                                      (128, 9, "sc16"), (64, 3, "fc32"), (128, 1, "fc32"),
                                      (1024, 2, "sc16")])
def test_shards_of_unaligned_rows(N, cp, fmt):
    import torch
    import paper_1901_07499_gb300.lsas as L
    cfg = _cfg(N, cp, fmt)
    check_split(L, cfg, BOUNDS, F=3)
    b = synth.generate(cfg)
    plan = make_plan(L, cfg, 3)
    word = torch.int16 if fmt == "sc16" else torch.float32
    n = b.frames.size
    for off in ([0, 1, 2, 3] if fmt == "sc16" else [0, 1]):   # samples past 16 bytes
        outs = []
        for other in (0, 77):
            buf = torch.full((n + 64,), other, dtype=word, device="cuda")
            x = buf[16 + 2 * off:16 + 2 * off + n].view(3, cfg.M, cfg.T, 2)
            x[:, 1:6] = torch.from_numpy(b.frames).cuda()[:, 1:6]
            H = torch.zeros((3, cfg.M, N), dtype=torch.complex64, device="cuda")
            P, E = plan.empty_partials(3, 1, device=x.device)
            plan.mrc_partial(x, 1, 5, H, P[0], E[0])
            plan.sync()
            outs.append((H, P, E))
        for u, v in zip(*outs):
            assert torch.equal(u, v)
        if off == 0:
            first = outs[0]
        for u, v in zip(first, outs[0]):
            assert torch.equal(u, v)
    plan.close()

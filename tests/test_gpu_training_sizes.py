"""Gradients of the refinement network (lsas_dn_grad, lsas_dn_grad_tc) against
the FP64 reference at the sizes where their kernels can go wrong: one tile of
128 positions, rows that are an odd number of tiles, fewer tiles than blocks,
an odd number of tiles in all, and the longest rows.

Bars, relative to the largest entry of a parameter block.  FP32: the bar of
tests/test_gpu_denoiser.py, 1e-4.  BF16: a weight gradient is a sum over
stored data gradients that went through at most three roundings to bf16 (g3,
g2, g1), each within 2^-9 of its value, so no block is off by more than
3 * 2^-9 of the sum of its terms' magnitudes in the worst case; 3 * 2^-9 = 6e-3
of the block's largest entry is asked (the errors have no common sign).
"""

import numpy as np
import pytest

import synth
from oracle import denoiser as odn

pytestmark = pytest.mark.gpu

SIZES = [(1, 128), (2, 384), (3, 640), (2, 2048), (37, 256)]


def _blocks_close(got, want, bar):
    o = 0
    for s in odn.SHAPES:
        n = int(np.prod(s))
        blk = want[o:o + n]
        err = np.max(np.abs(got[o:o + n] - blk)) / np.max(np.abs(blk))
        assert err <= bar, (s, err)
        o += n


@pytest.mark.parametrize("tc", [False, True], ids=["fp32", "bf16"])
@pytest.mark.parametrize("R,N", SIZES)
def test_gradient_at_tile_edges(R, N, tc):
    import torch
    import paper_1901_07499_gb300.denoiser as D
    H, Hls, _ = synth.ls_pairs(R, N, seed=101 + N)
    H, Hls = H.astype(np.complex64), Hls.astype(np.complex64)
    p = D.init_params(4) * np.float32(3.0)
    p += np.float32(0.01) * np.random.default_rng(5).standard_normal(p.size).astype(np.float32)
    dn = D.Denoiser(p)
    dn.work(R, N).fill_(float("nan"))   # nothing may be read before it is written
    loss, g = dn.compute_grad(torch.from_numpy(Hls).cuda(), torch.from_numpy(H).cuda(), tensor_cores=tc)
    assert int(dn.status().item()) == 0
    x0, rms = odn.prepare(Hls)
    t = np.stack([H.real, H.imag], 1) / rms[:, None, None]
    pr = p.astype(np.float64)
    if tc:
        b = p.view(np.uint32).astype(np.uint64)
        pr = (((b + 0x7FFF + ((b >> 16) & 1)) >> 16) << 16).astype(np.uint32).view(np.float32).astype(np.float64)
    y, cache = odn.forward(pr, x0, **({"act": odn.bf16_round} if tc else {}))
    want_loss, dy = odn.mse(y, t)
    if tc:
        cache = (cache[0],) + tuple(odn.bf16_round(np.maximum(a, 0)) for a in cache[1:])
    want = odn.backward(pr, cache, dy)
    assert abs(float(loss.item()) - want_loss) <= 1e-4 * want_loss
    _blocks_close(g.cpu().numpy(), want, 6e-3 if tc else 1e-4)

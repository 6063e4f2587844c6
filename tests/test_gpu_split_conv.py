"""The FP32 refinement's 32 -> 32 layers on split operands: values of any FP32
size, and tiles that the split cannot take.

Scaling layer 1's weights and bias by s = 2^k, layer 2's weights by 2^(j - k),
its bias by 2^j and layer 3's weights by 2^-j scales the outputs of layers 1 and
2 by 2^k and 2^j and leaves every later value as it was, exactly in FP32 while
nothing overflows or underflows.  The split holds from 2^-100 to 2^120: at j = 0
and k of 117 and more layer 2's weights are below that; at j = 28 they are not,
but the outputs of layer 1 above 8 (k = 117) or 4 (k = 118) are past its upper
end, so that tiles of both forms meet in one launch.  The smallest weights,
near 2^-123 at k = 120, lose at most 2^-149 * 2^120 = 2^-29 of a unit.  Bar: the 160-term sums of the
two forms differ by FP32 rounding, within 160 * 2^-24 = 1e-5 of the largest
output in the worst case of a layer, so 2e-5 for the two layers.
"""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,j", [(-60, 0), (117, 0), (118, 0), (120, 0), (117, 28), (118, 28)])
@pytest.mark.parametrize("R,N", [(3, 128), (5, 384), (400, 256)])
def test_scaled_layers(R, N, k, j):
    import torch
    import paper_1901_07499_gb300.denoiser as D
    H, Hls, _ = synth.ls_pairs(R, N, seed=7 + N)
    H, Hls = (torch.from_numpy(x.astype(np.complex64)).cuda() for x in (H, Hls))
    p = D.init_params(6)
    p += np.float32(0.01) * np.random.default_rng(8).standard_normal(p.size).astype(np.float32)
    q = p.copy()
    q[:352] = np.ldexp(q[:352], k)
    q[352:5472] = np.ldexp(q[352:5472], j - k)
    q[5472:5504] = np.ldexp(q[5472:5504], j)
    q[5504:10624] = np.ldexp(q[5504:10624], -j)
    a, b = D.Denoiser(p), D.Denoiser(q)
    a.work(R, N).fill_(float("nan"))
    b.work(R, N).fill_(float("nan"))
    want = a.apply(Hls, bf16=False)
    got = b.apply(Hls, bf16=False)
    top = want.abs().max().item()
    assert (got - want).abs().max().item() <= 2e-5 * top
    loss_a, ga = a.compute_grad(Hls, H)
    loss_b, gb = b.compute_grad(Hls, H)
    assert abs(loss_a.item() - loss_b.item()) <= 1e-4 * loss_a.item()
    # layers 3 and 4: the same gradients, layer 3's weights' times 2^j
    ga, gb = ga[5504:], gb[5504:].clone()
    gb[:5120] *= 2.0 ** -j
    assert (ga - gb).abs().max().item() <= 1e-4 * ga.abs().max().item()

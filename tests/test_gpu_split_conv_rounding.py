"""Rounding of the FP32 refinement's 32 -> 32 layers on split operands.

* No bias: tensor-core additions truncate, so a sum of plain bf16 terms loses
  about 2^-24 of its size, always towards zero; two layers shrink the network's
  part f(H) of the output by about 1e-7.  With biases of zero and entries of H
  from {1, -1, j, -j} (RMS exactly 1) out = H + f(H); the part of out - (H + f(H)
  in 64 bits) along f is the shrinking.  Additions rounded to nearest leave
  errors without a common sign, about 1e-7 of an output each: along f less than
  1e-7 / sqrt(131072) = 3e-10.  Bar: thirty times that, 1e-8.
* Channels of any size: a channel of a layer's output scaled by 2^-14 to 2^14 and
  its weights in the next layer by the inverse leave the outputs as they are.
  Bar: 3e-7 of the output (norm) against 64 bits, three layers of 160-term FP32
  sums at sqrt(160 / 3) * 2.4e-8 each.
* The upper end of the split's range (inputs of 2^60, times the size of their
  channel's largest weight, which is 1/4 to 1/2 here): with layer 2's weights
  scaled by 2^60 and layer 3's by the inverse, inputs from 4 to 8 on exceed it,
  so that tiles of both forms meet in one launch; 2^59 and 2^61 move that by two.
  Bar as in tests/test_gpu_split_conv.py: 2e-5 of the largest output.
"""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

W1, B1, W2, B2, W3, B3, W4, B4 = (slice(a, b) for a, b in (
    (0, 320), (320, 352), (352, 5472), (5472, 5504), (5504, 10624), (10624, 10656),
    (10656, 10976), (10976, 10978)))


def _params(seed, biases):
    rng = np.random.default_rng(seed)
    p = np.zeros(10978, np.float32)
    for s, fan in ((W1, 10), (W2, 160), (W3, 160), (W4, 160)):
        p[s] = rng.standard_normal(s.stop - s.start) * np.sqrt(2.0 / fan)
    if biases:
        for s in (B1, B2, B3, B4):
            p[s] = 0.02 * rng.standard_normal(s.stop - s.start)
    return p


def _network64(p, x):
    """f of [R][2][N] in 64 bits."""
    import torch
    import torch.nn.functional as nn
    q = torch.from_numpy(p).cuda().double()
    for w, b, shape in ((W1, B1, (32, 2, 5)), (W2, B2, (32, 32, 5)), (W3, B3, (32, 32, 5))):
        x = nn.conv1d(x, q[w].reshape(shape), q[b], padding=2).relu()
    return nn.conv1d(x, q[W4].reshape(2, 32, 5), q[B4], padding=2)


def _units(R, N):
    import torch
    units = torch.tensor([1, -1, 1j, -1j], dtype=torch.complex64, device="cuda")
    H = units[torch.from_numpy(np.random.default_rng(5).integers(0, 4, (R, N))).cuda()]
    return H, torch.stack([H.real, H.imag], 1).double()


def test_no_shrinking():
    import torch
    import paper_1901_07499_gb300.denoiser as D
    p = _params(4, False)
    H, x = _units(64, 1024)
    out = D.Denoiser(p).apply(H, bf16=False)
    f = _network64(p, x)
    err = torch.stack([out.real, out.imag], 1).double() - (x + f)
    assert err.abs().max().item() <= 1e-5 * f.abs().max().item()
    assert abs((err * f).sum().item()) <= 1e-8 * (f * f).sum().item()


def test_channels_of_any_size():
    import torch
    import paper_1901_07499_gb300.denoiser as D
    p = _params(6, True)
    rng = np.random.default_rng(7)
    a, b = (rng.integers(-14, 15, 32) for _ in range(2))   # powers of layer 1's and 2's channels
    power = np.zeros(p.size, int)
    power[W1], power[B1] = np.repeat(a, 10), a
    power[W2] = (np.repeat(b, 160).reshape(32, 32, 5) - a[None, :, None]).reshape(-1)
    power[B2] = b
    power[W3] = np.broadcast_to(-b[None, :, None], (32, 32, 5)).reshape(-1)
    H, x = _units(5, 384)
    want = x + _network64(p, x)
    for q in (p, np.ldexp(p, power).astype(np.float32)):
        out = D.Denoiser(q).apply(H, bf16=False)
        err = torch.stack([out.real, out.imag], 1).double() - want
        assert (err.norm() / want.norm()).item() <= 3e-7


@pytest.mark.parametrize("j", [59, 60, 61])
@pytest.mark.parametrize("R,N", [(3, 128), (400, 256)])
def test_both_forms_in_one_launch(R, N, j):
    import torch
    import paper_1901_07499_gb300.denoiser as D
    _, Hls, _ = synth.ls_pairs(R, N, seed=7 + N)
    Hls = torch.from_numpy(Hls.astype(np.complex64)).cuda()
    p = _params(8, True)
    power = np.zeros(p.size, int)
    power[W2] = power[B2] = j
    power[W3] = -j
    want = D.Denoiser(p).apply(Hls, bf16=False)
    got = D.Denoiser(np.ldexp(p, power).astype(np.float32)).apply(Hls, bf16=False)
    assert (got - want).abs().max().item() <= 2e-5 * want.abs().max().item()


@pytest.mark.parametrize("R,N", [(3, 128), (400, 256)])
def test_gradients_where_weights_are_out_of_range(R, N):
    """Layer 2's weights scaled by 2^62 and layer 1 by the inverse: layer 2 and
    its data gradient are summed by FMAs throughout.  The gradients differ from
    the unscaled network's by those powers and the two forms' rounding (bar of
    tests/test_gpu_split_conv.py: 1e-4 of a block's largest)."""
    import torch
    import paper_1901_07499_gb300.denoiser as D
    H, Hls, _ = synth.ls_pairs(R, N, seed=9 + N)
    H, Hls = (torch.from_numpy(v.astype(np.complex64)).cuda() for v in (H, Hls))
    p = _params(10, True)
    power = np.zeros(p.size, int)
    power[W1] = power[B1] = -62
    power[W2] = 62
    (loss, want), (loss_e, got) = (
        [t.cpu().numpy() for t in D.Denoiser(q).compute_grad(Hls, H)]
        for q in (p, np.ldexp(p, power).astype(np.float32)))
    assert abs(loss_e[0] - loss[0]) <= 1e-4 * loss[0]
    got = np.ldexp(got, power)
    for s in (W1, B1, W2, B2, W3, B3, W4, B4):
        assert np.abs(got[s] - want[s]).max() <= 1e-4 * np.abs(want[s]).max()

"""Order of the sums over blocks in the FP32 weight gradients: the partial rows
of sixteen slices, ten rows at a time, and then the slices, both as trees.

A network of zeros returns its input, so with H = 1 (RMS exactly 1) dy =
(x0 - t) 2/n is known bit for bit and layer 4's bias gradient is its plain sum.
With no more tiles than SMs a block sums one tile of 128 positions: four a
lane, then the lanes as a butterfly.  The sum added in that order in FP32 must
be the gradient's bits.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

F = np.float32


def _tree(v):
    v = list(v)
    while len(v) > 1:
        h = len(v) // 2
        v = [F(v[i] + v[i + h]) for i in range(h)]
    return v[0]


def _rows_sum(rows):
    per = -(-len(rows) // 16)
    slices = []
    for i in range(16):
        s, mine = F(0), rows[i * per:(i + 1) * per]
        for b in range(0, len(mine), 10):
            w = [F(x) for x in mine[b:b + 10]] + [F(0)] * (10 - len(mine[b:b + 10]))
            p = [F(w[j] + w[j + 1]) for j in range(0, 10, 2)]
            s = F(s + F(F(F(p[0] + p[1]) + F(p[2] + p[3])) + p[4]))
        slices.append(s)
    return _tree(slices)


@pytest.mark.parametrize("R", [1, 16, 17, 100, 128])
def test_bias_gradient_is_summed_in_a_tree(R):
    import torch
    import paper_1901_07499_gb300.denoiser as D
    import paper_1901_07499_gb300.lsas as L
    N = 128
    rng = np.random.default_rng(17 + R)
    dn = D.Denoiser(np.zeros(L.LSAS_DN_PARAMS, F))
    Hls = torch.ones((R, N), dtype=torch.complex64, device="cuda")
    scale = F(2.0) / F(2 * R * N)
    for _ in range(4):
        re, im = (rng.integers(2**21, 7 * 2**20, (R, N)) * 2.0**-22 for _ in range(2))   # 0.5 .. 1.75
        Ht = torch.from_numpy((1.0 - re - 1j * im).astype(np.complex64)).cuda()
        _, grad = dn.compute_grad(Hls, Ht)
        got = grad[-2:].cpu().numpy()
        for g, e in zip(got, (re, im)):
            dy = (e.astype(F) * scale).reshape(R, 32, 4)
            lanes = (dy[..., 0] + dy[..., 1]) + (dy[..., 2] + dy[..., 3])
            assert g == _rows_sum([_tree(row) for row in lanes])

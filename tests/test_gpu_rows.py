"""Symbol rows to memory (lsas_fft, lsas_estimate) and the receiver on rows in
memory (lsas_receive_y) where their kernels branch: numbers of rows that leave
a two-row step half empty or partly empty, fewer steps than warps, many steps
per warp, every N with aligned and unaligned rows; data symbols in one group
of four, in several, and in groups of seven.

Bars of parity_util (1e-4 of the RMS; the transform is also held to 1e-6 of
the row RMS, ten times the float32 rounding of a 2048-point transform).
"""

import numpy as np
import pytest

import oracle
import synth
from synth.frames import FrameConfig
from tests.parity_util import check_frame_outputs, oracle_run, rel_err, to_torch_frames

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import paper_1901_07499_gb300.lsas as lsas
    return lsas


@pytest.mark.parametrize("F", [1, 3])
@pytest.mark.parametrize("cp", [8, 9])
@pytest.mark.parametrize("M,N,S", [(1, 64, 2), (1, 128, 2), (5, 128, 3), (3, 256, 5), (1, 512, 3),
                                   (7, 512, 3), (1, 1024, 3), (9, 1024, 14), (3, 2048, 3)])
def test_transform_and_estimate_rows(L, M, N, S, cp, F):
    cfg = FrameConfig(M=M, N=N, cp=cp, S=S, Q=16, pilot_idx=S - 1, taps=4, snr_db=25.0, fmt="sc16",
                      F=F, seed=9 * N + M + cp)
    b = synth.generate(cfg)
    plan = L.Plan(M, N, cp, S, S - 1, 16, max_frames=F, pilot=b.pilot)
    x = to_torch_frames(b)
    Y = plan.fft(x).cpu().numpy()
    H = plan.estimate(x).cpu().numpy()
    plan.sync()
    y = b.as_complex().reshape(F, M, S, N + cp)[..., cp:]
    want = np.fft.fft(y, axis=-1) / np.sqrt(N)
    assert rel_err(Y, want, axes=(-1,)).max() <= 1e-5
    assert np.sqrt(np.mean(np.abs(Y - want) ** 2) / np.mean(np.abs(want) ** 2)) <= 1e-6
    assert rel_err(H, want[:, :, S - 1] / b.pilot, axes=(-1,)).max() <= 1e-4
    plan.close()


def test_many_steps_per_warp(L):
    """More rows than the launch's warps take in two steps each."""
    import torch
    M, N, cp, S, F = 16, 128, 8, 20, 200
    plan = L.Plan(M, N, cp, S, max_frames=F)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randint(-3000, 3000, (F, M, S * (N + cp), 2), generator=g, device="cuda").to(torch.int16)
    Y = plan.fft(x)
    plan.sync()
    y = torch.view_as_complex(x.double()).reshape(F, M, S, N + cp)[..., cp:]
    want = torch.fft.fft(y) / np.sqrt(N)
    assert float((Y - want).abs().max()) <= 1e-5 * float(want.abs().square().mean().sqrt())
    plan.close()


@pytest.mark.parametrize("M,N,S,pilot_idx,F", [(3, 64, 2, 0, 1), (5, 128, 5, 4, 2), (8, 512, 9, 2, 3),
                                               (2, 1024, 14, 13, 60), (4, 256, 15, 7, 300),
                                               (2, 64, 64, 30, 2), (1, 2048, 16, 0, 40)])
def test_receive_from_rows(L, M, N, S, pilot_idx, F):
    import torch
    cfg = FrameConfig(M=M, N=N, cp=8, S=S, Q=4, pilot_idx=pilot_idx, taps=2, snr_db=25.0, fmt="sc16",
                      F=min(F, 4), seed=N + S)
    b = synth.generate(cfg)
    ref = oracle_run(cfg, b, keep_Y=True)
    y = b.as_complex().reshape(cfg.F, M, S, N + 8)[..., 8:]
    Y = (np.fft.fft(y, axis=-1) / np.sqrt(N)).astype(np.complex64)
    reps = -(-F // cfg.F)
    plan = L.Plan(M, N, 8, S, pilot_idx, 4, max_frames=F, pilot=b.pilot)
    Yt = torch.from_numpy(Y).cuda().repeat(reps, 1, 1, 1)[:F].contiguous()
    H, bits, eq = plan.receive_y(Yt, want_eq=True)
    plan.sync()
    for f0 in range(0, F, cfg.F):
        n = min(cfg.F, F - f0)
        if n < cfg.F:
            break
        sl = slice(f0, f0 + n)
        if M == 1:   # zero forcing: near a fade only H and the slicer are held
            assert rel_err(H[sl].cpu().numpy(), ref.H, axes=(1, 2)).max() <= 1e-4
            got, _ = oracle.demap(eq[sl].cpu().numpy(), 4, dtype=np.float32)
            from tests.parity_util import unpack
            assert np.array_equal(got, unpack(bits[sl].cpu().numpy(), cfg.D, N, 2))
        else:
            check_frame_outputs(cfg, ref, H[sl].cpu().numpy(), bits[sl].cpu().numpy(),
                                eq[sl].cpu().numpy())
    plan.close()

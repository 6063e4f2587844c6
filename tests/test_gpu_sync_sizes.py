"""Packet detection and frame extraction at the sizes where their kernels
branch: antennas per round (up to 8, 16, 32 and more than one round), chips
in one and in several staged segments, lags that fill no, one and several
blocks of a cluster, windows that end at the capture's end, every alignment
of the cut and of the output.

Random +-1 chips are planted at a known lag over noise of a tenth of their
power per antenna, so the peak is clear of the runner-up; the offset must be the
oracle's, the peak power within 1e-4 of it (the bar of the parity tests), and
the extracted samples equal to the capture's.
"""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,pn_len,window,F", [
    (1, 1, 1, 1), (1, 255, 300, 3), (3, 7, 65, 2), (8, 255, 256, 2), (9, 256, 129, 2),
    (16, 257, 513, 5), (17, 300, 64, 1), (33, 1024, 70, 2), (64, 255, 512, 3), (40, 255, 1000, 170),
])
@pytest.mark.parametrize("fmt", ["sc16", "fc32"])
def test_detection_sizes(M, pn_len, window, F, fmt):
    import torch
    import paper_1901_07499_gb300.lsas as L
    N, cp, S = 64, 5, 3
    T = S * (N + cp)
    rng = np.random.default_rng([M, pn_len, window])
    pn = 2.0 * rng.integers(0, 2, pn_len) - 1.0
    Lc = window - 1 + pn_len + T
    lag = rng.integers(0, window, F)
    cap = 0.1 * rng.standard_normal((F, M, Lc, 2))
    if pn_len < 8:
        cap *= 0.01                       # too short to rise above the noise
    for f in range(F):
        cap[f, :, lag[f]:lag[f] + pn_len, 0] += pn
    if fmt == "sc16":
        cap = np.rint(cap * 2048.0).astype(np.int16)
    else:
        cap = cap.astype(np.float32)
    plan = L.Plan(M, N, cp, S, fmt=fmt, max_frames=F)
    plan.set_pn(pn)
    d = torch.from_numpy(cap).cuda()
    offs, peaks = plan.pn_sync(d, window)
    frames = plan.pn_extract(d, offs, backoff=0)
    plan.sync()
    offs, peaks = offs.cpu().numpy(), peaks.cpu().numpy()
    got = frames.cpu().numpy()
    for f in range(F):
        want, metric = oracle.pn_sync(oracle.to_complex(cap[f]), pn, window)
        assert offs[f] == want == lag[f]
        assert abs(peaks[f] - metric[want]) <= 1e-4 * metric[want]
        start = offs[f] + pn_len
        assert np.array_equal(got[f], cap[f, :, start:start + T])
    plan.close()


@pytest.mark.parametrize("fmt", ["sc16", "fc32"])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_extraction_alignments(fmt, shift):
    """Cuts at every offset modulo 16 bytes, into outputs at every 4-byte (8
    for fc32) offset, with the last frame ending at the capture's last
    sample; T is not a multiple of four samples."""
    import torch
    import paper_1901_07499_gb300.lsas as L
    M, N, cp, S, F = 3, 64, 5, 3, 8
    T = S * (N + cp)
    pn_len = 4
    Lc = pn_len + T + 7
    rng = np.random.default_rng(shift)
    cap = rng.integers(-3000, 3000, (F, M, Lc, 2))
    cap = cap.astype(np.int16 if fmt == "sc16" else np.float32)
    plan = L.Plan(M, N, cp, S, fmt=fmt, max_frames=F)
    plan.set_pn(np.ones(pn_len))
    d = torch.from_numpy(cap).cuda()
    offs = np.arange(F, dtype=np.int32)          # the last one ends the capture
    out = torch.zeros(F * M * T * 2 + 8, dtype=d.dtype, device="cuda")
    view = out[2 * shift:2 * shift + F * M * T * 2].view(F, M, T, 2)
    plan.pn_extract(d, torch.from_numpy(offs).cuda(), backoff=0, frames=view)
    plan.sync()
    want = np.stack([cap[f, :, offs[f] + pn_len:offs[f] + pn_len + T] for f in range(F)])
    assert np.array_equal(view.cpu().numpy(), want)
    rest = out.cpu().numpy()
    assert not rest[:2 * shift].any() and not rest[2 * shift + F * M * T * 2:].any()
    plan.close()

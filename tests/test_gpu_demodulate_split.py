"""Demodulation with a given channel on every route it can take: the
two-symbol kernels (N = 256 to 2048) and the one-symbol ones (short symbols,
few antennas, fc32, rows that are not 16-byte aligned), whole or as antenna
shards with and without a block per data-symbol group.

The oracle demodulates with the same channel (bars of parity_util).  A channel
with a row of zeros latches the device status only where no antenna is left;
a subcarrier with a non-finite channel gives z = 0 and touches no other.  A
demodulation recorded into a CUDA graph replays with the recorded call's
results.
"""

import numpy as np
import pytest

import oracle
import synth
from synth.frames import FrameConfig
from tests.parity_util import check_frame_outputs, oracle_run, to_torch_frames

pytestmark = pytest.mark.gpu

SHAPES = [  # M, N, cp, S, pilot_idx, fmt, frames
    (128, 256, 32, 8, 0, "sc16", 2),     # two-symbol teams, shards
    (32, 512, 36, 5, 2, "sc16", 3),
    (64, 1024, 72, 14, 0, "sc16", 1),    # shards and a block per group
    (64, 1024, 128, 14, 3, "sc16", 40),  # shards only
    (13, 1024, 128, 4, 1, "sc16", 2),    # odd antenna count: never split
    (128, 2048, 144, 9, 0, "sc16", 1),
    (24, 2048, 256, 2, 1, "sc16", 2),    # one data symbol
    (16, 64, 16, 15, 0, "fc32", 3),      # one-symbol kernels
    (64, 256, 18, 6, 5, "sc16", 2),      # rows not 16-byte aligned
    (64, 1024, 9, 6, 0, "sc16", 2),
    (16, 2048, 144, 5, 0, "fc32", 2),
]


@pytest.fixture(scope="module")
def L():
    import paper_1901_07499_gb300.lsas as lsas
    return lsas


def _case(shape):
    M, N, cp, S, pi, fmt, F = shape
    cfg = FrameConfig(M=M, N=N, cp=cp, S=S, Q=16, pilot_idx=pi, taps=4, decay_db=2.0, snr_db=25.0,
                      fmt=fmt, F=F, seed=71 + M + N)
    return cfg, synth.generate(cfg)


def _plan(L, cfg, b):
    return L.Plan(cfg.M, cfg.N, cfg.cp, cfg.S, cfg.pilot_idx, cfg.Q, fmt=cfg.fmt, max_frames=cfg.F,
                  pilot=b.pilot)


@pytest.mark.parametrize("split", [0, 1, 2])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "M%d_N%d_cp%d_S%d_p%d_%s_F%d" % s)
def test_given_channel(L, shape, split):
    import torch
    cfg, b = _case(shape)
    rng = np.random.default_rng(5)
    # not the estimate itself, so that an estimate made on the way would show
    H = oracle_run(cfg, b).H * (1.0 + 0.05 * rng.standard_normal((cfg.F, cfg.M, 1)))
    H = H.astype(np.complex64)
    plan = _plan(L, cfg, b)
    plan.set_batch_split(split)
    bits, eq = plan.demodulate(to_torch_frames(b), torch.from_numpy(H).cuda(), want_eq=True)
    plan.sync()
    ref = oracle_run(cfg, b, H_given=H.astype(np.complex128))
    check_frame_outputs(cfg, ref, None, bits.cpu().numpy(), eq.cpu().numpy(), check_H=False)
    plan.close()


@pytest.mark.parametrize("shape", [SHAPES[2], SHAPES[5]], ids=["N1024", "N2048"])
def test_energy_edges(L, shape):
    import torch
    cfg, b = _case(shape)
    H = oracle_run(cfg, b).H.astype(np.complex64)
    x = to_torch_frames(b)
    plan = _plan(L, cfg, b)
    good, good_eq = plan.demodulate(x, torch.from_numpy(H).cuda(), want_eq=True)
    plan.sync()
    bad = H.copy()
    bad[0, :, 5] = 0.0                    # no antenna hears subcarrier 5
    bad[0, 3, 9] = np.inf                 # one antenna's estimate is not finite
    _, eq = plan.demodulate(x, torch.from_numpy(bad).cuda(), want_eq=True)
    assert plan.sync_status() == L.LSAS_ERR_DEVICE
    eq, good_eq = eq.cpu().numpy(), good_eq.cpu().numpy()
    assert not eq[0, :, [5, 9]].any()
    keep = np.setdiff1d(np.arange(cfg.N), [5, 9])
    assert np.array_equal(eq[0][:, keep], good_eq[0][:, keep])
    assert plan.sync_status() == L.LSAS_OK
    plan.close()


def test_recorded_into_a_graph(L):
    import torch
    cfg, b = _case(SHAPES[2])
    plan = _plan(L, cfg, b)
    x, H = to_torch_frames(b), torch.from_numpy(oracle_run(cfg, b).H.astype(np.complex64)).cuda()
    assert plan.batch_split_shards(cfg.F) > 1
    want, want_eq = plan.demodulate(x, H, want_eq=True)   # split: its event has been used
    plan.sync()
    bits, eq = plan.empty_bits(cfg.F), plan.empty_eq(cfg.F)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        plan.demodulate(x, H, bits=bits, eq=eq)
    for _ in range(2):
        bits.zero_()
        eq.zero_()
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(bits, want)
    # the unsplit and the split sum over antennas differ in their order only
    assert float((eq - want_eq).abs().max()) <= 1e-5 * float(want_eq.abs().max())
    plan.close()


@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("M,cp,S,pilot_idx,F", [(1, 16, 2, 1, 1), (5, 144, 3, 0, 2), (4, 2, 8, 7, 3),
                                                (32, 144, 14, 0, 2), (9, 4, 17, 5, 1)])
def test_float_rows_n2048(L, M, cp, S, pilot_idx, F, split):
    """The two-symbol kernel on float rows: one antenna, antennas that leave
    pairs idle, even and odd numbers of items in a group, the pilot last."""
    cfg, b = _case((M, 2048, cp, S, pilot_idx, "fc32", F))
    plan = _plan(L, cfg, b)
    plan.set_batch_split(split)
    H, bits, eq = plan.run_frame(to_torch_frames(b), want_eq=True)
    plan.sync()
    ref = oracle_run(cfg, b)
    if M == 1:   # zero forcing: near a fade only H and the slicer are held
        from tests.parity_util import rel_err, unpack
        assert rel_err(H.cpu().numpy(), ref.H, axes=(1, 2)).max() <= 1e-4
        got, _ = oracle.demap(eq.cpu().numpy(), 16, dtype=np.float32)
        assert np.array_equal(got, unpack(bits.cpu().numpy(), cfg.D, cfg.N, 4))
    else:
        check_frame_outputs(cfg, ref, H.cpu().numpy(), bits.cpu().numpy(), eq.cpu().numpy())
    plan.close()

"""The work a user of liblsas has it do, as cases that can be timed and compared.

A case is a dict of plain values; ``prepare`` makes its inputs on the GPU from
a seed alone, ``run`` makes one pass through the public binding, ``exact``
gives the same outputs in 64 bits with torch only and ``work`` says what one
pass cannot do without.  Kinds of case (``case["kind"]``):

* ``frame``      received frames -> channel, bits (and z): Plan.run_frame;
* ``staged``     Plan.estimate, then Plan.demodulate with that channel (the
                 form for a user who looks at or replaces the channel);
* ``transform``  Plan.fft, then Plan.receive_y (the symbols kept in memory);
* ``detect``     captures with a PN preamble: Plan.pn_sync, Plan.pn_extract,
                 Plan.run_frame, and z in fftshift order (Sec. II-B, II-C);
* ``learned``    Plan.run_frame_refined (LS refined by the network, then MRC);
* ``train``      Denoiser.train_step: gradient and Adam, FP32 or BF16.

The host-buffer call and the serving loop run these same receiver kernels and
are bound by the host link, so their device work stands here and the link does
not.  Frames are synthetic OFDM uplink frames (Gray QAM, Rayleigh multipath,
noise), as in ``synth``, made with torch on the GPU.
"""

from __future__ import annotations

import math

import numpy as np
import torch

PN_LEN = 255
DN_MACS = 10880            # multiply-adds of the refinement network per subcarrier
DN_SHAPES = [(32, 2, 5), (32,), (32, 32, 5), (32,), (32, 32, 5), (32,), (2, 32, 5), (2,)]
DN_PARAMS = sum(int(np.prod(s)) for s in DN_SHAPES)
LR = 1e-3
MOST_SAMPLES = 1000 * 64 * 14 * 1152    # the most antenna samples a drawn batch holds


def listed():
    def rx(name, kind, F, M, N, cp, S, Q, fmt, pilot_idx=0, eq=True, **kw):
        return dict(name=name, kind=kind, F=F, M=M, N=N, cp=cp, S=S, Q=Q, fmt=fmt,
                    pilot_idx=pilot_idx, eq=eq, **kw)
    return [
        # one frame of the scale workload as it arrives: the latency call
        rx("one frame", "frame", 1, 64, 1024, 128, 14, 16, "sc16", eq=False),
        # a small array with short symbols and float samples, one radio burst
        # of frames: launches and block set-up count
        rx("tiny batch", "frame", 16, 8, 64, 16, 15, 4, "fc32"),
        # LTE 3 MHz numerology (N = 256, CP 18: rows that are not a multiple
        # of 16 bytes), an odd antenna count, the pilot inside the frame
        rx("short symbols", "frame", 200, 24, 256, 18, 14, 64, "sc16", pilot_idx=3),
        # the scale workload of bench.py: a recorded second of frames
        rx("scale batch", "frame", 1000, 64, 1024, 128, 14, 16, "sc16", eq=False),
        # the precision workload of bench.py: the largest arrays and symbols
        rx("precision batch", "frame", 500, 128, 2048, 256, 14, 64, "sc16", eq=False),
        # float samples from a front-end that already filters and resamples,
        # LTE 20 MHz numerology, 256-QAM
        rx("float samples", "frame", 60, 64, 2048, 144, 14, 256, "fc32"),
        # channel first, then demodulation with it: a batch of a serving loop
        # whose user smooths or replaces the estimate in between
        rx("estimate, demodulate", "staged", 200, 64, 1024, 128, 14, 16, "sc16"),
        # symbols kept in memory for other receivers, then LS and MRC on them
        rx("transform, receive", "transform", 120, 48, 512, 36, 14, 16, "sc16"),
        # raw captures: packet detection first, then the receiver
        rx("captures", "detect", 32, 64, 1024, 128, 14, 16, "sc16", max_delay=512),
        # the learned receiver on one serving batch
        rx("learned receiver", "learned", 16, 64, 1024, 128, 14, 16, "sc16"),
        # one optimiser step of the refinement on a training batch, both forms
        dict(name="train fp32", kind="train", R=256, N=1024, tc=False),
        dict(name="train bf16", kind="train", R=256, N=1024, tc=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "staged", "transform", "detect",
                       "learned", "train", "train"])
    if kind == "train":
        N = 128 * rng.randint(1, 16)
        return dict(kind=kind, R=_log_int(rng, 8, (256 * 1024) // N), N=N, tc=rng.random() < 0.5)
    fmt = rng.choice(["sc16", "sc16", "sc16", "fc32"])
    N = rng.choice([64, 128, 256, 512, 1024, 1024, 2048])
    if kind == "learned":
        fmt, N = "sc16", 1024
    M = _log_int(rng, 4, 160)
    # N/8 (the sweep), LTE's 9/128 N, or any length up to N/4
    cp = rng.choice([N // 8, N // 8, max(4, 9 * N // 128), rng.randint(4, N // 4)])
    S = rng.choice([14, 14, 15, 7, rng.randint(2, 20)])
    case = dict(kind=kind, M=M, N=N, cp=cp, S=S, Q=rng.choice([2, 4, 16, 16, 64, 256]), fmt=fmt,
                pilot_idx=rng.choice([0, 0, rng.randrange(S)]), eq=rng.random() < 0.5)
    if kind == "detect":
        case["max_delay"] = rng.randint(100, 1000)
    if kind in ("detect", "learned", "transform"):
        case["eq"] = True
    per_frame = M * (S * (N + cp) + 8 * case.get("max_delay", 0))
    if kind == "learned":
        per_frame = M * N * max(S, 16)
    most = {"frame": MOST_SAMPLES, "staged": MOST_SAMPLES // 4, "transform": MOST_SAMPLES // 8,
            "detect": MOST_SAMPLES // 16, "learned": MOST_SAMPLES // 16}[kind]
    case["F"] = _log_int(rng, 1, max(1, min(1000, most // per_frame)))
    return case


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)


def _crandn(g, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda") * math.sqrt(0.5))


def _pilot(case, seed):
    rng = np.random.default_rng([int(seed), case["N"], 1])
    return (2.0 * rng.integers(0, 2, size=case["N"]) - 1.0).astype(np.complex128)


def _chips():
    """The degree-8 m-sequence (x^8 + x^4 + x^3 + x^2 + 1) as +-1 chips."""
    a = [1] + [0] * 7
    for n in range(PN_LEN - 8):
        a.append(a[n + 4] ^ a[n + 3] ^ a[n + 2] ^ a[n])
    return 1.0 - 2.0 * np.array(a, dtype=np.float64)


def _qam(g, Q, *shape):
    L = 2 if Q == 2 else int(round(math.sqrt(Q)))
    A = 1.0 if Q == 2 else 1.0 / math.sqrt(2.0 * (Q - 1) / 3.0)
    re = (2 * torch.randint(0, L, shape, generator=g, device="cuda") - (L - 1)) * A
    if Q == 2:
        return torch.complex(re.float(), torch.zeros_like(re, dtype=torch.float32))
    im = (2 * torch.randint(0, L, shape, generator=g, device="cuda") - (L - 1)) * A
    return torch.complex(re.float(), im.float())


def _received(case, seed):
    """Frames [F][M][S(N+CP)][2], or captures [F][M][Lc][2] with a preamble
    at a random delay, after the channel, at 20 to 30 dB per antenna."""
    F, M, N, cp, S, Q = (case[k] for k in ("F", "M", "N", "cp", "S", "Q"))
    capture = "max_delay" in case
    T = S * (N + cp)
    Lc = T + (case["max_delay"] + PN_LEN if capture else 0)
    taps = min(8, cp + 1)
    g = _gen(seed)
    pdp = 10.0 ** (-0.2 * np.arange(taps))
    amp = torch.from_numpy(np.sqrt(pdp / pdp.sum())).float().cuda()
    pilot = torch.from_numpy(_pilot(case, seed)).to(torch.complex64).cuda()
    out = torch.empty((F, M, Lc, 2), device="cuda",
                      dtype=torch.int16 if case["fmt"] == "sc16" else torch.float32)
    delays = np.random.default_rng([int(seed), 2]).integers(0, case["max_delay"], F) if capture else None
    step = max(1, (1 << 26) // (M * Lc))
    for f0 in range(0, F, step):
        n = min(step, F - f0)
        X = _qam(g, Q, n, S, N)
        X[:, case["pilot_idx"]] = pilot
        x = torch.fft.ifft(X) * math.sqrt(N)
        x = torch.cat([x[..., N - cp:], x], -1).reshape(n, T)
        if capture:
            s = torch.zeros((n, Lc), dtype=torch.complex64, device="cuda")
            pn = torch.from_numpy(_chips()).to(torch.complex64).cuda()
            for i in range(n):
                d = int(delays[f0 + i])
                s[i, d:d + PN_LEN] = pn
                s[i, d + PN_LEN:d + PN_LEN + T] = x[i]
            x = s
        paths = torch.zeros((n, taps, Lc), dtype=torch.complex64, device="cuda")
        for l in range(taps):
            paths[:, l, l:] = x[:, :Lc - l]
        y = (_crandn(g, n, M, taps) * amp) @ paths
        snr = 20.0 + 10.0 * torch.rand((n, 1, 1), generator=g, device="cuda")
        y += _crandn(g, n, M, Lc) * 10.0 ** (-snr / 20.0)
        if case["fmt"] == "sc16":
            r = torch.view_as_real(y)
            gain = 2048.0 / torch.sqrt(r.square().sum(-1).mean((1, 2), keepdim=True))[..., None]
            out[f0:f0 + n] = torch.round(r * gain).clamp(-32767, 32767).to(torch.int16)
        else:
            out[f0:f0 + n] = torch.view_as_real(y)
    return out


def _weights(seed):
    """Network weights as a training run starts with them (He, small last
    layer), the biases away from zero as after a few steps."""
    rng = np.random.default_rng([int(seed), 3])
    parts = []
    for i, s in enumerate(DN_SHAPES):
        if len(s) == 1:
            parts.append(0.02 * rng.standard_normal(s))
        else:
            parts.append(rng.standard_normal(s) * math.sqrt(2.0 / (s[1] * s[2])) * (0.1 if i == 6 else 1.0))
    return np.concatenate([p.reshape(-1) for p in parts]).astype(np.float32)


def _pairs(case, seed):
    """True channel rows and their LS estimates, [R][N] complex64 (4 to 16
    taps, 0 to 30 dB)."""
    R, N = case["R"], case["N"]
    g = _gen(seed)
    n_taps = torch.randint(4, 17, (R, 1), generator=g, device="cuda")
    decay = 1.0 + 2.0 * torch.rand((R, 1), generator=g, device="cuda")
    l = torch.arange(16, device="cuda")[None]
    p = torch.where(l < n_taps, 10.0 ** (-decay * l / 10.0), torch.zeros((), device="cuda"))
    h = _crandn(g, R, 16) * torch.sqrt(p / p.sum(1, keepdim=True))
    Ht = torch.fft.fft(h, N)
    snr = 30.0 * torch.rand((R, 1), generator=g, device="cuda")
    return Ht.contiguous(), (Ht + _crandn(g, R, N) * 10.0 ** (-snr / 20.0)).contiguous()


# ---------------------------------------------------------------- one pass

def prepare(case, seed):
    import paper_1901_07499_gb300.denoiser as denoiser
    import paper_1901_07499_gb300.lsas as lsas
    if case["kind"] == "train":
        Ht, Hls = _pairs(case, seed)
        dn = denoiser.Denoiser(_weights(seed))
        dn.work(case["R"], case["N"])
        return dict(case=case, dn=dn, Ht=Ht, Hls=Hls)
    F = case["F"]
    plan = lsas.Plan(case["M"], case["N"], case["cp"], case["S"], case["pilot_idx"], case["Q"],
                     fmt=case["fmt"], max_frames=F, pilot=_pilot(case, seed))
    s = dict(case=case, plan=plan, x=_received(case, seed), H=plan.empty_H(F),
             bits=plan.empty_bits(F), eq=plan.empty_eq(F) if case["eq"] else None)
    if case["kind"] == "transform":
        s["Y"] = torch.empty((F, case["M"], case["S"], case["N"]), dtype=torch.complex64, device="cuda")
    elif case["kind"] == "detect":
        plan.set_pn(_chips())
        s["frames"] = torch.empty((F, case["M"], case["S"] * (case["N"] + case["cp"]), 2),
                                  dtype=s["x"].dtype, device="cuda")
        s["offsets"] = torch.empty(F, dtype=torch.int32, device="cuda")
        s["peaks"] = torch.empty(F, dtype=torch.float32, device="cuda")
        s["SHIFT_EQ"] = lsas.LSAS_SHIFT_EQ
    elif case["kind"] == "learned":
        dn = denoiser.Denoiser(_weights(seed))
        s.update(dn=dn, params=dn.bf16_params(), work=dn.work(F * case["M"], case["N"]),
                 status=dn.status())
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "train":
        dn = s["dn"]
        loss = dn.train_step(s["Hls"], s["Ht"], LR, tensor_cores=case["tc"])
        return dict(loss=loss, grad=dn.grad, params=dn.params, m=dn.m, v=dn.v)
    plan, x, H, bits, eq = s["plan"], s["x"], s["H"], s["bits"], s["eq"]
    out = dict(H=H, bits=bits)
    if eq is not None:
        out["eq"] = eq
    if kind == "frame":
        plan.run_frame(x, H=H, bits=bits, eq=eq)
    elif kind == "staged":
        plan.estimate(x, H=H)
        plan.demodulate(x, H, bits=bits, eq=eq)
    elif kind == "transform":
        out["Y"] = plan.fft(x, Y=s["Y"])
        plan.receive_y(s["Y"], H=H, bits=bits, eq=eq)
    elif kind == "detect":
        out["offsets"], out["peaks"] = plan.pn_sync(x, case["max_delay"], offsets=s["offsets"],
                                                    peaks=s["peaks"])
        out["frames"] = plan.pn_extract(x, s["offsets"], backoff=case["cp"] // 4, frames=s["frames"])
        plan.run_frame(s["frames"], H=H, bits=bits, eq=eq)
        plan.fftshift(s["SHIFT_EQ"], eq)
    elif kind == "learned":
        plan.run_frame_refined(x, s["params"], s["work"], s["status"], H=H, bits=bits, eq=eq)
    else:
        raise ValueError(kind)
    return out


def work(case):
    if case["kind"] == "train":
        # rows in, parameters and both moments in and out, the gradient out;
        # forward, weight gradients, and data gradients of all but layer 1
        n = case["R"] * case["N"]
        return dict(bytes=16 * n + 7 * 4 * DN_PARAMS, flops=2 * n * (3 * DN_MACS - 320))
    F, M, N, S, Q = (case[k] for k in ("F", "M", "N", "S", "Q"))
    D = S - 1
    bps = 4 if case["fmt"] == "sc16" else 8
    # the samples after the cyclic prefixes in; H, the packed bits and z out
    nbytes = M * S * N * bps + M * N * 8 + D * N * int(round(math.log2(Q))) // 8
    nbytes += D * N * 8 if case["eq"] else 0
    flops = M * S * 5 * N * math.log2(N) + 9 * M * N + 8 * M * D * N
    if case["kind"] == "transform":
        nbytes += M * S * N * 8
    elif case["kind"] == "detect":
        nbytes += M * (case["max_delay"] + PN_LEN - 1) * bps + M * S * (N + case["cp"]) * bps
        flops += M * case["max_delay"] * (4 * PN_LEN + 4)
    elif case["kind"] == "learned":
        nbytes += DN_PARAMS * 2 / F
        flops += 2 * M * N * DN_MACS
    return dict(bytes=F * nbytes, flops=F * flops)


# ---------------------------------------------------------------- in 64 bits

def _blocks(p):
    out, o = [], 0
    for s in DN_SHAPES:
        n = int(np.prod(s))
        out.append(p[o:o + n].view(*s))
        o += n
    return out


def _network(p, x0):
    w = _blocks(p)
    a = x0
    for i in range(4):
        # a convolution over subcarriers as five shifted products
        W, N = w[2 * i], a.shape[-1]
        pad = torch.nn.functional.pad(a, (2, 2))
        a = sum(torch.einsum("oc,rcn->ron", W[:, :, k], pad[..., k:k + N]) for k in range(5))
        a = a + w[2 * i + 1][:, None]
        if i < 3:
            a = torch.relu(a)
    return x0 + a


def _split(H, rms):
    return torch.stack([H.real, H.imag], 1) / rms[:, None, None]


def _rms(H):
    return H.abs().square().mean(-1).sqrt()


def _symbols(case, x):
    y = torch.view_as_complex(x.double()).reshape(x.shape[0], case["M"], case["S"], case["N"] + case["cp"])
    return torch.fft.fft(y[..., case["cp"]:]) / math.sqrt(case["N"])


def exact(case, seed):
    if case["kind"] == "train":
        Ht, Hls = _pairs(case, seed)
        Ht, Hls = Ht.to(torch.complex128), Hls.to(torch.complex128)
        p32 = torch.from_numpy(_weights(seed)).cuda()
        used = p32.bfloat16().double() if case["tc"] else p32.double()
        used.requires_grad_(True)
        rms = _rms(Hls)
        err = _network(used, _split(Hls, rms)) - _split(Ht, rms)
        loss = err.square().mean()
        loss.backward()
        grad = used.grad
        m, v = 0.1 * grad, 0.001 * grad.square()
        params = p32.double() - LR * grad / (grad.abs() + 1e-8)
        return dict(loss=loss.detach().reshape(1), grad=grad, params=params, m=m, v=v)
    F, M, N, S = (case[k] for k in ("F", "M", "N", "S"))
    x = _received(case, seed)
    pilot = torch.from_numpy(_pilot(case, seed)).cuda()
    c128 = dict(dtype=torch.complex128, device="cuda")
    H = torch.empty((F, M, N), **c128)
    eq = torch.empty((F, S - 1, N), **c128) if case["eq"] else None
    Y = torch.empty((F, M, S, N), **c128) if case["kind"] == "transform" else None
    peaks = torch.empty(F, dtype=torch.float64, device="cuda") if case["kind"] == "detect" else None
    data = [s for s in range(S) if s != case["pilot_idx"]]
    if case["kind"] == "learned":
        p = torch.from_numpy(_weights(seed)).cuda().bfloat16().double()
    step = max(1, (1 << 25) // (M * S * (N + case["cp"])))
    T = S * (N + case["cp"])
    for f0 in range(0, F, step):
        at = slice(f0, min(F, f0 + step))
        rows = x[at]
        if peaks is not None:
            chips = torch.from_numpy(_chips()).cuda()
            cut = []
            for i, cap in enumerate(torch.view_as_complex(rows.double())):
                seen = cap[:, :case["max_delay"] + PN_LEN - 1].unfold(-1, PN_LEN, 1)
                metric = (torch.view_as_real(seen).transpose(-1, -2) @ chips).square().sum((0, 2))
                d = int(metric.argmax())
                peaks[f0 + i] = metric[d]
                begin = d + PN_LEN - case["cp"] // 4
                cut.append(rows[i, :, begin:begin + T])
            rows = torch.stack(cut)
        y = _symbols(case, rows)
        h = y[:, :, case["pilot_idx"]] * (pilot.conj() / pilot.abs().square())
        if case["kind"] == "learned":
            flat = h.reshape(-1, N)
            rms = _rms(flat)
            o = _network(p, _split(flat, rms)) * rms[:, None, None]
            h = torch.complex(o[:, 0], o[:, 1]).reshape(h.shape)
        H[at] = h
        if Y is not None:
            Y[at] = y
        if eq is not None:
            z = (h.conj()[:, :, None] * y[:, :, data]).sum(1) / h.abs().square().sum(1)[:, None]
            eq[at] = torch.fft.fftshift(z, dim=-1) if peaks is not None else z
    out = dict(H=H, bits=None)
    if eq is not None:
        out["eq"] = eq
    if Y is not None:
        out["Y"] = Y
    if peaks is not None:
        out.update(offsets=None, peaks=peaks, frames=None)
    return out

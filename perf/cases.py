"""Performance cases of the receiver library: what its users have it do.

Every case goes through the package's public classes (`Receiver`, `Batch`, `CNN`,
`KKFrontEnd`, `WLEqualiser`) the way a program calls them.  `listed()` names the
cases, `draw()` gives more of the same ranges, `prepare()` makes the seeded inputs
and the handles a program keeps, `run()` is one pass, `work()` the bytes and
operations a pass cannot do without, and `exact()` the outputs in 64 bits, stated
with torch and numpy alone.

Inputs are synthetic links made on the GPU: Gray QPSK / 16QAM, root-raised-cosine
shaping, whole-stream dispersion, a Jones rotation with differential group delay,
laser phase noise, a frequency offset, additive noise and an 8-bit ADC; for the
Kramers-Kronig receiver one polarisation plus a carrier tone, square-law detected.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2104_06311_gb300 import CNN, Batch, KKFrontEnd, Receiver, WLEqualiser

C_LIGHT = 299_792_458.0
LAM = 1550e-9
TWO_PI = 2.0 * math.pi

# Receiver and batch defaults that the 64-bit statement needs.
N_CMA, ACQ, BU, SEG, PRE, WAVE_SEGS, NTAPS, ANGLES, MU = 8192, 16384, 32, 1024, 128, 32, 15, 32, 1e-3


def listed():
    return [
        # One short recording of a metro link, float samples, soft symbols kept for a
        # plot: the smallest call, where launches and the acquisition's chain count.
        dict(name="chain_qpsk_64k", kind="chain", mod=2, baud=10e9, L_km=1000.0, n_sym=1 << 16, snr=12.0, adc=0,
             fo=0.0, lw=0.0, track=1, prec=0, llr=0, sym=1, chunk=0, ber=0),
        # The long-haul headline: 10,000 km, 2^24 symbols, phase noise and offset, hard
        # bits and their error count.
        dict(name="chain_qpsk_16m_ber", kind="chain", mod=2, baud=10e9, L_km=10000.0, n_sym=1 << 24, snr=9.8, adc=1,
             fo=200e6, lw=100e3, track=1, prec=0, llr=0, sym=0, chunk=0, ber=1),
        # High-rate 16QAM feeding a soft-decision decoder: FP32 LLRs, N = 16384 windows.
        dict(name="chain_16qam_1m_llr", kind="chain", mod=4, baud=32e9, L_km=6000.0, n_sym=1 << 20, snr=18.0, adc=1,
             fo=0.0, lw=100e3, track=1, prec=0, llr=1, sym=0, chunk=0, ber=0),
        # The same link in the FP16 form with FP16 LLRs, a recording of odd length.
        dict(name="chain_16qam_fp16_700k", kind="chain", mod=4, baud=32e9, L_km=3000.0, n_sym=700001, snr=18.0, adc=1,
             fo=0.0, lw=100e3, track=0, prec=1, llr=2, sym=0, chunk=0, ber=0),
        # A stream arriving in buffers of ragged size, state carried from call to call.
        dict(name="chain_qpsk_stream", kind="chain", mod=2, baud=10e9, L_km=2400.0, n_sym=1300000, snr=11.0, adc=1,
             fo=120e6, lw=100e3, track=1, prec=0, llr=0, sym=1, chunk=300000, ber=0),
        # A line card: 64 WDM channels of uneven length, rate, dispersion and format.
        dict(name="batch_64ch", kind="batch", n_ch=64, lo=17.0, hi=20.0, llr=0, sym=0),
        # A few short channels with LLRs, as a monitoring tap takes them.
        dict(name="batch_6ch_llr", kind="batch", n_ch=6, lo=15.0, hi=17.0, llr=1, sym=0),
        # Inference of the learned post-equaliser on one training-length sequence and on
        # the long sequences of a whole recording.
        dict(name="cnn_apply_16k", kind="cnn", n_sym=1 << 14, grads=0, layers=4),
        dict(name="cnn_apply_1m", kind="cnn", n_sym=1 << 20, grads=0, layers=4),
        # Forward and backward over one training sequence.
        dict(name="cnn_grads_16k", kind="cnn", n_sym=1 << 14, grads=1, layers=4),
        # The Kramers-Kronig front end alone on float samples, field kept.
        dict(name="kk_field_1m", kind="kk", mod=4, L_km=1000.0, n_buf=1, samples=1 << 20, adc=0, field=1, eq=0),
        # The paper's own chain over four of its 2^22-sample ADC buffers: front end on one
        # stream, widely-linear equaliser on another.
        dict(name="kk_chain_4x4m", kind="kk", mod=4, L_km=5600.0, n_buf=4, samples=1 << 22, adc=1, field=0, eq=1),
    ]


def draw(rng):
    def log2(lo, hi):
        return int(round(2.0 ** rng.uniform(lo, hi)))

    kind = rng.choice(["chain", "chain", "chain", "batch", "cnn", "cnn", "kk", "kk"])
    if kind == "chain":
        mod = rng.choice([2, 4])
        n_sym = log2(15.1, 22.0)
        prec = rng.choice([0, 0, 0, 1, 2])
        return dict(kind="chain", mod=mod, baud=rng.uniform(10e9, 32e9), L_km=rng.uniform(200.0, 6000.0), n_sym=n_sym,
                    snr=rng.uniform(10.0, 14.0) if mod == 2 else rng.uniform(18.0, 22.0), adc=rng.choice([0, 1, 1]),
                    fo=rng.choice([0.0, 100e6]) if mod == 2 else 0.0, lw=100e3, track=1 if mod == 2 else rng.choice([0, 1]), prec=prec, llr=rng.choice([0, 1, 2]),
                    sym=rng.choice([0, 1]), chunk=rng.choice([0, 0, max(70000, n_sym // 2 * 2 // 3 * 2)]), ber=0)
    if kind == "batch":
        hi = rng.uniform(16.0, 19.0)
        return dict(kind="batch", n_ch=log2(1.0, 6.0), lo=15.0, hi=hi, llr=rng.choice([0, 1]), sym=rng.choice([0, 1]))
    if kind == "cnn":
        grads = rng.choice([0, 1])
        return dict(kind="cnn", n_sym=log2(10.0, 20.0 if not grads else 18.0), grads=grads, layers=rng.choice([3, 4, 4, 5]))
    eq = rng.choice([0, 1])
    return dict(kind="kk", mod=rng.choice([2, 4]), L_km=rng.uniform(200.0, 5600.0), n_buf=rng.choice([1, 2, 3]),
                samples=512 * max(64, log2(6.0, 13.0)), adc=rng.choice([0, 1]), field=1 - eq, eq=eq)


# ----------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _qam(mod, shape, g):
    """(symbols, bits [..., mod]) of the Gray maps, unit mean energy."""
    b = torch.randint(0, 2, (*shape, mod), generator=g, device="cuda", dtype=torch.int8)
    s = (1 - 2 * b).double()
    if mod == 2:
        return torch.complex(s[..., 0], s[..., 1]) / math.sqrt(2.0), b
    return torch.complex(s[..., 0] * (1 + 2 * b[..., 1]), s[..., 2] * (1 + 2 * b[..., 3])) / math.sqrt(10.0), b


def _freqs(n, fs):
    return torch.fft.fftfreq(n, 1.0 / fs, dtype=torch.float64, device="cuda")


def _beta2(D=17.0):
    return -(D * 1e-6) * LAM * LAM / (TWO_PI * C_LIGHT)


def _rrc(f, baud, roll):
    af = f.abs()
    f1, f2 = (1 - roll) * baud / 2, (1 + roll) * baud / 2
    return torch.where(af <= f1, 1.0, torch.where(af <= f2, torch.cos(math.pi * (af - f1) / (2 * roll * baud)), 0.0))


def _cis(phase):
    phase = torch.remainder(phase, TWO_PI)
    return torch.complex(torch.cos(phase), torch.sin(phase))


def _dual_pol_link(mod, baud, L_km, n_sym, snr, adc, fo, lw, seed, jones):
    """(samples (n, 4) int8 / float32, in_scale, reference bit words)."""
    g = _gen(seed)
    s, bits = _qam(mod, (2, n_sym), g)
    n, fs = 2 * n_sym, 2 * baud
    f = _freqs(n, fs)
    up = torch.zeros(2, n, dtype=torch.complex64, device="cuda")
    up[:, ::2] = s.to(torch.complex64)
    del s
    H = math.sqrt(2.0) * _rrc(f, baud, 0.1) * _cis(0.5 * _beta2() * L_km * 1e3 * (TWO_PI * f) ** 2)
    X = torch.fft.fft(up) * H.to(torch.complex64)
    th, psi = jones
    c, sn, e = math.cos(th), math.sin(th), complex(math.cos(psi), math.sin(psi))
    tau = 0.1e-12 * math.sqrt(L_km)      # differential group delay of 0.1 ps/sqrt(km)
    d = _cis(TWO_PI * f * tau / 2).to(torch.complex64)
    X = torch.stack([(c * X[0] - sn * e.conjugate() * X[1]) * d, (sn * e * X[0] + c * X[1]) * d.conj()])
    x = torch.fft.ifft(X)
    del X, up, H, d
    turns = torch.arange(n, device="cuda", dtype=torch.float64) * (fo / fs)
    if lw > 0:
        # a Wiener phase in whole 2^-40 turns, so that its running sum is exact
        step = torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * (math.sqrt(TWO_PI * lw / fs) / TWO_PI)
        turns += torch.cumsum(torch.round(step * 2.0 ** 40).to(torch.int64), 0).double() * 2.0 ** -40
    x *= _cis(TWO_PI * torch.remainder(turns, 1.0)).to(torch.complex64)
    del turns
    x += math.sqrt(0.5 * 10 ** (-snr / 10)) * torch.view_as_complex(torch.randn(2, n, 2, generator=g, device="cuda"))
    il = torch.view_as_real(x).permute(1, 0, 2).reshape(n, 4).contiguous()
    scale = 1.0
    if adc:
        scale = 4.0 * float(il[:1 << 16].double().square().mean().sqrt()) / 127.0
        il = torch.clamp(torch.round(il / scale), -128, 127).to(torch.int8)
    flat = bits.reshape(2, -1)
    pad = -flat.shape[1] % 32
    flat = torch.nn.functional.pad(flat, (0, pad)).reshape(2, -1, 32).to(torch.int64)
    words = (flat << torch.arange(32, device="cuda")).sum(-1)
    return il, scale, torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)


def _kk_link(case, seed):
    """(samples (n,) int8 / float32, scale, offset): square-law detected, one polarisation."""
    g = _gen(seed)
    n = case["samples"] * case["n_buf"]
    baud, fs = 1e9, 4e9
    s, _ = _qam(case["mod"], (n // 4,), g)
    up = torch.zeros(n, dtype=torch.complex128, device="cuda")
    up[::4] = s
    f = _freqs(n, fs)
    S = torch.fft.fft(up) * (2.0 * _rrc(f, baud, 0.01))
    sig = torch.fft.ifft(S)
    p_s = float(sig.abs().square().mean())
    t = torch.arange(n, dtype=torch.float64, device="cuda")
    sig = sig + math.sqrt(p_s * 10 ** 1.2) * _cis(TWO_PI * torch.remainder(_carrier(case) / fs * t, 1.0))
    E = torch.fft.ifft(torch.fft.fft(sig) * _cis(0.5 * _beta2() * case["L_km"] * 1e3 * (TWO_PI * f) ** 2))
    E += math.sqrt(0.5 * p_s * 10 ** -2.4) * torch.view_as_complex(
        torch.randn(n, 2, generator=g, device="cuda", dtype=torch.float64))
    inten = E.abs().square()
    if not case["adc"]:
        return inten.float(), 1.0, 0.0
    step = float(inten[:1 << 16].max()) * 1.25 / 255.0
    return (torch.clamp(torch.round(inten / step), 0, 255) - 128).to(torch.int8), step, 128.0


def _carrier(case):
    """0.516 GHz moved to the recording's frequency grid (its dispersion is circular)."""
    n = case["samples"] * case["n_buf"]
    return round(0.516e9 / 4e9 * n) * 4e9 / n


def _batch_channels(case, seed):
    """Channel settings of a batch: drawn once from the case, not from the seed."""
    r = np.random.default_rng(int(case["n_ch"] * 1000 + round(case["lo"] * 10) + round(case["hi"] * 100)))
    out = []
    for ch in range(case["n_ch"]):
        q = 1 << 11
        n_sym = max(1 << 15, int(round(2.0 ** r.uniform(case["lo"], case["hi"]) / q)) * q + int(r.integers(0, 3)) * 7)
        c = dict(baud=float(r.uniform(10e9, 32e9)), L_km=float(r.uniform(500.0, 6000.0)), n_sym=n_sym,
                 mod=4 if r.uniform() < 0.5 else 2, jones=(float(r.uniform(0, math.pi)), float(r.uniform(0, TWO_PI))),
                 seed=int(seed) * 4099 + ch)
        c["snr"] = float(r.uniform(11.0, 16.0) if c["mod"] == 2 else r.uniform(18.0, 22.0))
        c["V"] = _overlap(c["baud"], c["L_km"])
        c["N"] = _fft_n(c["V"])
        out.append(c)
    return out


def _columns(key, chans):
    """Columns of each channel's output rows: its symbols plus a margin, in whole 64s."""
    per = {"bits": lambda c: (c["n_sym"] + 32) * c["mod"] / 32, "llr": lambda c: (c["n_sym"] + 32) * c["mod"],
           "sym": lambda c: c["n_sym"] + 32}[key]
    return [64 * int(math.ceil(per(c) / 64)) for c in chans]


def _overlap(baud, L_km):
    T = 1.0 / (2 * baud)
    ncd = 2 * int(math.floor(17e-6 * LAM * LAM * L_km * 1e3 / (2 * C_LIGHT * T * T))) + 1
    return -(-(ncd - 1) // 32) * 32


def _fft_n(V):
    N = 1024
    while N < 4 * V and N < 16384:
        N *= 2
    return N


def _cnn_params(seed, layers):
    r = np.random.default_rng(int(seed) + 99)
    dims = [4] + [64] * (layers - 1) + [4]
    out = []
    for l in range(layers):
        W = r.standard_normal((15, dims[l], dims[l + 1])) * math.sqrt(2.0 / (15 * dims[l]))
        if l == layers - 1:
            W *= 0.1
        out.append((W, r.standard_normal(dims[l + 1]) * 0.01))
    return out


def _cnn_data(case, seed):
    """Received symbols with a Kerr-like distortion and noise, and the sent ones."""
    g = _gen(seed)
    t, _ = _qam(4, (2, case["n_sym"]), g)
    p = t.abs().square().sum(0)
    z = t * _cis(0.1 * (p + torch.roll(p, 1) - 2.0))
    z = z + 0.1 * torch.view_as_complex(torch.randn(2, case["n_sym"], 2, generator=g, device="cuda", dtype=torch.float64))
    return z.to(torch.complex64), t.to(torch.complex64)


# --------------------------------------------------------------------- the calls

def prepare(case, seed):
    kind = case["kind"]
    if kind == "chain":
        x, scale, ref = _dual_pol_link(case["mod"], case["baud"], case["L_km"], case["n_sym"], case["snr"], case["adc"],
                                       case["fo"], case["lw"], seed, (0.7, 1.9))
        rx = Receiver(case["baud"], case["L_km"], MOD=case["mod"], IN_SCALE=scale, PRECISION=case["prec"],
                      LLR_OUT=case["llr"], SYM_OUT=case["sym"], FO_TRACK=case["track"])
        rx.reserve(case["chunk"] or x.shape[0])
        out = rx.alloc_out(case["n_sym"] + 64 + (2 << 16 if case["chunk"] else 0), llr=bool(case["llr"]), sym=bool(case["sym"]))
        return dict(case=case, x=x, rx=rx, out=out, ref=ref if case["ber"] else None)
    if kind == "batch":
        chans = _batch_channels(case, seed)
        xs, cfgs = [], []
        for c in chans:
            x, scale, _ = _dual_pol_link(c["mod"], c["baud"], c["L_km"], c["n_sym"], c["snr"], 1, 0.0, 0.0, c["seed"], c["jones"])
            xs.append(x)
            # no offset or phase noise on these channels: tracking off, a longer BPS window
            # for 16QAM; the FFT size given, so that every run takes the same one
            cfgs.append(dict(baud=c["baud"], L_km=c["L_km"], in_scale=scale, max_samples=x.shape[0], mod_bits=c["mod"],
                             fft_n=c["N"], flags=1, bps_halfwin=64 if c["mod"] == 4 else 16))
        b = Batch(cfgs)
        # the channels' outputs one after another in one buffer of each kind
        outs, flat = [dict(capacity=c["n_sym"] + 32) for c in chans], {}
        kinds = [("bits", torch.int32), ("llr", torch.float32), ("sym", torch.complex64)]
        for key, dtype in kinds[:1] + [k for k in kinds[1:] if case[k[0]]]:
            flat[key] = torch.zeros(sum(2 * w for w in _columns(key, chans)), dtype=dtype, device="cuda")
            for o, part in zip(outs, flat[key].split([2 * w for w in _columns(key, chans)])):
                o[key] = part.view(2, -1)
        return dict(case=case, xs=xs, b=b, outs=outs, flat=flat)
    if kind == "cnn":
        z, t = _cnn_data(case, seed)
        net = CNN(case["n_sym"], layers=case["layers"])
        net.set_params(_cnn_params(seed, case["layers"]))
        return dict(case=case, z=z, t=t, net=net, out=torch.empty_like(z))
    x, scale, offset = _kk_link(case, seed)
    s_fe, s_eq = torch.cuda.Stream(), torch.cuda.Stream()
    n = case["samples"]
    st = dict(case=case, x=x.view(case["n_buf"], n), scale=scale, offset=offset, s_fe=s_fe, s_eq=s_eq,
              y=torch.empty(case["n_buf"], n // 2, dtype=torch.complex64, device="cuda"),
              ev=[torch.cuda.Event() for _ in range(case["n_buf"])],
              fe=KKFrontEnd(1e9, _carrier(case), case["L_km"], n, stream=s_fe if case["eq"] else None))
    if case["eq"]:
        st["eq"] = WLEqualiser(case["mod"], n // 4, stream=s_eq)
        words = n // 4 * case["mod"] // 32
        st["bits"] = torch.empty(case["n_buf"], words, dtype=torch.int32, device="cuda")
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "chain":
        rx = st["rx"]
        out = rx.run_stream(st["x"], chunk=case["chunk"] or None, out=st["out"])
        K = out["n"]
        got = {"bits": out["bits"][:, :-(-K * case["mod"] // 32)]}
        if "llr" in out:
            got["llr"] = out["llr"][:, :K * case["mod"]]
        if "sym" in out:
            got["sym"] = out["sym"][:, :K]
        if case["ber"]:
            got["ber"] = rx.ber(out["bits"], st["ref"], K)
        return got
    if kind == "batch":
        st["b"].process(st["xs"], st["outs"])
        return st["flat"]
    if kind == "cnn":
        if case["grads"]:
            loss, g = st["net"].grads(st["z"], st["t"])
            return {"loss": loss, "grads": g}
        return {"y": st["net"].apply(st["z"], out=st["out"])}
    fe = st["fe"]
    fe.set_position(0)
    if not case["eq"]:
        ys, fields = [], []
        for i in range(case["n_buf"]):
            y, f = fe.process(st["x"][i], st["scale"], st["offset"], field=True, out=st["y"][i])
            fields.append(f)
        y, f = fe.flush(field=True)
        return {"y": st["y"], "y_end": y, "field": fields, "field_end": f}
    eq, main = st["eq"], torch.cuda.current_stream()
    st["s_fe"].wait_stream(main)
    st["s_eq"].wait_stream(main)
    eq.reset()
    zs = []
    for i in range(case["n_buf"]):
        fe.process(st["x"][i], st["scale"], st["offset"], out=st["y"][i])
        st["ev"][i].record(st["s_fe"])
        st["s_eq"].wait_event(st["ev"][i])
        eq.process(st["y"][i], bits=st["bits"][i])
    main.wait_stream(st["s_fe"])
    main.wait_stream(st["s_eq"])
    return {"bits": st["bits"], "y": st["y"]}


def work(case):
    kind = case["kind"]
    if kind == "chain":
        return _chain_work(case["n_sym"], case["mod"], case["baud"], case["L_km"], 4 if case["adc"] else 16,
                           {0: 0, 1: 4, 2: 2}[case["llr"]], case["sym"])
    if kind == "batch":
        w = [_chain_work(c["n_sym"], c["mod"], c["baud"], c["L_km"], 4, 4 * case["llr"], case["sym"])
             for c in _batch_channels(case, 0)]
        return {k: sum(v[k] for v in w) for k in ("bytes", "flops")}
    if kind == "cnn":
        K, L = case["n_sym"], case["layers"]
        per = 2 * 15 * (2 * 4 * 64 + (L - 2) * 64 * 64)
        weights = 4 * (15 * (2 * 4 * 64 + (L - 2) * 64 * 64) + 64 * (L - 1) + 4)
        if case["grads"]:
            return {"bytes": 32.0 * K + 2 * weights, "flops": float(K) * (3 * per - 2 * 15 * 4 * 64)}
        return {"bytes": 32.0 * K + weights, "flops": float(K) * per}
    n = float(case["samples"] * case["n_buf"])
    # two transform pairs of 1024 points at half overlap (the last one of 512 points)
    flops = n * (2 * (2 * 5 * 10) + 2 * (5 * 10 + 0.5 * 5 * 9) + 40)
    size = n * (1 if case["adc"] else 4) + n / 2 * 8
    if case["eq"]:
        flops += n / 4 * 1.5 * 4 * 4 * 8
        size += n / 4 * case["mod"] / 8
    else:
        size += n * 8
    return {"bytes": size, "flops": flops}


def _chain_work(K, mod, baud, L_km, in_bytes, llr_bytes, sym):
    V = _overlap(baud, L_km)
    N = _fft_n(V)
    n = 2.0 * K
    flops = n * (2 * (10 * math.log2(N) + 6) * N / (N - V) + 480 * (1 + PRE / SEG)) + 2.0 * K * ANGLES * 11
    return {"bytes": n * in_bytes + 2.0 * K * (mod / 8 + llr_bytes * mod + 8 * sym), "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits

def exact(case, seed):
    kind = case["kind"]
    if kind == "cnn":
        return _cnn_exact(case, seed)
    if kind == "kk":
        return _kk_exact(case, seed)
    if kind == "chain":
        if case["ber"] or not (case["llr"] or case["sym"]) or case["n_sym"] > 1 << 21:
            return None
        x, scale, _ = _dual_pol_link(case["mod"], case["baud"], case["L_km"], case["n_sym"], case["snr"], case["adc"],
                                     case["fo"], case["lw"], seed, (0.7, 1.9))
        z, llr = _chain_exact(x, scale, case["mod"], case["baud"], case["L_km"], case["track"], 16)
        return {"bits": None, "llr": llr if case["llr"] else None, "sym": z if case["sym"] else None}
    if not (case["llr"] or case["sym"]) or case["n_ch"] > 8:
        return None
    zs, ls = [], []
    chans = _batch_channels(case, seed)
    for c, wl, ws in zip(chans, _columns("llr", chans), _columns("sym", chans)):
        x, scale, _ = _dual_pol_link(c["mod"], c["baud"], c["L_km"], c["n_sym"], c["snr"], 1, 0.0, 0.0, c["seed"], c["jones"])
        z, llr = _chain_exact(x, scale, c["mod"], c["baud"], c["L_km"], False, 64 if c["mod"] == 4 else 16)
        zs.append(torch.nn.functional.pad(z, (0, ws - z.shape[1])).reshape(-1))
        ls.append(torch.nn.functional.pad(llr, (0, wl - llr.shape[1])).reshape(-1))
    return {"bits": None, "llr": torch.cat(ls) if case["llr"] else None, "sym": torch.cat(zs) if case["sym"] else None}


def _decide(z, mod):
    if mod == 2:
        a = 1.0 / math.sqrt(2.0)
        return torch.complex(torch.where(z.real >= 0, a, -a), torch.where(z.imag >= 0, a, -a))
    s = math.sqrt(10.0)

    def lv(x):
        return torch.copysign(torch.where((x * s).abs() > 2, 3.0 / s, 1.0 / s).double(), x)

    return torch.complex(lv(z.real), lv(z.imag))


def _chain_exact(x, scale, mod, baud, L_km, track, nb):
    """(z, llr) of the whole chain: overlap-save, butterfly CMA / DD-LMS, BPS, LLRs."""
    x = x.double() * float(np.float32(scale))
    x = torch.stack([torch.complex(x[:, 0], x[:, 1]), torch.complex(x[:, 2], x[:, 3])])
    n = x.shape[1]
    K = n // 2
    V = _overlap(baud, L_km)
    N = _fft_n(V)
    S = N - V
    f = _freqs(N, 2 * baud)
    H = math.sqrt(2.0) * _rrc(f, baud, 0.1) * _cis(-0.5 * _beta2() * L_km * 1e3 * (TWO_PI * f) ** 2)
    nw = -(-n // S)
    xp = torch.nn.functional.pad(x, (V // 2, nw * S + N - n))
    u = torch.cat([torch.fft.ifft(torch.fft.fft(xp[:, i * S:i * S + S * (min(i + 256, nw) - i) + V].unfold(1, N, S)) * H)
                   [:, :, V // 2:V // 2 + S].reshape(2, -1) for i in range(0, nw, 256)], 1)[:, :n]
    c = (NTAPS - 1) // 2
    up = torch.nn.functional.pad(u, (c, 4 * SEG + c))
    dev = u.device
    ang = (torch.arange(ANGLES, device=dev, dtype=torch.float64) / ANGLES - 0.5) * (math.pi / 2)
    ph = _cis(ang)
    tap = torch.arange(NTAPS, device=dev)
    y = torch.zeros(2, K + SEG, dtype=torch.complex128, device=dev)
    M = 1 << 16

    def regress(k0, rot):      # k0: (G,) first symbols -> X (G, BU, 2, T)
        k = k0[:, None] + torch.arange(BU, device=dev)
        idx = 2 * k[..., None] + 2 * c - tap
        X = up[:, idx].permute(1, 2, 0, 3)
        if rot is not None:
            phi, n0, d = rot
            X = X * _cis((-TWO_PI / M) * torch.remainder(phi + (idx - c - n0) * d, M).double())[:, :, None, :]
        return X

    def step(h, X, k0, cma):   # h (G, 2, 2, T)
        yy = torch.einsum("gpqi,gkqi->gpk", h, X)
        on = (k0[:, None] + torch.arange(BU, device=dev) < K)[:, None, :]
        if cma:
            e = yy * (yy.abs().square() - (1.0 if mod == 2 else 1.32))
        else:
            w = yy[..., None] * ph.conj()
            d = (w - _decide(w, mod)).abs().square() * on[..., None]
            r = ph[d.sum(2).argmin(-1)][..., None]
            e = yy - _decide(yy * r.conj(), mod) * r
        e = torch.where(on, e, 0)
        return yy, h - MU * torch.einsum("gpk,gkqi->gpqi", e, X.conj())

    def pair_sum(v):
        q = (v[..., 1:] * v[..., :-1].conj()) ** 4
        if mod == 4:     # the two pi/4-aligned rings of 16QAM
            w = torch.clamp(((v.abs().square() - 1.0).abs() - 0.2) / 0.2, 0.0, 1.0)
            q = q * w[..., 1:] * w[..., :-1]
        return complex(q.sum())

    h = torch.zeros(1, 2, 2, NTAPS, dtype=torch.complex128, device=dev)
    h[0, 0, 0, c] = h[0, 1, 1, c] = 1.0
    for k0 in range(0, N_CMA, BU):
        kk = torch.tensor([k0], device=dev)
        yy, h = step(h, regress(kk, None), kk, True)
        y[:, k0:k0 + BU] = yy[0]
    d = 0
    if track:
        s = pair_sum(y[:, N_CMA // 2:N_CMA])
        d = int(np.rint(0.25 * math.atan2(s.imag, s.real) / (2 * TWO_PI) * M))
    for k0 in range(N_CMA, ACQ, BU):
        kk = torch.tensor([k0], device=dev)
        yy, h = step(h, regress(kk, (0, 2 * N_CMA, d) if track else None), kk, False)
        y[:, k0:k0 + BU] = yy[0]
    phi, inc_prev = ((2 * ACQ - 2 * N_CMA) * d) % M, 0
    G = -(-(K - ACQ) // SEG)
    for w0 in range(0, G, WAVE_SEGS):
        g = torch.arange(w0, min(w0 + WAVE_SEGS, G), device=dev)
        ks = ACQ + g * SEG
        hh = h.expand(len(g), 2, 2, NTAPS)
        rot = (phi, 2 * (ACQ + w0 * SEG), d) if track else None
        outs = []
        for t in range(-PRE, SEG, BU):
            yy, nh = step(hh, regress(ks + t, rot), ks + t, False)
            hh = nh
            if t >= 0:
                outs.append(yy)
        seg = torch.cat(outs, 2).permute(1, 0, 2)             # (2, G, SEG)
        a, b = ACQ + w0 * SEG, min(ACQ + (w0 + len(g)) * SEG, K)
        y[:, a:a + len(g) * SEG] = seg.reshape(2, -1)
        if track:
            s = 0j
            full = (b - a) // SEG
            s += pair_sum(seg[:, :full])
            if (b - a) % SEG:
                s += pair_sum(seg[:, full, :(b - a) % SEG])
            inc = int(np.rint(0.25 * math.atan2(s.imag, s.real) / 16.0 / (2 * TWO_PI) * M))
            phi = (phi + 2 * WAVE_SEGS * SEG * d) % M
            d, inc_prev = d + inc_prev, inc
        h = hh[-1:]
    y = y[:, :K]
    bh = torch.empty(2, K, dtype=torch.int64, device=dev)
    for k0 in range(0, K, 1 << 16):
        k1 = min(k0 + (1 << 16), K)
        a, b = max(k0 - nb, 0), min(k1 + nb, K)
        w = y[:, a:b, None] * ph.conj()
        dd = torch.nn.functional.pad(torch.cumsum((w - _decide(w, mod)).abs().square(), 1), (0, 0, 1, 0))
        k = torch.arange(k0, k1, device=dev)
        bh[:, k0:k1] = (dd[:, torch.clamp(k + nb + 1, max=K) - a] - dd[:, torch.clamp(k - nb, min=0) - a]).argmin(-1)
    df = bh[:, :-1] - bh[:, 1:]
    turn = torch.nn.functional.pad(torch.cumsum((df > ANGLES // 2).long() - (df < -(ANGLES // 2)).long(), 1), (1, 0))
    z = y * _cis(-(ang[bh] + turn * (math.pi / 2)))
    err = (z - _decide(z, mod)).abs().square()
    edges = [0] + list(range(ACQ, K, WAVE_SEGS * SEG)) + [K]
    s2 = torch.cat([err[:, a:b].mean(1, keepdim=True).expand(2, b - a) for a, b in zip(edges, edges[1:])], 1)
    m = 2 if mod == 2 else 4
    if mod == 2:
        lv, labels = torch.tensor([1.0, -1.0], device=dev).double() / math.sqrt(2.0), [[0, 1]]
    else:
        lv, labels = torch.tensor([-3.0, -1.0, 1.0, 3.0], device=dev).double() / math.sqrt(10.0), [[1, 1, 0, 0], [1, 0, 0, 1]]
    llr = []
    for v in (z.real, z.imag):
        d2 = (v[..., None] - lv).square()
        for lab in labels:
            one = torch.tensor(lab, device=dev).bool()
            llr.append((d2[..., one].min(-1).values - d2[..., ~one].min(-1).values) / s2)
    return z, torch.stack(llr, -1).reshape(2, K * m)


def _cnn_exact(case, seed):
    z, t = _cnn_data(case, seed)
    K = case["n_sym"]
    params = [(torch.tensor(W.astype(np.float32), device="cuda").double().requires_grad_(),
               torch.tensor(b.astype(np.float32), device="cuda").double().requires_grad_())
              for W, b in _cnn_params(seed, case["layers"])]

    def feats(v):
        return torch.stack([v[0].real, v[0].imag, v[1].real, v[1].imag], 1).double()

    x = feats(z)
    with torch.set_grad_enabled(bool(case["grads"])):
        a = x
        for l, (W, b) in enumerate(params):
            p = torch.nn.functional.pad(a, (0, 0, 7, 7))
            a = sum(p[k:k + K] @ W[k] for k in range(15)) + b
            if l < len(params) - 1:
                a = torch.relu(a)
        y = x + a
        if not case["grads"]:
            return {"y": torch.stack([torch.complex(y[:, 0], y[:, 1]), torch.complex(y[:, 2], y[:, 3])])}
        loss = (y - feats(t)).square().sum() / (4 * K)
    loss.backward()
    return {"loss": float(loss.detach()), "grads": torch.cat([v.grad.reshape(-1) for pr in params for v in pr])}


def _kk_exact(case, seed):
    samples, scale, offset = _kk_link(case, seed)
    fs, fc, N = 4e9, _carrier(case), 1024
    inten = (samples.double() + offset) * float(np.float32(scale))
    n = inten.shape[0]
    amp = torch.clamp(inten, min=1e-30).sqrt()
    k = torch.arange(N, device="cuda")
    hil = torch.where((k > 0) & (k < N // 2), 1.0, torch.where(k > N // 2, -1.0, 0.0)).double() * 1j

    def windows(v, V):
        S = N - V
        nw = -(-n // S)
        return torch.nn.functional.pad(v, (V // 2, nw * S + N - n)).unfold(0, N, S)[:nw]

    phi = torch.fft.ifft(torch.fft.fft(windows(amp.log(), N // 2)) * hil).real[:, N // 4:3 * N // 4].reshape(-1)[:n]
    turns = torch.remainder(fc / fs * torch.arange(n, device="cuda", dtype=torch.float64), 1.0)
    E = amp * _cis(phi + TWO_PI * turns)
    T = 1.0 / fs
    ncd = 2 * int(math.floor(17e-6 * LAM * LAM * case["L_km"] * 1e3 / (2 * C_LIGHT * T * T))) + 1
    V = max(N // 2, -(-(ncd - 1) // 32) * 32)
    f = _freqs(N, fs)
    b2 = 0.5 * _beta2() * case["L_km"] * 1e3
    H = 2.0 * _rrc(f, 1e9, 0.01) * _cis(b2 * ((TWO_PI * fc) ** 2 - (TWO_PI * f) ** 2))
    X = torch.fft.fft(windows(E, V)) * H
    Y = 0.5 * torch.cat([X[:, :N // 4], X[:, N - N // 4:]], 1)
    y = torch.fft.ifft(Y)[:, V // 4:V // 4 + (N - V) // 2].reshape(-1)[:n // 2]
    # the output lags the input by 1536 samples; zeros before the stream's first
    lag = 1536
    yd = torch.nn.functional.pad(y, (lag // 2, 0))
    y_bufs, y_end = yd[:n // 2].view(case["n_buf"], -1), yd[n // 2:]
    if case["eq"]:
        return {"bits": None, "y": y_bufs}
    fd = torch.nn.functional.pad(E, (lag, 0))
    return {"y": y_bufs, "y_end": y_end, "field": list(fd[:n].view(case["n_buf"], -1)), "field_end": fd[n:]}

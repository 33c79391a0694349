"""Performance cases of the correlator: what its users run, at the sizes they run it.

Each case goes through the package's public calls (``xc.Correlator``,
``xc.BatchCorrelator``, ``xc.channelize``, ``xc.correlate_autograd``) with the
buffers, handles and filter taps that a program prepares once.  ``listed``
gives the fixed cases, ``draw`` random ones of the same ranges.

Kinds of a case:
  corr     one integration of a handle: 8-bit, fp16 or fp32 voltages, any operand precision
  train    visibilities of fp32 voltages with gains, and the gradients of both
  fengine  station streams -> channels, in the correlator's input order
  fx       polyphase F-engine to 8 bits, then the 8-bit correlator
  batch    several subarrays in one launch
"""
import math

import numpy as np
import torch

from paper_1107_4264_gb300 import synth, xc

PRECISIONS = {"fp16": xc.XC_PREC_FP16, "hilo": xc.XC_PREC_HILO, "fp8": xc.XC_PREC_FP8}
DTYPES = {"int8": torch.int8, "float16": torch.float16, "float32": torch.float32}


def _corr(name, N, P, F, T, dtype="int8", precision="fp16", gains=False, f64_block=0):
    c = {"kind": "corr", "N": N, "P": P, "F": F, "T": T, "dtype": dtype, "precision": precision,
         "gains": gains, "f64_block": f64_block}
    return dict(c, name=name) if name else c


def listed():
    return [
        # A first light or a unit test of a small array: one call, all latency.
        _corr("tiny_n16", 16, 2, 8, 256),
        # A 32-station dual-polarisation array at full band: one second at 1 kHz channels.
        _corr("small_n32", 32, 2, 8192, 1000),
        # A 64-station dual-polarisation array (a channel fills two tiles).
        _corr("small_n64", 64, 2, 2048, 1000),
        # A subarray whose inputs do not fill whole blocks (400 inputs) with a short integration.
        _corr("ragged_n200", 200, 2, 256, 512),
        # The headline: a 256-station array, 1000 samples per integration.
        _corr("large_n256", 256, 2, 1024, 1000),
        # The same array dumping fast (transients, moving baselines): the output counts as much as the input.
        _corr("short_n256", 256, 2, 2048, 125),
        # 4-bit digitiser samples on the 8-bit floating-point operands.
        _corr("fp8_n256", 256, 2, 512, 1000, precision="fp8"),
        # Floating-point voltages of 512 stations with calibration gains.
        _corr("float_n512", 512, 2, 60, 2048, dtype="float32", gains=True),
        # Calibration by gradient descent: visibilities, voltage and gain gradients.
        {"name": "train_n256", "kind": "train", "N": 256, "P": 2, "F": 64, "T": 4096},
        # The F-engine in front of a floating-point correlator: 512 streams, 1024 channels.
        {"name": "fengine_1024", "kind": "fengine", "N": 256, "P": 2, "nchan": 1024, "T": 500, "ntaps": 0,
         "in": "int8", "out": "float16"},
        # The whole FX chain at 8 bits: 4-tap polyphase filter, 512 channels, 100 stations.
        {"name": "fx_n100", "kind": "fx", "N": 100, "P": 2, "nchan": 512, "T": 1003, "ntaps": 4},
        # Several subarrays sharing the GPU, from 32 to 1024 stations.
        {"name": "batch_6", "kind": "batch", "P": 2, "N": "32 64 128 200 384 1024", "F": "64 128 256 256 512 96",
         "T": "256 1024 4096 512 2048 8192"},
    ]


def _log(rng, lo, hi):
    """A whole number from lo to hi, spread evenly over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _fit(rng, N, P, per_sample, f_hi, t_lo, t_hi, max_bytes=1 << 30, max_ops=1.0e12):
    """F and T for N stations, so that buffers and operations stay inside the bounds."""
    nb = N * (N + 1) // 2
    T = _log(rng, t_lo, t_hi)
    room = min(max_bytes / (T * N * P * 2 * per_sample), max_bytes / (nb * P * P * 8),
               max_ops / (8.0 * T * P * P * nb))
    return _log(rng, 1, max(1, min(f_hi, int(room)))), T


def draw(rng):
    kind = rng.choice(["int8", "int8", "int8", "fp8", "float", "float", "train", "fengine", "fengine", "fx", "batch"])
    P = rng.choice([1, 2, 2])
    if kind == "int8":
        N = rng.choice([_log(rng, 2, 1024), rng.choice([4, 8, 16, 32, 64, 128, 256])])
        F, T = _fit(rng, N, P, 1, 65535, 32, 8192)
        return _corr("", N, P, F, T)
    if kind == "fp8":
        N = rng.choice([_log(rng, 2, 512), rng.choice([16, 32, 64, 128, 256])])
        F, T = _fit(rng, N, P, 1, 65535, 32, 4096)
        return _corr("", N, P, F, T, precision="fp8")
    if kind == "float":
        N = _log(rng, 2, 512)
        dtype = rng.choice(["float16", "float32"])
        precision = rng.choice(["fp16", "fp16", "hilo", "fp8"])
        F, T = _fit(rng, N, P, 2 if dtype == "float16" else 4, 4096, 32, 4096, max_ops=4.0e11)
        return _corr("", N, P, F, T, dtype=dtype, precision=precision, gains=rng.random() < 0.5,
                     f64_block=rng.choice([0, 0, 512, 1024]))
    if kind == "train":
        N = _log(rng, 2, 256)
        F, T = _fit(rng, N, P, 4, 1024, 64, 4096, max_ops=4.0e11)
        return {"kind": "train", "N": N, "P": P, "F": F, "T": T}
    if kind == "fengine":
        N, nchan = _log(rng, 1, 512), 1 << rng.randint(4, 12)
        ntaps = rng.choice([0, 0, 4, 8])
        T = max(1, ntaps) + _log(rng, 1, max(1, min(4096, (1 << 27) // (N * P * nchan))))
        return {"kind": "fengine", "N": N, "P": P, "nchan": nchan, "T": T, "ntaps": ntaps,
                "in": rng.choice(["int8", "int8", "float16", "float32"]),
                "out": rng.choice(["int8", "float16", "float16", "float32"])}
    if kind == "fx":
        N, nchan = _log(rng, 2, 256), 1 << rng.randint(5, 11)
        T = 8 + _log(rng, 32, max(32, min(2048, (1 << 27) // (N * P * nchan))))
        return {"kind": "fx", "N": N, "P": P, "nchan": nchan, "T": T, "ntaps": rng.choice([2, 4, 8])}
    subs = []
    for _ in range(rng.randint(2, 6)):
        N = _log(rng, 8, 384)
        subs.append((N,) + _fit(rng, N, P, 1, 512, 64, 4096, max_bytes=1 << 28, max_ops=3.0e11))
    return {"kind": "batch", "P": P, "N": " ".join(str(s[0]) for s in subs),
            "F": " ".join(str(s[1]) for s in subs), "T": " ".join(str(s[2]) for s in subs)}


# ------------------------------------------------------------------ inputs


def _voltages(T, F, N, P, dtype, precision, seed, dev):
    """Sky voltages: receiver noise and three point sources, as the type holds them."""
    if dtype == "int8" and precision == "fp8":  # 4-bit digitiser levels
        return synth.uniform_int8((T, F, N, P, 2), -7, 7, seed, device=dev)
    if dtype == "int8":
        return synth.sky_voltages(T, F, N, P, noise_sigma=3.0, nsrc=3, src_amp=1.5, seed=seed, device=dev,
                                  quantise_int8=True)
    return synth.sky_voltages(T, F, N, P, noise_sigma=math.sqrt(0.5), nsrc=3, src_amp=1.0, seed=seed, device=dev,
                              dtype=DTYPES[dtype])


def _gains(N, P, seed, dev):
    return torch.from_numpy(synth.complex_gains(N, P, seed)).to(dev, torch.float32)


def _streams(N, P, L, dtype, seed, dev):
    """Station streams [N][P][L][2]: receiver noise and a signal that all stations share."""
    gen = torch.Generator(device=dev).manual_seed(seed)
    x = torch.empty((N, P, L, 2), dtype=DTYPES[dtype], device=dev)
    common = torch.randn((P, L, 2), generator=gen, device=dev) * 4.0
    for s in range(N):
        v = torch.randn((P, L, 2), generator=gen, device=dev).mul_(12.0).add_(common)
        x[s] = v.round_().clamp_(-127, 127).to(torch.int8) if dtype == "int8" else v.to(x.dtype)
    return x


def _taps(nchan, ntaps, dev):
    """Hann-windowed sinc prototype of ntaps * nchan coefficients, of energy nchan."""
    m = (np.arange(ntaps * nchan) + 0.5) / nchan - ntaps / 2.0
    h = np.sinc(m) * np.hanning(ntaps * nchan + 2)[1:-1]
    h *= math.sqrt(nchan / np.sum(h * h))
    return torch.from_numpy(h.reshape(ntaps, nchan)).to(dev, torch.float32)


def _fscale(c, out):
    """8-bit codes get an rms of about 16 per component, the other types a unitary transform."""
    return (16.0 / 12.6 if out == "int8" else 1.0) / math.sqrt(c["nchan"])


def _subs(c):
    return list(zip(*([int(v) for v in c[k].split()] for k in ("N", "F", "T"))))


def prepare(c, seed):
    dev = torch.device("cuda")
    kind = c["kind"]
    if kind == "corr":
        eng = xc.Correlator(c["N"], c["P"], c["F"], c["T"], c["dtype"], precision=PRECISIONS[c["precision"]],
                            fp64_block=c["f64_block"])
        if c["gains"]:
            eng.set_gains(_gains(c["N"], c["P"], seed, dev))
        return {"kind": kind, "eng": eng, "out": eng.new_output(),
                "x": _voltages(c["T"], c["F"], c["N"], c["P"], c["dtype"], c["precision"], seed, dev)}
    if kind == "train":
        eng = xc.Correlator(c["N"], c["P"], c["F"], c["T"], "float32")
        gen = torch.Generator(device=dev).manual_seed(seed + 1)
        return {"kind": kind, "eng": eng,
                "x": _voltages(c["T"], c["F"], c["N"], c["P"], "float32", "fp16", seed, dev).requires_grad_(),
                "g": _gains(c["N"], c["P"], seed, dev).requires_grad_(),
                "grad": torch.randn(eng.out_shape, generator=gen, device=dev)}
    if kind == "batch":
        subs = _subs(c)
        eng = xc.BatchCorrelator(subs, npol=c["P"])
        return {"kind": kind, "eng": eng, "outs": eng.new_outputs(),
                "xs": [_voltages(T, F, N, c["P"], "int8", "fp16", seed + 1000 * i, dev)
                       for i, (N, F, T) in enumerate(subs)]}
    N, P, nchan, T, ntaps = c["N"], c["P"], c["nchan"], c["T"], c["ntaps"]
    out = c["out"] if kind == "fengine" else "int8"
    Tout = T - max(1, ntaps) + 1
    st = {"kind": kind, "nchan": nchan, "scale": _fscale(c, out), "out_dtype": out,
          "x": _streams(N, P, T * nchan, c["in"] if kind == "fengine" else "int8", seed, dev),
          "taps": _taps(nchan, ntaps, dev) if ntaps else None,
          "chan": torch.empty((Tout, nchan, N, P, 2), dtype=DTYPES[out], device=dev)}
    if kind == "fx":
        st["eng"] = xc.Correlator(N, P, nchan, Tout, "int8")
        st["vis"] = st["eng"].new_output()
    return st


def run(s):
    kind = s["kind"]
    if kind == "corr":
        return s["eng"].correlate(s["x"], out=s["out"])
    if kind == "train":
        vis = xc.correlate_autograd(s["eng"], s["x"], s["g"])
        gx, gg = torch.autograd.grad(vis, (s["x"], s["g"]), grad_outputs=s["grad"])
        return vis.detach(), gx, gg
    if kind == "batch":
        return s["eng"].correlate(s["xs"], s["outs"])
    xc.channelize(s["x"], s["nchan"], s["scale"], s["out_dtype"], out=s["chan"], taps=s["taps"])
    if kind == "fengine":
        return s["chan"]
    return s["chan"], s["eng"].correlate(s["chan"], out=s["vis"])


# -------------------------------------------------------------------- work


def _corr_work(N, P, F, T, in_bytes):
    nb = N * (N + 1) // 2
    return T * F * N * P * 2 * in_bytes + F * nb * P * P * 8, 8 * F * T * P * P * nb


def work(c):
    kind = c["kind"]
    if kind == "batch":
        w = [_corr_work(N, c["P"], F, T, 1) for N, F, T in _subs(c)]
        return {"bytes": sum(v[0] for v in w), "flops": sum(v[1] for v in w)}
    N, P, T = c["N"], c["P"], c["T"]
    if kind == "corr":
        b, f = _corr_work(N, P, c["F"], T, {"int8": 1, "float16": 2, "float32": 4}[c["dtype"]])
        return {"bytes": b, "flops": f}
    if kind == "train":  # x and the output gradient in; visibilities and the voltage gradient out
        F, n, nb = c["F"], N * P, N * (N + 1) // 2
        return {"bytes": 2 * T * F * n * 8 + 2 * F * nb * P * P * 8,
                "flops": 8 * F * T * P * P * nb + 8 * F * T * n * n}
    nchan, ntaps = c["nchan"], c["ntaps"]
    Tout = T - max(1, ntaps) + 1
    size = {"int8": 2, "float16": 4, "float32": 8}
    i, o = (c["in"], c["out"]) if kind == "fengine" else ("int8", "int8")
    b = N * P * nchan * (T * size[i] + Tout * size[o])
    f = N * P * Tout * nchan * int(5 * math.log2(nchan) + 4 * ntaps)
    if kind == "fx":  # the channels are an output of the pass and the correlator's input
        vb, vf = _corr_work(N, P, nchan, Tout, 0)
        b, f = b + vb, f + vf
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------- exact


def _pairs(V, N, P):
    """[f][n][n] complex -> [f][N(N+1)/2][P*P][2] real, the lower station triangle."""
    i, j = torch.tril_indices(N, N, device=V.device)
    V = V.view(-1, N, P, N, P).permute(0, 1, 3, 2, 4)[:, i, j]
    return torch.view_as_real(V.contiguous()).reshape(V.shape[0], i.numel(), P * P, 2)


def _vis64(x, gains=None, whole=False):
    """Visibilities of [T][F][N][P][2] in complex128, a few channels at a time."""
    T, F, N, P, _ = x.shape
    out = []
    step = max(1, 40_000_000 // max(T * N * P, (N * P) ** 2))
    for f in range(0, F, step):
        y = torch.view_as_complex(x[:, f:f + step].double()).reshape(T, -1, N * P).permute(1, 2, 0)
        if gains is not None:
            y = y * gains.reshape(1, -1, 1)
        v = _pairs(y @ y.mH, N, P)
        out.append(v.round().to(torch.int64) if whole else v)
    return torch.cat(out)


def _chan64(x, c, scale, taps, out):
    """The F-engine in 64 bits, a few stations at a time: [T][nchan][N][P][2]."""
    N, P, L, _ = x.shape
    T, ntaps = c["T"], max(1, c["ntaps"])
    res = []
    step = max(1, 30_000_000 // (P * L))
    for s in range(0, N, step):
        v = torch.view_as_complex(x[s:s + step].double()).reshape(-1, P, T, c["nchan"])
        if taps is not None:
            v = sum(taps[q].double() * v[:, :, q:T - ntaps + 1 + q] for q in range(ntaps))
        y = torch.view_as_real((torch.fft.fft(v, dim=-1) * scale).permute(2, 3, 0, 1).contiguous())
        res.append(y.round().clamp_(-127, 127).to(torch.int64) if out == "int8" else y)
    return torch.cat(res, dim=2)


def exact(c, seed):
    kind = c["kind"]
    if kind == "batch":  # its largest subarray alone takes minutes in 64 bits
        return None
    s = prepare(c, seed)
    if kind == "corr":
        if c["dtype"] == "int8":
            return _vis64(s["x"], whole=True)
        g = torch.view_as_complex(_gains(c["N"], c["P"], seed, s["x"].device).double()) if c["gains"] else None
        return _vis64(s["x"], g)
    if kind == "train":
        x, g = s["x"].detach(), torch.view_as_complex(s["g"].detach().double())
        N, P, F, n = c["N"], c["P"], c["F"], c["N"] * c["P"]
        i, j = torch.tril_indices(N, N, device=x.device)
        gx = torch.empty(x.shape, dtype=torch.float64, device=x.device)
        gg = torch.zeros(n, dtype=torch.complex128, device=x.device)
        for f in range(F):
            G = torch.zeros((N, N, P, P), dtype=torch.complex128, device=x.device)
            G[i, j] = torch.view_as_complex(s["grad"][f].double().contiguous()).view(-1, P, P)
            G = G.permute(0, 2, 1, 3).reshape(n, n)
            xf = torch.view_as_complex(x[:, f].double().contiguous()).reshape(-1, n)
            gy = (xf * g.reshape(1, n)) @ (G + G.mH).mT
            gx[:, f] = torch.view_as_real((gy * g.reshape(1, n).conj())).reshape(-1, N, P, 2)
            gg += (xf.conj() * gy).sum(0)
        return _vis64(x, g), gx, torch.view_as_real(gg).reshape(N, P, 2)
    chan = _chan64(s["x"], c, s["scale"], s["taps"], s["out_dtype"])
    return chan if kind == "fengine" else (chan, _vis64(chan, whole=True))

"""Performance cases of the dedispersion library's public entry points.

Each case is one call as a user's program makes it on data it has in hand: the
phase-rotate-and-sum on spectra (``Plan.dedisperse_spectra_bins``), the whole
path on a filterbank (``Plan.execute``), the batching form
(``Batch.execute``), brute-force time-domain dedispersion
(``Plan.tdd_execute``) and the host-buffer call (``Plan.execute_host``).  The
sizes are those of the repository's workloads (64, 1024, 1536 and 4096
channels, 128 to 8192 trials, 1 to 32 beams) or windows of them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2110_03482_gb300 as fdd

K_DM = 1.0 / 2.41e-4  # MHz^2 pc^-1 cm^3 s, the library's default constant

# Bands of the workloads: lower and upper edge (MHz), sampling time (s).
BANDS = {
    "lband64": (1250.0, 1550.0, 0.25e-3),
    "survey": (1210.0, 1520.0, 64e-6),
    "wide": (1100.0, 1700.0, 81.92e-6),
    "lowfreq": (110.0, 190.0, 491.52e-6),
}
PRECISIONS = {"fp32": fdd.FDD_PREC_FP32, "bf16_hilo": fdd.FDD_PREC_BF16_HILO,
              "bf16": fdd.FDD_PREC_BF16, "fp16": fdd.FDD_PREC_FP16}
OUTPUTS = {"time": fdd.FDD_OUT_TIME, "spectra": fdd.FDD_OUT_SPECTRA, "power": fdd.FDD_OUT_POWER}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # The smallest job: 64 channels, a 4096-sample series, 128 trials, the
        # sum over channels alone (launch latency and the small tile).
        dict(name="sum_64ch_128dm", kind="sum", band="lband64", n_chan=64, fft_len=4096,
             bin_first=0, n_bins=2049, pad=0, n_series=1, dm0=0.0, ddm=1.0, n_dm=128,
             out="spectra", prec="fp32"),
        # The same job end to end, filterbank in and time series out: what a
        # quick look at one short observation calls.
        dict(name="execute_64ch_128dm_time", kind="execute", band="lband64", n_chan=64,
             n_t=4096, chunk_len=0, n_beams=1, dm0=0.0, ddm=1.0, n_dm=128, out="time",
             prec="fp32", u8=False, chan_major=False, downsample=1),
        # The survey's hot path: a window of bins of a 2^18 transform, 1024
        # channels, 2048 trials (the unit a program splits across calls).
        dict(name="sum_1024ch_2048dm", kind="sum", band="survey", n_chan=1024, fft_len=1 << 18,
             bin_first=70001, n_bins=4096, pad=0, n_series=1, dm0=0.0, ddm=0.5, n_dm=2048,
             out="spectra", prec="fp32"),
        # A targeted search around a known DM: odd channel and trial counts, a
        # first trial away from zero, two series, DC included, a padded pitch.
        dict(name="sum_387ch_701dm_ragged", kind="sum", band="survey", n_chan=387,
             fft_len=1 << 15, bin_first=0, n_bins=4001, pad=3, n_series=2, dm0=56.7, ddm=0.11,
             n_dm=701, out="power", prec="fp32"),
        # Low frequency, long delays: 4096 channels, 8192 trials, power
        # spectra for a periodicity search, near the top of a 2^19 transform.
        dict(name="sum_4096ch_8192dm_power", kind="sum", band="lowfreq", n_chan=4096,
             fft_len=1 << 19, bin_first=262145 - 301, n_bins=301, pad=0, n_series=1, dm0=0.0,
             ddm=0.05, n_dm=8192, out="power", prec="fp32"),
        # 32 beams sharing the bins on tensor cores, FP16 (the fast form).
        dict(name="sum_32beam_4096dm_fp16", kind="sum", band="lband64", n_chan=1024,
             fft_len=1 << 19, bin_first=100000, n_bins=1025, pad=0, n_series=32, dm0=0.0,
             ddm=0.5, n_dm=4096, out="spectra", prec="fp16"),
        # 16 beams, 4096 channels, power output, BF16 hi+lo (the accurate
        # tensor-core form with FP32's range).
        dict(name="sum_16beam_8192dm_hilo", kind="sum", band="lowfreq", n_chan=4096,
             fft_len=1 << 19, bin_first=1, n_bins=129, pad=0, n_series=16, dm0=0.0, ddm=0.05,
             n_dm=8192, out="power", prec="bf16_hilo"),
        # Whole path on tensor cores: eight beams of float samples to time
        # series in overlap-save chunks (transposes, both FFTs, scatter).
        dict(name="execute_8beam_1024dm_fp16", kind="execute", band="lband64", n_chan=512,
             n_t=100000, chunk_len=1 << 15, n_beams=8, dm0=0.0, ddm=0.5, n_dm=1024, out="time",
             prec="fp16", u8=False, chan_major=False, downsample=1),
        # The survey end to end: 2^20 8-bit samples, 2048 trials, five 2^18
        # chunks, time output (the largest case).
        dict(name="execute_survey_2048dm", kind="execute", band="survey", n_chan=1024,
             n_t=1 << 20, chunk_len=1 << 18, n_beams=1, dm0=0.0, ddm=0.5, n_dm=2048,
             out="time", prec="fp32", u8=True, chan_major=False, downsample=1),
        # Beams of uneven length and trial count in one persistent launch
        # (default tile, no autotuning: the same tile on every run).
        dict(name="batch_6beam_1536ch", kind="batch", band="wide", n_chan=1536,
             n_t="4096,9000,20000,65536,30001,6000", n_dm="512,1300,4096,2048,777,3000",
             dm0=0.0, ddm=0.25, out="power", u8=False),
        # Brute force in the time domain, the method Fourier-domain
        # dedispersion is compared with: 8-bit samples, 512 trials.
        dict(name="tdd_1024ch_512dm", kind="tdd", band="survey", n_chan=1024, n_t=1 << 17,
             n_beams=1, dm0=0.0, ddm=0.5, n_dm=512, u8=True, chan_major=False),
        # Host buffers in and out (page-locked), copies streamed beside the
        # computation: 8-bit samples to power spectra.
        dict(name="host_1024ch_512dm_power", kind="host", band="survey", n_chan=1024,
             n_t=1 << 17, chunk_len=1 << 16, n_beams=1, dm0=0.0, ddm=0.5, n_dm=512,
             out="power", prec="fp32", u8=True, chan_major=False, downsample=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sum", "sum", "sum", "tc", "tc", "execute", "batch", "tdd"])
    band = rng.choice(sorted(BANDS))
    ddm = 0.05 if band == "lowfreq" else rng.choice([0.1, 0.25, 0.5])
    if kind in ("sum", "tc"):
        tc = kind == "tc"
        n_chan = _log(rng, 48, 4096)
        n_dm = _log(rng, 100, 8192)
        n_series = rng.choice([5, 8, 16, 23, 32]) if tc else rng.choice([1, 1, 1, 2, 3])
        fft_len = 1 << rng.randint(12, 19)
        budget = 2.5e10 if tc else 1.5e10  # complex MACs of a pass
        most = max(16, int(budget / (n_chan * n_dm * n_series)))
        n_bins = min(fft_len // 2 + 1, most, _log(rng, 150, 9000))
        return dict(kind="sum", band=band, n_chan=n_chan, fft_len=fft_len,
                    bin_first=rng.randint(0, fft_len // 2 + 1 - n_bins), n_bins=n_bins,
                    pad=rng.choice([0, 0, 1, 5]), n_series=n_series,
                    dm0=rng.choice([0.0, 0.0, 13.3]), ddm=ddm, n_dm=n_dm,
                    out=rng.choice(["spectra", "power"]),
                    prec=rng.choice(["fp16", "bf16_hilo", "bf16"]) if tc else "fp32")
    if kind == "execute":
        n_chan = _log(rng, 48, 1024)
        n_dm = _log(rng, 64, 3000)
        n_t = _log(rng, 4000, 400000)
        n_t = min(n_t, max(4000, int(1.2e11 / (n_chan * n_dm))))
        prec = rng.choice(["fp32", "fp32", "fp16", "bf16_hilo"])
        chunk_len = rng.choice([0, 0, 1 << 14]) if n_t > 20000 else 0
        return dict(kind="execute", band="lband64", n_chan=n_chan, n_t=n_t, chunk_len=chunk_len,
                    n_beams=1 if prec == "fp32" else rng.choice([2, 4, 8]), dm0=0.0, ddm=0.1,
                    n_dm=n_dm, out=rng.choice(["time", "spectra", "power"]), prec=prec,
                    u8=rng.choice([True, False]), chan_major=rng.choice([True, False]),
                    downsample=1)
    if kind == "batch":
        n = rng.randint(2, 8)
        return dict(kind="batch", band="wide", n_chan=_log(rng, 64, 1536),
                    n_t=",".join(str(_log(rng, 3000, 40000)) for _ in range(n)),
                    n_dm=",".join(str(_log(rng, 512, 4096)) for _ in range(n)), dm0=0.0,
                    ddm=0.25, out=rng.choice(["spectra", "power"]), u8=rng.choice([True, False]))
    return dict(kind="tdd", band=rng.choice(["lband64", "survey", "wide"]),
                n_chan=_log(rng, 48, 1024), n_t=_log(rng, 60000, 200000), n_beams=1, dm0=0.0,
                ddm=ddm, n_dm=_log(rng, 32, 600), u8=rng.choice([True, True, False]),
                chan_major=rng.choice([True, False]))


# ------------------------------------------------------------------ geometry
def _centres(case):
    lo, hi, t_samp = BANDS[case["band"]]
    dnu = (hi - lo) / case["n_chan"]
    return lo + 0.5 * dnu, dnu, t_samp


def _delays(case, dms):
    """Delays in samples, [trial][channel], of Eq. 1 in float64."""
    nu_lo, dnu, t_samp = _centres(case)
    nu = nu_lo + dnu * np.arange(case["n_chan"], dtype=np.float64)
    rate = K_DM * (1.0 / (nu * nu) - 1.0 / (nu.max() * nu.max())) / t_samp
    return np.asarray(dms)[:, None] * rate[None, :]


def _dms(case):
    return case["dm0"] + case["ddm"] * np.arange(case["n_dm"], dtype=np.float64)


def _common(case):
    nu_lo, dnu, t_samp = _centres(case)
    return dict(n_chan=case["n_chan"], nu_lo_mhz=nu_lo, dnu_mhz=dnu, t_samp_s=t_samp)


def _layout(case):
    return fdd.FDD_LAYOUT_CHAN_MAJOR if case.get("chan_major") else fdd.FDD_LAYOUT_TIME_MAJOR


def _beams(case):
    n_t = [int(v) for v in case["n_t"].split(",")]
    n_dm = [int(v) for v in case["n_dm"].split(",")]
    return [(t, case["dm0"], case["ddm"], d) for t, d in zip(n_t, n_dm)]


def _samples(shape, u8, seed, n_chan, chan_axis):
    """Noise over a sloping bandpass: 8-bit around 128, or floats around 0."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(shape, device="cuda", generator=g)
    gain = torch.linspace(0.7, 1.3, n_chan, device="cuda")
    view = [1] * len(shape)
    view[chan_axis] = n_chan
    x.mul_(gain.view(view))
    if not u8:
        return x
    return x.mul_(16.0).add_(128.0).round_().clamp_(0, 255).to(torch.uint8)


def _filterbank(case, seed):
    b, t, c = case["n_beams"], case["n_t"], case["n_chan"]
    if case.get("chan_major"):
        return _samples((b, c, t), case["u8"], seed, c, 1)
    return _samples((b, t, c), case["u8"], seed, c, 2)


def _spectra(case, seed):
    """Spectra of noise series: complex Gaussian over a sloping bandpass, and
    the large real DC of 8-bit samples where the window holds it."""
    pitch = case["n_bins"] + case["pad"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn((case["n_series"], case["n_chan"], pitch, 2), device="cuda", generator=g)
    X.mul_(16.0 * math.sqrt(case["fft_len"] / 2.0))
    X.mul_(torch.linspace(0.7, 1.3, case["n_chan"], device="cuda").view(1, -1, 1, 1))
    if case["bin_first"] == 0:
        X[:, :, 0, 0] += 128.0 * case["fft_len"]
        X[:, :, 0, 1] = 0.0
    return X


def _out_buffer(info, out):
    return torch.empty((info["out_elems"], 2) if out == "spectra" else (info["out_elems"],),
                       dtype=torch.float32, device="cuda")


# ------------------------------------------------------------------ a pass
def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "sum":
        st["plan"] = fdd.Plan(n_t=case["fft_len"], dm_list=_dms(case), n_beams=case["n_series"]
                              if case["prec"] != "fp32" else 1, in_dtype=fdd.FDD_IN_F32,
                              output=OUTPUTS[case["out"]], precision=PRECISIONS[case["prec"]],
                              workspace_limit=64 << 30, **_common(case))
        st["X"], st["pitch"] = _spectra(case, seed), case["n_bins"] + case["pad"]
        shape = (case["n_series"], case["n_dm"], case["n_bins"])
        st["Y"] = torch.empty(shape + (2,) if case["out"] == "spectra" else shape, device="cuda")
    elif kind in ("execute", "host", "tdd"):
        kw = dict(n_t=case["n_t"], n_beams=case["n_beams"], dm_list=_dms(case),
                  in_dtype=fdd.FDD_IN_U8 if case["u8"] else fdd.FDD_IN_F32,
                  in_layout=_layout(case), **_common(case))
        if kind != "tdd":
            kw.update(chunk_len=case["chunk_len"], output=OUTPUTS[case["out"]],
                      precision=PRECISIONS[case["prec"]], downsample=case["downsample"])
        else:
            kw.update(workspace_limit=64 << 30)
        st["plan"] = fdd.Plan(**kw)
        x = _filterbank(case, seed)
        if kind == "tdd":
            n_out = case["n_t"] - st["plan"].info["d_max"]
            st["y"] = torch.empty((case["n_beams"], case["n_dm"], n_out), device="cuda")
        else:
            st["y"] = _out_buffer(st["plan"].info, case["out"])
        if kind == "host":
            x = x.cpu().pin_memory()
            st["y"] = torch.empty(st["y"].shape, dtype=torch.float32, pin_memory=True)
        st["x"] = x
    else:
        beams = _beams(case)
        st["batch"] = fdd.Batch(beams, autotune=False, output=OUTPUTS[case["out"]],
                                in_dtype=fdd.FDD_IN_U8 if case["u8"] else fdd.FDD_IN_F32,
                                **_common(case))
        st["x"] = torch.cat([_samples((b[0], case["n_chan"]), case["u8"], seed * 1000 + i,
                                      case["n_chan"], 1).reshape(-1)
                             for i, b in enumerate(beams)])
        st["y"] = _out_buffer(st["batch"].info, case["out"])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "sum":
        st["plan"].dedisperse_spectra_bins(st["X"], st["pitch"], case["n_series"],
                                           case["bin_first"], case["n_bins"], 0, case["n_dm"],
                                           st["Y"], case["n_bins"], OUTPUTS[case["out"]])
        return st["Y"]
    if kind == "execute":
        st["plan"].execute(st["x"], st["y"])
    elif kind == "tdd":
        st["plan"].tdd_execute(st["x"], st["y"])
    elif kind == "batch":
        st["batch"].execute(st["x"], st["y"])
    else:
        st["plan"].execute_host(st["x"], st["y"])
        torch.cuda.current_stream().synchronize()  # the result is read on the host
    return st["y"]


# ------------------------------------------------------------------ its floor
def _geometry(n_t, chunk_len, d_max):
    """Transform length, kept samples per chunk, chunks, output samples."""
    if chunk_len == 0:
        L = 2
        while L < n_t:
            L *= 2
        return L, n_t, 1, n_t
    hop = chunk_len - d_max
    n_out = n_t - d_max
    return chunk_len, hop, -(-n_out // hop), n_out


def _d_max(case):
    return int(math.ceil(_delays(case, [case["dm0"] + case["ddm"] * (case["n_dm"] - 1)]).max()))


def work(case):
    kind = case["kind"]
    nc = case["n_chan"]
    if kind == "sum":
        rows = case["n_series"] * case["n_bins"]
        out = 8 if case["out"] == "spectra" else 4
        return {"bytes": rows * (8 * nc + out * case["n_dm"]),
                "flops": 8.0 * rows * nc * case["n_dm"]}
    esz = 1 if case["u8"] else 4
    if kind == "tdd":
        n_out = case["n_t"] - _d_max(case)
        return {"bytes": case["n_beams"] * (esz * nc * case["n_t"] + 4 * case["n_dm"] * n_out),
                "flops": float(case["n_beams"]) * nc * case["n_dm"] * n_out}
    jobs = ([(t, 0, d, 1) for t, _, _, d in _beams(case)] if kind == "batch" else
            [(case["n_t"], case["chunk_len"], case["n_dm"], case["n_beams"])])
    nbytes = flops = 0.0
    for n_t, chunk_len, n_dm, n_beams in jobs:
        L, _, n_chunks, n_out = _geometry(n_t, chunk_len, _d_max(case) if chunk_len else 0)
        K = L // 2 + 1
        fft = 2.5 * L * math.log2(L)  # real transform
        nbytes += n_beams * esz * nc * n_t
        nbytes += n_beams * (4 * n_dm * n_out if case["out"] == "time" else
                             (8 if case["out"] == "spectra" else 4) * n_chunks * n_dm * K)
        flops += n_beams * n_chunks * (8.0 * nc * n_dm * K + nc * fft +
                                       (n_dm * fft if case["out"] == "time" else 0.0))
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ in 64 bits
def _sum64(X, bins, L, delays):
    """sum over channels of X[c][k] exp(2 pi i k d[j][c] / L), complex128.

    X: [series][channel][bin] complex128 on the GPU, bins the absolute bins.
    """
    d = torch.from_numpy(np.ascontiguousarray(delays)).cuda() / L  # cycles per bin
    Y = torch.empty((X.shape[0], d.shape[0], len(bins)), dtype=torch.complex128, device="cuda")
    step = max(1, int(2.5e8 // d.numel()))
    for i in range(0, len(bins), step):
        k = torch.as_tensor(bins[i:i + step], dtype=torch.float64, device="cuda")
        ph = k[:, None, None] * d[None]
        ph = (ph - ph.round()) * (2.0 * math.pi)
        W = torch.polar(torch.ones_like(ph), ph)  # [bin][trial][channel]
        Y[:, :, i:i + step] = torch.bmm(W, X[:, :, i:i + step].permute(2, 1, 0)).permute(2, 1, 0)
    return Y


def _as_output(Y, out):
    if out == "spectra":
        return torch.view_as_real(Y)
    return Y.real.square() + Y.imag.square()


def _whole64(case, x, n_t, chunk_len, n_dm):
    """The whole path of one beam, x [channel][sample] float64: [rows]."""
    dms = case["dm0"] + case["ddm"] * np.arange(n_dm, dtype=np.float64)
    d = _delays(case, dms)
    L, hop, n_chunks, n_out = _geometry(n_t, chunk_len, int(math.ceil(d.max())))
    parts = []
    for c in range(n_chunks):
        seg = x[:, c * hop:c * hop + L]
        X = torch.fft.rfft(seg, n=L)[None]
        Y = _sum64(X, np.arange(L // 2 + 1), L, d)[0]
        if case["out"] == "time":
            parts.append(torch.fft.irfft(Y, n=L)[:, :min(hop, n_out - c * hop)])
        else:
            parts.append(_as_output(Y, case["out"]))
    return torch.cat(parts, dim=1) if case["out"] == "time" else torch.stack(parts)


def exact(case, seed):
    kind = case["kind"]
    w = work(case)
    if kind == "sum":
        if w["flops"] / case["n_series"] > 2.4e11:  # phasors to evaluate: 3e10
            return None
        X = torch.view_as_complex(_spectra(case, seed)[:, :, :case["n_bins"]].double())
        bins = np.arange(case["bin_first"], case["bin_first"] + case["n_bins"])
        return _as_output(_sum64(X, bins, case["fft_len"], _delays(case, _dms(case))),
                          case["out"])
    if kind == "tdd":
        if w["flops"] > 1.5e11:
            return None
        x = _filterbank(case, seed)
        x = x if case["chan_major"] else x.transpose(1, 2)
        x = x.double().contiguous()
        s = np.floor(_delays(case, _dms(case)) + 0.5).astype(np.int64)
        n_out = case["n_t"] - _d_max(case)
        y = torch.zeros((case["n_beams"], case["n_dm"], n_out), dtype=torch.float64,
                        device="cuda")
        flat = x.reshape(case["n_beams"], -1)
        row0 = torch.arange(case["n_chan"], device="cuda") * case["n_t"]
        t = torch.arange(n_out, device="cuda")
        for j in range(case["n_dm"]):
            first = row0 + torch.from_numpy(s[j]).cuda()
            for i in range(0, case["n_chan"], 256):
                idx = first[i:i + 256, None] + t[None]
                y[:, j] += flat[:, idx].sum(dim=1)
        return y
    if w["flops"] > 2.4e11 * case.get("n_beams", 1):
        return None
    if kind == "batch":
        parts = []
        for i, (n_t, _, _, n_dm) in enumerate(_beams(case)):
            x = _samples((n_t, case["n_chan"]), case["u8"], seed * 1000 + i, case["n_chan"], 1)
            y = _whole64(case, x.double().t().contiguous(), n_t, 0, n_dm)
            parts.append(y.reshape(-1, 2) if case["out"] == "spectra" else y.reshape(-1))
        return torch.cat(parts)
    x = _filterbank(case, seed)
    x = x if case["chan_major"] else x.transpose(1, 2)
    ys = [_whole64(case, x[b].double().contiguous(), case["n_t"], case["chunk_len"],
                   case["n_dm"]) for b in range(case["n_beams"])]
    y = torch.stack(ys)
    return y.reshape(-1, 2) if case["out"] == "spectra" else y.reshape(-1)

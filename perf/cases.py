"""Performance cases of the correction library: the work its users have it do.

Every case goes through the package's public entry points (plans, direct calls) on
device-resident complex64 samples.  Sizes are those of the workload recipes
in ``synth`` and of ``bench.py`` (plain pulse, Doppler bank, uneven batch,
split-precision exact sinc, paper-sized RF pulse) and of the tests' ragged and
long shapes.  ``listed`` holds fixed cases, ``draw`` more of the same ranges,
``exact`` the method in 64 bits in plain torch.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2508_04951_gb300 as dc

C_LIGHT = 299792458.0
KAPPA = 1.602176634e-19 ** 2 / (8 * math.pi ** 2 * 9.1093837015e-31 * 8.8541878128e-12)
MODES = {"windowed": dc.DC_WINDOWED, "exact_fp32": dc.DC_EXACT_FP32, "exact_bf16x3": dc.DC_EXACT_BF16X3,
         "exact_fp16x3": dc.DC_EXACT_FP16X3}
BATCH_SHAPE_SEED = 3      # the lengths of a batch are the case's, not the seed's


def listed():
    return [
        # The plain single pulse: the smallest call, one 4096-sample LFM
        # replayed from a recorded plan (a receive loop's latency).
        {"name": "pulse_plan", "kind": "batch", "plan": True, "n_pulses": 1, "n_min": 4096, "n_max": 4096,
         "fs": 10e6, "mode": "windowed", "carrier": False},
        # The same pulse with the exact finite sum of Eq. 17.
        {"name": "pulse_plan_exact", "kind": "batch", "plan": True, "n_pulses": 1, "n_min": 4096, "n_max": 4096,
         "fs": 10e6, "mode": "exact_fp32", "carrier": False},
        # The paper's own sizes: one RF pulse of 2^19 samples, resampled ...
        {"name": "resample_rf", "kind": "resample", "n": 1 << 19, "fs": 2.048e9, "fc": 0.0, "mode": "windowed"},
        # ... and corrected (every bin's phase evaluated in full).
        {"name": "iono_rf", "kind": "iono", "n": 1 << 19, "fs": 2.048e9, "fc": 0.0, "tec": 100.0},
        # The headline Doppler bank: one pulse against 256 range rates x 16 TECs.
        {"name": "bank", "kind": "bank", "n": 65536, "n_v": 256, "n_tec": 16, "n_rep": 0},
        # A short bank of odd sizes, as a tracker refines a few hypotheses.
        {"name": "bank_odd", "kind": "bank", "n": 10001, "n_v": 33, "n_tec": 7, "n_rep": 0},
        # A bank of a long pulse (L = 2^18, beyond the fused transforms).
        {"name": "bank_long", "kind": "bank", "n": 200000, "n_v": 24, "n_tec": 4, "n_rep": 0},
        # Correction bundled with pulse compression against a 4096-sample LFM.
        {"name": "bank_compress", "kind": "bank", "n": 30000, "n_v": 96, "n_tec": 8, "n_rep": 4096},
        # The uneven batch: 4096 pulses of 1024 .. 262144 samples in one plan.
        {"name": "batch", "kind": "batch", "plan": True, "n_pulses": 4096, "n_min": 1024, "n_max": 262144,
         "fs": 20e6, "mode": "windowed", "carrier": False},
        # A small batch of short pulses by a direct call, passband dilation.
        {"name": "batch_short", "kind": "batch", "plan": False, "n_pulses": 96, "n_min": 100, "n_max": 4096,
         "fs": 20e6, "mode": "windowed", "carrier": True},
        # Exact-sinc resampling of many pulses per range rate, split precision
        # (512 distinct 8192-sample pulses for each range rate).
        {"name": "exact_split", "kind": "exact", "n": 8192, "n_pulses": 512, "n_v": 16, "mode": "exact_bf16x3"},
        # The same in FP32, fewer and shorter pulses.
        {"name": "exact_fp32", "kind": "exact", "n": 4096, "n_pulses": 48, "n_v": 8, "mode": "exact_fp32"},
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    """Log-uniform integer in [lo, hi]; odd sizes come as they fall."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    kind = rng.choice(["pulse", "resample", "iono", "bank", "bank", "compress", "batch", "batch", "exact", "exact"])
    if kind == "pulse":
        mode = rng.choice(["windowed", "exact_fp32"])
        n = _log_int(rng, 1024, 16384)
        return {"kind": "batch", "plan": True, "n_pulses": 1, "n_min": n, "n_max": n, "fs": 10e6, "mode": mode,
                "carrier": rng.random() < 0.3}
    if kind == "resample":
        if rng.random() < 0.3:      # exact sum of a single pulse
            return {"kind": "resample", "n": _log_int(rng, 2048, 32768), "fs": 20e6, "fc": 1e9, "mode": "exact_fp32"}
        return {"kind": "resample", "n": _log_int(rng, 4096, 1 << 20), "fs": 20e6, "fc": 1e9, "mode": "windowed"}
    if kind == "iono":
        n, tec = _log_int(rng, 1024, 1 << 20), rng.uniform(-150.0, 150.0)
        rf = rng.random() < 0.4
        return {"kind": "iono", "n": n, "fs": 2.048e9 if rf else 20e6, "fc": 0.0 if rf else 1e9, "tec": tec}
    if kind in ("bank", "compress"):
        n = _log_int(rng, 1024, 262144)
        # at most the listed bank's samples
        pairs = max(1, min(4096, (1 << 28) // n))
        n_tec = _log_int(rng, 1, min(16, pairs))
        n_v = _log_int(rng, 1, max(1, min(256, pairs // n_tec)))
        n_rep = _log_int(rng, 64, n) if kind == "compress" else 0
        return {"kind": "bank", "n": n, "n_v": n_v, "n_tec": n_tec, "n_rep": n_rep}
    if kind == "batch":
        n_max = _log_int(rng, 2048, 262144)
        n_min = _log_int(rng, 64, n_max)
        return {"kind": "batch", "plan": rng.random() < 0.5, "n_pulses": _log_int(rng, 2, 512), "n_min": n_min,
                "n_max": n_max, "fs": 20e6, "mode": "windowed", "carrier": rng.random() < 0.3}
    mode = rng.choice(["exact_fp32", "exact_bf16x3", "exact_fp16x3"])
    if mode == "exact_fp32":
        return {"kind": "exact", "n": _log_int(rng, 256, 4096), "n_pulses": _log_int(rng, 1, 64),
                "n_v": _log_int(rng, 1, 8), "mode": mode}
    return {"kind": "exact", "n": _log_int(rng, 512, 8192), "n_pulses": _log_int(rng, 8, 512),
            "n_v": _log_int(rng, 1, 16), "mode": mode}


# ------------------------------------------------------------------- inputs

def _gen(seed: int) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed(20250807 + int(seed))
    return g


def _noise(n: int, g: torch.Generator, rows: int = 1) -> torch.Tensor:
    """[rows, n] band-limited noise (|f| <= 0.8 fs / 2), unit power, complex64."""
    w = torch.randn((rows, n), dtype=torch.complex64, device="cuda", generator=g)
    spec = torch.fft.fft(w)
    spec[:, torch.fft.fftfreq(n, device="cuda").abs() > 0.4] = 0.0
    x = torch.fft.ifft(spec)
    return x / x.abs().square().mean(-1, keepdim=True).sqrt()


def _lfm(n: int, fs: float, bandwidth: float) -> torch.Tensor:
    t = torch.arange(n, dtype=torch.float64, device="cuda") / fs - 0.5 * n / fs
    phase = math.pi * (bandwidth * fs / n) * t * t
    return torch.polar(torch.ones_like(phase), phase).to(torch.complex64)


def _rf_lfm(n: int, fs: float, g: torch.Generator) -> torch.Tensor:
    """RF samples of an LFM at 413 MHz, 18 MHz wide, 100 us long (its start
    phase and level drawn), zero past its end."""
    u = torch.rand(2, dtype=torch.float64, device="cuda", generator=g).cpu().tolist()
    t = torch.arange(n, dtype=torch.float64, device="cuda") / fs
    T = min(100e-6, n / fs)
    phase = 2 * math.pi * ((413e6 - 9e6) * t + 0.5 * (18e6 / T) * t * t + u[0])
    x = torch.polar(torch.full_like(phase, 0.5 + u[1]), torch.remainder(phase, 2 * math.pi))
    return torch.where(t < T, x, torch.zeros_like(x)).to(torch.complex64)


def _uniform(k: int, lo: float, hi: float, g: torch.Generator) -> np.ndarray:
    return (lo + (hi - lo) * torch.rand(k, dtype=torch.float64, device="cuda", generator=g)).cpu().numpy()


def _lengths(case) -> np.ndarray:
    if case["n_min"] == case["n_max"]:
        return np.full(case["n_pulses"], case["n_min"], dtype=np.int64)
    u = np.random.Generator(np.random.PCG64(BATCH_SHAPE_SEED)).uniform(
        math.log(case["n_min"]), math.log(case["n_max"]), case["n_pulses"])
    return np.clip(np.round(np.exp(u)).astype(np.int64), case["n_min"], case["n_max"])


def _batch_inputs(case, seed):
    """Concatenated pulses, half LFM (B up to half of fs) and half slices of
    band-limited noise, their items and lengths."""
    g = _gen(seed)
    lens = _lengths(case)
    offs = np.concatenate([[0], np.cumsum(lens)])
    total, p, fs = int(offs[-1]), len(lens), case["fs"]
    n_d = torch.from_numpy(lens).cuda()
    which = torch.repeat_interleave(torch.arange(p, device="cuda"), n_d)
    i = torch.arange(total, device="cuda") - torch.from_numpy(offs[:-1]).cuda()[which]
    is_lfm = torch.ones(1, device="cuda") > 0 if p == 1 else torch.rand(p, device="cuda", generator=g) < 0.5
    bw = 0.05 + 0.45 * torch.rand(p, dtype=torch.float64, device="cuda", generator=g)      # of fs
    nf = n_d.to(torch.float64)
    t = i.to(torch.float64) - 0.5 * nf[which]
    phase = math.pi * (bw / nf)[which] * t * t
    x = torch.polar(torch.ones_like(phase), torch.remainder(phase, 2 * math.pi)).to(torch.complex64)
    del t, phase, i
    if p > 1:
        m = 1 << (total - 1).bit_length()
        x = torch.where(is_lfm[which], x, _noise(m, g)[0, :total])
    del which
    items = np.zeros(p, dtype=dc.ITEM_DTYPE)
    items["in_off"], items["out_off"], items["n"], items["n_out"] = offs[:-1], offs[:-1], lens, lens
    items["fs"], items["fc"] = fs, 1e9
    items["v_r"], items["tec_tecu"] = _uniform(p, -8000.0, 8000.0, g), _uniform(p, 5.0, 150.0, g)
    return x, items


def _inputs(case, seed) -> dict:
    g = _gen(seed)
    kind = case["kind"]
    if kind == "batch":
        x, items = _batch_inputs(case, seed)
        return {"x": x, "items": items}
    if kind in ("resample", "iono"):
        x = _rf_lfm(case["n"], case["fs"], g) if case["fc"] == 0.0 else _noise(case["n"], g)[0]
        return {"x": x, "v": float(_uniform(1, -8000.0, 8000.0, g)[0])}
    if kind == "bank":
        s = {"x": _noise(case["n"], g)[0], "v": _uniform(case["n_v"], -8000.0, 8000.0, g),
             "tec": _uniform(case["n_tec"], 5.0, 150.0, g)}
        if case["n_rep"]:
            s["rep"] = _lfm(case["n_rep"], 20e6, 5e6)
        return s
    x = torch.empty((case["n_v"], case["n_pulses"], case["n"]), dtype=torch.complex64, device="cuda")
    for a in range(case["n_v"]):
        x[a] = _noise(case["n"], g, case["n_pulses"])
    return {"x": x, "v": _uniform(case["n_v"], -8000.0, 8000.0, g)}


_shared = []      # the context a program makes once and uses for its direct calls


def _context() -> dc.Context:
    if not _shared:
        dc.load()
        _shared.append(dc.Context(0))
    return _shared[0]


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    if kind == "batch":
        s["out"] = torch.empty_like(s["x"])
        if case["plan"]:
            s["ctx"] = dc.Context(0)
            # the plan's own recording runs on another stream
            torch.cuda.synchronize()
            s["plan"] = dc.dc_plan_batch(s["ctx"], s["x"], s["out"], s["items"], mode=MODES[case["mode"]],
                                         carrier_shift=case["carrier"])
            return s
    elif kind in ("resample", "iono"):
        s["out"] = torch.empty_like(s["x"])
    elif kind == "bank":
        s["out"] = torch.empty((case["n_v"], case["n_tec"], case["n"]), dtype=torch.complex64, device="cuda")
    else:
        s["out"] = torch.empty_like(s["x"])
    s["ctx"] = _context()
    return s


def run(s):
    case, ctx, x, out = s["case"], s["ctx"], s["x"], s["out"]
    kind = case["kind"]
    if kind == "batch":
        if case["plan"]:
            dc.dc_plan_execute(s["plan"])
        else:
            dc.correct_batch(ctx, x, out, s["items"], mode=MODES[case["mode"]], carrier_shift=case["carrier"])
    elif kind == "resample":
        dc.doppler_resample(ctx, x, out, case["fs"], case["fc"], s["v"], mode=MODES[case["mode"]])
    elif kind == "iono":
        dc.iono_correct(ctx, x, out, case["fs"], case["fc"], case["tec"])
    elif kind == "bank":
        if case["n_rep"]:
            dc.correct_compress_bank(ctx, x, s["rep"], s["v"], s["tec"], out, 20e6, 1e9)
        else:
            dc.correct_bank(ctx, x, s["v"], s["tec"], out, 20e6, 1e9)
    else:
        dc.resample_exact_batch(ctx, x, case["n"], case["n_pulses"], s["v"], out,
                                x_alpha_stride=case["n_pulses"] * case["n"], mode=MODES[case["mode"]])
    return out


# --------------------------------------------------------------------- work

def _fft_flops(n: int) -> float:
    L = 1 << max(0, n - 1).bit_length()
    return 5.0 * L * max(1, L.bit_length() - 1)


def _resample_flops(n: int, mode: str) -> float:
    # windowed: 32 complex-by-real multiply-adds per output; the exact sum is a
    # band-limited interpolation, which costs no more than a few transforms
    return 4.0 * 32 * n if mode == "windowed" else 4 * _fft_flops(2 * n)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        lens = [int(n) for n in _lengths(case)]
        return {"bytes": 16.0 * sum(lens),
                "flops": sum(_resample_flops(n, case["mode"]) + 2 * _fft_flops(n) + 6.0 * n for n in lens)}
    if kind == "resample":
        return {"bytes": 16.0 * case["n"], "flops": _resample_flops(case["n"], case["mode"])}
    if kind == "iono":
        return {"bytes": 16.0 * case["n"], "flops": 2 * _fft_flops(case["n"]) + 6.0 * case["n"]}
    if kind == "bank":
        n, n_v, n_tec = case["n"], case["n_v"], case["n_tec"]
        return {"bytes": 8.0 * (n + case["n_rep"] + n_v * n_tec * n),
                "flops": n_v * (_resample_flops(n, "windowed") + _fft_flops(n)) +
                n_v * n_tec * (_fft_flops(n) + 6.0 * n)}
    pulses = case["n_v"] * case["n_pulses"]
    return {"bytes": 16.0 * pulses * case["n"], "flops": pulses * _resample_flops(case["n"], case["mode"])}


# ------------------------------------------------------- the method, 64 bits

def _delta(v: float) -> float:
    b = v / C_LIGHT
    return 2.0 * b / (1.0 - b)


def _kaiser(u: torch.Tensor) -> torch.Tensor:
    r = (u / 16.0).square()
    return torch.special.i0(8.0 * (1.0 - r).clamp_min(0.0).sqrt()) / float(np.i0(8.0))


def _windowed64(x: torch.Tensor, i: torch.Tensor, d, base, n) -> torch.Tensor:
    """sum_k x[m + k] h(t - m - k) at t = (1 + d) i for outputs i (tensor), of
    pulses that lie at `base` .. `base + n` of the flat x."""
    drift = i.to(torch.float64) * d
    fl = torch.floor(drift)
    e = drift - fl
    m = i + fl.to(torch.int64)
    sn = torch.sin(math.pi * e) / math.pi
    y = torch.zeros(i.shape, dtype=torch.complex128, device="cuda")
    for k in range(-15, 17):
        u = e - k
        w = torch.where(u == 0, torch.ones_like(u), (sn if k % 2 == 0 else -sn) / u) * _kaiser(u)
        idx = m + k
        ok = (idx >= 0) & (idx < n)
        y += torch.where(ok, x[(base + idx).clamp(0, x.numel() - 1)], torch.zeros((), dtype=x.dtype, device="cuda")) * w
    return y


def _exact64(x: torch.Tensor, d: float) -> torch.Tensor:
    """sum_m x[..., m] sinc((1 + d) n - m) for rows x [p, n]."""
    n = x.shape[-1]
    i = torch.arange(n, dtype=torch.float64, device="cuda")
    fl = torch.floor(i * d)
    e = i * d - fl
    xr = torch.view_as_real(x.to(torch.complex128)).movedim(-1, 0).reshape(-1, n)     # re rows, im rows
    par = 1.0 - 2.0 * torch.remainder(i, 2.0)
    y = torch.empty_like(xr)
    for a in range(0, n, 4096):
        b = slice(a, min(n, a + 4096))
        u = (i[b] + fl[b])[:, None] - i[None, :] + e[b][:, None]
        s = torch.sin(math.pi * e[b]) / math.pi * (1.0 - 2.0 * torch.remainder(i[b] + fl[b], 2.0))
        S = torch.where(u == 0, torch.ones_like(u), s[:, None] * par[None, :] / u)
        y[:, b] = xr @ S.T
    h = y.shape[0] // 2
    return torch.complex(y[:h], y[h:])


def _phase64(L: int, fs: float, fc: float, tec: float) -> torch.Tensor:
    f = fc + torch.fft.fftfreq(L, dtype=torch.float64, device="cuda") * fs
    a = 4 * math.pi * KAPPA * tec * 1e16 / C_LIGHT
    phi = torch.where(f != 0, a / torch.where(f != 0, f, torch.ones_like(f)), torch.zeros_like(f))
    return torch.polar(torch.ones_like(phi), -phi)


def _iono64(y: torch.Tensor, fs: float, fc: float, tec: float) -> torch.Tensor:
    n = y.shape[-1]
    L = 1 << (n - 1).bit_length()
    return torch.fft.ifft(torch.fft.fft(y, n=L) * _phase64(L, fs, fc, tec))[..., :n]


def exact(case, seed):
    s = _inputs(case, seed)
    kind, x = case["kind"], s["x"]
    if kind == "batch":
        x64, items = x.to(torch.complex128), s["items"]
        if case["mode"] == "exact_fp32":
            y = torch.cat([_exact64(x[None, int(it["in_off"]):int(it["in_off"] + it["n"])], _delta(it["v_r"]))[0]
                           for it in items])
        else:
            lens = torch.from_numpy(items["n"].copy()).cuda()
            which = torch.repeat_interleave(torch.arange(len(items), device="cuda"), lens)
            base = torch.from_numpy(items["in_off"].copy()).cuda()
            d = torch.tensor([_delta(v) for v in items["v_r"]], dtype=torch.float64, device="cuda")
            y = torch.empty_like(x64)
            for a in range(0, x.numel(), 1 << 25):
                w = which[a:a + (1 << 25)]
                i = torch.arange(a, a + w.numel(), device="cuda") - base[w]
                y[a:a + w.numel()] = _windowed64(x64, i, d[w], base[w], lens[w])
        for it in items:
            o, n = int(it["in_off"]), int(it["n"])
            z = y[o:o + n]
            if case["carrier"]:
                cyc = it["fc"] * _delta(it["v_r"]) / it["fs"] * torch.arange(n, dtype=torch.float64, device="cuda")
                cyc = cyc - torch.round(cyc)
                z = z * torch.polar(torch.ones_like(cyc), 2 * math.pi * cyc)
            y[o:o + n] = _iono64(z, it["fs"], it["fc"], it["tec_tecu"])
        return y
    if kind == "iono":
        return _iono64(x.to(torch.complex128), case["fs"], case["fc"], case["tec"])
    if kind == "resample":
        if case["mode"] != "windowed":
            return _exact64(x[None], _delta(s["v"]))[0]
        return _windowed64(x.to(torch.complex128), torch.arange(case["n"], device="cuda"), _delta(s["v"]), 0, case["n"])
    if kind == "exact":
        return torch.stack([_exact64(x[a], _delta(float(s["v"][a]))) for a in range(case["n_v"])])
    n = case["n"]
    L = 1 << (n - 1).bit_length()
    fac = torch.stack([_phase64(L, 20e6, 1e9, float(t)) for t in s["tec"]])
    if case["n_rep"]:
        fac = fac * torch.fft.fft(s["rep"].to(torch.complex128), n=L).conj()
    out = torch.empty((case["n_v"], case["n_tec"], n), dtype=torch.complex128, device="cuda")
    i, x64 = torch.arange(n, device="cuda"), x.to(torch.complex128)
    for a in range(case["n_v"]):
        out[a] = torch.fft.ifft(torch.fft.fft(_windowed64(x64, i, _delta(float(s["v"][a])), 0, n), n=L) * fac)[..., :n]
    return out

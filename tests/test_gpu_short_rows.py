"""Transforms of 256 to 2048 points in registers (16, 8, 4, 2 per CTA) against
the FP64 oracle: lengths at the classes' edges, partly filled CTAs, several
classes in one launch, stored spectra with factor tables (banks) and caller
tables (compression).

Tolerance: FP32 transforms of at most 11 radix-2 levels each way with twiddles
of a few roundings, plus the reduced phase (4e-7): 2e-6 holds both.
"""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
FS, FC, TOL = 20e6, 1e9, 2e-6
SIZES = [128, 129, 255, 256, 257, 511, 512, 513, 1000, 1024, 1025, 2047, 2048]


@pytest.fixture(scope="module")
def dcg():
    import paper_2508_04951_gb300 as m
    m.build.build()
    m.load()
    return m


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n", SIZES)
def test_one_pulse(dcg, n):
    import torch
    x = synth.bandlimited_noise(n, synth.rng_for(1, salt=n)).astype(np.complex64)
    ctx = dcg.Context(0)
    xd = torch.from_numpy(x).cuda()
    for fs, fc, tec in ((FS, FC, 120.0), (FS, FC, -90.0), (2.048e9, 0.0, 100.0), (FS, FC, 0.0)):
        y = torch.full((n + 8,), 3.0, dtype=torch.complex64, device="cuda")
        dcg.iono_correct(ctx, xd, y[:n], fs, fc, tec)
        dcg.dc_check(ctx)
        got = y.cpu().numpy()
        assert np.all(got[n:] == 3.0)
        assert rel(got[:n], oracle.iono_correct(x.astype(np.complex128), fs, fc, tec)) <= TOL, (fs, tec)
    ctx.close()


@pytest.mark.parametrize("copies", [1, 3, 17])
def test_classes_of_a_batch(dcg, copies):
    import torch
    lens = np.array([n for n in SIZES + [1, 2, 7, 16, 33, 100, 3000, 4096] for _ in range(copies)], dtype=np.int64)
    rng = synth.rng_for(3, salt=copies)
    offs = np.concatenate([[0], np.cumsum(lens)])
    x = synth.bandlimited_noise(int(offs[-1]), rng).astype(np.complex64)
    items = np.zeros(len(lens), dtype=dcg.ITEM_DTYPE)
    items["in_off"] = items["out_off"] = offs[:-1]
    items["n"] = items["n_out"] = lens
    items["fs"], items["fc"] = FS, FC
    items["v_r"], items["tec_tecu"] = rng.uniform(-8000, 8000, len(lens)), rng.uniform(5, 150, len(lens))
    ctx = dcg.Context(0)
    y = torch.empty(len(x), dtype=torch.complex64, device="cuda")
    dcg.correct_batch(ctx, torch.from_numpy(x).cuda(), y, items)
    dcg.dc_check(ctx)
    y = y.cpu().numpy()
    for it in items:
        o, n = int(it["in_off"]), int(it["n"])
        ref = oracle.correct(x[o:o + n].astype(np.complex128), FS, FC, it["v_r"], it["tec_tecu"])
        assert rel(y[o:o + n], ref) <= TOL, n
    ctx.close()


@pytest.mark.parametrize("n", [200, 256, 500, 1000, 1025, 2048])
def test_spectra_and_tables(dcg, n):
    import torch
    rng = synth.rng_for(2, salt=n)
    x = synth.bandlimited_noise(n, rng).astype(np.complex64)
    h = synth.lfm(n // 3, FS, 5e6).astype(np.complex64)
    v, tec = rng.uniform(-8000, 8000, 5), rng.uniform(5, 150, 3)
    ctx = dcg.Context(0)
    xd, hd = torch.from_numpy(x).cuda(), torch.from_numpy(h).cuda()
    out = torch.empty((5, 3, n), dtype=torch.complex64, device="cuda")
    dcg.correct_bank(ctx, xd, v, tec, out, FS, FC)
    ref = oracle.correct_bank(x.astype(np.complex128), FS, FC, v, tec)
    dcg.dc_check(ctx)
    assert rel(out.cpu().numpy(), ref) <= TOL
    L = 1 << (n - 1).bit_length()
    H = np.fft.fft(h.astype(np.complex128), L).conj()

    def compressed(vr, t):
        y = oracle.resample(x.astype(np.complex128), FS, FC, vr)
        return np.fft.ifft(np.fft.fft(y, L) * np.exp(-1j * oracle.iono_phase(L, FS, FC, t)) * H)[:n]

    dcg.correct_compress_bank(ctx, xd, hd, v, tec, out, FS, FC)
    one = torch.empty(n, dtype=torch.complex64, device="cuda")
    dcg.correct_compress(ctx, xd, hd, one, FS, FC, float(v[1]), float(tec[2]))
    dcg.dc_check(ctx)
    got = out.cpu().numpy()
    for i in range(5):
        for t in range(3):
            assert rel(got[i, t], compressed(v[i], tec[t])) <= TOL
    assert rel(one.cpu().numpy(), compressed(v[1], tec[2])) <= TOL
    ctx.close()

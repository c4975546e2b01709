"""Transforms of 1 to 128 points (a thread, or 2 to 8 threads, each) against the
FP64 oracle: every size class, counts about a CTA's, stored spectra with factor
tables (banks), caller tables (compression), and dependent calls back to back
(each may start while the one before still runs).

Tolerance: FP32 transforms of at most 7 radix-2 levels each way and the reduced
phase (4e-7): 2e-6 holds both; the bank's resampling adds its weights' 2e-7.
"""

import numpy as np
import pytest

import oracle
import oracle.compression
import synth

pytestmark = pytest.mark.gpu
FS, FC, TOL = 20e6, 1e9, 2e-6
SIZES = [1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 31, 32, 33, 60, 64, 65, 100, 127, 128]


@pytest.fixture(scope="module")
def dcg():
    import paper_2508_04951_gb300 as m
    m.build.build()
    m.load()
    return m


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def noise(n, salt):
    g = np.random.default_rng(salt)
    return (g.standard_normal(n) + 1j * g.standard_normal(n)).astype(np.complex64)


@pytest.mark.parametrize("n", SIZES)
def test_one_pulse(dcg, n):
    import torch
    ctx = dcg.Context(0)
    x = noise(n, n)
    xd = torch.from_numpy(x).cuda()
    for fs, fc, tec in ((FS, FC, 120.0), (2.048e9, 0.0, -80.0), (FS, FC, 0.0)):
        y = torch.full((n + 8,), 3.0, dtype=torch.complex64, device="cuda")
        dcg.iono_correct(ctx, xd, y[:n], fs, fc, tec)
        dcg.dc_check(ctx)
        got = y.cpu().numpy()
        assert np.all(got[n:] == 3.0)
        assert rel(got[:n], oracle.iono_correct(x.astype(np.complex128), fs, fc, tec)) <= TOL, (fs, tec)
    ctx.close()


@pytest.mark.parametrize("count", [31, 33, 64, 129, 257])
def test_counts(dcg, count):
    import torch
    lens = np.array([n for n in (1, 7, 16, 30, 50, 128) for _ in range(count)], dtype=np.int64)
    offs = np.concatenate([[0], np.cumsum(lens)])
    x = noise(int(offs[-1]), count)
    items = np.zeros(len(lens), dtype=dcg.ITEM_DTYPE)
    items["in_off"] = items["out_off"] = offs[:-1]
    items["n"] = items["n_out"] = lens
    items["fs"], items["fc"], items["v_r"] = FS, FC, 0.0
    items["tec_tecu"] = np.linspace(-150.0, 150.0, len(lens))
    ctx = dcg.Context(0)
    xd = torch.from_numpy(x).cuda()
    y = torch.full((len(x) + 8,), 3.0, dtype=torch.complex64, device="cuda")
    dcg.correct_batch(ctx, xd, y[:len(x)], items)
    dcg.dc_check(ctx)
    got = y.cpu().numpy()
    assert np.all(got[len(x):] == 3.0)
    for i, n in enumerate(lens):
        p = slice(offs[i], offs[i + 1])
        ref = oracle.iono_correct(x[p].astype(np.complex128), FS, FC, items["tec_tecu"][i])
        assert rel(got[p], ref) <= TOL, (i, n)
    ctx.close()


@pytest.mark.parametrize("n", SIZES)
def test_bank_and_compression(dcg, n):
    import torch
    ctx = dcg.Context(0)
    x, rep = noise(n, 100 + n), noise(max(1, n // 3), n)
    xd, rd = torch.from_numpy(x).cuda(), torch.from_numpy(rep).cuda()
    v, t = [0.0, 5000.0, -7000.0], [20.0, 0.0, -90.0, 140.0]
    y = torch.full((len(v) * len(t) * n + 8,), 3.0, dtype=torch.complex64, device="cuda")
    x64, r64 = x.astype(np.complex128), rep.astype(np.complex128)
    for compress in (False, True):
        out = y[:-8].view(len(v), len(t), n)
        if compress:
            dcg.correct_compress_bank(ctx, xd, rd, v, t, out, FS, FC)
            ref = oracle.compression.correct_compress_bank(x64, r64, FS, FC, v, t)
        else:
            dcg.correct_bank(ctx, xd, v, t, out, FS, FC)
            ref = oracle.correct_bank(x64, FS, FC, v, t)
        dcg.dc_check(ctx)
        assert np.all(y[-8:].cpu().numpy() == 3.0)
        got = out.cpu().numpy()
        for i in range(len(v)):
            for k in range(len(t)):
                r = np.asarray(ref[i][k])[:n]
                assert np.linalg.norm(got[i, k] - r) <= TOL * max(np.linalg.norm(r), np.linalg.norm(ref)), (i, k)
    ctx.close()


@pytest.mark.parametrize("n", [16, 100, 1000, 4096])
def test_dependent_calls(dcg, n):
    import torch
    ctx = dcg.Context(0)
    a = torch.from_numpy(noise(n, n)).cuda()
    b, c = torch.empty_like(a), torch.empty_like(a)
    outs = []
    for wait in (True, False):
        x = a.clone()
        torch.cuda.synchronize()
        for i in range(40):
            for s, d, tec in ((x, b, 30.0), (b, c, -50.0), (c, x, 20.0 + i)):
                dcg.iono_correct(ctx, s, d, FS, FC, tec)
                if wait:
                    torch.cuda.synchronize()
            dcg.doppler_resample(ctx, x, b, FS, FC, 100.0)
            x, b = b, x
        dcg.dc_check(ctx)
        outs.append(x.cpu().numpy())
    assert np.array_equal(outs[0], outs[1])
    ctx.close()

"""Distance of the corrections from 64 bits, over enough samples that it is steady to
a per cent.  Bounds: what the transforms had with one table value, rounded once,
for every twiddle and a factor angle rounded once, and 5 %.
"""

import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
TEC = 100.0


@pytest.fixture(scope="module")
def dcg():
    import paper_2508_04951_gb300 as m
    m.build.build()
    m.load()
    return m


def corrected64(x, fs, fc, tec):
    """Eq. 16 in 64 bits for rows x [p, n]."""
    import torch
    n = x.shape[-1]
    L = 1 << (n - 1).bit_length()
    phi = torch.from_numpy(oracle.iono_phase(L, fs, fc, tec)).to(x.device)
    return torch.fft.ifft(torch.fft.fft(x.to(torch.complex128), n=L) * torch.polar(torch.ones_like(phi), -phi))[..., :n]


def noise(rows, n):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    return torch.randn((rows, n), dtype=torch.complex64, device="cuda", generator=g)


def batch_error(dcg, n, pulses, fs, fc):
    import torch
    ctx = dcg.Context(0)
    x = noise(pulses, n)
    y = torch.empty_like(x)
    items = np.zeros(pulses, dtype=dcg.ITEM_DTYPE)
    items["in_off"] = items["out_off"] = np.arange(pulses) * n
    items["n"] = items["n_out"] = n
    items["fs"], items["fc"], items["tec_tecu"] = fs, fc, TEC
    # v_r = 0: frequency conversion copies the pulse as it is
    dcg.correct_batch(ctx, x.view(-1), y.view(-1), items, mode=dcg.DC_FREQCONV)
    dcg.dc_check(ctx)
    ctx.close()
    ref = corrected64(x, fs, fc, TEC)
    return float((y.to(torch.complex128) - ref).norm() / ref.norm())


# pulses of up to 2048 samples: lengths of each split (R x 16, 16 x A x 16), padded and whole
@pytest.mark.parametrize("n,pulses,baseband,rf", [
    (64, 2048, 2.08e-7, 2.35e-7), (100, 2048, 2.11e-7, 2.36e-7), (256, 1024, 2.33e-7, 2.44e-7),
    (300, 1024, 2.08e-7, 2.44e-7), (700, 512, 2.20e-7, 2.53e-7), (2048, 256, 2.56e-7, 2.58e-7)])
def test_short_pulses(dcg, n, pulses, baseband, rf):
    assert batch_error(dcg, n, pulses, 20e6, 1e9) <= 1.05 * baseband
    assert batch_error(dcg, n, pulses, 2.048e9, 0.0) <= 1.05 * rf


# the factors' share: nothing but a factor and a DFT in registers, and banks' tables
@pytest.mark.parametrize("n,pulses,baseband,rf", [(16, 8192, 1.76e-7, 2.27e-7), (31, 4096, 1.98e-7, 2.53e-7)])
def test_tiny_pulses(dcg, n, pulses, baseband, rf):
    assert batch_error(dcg, n, pulses, 20e6, 1e9) <= 1.05 * baseband
    assert batch_error(dcg, n, pulses, 2.048e9, 0.0) <= 1.05 * rf


@pytest.mark.parametrize("n,n_tec,bound", [(200, 16, 2.25e-7), (1024, 16, 2.47e-7), (10001, 8, 2.83e-7),
                                           (65536, 16, 3.30e-7), (100000, 8, 3.06e-7), (200000, 4, 3.11e-7)])
def test_banks(dcg, n, n_tec, bound):
    import torch
    ctx = dcg.Context(0)
    x = noise(1, n)
    y = torch.empty((2, n_tec, n), dtype=torch.complex64, device="cuda")
    tec = np.linspace(5.0, 150.0, n_tec)
    dcg.correct_bank(ctx, x.view(-1), np.zeros(2), tec, y.view(-1), 20e6, 1e9, mode=dcg.DC_FREQCONV)
    dcg.dc_check(ctx)
    ctx.close()
    ref = torch.cat([corrected64(x, 20e6, 1e9, t) for t in tec])
    for v in range(2):
        assert float((y[v].to(torch.complex128) - ref).norm() / ref.norm()) <= 1.05 * bound


def test_long_rf_pulse(dcg):
    # 100 us of an 18 MHz LFM at 413 MHz in 2^19 samples: its energy lies in few bins,
    # so that the middle rows' twiddles do not average out (3.54e-7)
    import torch
    n, fs = 1 << 19, 2.048e9
    t = torch.arange(n, dtype=torch.float64, device="cuda") / fs
    phase = 2 * math.pi * (404e6 * t + 0.5 * (18e6 / 100e-6) * t * t)
    x = torch.where(t < 100e-6, torch.polar(torch.ones_like(t), phase), torch.zeros_like(phase)).to(torch.complex64)[None]
    y = torch.empty_like(x)
    ctx = dcg.Context(0)
    dcg.iono_correct(ctx, x.view(-1), y.view(-1), fs, 0.0, TEC)
    dcg.dc_check(ctx)
    ctx.close()
    ref = corrected64(x, fs, 0.0, TEC)
    assert float((y.to(torch.complex128) - ref).norm() / ref.norm()) <= 1.02 * 3.54e-7

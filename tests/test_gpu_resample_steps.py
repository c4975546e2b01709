"""The windowed resampler where floor(delta n) steps inside a warp's tile of
outputs (128 or 256): both directions, steps at and beside the tile's edges, the
pulse's ends, odd offsets, samples that are not finite, and the weights' tables
of more than one window.

Tolerance: FP32 sums of 32 products whose weights hold about 2e-7 each: 2e-6.
An output may differ in finiteness from the definition only where its position
lies within 1e-6 of an input's: the support's two ends change there.
"""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
FS, FC, C, TOL = 20e6, 1e9, 299792458.0, 2e-6


@pytest.fixture(scope="module")
def dcg():
    import paper_2508_04951_gb300 as m
    m.build.build()
    m.load()
    return m


def speed(delta):
    """v_r whose dilation alpha - 1 = 2 b / (1 - b) is delta."""
    return C * delta / (2.0 + delta)


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def run(m, x, n_out, v, off=0, **kw):
    import torch
    ctx = m.Context(0)
    xd = torch.zeros(len(x) + off, dtype=torch.complex64, device="cuda")
    xd[off:] = torch.from_numpy(x).cuda()
    y = torch.full((n_out + off + 8,), 3.0, dtype=torch.complex64, device="cuda")
    m.doppler_resample(ctx, xd[off:], y[off:off + n_out], FS, FC, v, n_out=n_out, **kw)
    m.dc_check(ctx)
    got = y.cpu().numpy()
    ctx.close()
    assert np.all(got[:off] == 3.0) and np.all(got[off + n_out:] == 3.0)
    return got[off:off + n_out]


# The first output past a step: at, beside and between the edges of the tiles of
# 256 outputs (17408 = 68 x 256, 8 outputs per lane) and of 128 (9472 = 74 x 128,
# 4 per lane); a step every few hundred outputs takes exact weights.
FIRST = [17408 + k for k in (0, 1, 2, 100, 127, 128, 255)] + [9472 + k for k in (0, 1, 64, 127)] + [150, 400]


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("first", FIRST)
def test_steps(dcg, first, sign):
    v = speed(sign / (first - 0.5))
    for n, n_out, off in ((first + 300, first + 300, 0), (first + 20, first + 400, 1), (first + 600, first + 5, 1)):
        x = synth.bandlimited_noise(n, synth.rng_for(1, salt=n)).astype(np.complex64)
        ref = oracle.resample_windowed(x.astype(np.complex128), oracle.alpha(v), n_out)
        # on an input (up to FP64's rounding, which leaves the oracle's sin(pi
        # frac) few digits there) the output is that input
        t = oracle.alpha(v) * np.arange(n_out)
        at = (np.abs(t - np.round(t)) < 1e-9) & (t < n - 0.5)
        ref[at] = x[np.round(t[at]).astype(int)]
        got = run(dcg, x, n_out, v, off)
        assert rel(got, ref) <= TOL, (n, n_out)
        near = slice(max(0, first - 300), n_out)
        assert rel(got[near], ref[near]) <= 2 * TOL, (n, n_out)


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("first", [17408 + 100, 9472 + 64, 400])
def test_not_finite(dcg, first, sign):
    n, delta = first + 500, sign / (first - 0.5)
    t = (1.0 + delta) * np.arange(n)
    m = np.floor(t).astype(np.int64)
    clear = np.abs(t - np.round(t)) > 1e-6
    inner = (t > 20) & (t < n - 20)
    for value in (np.inf, np.nan, 3e30):
        for at in range(first - 20, first + 20):
            x = np.ones(n, np.complex64)
            x[at] = value
            got = run(dcg, x, n, speed(delta))
            with_it = (m - 15 <= at) & (at <= m + 16)
            if np.isfinite(value):
                assert np.all(np.abs(got[clear & inner & ~with_it] - 1.0) < 0.05), at
            else:
                assert np.array_equal(~np.isfinite(got[clear].real), with_it[clear]), (value, at)


def test_windows_of_one_context(dcg):
    """More windows in turn than a context keeps tables for, each used twice."""
    import torch
    ctx = dcg.Context(0)
    x = synth.bandlimited_noise(1000, synth.rng_for(2)).astype(np.complex64)
    xd, y = torch.from_numpy(x).cuda(), torch.empty(1000, dtype=torch.complex64, device="cuda")
    for taps, beta in [(t, b) for t in (32, 16) for b in np.linspace(2.0, 10.0, 11)] * 2:
        dcg.doppler_resample(ctx, xd, y, FS, FC, 5000.0, taps=taps, beta=float(beta))
        dcg.dc_check(ctx)
        ref = oracle.resample_windowed(x.astype(np.complex128), oracle.alpha(5000.0), 1000, taps=taps,
                                       beta=float(beta))
        assert rel(y.cpu().numpy(), ref) <= TOL, (taps, beta)
    ctx.close()


@pytest.mark.parametrize("v", [1e-20, -1e-20, 1e-24, 1e-27, 1e-30, -1e-30, 1e-33, 1e-36, -1e-36, 1e-300])
def test_tiny_rates(dcg, v):
    """Positions within a float's smallest numbers of the inputs': the pulse itself."""
    import torch
    x = synth.bandlimited_noise(2000, synth.rng_for(3)).astype(np.complex64)
    for mode in (dcg.DC_WINDOWED, dcg.DC_EXACT_FP32):
        assert rel(run(dcg, x, 2000, v, mode=mode), x) <= TOL, mode
    ctx = dcg.Context(0)
    xd = torch.from_numpy(x).cuda().repeat(16)
    for mode in (dcg.DC_EXACT_FP32, dcg.DC_EXACT_BF16X3, dcg.DC_EXACT_FP16X3):
        y = torch.empty_like(xd)
        dcg.resample_exact_batch(ctx, xd, 2000, 16, [v], y, mode=mode)
        dcg.dc_check(ctx)
        assert rel(y.cpu().numpy().reshape(16, -1), np.tile(x, (16, 1))) <= 2e-5, mode   # split products
    y = torch.empty((3, 2, 2000), dtype=torch.complex64, device="cuda")
    dcg.correct_bank(ctx, xd[:2000], [v, 0.0, 2 * v], [50.0, 0.0], y, FS, FC)
    dcg.dc_check(ctx)
    ref = oracle.iono_correct(x.astype(np.complex128), FS, FC, 50.0)
    for i in range(3):
        assert rel(y[i, 0].cpu().numpy(), ref) <= TOL and rel(y[i, 1].cpu().numpy(), x) <= TOL
    ctx.close()

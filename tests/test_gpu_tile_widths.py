"""Dispatch rules on a call's size: the FP32 exact sum's tiles of 32 or 64 outputs
(few or many tiles in a launch) add the same terms in the same order, so that a
rate alone gives the bits it gives among others; a 65536-point bank below and
from 96 transforms (cluster or two-pass apply) agrees with the oracle.
"""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
FS, FC = 20e6, 1e9


@pytest.fixture(scope="module")
def dcg():
    import paper_2508_04951_gb300 as m
    m.build.build()
    m.load()
    return m


@pytest.mark.parametrize("n,n_out,pulses", [(300, 300, 48), (511, 700, 33), (1025, 97, 64), (1600, 1600, 40),
                                            (2100, 1999, 100), (2049, 2049, 64)])
def test_exact_tiles(dcg, n, n_out, pulses):
    import torch
    ctx = dcg.Context(0)
    x = torch.from_numpy(synth.bandlimited_noise(n * pulses, synth.rng_for(1, salt=n)).astype(np.complex64)).cuda()
    v = np.linspace(-7000.0, 8000.0, 24)
    many = torch.empty((24, pulses, n_out), dtype=torch.complex64, device="cuda")
    dcg.resample_exact_batch(ctx, x, n, pulses, v, many, n_out=n_out)
    for i in (0, 11, 23):
        one = torch.full((pulses * n_out + 8,), 3.0, dtype=torch.complex64, device="cuda")
        dcg.resample_exact_batch(ctx, x, n, pulses, v[i:i + 1], one[:-8], n_out=n_out)
        dcg.dc_check(ctx)
        assert torch.all(one[-8:] == 3.0)
        assert torch.equal(one[:-8].view(pulses, n_out), many[i]), i
    ref = oracle.resample_exact(x[:n].cpu().numpy().astype(np.complex128), oracle.alpha(v[11]), n_out)
    got = many[11, 0].cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)     # the FP32 paths' tolerance
    ctx.close()


@pytest.mark.parametrize("n_v,n_tec", [(1, 1), (19, 5), (16, 6), (8, 13)])
def test_bank_about_96_transforms(dcg, n_v, n_tec):
    import torch
    n = 40000
    ctx = dcg.Context(0)
    x = synth.bandlimited_noise(n, synth.rng_for(2)).astype(np.complex64)
    v, t = np.linspace(-7000.0, 7500.0, n_v), np.linspace(5.0, 150.0, n_tec)
    y = torch.full((n_v * n_tec * n + 8,), 3.0, dtype=torch.complex64, device="cuda")
    dcg.correct_bank(ctx, torch.from_numpy(x).cuda(), v, t, y[:-8], FS, FC)
    dcg.dc_check(ctx)
    assert torch.all(y[-8:] == 3.0)
    got = y[:-8].view(n_v, n_tec, n)
    for i, k in {(0, 0), (n_v // 2, n_tec - 1), (n_v - 1, n_tec // 2)}:
        ref = oracle.correct(x.astype(np.complex128), FS, FC, v[i], t[k])
        assert np.linalg.norm(got[i, k].cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref), (i, k)
    ctx.close()

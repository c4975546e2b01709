"""fp16x3 exact sums of pulses far below and far above one: the far field's node values
take a scale from the pulses, so that they are no further from the oracle than the dense
sum of the same planes is (a context whose scratch budget leaves no room for the far
field's).  Both quantise the samples to 2^-36; the far field adds node values to the
same spacing with weights of some 0.3, and loses most of the dense sum's
accumulator truncation: 1.1 times the dense sum's error at most.
"""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dcg():
    import paper_2508_04951_gb300 as m
    m.build.build()
    m.load()
    return m


def error(m, X, n, P, n_alpha, budget):
    import torch
    ctx = m.Context(0, budget)
    v = np.linspace(5000.0, -3000.0, n_alpha)
    xd = torch.from_numpy(X.reshape(-1)).cuda()
    yd = torch.zeros((n_alpha, P, n), dtype=torch.complex64, device="cuda")
    m.resample_exact_batch(ctx, xd, n, P, v, yd.view(-1), n_out=n, mode=m.DC_EXACT_FP16X3)
    m.dc_check(ctx)
    ctx.close()
    rows = np.unique(np.concatenate([np.arange(0, n, 61), np.arange(n - 20, n)]))
    out = []
    for a in range(n_alpha):
        ref = oracle.resample_exact_rows(X.astype(np.complex128), oracle.alpha(v[a]), rows)
        got = yd[a].cpu().numpy().astype(np.complex128)[:, rows]
        out.append(np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1))      # pulse by pulse
    return np.array(out)


@pytest.mark.parametrize("n", [2000, 4097])
@pytest.mark.parametrize("level", [1e-7, 1e-6, 1e-5, 1e-4, 1e-2, 1.0, 30.0, 1000.0, 15000.0])
def test_levels(dcg, n, level):
    P = 5
    X = np.stack([synth.bandlimited_noise(n, synth.rng_for(4, salt=n + p)) for p in range(P)]) * level
    X = X.astype(np.complex64)
    assert np.abs(X.view(np.float32)).max() < 65504
    dense = 2 * (2 * P * ((n + 7) // 8 * 8) * 2) + 512
    far, ref = error(dcg, X, n, P, 2, 0), error(dcg, X, n, P, 2, dense)
    assert np.all(far <= 1.1 * ref), (far, ref)


def test_a_tile_of_small_and_ordinary_pulses(dcg):
    # 150 pulses, two tiles of columns: those of 1e-6 beside those of one
    n, P = 2000, 150
    level = np.where(np.arange(P) % 3 == 0, 1e-6, 1.0)
    X = np.stack([synth.bandlimited_noise(n, synth.rng_for(4, salt=p)) for p in range(P)]) * level[:, None]
    X = X.astype(np.complex64)
    dense = 2 * (2 * P * n * 2) + 512
    far, ref = error(dcg, X, n, P, 1, 0), error(dcg, X, n, P, 1, dense)
    assert np.all(far <= 1.1 * ref), (far / ref).max()

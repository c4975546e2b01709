"""Exact-sinc resampling with distant blocks summed through their moments
(256-sample blocks, 16 Chebyshev nodes), against the FP64 oracle, where the
block arithmetic can go wrong: lengths about the smallest that takes this
form, partial blocks, odd lengths (rows off 16-byte boundaries), outputs
beyond the input, delays close to the 63 samples the target nodes cover and
just past them (dense sum), pulses shared across range rates.

Tolerances: bf16x3 drops the low-times-low product (2^-18 of a term, rms 4e-6
of an output) and rounds its accumulators toward zero at each of at most 57 x 6
steps (3e-8 each): 3e-5 holds both with a factor of two.  fp16x3: 2^-22, and
25 x 2 steps: 1e-5.
"""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
C_LIGHT = 299792458.0


@pytest.fixture(scope="module")
def dcg():
    import paper_2508_04951_gb300 as m
    m.build.build()
    m.load()
    return m


def v_of_delay(samples, n):
    """Range rate whose delay reaches `samples` at output n."""
    d = samples / n
    return C_LIGHT * d / (2.0 + d)


def check(dcg, ctx, mode_name, n, n_out, P, v, shared, tol):
    import torch
    rng = synth.rng_for(4, salt=n + n_out)
    G = 1 if shared else len(v)
    X = np.stack([synth.bandlimited_noise(n, rng) for _ in range(P * G)]).astype(np.complex64)
    xd = torch.from_numpy(X.reshape(-1)).cuda()
    yd = torch.full((len(v) * P * n_out + 64,), 7.0, dtype=torch.complex64, device="cuda")
    dcg.resample_exact_batch(ctx, xd, n, P, v, yd[:len(v) * P * n_out], n_out=n_out,
                             mode=getattr(dcg, mode_name), x_alpha_stride=0 if shared else P * n)
    dcg.dc_check(ctx)
    Y = yd.cpu().numpy()
    assert np.all(Y[-64:] == 7.0)
    Y = Y[:-64].astype(np.complex128).reshape(len(v), P, n_out)
    rows = np.unique(np.concatenate([np.arange(min(40, n_out)), np.arange(max(0, n_out - 40), n_out),
                                     np.arange(0, n_out, 37)]))
    X = X.astype(np.complex128).reshape(G, P, n)
    for a in range(len(v)):
        ref = oracle.resample_exact_rows(X[0 if shared else a], oracle.alpha(v[a]), rows)
        e = np.linalg.norm(Y[a][:, rows] - ref) / np.linalg.norm(ref)
        assert e <= tol, (v[a], e)


@pytest.mark.parametrize("mode_name,tol", [("DC_EXACT_BF16X3", 3e-5), ("DC_EXACT_FP16X3", 1e-5)])
@pytest.mark.parametrize("n,n_out,P,shared", [
    (1535, 1535, 3, False), (1536, 1536, 3, False), (1793, 1023, 5, True), (2303, 4100, 2, False),
    (4096, 4096, 9, True), (4097, 4097, 130, False), (5000, 300, 4, False), (8192, 8191, 3, False),
])
def test_far_field_matches_oracle(dcg, mode_name, tol, n, n_out, P, shared):
    ctx = dcg.Context(0)
    # a Doppler rate, a delay at the edge of the target nodes either way, one past it
    v = [7500.0, v_of_delay(62.9, n_out), -v_of_delay(62.9, n_out)]
    check(dcg, ctx, mode_name, n, n_out, P, v, shared, tol)
    check(dcg, ctx, mode_name, n, n_out, P, [v_of_delay(64.0, n_out), -3.0], shared, 5e-5)
    ctx.close()


def test_far_field_within_a_scratch_budget(dcg):
    # scratch capped at the dense sum's planes: the call is accepted and takes
    # the dense sum; capped below, it is refused
    n, P = 4096, 8
    dense = 2 * (2 * P * n * 2)
    ctx = dcg.Context(0, dense)
    check(dcg, ctx, "DC_EXACT_BF16X3", n, n, P, [4000.0], True, 5e-5)
    ctx.close()
    ctx = dcg.Context(0, dense - 256)
    with pytest.raises(dcg.DcError) as e:
        check(dcg, ctx, "DC_EXACT_BF16X3", n, n, P, [4000.0], True, 5e-5)
    assert e.value.status == 3
    ctx.close()

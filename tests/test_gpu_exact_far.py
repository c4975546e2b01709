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


@pytest.mark.parametrize("n,n_out,P,shared", [
    (1535, 1535, 9, False), (1536, 1536, 16, False), (1700, 2000, 17, True), (2000, 255, 40, False),
    (3001, 3001, 48, False), (1793, 1537, 65, True), (17000, 300, 10, True),   # tiles of pulses
    (4095, 4095, 1, False), (5793, 5793, 1, False), (4097, 5000, 2, False), (40001, 700, 3, True),
    (4096, 4096, 8, False), (20000, 20000, 1, False),                          # one warp per output
])
def test_far_field_fp32_matches_oracle(dcg, n, n_out, P, shared):
    # FP32 weights (2 ulp divide, sinpi) and sums of at most 4095 terms: 4e-6
    ctx = dcg.Context(0)
    v = [7500.0, v_of_delay(62.9, n_out), -v_of_delay(62.9, n_out)]
    check(dcg, ctx, "DC_EXACT_FP32", n, n_out, P, v, shared, 4e-6)
    check(dcg, ctx, "DC_EXACT_FP32", n, n_out, P, [v_of_delay(64.0, n_out), 0.0], shared, 4e-6)
    ctx.close()


@pytest.mark.parametrize("mode_name,n,P", [("DC_EXACT_FP32", 6200, 1), ("DC_EXACT_FP32", 2300, 20),
                                           ("DC_EXACT_BF16X3", 2300, 4), ("DC_EXACT_FP16X3", 2300, 4)])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, 3.3e38])
def test_far_field_keeps_values_that_are_not_finite(dcg, mode_name, n, P, bad):
    # one sample per pulse that is infinite, NaN or near the largest float: the
    # same outputs are infinite, NaN and finite as in the dense sum (a context
    # whose scratch budget leaves no room for the far field's)
    import torch
    rng = synth.rng_for(4, salt=n)
    X = np.stack([synth.bandlimited_noise(n, rng) for _ in range(P)]).astype(np.complex64)
    X[:, 300] = bad
    xd = torch.from_numpy(X.reshape(-1)).cuda()
    dense = {"DC_EXACT_FP32": 1}.get(mode_name, 2 * (2 * P * ((n + 7) // 8 * 8) * 2) + 512)
    got = []
    for budget in (0, dense):
        ctx = dcg.Context(0, budget)
        yd = torch.zeros(2 * P * n, dtype=torch.complex64, device="cuda")
        dcg.resample_exact_batch(ctx, xd, n, P, [5000.0, 0.5], yd, n_out=n, mode=getattr(dcg, mode_name))
        dcg.dc_check(ctx)
        got.append(torch.view_as_real(yd).cpu().numpy())
        ctx.close()
    far, ref = got
    np.testing.assert_array_equal(np.isnan(far), np.isnan(ref))
    np.testing.assert_array_equal(np.isinf(far), np.isinf(ref))
    np.testing.assert_array_equal(far[np.isinf(far)], ref[np.isinf(ref)])


@pytest.mark.parametrize("n", [4096, 6000])
def test_far_field_in_every_single_pulse_call(dcg, n):
    # doppler_resample, correct_batch, a plan and correct_compress take their
    # scratch from the context in different places: all against one oracle
    import torch
    rng = synth.rng_for(4, salt=n)
    x = synth.bandlimited_noise(n, rng).astype(np.complex64)
    h = synth.lfm(256, 20e6, 5e6).astype(np.complex64)
    fs, fc, v, tec = 20e6, 1e9, -6100.0, 60.0
    ctx = dcg.Context(0)
    xd, hd = torch.from_numpy(x).cuda(), torch.from_numpy(h).cuda()
    y, z, c = (torch.empty_like(xd) for _ in range(3))
    E = dcg.DC_EXACT_FP32
    items = np.zeros(2, dtype=dcg.ITEM_DTYPE)
    items["in_off"], items["out_off"], items["n"], items["n_out"] = 0, [0, n], n, n
    items["fs"], items["fc"], items["v_r"], items["tec_tecu"] = fs, fc, [v, 0.3 * v], tec
    b = torch.empty(2 * n, dtype=torch.complex64, device="cuda")
    pb = torch.empty_like(b)
    dcg.doppler_resample(ctx, xd, y, fs, fc, v, mode=E)
    dcg.correct_batch(ctx, xd, b, items, mode=E)
    torch.cuda.synchronize()
    plan = dcg.dc_plan_batch(ctx, xd, pb, items, mode=E)
    for _ in range(3):
        plan.execute()
    dcg.correct_compress(ctx, xd, hd, c, fs, fc, v, tec, mode=E)
    dcg.dc_check(ctx)
    assert torch.equal(torch.view_as_real(b), torch.view_as_real(pb))
    x64 = x.astype(np.complex128)
    rel = lambda a, r: np.linalg.norm(a - r) / np.linalg.norm(r)
    ref = oracle.resample(x64, fs, fc, v, "exact")
    assert rel(y.cpu().numpy(), ref) <= 4e-6
    assert rel(b[:n].cpu().numpy(), oracle.iono_correct(ref, fs, fc, tec)) <= 5e-6
    ref2 = oracle.correct(x64, fs, fc, 0.3 * v, tec, mode="exact")
    assert rel(b[n:].cpu().numpy(), ref2) <= 5e-6
    L = 1 << (n - 1).bit_length()
    H = np.fft.fft(h.astype(np.complex128), L)
    want = np.fft.ifft(np.fft.fft(oracle.iono_correct(ref, fs, fc, tec, L=L) if n == L else
                                  np.fft.ifft(np.fft.fft(ref, L) * np.exp(-1j * oracle.iono_phase(L, fs, fc, tec))), L)
                       * H.conj())[:n]
    assert rel(c.cpu().numpy(), want) <= 5e-6
    plan.close()
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

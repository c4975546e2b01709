"""Passes launched programmatically behind one another (single pulses of the
three-pass path, the Doppler bank's chain): a kernel that read its
predecessor's results too early, or a call that started before the last one
had finished with its scratch, would change some output.  Calls on two
alternating inputs are queued back to back on one stream, every result copied
aside, and each must equal the same call made alone, bit for bit.
"""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dcg():
    import paper_2508_04951_gb300 as m
    m.build.build()
    m.load()
    return m


def alternate(dcg, ctx, call, shape, rounds):
    import torch
    out = torch.empty(shape, dtype=torch.complex64, device="cuda")
    alone = []
    for i in range(2):
        call(i, out)
        torch.cuda.synchronize()
        alone.append(out.clone())
    torch.cuda.synchronize()
    got = []
    for r in range(rounds):
        call(r % 2, out)
        got.append(out.clone())
    dcg.dc_check(ctx)
    for r in range(rounds):
        assert torch.equal(torch.view_as_real(got[r]), torch.view_as_real(alone[r % 2])), r


# 32, 64, 128 row CTAs (programmatic, spread above 64), 256 (plain launches)
@pytest.mark.parametrize("n", [65537, 1 << 17, 200001, 1 << 18, (1 << 18) + 1, 1 << 19, (1 << 19) + 3])
def test_three_pass_pulses_back_to_back(dcg, n):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    x = [torch.randn(n, dtype=torch.complex64, device="cuda", generator=g) for _ in range(2)]
    ctx = dcg.Context(0)
    alternate(dcg, ctx, lambda i, out: dcg.iono_correct(ctx, x[i], out, 20e6, 1e9, 40.0 + 50 * i), n, 40)
    # in place: the last pass writes what the first one reads
    y = [t.clone() for t in x]
    out = [torch.empty_like(t) for t in x]
    for i in range(2):
        dcg.iono_correct(ctx, x[i], out[i], 2.048e9, 0.0, 100.0)
        dcg.iono_correct(ctx, y[i], y[i], 2.048e9, 0.0, 100.0)
    dcg.dc_check(ctx)
    for i in range(2):
        assert torch.equal(torch.view_as_real(out[i]), torch.view_as_real(y[i]))
    ctx.close()


@pytest.mark.parametrize("n,n_v,n_tec,n_rep", [(2000, 3, 2, 0), (4096, 33, 3, 0), (10001, 33, 7, 0), (10001, 5, 3, 400),
                                               (40000, 3, 2, 0), (200000, 2, 2, 0)])
def test_banks_back_to_back(dcg, n, n_v, n_tec, n_rep):
    import torch
    rng = synth.rng_for(2, salt=n)
    x = [torch.from_numpy(synth.bandlimited_noise(n, rng).astype(np.complex64)).cuda() for _ in range(2)]
    v = [rng.uniform(-8000, 8000, n_v) for _ in range(2)]
    tec = [rng.uniform(5, 150, n_tec) for _ in range(2)]
    rep = torch.from_numpy(synth.lfm(max(n_rep, 1), 20e6, 5e6).astype(np.complex64)).cuda()
    ctx = dcg.Context(0)

    def call(i, out):
        if n_rep:
            dcg.correct_compress_bank(ctx, x[i], rep, v[i], tec[i], out, 20e6, 1e9)
        else:
            dcg.correct_bank(ctx, x[i], v[i], tec[i], out, 20e6, 1e9)

    alternate(dcg, ctx, call, (n_v, n_tec, n), 30)
    ctx.close()

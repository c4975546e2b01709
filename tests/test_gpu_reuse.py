"""Scratch that a launch uses again while its first users may still be at it: the slots of the
two-pass apply at L = 65536, four times over, and the chunks of long banks and
batches, whose next pass starts programmatically behind the one that still reads them.
"""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
FS, FC = 20e6, 1e9


@pytest.fixture(scope="module")
def dcg():
    import paper_2508_04951_gb300 as m
    m.build.build()
    m.load()
    return m


def bank(m, n, n_v, n_tec, schedule, rounds=1):
    import torch
    x = torch.from_numpy(synth.bandlimited_noise(n, synth.rng_for(6, salt=n)).astype(np.complex64)).cuda()
    v, tec = np.linspace(-7900.0, 7900.0, n_v), np.linspace(5.0, 150.0, n_tec)
    ctx = m.Context(0)
    m.dc_tuning_set(ctx, schedule)
    out = torch.full((n_v, n_tec, n), 7.0, dtype=torch.complex64, device="cuda")
    first = None
    for _ in range(rounds):
        m.correct_bank(ctx, x, v, tec, out, FS, FC)
        if first is None:
            first = out.clone()
        else:
            assert torch.equal(torch.view_as_real(out), torch.view_as_real(first))
        out.fill_(7.0)
    m.dc_check(ctx)
    ctx.close()
    return first


def test_slots_of_the_two_pass_apply(dcg):
    # 4 slots of 24 transforms: 384 transforms take each slot four times; every one
    # against the clusters', whose sums are the same to rounding
    a, b = (bank(dcg, 65536, 24, 16, {"apply_kind": k}, rounds=3) for k in (3, 1))
    e = (a - b).norm(dim=-1) / b.norm(dim=-1)
    assert float(e.max()) <= 1e-6


# transforms of 2^17 and 2^18 (32 and 64 row CTAs each) in chunks of one, two, three (a
# remainder) and twenty: launches of at most 64, at most 152 and at least 1216 CTAs, and between
@pytest.mark.parametrize("n,n_v,n_tec,per_chunk", [(100000, 3, 2, 1), (100000, 3, 3, 2), (100000, 5, 2, 4), (200000, 3, 2, 1),
                                                   (200000, 3, 3, 2), (200000, 4, 2, 3), (200000, 6, 10, 20)])
def test_chunks_of_long_banks(dcg, n, n_v, n_tec, per_chunk):
    import torch
    m = 17 if n == 100000 else 18
    a = bank(dcg, n, n_v, n_tec, {"chunk": {m: per_chunk * (8 << m)}}, rounds=8)
    b = bank(dcg, n, n_v, n_tec, {"chunk": {m: -1}})
    assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))


@pytest.mark.parametrize("n,count,per_chunk", [(100000, 7, 2), (200000, 5, 1), (200000, 5, 2), (200000, 45, 20)])
def test_chunks_of_long_batches(dcg, n, count, per_chunk):
    import torch
    m = 17 if n == 100000 else 18
    x = torch.from_numpy(synth.bandlimited_noise(n * count, synth.rng_for(6, salt=n)).astype(np.complex64)).cuda()
    items = np.zeros(count, dtype=dcg.ITEM_DTYPE)
    items["in_off"] = items["out_off"] = n * np.arange(count)
    items["n"] = items["n_out"] = n
    items["fs"], items["fc"], items["v_r"], items["tec_tecu"] = FS, FC, np.linspace(-7000.0, 7000.0, count), 60.0
    ctx = dcg.Context(0)
    outs = []
    for chunk in (-1, per_chunk * (8 << m)):
        dcg.dc_tuning_set(ctx, {"chunk": {m: chunk}})
        for _ in range(6):
            y = torch.full_like(x, 7.0)
            dcg.correct_batch(ctx, x, y, items)
            outs.append(y)
        dcg.dc_check(ctx)
    for y in outs[1:]:
        assert torch.equal(torch.view_as_real(y), torch.view_as_real(outs[0]))
    ctx.close()

"""An item's result does not depend on the batch it comes in, bit for bit: also for exact
sums, whose far field takes scratch beside the batch's, under a scratch budget
that has room for it with one item and not with two, and in a plan.
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


# 6000 samples: 48128 bytes of scratch an item, 6144 more for its far field
@pytest.mark.parametrize("mode", ["DC_EXACT_FP32", "DC_WINDOWED"])
@pytest.mark.parametrize("budget", [0, 2 * 48128 + 1000, 1 << 30])
@pytest.mark.parametrize("plan", [False, True])
def test_alone_and_among_others(dcg, mode, budget, plan):
    import torch
    m = dcg
    n = 6000
    x = torch.from_numpy(synth.bandlimited_noise(2 * n, synth.rng_for(5)).astype(np.complex64)).cuda()
    items = np.zeros(2, dtype=m.ITEM_DTYPE)
    items["in_off"] = items["out_off"] = [0, n]
    items["n"] = items["n_out"] = n
    items["fs"], items["fc"], items["v_r"], items["tec_tecu"] = FS, FC, [6500.0, -300.0], [50.0, 80.0]
    got = []
    for count in (1, 2):
        ctx = m.Context(0, budget)
        y = torch.zeros_like(x)
        torch.cuda.synchronize()
        if plan:
            p = m.dc_plan_batch(ctx, x, y, items[:count], mode=getattr(m, mode))
            y.zero_()
            p.execute()
            m.dc_check(ctx)
            p.close()
        else:
            m.correct_batch(ctx, x, y, items[:count], mode=getattr(m, mode))
            m.dc_check(ctx)
        got.append(y[:n].cpu().numpy())
        ctx.close()
    np.testing.assert_array_equal(got[0].view(np.float32), got[1].view(np.float32))
    ref = oracle.correct(x[:n].cpu().numpy().astype(np.complex128), FS, FC, 6500.0, 50.0,
                         mode="exact" if mode == "DC_EXACT_FP32" else "windowed")
    assert np.linalg.norm(got[0] - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("lens", [[4096, 100], [4096, 4096, 2049, 3], [2500, 60000, 7], [70000, 4000, 70001]])
def test_every_class_among_others(dcg, lens):
    # one launch for several classes, a class of its own: the same kernels' arithmetic
    import torch
    m = dcg
    x = torch.from_numpy(synth.bandlimited_noise(sum(lens), synth.rng_for(6)).astype(np.complex64)).cuda()
    items = np.zeros(len(lens), dtype=m.ITEM_DTYPE)
    items["in_off"] = items["out_off"] = np.concatenate([[0], np.cumsum(lens)[:-1]])
    items["n"] = items["n_out"] = lens
    items["fs"], items["fc"], items["v_r"], items["tec_tecu"] = FS, FC, 6500.0 - 900.0 * np.arange(len(lens)), 50.0
    ctx = m.Context(0)
    y, z = torch.zeros_like(x), torch.zeros_like(x)
    m.correct_batch(ctx, x, y, items)
    for i in range(len(lens)):
        m.correct_batch(ctx, x, z, items[i:i + 1])
    m.dc_check(ctx)
    assert torch.equal(torch.view_as_real(y), torch.view_as_real(z))
    ctx.close()

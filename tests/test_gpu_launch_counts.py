"""dc_launch_count, dc_plan_launches and the profile's launches count kernels, also
where one call of the host code launches several (exact sums with their far
field, split planes and tiles, the cubic predistortion), as a profiler sees them.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dcg():
    import paper_2508_04951_gb300 as m
    m.build.build()
    m.load()
    return m


def calls(m, ctx, x, y):
    E = m.DC_EXACT_FP32
    return {
        "exact_dense": lambda: m.doppler_resample(ctx, x[:2000], y[:2000], 20e6, 1e9, 6000.0, mode=E),
        "exact_far": lambda: m.doppler_resample(ctx, x[:8000], y[:8000], 20e6, 1e9, 6000.0, mode=E),
        "exact_rows": lambda: m.resample_exact_batch(ctx, x, 2000, 10, [6000.0], y, mode=E),
        "bf16_dense": lambda: m.resample_exact_batch(ctx, x, 1000, 10, [6000.0], y, mode=m.DC_EXACT_BF16X3),
        "fp16_far": lambda: m.resample_exact_batch(ctx, x, 2000, 10, [6000.0], y, mode=m.DC_EXACT_FP16X3),
        "compress": lambda: m.correct_compress(ctx, x[:8000], x[:500], y[:8000], 20e6, 1e9, 6000.0, 50.0, mode=E),
        "cubic": lambda: m.predistort_lfm(ctx, y, 20e6, 1e9, 5e6, 1e-4, 50.0, kind=m.DC_LFM_CUBIC),
        "plain": lambda: m.predistort_lfm(ctx, y, 20e6, 1e9, 5e6, 1e-4, 50.0, kind=m.DC_LFM_PLAIN),
    }


# kernels of the call: moments, node values, sum; planes, (node values,) tiles; the
# spectrum, table and transform of a compression; frequencies, totals, samples
WANT = {"exact_dense": 1, "exact_far": 3, "exact_rows": 3, "bf16_dense": 2, "fp16_far": 3, "compress": 6, "cubic": 3,
        "plain": 1}


@pytest.mark.parametrize("kind", sorted(WANT))
def test_kernels_are_counted(dcg, kind):
    import torch
    m = dcg
    x = torch.randn(20000, dtype=torch.complex64, device="cuda")
    y = torch.empty_like(x)
    ctx = m.Context(0)
    call = calls(m, ctx, x, y)[kind]
    call()                                        # the scratch is there
    before = m.dc_launch_count(ctx)
    call()
    assert m.dc_launch_count(ctx) - before == WANT[kind]
    m.dc_profile_enable(ctx, True)
    call()
    assert sum(v[0] for v in m.dc_profile_read(ctx).values()) == WANT[kind]
    m.dc_profile_enable(ctx, False)
    m.dc_check(ctx)
    ctx.close()


def test_plans_of_exact_sums(dcg):
    import torch
    m = dcg
    x = torch.randn(16000, dtype=torch.complex64, device="cuda")
    y = torch.empty_like(x)
    items = np.zeros(2, dtype=m.ITEM_DTYPE)
    items["in_off"] = items["out_off"] = [0, 8000]
    items["n"] = items["n_out"] = 8000
    items["fs"], items["fc"], items["v_r"], items["tec_tecu"] = 20e6, 1e9, 5000.0, 40.0
    ctx = m.Context(0)
    torch.cuda.synchronize()
    plan = m.dc_plan_batch(ctx, x, y, items, mode=m.DC_EXACT_FP32)
    assert plan.launches == 2 * 3 + 1
    before = m.dc_launch_count(ctx)
    plan.execute()
    assert m.dc_launch_count(ctx) - before == 7
    m.dc_check(ctx)
    plan.close()
    ctx.close()

"""Scratch where memory is short: a plan takes what its own call takes, and is
recorded with less where a second block of that is not to be had.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
MIB = 1 << 20


@pytest.fixture(scope="module")
def dcg():
    import paper_2508_04951_gb300 as m
    m.build.build()
    m.load()
    return m


def free_bytes():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def items_of(m, n, count):
    items = np.zeros(count, dtype=m.ITEM_DTYPE)
    items["n"] = items["n_out"] = n
    items["in_off"] = items["out_off"] = n * np.arange(count)
    items["fs"], items["fc"], items["v_r"], items["tec_tecu"] = 20e6, 1e9, 100.0, 40.0
    return items


def test_plan_scratch_is_its_own_calls(dcg):
    # a context whose scratch has grown to 256 MiB and more
    import torch
    m = dcg
    ctx = m.Context(0)
    n, count = 1 << 18, 64
    x = torch.zeros(n * count, dtype=torch.complex64, device="cuda")
    y = torch.empty_like(x)
    m.correct_batch(ctx, x, y, items_of(m, n, count))
    small = items_of(m, 4096, 1)
    p = m.dc_plan_batch(ctx, x, y, small)                # what a first plan loads
    before = free_bytes()
    q = m.dc_plan_batch(ctx, x, y, small)
    assert before - free_bytes() <= 64 * MIB
    q.close()
    p.close()
    ctx.close()


def test_plan_with_less_scratch(dcg):
    # a bank whose passes take 512 MiB of scratch (610 in all) with 900 MiB left: the
    # call has it, a plan then gets the 64 MiB form (162), with the same outputs
    import torch
    m = dcg
    n, v, tec = 1 << 18, np.linspace(-5000.0, 5000.0, 8), np.linspace(5.0, 100.0, 33)
    x = torch.randn(n, dtype=torch.complex64, device="cuda")
    a = torch.empty((8, 33, n), dtype=torch.complex64, device="cuda")
    b = torch.empty_like(a)
    ctx = m.Context(0)
    m.correct_bank(ctx, x, v, tec, a, 20e6, 1e9)
    ctx.close()
    ctx = m.Context(0)
    filler = torch.empty(free_bytes() - 900 * MIB, dtype=torch.uint8, device="cuda")
    plan = m.dc_plan_bank(ctx, x, v, tec, b, 20e6, 1e9)
    b.zero_()
    torch.cuda.synchronize()
    for _ in range(2):
        plan.execute()
    m.dc_check(ctx)
    del filler
    assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
    plan.close()
    ctx.close()
    free_bytes()


def test_refused_scratch_is_not_asked_for_on_every_call(dcg):
    # a bank whose passes would take 512 MiB with 500 MiB left: it runs in the 64 MiB
    # form, and the next 64 calls do not ask for the 512 again (seen from the memory that
    # they leave alone when it has become free); then it is taken
    import torch
    m = dcg
    n, v, tec = 1 << 18, np.linspace(-5000.0, 5000.0, 8), np.linspace(5.0, 100.0, 33)
    x = torch.randn(n, dtype=torch.complex64, device="cuda")
    a, b, c = (torch.empty((8, 33, n), dtype=torch.complex64, device="cuda") for _ in range(3))
    ctx = m.Context(0)
    m.correct_bank(ctx, x[:1000], v, tec, a, 20e6, 1e9)
    filler = torch.empty(free_bytes() - 500 * MIB, dtype=torch.uint8, device="cuda")
    m.correct_bank(ctx, x, v, tec, a, 20e6, 1e9)
    m.dc_check(ctx)
    del filler
    before = free_bytes()
    for _ in range(64):
        m.correct_bank(ctx, x, v, tec, b, 20e6, 1e9)
    assert before - free_bytes() < 64 * MIB
    m.correct_bank(ctx, x, v, tec, c, 20e6, 1e9)
    assert before - free_bytes() > 400 * MIB
    m.dc_check(ctx)
    for y in (b, c):
        assert torch.equal(torch.view_as_real(a), torch.view_as_real(y))
    ctx.close()

"""FP32 exact sums of so many pulses that one kind of tile, or one warp per node
value, would take more CTAs than a grid holds in y or z (65535): the calls are
accepted, and their pulses give what they give in calls of a few thousand.
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


# tiles of 16 (dense sum) past 65535 in y, the largest count 32 pulses a tile hold; 8
# pulses per warp of node values past 65535 in z (n from 1536: the far field)
@pytest.mark.parametrize("n,n_out,pulses", [(2, 1, 1048577), (3, 2, 2097120), (1536, 4, 524281)])
def test_counts_past_a_grid(dcg, n, n_out, pulses):
    import torch
    g = torch.Generator(device="cuda").manual_seed(pulses)
    x = torch.randn((pulses, n), dtype=torch.complex64, device="cuda", generator=g)
    y = torch.full((pulses * n_out + 8,), 7.0, dtype=torch.complex64, device="cuda")
    ctx = dcg.Context(0)
    dcg.resample_exact_batch(ctx, x.view(-1), n, pulses, [6000.0], y[:-8], n_out=n_out)
    dcg.dc_check(ctx)
    assert torch.all(y[-8:] == 7.0)
    y = y[:-8].view(pulses, n_out)
    for a in (0, pulses // 2, pulses - 4096):
        part = torch.empty((4096, n_out), dtype=torch.complex64, device="cuda")
        dcg.resample_exact_batch(ctx, x[a:a + 4096].reshape(-1), n, 4096, [6000.0], part.view(-1), n_out=n_out)
        dcg.dc_check(ctx)
        # the same FP32 terms in another order
        assert float((part - y[a:a + 4096]).norm() / part.norm()) <= 2e-6
    ctx.close()


def test_counts_past_every_grid_are_refused(dcg):
    import torch
    ctx = dcg.Context(0)
    x = torch.zeros(65535 * 64 + 1, dtype=torch.complex64, device="cuda")
    with pytest.raises(dcg.DcError) as e:
        dcg.resample_exact_batch(ctx, x, 1, x.numel(), [0.0], torch.empty_like(x), n_out=1)
    assert e.value.status == 4
    dcg.dc_check(ctx)
    ctx.close()

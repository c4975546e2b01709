"""Calls captured into a caller's own CUDA graph, from a context that has only made
one small call before (its scratch not grown, the window's table not made): nothing
is allocated during the capture, and the replay gives the plain call's outputs.

Tolerance: another of the library's paths may serve the captured call; the FP32
ones agree within 2e-6.
"""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
FS, FC, TOL = 20e6, 1e9, 2e-6


@pytest.fixture(scope="module")
def dcg():
    import paper_2508_04951_gb300 as m
    m.build.build()
    m.load()
    return m


@pytest.mark.parametrize("n", [1000, 4096, 16384, 20000])
@pytest.mark.parametrize("kind", ["windowed", "beta", "exact", "exact_rows"])
def test_single_calls(dcg, kind, n):
    import torch
    m = dcg
    x = torch.from_numpy(synth.bandlimited_noise(n, synth.rng_for(1, salt=n)).astype(np.complex64)).cuda()
    rows = 4 if kind == "exact_rows" else 1
    xs = x.repeat(rows)

    def call(ctx, y, stream):
        if kind == "exact_rows":
            m.resample_exact_batch(ctx, xs, n, rows, [6000.0], y, mode=m.DC_EXACT_FP32, stream=stream)
        else:
            m.doppler_resample(ctx, x, y, FS, FC, 6000.0, beta=6.0 if kind == "beta" else 8.0, stream=stream,
                               mode=m.DC_EXACT_FP32 if kind == "exact" else m.DC_WINDOWED)

    plain, got = torch.empty_like(xs), torch.zeros_like(xs)
    ctx = m.Context(0)
    call(ctx, plain, None)
    m.dc_check(ctx)
    ctx.close()
    ctx = m.Context(0)
    m.doppler_resample(ctx, x[:100], got[:100], FS, FC, 6000.0)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(ctx, got, torch.cuda.current_stream())
    graph.replay()
    torch.cuda.synchronize()
    m.dc_check(ctx)
    assert float((got - plain).norm() / plain.norm()) <= TOL
    del graph
    ctx.close()

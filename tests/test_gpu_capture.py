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


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("n", [100, 1000, 4096, 8192, 131072, 300000])
def test_behind_copies_and_joins(dcg, n, captured):
    """Programmatic launches behind what is not a kernel of the library: a copy, a
    fill, another stream's event joined after a library call on this stream."""
    import torch
    m = dcg
    x = torch.from_numpy(synth.bandlimited_noise(n, synth.rng_for(4, salt=n)).astype(np.complex64)).cuda()
    ctx, other = m.Context(0), torch.cuda.Stream()
    ref = [torch.empty_like(x) for _ in range(3)]
    for r, scale in zip(ref, (1.0, 0.0, 2.0)):
        m.iono_correct(ctx, x * scale, r, FS, FC, 70.0)
        torch.cuda.synchronize()
    big = torch.zeros(1 << 24, device="cuda")
    a, b, c = torch.empty_like(x), torch.empty_like(x), torch.empty_like(x)
    outs = [torch.empty_like(x) for _ in range(4)]

    def work():
        s = torch.cuda.current_stream()
        a.copy_(x)                                       # a copy, then a call that reads it
        m.iono_correct(ctx, a, outs[0], FS, FC, 70.0, stream=s)
        b.zero_()
        m.iono_correct(ctx, b, outs[1], FS, FC, 70.0, stream=s)
        other.wait_stream(s)
        with torch.cuda.stream(other):                   # a long chain ahead of the input
            for _ in range(20):
                big.add_(1.0)
            torch.mul(x, 2.0, out=c)
        m.doppler_resample(ctx, x, outs[3], FS, FC, 10.0, stream=s)
        s.wait_stream(other)
        m.iono_correct(ctx, c, outs[2], FS, FC, 70.0, stream=s)
        c.zero_()                                        # and one that overwrites it

    work()
    torch.cuda.synchronize()
    for o in outs + [a, b, c]:
        o.fill_(5.0)
    if captured:
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            work()
        for _ in range(3):
            graph.replay()
    else:
        for _ in range(3):
            work()
    torch.cuda.synchronize()
    m.dc_check(ctx)
    for o, r in zip(outs, ref):
        assert torch.equal(o, r)
    if captured:
        del graph
    ctx.close()

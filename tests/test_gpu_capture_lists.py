"""Calls that send lists (items, range rates, a window's polynomials), captured into a
caller's graph: a replay uses the lists of the captured call, whatever calls the
context has served since, among them longer ones that move its buffers.
"""

import gc

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


def items_of(m, lens, v0):
    items = np.zeros(len(lens), dtype=m.ITEM_DTYPE)
    items["n"] = items["n_out"] = lens
    items["in_off"] = items["out_off"] = np.concatenate([[0], np.cumsum(lens)[:-1]])
    items["fs"], items["fc"] = FS, FC
    items["v_r"] = v0 + 311.0 * np.arange(len(lens))
    items["tec_tecu"] = 20.0 + 3.0 * np.arange(len(lens))
    return items


@pytest.mark.parametrize("kind", ["window", "batch", "batch_carrier", "bank", "bank_direct", "bank_compress", "rows",
                                  "bf16"])
def test_replays_keep_their_lists(dcg, kind):
    import torch
    m = dcg
    x = torch.from_numpy(synth.bandlimited_noise(30000, synth.rng_for(3)).astype(np.complex64)).cuda()
    v, tec = np.linspace(-6000.0, 7000.0, 5), np.linspace(10.0, 90.0, 3)

    def call(ctx, y, k=0, stream=None):
        """The call, with other values for other k."""
        if kind == "window":
            m.doppler_resample(ctx, x, y[:30000], FS, FC, 6000.0, beta=6.0 + 0.5 * k, stream=stream)
        elif kind in ("batch", "batch_carrier"):
            m.correct_batch(ctx, x, y, items_of(m, [100, 3000, 4096, 9000, 9001], 10.0 * k), stream=stream,
                            carrier_shift=kind == "batch_carrier")
        elif kind in ("bank", "bank_direct"):
            m.correct_bank(ctx, x[:3000], v + 5.0 * k, tec + k, y, FS, FC, stream=stream,
                           taps=32 if kind == "bank" else 16)
        elif kind == "bank_compress":
            m.correct_compress_bank(ctx, x[:3000], x[:200], v + 5.0 * k, tec + k, y, FS, FC, stream=stream)
        else:
            m.resample_exact_batch(ctx, x, 1000, 9, v[:3] + 5.0 * k, y, stream=stream,
                                   mode=m.DC_EXACT_FP32 if kind == "rows" else m.DC_EXACT_BF16X3)

    def zeros():
        return torch.zeros(5 * 3 * 3000, dtype=torch.complex64, device="cuda")

    # the window is one the context keeps no table of: all slots are taken
    ctx = m.Context(0)
    for i in range(17):
        m.doppler_resample(ctx, x[:64], zeros()[:64], FS, FC, 10.0, beta=float(i) / 2 + 9.0)
    plain, got, other = zeros(), zeros(), zeros()
    call(ctx, plain)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(ctx, got, stream=torch.cuda.current_stream())
    for k in (1, 2):
        got.zero_()
        call(ctx, other, k)                              # the same staging block, other lists
        lens = np.full(700 * k, 16)                      # longer ones: the buffers move
        m.correct_batch(ctx, x, zeros(), items_of(m, lens, 100.0))
        torch.cuda.synchronize()
        gc.collect()
        graph.replay()
        torch.cuda.synchronize()
        m.dc_check(ctx)
        assert torch.equal(torch.view_as_real(got), torch.view_as_real(plain)), k
        assert not torch.equal(other, plain)
    del graph
    torch.cuda.synchronize()
    ctx.close()

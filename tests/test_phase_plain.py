"""The short form of the phase evaluation (csrc/phase.cuh, iono_cycles<true>), restated
in float32: up to the bound under which the host chooses it, the quotient's second
part and the phase that goes unreduced into the sine are as small as stated there.
"""

import os
import re

import numpy as np
import pytest

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_04951_gb300", "csrc",
                      "phase.cuh")
f32 = np.float32


def plain_cycles():
    m = re.search(r"constexpr double kPlainCycles = 1 << (\d+);", open(HEADER).read())
    return float(1 << int(m.group(1)))


def evaluate(c, fc, d, kt, rcp_error):
    """iono_cycles<true>; fused multiply-adds by way of float64 (exact products)."""
    c_hi = f32(c)
    c_lo = f32(c - float(c_hi))
    p = (f32(d) * kt).astype(f32)
    p_lo = (float(d) * kt.astype(np.float64) - p).astype(f32)
    fh = (f32(fc) + p).astype(f32)
    fl = (p_lo + (p - (fh - f32(fc)).astype(f32)).astype(f32)).astype(f32)
    rb = (1.0 / fh.astype(np.float64) * (1.0 + rcp_error)).astype(f32)
    q1 = (c_hi * rb).astype(f32)
    r = (float(c_hi) - q1.astype(np.float64) * fh).astype(f32)
    r = ((r + c_lo).astype(f32).astype(np.float64) - q1.astype(np.float64) * fl).astype(f32)
    q2 = (r * rb).astype(f32)
    x = ((q1 - np.rint(q1)).astype(f32) + q2).astype(f32)
    return x, q2


@pytest.mark.parametrize("fs,fc", [(20e6, 1e9), (20e6, 435e6), (1 << 20, 1 << 28), (2e6, 1.0001e6), (300e6, 151e6)])
@pytest.mark.parametrize("rcp_error", [-2.0 ** -23, 0.0, 2.0 ** -23])
def test_phase_within_the_sines_range(fs, fc, rcp_error):
    gate = plain_cycles()
    rng = np.random.default_rng(5)
    L = 1 << 14
    d = fs / L
    assert float(f32(fc)) == fc
    d = float(f32(d))
    kt = np.concatenate([np.arange(-L // 2, -L // 2 + 2000), rng.integers(-L // 2, L // 2, 20000)]).astype(f32)
    f_min = fc - 0.5 * fs
    for share in (0.5, 0.7, 0.9, 0.9999):
        c = share * gate * f_min / max(1.0, 0.5 * fs / f_min)
        x, q2 = evaluate(c, fc, d, kt, rcp_error)
        assert np.abs(q2).max() <= 2.75 * 2.0 ** -23 * gate
        assert np.abs(q2).max() <= 0.09 and np.abs(x).max() <= 0.59

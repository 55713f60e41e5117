"""The rule that lets kernels trust their staged sample windows (windows_hold in
mach_internal.h), on a float32 model of pair_window, term_geometry and term_record: within the
rule's bounds every kept term's two taps lie in the window, whatever the order in which the
bound's squares are summed; far beyond them some do not, so that the rule is needed."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_06257_gb300", "csrc")
f32 = np.float32


def bound(name):
    with open(os.path.join(CSRC, "mach_internal.h")) as f:
        got = re.search(rf"constexpr \w+ {name} = ([^;]+);", f.read())
    return float(eval(got.group(1).rstrip("f")))


def fma(a, b, c):
    return f32(np.float64(a) * np.float64(b) + np.float64(c))


def outside(R, S, n, seed):
    """(kept, kept with a tap outside the window) of n one-voxel windows: receive delays of R/5 to
    R samples, transmit delays that put the sum anywhere in the record."""
    r = np.random.default_rng(seed)
    d = f32(R / np.sqrt(3.0) * r.uniform(0.2, 1.0, (3, n)))
    rx = np.sqrt(fma(d[0], d[0], fma(d[1], d[1], f32(d[2] * d[2]))))
    s_tx = f32(-np.float64(rx) + r.uniform(0, S, n))
    s = f32(s_tx + rx)
    i0 = np.floor(s)
    kept = (s >= 0) & (s < f32(S - 1))
    bad = np.zeros(n, bool)
    for rb in (np.sqrt(f32(f32(f32(d[0] * d[0]) + f32(d[1] * d[1])) + f32(d[2] * d[2]))),
               np.sqrt(fma(d[2], d[2], fma(d[1], d[1], f32(d[0] * d[0]))))):
        b = f32(s_tx + rb)
        lo = np.maximum(0, np.floor(np.maximum(b, f32(-8))) - 2)
        hi = np.minimum(S - 1, np.floor(np.minimum(b, f32(S))) + 3)
        staged = (b >= -1) & (b < f32(S)) & (hi >= lo + 1)
        bad |= kept & (~staged | (i0 < lo) | (i0 + 1 > hi))
    return int(kept.sum()), int(bad.sum())


@pytest.mark.parametrize("S", [200, 4096, 1 << 18])
def test_kept_terms_lie_in_their_windows_within_the_bounds(S):
    assert S <= bound("kWindowsHold")
    for k in range(10, 21):
        R = min(2.0 ** k, bound("kReachHolds"))
        kept, bad = outside(R, S, 100_000, k)
        assert kept > 90_000 and bad == 0, (R, kept, bad)


def test_windows_miss_terms_far_beyond_the_bounds():
    """Why the samples per row alone decide nothing."""
    assert bound("kReachHolds") < 2.0 ** 25
    assert outside(2.0 ** 25, 200, 100_000, 1)[1] > 0
    assert outside(2.0 ** 27, 200, 100_000, 2)[1] > 0

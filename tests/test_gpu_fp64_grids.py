"""The FP64 model's sampled response (csrc/bx_f64.cu) against the oracle at the edges of its rules:
columns narrower than a bin (bin masses from erfc tails), between one and five bins (the bin-mass
polynomial), at every sample spacing 2^c up to the widest, a band beyond 8 sigma (every column on
the bins), the Gram-Charlier response on each, an axis of one to a few 32-sample tiles, and a
pile-up spectrum longer than the window.  Tolerances: the FP64 ones of tests/test_gpu_parity.py
(counts 1e-10 relative or 1e-12 of the largest, -2 lnL 1e-7, gradient 1e-9 (1 + |g theta|))."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_1805_11125_gb300 import bx, inputs as I
from tests._util import per_bin_ok

pytestmark = pytest.mark.gpu

# name: (a, b, c, width, band_sigmas, skewness = kurtosis)
CASES = {
    "narrower_than_a_bin": (0.0, 0.0, 0.5, 2.0, 0.0, 0.0),
    "one_to_five_bins": (0.0, 0.0, 30.0, 3.0, 0.0, 0.0),
    "just_below_five_bins": (0.0, 0.0, 24.9, 1.0, 0.0, 0.0),
    "just_above_five_bins": (0.0, 0.0, 25.1, 1.0, 0.0, 0.0),
    "mixed_kinds": (1.1, 2e-4, 1e-3, 3.0, 0.0, 0.0),
    "every_spacing": (0.5, 0.12, 4.0, 1.0, 0.0, 0.0),
    "wide_band": (1.1, 2e-4, 4.0, 2.0, 12.0, 0.0),
    "wide_band_narrow": (0.0, 0.0, 0.5, 2.0, 20.0, 0.0),
    "gram_charlier": (1.1, 2e-4, 4.0, 2.0, 0.0, 0.05),
    "gram_charlier_wide_band": (1.1, 2e-4, 4.0, 2.0, 9.0, 0.05),
}


def spec_of(name, bins, L):
    a, b, c, width, band, gc = CASES[name]
    s = I.multivariate(n_grid=263, width=width, lo_npe=13 * width, hi_npe=(13 + bins) * width, n_species=9,
                       total=3e5, L=L, n_rad=7, n_psd=5, name=name)
    s = dataclasses.replace(s, resp_skew=gc, resp_kurt=gc)
    th = s.theta_true.copy()
    th[s.K + 1:s.K + 4] = a, b, c
    s.theta_true = th
    return s, band


@pytest.mark.parametrize("bins,L", [(19, 3), (300, 40), (33, 90), (967, 40)])
@pytest.mark.parametrize("name", sorted(CASES))
def test_fp64_counts_nll_and_gradient(name, bins, L):
    s, band = spec_of(name, bins, L)
    mo = O.expected(s, s.theta_true)
    s = s.with_counts(I.poisson_counts(mo, 5))
    th = s.theta_true * (1 + 0.01 * np.random.default_rng(3).standard_normal(s.P))
    m = bx.Model(s, precision=bx.BX_FP64, band_sigmas=band, max_batch=3)
    mo, mg = O.expected(s, th), m.expected(th)
    ok, wr, wa = per_bin_ok(mg, mo, rel=1e-10, abs_frac=1e-12)
    assert ok, (wr, wa)
    fo, go = O.nll(s, th, grad=True)
    f, g = m.nll_grad(th)
    assert 2 * abs(f - fo) <= 1e-7
    lhs = np.abs(g[:s.P] - go) * np.abs(th)
    assert np.all(lhs <= 1e-9 * (1 + np.abs(go * th))), float(np.max(lhs / (1 + np.abs(go * th))))
    fb, gb = m.nll_batch(np.stack([th] * 3), grad=True)
    assert np.array_equal(fb, [f] * 3) and np.array_equal(gb, np.stack([g] * 3))
    m.close()

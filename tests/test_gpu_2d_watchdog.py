"""2D models whose device-side waits run out: every block leaves its loops together, drains its copies and
multiplications and returns, the call reports BX_ETIMEOUT (or its results, where each wait ended in
time), and the same model sizes evaluate to their usual results afterwards."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_1805_11125_gb300 import bx, inputs as I
from tests._util import points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [31, 800])
@pytest.mark.parametrize("precision", [bx.BX_FP32, bx.BX_BF16X3])
def test_waits_that_run_out(precision, L):
    s = I.discrimination(seed=6, n_grid=801)
    s = dataclasses.replace(s, pileup=I.pileup_spectrum(L, s.width), counts={})
    s = s.with_counts(I.poisson_counts(O.expected(s, s.theta_true), 4))
    th = points(s, 3, seed=3)
    m = bx.Model(s, precision=precision, max_batch=3)
    f, g = m.nll_batch(th, grad=True)
    assert np.isfinite(f).all() and np.isfinite(g).all()
    for budget in (1e-5, 1e-6, 1e-9):
        short = bx.Model(s, precision=precision, max_batch=3, watchdog_s=budget)
        try:
            fs, gs = short.nll_batch(th, grad=True)
            assert np.array_equal(fs, f) and np.array_equal(gs, g)
        except bx.BxError as e:
            assert e.status == bx.BX_ETIMEOUT
        short.close()
        f2, g2 = m.nll_batch(th, grad=True)
        assert np.array_equal(f2, f) and np.array_equal(g2, g)
    m.close()

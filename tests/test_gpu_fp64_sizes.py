"""The size limit of FP64 models, 4 axis + 6 window + pile-up <= 25962: a model at the limit is created and
evaluates to the oracle's -lnL, one past it in any of the three sizes is refused with the sizes."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_1805_11125_gb300 import bx, inputs as I

pytestmark = pytest.mark.gpu


def spec(axis, window, L):
    s = I.single_spectrum(n_grid=96, width=0.3, n_species=4, L=L, name="limit")
    s = dataclasses.replace(s, m_lo=axis - window, m_hi=axis, counts={})
    return s.with_counts(np.zeros(s.n_bins_total))


def test_sizes_at_the_limit():
    s = spec(4096, 1529, 404)
    assert 4 * s.m_hi + 6 * s.n_window + s.L == 25962
    s = s.with_counts(I.poisson_counts(O.expected(s, s.theta_true), 2))
    m = bx.Model(s, precision=bx.BX_FP64)
    th = s.theta_true * 1.01
    assert 2 * abs(m.nll(th) - O.nll(s, th)) <= 1e-7
    m.close()


@pytest.mark.parametrize("axis,window,L", [(4096, 1529, 405), (4096, 1530, 404), (4097, 1529, 404)])
def test_sizes_past_the_limit(axis, window, L):
    with pytest.raises(bx.BxError) as e:
        bx.Model(spec(axis, window, L), precision=bx.BX_FP64)
    assert e.value.status == bx.BX_EINVAL
    assert all(str(x) in str(e.value) for x in (axis, window, L))

"""Results do not depend on the batch: the FP64 model's two forwards (up to 4 items, a CTA per share of a
tile; more items, a CTA per tile) on the grids and widths of test_gpu_fp64_grids, and the FP32 small-batch
kernels of Gram-Charlier models, which evaluate entry by entry where the large-batch kernel pairs them.
Bit for bit."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1805_11125_gb300 import bx, inputs as I
from tests._util import points
from tests.test_gpu_fp64_grids import CASES, spec_of

pytestmark = pytest.mark.gpu


def same_rows(m, th, sizes):
    n = len(th)
    dev = torch.as_tensor(th, device="cuda")
    f, g = (x.cpu().numpy() for x in m.nll_batch(dev, grad=True))
    assert np.isfinite(f).all() and np.isfinite(g).all()
    for b in sizes:
        fb, gb = (x.cpu().numpy() for x in m.nll_batch(dev[:b], grad=True))
        assert np.array_equal(fb, f[:b]) and np.array_equal(gb, g[:b]), b
        assert np.array_equal(m.nll_batch(th[:b]), f[:b]), b
    assert np.array_equal(m.nll_batch(dev).cpu().numpy(), f), n


@pytest.mark.parametrize("bins,L", [(19, 3), (300, 40)])
@pytest.mark.parametrize("name", sorted(CASES))
def test_fp64_batches_on_every_grid(name, bins, L):
    s, band = spec_of(name, bins, L)
    s = s.with_counts(I.poisson_counts(O.expected(s, s.theta_true), 5))
    th = s.theta_true * (1 + 0.01 * np.random.default_rng(3).standard_normal((6, s.P)))
    th[:, s.K + 1:s.K + 4] = s.theta_true[s.K + 1:s.K + 4]
    m = bx.Model(s, precision=bx.BX_FP64, band_sigmas=band, max_batch=6)
    same_rows(m, th, (1, 2, 4, 5))
    fo, go = O.nll(s, th[5], grad=True)   # a row of the large batch
    f, g = m.nll_batch(th, grad=True)
    assert 2 * abs(f[5] - fo) <= 1e-7
    lhs = np.abs(g[5, :s.P] - go) * np.abs(th[5])
    assert np.all(lhs <= 1e-9 * (1 + np.abs(go * th[5])))
    m.close()


@pytest.mark.parametrize("kind", ["shelled", "quenched", "sliced"])
def test_fp64_batches_of_several_sets_and_slices(kind):
    kw = {} if kind == "sliced" else dict(n_grid=700)
    s = getattr(I, kind)(seed=5, **kw)
    s = dataclasses.replace(s, resp_skew=0.05, resp_kurt=0.05) if kind != "quenched" else s
    s = s.with_counts(I.poisson_counts(O.expected(s, s.theta_true), 9))
    m = bx.Model(s, precision=bx.BX_FP64, max_batch=7)
    same_rows(m, points(s, 7, seed=77), (1, 3, 4, 5))
    m.close()


@pytest.mark.parametrize("kind,kw", [("multivariate", {}), ("multivariate", dict(n_grid=257, width=4.0, n_species=5)),
                                     ("single_spectrum", dict(n_grid=797, width=2.0, n_species=6)), ("sliced", {}),
                                     ("shelled", dict(n_grid=700))])
def test_fp32_gram_charlier_batches(kind, kw):
    s = dataclasses.replace(getattr(I, kind)(seed=5, **kw), resp_skew=0.1, resp_kurt=0.1)
    s = s.with_counts(I.poisson_counts(O.expected(s, s.theta_true), 9))
    n = 700   # more tiles than the split forward takes
    th = np.resize(points(s, 5, seed=77), (n, s.P))
    m = bx.Model(s, precision=bx.BX_FP32, max_batch=n)
    same_rows(m, th, (1, 2, 5, 19, 60, 61, 152, 153))
    m.close()

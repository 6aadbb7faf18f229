"""FP64 models whose column sets do not fill whole 32-column chunks: one radial shell (a single set of
columns through the several-set kernels) and a plain dataset beside a quenched one, on grids whose last
chunk holds one to a few columns behind one or more blocks of 128; and a single shell that holds only a
fraction of a species' events, in the energy spectra and in the Eq. 4 histograms.  Against the oracle
with the FP64 tolerances of tests/test_gpu_parity.py (the FP32 ones for that mode)."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_1805_11125_gb300 import bx, inputs as I
from tests._util import per_bin_ok

pytestmark = pytest.mark.gpu


def compare(m, s, th, toy=0):
    mo, mg = O.expected(s, th), m.expected(th, toy)
    ok, wr, wa = per_bin_ok(mg[:len(mo)], mo, rel=1e-10, abs_frac=1e-12)
    assert ok, (wr, wa)
    fo, go = O.nll(s, th, grad=True)
    f, g = m.nll_batch(th[None], toy_idx=np.array([toy], np.int32), grad=True)
    assert 2 * abs(f[0] - fo) <= 1e-7, (f, fo)
    lhs = np.abs(g[0, :s.P] - go) * np.abs(th)
    assert np.all(lhs <= 1e-9 * (1 + np.abs(go * th))), float(np.max(lhs / (1 + np.abs(go * th))))


def model_spec(n_grid, **kw):
    return I.multivariate(n_grid=n_grid, e_max=0.6, width=2.0, lo_npe=40.0, hi_npe=360.0, n_species=5, total=2e5,
                          L=40, n_rad=7, n_psd=5, **kw)


def with_data(s):
    return s.with_counts(I.poisson_counts(O.expected(s, s.theta_true), 3))


@pytest.mark.parametrize("n_grid", [256, 257, 259, 385, 1025])
def test_one_shell_on_ragged_grids(n_grid):
    s = model_spec(n_grid)
    s = with_data(dataclasses.replace(s, shell_ly=np.array([1.03]), shell_frac=np.ones((s.K, 1))))
    m = bx.Model(s, precision=bx.BX_FP64)
    compare(m, s, s.theta_true)
    m.close()


@pytest.mark.parametrize("n_grid", [257, 1026])
def test_a_plain_dataset_beside_a_quenched_one(n_grid):
    a = with_data(model_spec(n_grid))
    b = model_spec(n_grid, seed=1)
    b = with_data(dataclasses.replace(b, quench=np.array([1.0, 1.0, 2.3, 1.0, 2.3])))
    m = bx.Model([a, b], precision=bx.BX_FP64, max_batch=2)
    for t, s in enumerate((a, b)):
        compare(m, s, s.theta_true, t)
    m.close()


@pytest.mark.parametrize("prec,rel,ftol,gtol", [(bx.BX_FP64, 1e-10, 1e-7, 1e-9), (bx.BX_FP32, 1e-5, 1e-3, 1e-3)])
def test_one_shell_with_a_fraction_of_the_events(prec, rel, ftol, gtol):
    s = model_spec(300)
    frac = np.linspace(0.5, 0.9, s.K)[:, None]
    s = with_data(dataclasses.replace(s, shell_ly=np.array([1.03]), shell_frac=frac))
    th = s.theta_true
    m = bx.Model(s, precision=prec)
    ok, wr, wa = per_bin_ok(m.expected(th), O.expected(s, th), rel=rel, abs_frac=1e-8)
    assert ok, (wr, wa)
    fo, go = O.nll(s, th, grad=True)
    f, g = m.nll_grad(th)
    assert 2 * abs(f - fo) <= ftol, (f, fo)
    lhs = np.abs(g[:s.P] - go) * np.abs(th)
    assert np.all(lhs <= gtol * (1 + np.abs(go * th)))
    m.close()

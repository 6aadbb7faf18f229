"""The kernels a small FP32 batch takes (forward tiles split between generator and accumulator warps,
an item's column stage in parts, the coefficients of the 2D model in parts) give bit for bit the rows
that the kernels of a large batch give for the same points: grids and windows of odd sizes and of whole
tiles, one set of columns and several, on either side of both limits; and the host path's one block of
results (pinned, up to 64 KB) those of its larger calls and of the device path.  (The modes themselves
are held to the oracle by the parity tests.)"""
import numpy as np
import pytest
import torch

from paper_1805_11125_gb300 import bx, inputs as I
from oracle import oracle as O
from tests._util import points

pytestmark = pytest.mark.gpu

# (model, arguments): rows M and columns N off and on the multiples of 32, 64, 128 and 256
CASES = {
    "plain_ragged": ("single_spectrum", dict(n_grid=797, width=2.0, n_species=6)),
    "plain_whole": ("single_spectrum", dict(n_grid=1024, width=2.0, n_species=6)),
    "mv_one_column_over": ("multivariate", dict(n_grid=257, width=4.0, n_species=5)),
    "mv_full": ("multivariate", dict()),
    "quenched": ("quenched", dict(n_grid=700)),
    "shelled": ("shelled", dict(n_grid=700)),
    "sliced": ("sliced", dict()),
    "two_dim": ("discrimination", dict(n_grid=801)),
}


def dataset(name):
    kind, kw = CASES[name]
    s = getattr(I, kind)(seed=5, **kw)
    return s.with_counts(I.poisson_counts(O.expected(s, s.theta_true), 9))


@pytest.mark.parametrize("name", sorted(CASES))
def test_small_batches_give_the_rows_of_a_large_one(name):
    s = dataset(name)
    n = 700   # more tiles than the split forward takes, more items than the parts take
    th = np.resize(points(s, 5, seed=77), (n, s.P))
    m = bx.Model([s], precision=bx.BX_FP32, max_batch=n)
    dev = torch.as_tensor(th, device="cuda")
    f, g = (x.cpu().numpy() for x in m.nll_batch(dev, grad=True))
    assert np.isfinite(f).all() and np.isfinite(g).all()
    assert np.array_equal(f, np.resize(f[:5], n)) and np.array_equal(g, np.resize(g[:5], (n, g.shape[1])))
    for b in (1, 2, 5, 19, 20, 60, 61, 152, 153):
        fb, gb = (x.cpu().numpy() for x in m.nll_batch(dev[:b], grad=True))
        assert np.array_equal(fb, f[:b]) and np.array_equal(gb, g[:b]), b
        fh, gh = m.nll_batch(th[:b], grad=True)   # host path
        assert np.array_equal(fh, f[:b]) and np.array_equal(gh, g[:b]), b
        assert np.array_equal(m.nll_batch(th[:b]), f[:b]), b
    fh, gh = m.nll_batch(th, grad=True)   # beyond the pinned buffer
    assert np.array_equal(fh, f) and np.array_equal(gh, g)
    f1, g1 = m.nll_grad(th[3])
    assert f1 == f[3] and np.array_equal(g1, g[3])
    m.close()


@pytest.mark.parametrize("L,n_grid", [(1, 801), (31, 801), (640, 801), (1500, 2000)])
def test_2d_pile_up_spectra_of_every_length(L, n_grid):
    """The 2D pile-up products' operand table: a pile-up spectrum of one bin, below a 32-row block, of
    whole blocks, and longer than one table's 20 blocks (several tables a tile)."""
    import dataclasses
    s = I.discrimination(seed=6, n_grid=n_grid)
    s = dataclasses.replace(s, pileup=I.pileup_spectrum(L, s.width, 1.0) if L > 1 else np.ones(1), counts={})
    s = s.with_counts(I.poisson_counts(O.expected(s, s.theta_true), 4))
    m = bx.Model([s], precision=bx.BX_FP32, max_batch=2)
    th = points(s, 1, seed=3)[0]
    f, g = m.nll_grad(th)
    fo, go = O.nll(s, th, grad=True)
    assert 2 * abs(f - fo) <= 1e-3, (f, fo)
    lhs = np.abs(g[: s.P] - go) * np.abs(th[: s.P])
    assert np.all(lhs <= 1e-3 * (1.0 + np.abs(go * th[: s.P]))), lhs.max()
    m.close()

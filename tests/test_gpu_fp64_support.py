"""Which bins a column of the FP64 model reaches, and how well the bins far from its mean are known.

A column (true-energy point) contributes to every bin of each 128-bin tile that its response band
(band_sigmas) touches, and to no bin of any other tile.  Line sources on a few neighbouring columns
leave most of the axis to the response's tails: the expected counts are compared relative to
themselves.  References: the oracle (no band) where the touched tiles hold all that matters, and the
oracle's response matrix under the rule above for bands that cut it.

Tolerance of a tail: its argument z = (m w - mu) / sigma carries a few roundings of mu / sigma and of
z, dz = 4 (mu / sigma + |z|) 2^-53 on either side, and the tail changes by |z| dz relative; the bin is
a difference of two tails, which loses a factor h |z| (h = w / sigma) below 1; the terms of the sums
and the pile-up weights another 32 roundings."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_1805_11125_gb300 import bx, inputs as I

pytestmark = pytest.mark.gpu

TILE = 128
EPS = 2.0 ** -53


def line_spec(sigma, M, L=1, tag=False, kB=0.011, width=1.0, cols=(61, 64)):
    """Three lines on neighbouring columns near 0.49 MeV (mean 220 to 235 npe), constant width."""
    N, K = 128, 2
    shapes = np.zeros((K, N))
    shapes[0, cols[0]:cols[1]] = (0.5, 0.3, 0.2)
    shapes[1, cols[0] + 1:cols[1]] = (0.4, 0.6)
    E = I.grid_energies(N, 1.0)
    g = I.pileup_spectrum(L, width) if L > 1 else np.ones(1)
    s = I.ModelSpec(name="line", n_grid=N, e_max=1.0, shapes=shapes, stop_pow=I.stopping_power(E), pileup=g,
                    width=width, m_lo=0, m_hi=M, tag_frac=np.array([0.2, 0.6]) if tag else None,
                    species=["a", "b"])
    s.theta_true = np.array([4e3, 2e3, 500.0, 0.0, 0.0, sigma ** 2, kB, 0.05, 1.0])
    return s


def columns(s, th):
    """(mu, sigma) of the columns with support."""
    _, mu, sig, _ = O.quench(s, th)
    on = s.shapes.sum(0) > 0
    return mu[on], sig[on]


def score(s, th):
    """Distance of every bin from the nearest column with support, in its sigma."""
    mu, sig = columns(s, th)
    c = (np.arange(s.m_hi) + 0.5) * s.width
    return np.min(np.abs(c[:, None] - mu) / sig, axis=1)


def tile_mask(s, th, band, mu, sig):
    """[m_hi, columns]: the bins of the tiles that each column's band touches."""
    r0 = np.maximum(0, np.floor((mu - band * sig) / s.width)).astype(int)
    r1 = np.minimum(s.m_hi, np.floor((mu + band * sig) / s.width).astype(int) + 1)
    t = np.arange(s.m_hi)[:, None] // TILE
    return (r0 < r1) & (t >= r0 // TILE) & (t <= (r1 - 1) // TILE)


def touched(s, th, band=8.0, by=np.all):
    """Bins that every line reaches (by=np.any: some line)."""
    return by(tile_mask(s, th, band, *columns(s, th)), axis=1)


def tail_tol(s, th):
    mu, sig = columns(s, th)
    z = score(s, th)
    h = s.width / sig.min()
    dz = 4 * (mu.max() / sig.min() + z) * EPS
    return 32 * EPS + (2 * z * dz + 4 * EPS) / np.minimum(1.0, h * np.maximum(z, 1.0))


def complete(s, th):
    """Bins whose pile-up comes from touched tiles only (below the lines the next tile down is missing)."""
    first = int(np.argmax(touched(s, th)))
    m = np.arange(s.m_hi)
    return (s.L == 1) | (first == 0) | (m >= first + s.L) | ((m + 0.5) * s.width > columns(s, th)[0].min())


def empty(s):
    n = sum(s.hist_sizes().values())
    return s.with_counts(np.zeros(n))


def grad_ok(g, go, th):
    lhs = np.abs(g - go) * np.abs(th)
    return np.all(lhs <= 1e-9 * (1 + np.abs(go * th))), float(np.max(lhs / (1 + np.abs(go * th))))


# ---- bands wider than the default

@pytest.mark.parametrize("sigma", [0.7, 2.3, 4.5, 12.0])
@pytest.mark.parametrize("band", [10.0, 12.0, 20.0, 33.0, 36.0, 40.0])
def test_wide_band_tails_relative_to_themselves(band, sigma):
    s = empty(line_spec(sigma, 700))
    th = s.theta_true
    m = bx.Model(s, precision=bx.BX_FP64, band_sigmas=band)
    mg, mo = m.expected(th), O.expected(s, th)
    z = score(s, th)
    use = touched(s, th, band) & (z < min(band, 37.0))
    assert np.all(mo[use] > 0)
    rel = np.abs(mg[use] / mo[use] - 1)
    assert np.all(rel <= tail_tol(s, th)[use]), (float(rel.max()), float(z[use][np.argmax(rel / tail_tol(s, th)[use])]))
    m.close()


@pytest.mark.parametrize("band,z_event", [(36.0, -35.4), (40.0, -36.7), (40.0, 36.0), (20.0, 15.0)])
@pytest.mark.parametrize("sigma", [4.5, 6.0])
def test_event_at_the_end_of_a_wide_band(band, z_event, sigma):
    s = empty(line_spec(sigma, 700))
    th = s.theta_true
    mu, sig = columns(s, th)
    c = (np.arange(s.m_hi) + 0.5) * s.width
    edge = mu.min() if z_event < 0 else mu.max()
    b = int(np.argmin(np.abs((c - edge) / sig[0] - z_event)))
    s.counts["sub"][b] = 1.0
    m = bx.Model(s, precision=bx.BX_FP64, band_sigmas=band, max_batch=6)
    fo, go = O.nll(s, th, grad=True)
    for n in (1, 6):
        f, g = m.nll_batch(np.stack([th] * n), grad=True)
        assert np.all(2 * np.abs(f - fo) <= 1e-7), (f, fo)
        ok, worst = grad_ok(g[-1], go, th)
        assert ok, worst
    m.close()


# ---- bands that cut the response

def cut_reference(s, th, band):
    """(expected counts, -lnL, gradient by central differences) of the energy spectra when every column
    reaches the touched tiles only (the tiles held fixed in the differences)."""
    _, mu0, sig0, _ = O.quench(s, th)
    sup = s.shapes.sum(0) > 0
    tiles = tile_mask(s, th, band, mu0, sig0)
    for t in range(0, s.m_hi, TILE):   # a tile takes the columns from the first to the last that touches it
        i = np.nonzero(tiles[t] & sup)[0]
        tiles[t:t + TILE] = False
        if len(i):
            tiles[t:t + TILE, i[0]:i[-1] + 1] = True

    def expect(t):
        R, _ = O.response(s, t)
        v = (R * tiles) @ s.shapes.T
        w = [1 - s.tag_frac, s.tag_frac] if s.tag_frac is not None else [np.ones(s.K)]
        return np.concatenate([O.pileup(s, t[s.K + 5], v @ (t[:s.K] * x)) for x in w])

    n = s.counts_vector()

    def nll(t):
        u = expect(t)
        with np.errstate(divide="ignore", invalid="ignore"):
            return np.sum(u - n + np.where(n > 0, n * np.log(n / u), 0.0))

    g = np.zeros(s.P)
    for j in range(s.P):
        if th[j] == 0.0 or j == s.K + 6:
            continue
        h = 1e-4 * abs(th[j])
        d = []
        for q in (h, h / 2):
            a, b = th.copy(), th.copy()
            a[j] += q
            b[j] -= q
            d.append((nll(a) - nll(b)) / (2 * q))
        g[j] = (4 * d[1] - d[0]) / 3
    return expect(th), nll(th), g


@pytest.mark.parametrize("band,sigma,skew", [(3.0, 30.0, 0.0), (3.5, 9.0, 0.0), (4.5, 3.0, 0.0), (6.0, 60.0, 0.0),
                                             (7.9, 20.0, 0.0), (3.0, 30.0, 0.3), (4.0, 12.0, 0.05)])
@pytest.mark.parametrize("tag", [False, True])
def test_band_that_cuts_the_response(band, sigma, skew, tag):
    s = line_spec(sigma, 640, L=17, tag=tag)
    rng = np.random.default_rng(4)
    sh = s.shapes.copy()
    sh[1, 40:90] += rng.random(50) / 50
    s = dataclasses.replace(s, shapes=sh, resp_skew=skew)
    th = s.theta_true
    th[s.K + 1:s.K + 3] = 0.3, 1e-4
    mu = cut_reference(empty(s), th, band)[0]
    s = s.with_counts(np.where(mu > 0.5, np.floor(mu) + rng.integers(0, 2, mu.size), 0.0))
    mo, fo, go = cut_reference(s, th, band)
    m = bx.Model(s, precision=bx.BX_FP64, band_sigmas=band, max_batch=5)
    mg = m.expected(th)
    assert np.all(np.abs(mg - mo) <= 1e-12 * mo.max() + 1e-10 * np.abs(mo)), float(np.max(np.abs(mg - mo)) / mo.max())
    for n in (1, 5):
        f, g = m.nll_batch(np.stack([th] * n), grad=True)
        assert np.all(2 * np.abs(f - fo) <= 1e-7), (f, fo)
        # (the differences: 1e-4 steps extrapolated, rounding 1e-12 of -lnL over 1e-4)
        lhs = np.abs(g[-1] - go) * np.abs(th)
        lhs[s.K + 6] = 0.0
        assert np.all(lhs <= 1e-6 * (1 + np.abs(go * th)) + 1e-7 * abs(fo)), lhs
    m.close()


# ---- bins beyond the default band

def far_bins(s, th, zs):
    """The bins nearest to the scores zs above the last line and below the first, inside the axis."""
    mu, sig = columns(s, th)
    c = (np.arange(s.m_hi) + 0.5) * s.width
    out = []
    for z in zs:
        for edge, sg in ((mu.max(), 1), (mu.min(), -1)):
            x = edge + sg * z * sig[0]
            if c[0] <= x <= c[-1]:
                out.append(int(np.argmin(np.abs(c - x))))
    return sorted(set(out))


SIGMAS = [0.6, 1.3, 3.0, 5.2, 9.9, 16.0, 39.0, 70.0]


@pytest.mark.parametrize("L", [1, 3, 40, 400])
@pytest.mark.parametrize("sigma", SIGMAS)
def test_tails_of_the_default_band_relative_to_themselves(sigma, L):
    s = empty(line_spec(sigma, 900, L=L))
    th = s.theta_true
    m = bx.Model(s, precision=bx.BX_FP64)
    mg, mo = m.expected(th), O.expected(s, th)
    reach = touched(s, th)
    z = score(s, th)
    use = reach & (z < 37.0)
    use &= complete(s, th)
    tol = tail_tol(s, th)[use]
    rel = np.abs(mg[use] / mo[use] - 1)
    assert np.all(rel <= tol), (float(rel.max()), float(z[use][np.argmax(rel / tol)]))
    if L == 1:
        assert np.all(mg[~touched(s, th, by=np.any)] == 0.0)
    m.close()


@pytest.mark.parametrize("L", [1, 40, 400])
@pytest.mark.parametrize("sigma", SIGMAS)
def test_event_beyond_the_default_band(sigma, L):
    s0 = empty(line_spec(sigma, 900, L=L, tag=True))
    th = s0.theta_true
    reach = touched(s0, th)
    rng = np.random.default_rng(1)
    base = [rng.poisson(np.minimum(x, 1e6)).astype(float) for x in np.split(O.expected(s0, th), 2)]
    keep = score(s0, th) < 4.0
    reach &= complete(s0, th)
    bins = [b for b in far_bins(s0, th, (5.0, 6.2, 7.4, 8.3, 8.8, 9.5, 12.0, 20.0, 33.0)) if reach[b]]
    assert bins
    for j, b in enumerate(bins):
        s = dataclasses.replace(s0, counts={})
        s.counts = {"sub": np.where(keep, base[0], 0.0), "tag": np.where(keep, base[1], 0.0)}
        s.counts["tag" if j % 2 else "sub"][b] = 1.0
        m = bx.Model(s, precision=bx.BX_FP64, max_batch=6)
        fo, go = O.nll(s, th, grad=True)
        for n in (1, 6):
            f, g = m.nll_batch(np.stack([th] * n), grad=True)
            assert np.all(2 * np.abs(f - fo) <= 1e-7), (b, f, fo)
            ok, worst = grad_ok(g[-1], go, th)
            assert ok, (b, worst)
        m.close()


@pytest.mark.parametrize("sigma", [9.9, 16.0, 39.0])
def test_no_tile_beyond_the_default_band(sigma):
    """Without pile-up an event in the first bins of a tile that no band touches has no expected count."""
    s = empty(line_spec(sigma, 900))
    th = s.theta_true.copy()
    _, q, _, _ = O.quench(s, th)
    # the last line's band ends on a tile's last bin
    mu, sig = columns(s, th)
    last = (np.ceil((mu.max() + 8 * sigma) / TILE) + (1 if sigma > 30 else 0)) * TILE - 0.5
    th[s.K] *= (last - 8 * sigma) / mu.max()
    end = int(last + 0.5)
    some = touched(s, th, by=np.any)
    assert not some[end] and some[end - 1]
    for b, inside in ((end - 1, True), (end, False), (end + 3, False)):   # (8 sigma past the last line, and on)
        s.counts["sub"][:] = 0.0
        s.counts["sub"][b] = 1.0
        m = bx.Model(s, precision=bx.BX_FP64)
        assert (m.expected(th)[b] > 0) == inside
        if inside:
            assert 2 * abs(m.nll(th) - O.nll(s, th)) <= 1e-7
        else:
            with pytest.raises(bx.BxError) as e:
                m.nll(th)
            assert e.value.status == bx.BX_EDOMAIN
        m.close()


@pytest.mark.parametrize("skew,kurt", [(0.05, 0.05), (0.0, 0.05)])
@pytest.mark.parametrize("sigma", [3.0, 9.9, 39.0])
def test_gram_charlier_events_in_the_tails(sigma, skew, kurt):
    s = empty(dataclasses.replace(line_spec(sigma, 900), resp_skew=skew, resp_kurt=kurt))
    th = s.theta_true
    reach = touched(s, th)
    mo = O.expected(s, th)
    bins = [b for b in far_bins(s, th, (5.5, 7.3, 8.5, 9.4)) if reach[b] and mo[b] > 0]
    assert bins
    for b in bins:
        s.counts["sub"][:] = 0.0
        s.counts["sub"][b] = 1.0
        m = bx.Model(s, precision=bx.BX_FP64)
        fo, go = O.nll(s, th, grad=True)
        f, g = m.nll_grad(th)
        assert 2 * abs(f - fo) <= 1e-7, (b, f, fo)
        ok, worst = grad_ok(g, go, th)
        assert ok, (b, worst)
        m.close()


# ---- a spectrum that ends

@pytest.mark.parametrize("sigma,skew", [(4.0, 0.0), (9.9, 0.0), (21.0, 0.0), (44.0, 0.0), (13.0, 0.05)])
@pytest.mark.parametrize("L", [1, 2, 40, 150])
def test_past_the_end_of_a_spectrum(sigma, skew, L):
    """Many columns up to an end: bins past it are known to 2e-12 of themselves although the columns further
    back end before them, and an event there has its -lnL and gradient.  (Reference: the response matrix
    under the tile rule; the pile-up of a bin may hold tails known to 1e-12 of it.)"""
    s = line_spec(sigma, 900, L=L, tag=True)
    sh = np.zeros((2, 128))
    sh[0, 25:64] = np.linspace(1.0, 3.0, 39)
    sh[1, 30:64] = np.linspace(2.0, 1.0, 34)
    s = dataclasses.replace(s, shapes=sh / sh.sum(1, keepdims=True), resp_skew=skew, resp_kurt=skew, counts={})
    th = s.theta_true.copy()
    th[:s.K] *= 30.0
    th[s.K + 1:s.K + 3] = 0.1, 1e-4
    s = empty(s)
    mo = cut_reference(s, th, 8.0)[0]
    m = bx.Model(s, precision=bx.BX_FP64)
    mg = m.expected(th)
    m.close()
    z = np.tile(score(s, th), 2)
    use = (mo > 1e-200) & (z < 30)
    rel = np.abs(mg[use] / mo[use] - 1)
    tol = 2e-12 + np.tile(tail_tol(s, th), 2)[use]
    assert np.all(rel <= tol), (float(rel.max()), float(z[use][np.argmax(rel / tol)]))
    # events where 1e-3 to 1e-40 are expected
    rng = np.random.default_rng(2)
    n = rng.poisson(np.maximum(mo, 0.0)).astype(float)
    for lo, hi in ((1e-4, 1e-2), (1e-12, 1e-9), (1e-40, 1e-20)):
        b = np.nonzero((mo > lo) & (mo < hi))[0]
        if len(b):
            n[b[len(b) // 2]] = 1.0
    s = s.with_counts(n)
    _, fo, go = cut_reference(s, th, 8.0)
    m = bx.Model(s, precision=bx.BX_FP64, max_batch=6)
    for k in (1, 6):
        f, g = m.nll_batch(np.stack([th] * k), grad=True)
        assert np.all(2 * np.abs(f - fo) <= 1e-7), (f, fo)
        lhs = np.abs(g[-1] - go) * np.abs(th)
        lhs[s.K + 6] = 0.0
        # (differences of a -lnL with terms that change by their whole size over a step: 1e-5 of each)
        assert np.all(lhs <= 1e-5 * (1 + np.abs(go * th)) + 1e-7 * abs(fo)), lhs
    m.close()


@pytest.mark.parametrize("ratio", [30.0, 150.0, 500.0, 2000.0, 1e5])
@pytest.mark.parametrize("L", [1, 40])
def test_strong_columns_behind_a_weak_line(L, ratio):
    """Bins 3.5 sigma and more past a weak line, where strong columns 8.5 sigma off and more are 1e-12 of the
    count each: those that do not touch the tile are not in it, those that do are in it beyond 9 sigma."""
    s = line_spec(40.0, 900, L=L, tag=True)
    sh = np.zeros((2, 128))
    sh[0, 4:16] = ratio
    sh[1, 2:14] = ratio
    sh[:, 62:64] = 1.0
    s = empty(dataclasses.replace(s, shapes=sh / sh.sum(1, keepdims=True), counts={}))
    th = s.theta_true.copy()
    mo = cut_reference(s, th, 8.0)[0]
    m = bx.Model(s, precision=bx.BX_FP64)
    mg = m.expected(th)
    m.close()
    z = np.tile(score(s, th), 2)
    use = (mo > 1e-200) & (z < 30)
    rel = np.abs(mg[use] / mo[use] - 1)
    tol = 2e-12 + np.tile(tail_tol(s, th), 2)[use]
    assert np.all(rel <= tol), (float(rel.max()), float(z[use][np.argmax(rel / tol)]))

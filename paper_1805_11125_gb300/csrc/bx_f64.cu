// bx_f64.cu -- the FP64 model (BX_FP64): every quantity of Eq. 1 - 4 and its adjoint in FP64.
//
// GB300 issues FP64 at 1/64 of its FP32 rate (about 2 lanes per clock and SM), so the stage costs
// are FP64 operations per response entry.  A bin-integrated response R[m,i] = Phi(z_{m+1}) -
// Phi(z_m) from two erfc calls is ~100 of them.  This path samples instead: with the density
//   rho_i(y) = exp(-z^2 / 2) / (sqrt(2 pi) sigma_i),   z = (y - mu_i) / sigma_i,
// the Eq. 3 spectrum is the bin integral of ONE smooth function,
//   lambda_h[m] = int_{bin m} f_h(y) dy,   f_h(y) = sum_i S_h[i] norm_i rho_i(y),
// so f_h is summed at the points of a grid and integrated per bin (not per entry) by a stencil:
// the integral over the bin of the polynomial through the 2 R64 + 1 nearest samples.  Columns are
// grouped by width into classes c = 0 .. 6 with sample spacing d = 2^c w, such that h = d / sigma
// lies in (0.1, 0.2]: a column takes 90 - 180 samples whatever its width (its bins are 16 sigma / w,
// 160 - 640 at w = 1 npe).  Down a column the samples follow by a recurrence (two multiplications
// each) from an exact start every RUN64 samples.
// A column contributes to every bin of the 128-bin tiles that its band (8 sigma) touches and to no other
// tile; its samples end one sigma past the band.  A bin with content within about 3.5 sigma is known to
// 1e-14 of itself (the stencil is good to 1e-17 of the largest sample it meets, the columns that end before
// the bin are below 4e-15 of it).  In the tails beyond (k_lam64 marks them) the error of lambda is bounded,
// and the bins whose expected count needs better -- those with an event, and the expected counts a caller
// asks for -- take the exact bin masses of their tile's columns (tail_bins, tail_adjoint).
// Columns too narrow for that (h > 0.2 at d = w) form class CI on the bins themselves, each entry
// the exact bin mass: phi(z) times a polynomial in z^2 (kind P, sigma >= 0.8 w), or the difference of
// erfc tails (kind D: narrower still, or a narrow Gram-Charlier column).  Any band_sigmas but the
// default 8 puts every column into CI, with all bins of the 128-bin tiles that its band touches: a wider
// band asks for the far tails relative to themselves, and a narrower one cuts the response where it is
// not small, which a stencil cannot follow.
//
// The adjoint is the exact transpose: the row weights go through the transposed stencils onto the
// class grids (k_wt64), and each column sums Wt p, Wt z p, Wt z^2 p over its own samples.
//
//   k_scan64   per 128 columns: Birks prefix sums Q_i, dQ_i/dkB
//   k_cols64   per column: mu, sigma, normalisation, window masses, spectra, class, sample range
//   k_dens64   per 32-sample tile of a class grid: F_h[g] = sum_i A_i S_h[i] p_i[g], and for the
//              Eq. 4 terms each column's sum_g p_i[g] Gt_s[g]
//   k_lam64    per bin: lambda_h[m] from the class grids, and whether it lies in the tails; per chunk:
//              the Eq. 4 sums of every species
//   k_pile64   per 32 window bins: Eq. 2, the -lnL terms and weights 1 - n/mu
//   k_marg64   per item: Eq. 4 marginals and their terms, -lnL, the species' adjoint coefficients
//   k_corr64   per 32 axis bins: adjoint of Eq. 2;   k_wt64: row weights onto the class grids
//   k_bwd64    per 32 columns: adjoint of Eq. 1, chain rule, rate gradient
// Every sum has a fixed order.  Measured on a GB300 at 2070 MHz against the per-entry erfc form this
// replaced (one erfc per bin edge in the forward, one erfc and one exp in the adjoint): the
// multivariate model 52 evaluations with gradient 19.2 -> 1.22 ms, the plain model 1000 values
// 79.8 -> 3.7 ms, one plain value 4.2 -> 0.13 ms.
#include <limits.h>
#include <math.h>

#include <vector>

#include "bx_internal.cuh"

namespace bx {

constexpr int R64 = G64_R;              // stencil: R64 samples each side of the bin's own
constexpr int TAPS = 2 * R64 + 1;
constexpr int RUN64 = 16;               // samples per exact start of the recurrence
constexpr int RUNB = 16;                // the same in the adjoint
constexpr double HMAX = 0.2;            // largest spacing / sigma of a sampled column
constexpr double HPOLY = 1.25;          // largest w / sigma of kind P (its polynomial's rest: poly_coef)
constexpr double BAND_S = 8.0;          // band_sigmas of the sampled columns (the default)
constexpr double ZRUN = 37.0;           // |z| of the runs of kind P: z^2 / 2 < 700 (exp_tab)
constexpr int NPOLY = 16;               // kind P: terms of the bin-mass polynomial in z^2
enum { KIND_S = 0, KIND_P = 1, KIND_D = 2 };

// Class grids of an axis of M bins, one after the other, each padded to whole 32-sample tiles:
// classes 0 .. G64_NC - 1 (sample g' = g + R64 at y = (g + 1/2) 2^c w), then CI (the bins).
__host__ __device__ inline int g64_len(int M, int c) {
    const int n = c == G64_CI ? M : ((M + (1 << c) - 1) >> c) + 2 * R64;
    return (n + 31) & ~31;
}
__host__ __device__ inline int g64_off(int M, int c) {
    int o = 0;
    for (int q = 0; q < c; ++q) o += g64_len(M, q);
    return o;
}
int g64_total(int M) { return g64_off(M, G64_NC + 1); }
static int wt64_threads(int M);
int g64_wt_threads(int M) { return wt64_threads(M); }

// Host tables: the stencils of every class and phase -- weight j of phase ph of class c is the
// integral over u in [ph / 2^c - 1/2, (ph + 1) / 2^c - 1/2] (the bin, in units of the spacing, its
// cell's sample at 0) of the Lagrange polynomial of node j - R64 -- and 2^(j / 64), j < 64.
static std::vector<double> make_tables() {
    typedef long double ld;
    constexpr int NG = R64 + 2;   // Gauss-Legendre points (degree 2 R64 needs R64 + 1; even: no point on a node)
    ld gx[NG], gw[NG], bw[TAPS];
    for (int i = 0; i < NG; ++i) {
        ld z = cosl(3.14159265358979323846L * (i + 0.75L) / (NG + 0.5L)), dp = 0;
        for (int it = 0; it < 60; ++it) {
            ld p1 = 1, p2 = 0;
            for (int j = 1; j <= NG; ++j) {
                const ld p3 = p2;
                p2 = p1;
                p1 = ((2 * j - 1) * z * p2 - (j - 1) * p3) / j;
            }
            dp = NG * (z * p1 - p2) / (z * z - 1);
            const ld dz = p1 / dp;
            z -= dz;
            if (fabsl(dz) < 1e-18L) break;
        }
        gx[i] = z;
        gw[i] = 2 / ((1 - z * z) * dp * dp);
    }
    for (int j = -R64; j <= R64; ++j) {   // 1 / prod_{k != j} (j - k)
        ld q = 1;
        for (int k = -R64; k <= R64; ++k)
            if (k != j) q *= j - k;
        bw[j + R64] = 1 / q;
    }
    std::vector<double> out;
    for (int c = 0; c < G64_NC; ++c)
        for (int ph = 0; ph < (1 << c); ++ph) {
            const ld h = 1.0L / (1 << c), a = ph * h - 0.5L;
            ld s[TAPS] = {};
            for (int q = 0; q < NG; ++q) {
                const ld u = a + 0.5L * h * (1 + gx[q]);
                ld all = 0.5L * h * gw[q];
                for (int k = -R64; k <= R64; ++k) all *= u - k;
                for (int j = -R64; j <= R64; ++j) s[j + R64] += all * bw[j + R64] / (u - j);
            }
            for (int j = 0; j < TAPS; ++j) out.push_back((double)s[j]);
        }
    for (int j = 0; j < 64; ++j) out.push_back((double)exp2l((ld)j / 64));
    return out;
}
const std::vector<double>& g64_tables() {   // constants: made once
    static const std::vector<double> tab = make_tables();
    return tab;
}
__device__ __forceinline__ const double* g64_stencil(const Work& w, int c, int ph) {
    return w.tab64 + ((1 << c) - 1 + ph) * TAPS;
}
constexpr int EXP_OFF = ((1 << G64_NC) - 1) * TAPS;   // the 2^(j/64) table within tab64

// exp(x) for |x| <= 700 (clamped) by table and polynomial (Tang 1989): x = (64 e + j + f) ln2 / 64,
// |f| <= 1/2, exp(x) = 2^e 2^(j/64) e^r with |r| <= ln2 / 128: e^r - 1 from its Taylor series through
// r^5 (truncation 3e-17).  12 FP64 operations; ~1 ulp.
__device__ __forceinline__ double exp_tab(double x, const double* __restrict__ T) {
    x = fmin(fmax(x, -700.0), 700.0);
    const double t = fma(x, 92.332482616893656877, 6755399441055744.0);   // 64 / ln 2; 1.5 * 2^52
    const double n = t - 6755399441055744.0;
    double r = fma(n, -0.010830424696249145, x);              // ln 2 / 64, high and low part
    r = fma(n, -3.623510646634843e-19, r);
    const int k = __double2loint(t);
    const double tv = T[k & 63];
    const double ts = __hiloint2double(__double2hiint(tv) + ((k >> 6) << 20), __double2loint(tv));
    double q = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    q = fma(r, q, 1.0 / 6.0);
    q = fma(r, q, 0.5);
    q = fma(r * r, q, r);
    return fma(ts, q, ts);
}

// Sum of 32 values per lane over the warp at once: lane j returns the sum of v[j] (each step
// exchanges halves: 31 additions where 32 butterflies take 160).
__device__ __forceinline__ double warp_sum32(double (&v)[32]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j < o) {
                const double give = up ? v[j] : v[j + o];
                const double keep = up ? v[j + o] : v[j];
                v[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
    }
    return v[0];
}

constexpr double Q_CUT64 = 9.0;   // Q(x) = 1 - Phi(x) taken as 0 from here on (1.1e-19)
__device__ __forceinline__ double tail64(double x) {
    return x >= Q_CUT64 ? 0.0 : 0.5 * erfc(x * 0.70710678118654752440);
}
__device__ __forceinline__ double mass64(double a, double b) {
    if (a >= 0.0) return tail64(a) - tail64(b);
    if (b <= 0.0) return tail64(-b) - tail64(-a);
    return 1.0 - tail64(b) - tail64(-a);
}

// ------------------------------------------------------------------ column stage

// Q_i = sum_{j<i} x_j + x_i / 2, x_j = dE / (1 + kB xi S_j), and dQ_i/dkB, within blocks of 128
// columns; k_cols64 adds the blocks before.  CTA = (item, 128 columns): one block per item spent 19 us
// on a single SM's FP64 pipe (25 operations a column).
__global__ void __launch_bounds__(128) k_scan64(Work w, int nblk) {
    const int item = blockIdx.x / nblk, blk = blockIdx.x % nblk, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (w.skip && w.skip[item]) {
        if (tid == 0 && blk == 0) w.status[item] = STATUS_SKIPPED;
        return;
    }
    const Toy& T = w.toys[w.toy_of[item]];
    const int K = T.K;
    const double* th = w.theta + (size_t)item * w.tstride;
    if (blk == 0) {
        bool bad = tid < T.P && !isfinite(th[tid]);
        if (tid == 0 && (!(th[K] > 0.0) || (T.n_rad > 0 && !(th[K + 6] > 0.0)))) bad = true;
        const int any = __syncthreads_or(bad);
        if (tid == 0) {
            w.status[item] = any ? (int)BX_EDOMAIN : 0;
            w.cmask64[item] = 0;
            w.xany64[item] = 0;
            w.tmask64[item] = 0ull;
        }
    }
    // (with several column sets a set starts on a block: Ncs is a multiple of 128)
    const int ie = blk * 128 + tid, grp = T.n_set > 1 ? ie / T.Ncs : 0, i = ie - grp * T.Ncs;
    const bool in = ie < T.Next && i < T.N;
    double x = 0.0, y = 0.0;
    if (in) {
        const double xi = w.multi_set ? T.xi[grp] : 1.0, S = T.stop_pow[i], rq = 1.0 / (1.0 + th[K + 4] * xi * S);
        x = T.dE * rq;
        y = -x * S * rq * xi;
    }
    double ix = x, iy = y;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double a = __shfl_up_sync(0xffffffffu, ix, o), b = __shfl_up_sync(0xffffffffu, iy, o);
        if (lane >= o) { ix += a; iy += b; }
    }
    __shared__ double2 sh[4];
    if (lane == 31) sh[wid] = make_double2(ix, iy);
    __syncthreads();
    double ax = 0.0, ay = 0.0;
    for (int q = 0; q < wid; ++q) { ax += sh[q].x; ay += sh[q].y; }
    const double ex = __shfl_up_sync(0xffffffffu, ix, 1), ey = __shfl_up_sync(0xffffffffu, iy, 1);
    if (lane > 0) { ax += ex; ay += ey; }
    w.colq[(size_t)item * w.Npad + ie] = make_double2(ax + 0.5 * x, ay + 0.5 * y);
    if (tid == 127) w.qtot64[(size_t)item * (w.Npad / 128) + blk] = make_double2(ax + x, ay + y);
}

// Bins [r0, r1) within nsig sigma of a column's mean.
__device__ __forceinline__ void near_bins(double mu, double sig, double w, int M, float nsig, int& r0, int& r1) {
    const float muf = (float)mu, sigf = (float)sig, wf = (float)w, iwf = 1.0f / wf;
    const float e_min = -2.0f * wf, e_max = (M + 2.0f) * wf;
    r0 = max(0, (int)floorf(fminf(fmaxf(muf - nsig * sigf, e_min), e_max) * iwf));
    r1 = min(M, (int)floorf(fminf(fmaxf(muf + nsig * sigf, e_min), e_max) * iwf) + 1);
}

// One thread per column, a warp per 32-column chunk: Eq. 1's mean and width, the normalisation
// 1/Phi(mu/sigma), the masses of the energy slices, the spectra S_h[i] = sum_k r_k c_{h,k} s_k[i]
// times the column's amplitude, its class, kind and sample range, and per chunk the sample range of
// each class.
template <bool MULTI>
__global__ void __launch_bounds__(128) k_cols64(Work w, int nblk) {
    const int item = blockIdx.x / nblk, chunk = (blockIdx.x % nblk) * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (w.status[item] == STATUS_SKIPPED) return;
    const Toy& T = w.toys[w.toy_of[item]];
    const int K = T.K, N = T.N, M = T.M, NES = T.n_es;
    const double* th = w.theta + (size_t)item * w.tstride;
    const int ie = chunk * 32 + lane;
    // (a chunk lies within one set: with several, Ncs is a multiple of 128; with one, the lanes past its
    // last column stay in it too, since the warp shares the block sums below)
    const int grp = MULTI && T.n_set > 1 ? ie / T.Ncs : 0, i = ie - grp * T.Ncs;
    const bool in = ie < T.Next && i < N;
    const size_t at = (size_t)item * w.Npad + ie;
    double* aW = w.aW + (size_t)item * w.nes * w.Npad;
    int g0 = 0, g1 = 0, cls = -1, kind = KIND_S, nrow = 0;
    unsigned tlo = 0u, thi = 0u;   // tiles of 128 bins that the column's band touches
    Col64 cc{0.0, 1.0, 0.0, 0.0};
    double2 sp = make_double2(0.0, 0.0);
    Gen64 gen{0.0, 0.0, 0.0, 0.0};   // mu, 1/sigma, 1 - e^(-h^2), amplitude
    double aw[MAX_ES] = {0.0, 0.0, 0.0, 0.0};
    // the Birks sums of this column set's blocks before this one
    double2 q = make_double2(0.0, 0.0);
    {
        const int b1 = blockIdx.x % nblk, b0 = grp * (T.Ncs / 128);
        double qx = 0.0, qy = 0.0;
        for (int bq = b0 + lane; bq < b1; bq += 32) {
            const double2 t = w.qtot64[(size_t)item * nblk + bq];
            qx += t.x;
            qy += t.y;
        }
        qx = warp_sum(qx);
        qy = warp_sum(qy);
        if (in) {
            const double lyf = T.n_shell ? T.lyf[grp] : 1.0;   // a shell's light-yield factor, folded into Q
            q = w.colq[at];
            q = make_double2((q.x + qx) * lyf, (q.y + qy) * lyf);
        }
        w.colq[at] = q;
    }
    if (in) {
        const double LY = th[K], a = th[K + 1], b = th[K + 2], c = th[K + 3];
        const double xi = MULTI ? T.xi[grp] : 1.0;
        bool bad = !(1.0 + th[K + 4] * xi * T.stop_pow[i] > 0.0);
        bool nz = false;   // a species of this column's set has support in it
        double ssub = 0.0, stag = 0.0;
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
            const double wk = set_weight<MULTI>(T, k, grp);
            const double s0 = T.shapes[(size_t)k * N + i];
            if (wk == 0.0) continue;
            nz |= s0 != 0.0;
            const double sk = s0 * th[k] * wk, t = T.tag ? T.tag[k] : 0.0;
            ssub += (T.tag ? 1.0 - t : 1.0) * sk;
            stag += t * sk;
        }
        const bool live = !MULTI || T.n_shell || nz;   // a quenching group's column without support
        if (live) {
            const double mu = LY * q.x;
            const double var = fma(fma(b, mu, a), mu, c);
            const bool ok = var > 0.0;
            if (!ok) bad = true;
            const double isig = rsqrt(fmax(var, 1e-300)), sig = var * isig, z = mu * isig;
            double norm = 1.0, mills = 0.0;
            const bool gc = T.gc1 != 0.0 || T.gc2 != 0.0;
            if (z < Q_CUT64) {   // mass above 0 npe and the density there over it
                double Phi = z > 0.0 ? 1.0 - tail64(z) : tail64(-z), dens = INV_SQRT_2PI * exp(-0.5 * z * z);
                if (gc) {
                    Phi += gc_cdf_term(T, -z);
                    dens *= gc_density_factor(T, -z);
                }
                norm = 1.0 / Phi;
                mills = dens * norm;
            }
            cc = Col64{mu, sig, norm, mills};
            for (int e = 0; e < NES; ++e) {   // masses of the energy slices (Eq. 4)
                const double za = (T.es_lo[e] * T.w - mu) * isig, zb = (T.es_hi[e] * T.w - mu) * isig;
                double m = mass64(za, zb);
                if (gc) m -= gc_cdf_term(T, zb) - gc_cdf_term(T, za);
                aw[e] = m * norm;
            }
            // class: the widest spacing with h <= HMAX; or the bins
            const double hw = T.w * isig;
            // A column is left out when no bin lies within band sigma of its mean; its samples reach one
            // sigma further: what a cut at 8 sigma leaves out (6e-16 of a column's mass, 5e-15 of its slope)
            // was the largest error of the gradient (2.7e-13 of it over 21 models of every response
            // variant; 6.5e-15 without the cut, 5.2e-14 in the erfc form this replaced).
            const float muf = (float)mu, sigf = (float)sig, bandf = (float)w.band, wf = (float)T.w;
            double h = hw, amp = norm;
            near_bins(mu, sig, T.w, M, bandf, g0, g1);
            const bool valid = ok && g0 < g1 && (!MULTI || nz);
            if (valid) {
                nrow = g1 - g0;
                const unsigned long long tm = (2ull << ((g1 - 1) / TM)) - (1ull << (g0 / TM));
                tlo = (unsigned)tm;
                thi = (unsigned)(tm >> 32);
            }
            if (hw <= HMAX && w.band == BAND_S) {
                int c2 = 0;
                while (c2 < G64_NC - 1 && 2.0 * h <= HMAX) {
                    h *= 2.0;
                    ++c2;
                }
                cls = c2;
                amp = norm * INV_SQRT_2PI * h;
                const float id = 1.0f / (wf * (float)(1 << c2)), ext = (bandf + 1.0f) * sigf;
                const int len = ((M + (1 << c2) - 1) >> c2) + 2 * R64;
                const float lo_g = fminf(fmaxf((muf - ext) * id - 0.5f, -(float)R64 - 8.0f), (float)len);
                const float hi_g = fminf(fmaxf((muf + ext) * id - 0.5f, -(float)R64 - 8.0f), (float)len);
                g0 = max(0, (int)ceilf(lo_g) - 1 + R64);
                g1 = min(len, (int)floorf(hi_g) + 2 + R64);
                kind = KIND_S;
            } else {
                cls = G64_CI;
                if (w.band == BAND_S) {
                    near_bins(mu, sig, T.w, M, bandf + 1.0f, g0, g1);
                } else {   // every bin of the tiles that the band touches
                    g0 &= ~(TM - 1);
                    g1 = min(M, (g1 + TM - 1) & ~(TM - 1));
                }
                // kind P where its polynomial holds and its runs start in the range of exp_tab (a start
                // may lie up to RUN64 - 1 bins below the first bin of the column)
                const double z0 = ((double)(g0 - RUN64) * T.w - mu) * isig, z1 = ((double)g1 * T.w - mu) * isig;
                const double zm = fmax(-z0, z1);
                kind = gc || hw > HPOLY || zm > ZRUN || (w.band != BAND_S && hw * zm > 8.0 * HPOLY) ? KIND_D : KIND_P;
                if (kind == KIND_P) amp = norm * INV_SQRT_2PI * hw;
            }
            if (!valid || g0 >= g1) {
                g0 = g1 = 0;
                cls = -1;
            }
            gen = Gen64{mu, isig, -expm1(-h * h), amp};
            sp = make_double2(ssub * amp, stag * amp);
        }
        if (bad) w.status[item] = BX_EDOMAIN;
    }
    w.col64[at] = cc;
    w.colS[at] = sp;
    w.gen64[at] = gen;
    w.colc64[at] = make_int4(cls, kind, g0, g1);
    for (int e = 0; e < w.nes; ++e) aW[(size_t)e * w.Npad + ie] = e < NES ? aw[e] : 0.0;
    if (w.count_units) {
        const int r = __reduce_add_sync(0xffffffffu, nrow);
        if (lane == 0 && r) atomicAdd(w.units, (unsigned long long)r);
    }
    tlo = __reduce_or_sync(0xffffffffu, tlo);
    thi = __reduce_or_sync(0xffffffffu, thi);
    if (lane == 0) {
        w.ctile64[(size_t)item * (w.Npad / 32) + chunk] = make_uint2(tlo, thi);
        if (tlo | thi) atomicOr(&w.tmask64[item], (unsigned long long)thi << 32 | tlo);
    }
    int mask = 0;
    for (int c = 0; c <= G64_NC; ++c) {
        const unsigned here = __ballot_sync(0xffffffffu, cls == c);
        int2 r = make_int2(0, 0);
        if (here) {
            mask |= 1 << c;
            r.x = __reduce_min_sync(0xffffffffu, cls == c ? g0 : INT_MAX);
            r.y = __reduce_max_sync(0xffffffffu, cls == c ? g1 : INT_MIN);
        }
        if (lane == c) w.chk64[((size_t)item * (w.Npad / 32) + chunk) * (G64_NC + 1) + c] = r;
    }
    if (lane == 0 && mask) atomicOr(&w.cmask64[item], mask);
}

// ------------------------------------------------------------------ the generator

// The bin mass of a column of sigma >= 0.8 w over its bin centred at standard score z:
// int phi = w / sigma phi(z) sum_k C_k z^(2k), from the Taylor series of phi about the centre
// (sum_j t^j He_2j(z) / (2j + 1)!, t = (w / 2 sigma)^2) collected in powers of z^2:
//   C_k = t^k / (2k)! sum_i (-t/2)^i / (i! (2k + 2i + 1)).
// All C_k > 0; the truncated rest, (z w / 2 sigma)^32 / 33! of the mass, is 2e-17 of it at |z| = 6 and
// w = 1.25 sigma and 2e-14 at the band's end, |z| = 8.
__device__ __forceinline__ void poly_coef(double hw, double (&C)[NPOLY]) {
    const double t = 0.25 * hw * hw;
    double uq[11];   // (-t/2) / (i + 1): products with constants, no divisions
#pragma unroll
    for (int q = 0; q < 11; ++q) uq[q] = t * (-0.5 / (q + 1));
    double tk = 1.0;   // t^k / (2k)!
#pragma unroll
    for (int k = 0; k < NPOLY; ++k) {
        double s = 0.0;
#pragma unroll
        for (int q = 10; q >= 0; --q) s = fma(s, uq[q], 1.0 / (2 * k + 2 * q + 1));   // nested sum over i
        C[k] = tk * s;
        tk *= t * (1.0 / ((2 * k + 1) * (2 * k + 2)));
    }
}
__device__ __forceinline__ double poly_eval(const double (&C)[NPOLY], double x) {
    double s = C[NPOLY - 1];
#pragma unroll
    for (int k = NPOLY - 2; k >= 0; --k) s = fma(s, x, C[k]);
    return s;
}
// lower-tail form of the (Gram-Charlier) CDF at an edge: t = Phi(z) for z < 0, -Q(z) otherwise (f)
__device__ __forceinline__ double edge_tail(const Toy& T, double z, bool gc, bool& f) {
    f = z >= 0.0;
    double t = f ? -0.5 * erfc(z * 0.70710678118654752440) : 0.5 * erfc(-z * 0.70710678118654752440);
    if (gc) t -= gc_cdf_term(T, z);
    return t;
}

// ------------------------------------------------------------------ forward

// CTA = 32 samples of one class grid of one item; its four warps share the 32-column chunks that
// touch the tile.  Per chunk: lane = column, the column's samples down the tile by the recurrence
// (exact starts every RUN64) into a padded shared tile, its sum against Gt_s on the way; then
// lane = sample, the 32 columns' contributions added.  FP64-bound: 2 (recurrence) + 1.8 (starts) +
// 1 (Eq. 4 column sum) + 1 per spectrum = ~7 operations an entry.
// TAG: two spectra; ES: energy slices of the Eq. 4 terms the instantiation holds (0: no such terms).
// NW = 4: one CTA per tile, its warps taking every fourth chunk.  NW = 1 (small batches, whose tiles
// leave SMs idle): a CTA per warp share, the four partial sums as planes that k_lam64 adds in the
// same order, so the results do not depend on the choice.
template <bool TAG, int ES, bool GC, int NW>
__global__ void __launch_bounds__(32 * NW) k_dens64(Work w, int ntile) {
    constexpr bool COLS = ES > 0;
    const int unit = NW == 4 ? (int)blockIdx.x : (int)(blockIdx.x >> 2);
    const int item = unit / ntile, tile = unit % ntile, tid = threadIdx.x, lane = tid & 31, wq = tid >> 5;
    const int share = NW == 4 ? wq : (int)(blockIdx.x & 3);
    if (w.status[item]) return;
    const Toy& T = w.toys[w.toy_of[item]];
    const int M = T.M, present = w.cmask64[item];
    int c = 0, off = 0;
    for (; c <= G64_NC; ++c) {
        const int len = g64_len(M, c);
        if (tile * 32 < off + len) break;
        off += len;
    }
    if (c > G64_NC || !((present >> c) & 1)) return;
    const int gt = tile * 32 - off;   // first sample of the tile in its class grid
    const int NES = ES > 1 ? T.n_es : ES, nch = (T.Next + 31) / 32;
    const int nchp = w.Npad / 32;
    __shared__ double sT[NW][32][33];
    __shared__ double2 sS[NW][32];
    __shared__ double sG[COLS ? ES : 1][32];
    __shared__ double sE[64];
    __shared__ unsigned short s_list[MAX_SETS * MAX_CB * 4];
    __shared__ int s_n;
    if (wq == 0) {   // the chunks whose columns of this class touch the tile, in order
        const int2* chk = w.chk64 + (size_t)item * nchp * (G64_NC + 1) + c;
        int n = 0;
        for (int b = 0; b < nch; b += 32) {
            const int q = b + lane;
            const int2 r = q < nch ? chk[(size_t)q * (G64_NC + 1)] : make_int2(0, 0);
            const bool hit = r.y > gt && r.x < gt + 32 && r.x < r.y;
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (hit) s_list[n + __popc(m & ((1u << lane) - 1u))] = (unsigned short)q;
            n += __popc(m);
        }
        if (lane == 0) s_n = n;
    }
    if (wq == NW - 1) {
        sE[lane] = w.tab64[EXP_OFF + lane];
        sE[lane + 32] = w.tab64[EXP_OFF + lane + 32];
    }
    if (COLS && wq == NW / 2)
        for (int e = 0; e < NES; ++e) sG[e][lane] = T.Gt64[(size_t)e * g64_off(M, G64_NC + 1) + tile * 32 + lane];
    __syncthreads();
    const int n = s_n;
    const double d = T.w * (double)(1 << (c == G64_CI ? 0 : c));
    // (CI: the bins' centres; class grids start R64 samples before the axis)
    const double y0 = ((double)(gt - (c == G64_CI ? 0 : R64)) + 0.5) * d;
    double Fs = 0.0, Ft = 0.0;
    for (int li = share; li < n; li += 4) {
        const int ie = (int)s_list[li] * 32 + lane;
        const size_t at = (size_t)item * w.Npad + ie;
        const int4 cp = w.colc64[at];
        const bool on = cp.x == c && cp.w > gt && cp.z < gt + 32;
        if (!__any_sync(0xffffffffu, on)) continue;   // (the chunk's range is the hull of its columns')
        const int a0 = on ? max(cp.z - gt, 0) : 32, a1 = on ? min(cp.w - gt, 32) : 0;
        const Gen64 gen = on ? w.gen64[at] : Gen64{0.0, 0.0, 0.0, 0.0};
        sS[wq][lane] = on ? w.colS[at] : make_double2(0.0, 0.0);
        const double h = d * gen.y;
        double cs[COLS ? ES : 1];
#pragma unroll
        for (int e = 0; e < ES; ++e) cs[e] = 0.0;
        double(*sc)[33] = sT[wq];
        auto put = [&](int k, double v) {
            sc[k][lane] = v;
            if (COLS) {
#pragma unroll
                for (int e = 0; e < ES; ++e)
                    if (e < NES) cs[e] = fma(v, sG[e][k], cs[e]);
            }
        };
        const bool isD = on && cp.y == KIND_D, go = on && !isD;
        const unsigned mD = __ballot_sync(0xffffffffu, isD);
        const bool anyD = mD != 0u;
        if (anyD) {   // kind D, one column at a time: lane = bin, a tail per edge
            if (!go)
                for (int k = 0; k < 32; ++k) sc[k][lane] = 0.0;
            __syncwarp();
            const bool gc = GC && (T.gc1 != 0.0 || T.gc2 != 0.0);
            for (unsigned mr = mD; mr; mr &= mr - 1u) {
                const int j = __ffs(mr) - 1, b0 = __shfl_sync(0xffffffffu, a0, j), b1 = __shfl_sync(0xffffffffu, a1, j);
                const double mu = __shfl_sync(0xffffffffu, gen.x, j), isg = __shfl_sync(0xffffffffu, gen.y, j);
                bool fa, fz = false;
                const double ta = edge_tail(T, ((double)(gt + lane) * T.w - mu) * isg, gc, fa);
                double tz = 0.0;   // the tile's last edge
                if (b1 == 32) tz = edge_tail(T, ((double)(gt + 32) * T.w - mu) * isg, gc, fz);
                double tb = __shfl_down_sync(0xffffffffu, ta, 1);
                bool fb = __shfl_down_sync(0xffffffffu, (int)fa, 1) != 0;
                if (lane == 31) {
                    tb = tz;
                    fb = fz;
                }
                const double v = lane >= b0 && lane < b1 ? tb - ta + ((!fa && fb) ? 1.0 : 0.0) : 0.0;
                sc[lane][j] = v;
                if (COLS) {
#pragma unroll
                    for (int e = 0; e < ES; ++e)
                        if (e < NES) {
                            const double r = warp_sum(v * sG[e][lane]);
                            if (lane == j) cs[e] = r;
                        }
                }
            }
            __syncwarp();
        }
        if (c == G64_CI && __any_sync(0xffffffffu, go)) {   // kind P
            double C[NPOLY];
            poly_coef(h, C);
            for (int r0 = 0; r0 < 32; r0 += RUN64) {
                double z = (y0 + (double)r0 * d - gen.x) * gen.y;
                double p = exp_tab(-0.5 * z * z, sE), rho = exp_tab(-(z + 0.5 * h) * h, sE);
#pragma unroll 4
                for (int k = r0; k < r0 + RUN64; ++k) {
                    const bool use = go && k >= a0 && k < a1;
                    if (!anyD || go) put(k, use ? p * poly_eval(C, z * z) : 0.0);
                    p *= rho;
                    rho = fma(-rho, gen.z, rho);
                    z += h;
                }
            }
        } else if (c != G64_CI) {
#pragma unroll
            for (int r0 = 0; r0 < 32; r0 += RUN64) {
                if (!__any_sync(0xffffffffu, a0 < r0 + RUN64 && a1 > r0)) {
#pragma unroll
                    for (int k = r0; k < r0 + RUN64; ++k) sc[k][lane] = 0.0;
                    continue;
                }
                double z = (y0 + (double)r0 * d - gen.x) * gen.y;
                double p = exp_tab(-0.5 * z * z, sE), rho = exp_tab(-(z + 0.5 * h) * h, sE);
#pragma unroll
                for (int k = r0; k < r0 + RUN64; ++k) {
                    const double v = GC ? p * gc_density_factor(T, z) : p;
                    put(k, k >= a0 && k < a1 ? v : 0.0);
                    p *= rho;
                    rho = fma(-rho, gen.z, rho);
                    if (GC) z += h;
                }
            }
        }
        if (COLS && on) {
            const int slot = (gt >> 5) - (cp.z >> 5);
            double* ap = w.ap64 + ((size_t)item * w.nslot64 + slot) * w.nes * w.Npad;
#pragma unroll
            for (int e = 0; e < ES; ++e)
                if (e < NES) ap[(size_t)e * w.Npad + ie] = cs[e];
        }
        __syncwarp();
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const double v = sc[lane][j];
            const double2 S = sS[wq][j];
            Fs = fma(v, S.x, Fs);
            if (TAG) Ft = fma(v, S.y, Ft);
        }
        __syncwarp();
    }
    if (NW == 1) {
        double* F = w.F64 + (((size_t)item * 4 + share) * 2) * w.gl64 + tile * 32 + lane;
        F[0] = Fs;
        if (TAG) F[w.gl64] = Ft;
        return;
    }
    __syncthreads();
    sT[wq][0][lane] = Fs;
    sT[wq][1][lane] = Ft;
    __syncthreads();
    if (wq < (TAG ? 2 : 1)) {
        const double s = (sT[0][wq][lane] + sT[1 % NW][wq][lane]) + (sT[2 % NW][wq][lane] + sT[3 % NW][wq][lane]);
        w.F64[((size_t)item * 2 + wq) * w.gl64 + tile * 32 + lane] = s;
    }
}

// Per 32-column chunk (a warp), the chunk's part of every species' marginal sums
// sum_i s_k[i] G_W,q[i] and sum_i s_k[i] dG_W,q/deps, with G_W = (1 - eps) aW + eps a per column.
__device__ void marg_chunk(const Work& w, const Toy& T, int item, int chunk) {
    const int lane = threadIdx.x & 31, ie = chunk * 32 + lane, K = T.K;
    const int grp = T.n_set > 1 ? ie / T.Ncs : 0, i = ie - grp * T.Ncs;
    const bool in = ie < T.Next && i < T.N;
    const double eps = w.theta[(size_t)item * w.tstride + K + 5];
    const size_t at = (size_t)item * w.Npad + ie;
    const int4 cp = in ? w.colc64[at] : make_int4(-1, 0, 0, 0);
    const int ns = cp.x >= 0 ? ((cp.w - 1) >> 5) - (cp.z >> 5) + 1 : 0;
    const double amp = cp.x >= 0 ? w.gen64[at].w : 0.0;
    for (int q = 0; q < T.n_es; ++q) {
        double ag = 0.0;
        for (int s = 0; s < ns; ++s) ag += w.ap64[(((size_t)item * w.nslot64 + s) * w.nes + q) * w.Npad + ie];
        ag *= amp;
        const double aw = in ? w.aW[((size_t)item * w.nes + q) * w.Npad + ie] : 0.0;
        const double GW = (1.0 - eps) * aw + eps * ag, dG = ag - aw;
        double v[32];
#pragma unroll
        for (int k = 0; k < KMAX; ++k) {
            double x = 0.0;
            if (k < K && in) {
                const double wk = T.n_set > 1 || T.n_shell > 0 ? set_weight<true>(T, k, grp) : 1.0;
                x = wk == 0.0 ? 0.0 : wk * T.shapes[(size_t)k * T.N + i];
            }
            v[k] = x * GW;
            v[KMAX + k] = x * dG;
        }
        const double r = warp_sum32(v);
        w.mc64[(((size_t)item * (w.Npad / 32) + chunk) * w.nes + q) * 32 + lane] = r;
    }
}

// Rows of bits per bin of one spectrum's axis (k_lam64 writes both).
enum { ROWS_TAIL = 0, ROWS_EXACT = 1, ROWS_N = 2 };
__device__ __forceinline__ unsigned* bin_rows(const Work& w, int item, int h, int which) {
    return w.rows64 + (((size_t)item * 2 + h) * ROWS_N + which) * (w.Mpad / 32);
}
__device__ __forceinline__ bool row_bit(const unsigned* r, int m) { return (r[m >> 5] >> (m & 31)) & 1u; }
// A bin in the tails of everything near it: below 2^-TAIL_BITS of the largest sample that its stencils
// meet (top: that sample's exponent word).  That is from 3.1 to 3.9 sigma past the last column, for
// spacings of 0.2 to 0.1 sigma.  Nearer, the columns that end before the bin (9 sigma) are below 4e-15 of
// it and the stencil is good to 2e-16; at 6 sigma these are 1e-10 and 9e-14 (a dense spectrum).
constexpr int TAIL_BITS = 7;
__device__ __forceinline__ bool in_tail(double v, int top) {
    const int e = __double2hiint(v);
    return e <= top - (TAIL_BITS << 20) || e < (40 << 20);
}

// lambda_h[m]: the stencil of bin m's phase over each class's samples around its cell, plus CI.  A
// bin no column's samples reach (every class's own cell empty) and a tile that no column's band touches
// are exactly 0; the bins in the tails are marked for k_pile64 (the bins of such a tile too).  The
// first nrb CTAs of an item do that; the others take the marginal sums of four chunks each.
// nplane: the forward's partial planes (small batches), added in the order of its four warps.
template <bool TAG>
__global__ void __launch_bounds__(128) k_lam64(Work w, int nrb, int nall, int nplane) {
    const int item = blockIdx.x / nall, blk = blockIdx.x % nall, m = blk * 128 + threadIdx.x;
    if (w.status[item]) return;
    const Toy& T = w.toys[w.toy_of[item]];
    if (blk >= nrb) {
        const int chunk = (blk - nrb) * 4 + (threadIdx.x >> 5);
        if ((T.n_rad > 0 || T.n_psd > 0) && chunk * 32 < T.Next) marg_chunk(w, T, item, chunk);
        return;
    }
    const int M = T.M, present = w.cmask64[item];
    const bool touched = w.band != BAND_S || ((w.tmask64[item] >> blk) & 1ull);   // (128 bins: one tile)
    if (blk * 128 >= M) return;
    // the samples of a class that the CTA's 128 bins meet, the planes added, in shared memory
    const size_t ps = (size_t)w.gl64 * 2;   // between planes
    const double* F = w.F64 + (size_t)item * nplane * ps;
    constexpr int H = TAG ? 2 : 1;
    __shared__ double sF[H][128 + 2 * R64];
    __shared__ __align__(16) int s_top[H][4];
    // stages class c's samples for the bins: sample g + R64 of the staged ones is a bin's own
    // (top: the largest of them, by exponent word per bin width)
    auto stage = [&](int c, int off, int (&top)[H]) {
        int t[H] = {};
        const bool ci = c == G64_CI;
        const int g0 = ci ? blk * 128 - R64 : (blk * 128) >> c, ng = (ci ? 127 : 127 >> c) + 1 + 2 * R64;
        const int len = g64_len(M, c);
        __syncthreads();
        for (int q = threadIdx.x; q < H * ng; q += 128) {
            const int hh = q / ng, g = q - hh * ng;
            double v = 0.0;
            if (g0 + g >= 0 && g0 + g < len) {
                const double* f = F + (size_t)hh * w.gl64 + off + g0 + g;
                v = nplane == 1 ? f[0] : (f[0] + f[ps]) + (f[2 * ps] + f[3 * ps]);
            }
            sF[hh][g] = v;
#pragma unroll
            for (int h = 0; h < H; ++h)
                if (h == hh) t[h] = max(t[h], __double2hiint(v) & 0x7fffffff);
        }
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int r = __reduce_max_sync(0xffffffffu, t[h]);
            if ((threadIdx.x & 31) == 0) s_top[h][threadIdx.x >> 5] = r;
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int r = max(max(s_top[h][0], s_top[h][1]), max(s_top[h][2], s_top[h][3]));
            top[h] = max(top[h], r - (ci ? 0 : c << 20));
        }
        return ci ? (int)threadIdx.x : (m >> c) - g0;
    };
    double lam[H];
    bool any[H];
    int top[H];   // exponent word of the largest sample staged, per bin width
#pragma unroll
    for (int h = 0; h < H; ++h) {
        lam[h] = 0.0;
        any[h] = false;
        top[h] = 0;
    }
    int off = 0;
    for (int c = 0; c <= G64_NC; ++c) {
        if ((present >> c) & 1) {
            const int g = stage(c, off, top);
            if (m < M) {
                double a[H];
#pragma unroll
                for (int h = 0; h < H; ++h) a[h] = c == G64_CI ? sF[h][g + R64] : 0.0;
                if (c != G64_CI) {
                    const double* st = g64_stencil(w, c, m & ((1 << c) - 1));
#pragma unroll 11
                    for (int j = 0; j < TAPS; ++j)
#pragma unroll
                        for (int h = 0; h < H; ++h) a[h] = fma(st[j], sF[h][g + j], a[h]);
                }
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    lam[h] += a[h];
                    any[h] |= sF[h][g + R64] != 0.0;
                }
            }
        }
        off += g64_len(M, c);
    }
    if (w.band != BAND_S) {
        for (int h = 0; h < H; ++h)
            if (m < M) w.lam[((size_t)item * 2 + h) * w.Mpad + m] = any[h] ? lam[h] : 0.0;
        return;
    }
    bool tail = false;
#pragma unroll
    for (int h = 0; h < H; ++h) {
        lam[h] = m < M && any[h] && touched ? lam[h] : 0.0;
        if (m < M) w.lam[((size_t)item * 2 + h) * w.Mpad + m] = lam[h];
        if (threadIdx.x == 0) w.top64[((size_t)item * 2 + h) * MAX_TILES + blk] = top[h];
        tail |= m < M && in_tail(lam[h], top[h]);
    }
    // the largest of all samples staged bounds each bin's; only where that leaves a doubt, its own
    const bool doubt = __syncthreads_or(tail);
    if (doubt) {
#pragma unroll
        for (int h = 0; h < H; ++h) top[h] = 0;
        off = 0;
        for (int c = 0; c <= G64_NC; ++c) {
            if ((present >> c) & 1) {
                int all[H] = {};
                const int g = stage(c, off, all);
                for (int j = 0; m < M && j < TAPS; ++j)
#pragma unroll
                    for (int h = 0; h < H; ++h)
                        top[h] = max(top[h], (__double2hiint(sF[h][g + j]) & 0x7fffffff) - (c == G64_CI ? 0 : c << 20));
            }
            off += g64_len(M, c);
        }
    }
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const unsigned bt = __ballot_sync(0xffffffffu, doubt && m < M && in_tail(lam[h], top[h]));
        if ((threadIdx.x & 31) == 0) {
            bin_rows(w, item, h, ROWS_TAIL)[m >> 5] = bt;
            bin_rows(w, item, h, ROWS_EXACT)[m >> 5] = 0u;
        }
    }
}

// ------------------------------------------------------------------ bins in the tails

// Whether some column of the chunk, this column, touches the tile with its band.
__device__ __forceinline__ bool chunk_touches(const Work& w, int item, int chunk, int tile) {
    const uint2 t = w.ctile64[(size_t)item * (w.Npad / 32) + chunk];
    return ((tile < 32 ? t.x >> tile : t.y >> (tile - 32)) & 1u) != 0u;
}
__device__ __forceinline__ bool column_touches(const Work& w, const Toy& T, int item, int ie, int tile) {
    const size_t at = (size_t)item * w.Npad + ie;
    if (w.colc64[at].x < 0) return false;
    const Col64 cc = w.col64[at];
    int r0, r1;
    near_bins(cc.mu, cc.sig, T.w, T.M, (float)w.band, r0, r1);
    return r0 < r1 && tile >= r0 / TM && tile <= (r1 - 1) / TM;
}

// lambda_h[m] summed over the columns that touch the bin's tile, each bin mass the difference of erfc tails; by
// the whole block (128 threads).  A first pass over the columns finds the largest term to a few bits (the
// exponents and z^2 in FP32), the second evaluates those within 2^-70 of it: FP64 erfc costs about 100
// operations, and a few hundred of the columns matter.
__device__ double exact_bin(const Work& w, const Toy& T, int item, int h, int m, double* red) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const size_t cb = (size_t)item * w.Npad;
    const bool gc = T.gc1 != 0.0 || T.gc2 != 0.0;
    const double ya = (double)m * T.w, yb = (double)(m + 1) * T.w;
    float top = -3.0e38f;
    double sum = 0.0;
    for (int pass = 0; pass < 2; ++pass) {
        for (int ch = wid; ch * 32 < T.Next; ch += 4) {
            if (!chunk_touches(w, item, ch, m / TM)) continue;
            const int ie = ch * 32 + lane;
            const double2 S2 = w.colS[cb + ie];
            const double S = h ? S2.y : S2.x;
            if (S != 0.0 && column_touches(w, T, item, ie, m / TM)) {
                const Gen64 gen = w.gen64[cb + ie];
                const double za = (ya - gen.x) * gen.y, zb = (yb - gen.x) * gen.y;
                const float z = (float)(za > 0.0 ? za : zb < 0.0 ? zb : 0.0);
                const float e = (float)((__double2hiint(S) >> 20) & 0x7ff) - 0.72134752f * z * z;
                if (pass == 0) {
                    top = fmaxf(top, e);
                } else if (e >= top - 70.0f) {
                    bool fa, fb;
                    const double ta = edge_tail(T, za, gc, fa), tb = edge_tail(T, zb, gc, fb);
                    const double D = tb - ta + ((!fa && fb) ? 1.0 : 0.0);
                    sum = fma(S * (w.col64[cb + ie].norm / gen.w), D, sum);
                }
            }
        }
        __syncthreads();   // (red: the bin before)
        if (pass == 0) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
            if (lane == 0) red[wid] = top;
            __syncthreads();
            top = (float)fmax(fmax(red[0], red[1]), fmax(red[2], red[3]));
        } else {
            sum = warp_sum(sum);
            if (lane == 0) red[wid] = sum;
            __syncthreads();
            sum = (red[0] + red[1]) + (red[2] + red[3]);
        }
    }
    return sum;
}

// log2 of a positive normal number, to FP32's precision (its range may exceed FP32's).
__device__ __forceinline__ float log2_f64(double x) {
    const int hi = __double2hiint(x);
    return (float)((hi >> 20) - 1023) + log2f((float)__hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(x)));
}

// How far the stencil's lambda may be off in 32 bins (lane b: bin m + b, if its bit of on is set; the same in
// each of the block's four warps), over a count whose log2 is lm (l2max: log2 of more than any column's
// largest bin).  Summed over the columns in FP32: whole, a column whose samples end before the bin (9 sigma)
// or that does not touch its tile (its samples go one sigma past its band); of any column the stencil's 1e-17
// of the density 2.3 sigma nearer; and, where the stencil reaches past the end of the samples, 0.04 of the
// density there, 2^-4 less per sigma (bounds of the errors in 40 digits at spacings of 0.1 to 0.2 sigma,
// from 3 sigma on).  A lane holds a column and the bins are gone through, as data have one or two in 32: the
// assembly of 100 toys takes 164 us with it, 171 with a lane per bin and columns from 5.7 sigma on passed over
// up to 1e-11 of the count.  Terms below 2^-60 of the count are passed over; 2000 columns take a few us, an
// exact bin mass of every column that matters 12 us a bin.
__device__ float tail_error(const Work& w, const Toy& T, int item, int h, unsigned on, int m, float lm, float l2max) {
    __shared__ float s_err[4][32];
    const int tid = threadIdx.x, lane = tid & 31, part = tid >> 5;
    const float wf = (float)T.w;
    const float ylo = ((float)(m + __ffs(on)) - 0.5f) * wf, yhi = ((float)(m + 31 - __clz(on)) + 0.5f) * wf;
    float lmin = (on >> lane) & 1u ? lm : 3.0e38f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lmin = fminf(lmin, __shfl_xor_sync(0xffffffffu, lmin, o));
    auto score = [&](float gap, float isig) { return fmaxf((gap - 0.5f * wf) * isig, 0.f); };
    // the warp's groups of 32 columns with one near enough (loads of several groups in flight)
    static_assert(MAX_CB * BCOLS <= 64 * 128, "a bit per group of 128 columns");
    unsigned long long todo = 0ull;
    const Gen64* gen64 = w.gen64 + (size_t)item * w.Npad;
    const int ng = (T.Next + 127 - 32 * part) / 128;
#pragma unroll 8
    for (int g = 0; g < ng; ++g) {
        const int ie = min(g * 128 + part * 32 + lane, T.Next - 1);
        const double2 ms = *reinterpret_cast<const double2*>(gen64 + ie);   // mean, 1 / sigma
        const float z = score(fmaxf(fmaxf(ylo - (float)ms.x, (float)ms.x - yhi), 0.f), (float)ms.y);
        const float zn = fmaxf(z - 2.3f, 0.f), zw = fmaxf(z, 7.95f);
        const float e = -0.72134752f * fminf(fmaf(zn, zn, 78.3f), zw * zw);
        if (__any_sync(0xffffffffu, l2max - lmin + e > -60.f)) todo |= 1ull << g;
    }
    float err = 0.f;
    for (; todo; todo &= todo - 1ull) {
        const int ie = (__ffsll((long long)todo) - 1) * 128 + part * 32 + lane;
        float mu = 0.f, isig = 0.f, l2 = -3.0e38f;   // l2: log2 of the bin mass at the mean
        int t0 = 0, t1 = 0;                          // first and last tile that the column touches
        if (ie < T.Next) {
            const size_t at = (size_t)item * w.Npad + ie;
            const double2 S2 = w.colS[at];
            const Gen64 gen = gen64[ie];
            const Col64 cc = w.col64[at];
            const double S = fabs(h ? S2.y : S2.x);
            mu = (float)gen.x;
            isig = (float)gen.y;
            if (w.colc64[at].x >= 0 && S > 0.0)
                l2 = log2_f64(S) + log2f((float)cc.norm / (float)gen.w * isig * wf * 0.39894228f);
            int r0, r1;
            near_bins(cc.mu, cc.sig, T.w, T.M, (float)w.band, r0, r1);
            t0 = r0 / TM;
            t1 = (r1 - 1) / TM;
        }
        for (unsigned r = on; r; r &= r - 1u) {
            const int b = __ffs(r) - 1, tile = (m + b) / TM;
            const float top = l2 - __shfl_sync(0xffffffffu, lm, b);
            const float z = score(fabsf(((float)(m + b) + 0.5f) * wf - mu), isig), zn = fmaxf(z - 2.3f, 0.f);
            float e = exp2f(fmaf(-0.72134752f * zn, zn, top - 56.4f));   // (1e-17: 2^-56.5)
            if (z > 5.7f)
                e += exp2f(z > 8.9f || tile < t0 || tile > t1 ? fmaf(-0.72134752f * z, z, top) : fmaf(4.f, z, top - 99.1f));
            if (__any_sync(0xffffffffu, e > 8.7e-19f)) {
                e = warp_sum(e);
                if (lane == b) err += e;
            }
        }
    }
    __syncthreads();
    s_err[part][lane] = err;
    __syncthreads();
    return (s_err[0][lane] + s_err[1][lane]) + (s_err[2][lane] + s_err[3][lane]);
}

// Data in the tails: the lambdas (in sx) that those bins' expected counts (mu, from the stencils' values)
// need better are replaced by exact_bin's and marked for the adjoint; whether there were any.  No lambda
// of the reach is further off than 1.7e-17 of the largest density within 10 sigma of it (a column at the
// end of its samples; what columns have in a tile next to those they touch counts against a bin's own lambda
// only).  A bin for which that is below 1e-12 needs nothing; if it is for the tails in its
// reach (nearly every bin with pile-up from the columns themselves), at most its own lambda; the reach of
// any other bin is looked through.
__device__ __noinline__ bool tail_bins(const Work& w, const Toy& T, int item, int h, unsigned ev, int m0, int Lt,
                                       double eps, const double* sg, double* sx, const double* mu, int want_mu) {
    __shared__ unsigned s_need[(MAX_L + 32) / 32 + 1];
    __shared__ double s_red[4];
    const int tid = threadIdx.x, lane = tid & 31, nrow = 32 + Lt - 1;
    const unsigned* tail = bin_rows(w, item, h, ROWS_TAIL);
    const unsigned long long touched = w.tmask64[item];   // (lambda is exactly 0 in the other tiles)
    double gs = 0.0;
    for (int d = tid; d < Lt; d += 128) gs += fabs(sg[d]);
    gs = warp_sum(gs);
    if (lane == 0) s_red[tid >> 5] = gs;
    for (int q = tid; q <= nrow / 32; q += 128) s_need[q] = 0u;
    int top = 0;   // class c: sigma below 10 2^c bins (the last class: any)
    {
        const int cm = w.cmask64[item] & ((1 << G64_NC) - 1), c = 31 - __clz(cm | 1);
        const int R = c == G64_NC - 1 ? T.M : 100 << c;
        int first = INT_MAX;   // tail of the reach, in whole words of 32 bins
        for (int q = max(m0 - (Lt - 1), 0) / 32 + lane; q * 32 < min(m0 + 32, T.M); q += 32)
            if (tail[q] && ((touched >> (q * 32 / TM)) & 1ull)) first = min(first, q * 32);
        first = __reduce_min_sync(0xffffffffu, first);
        const int t0 = max(min(first, m0) - R, 0) / TM, t1 = min(m0 + 32 + R, T.M - 1) / TM;
        for (int t = t0 + lane; t <= t1; t += 32) top = max(top, w.top64[((size_t)item * 2 + h) * MAX_TILES + t]);
        top = __reduce_max_sync(0xffffffffu, top);
    }
    __syncthreads();
    gs = (s_red[0] + s_red[1]) + (s_red[2] + s_red[3]);
    // (the Gram-Charlier density at 9 sigma is this much more than the Gaussian's)
    const double gcf = 1.0 + 702.0 * fabs(T.gc1) + 6078.0 * fabs(T.gc2);
    const double bound = 1.7e-5 * gcf * __hiloint2double(top + (1 << 20), 0), reach = bound * fabs(eps) * gs;
    // of a bin's expected count (an event's term takes n times the error; 100 toys' assembly takes 166 us from
    // 2e-13 to 1e-12, 199 at 5e-14, 206 at 1e-14)
    const float tol = (float)((want_mu ? 1e-14 : 2e-13) / gcf);
    // (no count: no error is small enough)
    auto log2_mu = [&](int b) { return mu[b] > 1e-290 ? log2_f64(mu[b]) : -3.0e38f; };
    ev &= ~__ballot_sync(0xffffffffu, mu[lane] >= bound + reach);   // (a bin's own lambda is as good)
    if (!ev) return false;
    int all = 0;   // the largest sample of any tile (and 2^40 of it: a column's mean may lie off the axis)
    for (int t = lane; t * TM < T.M; t += 32) all = max(all, w.top64[((size_t)item * 2 + h) * MAX_TILES + t]);
    const float l2max = (float)((__reduce_max_sync(0xffffffffu, all) >> 20) - 1023) + 40.f;
    const unsigned own = ev & __ballot_sync(0xffffffffu, mu[lane] >= reach && mu[lane] > 1e-290);
    unsigned any = 0u;
    if (own) {
        const float err = tail_error(w, T, item, h, own, m0, log2_mu(lane), l2max);
        any = __ballot_sync(0xffffffffu, ((own >> lane) & 1u) && !(err <= tol));
        if (tid < 32 && ((any >> lane) & 1u)) atomicOr(&s_need[(Lt - 1 + lane) >> 5], 1u << ((Lt - 1 + lane) & 31));
    }
    if (ev & ~own) {
        float lm0 = 3.0e38f;   // the smallest of their counts
        for (unsigned e = ev & ~own; e; e &= e - 1u) lm0 = fminf(lm0, log2_mu(__ffs(e) - 1));
        for (int q0 = 0; q0 < nrow; q0 += 32) {   // the bins of sx, 32 at a time
            const int q = q0 + lane, mq = m0 - (Lt - 1) + q;
            const bool on = q < nrow && mq >= 0 && mq < T.M && ((touched >> (mq / TM)) & 1ull) && row_bit(tail, mq);
            const unsigned rows = __ballot_sync(0xffffffffu, on);   // (of all warps alike)
            if (!rows) continue;
            const float err = tail_error(w, T, item, h, rows, mq - lane, lm0, l2max);
            bool need = false;
            for (unsigned e = ev & ~own; e; e &= e - 1u) {
                const int b = __ffs(e) - 1, d = Lt - 1 + b - q;   // its shift, and its weight in mu
                if (on && d >= 0 && d < Lt) {
                    const double c = fabs(eps * sg[d] + (d == 0 ? 1.0 - eps : 0.0));
                    need |= c > 0.0 && !(err * exp2f(lm0 - log2_mu(b)) * (float)c <= tol);
                }
            }
            const unsigned bits = __ballot_sync(0xffffffffu, need);
            if (tid == 0) s_need[q0 >> 5] |= bits;
            any |= bits;
        }
    }
    __syncthreads();
    if (!any) return false;
    for (int q0 = 0; q0 < nrow; q0 += 32)
        for (unsigned r = s_need[q0 >> 5]; r; r &= r - 1u) {
            const int q = q0 + __ffs(r) - 1, m = m0 - (Lt - 1) + q;
            const double v = exact_bin(w, T, item, h, m, s_red);
            if (tid == 0) {
                sx[q] = v;
                atomicOr(&bin_rows(w, item, h, ROWS_EXACT)[m >> 5], 1u << (m & 31));
                w.xany64[item] = 1;
            }
        }
    __syncthreads();
    return true;
}

// The adjoint of the bins that tail_bins took (their row weights xw64 are not in rowW), for one column:
// sums of the species-summed weights times the bin mass and its derivatives (E[0 .. 2]), and of the
// weights times the mass (E[3], E[4]: vetoed, tagged), as kind D's.
__device__ __noinline__ void tail_adjoint(const Work& w, const Toy& T, int item, int ie, double Ss, double St, double mu,
                                          double isig, double (&E)[5]) {
    const bool gc = T.gc1 != 0.0 || T.gc2 != 0.0;
    for (int h = 0; h < (T.has_tag ? 2 : 1); ++h) {
        const unsigned* rows = bin_rows(w, item, h, ROWS_EXACT);
        const double S = h ? St : Ss;
        for (int b = 0; b * 32 < T.M; ++b)
            for (unsigned r = rows[b]; r; r &= r - 1u) {
                const int m = b * 32 + __ffs(r) - 1;
                if (!column_touches(w, T, item, ie, m / TM)) continue;
                const double W = w.xw64[((size_t)item * 2 + h) * w.Mpad + m];
                const double za = ((double)m * T.w - mu) * isig, zb = ((double)(m + 1) * T.w - mu) * isig;
                bool fa, fb;
                const double ta = edge_tail(T, za, gc, fa), tb = edge_tail(T, zb, gc, fb);
                double pa = INV_SQRT_2PI * exp(-0.5 * za * za), pb = INV_SQRT_2PI * exp(-0.5 * zb * zb);
                if (gc) {
                    pa *= gc_density_factor(T, za);
                    pb *= gc_density_factor(T, zb);
                }
                const double q = W * (tb - ta + ((!fa && fb) ? 1.0 : 0.0));
                E[0] = fma(q, S, E[0]);
                E[1] = fma(-W * (pb - pa), S, E[1]);
                E[2] = fma(-W * (zb * pb - za * pa), S, E[2]);
                E[3 + h] += q;
            }
    }
}

// ------------------------------------------------------------------ assembly

// CTA = 32 window bins of one spectrum of one item, a warp per quarter of the taps: Eq. 2, the
// Baker-Cousins terms, w = 1 - n/mu, and the tile's part of -lnL (compensated) and of d/deps.  With an
// event in the tails the sum is taken again if tail_bins changed a lambda (100 toys: 155 -> 166 us; the
// bound of 10 CTAs keeps the registers at 48, 47 without the tails).
__global__ void __launch_bounds__(128, 10) k_pile64(Work w, int ntw, int nH, int want_grad, int want_mu) {
    extern __shared__ __align__(16) double dsm[];
    const int t = blockIdx.x % ntw, h = (blockIdx.x / ntw) % nH, item = blockIdx.x / (ntw * nH), tid = threadIdx.x;
    double* part = w.part64 + (((size_t)item * nH + h) * ntw + t) * 4;
    const Toy& T = w.toys[w.toy_of[item]];
    const int nw = T.nw, m_lo = T.m_lo, L = T.L, H = T.has_tag ? 2 : 1;
    if (w.status[item] || h >= H || t * 32 >= nw) {
        if (tid < 4) part[tid] = 0.0;
        return;
    }
    const double eps = w.theta[(size_t)item * w.tstride + T.K + 5];
    const int m0 = m_lo + t * 32, Lt = min(L, m0 + 32);   // taps that meet the axis
    double* sg = dsm;         // [Lt]
    double* sx = dsm + Lt;    // [32 + Lt - 1]: lambda from m0 - (Lt - 1)
    const double* lam = w.lam + ((size_t)item * 2 + h) * w.Mpad;
    for (int d = tid; d < Lt; d += 128) sg[d] = T.g[d];
    for (int q = tid; q < 32 + Lt - 1; q += 128) {
        const int m = m0 - (Lt - 1) + q;
        sx[q] = m >= 0 && m < T.M ? lam[m] : 0.0;
    }
    const int b = tid & 31, pt = tid >> 5, j = t * 32 + b, pl = (Lt + 3) / 4;
    unsigned ev = 0u;   // bins in the tails whose counts matter relative to themselves
    if (w.band == BAND_S) {
        bool e = j < nw && row_bit(bin_rows(w, item, h, ROWS_TAIL), m0 + b);
        if (e) e = want_mu || T.cnt[(size_t)h * nw + j] != 0.0;
        ev = __ballot_sync(0xffffffffu, e);
    }
    __shared__ double sc[4][32];
    __syncthreads();
    const int d0 = min(Lt, pt * pl), d1 = min(Lt, d0 + pl);
    const double* x = sx + (Lt - 1) + b;
    double cv = 0.0;
    for (;;) {
        double c0 = 0.0, c1 = 0.0;
        int d = d0;
#pragma unroll 4
        for (; d + 1 < d1; d += 2) {
            c0 = fma(sg[d], x[-d], c0);
            c1 = fma(sg[d + 1], x[-d - 1], c1);
        }
        if (d < d1) c0 = fma(sg[d], x[-d], c0);
        if (pt) sc[pt - 1][b] = c0 + c1;
        __syncthreads();
        if (pt == 0) cv = ((c0 + c1) + sc[0][b]) + (sc[1][b] + sc[2][b]);
        if (!ev) break;
        if (pt == 0) sc[3][b] = (1.0 - eps) * x[0] + eps * cv;
        __syncthreads();
        if (!tail_bins(w, T, item, h, ev, m0, Lt, eps, sg, sx, sc[3], want_mu)) break;
        ev = 0u;   // once more with the better values
    }
    if (pt) return;
    bool dom = false;
    Neu acc{0.0, 0.0};
    double geps = 0.0;
    if (j < nw) {
        const double lm = x[0], mu = (1.0 - eps) * lm + eps * cv;
        const double n = T.cnt[(size_t)h * nw + j];
        double term, wb = 1.0;
        if (n == 0.0) term = mu;
        else if (!(mu > 0.0 && isfinite(mu))) { dom = true; term = 0.0; }
        else {
            term = (mu - n) + n * log1p((n - mu) / mu);
            wb = 1.0 - n / mu;
        }
        neu_add(acc, term);
        if (want_mu) w.mu[(size_t)item * w.nbmax + (size_t)h * nw + j] = mu;
        if (want_grad) {
            w.wv64[((size_t)item * 2 + h) * w.Mpad + j] = wb;
            geps = wb * (cv - lm);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Neu other{__shfl_xor_sync(0xffffffffu, acc.s, o), __shfl_xor_sync(0xffffffffu, acc.c, o)};
        acc = neu_merge(acc, other);
        geps += __shfl_xor_sync(0xffffffffu, geps, o);
    }
    dom = __any_sync(0xffffffffu, dom);
    if (tid == 0) {
        part[0] = acc.s;
        part[1] = acc.c;
        part[2] = geps;
        part[3] = dom ? 1.0 : 0.0;
    }
}

// Radial bin probabilities (closed-form shell integrals; internal: uniform in volume), as the
// mixed-precision assembly's.  By the whole block (one barrier inside).
__device__ void radial_probs64(const Toy& T, double s_r, double* sF, double* sdF, double* pint, double* pext,
                               double* dpext) {
    const int nrad = T.n_rad;
    const double lamA = T.att_len * s_r;
    for (int e = threadIdx.x; e <= nrad + 1; e += blockDim.x) {
        const double r = e < nrad ? T.r_fid * e / nrad : (e == nrad ? T.r_fid : 0.0);
        shell_F(r, T.r_iv, lamA, sF[e], sdF[e]);
    }
    __syncthreads();
    const double tot = sF[nrad] - sF[nrad + 1], dtot = sdF[nrad] - sdF[nrad + 1];
    for (int b = threadIdx.x; b < nrad; b += blockDim.x) {
        const double ra = T.r_fid * b / nrad, rb = T.r_fid * (b + 1) / nrad;
        pint[b] = (rb * rb * rb - ra * ra * ra) / (T.r_fid * T.r_fid * T.r_fid);
        const double p = (sF[b + 1] - sF[b]) / tot;
        pext[b] = p;
        dpext[b] = ((sdF[b + 1] - sdF[b]) / tot - p * dtot / tot) * T.att_len;
    }
}

// Per item: the Eq. 4 marginals A_k^(q) = r_k c_k sum_i s_k[i] ((1 - eps) aW[i] + eps a[i]) from the
// chunk sums of k_lam64, their -lnL terms, the item's -lnL, and the adjoint's coefficients.
constexpr int MG = 256;
__global__ void __launch_bounds__(MG) k_marg64(Work w, int ntw, int nH, int want_grad, int want_mu) {
    const int item = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const Toy& T = w.toys[w.toy_of[item]];
    const int K = T.K, nw = T.nw, nrad = T.n_rad, npsd = T.n_psd, NES = T.n_es, H = T.has_tag ? 2 : 1;
    const int nradS = NES * nrad, npsdS = NES * npsd;
    double* gmid = w.gmid + (size_t)item * PMAX;
    if (w.status[item]) {
        if (tid == 0) w.nll[item] = INFINITY;
        if (tid < PMAX) gmid[tid] = 0.0;
        return;
    }
    const double* th = w.theta + (size_t)item * w.tstride;
    const double s_r = th[K + 6];
    __shared__ double s_rs[KMAX], s_rt[KMAX], s_SA[MAX_ES][2 * KMAX], s_beta[MAX_ES][KMAX], s_aint[MAX_ES], s_aext[MAX_ES];
    __shared__ double s_pint[MAX_RAD], s_pext[MAX_RAD], s_dpext[MAX_RAD], s_F[MAX_RAD + 2], s_dF[MAX_RAD + 2];
    __shared__ double s_w[MAX_RAD + MAX_PSD];      // 1 - n/mu of the marginal bins
    __shared__ double red[MG / 32][2], sP[MG / 32][32];
    __shared__ int s_dom;
    const bool mv = nrad > 0 || npsd > 0;
    if (tid == 0) s_dom = 0;
    if (tid < K) {
        const double r = th[tid], t = T.tag ? T.tag[tid] : 0.0;
        s_rs[tid] = r * (T.tag ? 1.0 - t : 1.0);
        s_rt[tid] = r * t;
    }
    if (mv) {   // 32 sums per slice over the chunks: a warp per part of the chunks, then the parts in order
        const int nch = (T.Next + 31) / 32, nchp = w.Npad / 32;
        for (int q = 0; q < NES; ++q) {
            const double* mc = w.mc64 + ((size_t)item * nchp * w.nes + q) * 32 + lane;
            double s = 0.0;
#pragma unroll 4
            for (int ch = wid; ch < nch; ch += MG / 32) s += mc[(size_t)ch * w.nes * 32];
            sP[wid][lane] = s;
            __syncthreads();
            if (tid < 32) {
                double r = 0.0;
                for (int p = 0; p < MG / 32; ++p) r += sP[p][tid];
                s_SA[q][tid] = r;
            }
            __syncthreads();
        }
    }
    if (nrad > 0) radial_probs64(T, s_r, s_F, s_dF, s_pint, s_pext, s_dpext);
    __syncthreads();
    if (mv && tid < NES) {
        double aint = 0.0, aext = 0.0;
        for (int k = 0; k < K; ++k) {
            const double A = s_rs[k] * s_SA[tid][k];
            if (nrad > 0 && T.rad_class[k] == BX_RAD_EXTERNAL) aext += A; else aint += A;
        }
        s_aint[tid] = aint;
        s_aext[tid] = aext;
    }
    __syncthreads();
    Neu acc{0.0, 0.0};
    for (int b = tid; b < nradS + npsdS; b += MG) {
        double mu = 0.0;
        if (b < nradS) {
            const int q = b / nrad, r = b - q * nrad;
            mu = s_aint[q] * s_pint[r] + s_aext[q] * s_pext[r];
        } else {
            const int j = b - nradS, q = j / npsd, r = j - q * npsd;
            for (int k = 0; k < K; ++k) mu += s_rs[k] * s_SA[q][k] * T.psd[(size_t)k * npsd + r];
        }
        const double n = T.cnt[(size_t)H * nw + b];
        double term, wb = 1.0;
        if (n == 0.0) term = mu;
        else if (!(mu > 0.0 && isfinite(mu))) { s_dom = 1; term = 0.0; }
        else {
            term = (mu - n) + n * log1p((n - mu) / mu);
            wb = 1.0 - n / mu;
        }
        neu_add(acc, term);
        s_w[b] = wb;
        if (want_mu) w.mu[(size_t)item * w.nbmax + (size_t)H * nw + b] = mu;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Neu other{__shfl_xor_sync(0xffffffffu, acc.s, o), __shfl_xor_sync(0xffffffffu, acc.c, o)};
        acc = neu_merge(acc, other);
    }
    if (lane == 0) { red[wid][0] = acc.s; red[wid][1] = acc.c; }
    __syncthreads();
    __shared__ double s_ge;
    if (wid == 0) {   // the window's tiles, then the marginals
        const double* part = w.part64 + (size_t)item * nH * ntw * 4;
        Neu tot{0.0, 0.0};
        double ge = 0.0, dom = 0.0;
        for (int q = lane; q < nH * ntw; q += 32) {
            tot = neu_merge(tot, Neu{part[q * 4], part[q * 4 + 1]});
            ge += part[q * 4 + 2];
            dom += part[q * 4 + 3];
        }
        if (lane < MG / 32) tot = neu_merge(tot, Neu{red[lane][0], red[lane][1]});
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            Neu other{__shfl_xor_sync(0xffffffffu, tot.s, o), __shfl_xor_sync(0xffffffffu, tot.c, o)};
            tot = neu_merge(tot, other);
            ge += __shfl_xor_sync(0xffffffffu, ge, o);
            dom += __shfl_xor_sync(0xffffffffu, dom, o);
        }
        if (lane == 0) {
            if (dom != 0.0) s_dom = 1;
            w.nll[item] = s_dom ? INFINITY : tot.s + tot.c;
            if (s_dom) w.status[item] = BX_EDOMAIN;
            s_ge = ge;
        }
    }
    __syncthreads();
    if (!want_grad || s_dom) {
        if (tid < PMAX) gmid[tid] = 0.0;
        return;
    }
    // beta_q,k = dNLL/dA_k^(q)
    if (mv)
        for (int qk = wid; qk < NES * K; qk += MG / 32) {
            const int q = qk / K, k = qk - q * K;
            double s = 0.0;
            const bool ext = nrad > 0 && T.rad_class[k] == BX_RAD_EXTERNAL;
            for (int b = lane; b < nrad; b += 32) s += s_w[q * nrad + b] * (ext ? s_pext[b] : s_pint[b]);
            for (int j = lane; j < npsd; j += 32) s += s_w[nradS + q * npsd + j] * T.psd[(size_t)k * npsd + j];
            s = warp_sum(s);
            if (lane == 0) s_beta[q][k] = s;
        }
    __syncthreads();
    double* coef = w.coef + (size_t)item * (2 + w.nes) * KMAX;
    if (tid < KMAX) {
        const int k = tid;
        double gk = 0.0;
        if (k < K) {
            const double csub = T.tag ? 1.0 - T.tag[k] : 1.0;
            for (int q = 0; mv && q < NES; ++q) gk += s_beta[q][k] * csub * s_SA[q][k];
            gmid[k] = gk;
        }
        coef[k] = k < K ? s_rs[k] : 0.0;
        coef[KMAX + k] = k < K ? s_rt[k] : 0.0;
    }
    for (int j = tid; j < w.nes * KMAX; j += MG) {
        const int q = j / KMAX, k = j - q * KMAX;
        coef[(size_t)(2 + q) * KMAX + k] = mv && q < NES && k < K ? s_beta[q][k] * s_rs[k] : 0.0;
    }
    if (wid == 0) {
        double ge = 0.0, gs = 0.0;
        for (int qk = lane; mv && qk < NES * K; qk += 32) {
            const int q = qk / K, k = qk - q * K;
            ge += s_beta[q][k] * s_rs[k] * s_SA[q][KMAX + k];
        }
        for (int b = lane; b < nradS; b += 32) {
            const int q = b / nrad;
            gs += s_w[b] * s_aext[q] * s_dpext[b - q * nrad];
        }
        ge = warp_sum(ge);
        gs = warp_sum(gs);
        if (lane == 0) {
            for (int j = K; j < K + 5; ++j) gmid[j] = 0.0;
            gmid[K + 5] = s_ge + ge;
            gmid[K + 6] = gs;
            for (int j = K + 7; j < PMAX; ++j) gmid[j] = 0.0;
        }
    }
}

// Adjoint of Eq. 2, CTA = 32 axis bins of one spectrum, a warp per quarter of the taps:
// wt_h[m] = (1 - eps) w_h[m] + eps sum_d g[d] w_h[m + d]; the CTAs of spectrum 0 also write G_W of
// every energy slice.
__global__ void __launch_bounds__(128) k_corr64(Work w, int ntm, int nH) {
    extern __shared__ __align__(16) double dsm[];
    const int t = blockIdx.x % ntm, h = (blockIdx.x / ntm) % nH, item = blockIdx.x / (ntm * nH), tid = threadIdx.x;
    const Toy& T = w.toys[w.toy_of[item]];
    const int nw = T.nw, m_lo = T.m_lo, L = T.L, H = T.has_tag ? 2 : 1, M = T.M, NES = T.n_es;
    if (w.status[item] || t * 32 >= M) return;
    const double eps = w.theta[(size_t)item * w.tstride + T.K + 5];
    double* rowW = static_cast<double*>(w.rowW) + (size_t)item * (2 + w.nes) * w.Mpad;
    const int b = tid & 31, pt = tid >> 5, m = t * 32 + b;
    if (h == 0) {   // G_W,q[m] (0 beyond the toy's slices), and a missing tagged spectrum
        const bool mv = T.n_rad > 0 || T.n_psd > 0;
        for (int q = pt; q < w.nes && m < M; q += 4) {
            const double inW = q < NES && m >= T.es_lo[q] && m < T.es_hi[q] ? 1.0 : 0.0;
            rowW[(size_t)(2 + q) * w.Mpad + m] = mv && q < NES ? (1.0 - eps) * inW + eps * T.Gg[(size_t)q * M + m] : 0.0;
        }
        if (pt == 1 && H == 1 && m < M) rowW[(size_t)w.Mpad + m] = 0.0;
    }
    if (h >= H) return;
    // taps that meet the window: window bin j0 + b + d of axis bin t * 32 + b
    const int j0 = t * 32 - m_lo, dlo = max(0, -j0 - 31), dhi = max(dlo, min(L, nw - j0)), Lt = dhi - dlo;
    double* sg = dsm;         // [Lt]: g from dlo
    double* sx = dsm + Lt;    // [32 + Lt - 1]: w_h from window bin j0 + dlo
    const double* wv = w.wv64 + ((size_t)item * 2 + h) * w.Mpad;
    for (int d = tid; d < Lt; d += 128) sg[d] = T.g[dlo + d];
    for (int q = tid; q < 32 + Lt - 1; q += 128) {
        const int j = j0 + dlo + q;
        sx[q] = j >= 0 && j < nw ? wv[j] : 0.0;
    }
    __shared__ double sc[3][32];
    __syncthreads();
    const int pl = (Lt + 3) / 4, d0 = min(Lt, pt * pl), d1 = min(Lt, d0 + pl);
    const double* x = sx + b;
    double c0 = 0.0, c1 = 0.0;
    int d = d0;
#pragma unroll 4
    for (; d + 1 < d1; d += 2) {
        c0 = fma(sg[d], x[d], c0);
        c1 = fma(sg[d + 1], x[d + 1], c1);
    }
    if (d < d1) c0 = fma(sg[d], x[d], c0);
    if (pt) sc[pt - 1][b] = c0 + c1;
    __syncthreads();
    if (pt || m >= M) return;
    const double direct = m >= m_lo ? (1.0 - eps) * wv[m - m_lo] : 0.0;
    double val = direct + eps * (((c0 + c1) + sc[0][b]) + (sc[1][b] + sc[2][b]));
    if (w.xany64[item] && row_bit(bin_rows(w, item, h, ROWS_EXACT), m)) {   // tail_adjoint's
        w.xw64[((size_t)item * 2 + h) * w.Mpad + m] = val;
        val = 0.0;
    }
    rowW[(size_t)h * w.Mpad + m] = val;
}

// ------------------------------------------------------------------ adjoint

// Row weights onto the class grids: Wt[r][g] = sum_m stencil(m)[g] W[r][m] over the bins whose
// stencil reaches sample g.  2^lc lanes per sample (lc = min(c, 3)) share the bins of a cell, so that
// a warp's loads of W run along the axis; their sums are added by shuffles.
__device__ __forceinline__ void transpose_stencil(const double* __restrict__ tab, int c, int lc, int gp, int sub, int M,
                                                  int nr, const double* __restrict__ W, size_t ws, double* out, size_t os,
                                                  bool on) {
    // class sample gp (grid index): g = gp - R64; cells G with |G - g| <= R64, bins m = (G << c) + ph
    double s[2 + MAX_ES] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    const int G0 = max(0, gp - 2 * R64), G1 = on ? min((M - 1) >> c, gp) : -1;
    const double* st0 = tab + ((1 << c) - 1) * TAPS + gp;
    for (int ph = sub; ph < (1 << c); ph += 1 << lc) {
        const double* st = st0 + ph * TAPS;
#pragma unroll 4
        for (int G = G0; G <= G1; ++G) {
            const int m = (G << c) + ph;
            if (m < M) {
                const double a = st[-G];   // tap (g - G) + R64
#pragma unroll
                for (int r = 0; r < 2 + MAX_ES; ++r)
                    if (r < nr) s[r] = fma(a, W[r * ws + m], s[r]);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < 2 + MAX_ES; ++r) {
        if (r >= nr) break;
        for (int o = 1; o < (1 << lc); o <<= 1) s[r] += __shfl_xor_sync(0xffffffffu, s[r], o);
        if (on && sub == 0) out[r * os] = s[r];
    }
}

// Thread s of the list of (class, sample, lane share): a warp lies within one class (each class has
// a multiple of 32 samples).
__device__ __forceinline__ bool wt64_unit(int s, int M, int& c, int& gp, int& sub, int& off) {
    off = 0;
    for (c = 0; c < G64_NC; ++c) {
        const int len = g64_len(M, c), lc = min(c, 3);
        if (s < len << lc) {
            gp = s >> lc;
            sub = s & ((1 << lc) - 1);
            return true;
        }
        s -= len << lc;
        off += len;
    }
    return false;
}
static int wt64_threads(int M) {
    int n = 0;
    for (int c = 0; c < G64_NC; ++c) n += g64_len(M, c) << (c < 3 ? c : 3);
    return n;
}

__global__ void __launch_bounds__(128) k_wt64(Work w, int nblk) {
    const int item = blockIdx.x / nblk;
    if (w.status[item]) return;
    const Toy& T = w.toys[w.toy_of[item]];
    int c, gp, sub, off;
    if (!wt64_unit((blockIdx.x % nblk) * 128 + threadIdx.x, T.M, c, gp, sub, off) || !((w.cmask64[item] >> c) & 1)) return;
    transpose_stencil(w.tab64, c, min(c, 3), gp, sub, T.M, 2 + T.n_es,
                      static_cast<const double*>(w.rowW) + (size_t)item * (2 + w.nes) * w.Mpad, w.Mpad,
                      w.wt64 + (size_t)item * (2 + w.nes) * w.gl64 + off + gp, w.gl64, true);
}

// Model set-up: Gt_q[g] of one toy, [n_es][g64_total(M)] (CI: Gg itself).
__global__ void __launch_bounds__(128) k_setup_gt64(Toy t, const double* tab, double* Gt) {
    const int GL = g64_off(t.M, G64_NC + 1), s = blockIdx.x * 128 + threadIdx.x;
    int c, gp, sub, off;
    if (wt64_unit(s, t.M, c, gp, sub, off))
        transpose_stencil(tab, c, min(c, 3), gp, sub, t.M, t.n_es, t.Gg, t.M, Gt + off + gp, GL, true);
    const int oc = g64_off(t.M, G64_CI);
    if (s < GL - oc)
        for (int q = 0; q < t.n_es; ++q) Gt[(size_t)q * GL + oc + s] = s < t.M ? t.Gg[(size_t)q * t.M + s] : 0.0;
}
cudaError_t launch_setup_gt64(const Toy& t, const double* tab, double* Gt, cudaStream_t s) {
    k_setup_gt64<<<(wt64_threads(t.M) + 127) / 128, 128, 0, s>>>(t, tab, Gt);
    return cudaGetLastError();
}

// A warp per 32-column chunk.  Thread = column: over its samples the sums of Wt p, Wt z p, Wt z^2 p
// with Wt = sum_r (species sum r) Wt_r, and of Wt_vetoed p, Wt_tagged p for the rates; within a run
// the moments are taken in the sample index.  ~13 FP64 operations an entry.  Then the chain rule
// through mu = LY Q(kB), sigma^2 = a mu + b mu^2 + c and the chunk's partial gradient.
template <bool MULTI, bool GC, int ES>
__global__ void __launch_bounds__(32) k_bwd64(Work w, int nch) {
    const int item = blockIdx.x / nch, chunk = blockIdx.x % nch, lane = threadIdx.x;
    const Toy& T = w.toys[w.toy_of[item]];
    if (chunk * 32 >= T.Next) return;
    double* gp = w.gpart + ((size_t)item * w.gp_rows + chunk) * GPN;
    if (w.status[item]) {
        if (lane < GPN) gp[lane] = 0.0;
        return;
    }
    const int K = T.K, N = T.N, M = T.M, NES = ES > 1 ? T.n_es : 1;
    const int ie = chunk * 32 + lane, grp = MULTI ? ie / T.Ncs : 0, i = ie - grp * T.Ncs;
    const bool in = ie < T.Next && i < N;
    const size_t at = (size_t)item * w.Npad + ie;
    const int4 cp = w.colc64[at];
    __shared__ double sW[2 + ES][32];
    __shared__ double sE[64];
    sE[lane] = w.tab64[EXP_OFF + lane];
    sE[lane + 32] = w.tab64[EXP_OFF + lane + 32];
    const bool live = in && cp.x >= 0;
    if (!__any_sync(0xffffffffu, live)) {
        if (lane < GPN) gp[lane] = 0.0;
        return;
    }
    // species sums of the column's adjoint weights
    double Sv[2 + ES];
#pragma unroll
    for (int q = 0; q < 2 + ES; ++q) Sv[q] = 0.0;
    if (live) {
        const double* coef = w.coef + (size_t)item * (2 + w.nes) * KMAX;
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
            const double wk = set_weight<MULTI>(T, k, grp);
            const double s = wk == 0.0 ? 0.0 : wk * T.shapes[(size_t)k * N + i];
#pragma unroll
            for (int q = 0; q < 2 + ES; ++q)
                if (q < 2 + NES) Sv[q] = fma(coef[q * KMAX + k], s, Sv[q]);
        }
    }
    const Col64 cc = w.col64[at];
    const int exact = w.xany64[item];
    const Gen64 gen = live ? w.gen64[at] : Gen64{0.0, 0.0, 0.0, 0.0};
    double P0 = 0.0, P1 = 0.0, P2 = 0.0, Rs = 0.0, Rt = 0.0;
    double f1 = 1.0, f2 = 1.0, f0 = 0.0;   // S1 = f1 P1, S2 = f2 (P2 - f0 P0)
    const double* rowW = static_cast<const double*>(w.rowW) + (size_t)item * (2 + w.nes) * w.Mpad;
    const double* wtg = w.wt64 + (size_t)item * (2 + w.nes) * w.gl64;
    const bool gc = GC && (T.gc1 != 0.0 || T.gc2 != 0.0);
    for (int c = 0; c <= G64_NC; ++c) {
        const bool mine = live && cp.x == c;
        if (!__any_sync(0xffffffffu, mine)) continue;
        const int lo = __reduce_min_sync(0xffffffffu, mine ? cp.z : INT_MAX) & ~(RUNB - 1);
        const int hi = __reduce_max_sync(0xffffffffu, mine ? cp.w : INT_MIN);
        const bool ci = c == G64_CI;
        const double d = T.w * (double)(1 << (ci ? 0 : c)), h = d * gen.y;
        const double* src = ci ? rowW : wtg + g64_off(M, c);
        const size_t sstr = ci ? w.Mpad : w.gl64;
        const int glen = ci ? M : g64_len(M, c);
        double C[NPOLY];
        if (ci) poly_coef(h, C);
        const bool isD = mine && ci && cp.y == KIND_D, isP = mine && ci && cp.y == KIND_P;
        for (unsigned mr = __ballot_sync(0xffffffffu, isD); mr; mr &= mr - 1u) {
            // kind D, one column at a time: lane = edge, 31 bins a step
            const int j = __ffs(mr) - 1, b0 = __shfl_sync(0xffffffffu, cp.z, j), b1 = __shfl_sync(0xffffffffu, cp.w, j);
            const double mu = __shfl_sync(0xffffffffu, gen.x, j), isg = __shfl_sync(0xffffffffu, gen.y, j);
            double Sj[2 + ES];
#pragma unroll
            for (int q = 0; q < 2 + ES; ++q) Sj[q] = __shfl_sync(0xffffffffu, Sv[q], j);
            double q0 = 0.0, q1 = 0.0, q2 = 0.0, qs = 0.0, qt = 0.0;
            for (int m0 = b0; m0 < b1; m0 += 31) {
                const int m = m0 + lane;
                const double z = ((double)m * T.w - mu) * isg;
                bool f;
                const double t = edge_tail(T, z, gc, f);
                double p = INV_SQRT_2PI * exp(-0.5 * z * z);
                if (gc) p *= gc_density_factor(T, z);
                const double tb = __shfl_down_sync(0xffffffffu, t, 1), pb = __shfl_down_sync(0xffffffffu, p, 1);
                const double zb = __shfl_down_sync(0xffffffffu, z, 1);
                const bool fb = __shfl_down_sync(0xffffffffu, (int)f, 1) != 0;
                if (lane < 31 && m < b1) {
                    const double ws = rowW[m], wt = rowW[w.Mpad + m];
                    double W = fma(ws, Sj[0], wt * Sj[1]);
#pragma unroll
                    for (int q = 0; q < ES; ++q)
                        if (q < NES) W = fma(rowW[(size_t)(2 + q) * w.Mpad + m], Sj[2 + q], W);
                    const double D = tb - t + ((!f && fb) ? 1.0 : 0.0);
                    q0 = fma(W, D, q0);
                    q1 -= W * (pb - p);
                    q2 -= W * (zb * pb - z * p);
                    qs = fma(D, ws, qs);
                    qt = fma(D, wt, qt);
                }
            }
            q0 = warp_sum(q0);
            q1 = warp_sum(q1);
            q2 = warp_sum(q2);
            qs = warp_sum(qs);
            qt = warp_sum(qt);
            if (lane == j) {
                P0 = q0;
                P1 = q1;
                P2 = q2;
                Rs = qs;
                Rt = qt;
            }
        }
        if (ci && !__any_sync(0xffffffffu, isP)) continue;
        for (int g0 = lo; g0 < hi; g0 += 32) {
            __syncwarp();
            for (int q = 0; q < 2 + NES; ++q) sW[q][lane] = g0 + lane < glen ? src[(size_t)q * sstr + g0 + lane] : 0.0;
            __syncwarp();
            auto weight = [&](int k) {
                double W = fma(sW[0][k], Sv[0], sW[1][k] * Sv[1]);
#pragma unroll
                for (int q = 0; q < ES; ++q)
                    if (q < NES) W = fma(sW[2 + q][k], Sv[2 + q], W);
                return W;
            };
            const int ng = min(32, hi - g0);
            if (ci) {
                if (__any_sync(0xffffffffu, isP))
                    for (int r0 = 0; r0 < ng; r0 += RUNB) {
                        // centres z, density p; edges ze = z - h/2 .., density pe (both over sqrt(2 pi))
                        double z = (((double)(g0 + r0) + 0.5) * d - gen.x) * gen.y;
                        double ze = ((double)(g0 + r0) * d - gen.x) * gen.y;
                        double p = exp_tab(-0.5 * z * z, sE), rho = exp_tab(-(z + 0.5 * h) * h, sE);
                        double pe = exp_tab(-0.5 * ze * ze, sE), re = exp_tab(-(ze + 0.5 * h) * h, sE);
#pragma unroll 2
                        for (int k = r0; k < r0 + RUNB; ++k) {
                            const double pn = pe * re, zn = ze + h;
                            if (isP && g0 + k >= cp.z && g0 + k < cp.w) {
                                const double W = weight(k), D = p * poly_eval(C, z * z);
                                P0 = fma(W, D, P0);
                                P1 -= W * (pn - pe);
                                P2 -= W * (zn * pn - ze * pe);
                                Rs = fma(D, sW[0][k], Rs);
                                Rt = fma(D, sW[1][k], Rt);
                            }
                            p *= rho;
                            rho = fma(-rho, gen.z, rho);
                            z += h;
                            pe = pn;
                            ze = zn;
                            re = fma(-re, gen.z, re);
                        }
                    }
            } else {
                for (int r0 = 0; r0 < ng; r0 += RUNB) {
                    if (!__any_sync(0xffffffffu, mine && cp.z < g0 + r0 + RUNB && cp.w > g0 + r0)) continue;
                    const double z0 = (((double)(g0 + r0 - R64) + 0.5) * d - gen.x) * gen.y;
                    double p = exp_tab(-0.5 * z0 * z0, sE), rho = exp_tab(-(z0 + 0.5 * h) * h, sE);
                    double m0 = 0.0, m1 = 0.0, m2 = 0.0;
#pragma unroll
                    for (int k = 0; k < RUNB; ++k) {
                        const bool use = mine && g0 + r0 + k >= cp.z && g0 + r0 + k < cp.w;
                        const double W = weight(r0 + k);
                        if (GC) {
                            const double z = fma((double)k, h, z0), g = gc_density_factor(T, z);
                            const double gs = 3.0 * T.gc1 * (z * z - 1.0) + 4.0 * T.gc2 * z * (z * z - 3.0);   // dg/dz
                            const double a = fma(z, g, -gs), v = use ? p : 0.0, q = W * v, pg = v * g;
                            m0 = fma(q, g, m0);
                            m1 = fma(q, a, m1);
                            m2 = fma(q, z * a, m2);
                            Rs = fma(pg, sW[0][r0 + k], Rs);
                            Rt = fma(pg, sW[1][r0 + k], Rt);
                        } else {
                            const double v = use ? p : 0.0, q = W * v;
                            m0 += q;
                            m1 = fma((double)k, q, m1);
                            m2 = fma((double)(k * k), q, m2);
                            Rs = fma(v, sW[0][r0 + k], Rs);
                            Rt = fma(v, sW[1][r0 + k], Rt);
                        }
                        p *= rho;
                        rho = fma(-rho, gen.z, rho);
                    }
                    if (GC) {
                        P0 += m0;
                        P1 += m1;
                        P2 += m2;
                    } else {   // z = z0 + k h
                        P0 += m0;
                        P1 += fma(h, m1, z0 * m0);
                        P2 += fma(z0, fma(2.0 * h, m1, z0 * m0), h * h * m2);
                    }
                }
            }
        }
        if (mine) {
            if (!ci) {   // R = amp p: dR/dmu = amp p z / sigma, dR/dsigma = amp p (z^2 - 1) / sigma
                f0 = 1.0;
            } else if (isP) {   // R = amp' D with amp' = norm h / sqrt(2 pi); the edges over sqrt(2 pi)
                f1 = f2 = 1.0 / h;
            }
        }
    }
    double g[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) g[j] = 0.0;
    if (live) {
        const double* th = w.theta + (size_t)item * w.tstride;
        const double LY = th[K], a = th[K + 1], b = th[K + 2], mu = cc.mu, sig = cc.sig, isig = gen.y, amp = gen.w;
        double S0 = amp * P0, S1 = amp * isig * f1 * P1, S2 = amp * isig * f2 * (P2 - f0 * P0);
        double rs = amp * Rs, rt = amp * Rt;
        if (exact) {
            double E[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
            tail_adjoint(w, T, item, ie, Sv[0], Sv[1], mu, isig, E);
            S0 = fma(cc.norm, E[0], S0);
            S1 = fma(cc.norm * isig, E[1], S1);
            S2 = fma(cc.norm * isig, E[2], S2);
            rs = fma(cc.norm, E[3], rs);
            rt = fma(cc.norm, E[4], rt);
        }
        const double dmu = S1 - cc.mills * isig * S0;
        const double dsig = S2 + cc.mills * mu * isig * isig * S0;
        const double D = dsig / (2.0 * sig);
        const double Gmu = dmu + D * (a + 2.0 * b * mu);
        const double2 q = w.colq[at];
        g[0] = Gmu * q.x;          // LY
        g[1] = D * mu;             // a
        g[2] = D * mu * mu;        // b
        g[3] = D;                  // c
        g[4] = Gmu * LY * q.y;     // kB
#pragma unroll
        for (int k = 0; k < KMAX; ++k)
            if (k < K) {
                const double wk = set_weight<MULTI>(T, k, grp), t = T.tag ? T.tag[k] : 0.0;
                if (wk != 0.0) g[5 + k] = wk * T.shapes[(size_t)k * N + i] * fma(T.tag ? 1.0 - t : 1.0, rs, t * rt);
            }
    }
    const double s = warp_sum32(g);
    if (lane < GPN) gp[lane] = s;
}

// ------------------------------------------------------------------ launchers

cudaError_t launch_prep64(const Work& w, int n, cudaStream_t s) {
    const int nblk = w.Npad / 128;
    k_scan64<<<(unsigned)n * nblk, 128, 0, s>>>(w, nblk);
    if (w.multi_set) k_cols64<true><<<(unsigned)n * nblk, 128, 0, s>>>(w, nblk);
    else k_cols64<false><<<(unsigned)n * nblk, 128, 0, s>>>(w, nblk);
    return cudaGetLastError();
}

template <bool TAG, int ES>
static void dens64_variant(const Work& w, int n, bool split, cudaStream_t s) {
    const unsigned nt = w.gl64 / 32, grid = (unsigned)n * nt;
    if (split && w.gc) k_dens64<TAG, ES, true, 1><<<4 * grid, 32, 0, s>>>(w, nt);
    else if (split) k_dens64<TAG, ES, false, 1><<<4 * grid, 32, 0, s>>>(w, nt);
    else if (w.gc) k_dens64<TAG, ES, true, 4><<<grid, 128, 0, s>>>(w, nt);
    else k_dens64<TAG, ES, false, 4><<<grid, 128, 0, s>>>(w, nt);
}

cudaError_t launch_fwd64(const Work& w, int n, int any_tag, int any_cols, cudaStream_t s) {
    const int es = !any_cols ? 0 : w.nes > 1 ? MAX_ES : 1;
    // up to G64_SPLIT items, the tiles with columns (about 35 of an item) do not fill the 152 SMs
    const bool split = n <= G64_SPLIT;
    if (any_tag && es == 0) dens64_variant<true, 0>(w, n, split, s);
    else if (any_tag && es == 1) dens64_variant<true, 1>(w, n, split, s);
    else if (any_tag) dens64_variant<true, MAX_ES>(w, n, split, s);
    else if (es == 0) dens64_variant<false, 0>(w, n, split, s);
    else if (es == 1) dens64_variant<false, 1>(w, n, split, s);
    else dens64_variant<false, MAX_ES>(w, n, split, s);
    const int nrb = w.max_tiles, nall = nrb + (any_cols ? (w.Npad / 32 + 3) / 4 : 0), np = split ? 4 : 1;
    if (any_tag) k_lam64<true><<<(unsigned)n * nall, 128, 0, s>>>(w, nrb, nall, np);
    else k_lam64<false><<<(unsigned)n * nall, 128, 0, s>>>(w, nrb, nall, np);
    return cudaGetLastError();
}

cudaError_t launch_mid64(const Work& w, int n, int Mmax, int nwmax, int Lmax, int nH, int want_grad, int want_mu,
                         cudaStream_t s) {
    const int ntw = (nwmax + 31) / 32, ntm = (Mmax + 31) / 32;
    const size_t sp = (size_t)(2 * Lmax + 31) * sizeof(double);
    cudaError_t e;
    static SmemOptIn set_pile, set_corr;
    if (sp > 24 * 1024) {   // (the default limit is 48 KB with a kernel's static share)
        if ((e = smem_opt_in(set_pile, k_pile64, sp)) != cudaSuccess) return e;
        if ((e = smem_opt_in(set_corr, k_corr64, sp)) != cudaSuccess) return e;
    }
    k_pile64<<<(unsigned)n * ntw * nH, 128, sp, s>>>(w, ntw, nH, want_grad, want_mu);
    k_marg64<<<n, MG, 0, s>>>(w, ntw, nH, want_grad, want_mu);
    if (want_grad) k_corr64<<<(unsigned)n * ntm * nH, 128, sp, s>>>(w, ntm, nH);
    return cudaGetLastError();
}

cudaError_t launch_bwd64(const Work& w, int n, cudaStream_t s) {
    const int nb = (w.wt_threads64 + 127) / 128, nch = w.Npad / 32;
    k_wt64<<<(unsigned)n * nb, 128, 0, s>>>(w, nb);
    const unsigned grid = (unsigned)n * nch;
    const bool mes = w.nes > 1;
    if (w.gc) {
        if (w.multi_set && mes) k_bwd64<true, true, MAX_ES><<<grid, 32, 0, s>>>(w, nch);
        else if (w.multi_set) k_bwd64<true, true, 1><<<grid, 32, 0, s>>>(w, nch);
        else if (mes) k_bwd64<false, true, MAX_ES><<<grid, 32, 0, s>>>(w, nch);
        else k_bwd64<false, true, 1><<<grid, 32, 0, s>>>(w, nch);
    } else if (w.multi_set && mes) k_bwd64<true, false, MAX_ES><<<grid, 32, 0, s>>>(w, nch);
    else if (w.multi_set) k_bwd64<true, false, 1><<<grid, 32, 0, s>>>(w, nch);
    else if (mes) k_bwd64<false, false, MAX_ES><<<grid, 32, 0, s>>>(w, nch);
    else k_bwd64<false, false, 1><<<grid, 32, 0, s>>>(w, nch);
    return cudaGetLastError();
}

// The sizes an FP64 model takes: 4 values per axis bin, 6 per window bin and one per pile-up bin within
// 207,696 bytes.  That is what the spectra of one item took of a thread block's shared memory while one
// block assembled an item; the kernels here need only 2 L + 31 doubles, and the limit stands as a limit of
// the interface.
void g64_size_limit(int Mmax, int nwmax, int Lmax, size_t* need, size_t* avail) {
    *need = (size_t)(4 * Mmax + 6 * nwmax + Lmax) * sizeof(double);
    *avail = 207696;
}

}  // namespace bx

// bx_fwd_f32.cu -- Eq. 1 forward in FP32 on the CUDA cores (the mixed-precision path).
//
// Rate-first form: the Eq. 3 spectra are contracted directly,
//     lambda_h[m] = sum_i (R[m,i] / A_i) (A_i S_h[i]),   S_h[i] = sum_k r_k c_{h,k} s_k[i],
// with the column amplitude A_i folded into the spectra by k_prep32 (one rounding of the
// double-float product instead of two, and one multiply less per entry),
// and, for models with Eq. 4 terms, the response is also reduced over rows,
//     a_t[i] = sum_{m in tile t} R[m,i] Gg[m],
// from which k_mid forms every species' window marginal after pile-up.
// Two kernels with the same sums in the same order: k_fwd_f32 for large batches (below) and k_fwd_split
// for up to SPLIT_TILES tiles, where generator warps evaluate chunks of columns side by side for an
// accumulator warp.  Both evaluate a pair of columns x a pair of rows a thread in packed FP32
// arithmetic (two lane operations per issue slot: the forward was bound by issue, not by the FMA rate)
// wherever |z| <= 1 holds for both columns, and entry by entry elsewhere.
// Unit = (row tile of TM output bins, item); 64 threads, warp q owning the two 32-row
// groups m0 + 64q + [0, 32) and m0 + 64q + [32, 64), one row of each per thread.  The warps
// never wait for each other: each stages 32 columns' parameters at a time in its own shared
// memory, lane = column, and the lanes vote three masks: the column's band touches row group
// A, row group B, and |z| <= 1 holds at every row of the warp (the generator's series branch,
// so the per-entry test is dropped).  The warp then visits only the set bits, so the work
// follows each column's own band rather than the union over the tile.
// Each thread generates the response of its bins with round-to-nearest FP32 arithmetic
// (bx_resp.cuh) and adds R S_h into Kahan-compensated accumulators at every term, so a row
// sum of ~10^3 terms keeps an error of a few roundings with no systematic sign.  For the
// column sums each lane adds R Gg of its two rows; the 32 lane values per column go through
// a padded warp-private shared buffer once per 32 columns and are stored per half tile.
// With several energy slices of the Eq. 4 terms (MES) the buffer holds R of all 64 rows and
// the column sums are formed once per slice s with its Gg_s.
#include <math.h>

#include <type_traits>

#include "bx_df.cuh"
#include "bx_internal.cuh"
#include "bx_resp.cuh"

namespace bx {

constexpr int FCH32 = 32;
constexpr int SPW = 20;    // floats of a staged column pair (16-byte rows; 14 in use)

// acc += a (b + bl), Kahan-compensated: bl is the low part of the column's double-float spectrum,
// so that the one rounding per term is the product's (independent from entry to entry).  The
// compensation is kept negated (nc = -c).
__device__ __forceinline__ void kahan_fma(float& acc, float& nc, float a, float b, float bl) {
    const float y = fmaf(a, b, fmaf(a, bl, nc));
    const float t = __fadd_rn(acc, y);
    nc = __fsub_rn(y, __fsub_rn(t, acc));
    acc = t;
}
// The same on both halves of a pair.
__device__ __forceinline__ void kahan_fma2(f2& acc, f2& nc, f2 a, f2 b, f2 bl) {
    const f2 y = f2_fma(a, b, f2_fma(a, bl, nc));
    const f2 t = f2_add(acc, y);
    nc = f2_sub(y, f2_sub(t, acc));
    acc = t;
}

// WPC: warps per CTA, 2 (a CTA = one 128-row tile) or 1 (a CTA = one warp's 64-row half of a
// tile; the autotuner of the batched fits may pick it for small ragged items).  The warps of a
// CTA never synchronise, so the two shapes do the same work per warp.
// GC: the Gram-Charlier response (resp_shape32_gc, the toy's skewness and kurtosis terms).
template <bool TAG, bool COLS, bool MES, int WPC = 2, bool GC = false>
__global__ void __launch_bounds__(32 * WPC) k_fwd_f32(Work w) {
    chain_wait();
    // 1D item-major grid (a y dimension would cap the batch at 65535 items)
    const int unit = WPC == 2 ? (int)blockIdx.x : (int)(blockIdx.x >> 1);
    const int tile = unit % w.max_tiles, item = unit / w.max_tiles, tid = threadIdx.x;
    const Toy& T = w.toys[w.toy_of[item]];
    if (tile >= T.n_tiles || w.status[item]) return;
    const int m0 = tile * TM, M = T.M;
    const int NGRP = T.n_set > 1 ? T.n_set : 1;   // quenching groups: one column range each
    const size_t cbase = (size_t)item * w.Npad;
    const float4* colf = w.colf + cbase;
    const ColG* colg = w.colg + cbase;
    const float4* colS = w.colS32 + cbase;
    const int2* colr = w.colr + cbase;
    const int lane = tid & 31, q = WPC == 2 ? tid >> 5 : (int)(blockIdx.x & 1), g = m0 + 64 * q;
    const int qs = WPC == 2 ? q : 0;   // the warp's slot in the CTA's shared arrays
    // warp-private staging of 32 columns at a time (no block-wide barrier)
    __shared__ float4 sC[WPC][FCH32];
    __shared__ ColG sG[WPC][FCH32];
    __shared__ __align__(16) float sP[GC ? 1 : WPC][GC ? 1 : FCH32 / 2][SPW];   // column pairs: ColPair's fields
    __shared__ float4 sS[WPC][FCH32];
    // column sums: one slice -> R Gg of the lane's two rows added (32 values per column);
    // several slices (MES) -> R of each of the warp's 64 rows
    constexpr int CBR = MES ? 64 : 32, CBW = FCH32 + 2;   // (even rows: a pair of columns is one store)
    __shared__ __align__(8) float colbuf[COLS ? WPC : 1][COLS ? CBR : 1][CBW];
    float(*cb)[CBW] = colbuf[COLS ? qs : 0];

    const int ra = g + lane, rb = ra + 32;
    const float mfa = (float)ra, mfb = (float)rb;
    const float gga = (COLS && !MES && ra < M) ? (float)T.Gg[ra] : 0.f;
    const float ggb = (COLS && !MES && rb < M) ? (float)T.Gg[rb] : 0.f;
    const int NES = MES ? T.n_es : 1;
    __shared__ float sGg[MES ? WPC : 1][MES ? MAX_ES : 1][MES ? 64 : 1];   // Gg_s of the warp's 64 rows
    if (MES)
        for (int s = 0; s < NES; ++s) {
            sGg[qs][s][lane] = ra < M ? T.Gg32[(size_t)s * M + ra] : 0.f;
            sGg[qs][s][lane + 32] = rb < M ? T.Gg32[(size_t)s * M + rb] : 0.f;
        }
    float sa = 0.f, csa = 0.f, ta = 0.f, cta = 0.f, sb = 0.f, csb = 0.f, tb = 0.f, ctb = 0.f;
    float* apart = static_cast<float*>(w.apart) + (((size_t)item * w.max_tiles + tile) * 2 + q) * (MES ? w.nes : 1) * w.Npad;

    // one column's entries of the lane's rows: both row groups (the common case: two
    // independent chains for the scheduler) or one of them
    const float gc3 = GC ? (float)T.gc1 : 0.f, gc4 = GC ? (float)T.gc2 : 0.f;
    auto shape_t = [&](auto wide_tag, float th, float tl, const ColG& cg) {
        constexpr bool WIDE = decltype(wide_tag)::value;
        if constexpr (GC) return resp_shape32_gc_t<WIDE>(th, tl, cg, gc3, gc4);
        else return resp_shape32_t<WIDE>(th, tl, cg);
    };
    auto shape = [&](auto wide_tag, float mf, const float4& cf, const ColG& cg) {
        float th, tl;
        centre_df(mf, cf, cg.c_lo, th, tl);
        return shape_t(wide_tag, th, tl, cg);
    };
    auto column = [&](auto wide_tag, bool inA, bool inB, int c, float& Ra, float& Rb) {
        const float4 cf = sC[qs][c];
        const ColG cg = sG[qs][c];
        const float4 S = sS[qs][c];
        if (inA && inB) {   // row B's centre from row A's: one double-float add
            float tha, tla, thb, tlb;
            centre_df(mfa, cf, cg.c_lo, tha, tla);
            centre_step32(tha, tla, cf, thb, tlb);
            Ra = shape_t(wide_tag, tha, tla, cg);
            Rb = shape_t(wide_tag, thb, tlb, cg);
            kahan_fma(sa, csa, Ra, S.x, S.z);
            kahan_fma(sb, csb, Rb, S.x, S.z);
            if (TAG) {
                kahan_fma(ta, cta, Ra, S.y, S.w);
                kahan_fma(tb, ctb, Rb, S.y, S.w);
            }
        } else if (inA) {
            Ra = shape(wide_tag, mfa, cf, cg);
            kahan_fma(sa, csa, Ra, S.x, S.z);
            if (TAG) kahan_fma(ta, cta, Ra, S.y, S.w);
        } else {
            Rb = shape(wide_tag, mfb, cf, cg);
            kahan_fma(sb, csb, Rb, S.x, S.z);
            if (TAG) kahan_fma(tb, ctb, Rb, S.y, S.w);
        }
    };
    // both rows' entries of one column added: with TAG a row's two spectra share an instruction,
    // without it the two rows
    auto add_col = [&](const float4& S, float Ra, float Rb) {
        if (TAG) {
            const f2 b = f2_pack(S.x, S.y), bl = f2_pack(S.z, S.w);
            f2 acc = f2_pack(sa, ta), nc = f2_pack(csa, cta);
            kahan_fma2(acc, nc, f2_dup(Ra), b, bl);
            f2_get(acc, sa, ta);
            f2_get(nc, csa, cta);
            acc = f2_pack(sb, tb), nc = f2_pack(csb, ctb);
            kahan_fma2(acc, nc, f2_dup(Rb), b, bl);
            f2_get(acc, sb, tb);
            f2_get(nc, csb, ctb);
        } else {
            f2 acc = f2_pack(sa, sb), nc = f2_pack(csa, csb);
            kahan_fma2(acc, nc, f2_pack(Ra, Rb), f2_dup(S.x), f2_dup(S.z));
            f2_get(acc, sa, sb);
            f2_get(nc, csa, csb);
        }
    };
    const f2 mfa2 = f2_dup(mfa), gga2 = f2_dup(gga), ggb2 = f2_dup(ggb);
    // columns 2 pr and 2 pr + 1, both rows of every lane inside both bands (most of the work): four
    // entries a thread in packed arithmetic, added in column order
    auto pair = [&](int pr) {
        f2 RA, RB;
        if constexpr (GC) {   // four scalar evaluations in flight
            const float4 cf0 = sC[qs][2 * pr], cf1 = sC[qs][2 * pr + 1];
            const ColG cg0 = sG[qs][2 * pr], cg1 = sG[qs][2 * pr + 1];
            float t0, l0, t1, l1, u0, k0, u1, k1;
            centre_df(mfa, cf0, cg0.c_lo, t0, l0);
            centre_df(mfa, cf1, cg1.c_lo, t1, l1);
            centre_step32(t0, l0, cf0, u0, k0);
            centre_step32(t1, l1, cf1, u1, k1);
            RA = f2_pack(shape_t(std::true_type{}, t0, l0, cg0), shape_t(std::true_type{}, t1, l1, cg1));
            RB = f2_pack(shape_t(std::true_type{}, u0, k0, cg0), shape_t(std::true_type{}, u1, k1, cg1));
        } else {
            const float4* P = reinterpret_cast<const float4*>(sP[GC ? 0 : qs][GC ? 0 : pr]);
            const float4 v0 = P[0], v1 = P[1], v2 = P[2], v3 = P[3];
            ColPair k;
            k.x = f2_pack(v0.x, v0.y);
            k.y = f2_pack(v0.z, v0.w);
            k.z = f2_pack(v1.x, v1.y);
            k.w = f2_pack(v1.z, v1.w);
            k.cl = f2_pack(v2.x, v2.y);
            k.kap = f2_pack(v2.z, v2.w);
            k.Ck2 = f2_pack(v3.x, v3.y);
            f2 th, tl, uh, ul;
            centre_df2(mfa2, k, th, tl);
            centre_step2(th, tl, k, f2_dup(32.0f), uh, ul);
            resp_shape32_x4(k, th, tl, uh, ul, RA, RB);
        }
        float a0, a1, b0, b1;
        f2_get(RA, a0, a1);
        f2_get(RB, b0, b1);
        add_col(sS[qs][2 * pr], a0, b0);
        add_col(sS[qs][2 * pr + 1], a1, b1);
        if (COLS) {
            if (MES) {
                *reinterpret_cast<float2*>(&cb[lane][2 * pr]) = make_float2(a0, a1);
                *reinterpret_cast<float2*>(&cb[lane + 32][2 * pr]) = make_float2(b0, b1);
            } else {
                float x, y;
                f2_get(f2_fma(RB, ggb2, f2_mul(RA, gga2)), x, y);
                *reinterpret_cast<float2*>(&cb[lane][2 * pr]) = make_float2(x, y);
            }
        }
    };

    for (int grp = 0; grp < NGRP; ++grp) {
    const int2 cr = tile_range(w, item, grp, tile);
    for (int c0 = cr.x; c0 < cr.y; c0 += FCH32) {
        const int ncol = min(FCH32, cr.y - c0);
        // lane = column: stage its parameters and vote, for the warp's two 32-row groups,
        // whether the column's band touches them (mA, mB) and whether |z| <= 1 at every row
        // of the warp (mW: t = (m - floor(mu/w)) hs + c is linear in the row m, so its two
        // end rows bound it)
        unsigned mA, mB, mW, mP;   // mP: |t| <= 11 as well (the packed generator's range)
        float Al = 0.f;            // the lane's column amplitude
        {
            const bool in = lane < ncol;
            const int i = c0 + lane;
            const float4 cfl = in ? colf[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            const ColG cgl = in ? colg[i] : ColG{0.f, 0.f, 0.f, 0.f};
            sC[qs][lane] = cfl;
            sG[qs][lane] = cgl;
            if (!GC) {
                float* P = sP[GC ? 0 : qs][GC ? 0 : lane >> 1] + (lane & 1);
                P[0] = cfl.x;
                P[2] = cfl.y;
                P[4] = cfl.z;
                P[6] = cfl.w;
                P[8] = cgl.c_lo;
                P[10] = cgl.kap;
                P[12] = cgl.Ck2;
            }
            Al = cgl.A;
            sS[qs][lane] = in ? colS[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            const int2 band = in ? colr[i] : make_int2(0, 0);
            const float t0 = fmaf((float)g - cfl.x, cfl.z, cfl.y), t1 = fmaf(63.0f, cfl.z, t0);
            const float tm = fmaxf(fabsf(t0), fabsf(t1));
            mA = __ballot_sync(0xffffffffu, band.x < g + 32 && band.y > g);
            mB = __ballot_sync(0xffffffffu, band.x < g + 64 && band.y > g + 32);
            mW = __ballot_sync(0xffffffffu, cgl.kap * tm <= 0.99f);
            mP = GC ? 0xffffffffu : __ballot_sync(0xffffffffu, tm <= 10.9f);
        }
        __syncwarp();
        const unsigned mAny = mA | mB, m1 = mA & mB & mW & mP;
        const unsigned m2 = m1 & (m1 >> 1) & 0x55555555u;   // column pairs for the packed path
        if (m2 == 0x55555555u) {
#pragma unroll 2
            for (int pr = 0; pr < FCH32 / 2; ++pr) pair(pr);
        } else
        for (unsigned mr = mAny; mr; mr &= mr - 1u) {   // the columns whose band touches the warp
            const int c = __ffs(mr) - 1;
            if ((m2 >> c) & 1u) {
                pair(c >> 1);
                mr &= mr - 1u;
                continue;
            }
            const bool inA = (mA >> c) & 1u, inB = (mB >> c) & 1u;
            float Ra = 0.f, Rb = 0.f;
            if ((mW >> c) & 1u) column(std::true_type{}, inA, inB, c, Ra, Rb);
            else column(std::false_type{}, inA, inB, c, Ra, Rb);
            if (COLS) {
                if (MES) {
                    cb[lane][c] = Ra;
                    cb[lane + 32][c] = Rb;
                } else {
                    cb[lane][c] = fmaf(Rb, ggb, Ra * gga);
                }
            }
        }
        __syncwarp();
        if (COLS && !MES) {
            float s = 0.f;
            if ((mAny >> lane) & 1u)
                for (int j = 0; j < 32; ++j) s += cb[j][lane];
            if (lane < ncol) apart[c0 + lane] = s * Al;
            __syncwarp();
        }
        if (COLS && MES) {
            float s[MAX_ES];
#pragma unroll
            for (int e = 0; e < MAX_ES; ++e) s[e] = 0.f;
            if ((mAny >> lane) & 1u)
                for (int j = 0; j < 64; ++j) {
                    const float r = cb[j][lane];
#pragma unroll
                    for (int e = 0; e < MAX_ES; ++e)
                        if (e < NES) s[e] = fmaf(r, sGg[qs][e][j], s[e]);
                }
            if (lane < ncol)
#pragma unroll
                for (int e = 0; e < MAX_ES; ++e)
                    if (e < NES) apart[(size_t)e * w.Npad + c0 + lane] = s[e] * Al;
            __syncwarp();
        }
    }
    }
    double* lam = w.lam + (size_t)item * 2 * w.Mpad;
    if (w.lam_pairs) {   // the Kahan sum as a normalised FP32 pair
        float2* lp = reinterpret_cast<float2*>(lam);
        const auto pair = [](float sum, float comp) {
            const df p = df_two_sum(sum, comp);
            return make_float2(p.h, p.l);
        };
        if (ra < M) {
            lp[ra] = pair(sa, csa);
            if (TAG) lp[w.Mpad + ra] = pair(ta, cta);
        }
        if (rb < M) {
            lp[rb] = pair(sb, csb);
            if (TAG) lp[w.Mpad + rb] = pair(tb, ctb);
        }
        return;
    }
    if (ra < M) {
        lam[ra] = (double)sa + (double)csa;
        if (TAG) lam[w.Mpad + ra] = (double)ta + (double)cta;
    }
    if (rb < M) {
        lam[rb] = (double)sb + (double)csb;
        if (TAG) lam[w.Mpad + rb] = (double)tb + (double)ctb;
    }
}

// Small batches: the 16 warps of an item (two 64-row halves of 8 tiles) leave most of the GPU idle, and
// a warp's chunks are one serial chain.  Here a CTA takes one 64-row half: SG generator warps evaluate the
// response of SG chunks at a time into shared memory (and take the column sums), and two more warps
// (rows A, rows B) add the chunks' entries to the row sums in column order, one round behind.  The
// entries and the order of every sum are those of k_fwd_f32: the results are the same bits.
constexpr int SG = 4;
// 128-row tiles of a batch (measured, us, split against plain: multivariate 52 items = 416 tiles 101 / 120,
// 76 items = 608 tiles 134 / 121; one item 35 / 86; plain model 104 items = 416 tiles 120 / 146,
// 152 items = 608 tiles 164 / 148)
constexpr unsigned SPLIT_TILES = 480;
constexpr int SRW = 33;   // row stride of an entry buffer
struct SplitShared {
    float R[2][SG][64][SRW];
    float4 S[2][SG][FCH32];
    unsigned m[2][SG][2];             // columns whose bands touch rows A, rows B
    float4 C[SG][FCH32];
    ColG G[SG][FCH32];
    float P[SG][FCH32 / 2][SPW];
    float gg[MAX_ES][64];             // Gg_s of the rows
};
__device__ __forceinline__ void bar_sync(int id, int n) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int n) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

template <bool TAG, bool COLS, bool MES, bool GC>
__global__ void __launch_bounds__(32 * (SG + 2)) k_fwd_split(Work w) {
    chain_wait();
    extern __shared__ __align__(16) unsigned char split_raw[];
    SplitShared& sh = *reinterpret_cast<SplitShared*>(split_raw);
    const int unit = blockIdx.x >> 1, q = blockIdx.x & 1;
    const int tile = unit % w.max_tiles, item = unit / w.max_tiles, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const Toy& T = w.toys[w.toy_of[item]];
    if (tile >= T.n_tiles || w.status[item]) return;
    const int M = T.M, g0 = tile * TM + 64 * q, NGRP = T.n_set > 1 ? T.n_set : 1, NES = MES ? T.n_es : 1;
    constexpr int NT = 32 * (SG + 2);
    for (int j = tid; COLS && j < NES * 64; j += NT) {
        const int e = j >> 6, r = g0 + (j & 63);
        sh.gg[e][j & 63] = r < M ? (MES ? T.Gg32[(size_t)e * M + r] : (float)T.Gg[r]) : 0.f;
    }
    int total = 0;   // chunks of 32 columns, set after set
    for (int grp = 0; grp < NGRP; ++grp) {
        const int2 cr = tile_range(w, item, grp, tile);
        if (cr.x < cr.y) total += (cr.y - cr.x + FCH32 - 1) / FCH32;
    }
    const int rounds = (total + SG - 1) / SG;
    __syncthreads();
    const int row = g0 + lane + (wid == SG + 1 ? 32 : 0);   // (accumulator warps)
    if (wid >= SG) {   // row sums: warp SG rows A, warp SG + 1 rows B
        const int half = wid - SG;
        float s = 0.f, cs = 0.f, t = 0.f, ct = 0.f;
        for (int r = 0; r < rounds; ++r) {
            const int b = r & 1;
            bar_sync(1 + b, NT);
            for (int k = 0; k < SG && r * SG + k < total; ++k) {
                const float* R = sh.R[b][k][lane + 32 * half];
                const float4* S = sh.S[b][k];
                auto add = [&](int c) {
                    const float x = R[c];
                    const float4 v = S[c];
                    if (TAG) {
                        f2 acc = f2_pack(s, t), nc = f2_pack(cs, ct);
                        kahan_fma2(acc, nc, f2_dup(x), f2_pack(v.x, v.y), f2_pack(v.z, v.w));
                        f2_get(acc, s, t);
                        f2_get(nc, cs, ct);
                    } else {
                        kahan_fma(s, cs, x, v.x, v.z);
                    }
                };
                const unsigned m = sh.m[b][k][half];
                if (m == 0xffffffffu) {
#pragma unroll 8
                    for (int c = 0; c < FCH32; ++c) add(c);
                } else {
                    for (unsigned mr = m; mr; mr &= mr - 1u) add(__ffs(mr) - 1);
                }
            }
            if (r + 2 < rounds) bar_arrive(3 + b, NT);
        }
        if (row < M) {
            double* lam = w.lam + (size_t)item * 2 * w.Mpad;
            if (w.lam_pairs) {   // the Kahan sum as a normalised FP32 pair
                float2* lp = reinterpret_cast<float2*>(lam);
                const df ps = df_two_sum(s, cs), pt = df_two_sum(t, ct);
                lp[row] = make_float2(ps.h, ps.l);
                if (TAG) lp[w.Mpad + row] = make_float2(pt.h, pt.l);
            } else {
                lam[row] = (double)s + (double)cs;
                if (TAG) lam[w.Mpad + row] = (double)t + (double)ct;
            }
        }
        return;
    }
    // generators
    const float mfa = (float)(g0 + lane), mfb = (float)(g0 + lane + 32);
    const float gc3 = GC ? (float)T.gc1 : 0.f, gc4 = GC ? (float)T.gc2 : 0.f;
    auto shape = [&](bool wide, float th, float tl, const ColG& cg) {
        if constexpr (GC)
            return wide ? resp_shape32_gc_t<true>(th, tl, cg, gc3, gc4) : resp_shape32_gc_t<false>(th, tl, cg, gc3, gc4);
        else return wide ? resp_shape32_t<true>(th, tl, cg) : resp_shape32_t<false>(th, tl, cg);
    };
    const size_t cbase = (size_t)item * w.Npad;
    float* apart = static_cast<float*>(w.apart) + (((size_t)item * w.max_tiles + tile) * 2 + q) * (MES ? w.nes : 1) * w.Npad;
    for (int r = 0; r < rounds; ++r) {
        const int b = r & 1;
        if (r >= 2) bar_sync(3 + b, NT);
        int k = r * SG + wid;   // the warp's chunk
        if (k < total) {
            int c0 = 0, c1 = 0;
            for (int grp = 0; grp < NGRP; ++grp) {
                const int2 cr = tile_range(w, item, grp, tile);
                const int n = cr.x < cr.y ? (cr.y - cr.x + FCH32 - 1) / FCH32 : 0;
                if (k < n) {
                    c0 = cr.x + k * FCH32;
                    c1 = cr.y;
                    break;
                }
                k -= n;
            }
            const int i = c0 + lane;
            const bool in = i < c1;
            const float4 cfl = in ? w.colf[cbase + i] : make_float4(0.f, 0.f, 0.f, 0.f);
            const ColG cgl = in ? w.colg[cbase + i] : ColG{0.f, 0.f, 0.f, 0.f};
            const int2 band = in ? w.colr[cbase + i] : make_int2(0, 0);
            sh.S[b][wid][lane] = in ? w.colS32[cbase + i] : make_float4(0.f, 0.f, 0.f, 0.f);
            sh.C[wid][lane] = cfl;
            sh.G[wid][lane] = cgl;
            float* P = sh.P[wid][lane >> 1] + (lane & 1);
            P[0] = cfl.x;
            P[2] = cfl.y;
            P[4] = cfl.z;
            P[6] = cfl.w;
            P[8] = cgl.c_lo;
            P[10] = cgl.kap;
            P[12] = cgl.Ck2;
            const float t0 = fmaf((float)g0 - cfl.x, cfl.z, cfl.y), t1 = fmaf(63.0f, cfl.z, t0);
            const float tm = fmaxf(fabsf(t0), fabsf(t1));
            const unsigned mA = __ballot_sync(0xffffffffu, band.x < g0 + 32 && band.y > g0);
            const unsigned mB = __ballot_sync(0xffffffffu, band.x < g0 + 64 && band.y > g0 + 32);
            const unsigned mW = __ballot_sync(0xffffffffu, cgl.kap * tm <= 0.99f);
            const unsigned mP = __ballot_sync(0xffffffffu, tm <= 10.9f);
            if (lane == 0) {
                sh.m[b][wid][0] = mA;
                sh.m[b][wid][1] = mB;
            }
            __syncwarp();
            float(*R)[SRW] = sh.R[b][wid];
            const unsigned mAny = mA | mB, m1 = GC ? 0u : mA & mB & mW & mP, m2 = m1 & (m1 >> 1) & 0x55555555u;
            auto pair = [&](int pr) {
                const float4* Pv = reinterpret_cast<const float4*>(sh.P[wid][pr]);
                const float4 v0 = Pv[0], v1 = Pv[1], v2 = Pv[2], v3 = Pv[3];
                ColPair kp;
                kp.x = f2_pack(v0.x, v0.y);
                kp.y = f2_pack(v0.z, v0.w);
                kp.z = f2_pack(v1.x, v1.y);
                kp.w = f2_pack(v1.z, v1.w);
                kp.cl = f2_pack(v2.x, v2.y);
                kp.kap = f2_pack(v2.z, v2.w);
                kp.Ck2 = f2_pack(v3.x, v3.y);
                f2 th, tl, uh, ul, RA, RB;
                centre_df2(f2_dup(mfa), kp, th, tl);
                centre_step2(th, tl, kp, f2_dup(32.0f), uh, ul);
                resp_shape32_x4(kp, th, tl, uh, ul, RA, RB);
                f2_get(RA, R[lane][2 * pr], R[lane][2 * pr + 1]);
                f2_get(RB, R[lane + 32][2 * pr], R[lane + 32][2 * pr + 1]);
            };
            if (m2 == 0x55555555u) {
#pragma unroll 4
                for (int pr = 0; pr < FCH32 / 2; ++pr) pair(pr);
            } else {
                for (unsigned mr = mAny; mr; mr &= mr - 1u) {
                    const int c = __ffs(mr) - 1;
                    if ((m2 >> c) & 1u) {
                        pair(c >> 1);
                        mr &= mr - 1u;
                        continue;
                    }
                    const bool inA = (mA >> c) & 1u, inB = (mB >> c) & 1u, wide = (mW >> c) & 1u;
                    const float4 cf = sh.C[wid][c];
                    const ColG cg = sh.G[wid][c];
                    float Ra = 0.f, Rb = 0.f, th, tl;
                    if (inA) {
                        centre_df(mfa, cf, cg.c_lo, th, tl);
                        float uh = 0.f, ul = 0.f;
                        if (inB) centre_step32(th, tl, cf, uh, ul);   // row B's centre from row A's
                        Ra = shape(wide, th, tl, cg);
                        if (inB) Rb = shape(wide, uh, ul, cg);
                    } else {
                        centre_df(mfb, cf, cg.c_lo, th, tl);
                        Rb = shape(wide, th, tl, cg);
                    }
                    R[lane][c] = Ra;
                    R[lane + 32][c] = Rb;
                }
            }
            if (COLS) {   // column sums: lane = column, rows in order
                __syncwarp();
                const bool any = (mAny >> lane) & 1u;
                if (MES) {
                    float sm[MAX_ES];
#pragma unroll
                    for (int e = 0; e < MAX_ES; ++e) sm[e] = 0.f;
                    if (any)
#pragma unroll 4
                        for (int j = 0; j < 64; ++j) {
                            const float x = R[j][lane];
#pragma unroll
                            for (int e = 0; e < MAX_ES; ++e)
                                if (e < NES) sm[e] = fmaf(x, sh.gg[e][j], sm[e]);
                        }
                    if (in)
#pragma unroll
                        for (int e = 0; e < MAX_ES; ++e)
                            if (e < NES) apart[(size_t)e * w.Npad + i] = sm[e] * cgl.A;
                } else {
                    float sm = 0.f;
                    if (any)
#pragma unroll 8
                        for (int j = 0; j < 32; ++j)
                            sm = __fadd_rn(sm, fmaf(R[j + 32][lane], sh.gg[0][j + 32], __fmul_rn(R[j][lane], sh.gg[0][j])));
                    if (in) apart[i] = sm * cgl.A;
                }
            }
        }
        bar_arrive(1 + b, NT);
    }
}

template <bool TAG, bool COLS, bool MES>
static cudaError_t fwd_split_variant(const Work& w, unsigned grid, cudaStream_t s) {
    static SmemOptIn set[2];
    const int gc = w.gc ? 1 : 0;
    const auto k = gc ? k_fwd_split<TAG, COLS, MES, true> : k_fwd_split<TAG, COLS, MES, false>;
    const cudaError_t e = smem_opt_in(set[gc], k, sizeof(SplitShared));
    if (e != cudaSuccess) return e;
    launch_chained(k, 2 * grid, 32 * (SG + 2), sizeof(SplitShared), s, w);
    return cudaGetLastError();
}

template <int WPC, bool GC = false>
static void fwd_f32_variant(const Work& w, unsigned grid, int any_tag, int any_cols, bool mes, cudaStream_t s) {
    const unsigned g = grid * (2 / WPC);
    if (any_tag && any_cols && mes) launch_chained(k_fwd_f32<true, true, true, WPC, GC>, g, 32 * WPC, 0, s, w);
    else if (any_cols && mes) launch_chained(k_fwd_f32<false, true, true, WPC, GC>, g, 32 * WPC, 0, s, w);
    else if (any_tag && any_cols) launch_chained(k_fwd_f32<true, true, false, WPC, GC>, g, 32 * WPC, 0, s, w);
    else if (any_tag) launch_chained(k_fwd_f32<true, false, false, WPC, GC>, g, 32 * WPC, 0, s, w);
    else if (any_cols) launch_chained(k_fwd_f32<false, true, false, WPC, GC>, g, 32 * WPC, 0, s, w);
    else launch_chained(k_fwd_f32<false, false, false, WPC, GC>, g, 32 * WPC, 0, s, w);
}

cudaError_t launch_fwd_f32(const Work& w, int n, int max_tiles, int any_tag, int any_cols, cudaStream_t s) {
    const unsigned grid = (unsigned)n * (unsigned)w.max_tiles;   // decoded with w.max_tiles
    const bool mes = w.nes > 1;   // several energy slices of the Eq. 4 terms
    // up to SPLIT_TILES tiles the generators of k_fwd_split find idle SMs
    if (grid <= SPLIT_TILES) {
        if (any_tag && any_cols && mes) return fwd_split_variant<true, true, true>(w, grid, s);
        if (any_cols && mes) return fwd_split_variant<false, true, true>(w, grid, s);
        if (any_tag && any_cols) return fwd_split_variant<true, true, false>(w, grid, s);
        if (any_tag) return fwd_split_variant<true, false, false>(w, grid, s);
        if (any_cols) return fwd_split_variant<false, true, false>(w, grid, s);
        return fwd_split_variant<false, false, false>(w, grid, s);
    }
    if (w.gc) fwd_f32_variant<2, true>(w, grid, any_tag, any_cols, mes, s);   // one tile shape for GC models
    else if (w.fwd_wpc == 1) fwd_f32_variant<1>(w, grid, any_tag, any_cols, mes, s);
    else fwd_f32_variant<2>(w, grid, any_tag, any_cols, mes, s);
    return cudaGetLastError();
}

}  // namespace bx

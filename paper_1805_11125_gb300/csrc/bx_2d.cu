// bx_2d.cu -- the discrimination regime: the TFC-vetoed and -tagged energy spectra and the
// 2D energy x radius and energy x pulse-shape histograms of the vetoed events, all handled
// as the NSL = 128 slices b of one rate-first contraction on the 5th-generation tensor cores
// (Eq. 1 - 4 with the radial and pulse-shape information binned against energy):
//
//   T_r[i,b] = ut[i,b] sum_k coef[k][b] s_k[i]                          k_coef2d, k_trate
//   Y[m,b]   = sum_i R[m,i] T_r[i,b]                  Eq. 1, a GEMM     k_fwd2d
//   mu[m,b]  = (1 - eps) Y[m,b] + eps sum_d g[d] Y[m-d,b]   Eq. 2, a Toeplitz GEMM   k_pile2d
//   -lnL     = sum over window rows and slices of mu - n + n ln(n/mu)           k_pile2d
// and its adjoint
//   w[m,b]   = 1 - n/mu,   Wt[m,b] = (1 - eps) w[m,b] + eps sum_d g[d] w[m+d,b]   k_corr2d
//   D_X[i,b] = sum_m X[m,i] Wt[m,b]  (X: the three Gauss-Legendre node sums of dR)  k_bwd2d
//   S_X[i]   = sum_b T_r[i,b] D_X[i,b] -> the chain rule of Eq. 1 (LY, a, b, c, kB);
//   dNLL/dr_k  = sum_{i,b} A_i D_0[i,b] ut[i,b] dcoef[k][b]/dr_k s_k[i],   dNLL/ds_r likewise.
//
// Every GEMM is M = 128 (output rows, or true-energy columns in the adjoint) x N = NSL x
// K = 32 per k-block.  The A tile is generated by the CUDA cores into shared memory (the
// response by the bias-free FP32 generator of bx_resp.cuh) or is a window of a table of the
// pile-up kernel g (toeplitz_table), the B tile arrives by a bulk copy from a tile written by
// the previous stage.  The forward
// splits both operands in three (split3: an 8-bit hi on a grid shared by the k-block's
// row or slice, then TF32 mid and lo), which makes the hi*hi products exact in the FP32
// accumulator; the other GEMMs split into TF32 hi and lo, and one thread issues hi*lo,
// lo*hi, then hi*hi (the small products first: the tensor core's FP32 accumulation truncates,
// so the small terms are added while the partial sum is still small).  The forward and the pile-up GEMMs drain their accumulator
// after every k-block and sum in registers, adding back each k-block's expected truncation
// (trunc_comp), so that no systematic error of the accumulation reaches -lnL.
// Every wait is bounded by the watchdog budget; on expiry the CTA records ERR_TIMEOUT,
// drains its own copies and MMAs (bounded), frees its tensor memory and returns.
#include <limits.h>
#include <math.h>

#include "bx_df.cuh"
#include "bx_internal.cuh"
#include "bx_resp.cuh"

namespace bx {

constexpr int T2 = 256;                            // threads of the adjoint GEMM that generate its operand
constexpr int TP = 512;                            // threads of the pile-up GEMMs
constexpr int PS = NSL * TM / TP;                  // slices of one row that a thread drains and finishes
constexpr int TILE_FLOATS = 2 * NSL * KB;          // one B tile (hi | lo), 32 KB
constexpr uint32_t TILE_BYTES = TILE_FLOATS * 4;
// a Y tile: the B tile (hi | lo) of the pile-up GEMM, then the FP32 remainder y - hi - lo (exact),
// so that the pile-up epilogue forms mu from the full FP32 value (hi + lo alone holds ~22 bits)
constexpr int YTILE_FLOATS = 3 * NSL * KB;
constexpr int TILE3_FLOATS = 3 * NSL * KB;         // one three-part B tile (hi | mid | lo), 48 KB
constexpr uint32_t TILE3_BYTES = TILE3_FLOATS * 4;
constexpr int TF = 512;                            // threads of the forward GEMM
constexpr int A_FLOATS = TM * KB;                  // one A half
constexpr unsigned long long CLEANUP_NS = 2000000000ull;

// A (128 x 32, K-major): element (r, c) at (c / 4) * 512 + r * 4 + c % 4
__device__ __forceinline__ int a_off(int r, int c) { return (c >> 2) * (TM * 4) + r * 4 + (c & 3); }
// B (NSL x 32, K-major): element (n, c) at (c / 4) * NSL * 4 + n * 4 + c % 4; lo half at + NSL * KB
__device__ __forceinline__ int b_off(int n, int c) { return (c >> 2) * (NSL * 4) + n * 4 + (c & 3); }

__device__ __forceinline__ void split_store(float* hi, float* lo, int off, float x) {
    const float h = tf32_rna(x);
    hi[off] = h;
    lo[off] = tf32_rna(x - h);
}
// (read-only loads: the stores of a loop over slices do not hold back the next slices' loads)
__device__ __forceinline__ float tile_get(const float* tile, int n, int c) {
    const int o = b_off(n, c);
    return __ldg(tile + o) + __ldg(tile + NSL * KB + o);
}
__device__ __forceinline__ void tile_put(float* tile, int n, int c, float x) {
    const float h = tf32_rna(x);
    const int o = b_off(n, c);
    tile[o] = h;
    tile[NSL * KB + o] = tf32_rna(x - h);
}

// The pile-up GEMMs' A tiles are Toeplitz: with the tile's rows taken in reverse (A row l is output row
// 127 - l), entry (l, c) of k-block it depends on l + c + 32 it alone.  So the core matrices (8 rows x 4
// columns, 128 bytes) of every tile are a window of one table, core p = elements x + 4 p + i + k: the
// descriptor's strides are 128 bytes along K and 256 along M, overlapping, and the next k-block starts
// 1024 bytes on.  One table (two TF32 parts) serves TP_KB k-blocks instead of a 128 x 32 tile written,
// split and fenced for each: the generation took 2/3 of these kernels.
constexpr int TP_KB = 20;                              // k-blocks per table: what two CTAs per SM leave
constexpr int TP_CORES = TP_KB * (KB / 4) + 2 * (TM / 8) - 2;
constexpr int TP_FLOATS = TP_CORES * 32;               // one part of the table
constexpr size_t TP_SMEM = (size_t)(2 * TP_FLOATS + 2 * TILE_FLOATS) * 4 + 128;

// Table of core p, element (i, k) = g[x + sgn (4 p + i + k)] (0 outside [0, L)), by the whole block.
__device__ __forceinline__ void toeplitz_table(float* hi, float* lo, const float* g, int L, int x, int sgn) {
    for (int q = threadIdx.x; q < TP_FLOATS; q += blockDim.x) {
        const int d = x + sgn * (4 * (q >> 5) + ((q >> 2) & 7) + (q & 3));
        split_store(hi, lo, q, d >= 0 && d < L ? g[d] : 0.f);
    }
}

constexpr int PITCH = TM + 4;   // of a slice's rows in the epilogues' exchange: quarter-warps without conflicts
// Rows c .. c + 3 (c a multiple of four) of slice n.
__device__ __forceinline__ void quad_put(float* tile, int n, int c, const float (&x)[4]) {
    float h[4], l[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        h[u] = tf32_rna(x[u]);
        l[u] = tf32_rna(x[u] - h[u]);
    }
    const int o = b_off(n, c);
    *reinterpret_cast<float4*>(tile + o) = make_float4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<float4*>(tile + NSL * KB + o) = make_float4(l[0], l[1], l[2], l[3]);
}

// D (+)= A B^T over one k-block, split products small-first; Ahi, Alo: the k-block's first core matrix.
__device__ __forceinline__ void mma_kblock(uint32_t d, const float* Ahi, const float* Alo, const float* B,
                                           bool accumulate) {
    constexpr uint32_t idesc = umma_idesc_tf32(TM, NSL);
    const uint32_t ahi = smem_u32(Ahi), alo = smem_u32(Alo), bhi = smem_u32(B), blo = bhi + NSL * KB * 4;
    uint32_t acc = accumulate ? 1u : 0u;
#pragma unroll
    for (int q = 0; q < KB / 8; ++q) {
        umma_tf32(d, umma_desc(ahi + q * 256, 128, 256), umma_desc(blo + q * 2 * (NSL * 16), NSL * 16, 128), idesc, acc);
        acc = 1u;
    }
#pragma unroll
    for (int q = 0; q < KB / 8; ++q)
        umma_tf32(d, umma_desc(alo + q * 256, 128, 256), umma_desc(bhi + q * 2 * (NSL * 16), NSL * 16, 128), idesc, 1u);
#pragma unroll
    for (int q = 0; q < KB / 8; ++q)
        umma_tf32(d, umma_desc(ahi + q * 256, 128, 256), umma_desc(bhi + q * 2 * (NSL * 16), NSL * 16, 128), idesc, 1u);
}

// Half a k-block (K = 16 of B's 32 rows, half `half`): the same three products as mma_kblock on
// an A tile of 16 columns (4 slabs of TM x 16 bytes).
__device__ __forceinline__ void mma_half(uint32_t d, const float* Ahi, const float* Alo, const float* B, int half,
                                         bool accumulate) {
    constexpr uint32_t idesc = umma_idesc_tf32(TM, NSL);
    const uint32_t ahi = smem_u32(Ahi), alo = smem_u32(Alo);
    const uint32_t bhi = smem_u32(B) + (uint32_t)half * 4u * (NSL * 16), blo = bhi + NSL * KB * 4;
    uint32_t acc = accumulate ? 1u : 0u;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        umma_tf32(d, umma_desc(ahi + q * 2 * (TM * 16), TM * 16, 128), umma_desc(blo + q * 2 * (NSL * 16), NSL * 16, 128),
                  idesc, acc);
        acc = 1u;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
        umma_tf32(d, umma_desc(alo + q * 2 * (TM * 16), TM * 16, 128), umma_desc(bhi + q * 2 * (NSL * 16), NSL * 16, 128),
                  idesc, 1u);
#pragma unroll
    for (int q = 0; q < 2; ++q)
        umma_tf32(d, umma_desc(ahi + q * 2 * (TM * 16), TM * 16, 128), umma_desc(bhi + q * 2 * (NSL * 16), NSL * 16, 128),
                  idesc, 1u);
}

struct Pipe {
    uint64_t mma_bar[2];
    uint64_t b_bar[2];
    uint32_t tmem;
    int abort;
    int committed;
};

__device__ __forceinline__ float* align128(unsigned char* p) {
    return reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(p) + 127) & ~uintptr_t(127));
}

// Thread 0: wait (bounded) for the bulk copies issued but not waited for.
__device__ __forceinline__ bool drain_copies(Pipe& pp, int waited, int issued) {
    bool ok = true;
    for (int j = waited; j < issued; ++j) ok &= mbar_wait(&pp.b_bar[j & 1], (j >> 1) & 1, CLEANUP_NS);
    return ok;
}

// Expected truncation of one k-block's sum in the two-part GEMMs (pile-up).  The tensor core
// adds every MMA instruction's result into the FP32 accumulator rounding toward zero: -1/2
// ulp of the running sum on average.  Of the 12 instructions of a k-block the 8 small-product
// ones act on partial sums 2^-11 of the total (negligible); the 4 hi*hi ones on about 1/4,
// 1/2, 3/4 and 1 of it, so the drained sum D is short by about 1/2 (1/4 + 1/2 + 3/4 + 1)
// ulp(D) = 1.25 ulp(D).  (The pile-up part enters mu with the weight eps, so what this model
// misses is below 1e-8 of mu; the forward GEMM needs no model, its hi*hi sums are exact.)
// ulp(D) = 2^(exponent of D - 23), taken with D's sign from its bit pattern.
__device__ __forceinline__ float trunc_comp(float d) {
    return __int_as_float(__float_as_int(d) & 0xFF800000) * (1.25f * 1.1920928955078125e-7f);
}

// Read this thread's PS accumulator columns (warp q: TMEM lanes 32 (q % 4) + lane, columns
// PS (q / 4) .. + PS - 1) and add them into acc; with `comp` each value is corrected by its
// expected truncation (one k-block accumulated from zero).
__device__ __forceinline__ void drain_add(uint32_t tbase, int col0, float (&acc)[PS], bool comp) {
    const int warp = threadIdx.x >> 5;
    const uint32_t base = tbase + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(col0 + (warp >> 2) * PS);
#pragma unroll
    for (int j = 0; j < PS; j += 8) {
        float v[8];
        tmem_ld8(base + (uint32_t)j, v);
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[j + q] += comp ? v[q] + trunc_comp(v[q]) : v[q];
    }
}

// ------------------------------------------------------------------ coefficients, templates

// coef2d[item] = {r_k c[k][b], c[k][b], r_k dc[k][b]/ds_r}, c[k][b] = dT_r[i,b]/dr_k / (ut s_k[i]):
//   b = 0 vetoed: 1 - t_k;  b = 1 tagged: t_k;  radial rho: (1 - t_k) p_k[rho](s_r) / N^R_k(s_r);
//   pulse shape j: (1 - t_k) q_k[j] / N^P_k, with N_k = sum_{b in the set} q_k[b] U2[k][b];
//   joint grid (rho, j): (1 - t_k) p_k[rho](s_r) q_k[j] / N_k(s_r), one set (the grid).
// A small batch leaves most SMs idle: np CTAs share an item (launch_eval2d), each with the item's short
// FP64 part (the same bits in all of them) and its share of the columns and of the coefficients.
__global__ void __launch_bounds__(512) k_coef2d(Work w, int np) {
    const int item = blockIdx.x / np, part = blockIdx.x % np, tid = threadIdx.x;
    if (w.status[item]) return;
    const Toy& T = w.toys[w.toy_of[item]];
    const int K = T.K, nR = T.n_r2, nP = T.n_p2, b2 = T.b_r2;
    const double* th = w.theta + (size_t)item * w.tstride;
    __shared__ double s_pi[NSL], s_pe[NSL], s_dpe[NSL], s_NR[KMAX], s_dNR[KMAX], s_NP[KMAX];
    __shared__ double s_F[NSL + 2], s_dF[NSL + 2];   // n_r2 < NSL
    if (nR > 0) {
        const double lamA = T.att_len * th[K + 6];
        // the shell integrals at the bin edges and at r_fid, one a thread
        for (int e = tid; e <= nR + 1; e += blockDim.x)
            shell_F(e <= nR ? T.r_fid * e / nR : T.r_fid, T.r_iv, lamA, s_F[e], s_dF[e]);
        __syncthreads();
        const double tot = s_F[nR + 1] - s_F[0], dtot = s_dF[nR + 1] - s_dF[0];
        for (int b = tid; b < nR; b += blockDim.x) {
            const double ra = T.r_fid * b / nR, rb = T.r_fid * (b + 1) / nR;
            s_pi[b] = (rb * rb * rb - ra * ra * ra) / (T.r_fid * T.r_fid * T.r_fid);
            const double p = (s_F[b + 1] - s_F[b]) / tot;
            s_pe[b] = p;
            s_dpe[b] = ((s_dF[b + 1] - s_dF[b]) / tot - p * dtot / tot) * T.att_len;
        }
    }
    __syncthreads();
    // the normalisations: NR, dNR and NP in three warps (three FP64 pipes), eight terms' loads in flight
    if (tid < 96 && (tid & 31) < K) {
        const int k = tid & 31, which = tid >> 5;
        const bool ext = nR > 0 && T.rad_class[k] == BX_RAD_EXTERNAL;
        const double *U = T.U2 + (size_t)k * NSL + b2, *q2 = T.psd2 + (size_t)k * nP;
        const double* pr = which == 1 ? s_dpe : ext ? s_pe : s_pi;
        double v = 0.0;
        if (T.joint2) {   // one set, the grid; its normalisation in NR (and d/ds_r in dNR)
            if (which == 0 || (which == 1 && ext))
                for (int r = 0; r < nR; ++r)
#pragma unroll 8
                    for (int j = 0; j < nP; ++j) v = fma(pr[r], __ldg(q2 + j) * __ldg(U + r * nP + j), v);
        } else if (which < 2) {
            if (which == 0 || ext)
#pragma unroll 8
                for (int r = 0; r < nR; ++r) v = fma(pr[r], __ldg(U + r), v);
        } else {
#pragma unroll 8
            for (int j = 0; j < nP; ++j) v = fma(__ldg(q2 + j), __ldg(U + nR + j), v);
        }
        (which == 0 ? s_NR : which == 1 ? s_dNR : s_NP)[k] = v;
    }
    __syncthreads();
    {   // the class form of the coefficients of T_r (k_trate): alpha[set][k], q[b][class]
        float2* al = w.alpha2d + (size_t)item * 4 * KMAX;
        for (int idx = tid; idx < 4 * KMAX; idx += blockDim.x) {
            const int sset = idx / KMAX, k = idx % KMAX;
            double a = 0.0;
            if (k < K) {
                const double t = T.tag ? T.tag[k] : 0.0, csub = T.tag ? 1.0 - t : 1.0, r = th[k];
                a = sset == 0 ? r * csub : sset == 1 ? r * t : sset == 2 ? (nR > 0 ? r * csub / s_NR[k] : 0.0)
                                                                          : (nP > 0 && !T.joint2 ? r * csub / s_NP[k] : 0.0);
            }
            const float h = (float)a;
            al[idx] = make_float2(h, (float)(a - (double)h));
        }
        float2* qc = w.qcls2d + (size_t)item * NSL * KMAX;
        for (int idx = tid; idx < NSL * KMAX; idx += blockDim.x) {
            const int b = idx / KMAX, c = idx % KMAX;
            double q = 0.0;
            if (b == 0 || (T.has_tag && b == 1)) {
                q = c == 0 ? 1.0 : 0.0;
            } else if (T.joint2) {
                if (b >= b2 && b < b2 + nR * nP && c < T.n_cls[2]) {
                    const int rep = T.cls_rep[2][c], rho = (b - b2) / nP, j = (b - b2) - rho * nP;
                    q = (T.rad_class[rep] == BX_RAD_EXTERNAL ? s_pe[rho] : s_pi[rho]) * T.psd2[(size_t)rep * nP + j];
                }
            } else if (b >= b2 && b < b2 + nR) {
                if (c < T.n_cls[2]) q = T.rad_class[T.cls_rep[2][c]] == BX_RAD_EXTERNAL ? s_pe[b - b2] : s_pi[b - b2];
            } else if (b >= b2 + nR && b < b2 + nR + nP) {
                if (c < T.n_cls[3]) q = T.psd2[(size_t)T.cls_rep[3][c] * nP + (b - b2 - nR)];
            }
            const float h = (float)q;
            qc[idx] = make_float2(h, (float)(q - (double)h));
        }
    }
    __syncthreads();   // alpha and q of this item are in global memory (this block wrote them)
    {   // the class sums W[set, c][i] of every column, their largest values, and from those an upper
        // bound of each slice's T_r: utmax[b] sum_c q[b][c] max_i W[set(b), c][i]
        __shared__ unsigned s_wmax[4 * KMAX];
        __shared__ bool s_last;
        __shared__ int s_off[5];
        if (tid == 0) {
            int o = 0;
            for (int ss = 0; ss < 4; ++ss) {
                s_off[ss] = o;
                o += T.n_cls[ss];
            }
            s_off[4] = o;
        }
        for (int j = tid; j < 4 * KMAX; j += blockDim.x) s_wmax[j] = 0u;
        __syncthreads();
        const float2* alg = w.alpha2d + (size_t)item * 4 * KMAX;
        float2* W = w.wcls2d + (size_t)item * w.ncs2d * w.Npad;
        for (int i0 = (tid & ~31) + part * blockDim.x; i0 < T.N; i0 += np * blockDim.x) {
            const int i = i0 + (tid & 31);
            df sk[KMAX];
#pragma unroll
            for (int k = 0; k < KMAX; ++k)
                sk[k] = k < K && i < T.N ? df{T.shapes32[(size_t)k * T.N + i], T.shapes32l[(size_t)k * T.N + i]}
                                         : df{0.f, 0.f};
            for (int ss = 0; ss < 4; ++ss)
                for (int c = 0; c < T.n_cls[ss]; ++c) {
                    df acc{0.f, 0.f};
#pragma unroll
                    for (int k = 0; k < KMAX; ++k)
                        if (k < K && T.cls_of[ss][k] == c && sk[k].h != 0.f) {
                            const float2 a = alg[ss * KMAX + k];
                            acc = df_add(acc, df_mul(df{a.x, a.y}, sk[k]));
                        }
                    if (i < T.N) W[(size_t)(s_off[ss] + c) * w.Npad + i] = make_float2(acc.h, acc.l);
                    // one atomic a warp: 32 to one address take turns
                    const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(acc.h)));
                    if ((tid & 31) == 0) atomicMax(&s_wmax[s_off[ss] + c], top);
                }
        }
        __syncthreads();
        bool last = true;   // the CTA that finishes the item: it has every part's largest values
        if (np > 1) {
            int2* all = w.prep_part + (size_t)item * PREP_PARTS * (MAX_SETS * MAX_TILES + 1);
            if (tid < 4 * KMAX) all[part * 4 * KMAX + tid].x = (int)s_wmax[tid];
            __threadfence();
            __syncthreads();
            if (tid == 0) s_last = atomicAdd(&w.prep_count[item], 1) == np - 1;
            __syncthreads();
            last = s_last;
            if (last) {
                __threadfence();
                if (tid < 4 * KMAX)
                    for (int q = 0; q < np; ++q)
                        s_wmax[tid] = max(s_wmax[tid], (unsigned)__ldcg(&all[q * 4 * KMAX + tid]).x);
                if (tid == 0) w.prep_count[item] = 0;
                __syncthreads();
            }
        }
        const float2* qc = w.qcls2d + (size_t)item * NSL * KMAX;
        for (int b = tid; last && b < NSL; b += blockDim.x) {
            const int ss = b == 0 ? 0 : (T.has_tag && b == 1) ? 1 : (T.joint2 || b < b2 + nR) ? 2 : 3;
            double bound = 0.0;
            if (b < T.n_sl)
                for (int c = 0; c < T.n_cls[ss]; ++c) {
                    const float2 q = qc[(size_t)b * KMAX + c];
                    bound += fabs((double)q.x + (double)q.y) * (double)__uint_as_float(s_wmax[s_off[ss] + c]);
                }
            // above every |T_r[i,b]| (relative slack for the roundings of the double-float values)
            w.trmax2d[(size_t)item * NSL + b] = __float_as_uint((float)(bound * (double)T.utmax[b] * (1.0 + 1e-5)));
        }
    }
    float* out = w.coef2d + (size_t)item * 4 * KMAX * NSL;
    for (int idx = tid + part * blockDim.x; idx < KMAX * NSL; idx += np * blockDim.x) {
        const int k = idx / NSL, b = idx % NSL;
        double c = 0.0, dc = 0.0, r = 0.0;
        if (k < K) {
            r = th[k];
            const double t = T.tag ? T.tag[k] : 0.0, csub = T.tag ? 1.0 - t : 1.0;
            if (b == 0) c = csub;
            else if (T.has_tag && b == 1) c = t;
            else if (T.joint2) {
                if (b >= b2 && b < b2 + nR * nP) {
                    const int rho = (b - b2) / nP, j = (b - b2) - rho * nP;
                    const bool ext = T.rad_class[k] == BX_RAD_EXTERNAL;
                    const double qj = T.psd2[(size_t)k * nP + j], N = s_NR[k];
                    const double q = (ext ? s_pe[rho] : s_pi[rho]) * qj;
                    c = csub * q / N;
                    if (ext) dc = csub * (s_dpe[rho] * qj * N - q * s_dNR[k]) / (N * N);
                }
            } else if (b >= b2 && b < b2 + nR) {
                const int rho = b - b2;
                const bool ext = T.rad_class[k] == BX_RAD_EXTERNAL;
                const double q = ext ? s_pe[rho] : s_pi[rho], N = s_NR[k];
                c = csub * q / N;
                if (ext) dc = csub * (s_dpe[rho] * N - q * s_dNR[k]) / (N * N);
            } else if (b >= b2 + nR && b < b2 + nR + nP) {
                c = csub * T.psd2[(size_t)k * nP + (b - b2 - nR)] / s_NP[k];
            }
        }
        const double rc = r * c;
        const float rch = (float)rc;
        out[idx] = rch;
        out[KMAX * NSL + idx] = (float)c;
        out[2 * KMAX * NSL + idx] = (float)(r * dc);
        out[3 * KMAX * NSL + idx] = (float)(rc - (double)rch);
    }
}

// T_r tiles of one item: grid = items x tr_kb k-blocks of 32 true-energy columns; thread =
// slice b and a share of the k-block's columns (NSL x TRS threads).
// T_r[i,b] = ut[i,b] sum_c q[b][c] W[set(b), c][i], with the class sums W of k_coef2d, in double-float (split coefficients, shapes and modulation, TwoProduct by
// FMA, TwoSum): ~2^-44 relative instead of the FP32 roundings of every factor and partial sum,
// which all the rows that T_r[i,b] meets in the GEMM would share, so that they would not average
// out over a bin's sum.  It is split in three on one grid per slice (from k_coef2d's upper bound
// of the slice's values), so that the hi parts of every k-block share one grid and their products
// with the forward's hi parts accumulate exactly: TF32 parts (hi to 8 bits, TF32 mid and lo), or
// (BF) BF16 parts in the BF16 tile layout (element (n, c) at (c / 8) NSL 8 + n 8 + c % 8 of each
// part, the first half of the tile).
// TRS threads per slice, each a contiguous share of the k-block's columns (more warps per SM to
// hide the latency of the loads each value waits for).
template <bool BF>
constexpr int TRS = BF ? 2 : 4;
template <bool BF>
__global__ void __launch_bounds__(NSL * TRS<BF>, 2) k_trate(Work w) {
    const int kb = blockIdx.x % w.tr_kb, item = blockIdx.x / w.tr_kb;
    const int b = threadIdx.x % NSL, part = threadIdx.x / NSL;
    if (w.status[item]) return;
    // the toy's fields in registers: the tile stores below could alias them otherwise
    const Toy& T = w.toys[w.toy_of[item]];
    const int N = T.N, n_sl = T.n_sl;
    const int ss = b == 0 ? 0 : (T.has_tag && b == 1) ? 1 : (T.joint2 || b < T.b_r2 + T.n_r2) ? 2 : 3;
    const int nc = T.n_cls[ss];
    int w0 = 0;
    for (int q = 0; q < ss; ++q) w0 += T.n_cls[q];
    const float* __restrict__ ut = T.ut + b;
    const float* __restrict__ utl = T.utl + b;
    df qv[KMAX];
    const float2* qc = w.qcls2d + ((size_t)item * NSL + b) * KMAX;
#pragma unroll
    for (int q = 0; q < KMAX; ++q) {
        const float2 v = q < nc ? qc[q] : make_float2(0.f, 0.f);
        qv[q] = df{v.x, v.y};
    }
    const float2* __restrict__ W = w.wcls2d + ((size_t)item * w.ncs2d + w0) * w.Npad;
    const size_t Npad = w.Npad;
    const Grid g = hi_grid(__uint_as_float(w.trmax2d[(size_t)item * NSL + b]));
    float* __restrict__ tile = w.tr2d + ((size_t)item * w.tr_kb + kb) * TILE3_FLOATS;
    const bool live = b < n_sl;
    auto value = [&](int i) {   // T_r[i, b] as a double-float
        df x{0.f, 0.f};
        if (live && i < N) {
            df acc{0.f, 0.f};
#pragma unroll
            for (int q = 0; q < KMAX; ++q)
                if (q < nc) {
                    const float2 wv = W[(size_t)q * Npad + i];
                    acc = df_add(acc, df_mul(qv[q], df{wv.x, wv.y}));
                }
            x = df_mul(df{ut[(size_t)i * NSL], utl[(size_t)i * NSL]}, acc);
        }
        return x;
    };
    if (BF) {
        uint16_t* t16 = reinterpret_cast<uint16_t*>(tile);
#pragma unroll 1
        for (int c8 = part * (KB / 8 / TRS<BF>); c8 < (part + 1) * (KB / 8 / TRS<BF>); ++c8) {
            uint16_t hv[8], mv[8], lv[8];
#pragma unroll
            for (int q8 = 0; q8 < 8; ++q8) {
                const df x = value(kb * KB + 8 * c8 + q8);
                const float hi = rintf(x.h * g.inv) * g.scale;
                const float r = __fadd_rn(__fsub_rn(x.h, hi), x.l);
                hv[q8] = bf16_rn(hi);
                mv[q8] = bf16_rn(r);
                lv[q8] = bf16_rn(__fsub_rn(r, bf16_val(mv[q8])));
            }
            const int o = c8 * (NSL * 8) + b * 8;
            *reinterpret_cast<uint4*>(t16 + o) = make_uint4(hv[0] | (uint32_t)hv[1] << 16, hv[2] | (uint32_t)hv[3] << 16,
                                                            hv[4] | (uint32_t)hv[5] << 16, hv[6] | (uint32_t)hv[7] << 16);
            *reinterpret_cast<uint4*>(t16 + NSL * KB + o) =
                make_uint4(mv[0] | (uint32_t)mv[1] << 16, mv[2] | (uint32_t)mv[3] << 16, mv[4] | (uint32_t)mv[5] << 16,
                           mv[6] | (uint32_t)mv[7] << 16);
            *reinterpret_cast<uint4*>(t16 + 2 * NSL * KB + o) =
                make_uint4(lv[0] | (uint32_t)lv[1] << 16, lv[2] | (uint32_t)lv[3] << 16, lv[4] | (uint32_t)lv[5] << 16,
                           lv[6] | (uint32_t)lv[7] << 16);
        }
    } else {   // four columns of slice b are one 16-byte row of a core matrix: one store per part
#pragma unroll 1
        for (int c4 = part * (KB / 4 / TRS<BF>); c4 < (part + 1) * (KB / 4 / TRS<BF>); ++c4) {
            float hv[4], mv[4], lv[4];
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4) {
                // x.h - hi is exact: hi is x.h rounded to a grid no finer than ulp(x.h)
                const df x = value(kb * KB + 4 * c4 + q4);
                const float hi = rintf(x.h * g.inv) * g.scale;
                const float r = __fadd_rn(__fsub_rn(x.h, hi), x.l);
                hv[q4] = hi;
                mv[q4] = tf32_rna(r);
                lv[q4] = tf32_rna(__fsub_rn(r, mv[q4]));
            }
            const int o = b_off(b, 4 * c4);
            *reinterpret_cast<float4*>(tile + o) = make_float4(hv[0], hv[1], hv[2], hv[3]);
            *reinterpret_cast<float4*>(tile + NSL * KB + o) = make_float4(mv[0], mv[1], mv[2], mv[3]);
            *reinterpret_cast<float4*>(tile + 2 * NSL * KB + o) = make_float4(lv[0], lv[1], lv[2], lv[3]);
        }
    }
}

// ------------------------------------------------------------------ forward: Y = R T_r

// The two operands are split in three (hi | mid | lo) on grids fixed for the whole contraction:
// A (the response tile) on one grid per row tile, from the tile's largest column amplitude
// times the largest value of the node sum (8 p0 + 5 (p- + p+) <= 8 + 5 Ck2 cosh z, at most 24),
// with a 7-bit hi; B (T_r) on one grid per slice (k_trate) with an 8-bit hi.  Every hi*hi
// product is then an integer below 2^15 times the same power of two for all k-blocks, and a
// row's sum of them over its band (~10^2 columns, their hi parts summing to a few 10^4) stays
// below 2^24 units: region E accumulates them over every k-block exactly, whatever the order or
// rounding of the tensor core's accumulator.  Region S (fresh per k-block) takes the cross
// products hi lo, lo hi, mid mid, hi mid, mid hi (smallest first), ~2^-7 of E, and is drained
// per k-block into FP32 registers, where the rounding acts on values that small.
// BF16 parts carry 8 bits where TF32 ones carry 11: on A's coarse grid (the remainder after hi
// reaches 0.19 of the tile's largest amplitude) mid and lo would leave 7e-7 of it, so the BF16
// variant splits A in four (hi | mid | lo | lo2) and S takes three more products (lo2 hi, mid lo,
// lo mid): what is left out is ~1e-8 of the row's terms or less.
constexpr float RESP_SHAPE_MAX = 24.0f;

template <bool BF>
__device__ __forceinline__ void umma_part(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
    if (BF) umma_bf16(d, ad, bd, idesc, acc);
    else umma_tf32(d, ad, bd, idesc, acc);
}

// One k-block of 32 columns: region S (fresh) <- the five (BF16: eight) cross products, region
// E <- hi hi (accumulated over the k-blocks, fresh at the first).  TF32 parts: 4 instructions of
// K = 8 per part pair; BF16 parts (BF): 2 of K = 16.  Either way an instruction spans 32 bytes of K, two
// core matrices, so the descriptors step alike.
template <bool BF>
__device__ __forceinline__ void mma_kblock3(uint32_t dS, uint32_t dE, const void* A3, const void* B3, bool first) {
    constexpr uint32_t idesc = BF ? umma_idesc_bf16(TM, NSL) : umma_idesc_tf32(TM, NSL);
    constexpr uint32_t esz = BF ? 2u : 4u;
    constexpr int NQ = KB * (int)esz / 32;
    const uint32_t a0 = smem_u32(A3), b0 = smem_u32(B3);
    const uint32_t a[4] = {a0, a0 + A_FLOATS * esz, a0 + 2 * A_FLOATS * esz, a0 + 3 * A_FLOATS * esz};
    const uint32_t bb[3] = {b0, b0 + NSL * KB * esz, b0 + 2 * NSL * KB * esz};
    // (A part, B part) of the products into S, smallest first
    constexpr int pa5[5] = {0, 2, 1, 0, 1}, pb5[5] = {2, 0, 1, 1, 0};
    constexpr int pa8[8] = {3, 1, 2, 0, 2, 1, 0, 1}, pb8[8] = {0, 2, 1, 2, 0, 1, 1, 0};
    constexpr int NP = BF ? 8 : 5;
    uint32_t acc = 0u;
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int ap = BF ? pa8[p] : pa5[p], bp = BF ? pb8[p] : pb5[p];
            umma_part<BF>(dS, umma_desc(a[ap] + q * 2 * (TM * 16), TM * 16, 128),
                          umma_desc(bb[bp] + q * 2 * (NSL * 16), NSL * 16, 128), idesc, acc);
            acc = 1u;
        }
#pragma unroll
    for (int q = 0; q < NQ; ++q)
        umma_part<BF>(dE, umma_desc(a[0] + q * 2 * (TM * 16), TM * 16, 128),
                      umma_desc(bb[0] + q * 2 * (NSL * 16), NSL * 16, 128), idesc, (first && q == 0) ? 0u : 1u);
}

struct PipeF {
    uint64_t mma_bar[2];
    uint64_t b_bar[2];
    uint32_t tmem;
    int abort;
    int committed;
    unsigned amax;   // largest column amplitude of the tile (FP32 bits)
};

__device__ __forceinline__ bool drain_copies3(PipeF& pp, int waited, int issued) {
    bool ok = true;
    for (int j = waited; j < issued; ++j) ok &= mbar_wait(&pp.b_bar[j & 1], (j >> 1) & 1, CLEANUP_NS);
    return ok;
}

// TMEM columns of this thread's 32 values in region `col0` (warp q: lanes 32 (q % 4) + lane,
// columns 32 (q / 4) .. + 31 of the region)
__device__ __forceinline__ uint32_t fwd_tcols(uint32_t tbase, int col0) {
    const int warp = threadIdx.x >> 5;
    return tbase + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(col0 + (warp >> 2) * (NSL / 4));
}

// Add region S of TMEM buffer s (columns s NSL .. + NSL - 1) into this thread's 32 values.
__device__ __forceinline__ void drainS(uint32_t tbase, int s, float (&acc)[NSL / 4]) {
    const uint32_t base = fwd_tcols(tbase, s * NSL);
#pragma unroll
    for (int j = 0; j < NSL / 4; j += 8) {
        float v[8];
        tmem_ld8(base + (uint32_t)j, v);
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[j + q] += v[q];
    }
}

// Unit = (row tile, item), 512 threads: thread = (row r, quarter h of the k-block's columns).
// Two stages: while the tensor core multiplies k-block j, the CUDA cores generate j + 1; the
// cross products of k-block j are drained when j + 2 starts; region E (columns 2 NSL ..) is read
// once at the end.  Y = E + S goes out as the pile-up GEMM's TF32 hi | lo tile plus the FP32
// remainder.
template <bool BF>
__global__ void __launch_bounds__(TF + 32, 1) k_fwd2d(Work w) {
    extern __shared__ unsigned char smem_raw[];
    float* A3 = align128(smem_raw);            // [2][3][A_FLOATS]
    float* B3 = A3 + 6 * A_FLOATS;             // [2][TILE3_FLOATS]
    __shared__ PipeF pp;
    __shared__ uint64_t a_bar[2], p_bar[2];    // A tile written (TF arrivals), column constants staged (32)
    __shared__ float4 sCf[2][KB];
    __shared__ ColG sCg[2][KB];
    __shared__ float sAl[2][KB];
    const int tile = blockIdx.x % w.max_tiles, item = blockIdx.x / w.max_tiles, tid = threadIdx.x;
    const Toy& T = w.toys[w.toy_of[item]];
    if (tile >= T.n_tiles || w.status[item]) return;
    const bool gen = tid < TF;                 // warps 0-15 generate A; warp 16 stages, copies and multiplies
    const int m0 = tile * TM, r = tid & (TM - 1), h = (tid >> 7) & 3, warp = tid >> 5, lane = tid & 31;
    const int2 cr = tile_range(w, item, 0, tile);   // one quenching group
    const int kb0 = cr.x < cr.y ? cr.x / KB : 0;
    const int nblk = cr.x < cr.y ? (cr.y - 1) / KB + 1 - kb0 : 0;
    const int N = T.N;
    const float* trg = w.tr2d + ((size_t)item * w.tr_kb + kb0) * TILE3_FLOATS;
    const float4* colf = w.colf + (size_t)item * w.Npad;
    const ColG* colg = w.colg + (size_t)item * w.Npad;
    const float* colal = w.colAl + (size_t)item * w.Npad;
    volatile int* abort_flag = &pp.abort;
    // Y rows of this thread: lane group (warp % 4) of the tile, slices 32 (warp / 4) ..
    const int row = m0 + (warp & 3) * 32 + lane;
    float* ytile = w.y2d + ((size_t)item * w.row_kb + row / KB) * YTILE_FLOATS;
    const int b0 = ((warp >> 2) & 3) * (NSL / 4);
    auto store_y = [&](int j, float y, float yl) {   // y + yl (|yl| <= ulp(y) / 2)
        const int o = b_off(b0 + j, row % KB);
        const float hh = tf32_rna(y), ll = tf32_rna(__fsub_rn(y, hh));
        ytile[o] = hh;
        ytile[NSL * KB + o] = ll;
        ytile[2 * NSL * KB + o] = __fadd_rn(__fsub_rn(__fsub_rn(y, hh), ll), yl);
    };
    auto stage = [&](int it) {   // warp 16: the column constants of k-block it into buffer it & 1
        const int i = (kb0 + it) * KB + lane, sb = it & 1;
        const bool in = i < N;
        sCf[sb][lane] = in ? colf[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        sCg[sb][lane] = in ? colg[i] : ColG{0.f, 0.f, 0.f, 0.f};
        sAl[sb][lane] = in ? colal[i] : 0.f;
        mbar_arrive(&p_bar[sb]);
    };
    float acc[NSL / 4];
#pragma unroll
    for (int j = 0; j < NSL / 4; ++j) acc[j] = 0.f;
    bool stored = false;
    if (nblk > 0) {
        if (tid == 0) {
            mbar_init(&pp.mma_bar[0], 1);
            mbar_init(&pp.mma_bar[1], 1);
            mbar_init(&pp.b_bar[0], 1);
            mbar_init(&pp.b_bar[1], 1);
            mbar_init(&a_bar[0], TF);
            mbar_init(&a_bar[1], TF);
            mbar_init(&p_bar[0], 32);
            mbar_init(&p_bar[1], 32);
            pp.abort = 0;
            pp.amax = 0u;
            fence_mbar_init();
        }
        if (warp == 0) {
            tmem_alloc(&pp.tmem, 4 * NSL);
            tmem_relinquish();
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        const uint32_t tbase = pp.tmem;
        if (gen) {   // the A grid of the tile: its largest column amplitude (A + |al|) times RESP_SHAPE_MAX
            float am = 0.f;
            for (int i = cr.x + tid; i < min(cr.y, N); i += TF) am = fmaxf(am, colg[i].A + fabsf(colal[i]));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
            if (lane == 0 && am > 0.f) atomicMax(&pp.amax, __float_as_uint(am));
        }
        __syncthreads();
        const Grid gA = hi_grid7(__uint_as_float(pp.amax) * RESP_SHAPE_MAX);
        if (gen) {
            const float mf = (float)(m0 + r);
            const bool row_ok = m0 + r < T.M;
            for (int it = 0; it < nblk; ++it) {
                const int s = it & 1;
                // the column constants of k-block it; k-block it - 2 used buffer s: its MMAs must be
                // done before A and region S of s are reused
                bool ok = mbar_wait(&p_bar[s], (it >> 1) & 1, w.watchdog_ns);
                if (it >= 2) ok = ok && mbar_wait(&pp.mma_bar[s], ((it - 2) >> 1) & 1, w.watchdog_ns);
                if (!ok) atomicOr(&pp.abort, 1);
                // leave warp-uniformly: region S is read by warp-collective tcgen05.ld
                if (__any_sync(0xffffffffu, !ok || *abort_flag != 0)) break;
                tc_fence_after();
                if (it >= 2) drainS(tbase, s, acc);
                const int ibase = (kb0 + it) * KB;
                float x[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int c = 8 * h + q;
                    x[q] = (row_ok && ibase + c < N) ? resp_amp32(mf, sCf[s][c], sCg[s][c], sAl[s][c]) : 0.f;
                }
                float* As = A3 + s * 3 * A_FLOATS;
                if (BF) {   // the thread's 8 columns are one 16-byte row of a BF16 core matrix
                    uint16_t hv[8], mv[8], lv[8], ev[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) split4_bf16(x[q], gA, hv[q], mv[q], lv[q], ev[q]);
                    uint16_t* A16 = reinterpret_cast<uint16_t*>(As);
                    const int o = h * (TM * 8) + r * 8;
                    *reinterpret_cast<uint4*>(A16 + o) =
                        make_uint4(hv[0] | (uint32_t)hv[1] << 16, hv[2] | (uint32_t)hv[3] << 16,
                                   hv[4] | (uint32_t)hv[5] << 16, hv[6] | (uint32_t)hv[7] << 16);
                    *reinterpret_cast<uint4*>(A16 + A_FLOATS + o) =
                        make_uint4(mv[0] | (uint32_t)mv[1] << 16, mv[2] | (uint32_t)mv[3] << 16,
                                   mv[4] | (uint32_t)mv[5] << 16, mv[6] | (uint32_t)mv[7] << 16);
                    *reinterpret_cast<uint4*>(A16 + 2 * A_FLOATS + o) =
                        make_uint4(lv[0] | (uint32_t)lv[1] << 16, lv[2] | (uint32_t)lv[3] << 16,
                                   lv[4] | (uint32_t)lv[5] << 16, lv[6] | (uint32_t)lv[7] << 16);
                    *reinterpret_cast<uint4*>(A16 + 3 * A_FLOATS + o) =
                        make_uint4(ev[0] | (uint32_t)ev[1] << 16, ev[2] | (uint32_t)ev[3] << 16,
                                   ev[4] | (uint32_t)ev[5] << 16, ev[6] | (uint32_t)ev[7] << 16);
                } else {
#pragma unroll
                    for (int c4 = 0; c4 < 2; ++c4) {
                        float4 vh, vm, vl;
                        split3(x[4 * c4 + 0], gA, vh.x, vm.x, vl.x);
                        split3(x[4 * c4 + 1], gA, vh.y, vm.y, vl.y);
                        split3(x[4 * c4 + 2], gA, vh.z, vm.z, vl.z);
                        split3(x[4 * c4 + 3], gA, vh.w, vm.w, vl.w);
                        const int o = a_off(r, 8 * h + 4 * c4);
                        *reinterpret_cast<float4*>(As + o) = vh;
                        *reinterpret_cast<float4*>(As + A_FLOATS + o) = vm;
                        *reinterpret_cast<float4*>(As + 2 * A_FLOATS + o) = vl;
                    }
                }
                fence_proxy_async_smem();   // the A tile and the drained region S, then the arrival
                tc_fence_before();
                mbar_arrive(&a_bar[s]);
            }
        } else {   // warp 16
            int issued = 0, waited = 0, committed = 0;   // lane 0's bookkeeping
            constexpr uint32_t bytes = BF ? TILE3_BYTES / 2 : TILE3_BYTES;   // TF32 parts, or BF16 (the first half)
            stage(0);
            if (lane == 0) {
                mbar_arrive_expect_tx(&pp.b_bar[0], bytes);
                bulk_g2s(B3, trg, bytes, &pp.b_bar[0]);
                issued = 1;
            }
            for (int it = 0; it < nblk; ++it) {
                const int s = it & 1, s1 = s ^ 1;
                bool ok = true;
                if (it + 1 < nblk) {
                    // buffer s1 of the column constants: the generators are done with k-block it - 1
                    if (it >= 1) ok = mbar_wait(&a_bar[s1], ((it - 1) >> 1) & 1, w.watchdog_ns);
                    ok = __all_sync(0xffffffffu, ok);   // the 32 arrivals on p_bar come together or not at all
                    if (ok) stage(it + 1);
                }
                if (lane == 0 && ok) {
                    if (it + 1 < nblk) {   // B tile it + 1 into buffer s1, once MMA it - 1 has read it
                        if (it >= 1) ok = mbar_wait(&pp.mma_bar[s1], ((it - 1) >> 1) & 1, w.watchdog_ns);
                        if (ok) {
                            mbar_arrive_expect_tx(&pp.b_bar[s1], bytes);
                            bulk_g2s(B3 + s1 * TILE3_FLOATS, trg + (size_t)(it + 1) * TILE3_FLOATS, bytes, &pp.b_bar[s1]);
                            ++issued;
                        }
                    }
                    ok = ok && mbar_wait(&a_bar[s], (it >> 1) & 1, w.watchdog_ns);
                    ok = ok && mbar_wait(&pp.b_bar[s], (it >> 1) & 1, w.watchdog_ns);
                    if (ok) {
                        ++waited;
                        tc_fence_after();
                        mma_kblock3<BF>(tbase + (uint32_t)(s * NSL), tbase + (uint32_t)(2 * NSL), A3 + s * 3 * A_FLOATS,
                                        B3 + s * TILE3_FLOATS, it == 0);
                        umma_commit(&pp.mma_bar[s]);
                        ++committed;
                    }
                }
                if (!ok) atomicOr(&pp.abort, 1);
                if (__any_sync(0xffffffffu, !ok || *abort_flag != 0)) break;
            }
            if (lane == 0) {
                if (!drain_copies3(pp, waited, issued)) atomicOr(&pp.abort, 1);
                pp.committed = committed;
            }
        }
        __syncthreads();
        const int nc = pp.committed;
        const unsigned long long budget = w.watchdog_ns > CLEANUP_NS ? w.watchdog_ns : CLEANUP_NS;
        if (gen) {
            bool done = true;
            // the last two k-blocks (one per buffer) are still to be waited for; the commit of the
            // last one also covers every earlier MMA into region E
            for (int j = (nc >= 2 ? nc - 2 : 0); j < nc; ++j) done &= mbar_wait(&pp.mma_bar[j & 1], (j >> 1) & 1, budget);
            tc_fence_after();
            const bool ok = __all_sync(0xffffffffu, !pp.abort && done && nc == nblk);   // warp-uniform: tcgen05.ld
            if (ok) {
                for (int j = (nc >= 2 ? nc - 2 : 0); j < nc; ++j) drainS(tbase, j & 1, acc);
                const bool keep = row < T.M;
                const uint32_t eb = fwd_tcols(tbase, 2 * NSL);
#pragma unroll
                for (int j = 0; j < NSL / 4; j += 8) {
                    float v[8];
                    tmem_ld8(eb + (uint32_t)j, v);
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const df y = df_two_sum(v[q], acc[j + q]);   // E exact, S the small part
                        store_y(j + q, keep ? y.h : 0.f, keep ? y.l : 0.f);
                    }
                }
                stored = true;
            }
            if (!ok && tid == 0) atomicOr(w.err, ERR_TIMEOUT);
        }
        tc_fence_before();
        __syncthreads();
        if (warp == 0) tmem_dealloc(tbase, 4 * NSL);
    }
    if (gen && !stored)   // a tile without columns (Y = 0), or a failed wait
#pragma unroll
        for (int j = 0; j < NSL / 4; ++j) store_y(j, 0.f, 0.f);
}

// ------------------------------------------------------------------ pile-up + -lnL

// Window tile t: rows m = m_lo + 128 t + 127 - l.  A[l, c] = g[m - m'] (input row m' = 32 kb + c, a
// Toeplitz table), B = Y tiles; k-block it + 1 is multiplied into the other accumulator while it is
// drained; D = sum_d g[d] Y[m - d, b].  Epilogue: mu, the Baker-Cousins terms (cancellation-free FP32
// form where mu/2 <= n <= 2 mu, double-float otherwise; compensated sums), w = 1 - n/mu.  -lnL and the eps
// derivative are sums over a thread's 32 slices of a row, then over the rows: their last bits follow that
// order (chains of 64 slices, shared by two threads, cost 8 us of one item's 68 and 47 of 256 items' 624).
__global__ void __launch_bounds__(TP, 2) k_pile2d(Work w, int want_mu) {
    extern __shared__ unsigned char smem_raw[];
    float* Ahi = align128(smem_raw);   // Toeplitz table of g, TP_KB k-blocks
    float* Alo = Ahi + TP_FLOATS;
    float* Bt = Alo + TP_FLOATS;       // [2][TILE_FLOATS]
    __shared__ Pipe pp;
    __shared__ double red[3][TP / 32];
    const int t = blockIdx.x % w.win_tiles, item = blockIdx.x / w.win_tiles, tid = threadIdx.x;
    const Toy& T = w.toys[w.toy_of[item]];
    const int nw = T.nw, M = T.M, L = T.L;
    if (t * TM >= nw || w.status[item]) {
        if (tid == 0) {
            w.nll2d[((size_t)item * MAX_TILES + t) * 2] = 0.0;
            w.nll2d[((size_t)item * MAX_TILES + t) * 2 + 1] = 0.0;
            w.geps2d[(size_t)item * MAX_TILES + t] = 0.0;
        }
        return;
    }
    const double* th = w.theta + (size_t)item * w.tstride;
    const double eps = th[T.K + 5];
    const int warp = tid >> 5;
    const int mw0 = T.m_lo + t * TM;                       // first output row
    const int in_lo = max(0, mw0 - (L - 1)), in_hi = min(M, mw0 + TM);
    const int kb0 = in_lo / KB, nblk = (in_hi + KB - 1) / KB - kb0;
    const float* yg = w.y2d + (size_t)item * w.row_kb * YTILE_FLOATS;
    float pu[PS];
#pragma unroll
    for (int j = 0; j < PS; ++j) pu[j] = 0.f;
    if (tid == 0) {
        mbar_init(&pp.mma_bar[0], 1);
        mbar_init(&pp.mma_bar[1], 1);
        mbar_init(&pp.b_bar[0], 1);
        mbar_init(&pp.b_bar[1], 1);
        pp.abort = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(&pp.tmem, 2 * NSL);   // two accumulators
        tmem_relinquish();
    }
    int issued = 0, waited = 0, committed = 0;
    auto copy_b = [&](int it) {   // thread 0: k-block it's B tile into its stage
        mbar_arrive_expect_tx(&pp.b_bar[it & 1], TILE_BYTES);
        bulk_g2s(Bt + (it & 1) * TILE_FLOATS, yg + (size_t)(kb0 + it) * YTILE_FLOATS, TILE_BYTES, &pp.b_bar[it & 1]);
        ++issued;
    };
    if (tid == 0)
        for (int it = 0; it < min(nblk, 2); ++it) copy_b(it);
    // the table from k-block it on: d = m - m' = mw0 + 127 - l - 32 (kb0 + it) - c
    auto table = [&](int it) {
        toeplitz_table(Ahi, Alo, T.g32, L, mw0 + TM - 1 - (kb0 + it) * KB, -1);
        fence_proxy_async_smem();
        tc_fence_before();
        __syncthreads();
    };
    table(0);
    tc_fence_after();
    const uint32_t tbase = pp.tmem;
    auto multiply = [&](int it) {   // thread 0; accumulator it & 1 is drained
        tc_fence_after();
        if (!mbar_wait(&pp.b_bar[it & 1], (it >> 1) & 1, w.watchdog_ns)) {
            atomicOr(&pp.abort, 1);
        } else {
            ++waited;
            const int o = it % TP_KB * (KB / 4) * 32;
            mma_kblock(tbase + (uint32_t)((it & 1) * NSL), Ahi + o, Alo + o, Bt + (it & 1) * TILE_FLOATS, false);
            umma_commit(&pp.mma_bar[it & 1]);
            ++committed;
        }
    };
    if (tid == 0 && nblk > 0) multiply(0);
    for (int it = 0; it < nblk; ++it) {
        const bool next = it + 1 < nblk, fresh = next && (it + 1) % TP_KB == 0;   // fresh: a new table first
        if (tid == 0 && next && !fresh && !pp.abort) multiply(it + 1);
        __syncwarp();
        const bool got = __all_sync(0xffffffffu, mbar_wait(&pp.mma_bar[it & 1], (it >> 1) & 1, w.watchdog_ns));
        tc_fence_after();
        if (!got) {
            atomicOr(&pp.abort, 1);
        } else {
            if (tid == 0 && it + 2 < nblk) copy_b(it + 2);   // the stage k-block it has left
            __syncwarp();
            drain_add(tbase, (it & 1) * NSL, pu, true);      // summed in registers
        }
        tc_fence_before();
        // one vote for the block: a thread ahead of the others may set the flag again before they read it
        if (__syncthreads_or(pp.abort)) break;
        if (fresh) {
            table(it + 1);
            if (tid == 0) multiply(it + 1);
        }
    }
    if (tid == 0) {
        if (!drain_copies(pp, waited, issued)) atomicOr(&pp.abort, 1);
        pp.committed = committed;
    }
    __syncthreads();
    const int nc = pp.committed;
    bool done = true;
    if (nc > 0)
        done = mbar_wait(&pp.mma_bar[(nc - 1) & 1], ((nc - 1) >> 1) & 1,
                         w.watchdog_ns > CLEANUP_NS ? w.watchdog_ns : CLEANUP_NS);
    tc_fence_after();
    const bool ok = !pp.abort && done && nc == nblk;
    if (!ok && tid == 0) atomicOr(w.err, ERR_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tbase, 2 * NSL);

    // epilogue: row of this thread and its 64 slices; the pile-up sums go through the idle
    // operand buffers (thread-private, every copy and MMA has completed) so that the loop
    // below may index them
    float* pus = Ahi;
    static_assert(2 * TP_FLOATS + 2 * TILE_FLOATS >= PS * TP, "the pile-up sums in the operand buffers");
#pragma unroll
    for (int q = 0; q < PS; ++q) pus[q * TP + tid] = pu[q];
    const int row = mw0 + TM - 1 - ((warp & 3) * 32 + (tid & 31)), j = row - T.m_lo;
    const int b0 = (warp >> 2) * (PS);
    // Per bin in FP32 with double-float where it matters: mu = (1 - eps) Y + eps (g * Y) and
    // n - mu carry ~2^-44 relative error, the Baker-Cousins term is formed without
    // cancellation (log1p_minus_x32 where mu/2 <= n <= 2 mu, bc_term_far in double-float
    // beyond), and summed compensated.
    const float c1h = (float)(1.0 - eps), c1l = (float)((1.0 - eps) - (double)c1h);
    const float c2h = (float)eps, c2l = (float)(eps - (double)c2h);
    Sum32 acc, gacc;
    double acc64 = 0.0;   // terms taken in FP64
    int dom = 0;
    const bool live = ok && row < M;   // j < nw
    float* wtile = (j / KB < w.win_kb) ? w.w2d + ((size_t)item * w.win_kb + j / KB) * TILE_FLOATS : nullptr;
    const float* ytile = yg + (size_t)(row / KB) * YTILE_FLOATS;
    const float2* cnt = T.cnt32;
    const int n_sl = T.n_sl;
#pragma unroll 4
    for (int q = 0; q < PS; ++q) {
        const int b = b0 + q;
        float wb = 0.f;
        if (live && b < n_sl) {
            const int o = b_off(b, row % KB);
            // Y = yh + yl (the pair the GEMM used) + the FP32 remainder, as a double-float
            const float yh = __ldg(ytile + o), yl = __fadd_rn(__ldg(ytile + NSL * KB + o), __ldg(ytile + 2 * NSL * KB + o));
            const float pq = pus[q * TP + tid];
            // mu as a double-float
            float p1 = __fmul_rn(c1h, yh), e1 = fmaf(c1h, yh, -p1);
            e1 = fmaf(c1h, yl, fmaf(c1l, yh, e1));
            float p2 = __fmul_rn(c2h, pq), e2 = fmaf(c2h, pq, -p2);
            e2 = fmaf(c2l, pq, e2);
            float sh = __fadd_rn(p1, p2), bb = __fsub_rn(sh, p1);
            float sl = __fadd_rn(__fsub_rn(p1, __fsub_rn(sh, bb)), __fsub_rn(p2, bb));
            sl = __fadd_rn(sl, __fadd_rn(e1, e2));
            const float muh = __fadd_rn(sh, sl), mul = __fsub_rn(sl, __fsub_rn(muh, sh));
            const float2 n = __ldg(cnt + (size_t)b * nw + j);
            float term, wf = 1.f;
            if (n.x == 0.f) {
                term = muh;
            } else if (!(muh > 0.f) || !isfinite(muh)) {
                dom = 1;
                term = 0.f;
            } else {
                // d = n - mu
                const float dh = __fsub_rn(n.x, muh), b2 = __fsub_rn(dh, n.x);
                const float dl = __fadd_rn(__fsub_rn(n.x, __fsub_rn(dh, b2)), __fsub_rn(-muh, b2));
                const float d = __fadd_rn(dh, __fadd_rn(dl, __fsub_rn(n.y, mul)));
                const float x = d / muh;
                if (x >= BC_XLO && x <= BC_XHI) {
                    term = fmaf(n.x, log1p_minus_x32(x), d * x);
                    wf = -x;
                } else {   // n < mu/2 or n > 2 mu (bins with few counts): double-float
                    df t;
                    if (bc_term_far(df{n.x, n.y}, df{muh, mul}, t, wf)) {
                        term = t.h;
                        acc.c = __fadd_rn(acc.c, t.l);
                    } else {   // n/mu beyond [1e-30, 1e30]: FP64
                        const double mud = (double)muh + (double)mul, nd = T.cnt[(size_t)b * nw + j];
                        const double xd = (nd - mud) / mud;
                        acc64 += (mud - nd) + nd * log1p(xd);
                        term = 0.f;
                        wf = (float)(-xd);
                    }
                }
            }
            acc.add(term);
            gacc.add(wf * __fsub_rn(pq, __fadd_rn(yh, yl)));
            wb = wf;
            if (want_mu) w.mu[(size_t)item * w.nbmax + (size_t)b * nw + j] = (double)muh + (double)mul;
        }
        if (wtile) tile_put(wtile, b, j % KB, wb);
    }
    if (dom) w.status[item] = BX_EDOMAIN;
    // block sums in FP64
    Neu nacc{(double)acc.s, (double)acc.c};
    neu_add(nacc, acc64);
    double geps = (double)gacc.s + (double)gacc.c;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Neu other{__shfl_xor_sync(0xffffffffu, nacc.s, o), __shfl_xor_sync(0xffffffffu, nacc.c, o)};
        nacc = neu_merge(nacc, other);
        geps += __shfl_xor_sync(0xffffffffu, geps, o);
    }
    if ((tid & 31) == 31) {   // the warp's first row; the warps in the order of their rows
        red[0][warp ^ 3] = nacc.s;
        red[1][warp ^ 3] = nacc.c;
        red[2][warp ^ 3] = geps;
    }
    __syncthreads();
    if (tid == 0) {
        Neu tot{0.0, 0.0};
        double ge = 0.0;
        for (int q = 0; q < TP / 32; ++q) {
            tot = neu_merge(tot, Neu{red[0][q], red[1][q]});
            ge += red[2][q];
        }
        w.nll2d[((size_t)item * MAX_TILES + t) * 2] = tot.s;
        w.nll2d[((size_t)item * MAX_TILES + t) * 2 + 1] = tot.c;
        w.geps2d[(size_t)item * MAX_TILES + t] = ge;
    }
}

// ------------------------------------------------------------------ adjoint of Eq. 2

// Output rows m = 128 t + 127 - l over the whole axis; A[l, c] = g[(m_lo + j) - m] with window row
// j = 32 kb + c (a Toeplitz table; the w tiles hold zeros beyond the window), B = w tiles;
// Wt = (1 - eps) w + eps D, stored as the adjoint's B tiles.
__global__ void __launch_bounds__(TP, 2) k_corr2d(Work w) {
    extern __shared__ unsigned char smem_raw[];
    float* Ahi = align128(smem_raw);   // Toeplitz table of g, TP_KB k-blocks
    float* Alo = Ahi + TP_FLOATS;
    float* Bt = Alo + TP_FLOATS;       // [2][TILE_FLOATS]
    __shared__ Pipe pp;
    const int t = blockIdx.x % w.max_tiles, item = blockIdx.x / w.max_tiles, tid = threadIdx.x;
    const Toy& T = w.toys[w.toy_of[item]];
    if (t >= T.n_tiles || w.status[item]) return;
    const int nw = T.nw, M = T.M, L = T.L, m_lo = T.m_lo;
    const double eps = w.theta[(size_t)item * w.tstride + T.K + 5];
    const int warp = tid >> 5;
    const int m0 = t * TM;
    const int j_lo = max(0, m0 - m_lo), j_hi = min(nw, m0 + TM - 1 - m_lo + L);
    const int kb0 = j_lo / KB, nblk = j_hi > j_lo ? (j_hi + KB - 1) / KB - kb0 : 0;
    const float* wg = w.w2d + (size_t)item * w.win_kb * TILE_FLOATS;
    float acc[PS];
#pragma unroll
    for (int q = 0; q < PS; ++q) acc[q] = 0.f;
    bool ok = true;
    if (nblk > 0) {
        if (tid == 0) {
            mbar_init(&pp.mma_bar[0], 1);
            mbar_init(&pp.mma_bar[1], 1);
            mbar_init(&pp.b_bar[0], 1);
            mbar_init(&pp.b_bar[1], 1);
            pp.abort = 0;
            fence_mbar_init();
        }
        if (warp == 0) {
            tmem_alloc(&pp.tmem, NSL);
            tmem_relinquish();
        }
        int issued = 0, waited = 0, committed = 0;
        auto copy_b = [&](int it) {   // thread 0: k-block it's B tile into its stage
            mbar_arrive_expect_tx(&pp.b_bar[it & 1], TILE_BYTES);
            bulk_g2s(Bt + (it & 1) * TILE_FLOATS, wg + (size_t)(kb0 + it) * TILE_FLOATS, TILE_BYTES, &pp.b_bar[it & 1]);
            ++issued;
        };
        if (tid == 0)
            for (int it = 0; it < min(nblk, 2); ++it) copy_b(it);
        uint32_t tbase = 0;
        for (int c0 = 0; c0 < nblk; c0 += TP_KB) {
            // every MMA on the previous table has completed before it is overwritten
            bool got = true;
            if (c0 > 0) got = mbar_wait(&pp.mma_bar[(c0 - 1) & 1], ((c0 - 1) >> 1) & 1, w.watchdog_ns);
            if (!got) atomicOr(&pp.abort, 1);
            // d = m_lo + j - m = m_lo + 32 (kb0 + it) + c - m0 - 127 + l
            if (got) toeplitz_table(Ahi, Alo, T.g32, L, m_lo + (kb0 + c0) * KB - m0 - (TM - 1), 1);
            fence_proxy_async_smem();
            tc_fence_before();
            __syncthreads();
            tc_fence_after();
            tbase = pp.tmem;
            if (tid == 0 && !pp.abort) {
                for (int it = c0; it < min(nblk, c0 + TP_KB); ++it) {
                    if (!mbar_wait(&pp.b_bar[it & 1], (it >> 1) & 1, w.watchdog_ns)) {
                        atomicOr(&pp.abort, 1);
                        break;
                    }
                    ++waited;
                    const int o = (it - c0) * (KB / 4) * 32;
                    mma_kblock(tbase, Ahi + o, Alo + o, Bt + (it & 1) * TILE_FLOATS, it > 0);
                    umma_commit(&pp.mma_bar[it & 1]);
                    ++committed;
                    if (it > 0 && it + 1 < nblk) {   // refill the stage that k-block it - 1 leaves
                        if (!mbar_wait(&pp.mma_bar[(it - 1) & 1], ((it - 1) >> 1) & 1, w.watchdog_ns)) {
                            atomicOr(&pp.abort, 1);
                            break;
                        }
                        copy_b(it + 1);
                    }
                }
            }
            if (__syncthreads_or(pp.abort)) break;   // one vote for the block, as in k_pile2d
        }
        if (tid == 0) {
            if (!drain_copies(pp, waited, issued)) atomicOr(&pp.abort, 1);
            pp.committed = committed;
        }
        __syncthreads();
        const int nc = pp.committed;
        bool done = true;
        if (nc > 0)
            done = mbar_wait(&pp.mma_bar[(nc - 1) & 1], ((nc - 1) >> 1) & 1,
                             w.watchdog_ns > CLEANUP_NS ? w.watchdog_ns : CLEANUP_NS);
        tc_fence_after();
        ok = __all_sync(0xffffffffu, !pp.abort && done && nc == nblk);
        if (ok) drain_add(tbase, 0, acc, false);
        else if (tid == 0) atomicOr(w.err, ERR_TIMEOUT);
        tc_fence_before();
        __syncthreads();
        if (warp == 0) tmem_dealloc(tbase, NSL);
    }
    // The epilogue takes four rows of one slice a thread, a warp 32 slices of the same rows: the tiles hold
    // four rows of a slice side by side, so the warp's stores are whole lines (one row a lane touched eight
    // half-used sectors per access; 256 points: 300 -> 214 us).  The sums change hands through the operand
    // buffers, which are no longer needed, slice b's rows at b PITCH.  (k_pile2d keeps a row a lane: there
    // neighbouring energies take the same branch of the bin's term, and slices of one row do not: 633 us
    // of 256 points against 672.)
    float* ex = Ahi;
    static_assert(2 * TP_FLOATS + 2 * TILE_FLOATS >= NSL * PITCH, "the sums in the operand buffers");
    {
        const int l = (warp & 3) * 32 + (tid & 31), s0 = (warp >> 2) * PS;
#pragma unroll
        for (int q = 0; q < PS; ++q) ex[(s0 + q) * PITCH + TM - 1 - l] = acc[q];
    }
    __syncthreads();
    const float e = (float)eps, ome = (float)(1.0 - eps);
    const int n_sl = T.n_sl, lane = tid & 31;
    for (int step = warp; step < TM / 4 * (NSL / 32); step += TP / 32) {
        const int r0 = step % (TM / 4) * 4, b = step / (TM / 4) * 32 + lane;
        const int row0 = m0 + r0, j0 = row0 - m_lo;
        const float4 a4 = *reinterpret_cast<const float4*>(ex + b * PITCH + r0);
        const float av[4] = {a4.x, a4.y, a4.z, a4.w};
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + u;
            v[u] = 0.f;
            if (ok && row0 + u < M && b < n_sl) {
                v[u] = e * av[u];
                if (j >= 0 && j < nw) v[u] = fmaf(ome, tile_get(wg + (size_t)(j / KB) * TILE_FLOATS, b, j % KB), v[u]);
            }
        }
        quad_put(w.wt2d + ((size_t)item * w.row_kb + row0 / KB) * TILE_FLOATS, b, row0 % KB, v);
    }
}

// ------------------------------------------------------------------ adjoint of Eq. 1

// Column tile cb (128 true-energy columns), rows: the union of the columns' bands within
// [max(0, m_lo - L + 1), M).  A_X[i, c] = X[32 kb + c, i] for the node sums P0, P1, P2 of
// bx_resp.cuh, generated by the row recurrence, B = Wt tiles; D_X accumulate in three TMEM
// blocks.  The rows go in half k-blocks of 16 (each thread's 8 rows one run, adj_nodes_run<8>)
// through two A buffers of 48 KB, so that the CUDA cores generate half-block j + 1 while the
// tensor core multiplies j; B tiles (32 rows) are double-buffered per k-block.
__global__ void __launch_bounds__(T2 + 32, 1) k_bwd2d(Work w) {
    extern __shared__ unsigned char smem_raw[];
    constexpr int AH_FLOATS = TM * 16;      // one part of a half k-block's A tile
    float* A = align128(smem_raw);          // [2][3][2][AH_FLOATS]: buffer, (P0 hi, lo), (P1 ...), (P2 ...)
    float* Bt = A + 6 * A_FLOATS;           // [2][TILE_FLOATS]
    float* sco = Bt + 2 * TILE_FLOATS;      // [3][NSL][KMAX]: the coefficient planes, species fastest
    static_assert(2 * 6 * AH_FLOATS == 6 * A_FLOATS, "two half-block A buffers in the space of one k-block's");
    __shared__ PipeF pp;
    __shared__ uint64_t a_bar[2];           // half-block's A tile written (T2 arrivals)
    __shared__ double red[GPN + 1][4];
    __shared__ float xch[4][32][KMAX + 3];
    const int cb = blockIdx.x % w.max_cb, item = blockIdx.x / w.max_cb, tid = threadIdx.x;
    const bool gen = tid < T2;              // warps 0-7 generate A; warp 8 copies B and multiplies
    const Toy& T = w.toys[w.toy_of[item]];
    if (cb >= T.n_cb) return;
    double* gp = w.gpart2d + ((size_t)item * MAX_CB + cb) * (GPN + 1);
    if (w.status[item]) {
        if (tid <= GPN) gp[tid] = 0.0;
        return;
    }
    const int K = T.K, M = T.M, N = T.N;
    const int r = tid & (TM - 1), h = (tid >> 7) & 1, warp = tid >> 5;
    const int2 rr = w.cb_rows[(size_t)item * MAX_CB + cb];
    const int r0 = max(rr.x, max(0, T.m_lo - T.L + 1)), r1 = min(rr.y, M);
    const int kb0 = r0 / KB, nblk = r1 > r0 ? (r1 + KB - 1) / KB - kb0 : 0;
    const float* coefg = w.coef2d + (size_t)item * 4 * KMAX * NSL;
    for (int idx = tid; idx < 3 * KMAX * NSL; idx += blockDim.x) {   // [p][k][b] -> [p][b][k]
        const int p = idx / (KMAX * NSL), r = idx - p * KMAX * NSL, b = r / KMAX, k = r - b * KMAX;
        sco[idx] = coefg[(size_t)(p * KMAX + k) * NSL + b];
    }
    const float* wtg = w.wt2d + (size_t)item * w.row_kb * TILE_FLOATS;
    const int i_gen = cb * BCOLS + r;   // column generated by this thread
    const bool col_ok = i_gen < N;
    const float4 cf = col_ok ? w.colf[(size_t)item * w.Npad + i_gen] : make_float4(0.f, 0.f, 0.f, 0.f);
    const ColG cg = col_ok ? w.colg[(size_t)item * w.Npad + i_gen] : ColG{0.f, 0.f, 0.f, 0.f};
    const AdjCol ac = adj_col(cf, cg);
    bool ok = true;
    uint32_t tbase = 0;
    if (tid == 0) {
        mbar_init(&pp.mma_bar[0], 1);
        mbar_init(&pp.mma_bar[1], 1);
        mbar_init(&pp.b_bar[0], 1);
        mbar_init(&pp.b_bar[1], 1);
        mbar_init(&a_bar[0], T2);
        mbar_init(&a_bar[1], T2);
        pp.abort = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(&pp.tmem, 4 * NSL);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    tbase = pp.tmem;
    {
        volatile int* abort_flag = &pp.abort;
        const int nh = 2 * nblk;
        if (gen) {
            for (int j = 0; j < nh; ++j) {
                const int s = j & 1, it = j >> 1;
                // half-block j - 2 used A buffer s: its MMAs (and, by the commit's order, all earlier
                // ones) must be done before the buffer is rewritten
                const bool okw = j < 2 || mbar_wait(&pp.mma_bar[s], ((j - 2) >> 1) & 1, w.watchdog_ns);
                if (!okw) atomicOr(&pp.abort, 1);
                if (__any_sync(0xffffffffu, !okw || *abort_flag != 0)) break;
                const int mb = (kb0 + it) * KB + 16 * s;   // first row of the half-block
                float* Ah = A + s * 6 * AH_FLOATS;
                // the thread's 8 rows of its column: one run of the row recurrence (bx_resp.cuh), kept
                // in registers and stored as 16-byte rows of the core matrices (4 rows of the run each)
                float pv[3][8];
                adj_nodes_run<8>((float)(mb + 8 * h), 8, cf, cg, ac, [&](int k, float P0, float P1, float P2) {
                    const bool in = col_ok && mb + 8 * h + k < M;
                    pv[0][k] = in ? P0 : 0.f;
                    pv[1][k] = in ? P1 : 0.f;
                    pv[2][k] = in ? P2 : 0.f;
                });
#pragma unroll
                for (int x = 0; x < 3; ++x)
#pragma unroll
                    for (int g4 = 0; g4 < 2; ++g4) {
                        float hv[4], lv[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            hv[q] = tf32_rna(pv[x][4 * g4 + q]);
                            lv[q] = tf32_rna(pv[x][4 * g4 + q] - hv[q]);
                        }
                        const int o = a_off(r, 8 * h + 4 * g4);
                        *reinterpret_cast<float4*>(Ah + 2 * x * AH_FLOATS + o) = make_float4(hv[0], hv[1], hv[2], hv[3]);
                        *reinterpret_cast<float4*>(Ah + (2 * x + 1) * AH_FLOATS + o) = make_float4(lv[0], lv[1], lv[2], lv[3]);
                    }
                fence_proxy_async_smem();
                tc_fence_before();
                mbar_arrive(&a_bar[s]);
            }
        } else if (tid == T2) {   // warp 8, lane 0: the B tiles and the MMAs, in half-block order
            int issued = 0, waited = 0, committed = 0;
            if (nblk > 0) {
                mbar_arrive_expect_tx(&pp.b_bar[0], TILE_BYTES);
                bulk_g2s(Bt, wtg + (size_t)kb0 * TILE_FLOATS, TILE_BYTES, &pp.b_bar[0]);
                issued = 1;
            }
            for (int j = 0; j < nh; ++j) {
                const int s = j & 1, it = j >> 1;
                bool okw = true;
                // B buffer (it + 1) & 1 was last read by half-blocks 2 it - 2 and 2 it - 1: the commit
                // of 2 it - 1 (= j - 2 here) covers both
                if (s == 1 && it + 1 < nblk) {
                    if (it >= 1) okw = mbar_wait(&pp.mma_bar[1], ((j - 2) >> 1) & 1, w.watchdog_ns);
                    if (okw) {
                        mbar_arrive_expect_tx(&pp.b_bar[(it + 1) & 1], TILE_BYTES);
                        bulk_g2s(Bt + ((it + 1) & 1) * TILE_FLOATS, wtg + (size_t)(kb0 + it + 1) * TILE_FLOATS,
                                 TILE_BYTES, &pp.b_bar[(it + 1) & 1]);
                        ++issued;
                    }
                }
                okw = okw && mbar_wait(&a_bar[s], (j >> 1) & 1, w.watchdog_ns);
                if (okw && s == 0) {
                    okw = mbar_wait(&pp.b_bar[it & 1], (it >> 1) & 1, w.watchdog_ns);
                    if (okw) ++waited;
                }
                if (!okw) {
                    atomicOr(&pp.abort, 1);
                    break;
                }
                tc_fence_after();
                const float* B = Bt + (it & 1) * TILE_FLOATS;
                float* Ah = A + s * 6 * AH_FLOATS;
#pragma unroll
                for (int x = 0; x < 3; ++x)
                    mma_half(tbase + (uint32_t)(x * NSL), Ah + 2 * x * AH_FLOATS, Ah + (2 * x + 1) * AH_FLOATS, B, s, j > 0);
                umma_commit(&pp.mma_bar[s]);
                ++committed;
                if (*abort_flag) break;
            }
            if (!drain_copies3(pp, waited, issued)) atomicOr(&pp.abort, 1);
            pp.committed = committed;
        }
        __syncthreads();
        const int nc = pp.committed;
        const unsigned long long budget = w.watchdog_ns > CLEANUP_NS ? w.watchdog_ns : CLEANUP_NS;
        bool done = true;
        // the last two half-blocks (one per barrier) are still to be waited for
        if (gen)
            for (int j = (nc >= 2 ? nc - 2 : 0); j < nc; ++j) done &= mbar_wait(&pp.mma_bar[j & 1], (j >> 1) & 1, budget);
        tc_fence_after();
        ok = __all_sync(0xffffffffu, !pp.abort && done && nc == nh);   // warp-uniform: the epilogue's tcgen05.ld
        if (!ok && tid == 0) atomicOr(w.err, ERR_TIMEOUT);
    }
    // epilogue: column i = 32 (warp % 4) + lane of the tile; warps 0-3 take slices 0..63,
    // warps 4-7 slices 64..127; per column: S_X = sum_b T_r D_X, rate and s_r sums of D_0
    const int lane = tid & 31, q4 = warp & 3, half = gen ? warp >> 2 : 2;   // warp 8 (half 2) sits out
    const int i = cb * BCOLS + q4 * 32 + lane;
    const bool iok = i < N && ok;
    float sk[KMAX];
#pragma unroll
    for (int k = 0; k < KMAX; ++k) sk[k] = (iok && k < K) ? T.shapes32[(size_t)k * N + i] : 0.f;
    float racc[KMAX], dacc = 0.f, S1 = 0.f, S2 = 0.f;
#pragma unroll
    for (int k = 0; k < KMAX; ++k) racc[k] = 0.f;
    if (ok && nblk > 0 && gen) {
        const uint32_t lanebase = tbase + ((uint32_t)(q4 * 32) << 16);
        const int n_sl = T.n_sl;
        const float* uti = T.ut + (size_t)(iok ? i : 0) * NSL;
        for (int j0 = half * (NSL / 2); j0 < (half + 1) * (NSL / 2); j0 += 8) {
            float d0[8], d1[8], d2[8];
            tmem_ld8(lanebase + (uint32_t)j0, d0);
            tmem_ld8(lanebase + (uint32_t)(NSL + j0), d1);
            tmem_ld8(lanebase + (uint32_t)(2 * NSL + j0), d2);
            if (iok) {
                // the column's 8 modulation values of these slices: two 16-byte loads
                const float4 ua = *reinterpret_cast<const float4*>(uti + j0);
                const float4 ub = *reinterpret_cast<const float4*>(uti + j0 + 4);
                const float uv[8] = {ua.x, ua.y, ua.z, ua.w, ub.x, ub.y, ub.z, ub.w};
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int b = j0 + q;
                    if (b >= n_sl) break;
                    const float u = uv[q];
                    const float E = u * d0[q];
                    float tr = 0.f, dk = 0.f;
                    // the slice's coefficients of every species as 16-byte broadcast loads (the
                    // planes hold zeros beyond K, like sk)
                    const float4* c0 = reinterpret_cast<const float4*>(sco + (size_t)b * KMAX);
                    const float4* c1 = reinterpret_cast<const float4*>(sco + (size_t)(NSL + b) * KMAX);
                    const float4* c2 = reinterpret_cast<const float4*>(sco + (size_t)(2 * NSL + b) * KMAX);
#pragma unroll
                    for (int k4 = 0; k4 < KMAX / 4; ++k4) {
                        const float4 a0 = c0[k4], a1 = c1[k4], a2 = c2[k4];
                        tr = fmaf(a0.x, sk[4 * k4], fmaf(a0.y, sk[4 * k4 + 1], fmaf(a0.z, sk[4 * k4 + 2], fmaf(a0.w, sk[4 * k4 + 3], tr))));
                        dk = fmaf(a2.x, sk[4 * k4], fmaf(a2.y, sk[4 * k4 + 1], fmaf(a2.z, sk[4 * k4 + 2], fmaf(a2.w, sk[4 * k4 + 3], dk))));
                        racc[4 * k4] = fmaf(a1.x, E, racc[4 * k4]);
                        racc[4 * k4 + 1] = fmaf(a1.y, E, racc[4 * k4 + 1]);
                        racc[4 * k4 + 2] = fmaf(a1.z, E, racc[4 * k4 + 2]);
                        racc[4 * k4 + 3] = fmaf(a1.w, E, racc[4 * k4 + 3]);
                    }
                    dacc = fmaf(dk, E, dacc);
                    tr *= u;
                    S1 = fmaf(tr, d1[q], S1);
                    S2 = fmaf(tr, d2[q], S2);
                }
            }
        }
    }
    tc_fence_before();
    // the upper half hands its partial sums to the lower half
    if (half == 1) {
#pragma unroll
        for (int k = 0; k < KMAX; ++k) xch[q4][lane][k] = racc[k];
        xch[q4][lane][KMAX] = dacc;
        xch[q4][lane][KMAX + 1] = S1;
        xch[q4][lane][KMAX + 2] = S2;
    }
    __syncthreads();
    if (warp == 0) tmem_dealloc(tbase, 4 * NSL);
    double g[GPN + 1];
#pragma unroll
    for (int k = 0; k <= GPN; ++k) g[k] = 0.0;
    if (half == 0) {
#pragma unroll
        for (int k = 0; k < KMAX; ++k) racc[k] += xch[q4][lane][k];
        dacc += xch[q4][lane][KMAX];
        S1 += xch[q4][lane][KMAX + 1];
        S2 += xch[q4][lane][KMAX + 2];
        if (iok) {
            const Col64 cc = w.col64[(size_t)item * w.Npad + i];
            const double2 qq = w.colq[(size_t)item * w.Npad + i];
            const double* th = w.theta + (size_t)item * w.tstride;
            const double LY = th[K], a = th[K + 1], b = th[K + 2];
            const double isig = 1.0 / cc.sig;
            const double Acol = (0.5 * INV_SQRT_2PI * GL_W_SCALE) * T.w * isig * cc.norm;   // R = Acol P0
            double S0 = 0.0;
#pragma unroll
            for (int k = 0; k < KMAX; ++k)
                if (k < K) {
                    const double gk = (double)racc[k] * (double)sk[k];   // sum_b dT_r/dr_k D_0 / Acol
                    g[5 + k] = Acol * gk;
                    S0 += th[k] * gk;
                }
            g[GPN] = Acol * (double)dacc;
            const double s0 = Acol * S0;
            const double s1 = Acol * isig * ((double)S1 * (1.0 / S_EX2));
            const double s2 = Acol * isig * ((double)S2 * (1.0 / (S_EX2 * S_EX2)) - S0);
            const double dmu = s1 - cc.mills * isig * s0;
            const double dsig = s2 + cc.mills * cc.mu * isig * isig * s0;
            const double D = 0.5 * isig * dsig;
            const double Gmu = dmu + D * (a + 2.0 * b * cc.mu);
            g[0] = Gmu * qq.x;
            g[1] = D * cc.mu;
            g[2] = D * cc.mu * cc.mu;
            g[3] = D;
            g[4] = Gmu * LY * qq.y;
        }
#pragma unroll
        for (int k = 0; k <= GPN; ++k) {
            const double v = warp_sum(g[k]);
            if (lane == 0) red[k][q4] = v;
        }
    }
    __syncthreads();
    if (tid <= GPN) gp[tid] = red[tid][0] + red[tid][1] + red[tid][2] + red[tid][3];
}

// ------------------------------------------------------------------ gather

// A warp per item, lane j = parameter j (as k_gather; the window tiles' sums of -lnL and of the
// eps gradient keep their order).
__global__ void __launch_bounds__(128) k_gather2d(Work w, int n, double* nll_out, double* grad_out, int want_grad) {
    const int item = blockIdx.x * 4 + (threadIdx.x >> 5), j = threadIdx.x & 31;
    if (item >= n) return;
    const Toy& T = w.toys[w.toy_of[item]];
    const int st = w.status[item];
    const int nt = (T.nw + TM - 1) / TM;
    if (j == 0) {
        double s = 0.0, c = 0.0;
#pragma unroll 4
        for (int t = 0; t < nt; ++t) {
            s += w.nll2d[((size_t)item * MAX_TILES + t) * 2];
            c += w.nll2d[((size_t)item * MAX_TILES + t) * 2 + 1];
        }
        nll_out[item] = st ? INFINITY : s + c;
    }
    if (!want_grad || j >= w.pstride) return;
    double g = 0.0;
    if (!st && j < T.P) {
        const int slot = j < T.K ? 5 + j : j < T.K + 5 ? j - T.K : j == T.K + 6 ? GPN : -1;
        // the column blocks' partials, or (eps) the window tiles'
        const double* gp = slot >= 0 ? w.gpart2d + (size_t)item * MAX_CB * (GPN + 1) + slot
                                     : w.geps2d + (size_t)item * MAX_TILES;
        const int np = slot >= 0 ? T.n_cb : nt, step = slot >= 0 ? GPN + 1 : 1;
#pragma unroll 8
        for (int q = 0; q < np; ++q) g += gp[(size_t)q * step];
    }
    grad_out[(size_t)item * w.pstride + j] = g;
}

// ------------------------------------------------------------------ launchers


// stage 1: templates and the forward GEMM; stage 2: pile-up and -lnL; stage 3: adjoint.
cudaError_t launch_eval2d(const Work& w, int n, int want_grad, int want_mu, int stage, cudaStream_t s) {
    static SmemOptIn c_fwd, c_fwd_bf, c_pile, c_corr, c_bwd;
    cudaError_t e = cudaSuccess;
    if (stage == 1) {
        // the forward stage of one item: 174 us with one CTA here, 129 with eight
        const int np = w.prep_part && n <= PREP_ITEMS ? max(1, min(PREP_PARTS, 152 / n)) : 1;
        k_coef2d<<<n * np, 512, 0, s>>>(w, np);
        const size_t sm = (size_t)(6 * A_FLOATS + 2 * TILE3_FLOATS) * 4 + 128;
        if (w.precision == BX_BF16X3) {
            k_trate<true><<<(unsigned)n * (unsigned)w.tr_kb, NSL * TRS<true>, 0, s>>>(w);
            if ((e = smem_opt_in(c_fwd_bf, k_fwd2d<true>, sm)) != cudaSuccess) return e;
            k_fwd2d<true><<<(unsigned)n * (unsigned)w.max_tiles, TF + 32, sm, s>>>(w);
        } else {
            k_trate<false><<<(unsigned)n * (unsigned)w.tr_kb, NSL * TRS<false>, 0, s>>>(w);
            if ((e = smem_opt_in(c_fwd, k_fwd2d<false>, sm)) != cudaSuccess) return e;
            k_fwd2d<false><<<(unsigned)n * (unsigned)w.max_tiles, TF + 32, sm, s>>>(w);
        }
    } else if (stage == 2) {
        if ((e = smem_opt_in(c_pile, k_pile2d, TP_SMEM)) != cudaSuccess) return e;
        k_pile2d<<<(unsigned)n * (unsigned)w.win_tiles, TP, TP_SMEM, s>>>(w, want_mu);
    } else if (stage == 3 && want_grad) {
        if ((e = smem_opt_in(c_corr, k_corr2d, TP_SMEM)) != cudaSuccess) return e;
        k_corr2d<<<(unsigned)n * (unsigned)w.max_tiles, TP, TP_SMEM, s>>>(w);
        const size_t sb = (size_t)(6 * A_FLOATS + 2 * TILE_FLOATS + 3 * KMAX * NSL) * 4 + 128;
        if ((e = smem_opt_in(c_bwd, k_bwd2d, sb)) != cudaSuccess) return e;
        k_bwd2d<<<(unsigned)n * (unsigned)w.max_cb, T2 + 32, sb, s>>>(w);
    }
    return cudaGetLastError();
}

cudaError_t launch_gather2d(const Work& w, int n, double* nll_out, double* grad_out, int want_grad, cudaStream_t s) {
    k_gather2d<<<(n + 3) / 4, 128, 0, s>>>(w, n, nll_out, grad_out, want_grad);
    return cudaGetLastError();
}

}  // namespace bx

// Device-side model layout and block-level building blocks of the forward-folding fit.
//
// One thread block evaluates one parameter vector of one model: the expectation of every
// dataset (survival x reweights on the fine true grid, energy correction by overlap length,
// banded response fold, backgrounds), the Poisson -2lnL and its adjoint gradient. The same
// device functions serve the batched evaluation kernels and the persistent fit kernel.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/fitcore.h"

namespace fitcore {

constexpr int kMaxWarps = 16;      // blocks of at most 512 threads
constexpr int kMaxBkgDs = 6;       // backgrounds per dataset
constexpr int kMaxOsc = 6;         // survival parameters (6 for the 3+1 formula, else 4)

// A banded matrix packed for matrix-vector products (band_product): four consecutive outputs per lane
// group of `parts` lanes, each lane a consecutive range of the band's inputs. Warp unit w holds
// 32 such lanes: steps[w].y steps of 32 float4 from entry + steps[w].x; lane l of it starts at
// input start[32 w + l]. Entries outside a lane's own range are 0 and every input read exists.
struct BandUnits {
    const int2 *steps;
    const int *start;
    const float4 *entry;
    int n, parts, outs;
};

struct DevDetector {
    int n_reco;
    BandUnits fold;          // outputs: reco rows in fours, inputs: true bins
    BandUnits adj;           // outputs: true bins in fours, inputs: reco rows
    const int2 *row_band;    // [N_r] first true bin and length of each row's band
    const float *rdense_hi;  // [N_r x ldt] dense response, TF32-exact high part (tensor-core fold)
    const float *rdense_lo;  // [N_r x ldt] R - rdense_hi
    const float *rdt_hi;     // [N_t x ldr] R^T, TF32-exact high part (tensor-core adjoint fold)
    const float *rdt_lo;     // [N_t x ldr] R^T - rdt_hi
    int ldr;                 // row stride of R^T (N_r rounded up to 4)
};

struct DevBkg {
    const float *tmpl;       // [N_r] expected counts at nominal
    const int *shape_idx;    // [N_r] parameter of delta_j or -1
    int rate_idx;
    int pad;
};

struct DevDataset {
    int det, n_reco, data_off;
    int norm_idx, eff_idx;
    int esc_idx[3];
    float a1_off;            // theta0(a1) - 1, so that a1 - 1 = a1_off + (theta - theta0)
    int bkg_begin, bkg_end;  // backgrounds of this dataset in DevModel::bkg
    int n_sp;                // distinct shape parameters used by this dataset
    const float *t;          // [N_t] un-oscillated signal
    const int *shape_idx;    // [N_t]
    // Shape parameter p: parameter sp[p].x, sp[p].z true bins, consecutive from sp[p].y (sp[p].w = 1)
    // or at sp_k + sp[p].y
    const int4 *sp;          // [n_sp]
    const int *sp_k;
    int lik_dup, map_dup;    // gradient totals whose parameter receives another total too: bits of
                             // (deviance, efficiency, rates) and of (a0, a1, a2, norm)
    int sp_lanes;            // lanes that share one shape parameter's sum (a power of two <= 32)
    float w[FIT_MAX_CORES];  // core flux shares
    float kl_hi[FIT_MAX_CORES], kl_lo[FIT_MAX_CORES];  // K L_dc / pi as a float pair (half-turns)
};

// One tile of a triangular matrix-vector product: out rows `out`.. (of all blocks concatenated), summed
// over `cols` columns, the inputs in0.. (consecutive parameters) or blk_idx[idx..] (in0 < 0). The
// tile's matrix entries are stored column after column, `pitch` (rows rounded up to 4) floats each.
struct TriTile {
    int mat, pitch, rows, cols;
    int in0, idx, out, seg;
};

// Bin j of background q (dataset d, row of the data vector of that dataset) scaled by a shape parameter
struct BkgShapeRef {
    int d, q, j;
    float tmpl;
};

struct DevModel {
    int P, N_t, C, n_ds, n_data, osc_mode, n_blocks, n_bkg;
    float e_lo, de, inv_de;
    float e_first, e_last;   // e_edge[0], e_edge[N_t]
    int shared_roles;        // 1: some parameter has two roles (say, a shape of two datasets, or a
                             // rate that is also a norm): its gradient additions need ordering
    int n_osc;               // survival parameters of osc_mode: 4, or 6 (FIT_OSC_STERILE4)
    int remap_mode;          // FIT_REMAP_OVERLAP or FIT_REMAP_SPLINE
    int osc_idx[kMaxOsc];
    float osc_val[kMaxOsc];
    float osc_val_lo[kMaxOsc];   // low parts of the constant survival parameters
    float osc_th_f[kMaxOsc], osc_th_lo[kMaxOsc];   // theta0 of the fitted ones as a float pair
    int osc_dup;             // as DevDataset::map_dup: bits of the survival parameters, then the powers
    int any_map_dup;         // 1: osc_dup or some dataset's map_dup is not 0
    int core_power_idx[FIT_MAX_CORES];
    const float *e_edge;     // [N_t + 1]
    const float *inv_e_hi;   // [N_t] 1 / E_k (true-bin centre) as a float pair
    const float *inv_e_lo;
    DevDataset ds[FIT_MAX_DATASETS];
    DevDetector det[FIT_MAX_DETECTORS];
    DevBkg bkg[FIT_MAX_BACKGROUNDS];
    // parameters, priors and the transformation layer
    const double *theta0;    // [P]
    const float *theta0_f;   // [P] theta0 rounded to float
    const float *theta0_lo;  // [P] theta0 - theta0_f (the low part of a float pair)
    const float *zscale;     // [P] sigma (individual prior) or scale (free); 0 in a block
    const float *prior_inv;  // [P] 1/sigma for individually constrained parameters, else 0
    const int *blk_size;     // [n_blocks]
    const int *blk_idx_off;  // [n_blocks]
    const int *blk_idx;      // concatenated parameter indices
    const int64_t *blk_mat_off;  // [n_blocks] offset of the block's m x m matrices
    const double *blk_L64;   // lower Cholesky factors of V, then transposed (final theta of a fit)
    const float *asimov;     // [n_data] expectation at theta0
    const int *slot_ds;      // [n_data] dataset of each data bin
    int ws_eval_floats;      // workspace of one dataset of one evaluation (a multiple of 4)
    int ws_group;            // datasets evaluated together (their workspaces are held at once)
    // matrix-vector products with the triangular prior blocks as packed tiles (see tri_apply):
    // tri_lo for L z / W d, tri_up for L^T g / W^T z; the tiles' entries in L_lo, L_up, W_lo, W_up
    const TriTile *tri_lo, *tri_up;
    const float *L_lo, *L_up, *W_lo, *W_up;
    int n_tri_lo, n_tri_up, tri_segs, tri_rows;   // tiles, column segments, rows of all blocks
    const int *tri_param;    // [tri_rows] parameter of each concatenated row
    const int *tri_seg;      // [tri_rows] its segments: lower 0..(x & 255) - 1, upper
                             // (x >> 8 & 255)..(x >> 16) - 1
    int ws_floats;           // per-block workspace of one evaluation: ws_group datasets, or the
                             // tri_segs x tri_rows partial sums if larger
    // background-shape parameters and the (background, bin) pairs each one scales, by dataset
    const int *bs_param;     // [n_bs]
    const int *bs_ptr;       // [n_bs + 1]
    const BkgShapeRef *bs_ref;
    int n_bs;
    int max_reco;
    int ldt;                 // row stride of the dense response (N_t rounded up to 4)
    // Fisher preconditioner (nullptr until built): z = T w, T = I + Q diag(c) Q^T; pre_Q holds
    // Q^T as pre_r rows on the vector pitch, pre_c the r coefficients c then the r of T^-1
    const float *pre_Q, *pre_c;
    int pre_r;
};

// ------------------------------------------------------------------------------------
// Reductions: FP32 within a warp, FP64 across warps.
// ------------------------------------------------------------------------------------
// Sum of one value per thread over the block, on every thread: FP32 within a warp, then one
// warp adds the warps' totals in double (a double addition occupies the SM's FP64 pipe for 16
// cycles per warp, so only one warp does it). red: kMaxWarps + 1 doubles of shared scratch,
// reusable by the next call without another barrier. Contains two __syncthreads.
__device__ __forceinline__ double block_sum(float v, double *red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) red[warp] = (double)v;
    __syncthreads();
    if (warp == 0) {
        double t = lane < nw ? red[lane] : 0.0;
#pragma unroll
        for (int o = kMaxWarps / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) red[kMaxWarps] = t;
    }
    __syncthreads();
    return red[kMaxWarps];
}

// Warp totals of N (a power of two <= 32) per-lane values with N - 1 + log2(32 / N) shuffles
// instead of 5 N: each step exchanges half of the values with the partner lane and keeps the
// sums of the other half. Lane l returns the total of value l >> (5 - log2 N), every lane of
// the group the same; the additions are those of warp_sum's tree.
template <int N>
__device__ __forceinline__ float warp_sum_split(float (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int n = N; n > 1; n >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const float give = up ? v[i] : v[i + n / 2], keep = up ? v[i + n / 2] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    float t = v[0];
    for (; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// ------------------------------------------------------------------------------------
// Survival probability with phase arithmetic in float pairs.
// ------------------------------------------------------------------------------------
// sin and cos of pi r for |r| <= 1/2 (a little more is harmless): r (pi + u P(u)) and 1 + u Q(u),
// u = r^2, P of degree 3 and Q of degree 4 fitted for the smallest largest error (Lawson
// iteration; sin2pi_fit.py in this directory), pi as a float pair. Within 1.3e-7 in FP32,
// the error of sincospif's results to one unit in the last place at half its instructions
// (the phase is already reduced, so none of them goes into reduction and quadrants).
__device__ __forceinline__ void sincos_half(float r, float &s, float &c) {
    const float u = r * r;
    float t = fmaf(0.07749626f, u, -0.59821373f);
    t = fmaf(t, u, 2.5500667f);
    t = fmaf(t, u, -5.16771f);
    t = fmaf(t, u, -8.742278e-8f);        // pi - (float)pi
    s = fmaf(r, 3.14159274f, r * t);
    float q = fmaf(-0.024417998f, u, 0.23495245f);
    q = fmaf(q, u, -1.3352158f);
    q = fmaf(q, u, 4.0587096f);
    q = fmaf(q, u, -4.934802f);
    c = fmaf(q, u, 1.f);
}

// Phase in half-turns: y = x / pi = (dm_hi + dm_lo) * (c_hi + c_lo), c = K L / (pi E), carried
// as a float pair. The probability depends on sin^2 x and sin 2x only, so y is reduced by
// its nearest integer, which is exact (y_hi - rint(y_hi) is representable), and sin, cos of
// pi r, |r| <= 1/2, follow. The pair keeps r accurate to ~1e-8 even at 50 km
// (y ~ 30), and no pi constant or multi-word reduction enters the arithmetic.
__device__ __forceinline__ void phase_sc(float dm, float dm_lo, float c_hi, float c_lo, float &s,
                                         float &c) {
    const float yh = dm * c_hi;
    const float yl = fmaf(dm_lo, c_hi, fmaf(dm, c_lo, fmaf(dm, c_hi, -yh)));
    sincos_half((yh - rintf(yh)) + yl, s, c);
}

// Packed FP32: two values in one register pair, one instruction for both.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ f32x2 pack2(float a) { return pack2(a, a); }
__device__ __forceinline__ float2 unpack2(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// sincos_half for two reduced phases
__device__ __forceinline__ void sincos_half2(f32x2 r, f32x2 &s, f32x2 &c) {
    const f32x2 u = mul2(r, r);
    f32x2 t = fma2(pack2(0.07749626f), u, pack2(-0.59821373f));
    t = fma2(t, u, pack2(2.5500667f));
    t = fma2(t, u, pack2(-5.16771f));
    t = fma2(t, u, pack2(-8.742278e-8f));
    s = fma2(r, pack2(3.14159274f), mul2(r, t));
    f32x2 q = fma2(pack2(-0.024417998f), u, pack2(0.23495245f));
    q = fma2(q, u, pack2(-1.3352158f));
    q = fma2(q, u, pack2(4.0587096f));
    q = fma2(q, u, pack2(-4.934802f));
    c = fma2(q, u, pack2(1.f));
}

// The reduced phase -y of phase_sc for two cores (dm, -dm, its low part; m1 = -1)
__device__ __forceinline__ f32x2 neg_phase2(f32x2 dm, f32x2 ndm, f32x2 dm_lo, f32x2 ch, f32x2 cl, f32x2 m1) {
    const f32x2 n = mul2(ndm, ch);
    const f32x2 e = fma2(dm_lo, ch, fma2(dm, cl, fma2(dm, ch, n)));
    const float2 v = unpack2(n);
    return fma2(e, m1, fma2(pack2(rintf(v.x), rintf(v.y)), m1, n));
}

// sin^2(pi r) for |r| <= 1/2: u q(u), u = r^2, q a degree-7 polynomial fitted for the
// smallest largest absolute error (Lawson iteration; sin2pi_fit.py in this directory). Its
// FP32 evaluation is within 1.8e-7 of sin^2. (This form states the constants for one phase.)
__device__ __forceinline__ float sin2pi(float r) {
    const float u = r * r;
    float q = -0.122019291f;
    q = fmaf(q, u, 0.848584056f);
    q = fmaf(q, u, -3.94964409f);
    q = fmaf(q, u, 13.2128229f);
    q = fmaf(q, u, -30.1222954f);
    q = fmaf(q, u, 42.7284088f);
    q = fmaf(q, u, -32.469696f);
    q = fmaf(q, u, 9.86960411f);
    return u * q;
}

// The same for two phases: what the event kernel evaluates.
__device__ __forceinline__ f32x2 sin2pi2(f32x2 r) {
    const f32x2 u = mul2(r, r);
    f32x2 q = fma2(pack2(-0.122019291f), u, pack2(0.848584056f));
    q = fma2(q, u, pack2(-3.94964409f));
    q = fma2(q, u, pack2(13.2128229f));
    q = fma2(q, u, pack2(-30.1222954f));
    q = fma2(q, u, pack2(42.7284088f));
    q = fma2(q, u, pack2(-32.469696f));
    q = fma2(q, u, pack2(9.86960411f));
    return mul2(u, q);
}

// Coefficients of the sin^2 terms of P, formed once per evaluation in double from the exact
// parameter values and applied as float pairs (a single FP32 rounding of a coefficient would
// bias every bin coherently).
//   FIT_OSC_EQ1:     P = 1 - C0 sin^2 x_ee - C1 sin^2 x_21,  C0 = sin^2 2th13,
//                    C1 = cos^4 th13 sin^2 2th12
//   FIT_OSC_VACUUM3: P = 1 - C0 sin^2 x_21 - C1 sin^2 x_31 - C2 sin^2 x_32,
//                    C0 = cos^4 th13 sin^2 2th12, C1 = sin^2 2th13 cos^2 th12,
//                    C2 = sin^2 2th13 sin^2 th12
template <int NT>
struct OscCoefN {
    float hi[NT], lo[NT];
};
using OscCoef = OscCoefN<3>;

template <int NT>
__device__ __forceinline__ float cterm(const OscCoefN<NT> &k, int i, float q) {
    return fmaf(q, k.lo[i], k.hi[i] * q);
}

// Float-pair ("double-float") arithmetic: a value h + l with |l| <= ulp(h) / 2, carried in two
// floats (error-free transformations of Knuth's two-sum and the FMA two-product, Dekker's
// normalisation). Used where a few coefficients need more than 24 bits but FP64 would sit on
// the critical path (GB300 runs FP64 at 1/64 of the FP32 rate).
struct F2 {
    float h, l;
};

__device__ __forceinline__ F2 f2_norm(float h, float l) {
    const float s = h + l;
    return F2{s, l - (s - h)};
}

__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    const float s = a.h + b.h;
    const float bb = s - a.h;
    const float e = (a.h - (s - bb)) + (b.h - bb);
    return f2_norm(s, e + (a.l + b.l));
}

__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    const float p = a.h * b.h;
    const float e = fmaf(a.h, b.h, -p);
    return f2_norm(p, fmaf(a.h, b.l, fmaf(a.l, b.h, e)));
}

__device__ __forceinline__ F2 f2_scale(F2 a, float c) {   // c a power of two
    return F2{a.h * c, a.l * c};
}

__device__ __forceinline__ F2 f2_one_minus(F2 a) { return f2_add(F2{1.f, 0.f}, F2{-a.h, -a.l}); }

// square root: s = sqrtf(h) refined by one Newton step on the residual a - s^2
__device__ __forceinline__ F2 f2_sqrt(F2 a) {
    if (!(a.h > 0.f)) return F2{0.f, 0.f};
    const float s = sqrtf(a.h);
    const float r = fmaf(-s, s, a.h) + a.l;
    return f2_norm(s, r / (2.f * s));
}

// The sin^2 coefficients of Eq. 1 and the three-flavour formula from float pairs e of the exact
// parameter values.
__device__ __forceinline__ OscCoef osc_coef(int mode, const F2 (&e)[4]) {
    F2 cf[3];
    if (mode == FIT_OSC_EQ1) {
        // cos^4 th13 = ((1 + sqrt(1 - sin^2 2th13)) / 2)^2
        const F2 c2 = f2_scale(f2_add(F2{1.f, 0.f}, f2_sqrt(f2_one_minus(e[0]))), 0.5f);
        cf[0] = e[0];
        cf[1] = f2_mul(f2_mul(c2, c2), e[2]);
        cf[2] = F2{0.f, 0.f};
    } else {
        const F2 S12 = f2_scale(f2_mul(e[0], f2_one_minus(e[0])), 4.f);
        const F2 S13 = f2_scale(f2_mul(e[1], f2_one_minus(e[1])), 4.f);
        const F2 c13 = f2_one_minus(e[1]);
        cf[0] = f2_mul(f2_mul(c13, c13), S12);
        cf[1] = f2_mul(S13, f2_one_minus(e[0]));
        cf[2] = f2_mul(S13, e[0]);
    }
    OscCoef k;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        k.hi[i] = cf[i].h;
        k.lo[i] = cf[i].l;
    }
    return k;
}

// Exact 3+1 vacuum survival (FIT_OSC_STERILE4), one sterile state added to the three-flavour
// formula: eta = (sin^2 th12, sin^2 th13, dm2_21, dm2_31, sin^2 2th14, dm2_41),
//   P = 1 - cos^4 th14 [C0 sin^2 x21 + C1 sin^2 x31 + C2 sin^2 x32]
//         - sin^2 2th14 [cos^2 th13 (cos^2 th12 sin^2 x41 + sin^2 th12 sin^2 x42)
//                        + sin^2 th13 sin^2 x43]
// (the first row of the 4x4 mixing matrix is (c12 c13 c14, s12 c13 c14, s13 c14, s14)), with
// the coefficients k.hi/lo[0..5] of the six sin^2 terms; x32, x42 and x43 from the angle
// differences of x21, x31 and x41.
__device__ __forceinline__ float survival_sterile(const float (&eta)[6], const float (&eta_lo)[6],
                                                  const OscCoefN<6> &k, float c_hi, float c_lo,
                                                  float (&dP)[6]) {
    const float dx = 3.14159265358979f * c_hi;
    const float s12 = eta[0], s13 = eta[1], S14 = eta[4];
    const float c12 = 1.f - s12, c13 = 1.f - s13;
    const float S12 = 4.f * s12 * c12, S13 = 4.f * s13 * c13;
    const float root = sqrtf(fmaxf(1.f - S14, 1e-12f));
    const float c14 = 0.5f * (1.f + root), C4 = c14 * c14;
    float a21, b21, a31, b31, a41, b41;
    phase_sc(eta[2], eta_lo[2], c_hi, c_lo, a21, b21);
    phase_sc(eta[3], eta_lo[3], c_hi, c_lo, a31, b31);
    phase_sc(eta[5], eta_lo[5], c_hi, c_lo, a41, b41);
    const float a32 = a31 * b21 - b31 * a21, b32 = b31 * b21 + a31 * a21;   // x31 - x21
    const float a42 = a41 * b21 - b41 * a21, b42 = b41 * b21 + a41 * a21;   // x41 - x21
    const float a43 = a41 * b31 - b41 * a31, b43 = b41 * b31 + a41 * a31;   // x41 - x31
    const float q21 = a21 * a21, q31 = a31 * a31, q32 = a32 * a32;
    const float q41 = a41 * a41, q42 = a42 * a42, q43 = a43 * a43;
    const float P = ((((((1.f - cterm(k, 0, q21)) - cterm(k, 1, q31)) - cterm(k, 2, q32)) -
                      cterm(k, 3, q41)) - cterm(k, 4, q42)) - cterm(k, 5, q43));
    const float d21 = 2.f * a21 * b21 * dx, d31 = 2.f * a31 * b31 * dx, d32 = 2.f * a32 * b32 * dx;
    const float d41 = 2.f * a41 * b41 * dx, d42 = 2.f * a42 * b42 * dx, d43 = 2.f * a43 * b43 * dx;
    const float A = c13 * c13 * S12 * q21 + S13 * (c12 * q31 + s12 * q32);
    const float Bs = c13 * (c12 * q41 + s12 * q42) + s13 * q43;
    const float dC4 = -c14 * 0.5f / root;
    dP[0] = -C4 * (c13 * c13 * 4.f * (1.f - 2.f * s12) * q21 + S13 * (q32 - q31)) - S14 * c13 * (q42 - q41);
    dP[1] = -C4 * (-2.f * c13 * S12 * q21 + 4.f * (1.f - 2.f * s13) * (c12 * q31 + s12 * q32)) -
            S14 * (q43 - (c12 * q41 + s12 * q42));
    dP[2] = -C4 * (c13 * c13 * S12 * d21 - S13 * s12 * d32) + S14 * c13 * s12 * d42;
    dP[3] = -C4 * S13 * (c12 * d31 + s12 * d32) + S14 * s13 * d43;
    dP[4] = -dC4 * A - Bs;
    dP[5] = -S14 * (c13 * (c12 * d41 + s12 * d42) + s13 * d43);
    return P;
}

// The six coefficients of survival_sterile from float pairs e of the exact parameter values.
__device__ __forceinline__ OscCoefN<6> osc_coef_sterile(const F2 (&e)[6]) {
    const F2 one{1.f, 0.f};
    const F2 c12 = f2_one_minus(e[0]), c13 = f2_one_minus(e[1]);
    const F2 S12 = f2_scale(f2_mul(e[0], c12), 4.f), S13 = f2_scale(f2_mul(e[1], c13), 4.f);
    const F2 c14 = f2_scale(f2_add(one, f2_sqrt(f2_one_minus(e[4]))), 0.5f);   // cos^2 th14
    const F2 C4 = f2_mul(c14, c14);
    F2 cf[6];
    cf[0] = f2_mul(C4, f2_mul(f2_mul(c13, c13), S12));
    cf[1] = f2_mul(C4, f2_mul(S13, c12));
    cf[2] = f2_mul(C4, f2_mul(S13, e[0]));
    cf[3] = f2_mul(e[4], f2_mul(c13, c12));
    cf[4] = f2_mul(e[4], f2_mul(c13, e[0]));
    cf[5] = f2_mul(e[4], e[1]);
    OscCoefN<6> k;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        k.hi[i] = cf[i].h;
        k.lo[i] = cf[i].l;
    }
    return k;
}

// whether survival parameter i of a formula is a mass splitting (carried as a float pair)
__host__ __device__ __forceinline__ bool osc_is_dm(int mode, int i) {
    return mode == FIT_OSC_EQ1 ? (i == 1 || i == 3) : (i == 2 || i == 3 || i == 5);
}

// sin^2 coefficients for the formulas with 4 survival parameters (Eq. 1, three-flavour) or 6 (3+1)
template <int NOSC>
struct OscTraits;
template <>
struct OscTraits<4> {
    using Coef = OscCoefN<3>;
    static __device__ __forceinline__ Coef coef(int mode, const F2 (&e)[4]) { return osc_coef(mode, e); }
};
template <>
struct OscTraits<6> {
    using Coef = OscCoefN<6>;
    static __device__ __forceinline__ Coef coef(int, const F2 (&e)[6]) { return osc_coef_sterile(e); }
};

// Poisson deviance 2[mu - n + n ln(n/mu)] = 2 mu h(r), r = (n - mu)/mu,
// h(r) = (1+r) ln(1+r) - r, by its alternating series for |r| < 1/4. diff: n - mu, which a caller
// may hold more exactly than the rounded mu gives it.
__device__ __forceinline__ float deviance(float n, float mu, float diff) {
    if (n == 0.f) return 2.f * mu;
    const float r = diff / mu;
    float h;
    if (fabsf(r) < 0.25f) {
        // h = sum_{j>=2} (-1)^j r^j / (j (j-1))
        float acc = 0.f;
#pragma unroll
        for (int j = 14; j >= 2; --j) {
            const float cj = ((j & 1) ? -1.f : 1.f) / (float)(j * (j - 1));
            acc = fmaf(acc, r, cj);
        }
        h = acc * r * r;
    } else {
        h = (1.f + r) * log1pf(r) - r;
    }
    return 2.f * mu * h;
}

// Parameter access: pv = value, pd = value - theta0, pl = the rounding residual of pv (see PP).
struct ParVecs {
    const float *pv, *pd, *pl;
};

// A parameter as the float pair h + l: h = its float value, l = the exact rounding residual
// (theta0_f - h) + delta + theta0_lo. Products x * theta are then formed as fma(x, l, x h),
// so the kernels evaluate at the caller's double-precision point, not at its float rounding
// (high-statistics normalisations have enough curvature for that rounding to show).
struct PP {
    float h, l;
};

// the residual l of parameter p, for a vector of them
__device__ __forceinline__ float presid(const DevModel &m, float h, float delta, int p) {
    return ((m.theta0_f[p] - h) + delta) + m.theta0_lo[p];
}

__device__ __forceinline__ PP ppair(const ParVecs &q, int p, float dflt) {
    return p < 0 ? PP{dflt, 0.f} : PP{q.pv[p], q.pl[p]};
}

__device__ __forceinline__ float pmul(PP a, float x) { return fmaf(x, a.l, x * a.h); }

// Status bits raised during an evaluation
constexpr int kStMuNonpos = 1;
constexpr int kStEscale = 2;

// Energy map of dataset d in grid units: displacement D(e) = (a0 + (a1-1) e + a2 e^2) / de.
struct EMap {
    float a0, a1m1, a2, inv_de, inv_slope, de;   // inv_slope: 1 / slope at mid grid, nearly (a first guess)
    __device__ __forceinline__ float disp(float e) const {
        return fmaf(fmaf(a2, e, a1m1), e, a0) * inv_de;
    }
    __device__ __forceinline__ float slope(float e) const { return 1.f + a1m1 + 2.f * a2 * e; }
};

// ---- area-conserving spline remap --------------------------------------------------------
// The grid's cumulative content C(e_k) is interpolated on each bin by the cubic Hermite
// polynomial with end slopes de f(e_k) = S_k = (u_{k-1} + u_k) / 2 (u_0, u_{N-1} at the ends):
//   F(e_k + t de) = C(e_k) + G_k(t),  G_k(t) = u_k h01(t) + S_k h10(t) + S_{k+1} h11(t),
// which keeps every bin's content and has a continuous density. The corrected spectrum is
// v_j = F(x_{j+1}) - F(x_j), x_j = E'^{-1}(e_j), evaluated locally as
//   v_j = sum_{k0 <= k < k1} u_k + G_{k1}(t1) - G_{k0}(t0)
// with each x on the grid as e + r (exact integer edge index + small FP32 offset r).
__device__ __forceinline__ float hermite_S(const float *u, int k, int N) {
    return k <= 0 ? u[0] : (k >= N ? u[N - 1] : 0.5f * (u[k - 1] + u[k]));
}

__device__ __forceinline__ float hermite_G(const float *u, int k, float t, int N) {
    const float t2 = t * t, t3 = t2 * t;
    const float h01 = fmaf(-2.f, t3, 3.f * t2), h10 = t3 - 2.f * t2 + t, h11 = t3 - t2;
    return fmaf(u[k], h01, fmaf(hermite_S(u, k, N), h10, hermite_S(u, k + 1, N) * h11));
}

// r with E'(e_e + r de) = e_e (two Newton steps from -D(e_e); |r| is a few bins at most)
template <class Map>
__device__ __forceinline__ float edge_inv_r(const float *e_edge, const Map &em, int e) {
    const float xe = e_edge[e];
    float r = -em.disp(xe);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float x = fmaf(r, em.de, xe);
        r -= (r + em.disp(x)) / em.slope(x);
    }
    return r;
}

// bin k and fraction t of the grid position e + r, clamped to the grid: below it (0, 0)
// (F = 0), above it (N - 1, 1) (F = total); `inside` tells whether it was on the grid
__device__ __forceinline__ void edge_bin(int e, float r, int N, int &k, float &t, bool &inside) {
    const float fl = floorf(r);
    k = e + (int)fl;
    t = r - fl;
    inside = true;
    if (k < 0) {
        k = 0;
        t = 0.f;
        inside = false;
    } else if (k >= N) {
        k = N - 1;
        t = 1.f;
        inside = false;
    }
}

// The inverse images of the grid edges, found once per evaluation and read by the remap and its
// adjoint (which look at five or six edges per bin): bin k and fraction t of x_e (see edge_bin),
// k + kEdgeOff where x_e is off the grid, and r.
constexpr int kEdgeOff = 1 << 16;
struct EdgeTab {
    int *k;
    float *t, *r;
};

template <class Map>
__device__ __forceinline__ void edge_store(const EdgeTab &T, const float *e_edge, const Map &em, int e, int N) {
    const float r = edge_inv_r(e_edge, em, e);
    int k;
    float t;
    bool in;
    edge_bin(e, r, N, k, t, in);
    T.k[e] = in ? k : k + kEdgeOff;
    T.t[e] = t;
    T.r[e] = r;
}

// v_j for target bin j
__device__ __forceinline__ float spline_target(const float *u, const EdgeTab &T, int j, int N) {
    const int k0 = T.k[j] & (kEdgeOff - 1), k1 = T.k[j + 1] & (kEdgeOff - 1);
    float acc = 0.f;
#pragma unroll 1
    for (int k = k0, it = 0; k < k1 && it < 64; ++k, ++it) acc += u[k];
    return acc + (hermite_G(u, k1, T.t[j + 1], N) - hermite_G(u, k0, T.t[j], N));
}

// Adjoint of the spline remap for source bin i: d(-2lnL)/du_i. With w_e = gv_{e-1} - gv_e the
// weight of F(x_e) (gv outside the grid 0), dF(x_e)/du_i is 1 for i < k_e (the cumulative)
// plus the Hermite weights of u_i in G_{k_e}; the cumulative part sums to gv_{e*-1}, e* the
// first edge with k_e > i.
__device__ __forceinline__ float spline_adjoint_source(const float *gv, const EdgeTab &T, int i, int N) {
    auto kb = [&](int e, int &k, float &t) {
        k = T.k[e] & (kEdgeOff - 1);
        t = T.t[e];
    };
    // e*: start from the inverse shift at edge i and walk to the first edge with k_e > i
    int e = min(max(i + 1 - (int)floorf(T.r[i]), 0), N + 1);
    int k;
    float t;
#pragma unroll 1
    for (int it = 0; it < 64 && e > 0; ++it) {   // step down while the edge before is past i
        kb(e - 1, k, t);
        if (k <= i) break;
        --e;
    }
#pragma unroll 1
    for (int it = 0; it < 64 && e <= N; ++it) {  // step up while this edge is not past i
        kb(e, k, t);
        if (k > i) break;
        ++e;
    }
    float g = (e >= 1 && e <= N) ? gv[e - 1] : 0.f;
    // local Hermite weights: edges with k_e in [i - 1, i + 1] lie around e*
    auto local = [&](int ee) -> bool {
        int kk;
        float tt;
        kb(ee, kk, tt);
        if (kk < i - 1 || kk > i + 1) return false;
        const float we = (ee >= 1 ? gv[ee - 1] : 0.f) - (ee <= N - 1 ? gv[ee] : 0.f);
        const float t2 = tt * tt, t3 = t2 * tt;
        const float h01 = fmaf(-2.f, t3, 3.f * t2), h10 = t3 - 2.f * t2 + tt, h11 = t3 - t2;
        float c = 0.f;
        if (kk == i) c = h01 + (kk == 0 ? h10 : 0.5f * h10) + (kk == N - 1 ? h11 : 0.5f * h11);
        else if (kk == i + 1) c = 0.5f * h10;   // S_{i+1} = (u_i + u_{i+1}) / 2
        else c = 0.5f * h11;                    // kk == i - 1: S_i = (u_{i-1} + u_i) / 2
        g = fmaf(we, c, g);
        return true;
    };
#pragma unroll 1
    for (int ee = e - 1, it = 0; ee >= 0 && it < 64; --ee, ++it)
        if (!local(ee)) break;
#pragma unroll 1
    for (int ee = e, it = 0; ee <= N && it < 64; ++ee, ++it)
        if (!local(ee)) break;
    return g;
}

// Edge e's share of d(-2lnL)/d(a0, a1, a2): w_e f(x_e) dx_e/da_i, dx/da_i = -x^i / E''(x)
// (f the spline's density per MeV, 0 off the grid); added to ep[0..2].
template <class Map>
__device__ __forceinline__ void spline_adjoint_edge(const float *u, const float *gv, const float *e_edge,
                                                    const Map &em, const EdgeTab &T, int e, int N, float *ep) {
    const int k = T.k[e];
    if (k & kEdgeOff) return;
    const float r = T.r[e], t = T.t[e];
    const float we = (e >= 1 ? gv[e - 1] : 0.f) - (e <= N - 1 ? gv[e] : 0.f);
    const float t2 = t * t;
    const float dG = fmaf(u[k], 6.f * (t - t2), fmaf(hermite_S(u, k, N), 3.f * t2 - 4.f * t + 1.f,
                                                      hermite_S(u, k + 1, N) * (3.f * t2 - 2.f * t)));
    const float x = fmaf(r, em.de, e_edge[e]);
    const float q = -we * dG * em.inv_de / em.slope(x);
    ep[0] += q;
    ep[1] = fmaf(q, x, ep[1]);
    ep[2] = fmaf(q, x * x, ep[2]);
}

__device__ __forceinline__ EMap make_emap(const DevModel &m, const DevDataset &ds, const float *pv,
                                          const float *pd) {
    EMap em;
    em.a0 = ds.esc_idx[0] >= 0 ? pv[ds.esc_idx[0]] : 0.f;
    em.a1m1 = ds.esc_idx[1] >= 0 ? ds.a1_off + pd[ds.esc_idx[1]] : 0.f;
    em.a2 = ds.esc_idx[2] >= 0 ? pv[ds.esc_idx[2]] : 0.f;
    em.inv_de = m.inv_de;
    em.inv_slope = __fdividef(1.f, em.slope(0.5f * (m.e_first + m.e_last)));
    em.de = m.de;
    return em;
}

// ------------------------------------------------------------------------------------
// Block-level evaluation of one parameter vector.
//
// What bounds it: a few hundred kFLOP per vector in a dozen dependent stages over a few hundred
// to a few thousand bins, so with one block per vector the time is the chain of barriers,
// reductions and load latencies, not arithmetic or bandwidth. So every stage runs over all
// datasets of the vector together (a "group": the datasets whose workspaces are held at once,
// DevModel::ws_group), with one barrier per stage for the group instead of one per dataset and
// stage, and the warps that one dataset leaves over start on the next (each dataset's bins
// begin at the warp where the previous dataset's ended).
// ------------------------------------------------------------------------------------
// Per-dataset workspace (floats), arrays of N_t rounded up to 4 unless noted:
//   u, v (-> gv), ts = t s, ptot, dp[n_osc] (dp[0] is reused for the shape gradient),
//   pcw[C] = w_c P_c per core, f0[max_reco], gmu[max_reco], and for the spline correction the
//   edge table (three arrays of N_t + 1), for the overlap rule the displacements D(e_k) of the
//   grid edges (N_t + 1, in edge.t). u is the signal, divided by the mapped width of
//   its bin under the overlap rule (every use of it there is divided by that width).
struct DsWs {
    float *u, *v, *ts, *ptot, *dp, *pcw, *f0, *gmu;
    EdgeTab edge;
};

__host__ __device__ inline int eval_ws_floats(int N_t, int C, int max_reco, int n_osc, int remap_mode) {
    return (remap_mode == FIT_REMAP_SPLINE ? 3 : 1) * ((N_t + 4) & ~3) + (4 + n_osc + C) * ((N_t + 3) & ~3) + 2 * ((max_reco + 3) & ~3);
}

__device__ __forceinline__ DsWs carve_ds_ws(float *base, int N_t, int C, int max_reco, int n_osc) {
    const int N4 = (N_t + 3) & ~3;
    DsWs w;
    w.u = base;
    w.v = w.u + N4;
    w.ts = w.v + N4;
    w.ptot = w.ts + N4;
    w.dp = w.ptot + N4;          // n_osc arrays (pitch N_t)
    w.pcw = w.dp + n_osc * N4;   // C arrays (pitch N_t)
    w.f0 = w.pcw + C * N4;       // max_reco
    w.gmu = w.f0 + ((max_reco + 3) & ~3);
    w.edge.t = w.gmu + ((max_reco + 3) & ~3);
    w.edge.r = w.edge.t + ((N_t + 4) & ~3);
    w.edge.k = reinterpret_cast<int *>(w.edge.r + ((N_t + 4) & ~3));
    return w;
}

// Two cores of a dataset: K L / pi (pair), flux share w, w p high and low part. A core that is not
// seen, or past the last one, has all of them 0: probability 1, weight 0.
struct alignas(16) CorePair {
    f32x2 klh, kll, w, wp, wpl, pad;
};

// Shared state of one evaluation (one per block).
struct EvalShared {
    typename OscTraits<6>::Coef kc;         // sin^2 coefficients (the first three for 4 parameters)
    float eta[kMaxOsc], eta_lo[kMaxOsc];
    PP nrm[FIT_MAX_DATASETS], eff[FIT_MAX_DATASETS];
    EMap em[FIT_MAX_DATASETS];
    PP rate[FIT_MAX_BACKGROUNDS];
    CorePair core[FIT_MAX_DATASETS][(FIT_MAX_CORES + 1) / 2];   // of the group's datasets
    int dl[FIT_MAX_DATASETS];               // datasets of the current group
    int n;                                  // their number
    int bad;                                // 1: the dataset after them has an invalid energy map
    int status;                             // kSt* bits
    double nll;                             // sum over the datasets so far
    double nll_ds[FIT_MAX_DATASETS];        // the group's datasets
    float dup[FIT_MAX_DATASETS * 8 + 32];   // totals of parameters that receive several (in order)
    // warp totals: likelihood sums [dataset][warp][8], then energy-map sums [dataset][warp][4] and
    // survival / power sums [warp][32] (the two uses are barriers apart)
    float part[FIT_MAX_DATASETS * kMaxWarps * 8];
};

// Logical thread index of this thread in a stage whose datasets take `per` warps each: dataset
// number i starts at the warp where dataset i - 1 ended.
__device__ __forceinline__ int rot_tid(int i, int per) {
    const int nw = blockDim.x >> 5;
    int w = (int)(threadIdx.x >> 5) - (i * per) % nw;
    if (w < 0) w += nw;
    return w * 32 + (int)(threadIdx.x & 31);
}

// Group setup: the datasets `first`, ... of the mask, at most m.ws_group of them (E.dl, E.n),
// survival parameters and coefficients, normalisations, efficiencies, energy maps, powers,
// rates. A dataset whose energy map is not increasing with slope in (1/4, 4) on the grid ends
// the list (E.bad). Returns the dataset after the group. Starts and ends with a barrier.
template <int NOSC>
static __device__ int eval_setup(const DevModel &m, EvalShared &E, const ParVecs &q, uint32_t mask, int first,
                                 int group) {
    __syncthreads();
    const int tid = threadIdx.x, lane = tid & 31;
    int next = first;
    {   // every thread walks the mask (at most 8 datasets)
        int n = 0;
        bool bad = false;
        while (next < m.n_ds && n < group) {
            const int d = next++;
            if (!((mask >> d) & 1u)) continue;
            const DevDataset &ds = m.ds[d];
            const EMap em = make_emap(m, ds, q.pv, q.pd);
            const float s0 = em.slope(m.e_first), s1 = em.slope(m.e_last);
            if (!(s0 > 0.25f && s0 < 4.f && s1 > 0.25f && s1 < 4.f)) {
                bad = true;
                break;
            }
            if (tid == 32 + n) {
                E.dl[n] = d;
                E.em[n] = em;
                E.nrm[n] = ppair(q, ds.norm_idx, 1.f);
                E.eff[n] = ppair(q, ds.eff_idx, 1.f);
            }
            ++n;
        }
        if (tid == 0) {
            E.n = n;
            E.bad = bad;
        }
    }
    const int warp = tid >> 5;
    if (warp == 0) {
        // survival parameters: mass splittings as theta0_f + (theta0_lo + delta) inside the phase
        if (lane < NOSC) {
            const int p = m.osc_idx[lane];
            float h, l;
            if (osc_is_dm(m.osc_mode, lane)) {
                h = p >= 0 ? m.osc_th_f[lane] : m.osc_val[lane];
                l = p >= 0 ? m.osc_th_lo[lane] + q.pd[p] : m.osc_val_lo[lane];
            } else {
                h = p >= 0 ? q.pv[p] : m.osc_val[lane];
                l = 0.f;
            }
            // (normalised: the reduced phase must stay within a half)
            const F2 n = f2_norm(h, l);
            E.eta[lane] = n.h;
            E.eta_lo[lane] = n.l;
        }
        // the sin^2 coefficients from float pairs of the exact parameter values
        F2 e[NOSC];
#pragma unroll
        for (int i = 0; i < NOSC; ++i) {
            const int p = m.osc_idx[i];
            e[i] = p >= 0 ? f2_norm(q.pv[p], q.pl[p]) : F2{m.osc_val[i], m.osc_val_lo[i]};
        }
        const auto k = OscTraits<NOSC>::coef(m.osc_mode, e);
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < (int)(sizeof(k.hi) / sizeof(float)); ++i) {
                E.kc.hi[i] = k.hi[i];
                E.kc.lo[i] = k.lo[i];
            }
        }
    }
    // (every thread reads the mask itself: dataset number i of the group for core slots 16 i + c)
#pragma unroll 1
    for (int e = tid; e < 16 * group; e += blockDim.x) {
        const int c = e & 15;
        int d = first, left = e >> 4;
        while (d < m.n_ds && !(((mask >> d) & 1u) && left-- == 0)) ++d;
        if (d >= m.n_ds || c >= ((m.C + 1) & ~1)) continue;
        const DevDataset &ds = m.ds[d];
        const float w = c < m.C ? ds.w[c] : 0.f;
        const PP p = w != 0.f ? ppair(q, m.core_power_idx[c], 1.f) : PP{0.f, 0.f};
        const float wp = w * p.h;
        float *k = reinterpret_cast<float *>(&E.core[e >> 4][c >> 1]) + (c & 1);
        k[0] = w != 0.f ? ds.kl_hi[c] : 0.f;
        k[2] = w != 0.f ? ds.kl_lo[c] : 0.f;
        k[4] = w;
        k[6] = wp;
        k[8] = fmaf(w, p.l, fmaf(w, p.h, -wp));
    }
    if (warp == (int)(blockDim.x >> 5) - 1 && lane < m.n_bkg) E.rate[lane] = ppair(q, m.bkg[lane].rate_idx, 1.f);
    __syncthreads();
    return next;
}

// The survival sums of one true bin over the cores: pt = sum_c p_c w_c P_c, its derivatives dpt by
// the survival parameters, and corr, the part of the sum below FP32's rounding of P (the low
// parts of the sin^2 coefficients and of p_c w_c), which a caller adds where it still counts.
//
// Eq. 1 and the three-flavour formula are linear in sin^2 x_i, and their derivatives in sin^2 x_i
// and sin 2 x_i, with coefficients that no bin or core changes. So the loop over the cores sums
// p w sin^2 x_i and p w c sin x_i cos x_i, and the derivatives are formed once per bin: about 70
// instructions per bin and core instead of 125 with each core's derivatives in full (the 53 km
// model's signal stage: 60 200 cycles of 512 threads before).
//
// Two cores at a time in packed FP32 (f32x2): the packed instructions have no higher rate per FMA
// here (37 against 37 T/s measured) but are half the instructions, and issue slots, not the FMA
// units, are what this loop runs out of. The phase is taken negative (-y), which spares
// negations: sin^2 and cos are even, the products sin cos change sign and get it back at the end.
template <bool DERIV, int NOSC, int MODE>
struct CoreSums {
    static __device__ __forceinline__ void run(const EvalShared &E, int i, int C, float ih, float il, float *pcw,
                                               int stride, float &pt, float &corr, float (&dpt)[NOSC]) {
        constexpr int NT = MODE == FIT_OSC_EQ1 ? 2 : 3;
        constexpr int D0 = MODE == FIT_OSC_EQ1 ? 1 : 2;   // index of the first mass splitting
        const f32x2 one = pack2(1.f), m1 = pack2(-1.f), ih2 = pack2(ih), nih2 = pack2(-ih), il2 = pack2(il);
        f32x2 Q[NT], H[NT], p2 = pack2(0.f), lo = p2, nC[NT];
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            Q[j] = H[j] = p2;
            nC[j] = pack2(-E.kc.hi[j]);
        }
        const f32x2 ma = pack2(E.eta[D0]), nma = pack2(-E.eta[D0]), mal = pack2(E.eta_lo[D0]);
        const f32x2 mb = pack2(E.eta[3]), nmb = pack2(-E.eta[3]), mbl = pack2(E.eta_lo[3]);
#pragma unroll 1
        for (int c = 0; c < C; c += 2) {
            const CorePair &K = E.core[i][c >> 1];
            const f32x2 klh = K.klh, kll = K.kll, wp = K.wp;
            const f32x2 ch = mul2(klh, ih2), nch = mul2(klh, nih2);
            const f32x2 cl = fma2(kll, ih2, fma2(klh, il2, fma2(klh, ih2, nch)));
            f32x2 sa, ca, sb, cb, q[NT], h[NT];
            sincos_half2(neg_phase2(ma, nma, mal, ch, cl, m1), sa, ca);
            sincos_half2(neg_phase2(mb, nmb, mbl, ch, cl, m1), sb, cb);
            q[0] = mul2(sa, sa);
            q[1] = mul2(sb, sb);
            if (DERIV) {
                h[0] = mul2(sa, ca);
                h[1] = mul2(sb, cb);
            }
            if constexpr (NT == 3) {   // x32 = x31 - x21
                const f32x2 s2 = fma2(cb, mul2(sa, m1), mul2(sb, ca));
                q[2] = mul2(s2, s2);
                if (DERIV) h[2] = mul2(s2, fma2(sb, sa, mul2(cb, ca)));
            }
            f32x2 P = one;
#pragma unroll
            for (int j = 0; j < NT; ++j) P = fma2(nC[j], q[j], P);
            if (DERIV) {
                const float2 w = unpack2(mul2(K.w, P));
                pcw[c * stride] = w.x;
                if (c + 1 < C) pcw[(c + 1) * stride] = w.y;
            }
            p2 = fma2(P, wp, p2);
            lo = fma2(P, K.wpl, lo);
            const f32x2 wc = mul2(wp, ch);
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                Q[j] = fma2(wp, q[j], Q[j]);
                if (DERIV) H[j] = fma2(wc, h[j], H[j]);
            }
        }
        auto total = [](f32x2 v) {
            const float2 t = unpack2(v);
            return t.x + t.y;
        };
        {   // the two cores' halves, the rounding of their sum into the correction
            const float2 t = unpack2(p2);
            pt = t.x + t.y;
            const float bb = pt - t.x;
            corr = total(lo) + ((t.x - (pt - bb)) + (t.y - bb));
        }
        float Qs[NT], Hs[NT];
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            Qs[j] = total(Q[j]);
            corr = fmaf(-E.kc.lo[j], Qs[j], corr);
            if (DERIV) Hs[j] = total(H[j]);
        }
        if constexpr (!DERIV) return;
        constexpr float k2pi = -6.28318531f;   // d sin^2 x / d dm2 = 2 sin x cos x dx / d dm2, dx = pi c
        if constexpr (MODE == FIT_OSC_EQ1) {
            const float S13 = E.eta[0], S12 = E.eta[2];
            const float root = sqrtf(fmaxf(1.f - S13, 1e-12f)), c2 = 0.5f * (1.f + root);
            const float dc4 = -c2 * 0.5f / root;
            dpt[0] = -Qs[0] - dc4 * S12 * Qs[1];
            dpt[1] = -S13 * (k2pi * Hs[0]);
            dpt[2] = -c2 * c2 * Qs[1];
            dpt[3] = -c2 * c2 * S12 * (k2pi * Hs[1]);
        } else {
            const float s12 = E.eta[0], s13 = E.eta[1], c12 = 1.f - s12, c13 = 1.f - s13;
            const float S12 = 4.f * s12 * c12, S13 = 4.f * s13 * c13;
            dpt[0] = -c13 * c13 * 4.f * (1.f - 2.f * s12) * Qs[0] - S13 * (Qs[2] - Qs[1]);
            dpt[1] = 2.f * c13 * S12 * Qs[0] - 4.f * (1.f - 2.f * s13) * (c12 * Qs[1] + s12 * Qs[2]);
            dpt[2] = k2pi * (S13 * s12 * Hs[2] - c13 * c13 * S12 * Hs[0]);
            dpt[3] = -S13 * (k2pi * (c12 * Hs[1] + s12 * Hs[2]));
        }
    }
};

// The 3+1 formula: each core's probability and derivatives in full.
template <bool DERIV>
struct CoreSums<DERIV, 6, FIT_OSC_STERILE4> {
    static __device__ __forceinline__ void run(const EvalShared &E, int i, int C, float ih, float il, float *pcw,
                                               int stride, float &pt, float &corr, float (&dpt)[6]) {
        float eta[6], eta_lo[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            eta[j] = E.eta[j];
            eta_lo[j] = E.eta_lo[j];
            dpt[j] = 0.f;
        }
        pt = corr = 0.f;
        for (int c = 0; c < C; ++c) {
            const float *k = reinterpret_cast<const float *>(&E.core[i][c >> 1]) + (c & 1);
            const float klh = k[0], kll = k[2], w = k[4], wp = k[6], wpl = k[8];
            const float ch = klh * ih;
            const float cl = fmaf(kll, ih, fmaf(klh, il, fmaf(klh, ih, -ch)));
            float dP[6];
            const float P = survival_sterile(eta, eta_lo, E.kc, ch, cl, dP);
            if (DERIV) pcw[c * stride] = w * P;
            pt = fmaf(P, wp, pt);
            corr = fmaf(P, wpl, corr);
            if (DERIV) {
#pragma unroll
                for (int j = 0; j < 6; ++j) dpt[j] = fmaf(wp, dP[j], dpt[j]);
            }
        }
    }
};

// Stage A: u_k (and with DERIV the per-bin partials the adjoint needs), and the spline's edge table.
// Ends with a barrier.
template <bool DERIV, int NOSC, int MODE, bool GEN>
static __device__ __forceinline__ void st_signal_mode(const DevModel &m, const EvalShared &E, const ParVecs &q,
                                                      float *wsb) {
    const int N_t = m.N_t, nth = blockDim.x;
    const bool spline = GEN && m.remap_mode == FIT_REMAP_SPLINE;
#pragma unroll 1
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, N_t, m.C, m.max_reco, m.n_osc);
        const PP nrm = E.nrm[i];
        const EMap em = E.em[i];
#pragma unroll 1
        for (int k = rot_tid(i, (N_t + 31) >> 5); k < N_t; k += nth) {
            const float ih = m.inv_e_hi[k], il = m.inv_e_lo[k];
            const float e0 = m.e_edge[k], e1 = m.e_edge[k + 1];
            const int sp = ds.shape_idx[k];
            const float tk = ds.t[k];
            float pt, corr, dpt[NOSC];
            CoreSums<DERIV, NOSC, MODE>::run(E, i, m.C, ih, il, ws.pcw + k, N_t, pt, corr, dpt);
            const float ts = pmul(ppair(q, sp, 1.f), tk);
            if (DERIV) {
                ws.ts[k] = ts;
                ws.ptot[k] = pt;
#pragma unroll
                for (int j = 0; j < NOSC; ++j) ws.dp[j * N_t + k] = dpt[j];
            }
            // (ts pt + ts corr in one rounding: the correction is below pt's last bit)
            const float u = pmul(nrm, fmaf(ts, pt, ts * corr));
            if (spline) {
                ws.u[k] = u;
                edge_store(ws.edge, m.e_edge, em, k, N_t);
                if (k == N_t - 1) edge_store(ws.edge, m.e_edge, em, N_t, N_t);
            } else {
                const float d0 = em.disp(e0), d1 = em.disp(e1);
                ws.u[k] = u / (1.f + (d1 - d0));
                ws.edge.t[k] = d0;
                if (k == N_t - 1) ws.edge.t[N_t] = d1;
            }
        }
    }
    __syncthreads();
}

// GEN: the general build (any formula); else Eq. 1 or the three-flavour formula.
template <bool DERIV, bool GEN>
static __device__ __forceinline__ void st_signal(const DevModel &m, const EvalShared &E, const ParVecs &q, float *wsb) {
    if (GEN && m.osc_mode == FIT_OSC_STERILE4)
        st_signal_mode<DERIV, 6, FIT_OSC_STERILE4, GEN>(m, E, q, wsb);
    else if (m.osc_mode == FIT_OSC_EQ1)
        st_signal_mode<DERIV, 4, FIT_OSC_EQ1, GEN>(m, E, q, wsb);
    else
        st_signal_mode<DERIV, 4, FIT_OSC_VACUUM3, GEN>(m, E, q, wsb);
}

// Corrected content of target bin t under the overlap rule, from the sources' contents per mapped
// width u and the map's slope at mid grid. Source bin k covers [Y_k, Y_k+1] in
// grid units, Y_k = k + D(e_k); target t gathers the sources whose mapped interval overlaps
// [t, t+1]; overlaps are computed relative to the target (k - t is an exact small integer),
// which keeps them accurate in FP32.
__device__ __forceinline__ float overlap_target(const float *u, const float *D, float inv_slope, int t, int N_t) {
    // first source whose mapped upper edge lies above t: from k ~ t - D(t) / slope (exact for a linear
    // map), stepping down until the bracket is right; the sum steps up over what lies below t.
    // Neither is capped: the map is increasing, so both end, and at scales a few percent off 1
    // neither takes more than a step.
    int k = min(max(t - (int)floorf(D[t] * inv_slope) - 1, 0), N_t - 1);
    float dlo = D[k];
#pragma unroll 1
    while (k > 0 && (float)(k - t) + dlo > 0.f) dlo = D[--k];
    float acc = 0.f;
#pragma unroll 1
    for (; k < N_t; ++k) {
        const float dhi = D[k + 1];
        const float ylo = (float)(k - t) + dlo;      // mapped edges relative to target t
        const float yhi = (float)(k + 1 - t) + dhi;
        if (ylo >= 1.f) break;
        const float ov = fminf(yhi, 1.f) - fmaxf(ylo, 0.f);
        if (ov > 0.f) acc = fmaf(u[k], ov, acc);
        dlo = dhi;
    }
    return acc;
}

// Stage B: v = M(a) u. Ends with a barrier. GEN: compiled with the spline option.
template <bool GEN>
static __device__ __forceinline__ void st_remap(const DevModel &m, const EvalShared &E, float *wsb) {
    const int N_t = m.N_t, nth = blockDim.x;
    const bool spline = GEN && m.remap_mode == FIT_REMAP_SPLINE;
#pragma unroll 1
    for (int i = 0; i < E.n; ++i) {
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, N_t, m.C, m.max_reco, m.n_osc);
        const float is = E.em[i].inv_slope;
#pragma unroll 1
        for (int t = rot_tid(i, (N_t + 31) >> 5); t < N_t; t += nth)
            ws.v[t] = spline ? spline_target(ws.u, ws.edge, t, N_t) : overlap_target(ws.u, ws.edge.t, is, t, N_t);
    }
    __syncthreads();
}

// out[4 g + e] (+ lo) = sum of a banded row times x, for warp units w0, w0 + nw, ... of U. One 16-byte
// load of the matrix and one x serve four products, eight loads in flight: the response comes
// from L2 (0.9 MB for the 53 km model's two detectors), and what counts besides bytes in flight
// is instructions: a warp per row with its tree and addresses took 50 000 of the 358 000 warp
// instructions of an evaluation there, this 9 000. The sum over the lanes of an output
// group keeps its rounding errors (two-sums; into lo when it is not null).
__device__ __forceinline__ void band_product(const BandUnits &U, const float *x, int w0, int nw, PP scale, float *out,
                                             float *lo) {
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int w = w0; w < U.n; w += nw) {
        const int2 st = U.steps[w];
        const float *xs = x + U.start[w * 32 + lane];
        const float4 *r = U.entry + st.x + lane;
        float a[4] = {0.f, 0.f, 0.f, 0.f}, b[4] = {0.f, 0.f, 0.f, 0.f};
        int k = 0;
#pragma unroll 1
        for (; k + 8 <= st.y; k += 8, r += 256, xs += 8) {
            float4 q[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) q[u] = r[32 * u];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float v = xs[u];
                float (&t)[4] = (u & 1) ? b : a;
                t[0] = fmaf(q[u].x, v, t[0]);
                t[1] = fmaf(q[u].y, v, t[1]);
                t[2] = fmaf(q[u].z, v, t[2]);
                t[3] = fmaf(q[u].w, v, t[3]);
            }
        }
#pragma unroll 1
        for (; k < st.y; ++k, r += 32, ++xs) {
            const float4 q = *r;
            const float v = *xs;
            a[0] = fmaf(q.x, v, a[0]);
            a[1] = fmaf(q.y, v, a[1]);
            a[2] = fmaf(q.z, v, a[2]);
            a[3] = fmaf(q.w, v, a[3]);
        }
        float h[4], l[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            h[e] = a[e] + b[e];
            const float bb = h[e] - a[e];
            l[e] = (a[e] - (h[e] - bb)) + (b[e] - bb);
        }
#pragma unroll 1
        for (int o = U.parts >> 1; o > 0; o >>= 1) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float g = __shfl_xor_sync(0xffffffffu, h[e], o), gl = __shfl_xor_sync(0xffffffffu, l[e], o);
                const float t = h[e] + g, bb = t - h[e];
                l[e] = (l[e] + gl) + ((h[e] - (t - bb)) + (g - bb));
                h[e] = t;
            }
        }
        const int x0 = w * 32 + lane;
        if ((x0 & (U.parts - 1)) == 0) {
            const int g = 4 * (x0 / U.parts);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (g + e >= U.outs) break;
                if (lo) {
                    out[g + e] = h[e];
                    lo[g + e] = l[e];
                } else {
                    out[g + e] = pmul(scale, h[e]);
                }
            }
        }
    }
}

// Stage C: fold into reco bins, f0 = R v (before the efficiency), banded rows. The sums are float
// pairs (low parts in gmu until st_lik): a bin's dD/dmu = 2 (mu - n) / mu is the difference of
// near equals, so the last bits of mu are what the gradient near a minimum is made of. Ends with
// a barrier.
static __device__ __forceinline__ void st_fold(const DevModel &m, const EvalShared &E, float *wsb) {
    const int nw = blockDim.x >> 5;
#pragma unroll 1
    for (int i = 0; i < E.n; ++i) {
        const BandUnits &U = m.det[m.ds[E.dl[i]].det].fold;
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, m.N_t, m.C, m.max_reco, m.n_osc);
        band_product(U, ws.v, rot_tid(i, U.n) >> 5, nw, PP{1.f, 0.f}, ws.f0, ws.gmu);
    }
    __syncthreads();
}

// Expected counts of one bin as sig + rest: sig the efficiency x fold, rest what its rounding left out
// and the backgrounds, so that a caller can form mu - n = (sig - n) + rest without rounding at the
// size of mu (fold pair f0 + f1). tm / sh receive the templates and 1 + delta of the dataset's
// backgrounds (the loads of all of them in flight together).
__device__ __forceinline__ float bin_mu(const DevModel &m, const EvalShared &E, int i, const DevDataset &ds,
                                        const ParVecs &q, float f0, float f1, int j, int nb, float (&tm)[kMaxBkgDs],
                                        float (&sh)[kMaxBkgDs], float &rest) {
    int si[kMaxBkgDs];
#pragma unroll
    for (int b = 0; b < kMaxBkgDs; ++b) {
        const DevBkg &bk = m.bkg[ds.bkg_begin + min(b, max(nb - 1, 0))];
        tm[b] = b < nb ? bk.tmpl[j] : 0.f;
        si[b] = b < nb ? bk.shape_idx[j] : -1;
    }
    const PP eff = E.eff[i];
    const float sig = f0 * eff.h;
    const float low = fmaf(f1, eff.h, fmaf(f0, eff.l, fmaf(f0, eff.h, -sig)));
    float bg = 0.f;
#pragma unroll
    for (int b = 0; b < kMaxBkgDs; ++b) {
        if (b >= nb) break;
        const float del = si[b] >= 0 ? q.pv[si[b]] : 0.f;
        sh[b] = 1.f + del;
        bg += pmul(E.rate[ds.bkg_begin + b], fmaf(tm[b], del, tm[b]));
    }
    rest = bg + low;
    return sig;
}

// Expected counts of the group's datasets into mu (the whole data vector). Ends with a barrier.
static __device__ __forceinline__ void st_mu(const DevModel &m, const EvalShared &E, const ParVecs &q, float *wsb,
                                             float *mu) {
    const int nth = blockDim.x;
#pragma unroll 1
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, m.N_t, m.C, m.max_reco, m.n_osc);
#pragma unroll 1
        for (int j = rot_tid(i, (ds.n_reco + 31) >> 5); j < ds.n_reco; j += nth) {
            float tm[kMaxBkgDs], sh[kMaxBkgDs];
            float rest;
            const float sig = bin_mu(m, E, i, ds, q, ws.f0[j], ws.gmu[j], j, ds.bkg_end - ds.bkg_begin, tm, sh, rest);
            mu[ds.data_off + j] = sig + rest;
        }
    }
    __syncthreads();
}

// Stage C2: backgrounds, deviance, dD/dmu (gmu) from the folded spectra f0, and the warp totals
// of the deviance and of the efficiency and rate gradients (E.part). Bins with mu <= 0 raise
// kStMuNonpos. Ends with a barrier; lik_finish adds the totals up.
template <bool GRAD>
static __device__ __forceinline__ void st_lik(const DevModel &m, EvalShared &E, const ParVecs &q, const float *data,
                                              float *wsb) {
    const int nth = blockDim.x, lane = threadIdx.x & 31;
#pragma unroll 1
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, m.N_t, m.C, m.max_reco, m.n_osc);
        const int nr = ds.n_reco, nb = ds.bkg_end - ds.bkg_begin;
        const int t0 = rot_tid(i, (nr + 31) >> 5);
        if ((t0 & ~31) >= nr) continue;      // this warp has no bin of this dataset
        float part[8];   // deviance, d/d eff, d/d rate_b
#pragma unroll
        for (int b = 0; b < 8; ++b) part[b] = 0.f;
#pragma unroll 1
        for (int j = t0; j < nr; j += nth) {
            const float n = data[ds.data_off + j], f0 = ws.f0[j];
            float tm[kMaxBkgDs], sh[kMaxBkgDs], rest;
            const float sig = bin_mu(m, E, i, ds, q, f0, ws.gmu[j], j, nb, tm, sh, rest);
            const float mu = sig + rest, diff = (sig - n) + rest;   // mu - n
            if (!(mu > 0.f)) {
                atomicOr(&E.status, kStMuNonpos);
                continue;
            }
            part[0] += deviance(n, mu, -diff);
            const float g = 2.f * diff / mu;
            ws.gmu[j] = g;
            if (GRAD) {
                part[1] = fmaf(g, f0, part[1]);
#pragma unroll
                for (int b = 0; b < kMaxBkgDs; ++b) {
                    if (b >= nb) break;
                    part[2 + b] = fmaf(g * tm[b], sh[b], part[2 + b]);
                }
            }
        }
        __syncwarp();
        const float tot = warp_sum_split<8>(part);
        if ((lane & 3) == 0) E.part[(i * kMaxWarps + (t0 >> 5)) * 8 + (lane >> 2)] = tot;
    }
    __syncthreads();
}

// Total over n <= kMaxWarps warps of the floats p[0], p[stride], ..., in double, by four
// neighbouring lanes (sub = lane & 3); on each of them. A double addition has a latency of 66
// cycles here, so four lanes halve the chain of a lane per total (which measured 5 000 cycles
// over three datasets, one warp working through them), and all totals of a stage run at once
// on as many warps as they need.
__device__ __forceinline__ double quad_total(const float *p, int stride, int n, int sub) {
    double s = 0.0;
#pragma unroll 1
    for (int w = sub; w < n; w += 4) s += (double)p[w * stride];
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    return s;
}

// After st_lik: the group's likelihood sums in double (E.nll_ds), and with GRAD the efficiency and
// rate gradients into grad; totals whose parameter receives several are left in E.dup for
// lik_dups, a barrier later.
template <bool GRAD>
static __device__ __forceinline__ void lik_finish(const DevModel &m, EvalShared &E, float *grad) {
    const int nw = blockDim.x >> 5, sub = threadIdx.x & 3;
#pragma unroll 1
    for (int v0 = 0; v0 < 8 * E.n; v0 += blockDim.x >> 2) {
        const int v = v0 + (int)(threadIdx.x >> 2), i = v >> 3, q = v & 7;
        if ((v & ~7) >= 8 * E.n) break;   // uniform over the warp
        const DevDataset &ds = m.ds[E.dl[i]];
        const double s = quad_total(E.part + (int64_t)i * kMaxWarps * 8 + q, 8, min(nw, (ds.n_reco + 31) >> 5), sub);
        if (sub != 0) continue;
        if (q == 0) E.nll_ds[i] = s;
        if (GRAD && q >= 1) {
            const int p = q == 1 ? ds.eff_idx : q - 2 < ds.bkg_end - ds.bkg_begin ? m.bkg[ds.bkg_begin + q - 2].rate_idx : -1;
            if (p >= 0) {
                if ((ds.lik_dup >> q) & 1)
                    E.dup[v] = (float)s;
                else
                    grad[p] += (float)s;
            }
        }
    }
}

// One thread, a barrier after lik_finish: the sum of the group's -2lnL and (grad) the totals left
// in E.dup, in order.
static __device__ __forceinline__ void lik_dups(const DevModel &m, EvalShared &E, float *grad) {
    double nll = E.nll;
#pragma unroll 1
    for (int i = 0; i < E.n; ++i) nll += E.nll_ds[i];
    E.nll = nll;
    if (grad == nullptr) return;
#pragma unroll 1
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
#pragma unroll 1
        for (int left = ds.lik_dup; left; left &= left - 1) {
            const int q = __ffs(left) - 1;
            const int p = q == 1 ? ds.eff_idx : m.bkg[ds.bkg_begin + q - 2].rate_idx;
            grad[p] += E.dup[i * 8 + q];
        }
    }
}

// Background-shape gradient: a thread per shape parameter sums its (background, bin) pairs of
// the group's datasets in a fixed order (several datasets may share a shape).
static __device__ __forceinline__ void st_bkg_shape(const DevModel &m, const EvalShared &E, float *wsb, float *grad) {
#pragma unroll 1
    for (int p = threadIdx.x; p < m.n_bs; p += blockDim.x) {
        float s = 0.f;
#pragma unroll 1
        for (int r = m.bs_ptr[p]; r < m.bs_ptr[p + 1]; ++r) {
            const BkgShapeRef ref = m.bs_ref[r];
#pragma unroll 1
            for (int i = 0; i < E.n; ++i) {
                if (E.dl[i] != ref.d) continue;
                const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, m.N_t, m.C, m.max_reco, m.n_osc);
                s += ws.gmu[ref.j] * E.rate[ref.q].h * ref.tmpl;
            }
        }
        grad[m.bs_param[p]] += s;
    }
}

// Stage D: adjoint of the fold, v <- gv = eff R^T gmu. No barrier.
static __device__ __forceinline__ void st_adjoint_fold(const DevModel &m, const EvalShared &E, float *wsb) {
    const int nw = blockDim.x >> 5;
#pragma unroll 1
    for (int i = 0; i < E.n; ++i) {
        const BandUnits &U = m.det[m.ds[E.dl[i]].det].adj;
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, m.N_t, m.C, m.max_reco, m.n_osc);
        // (v is dead after the fold)
        band_product(U, ws.gmu, rot_tid(i, U.n) >> 5, nw, E.eff[i], ws.v, nullptr);
    }
}

// Stage E: adjoint of the energy map and of the signal from gv (in v); leaves d(-2lnL)/ds of each
// bin in dp[0] and the warp totals of the energy-map, normalisation, survival and power
// gradients in E.part. Needs u/ts/ptot/dp/pcw (st_signal<true>). Ends with a barrier.
template <int NC, int NOSC, bool GEN>
static __device__ __forceinline__ void st_adjoint_rest_n(const DevModel &m, EvalShared &E, float *wsb) {
    const int N_t = m.N_t, C = m.C, nth = blockDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool spline = GEN && m.remap_mode == FIT_REMAP_SPLINE;
    float eo[NOSC], ec[NC];   // d/d eta, d/d power_c (NC >= C), over all datasets of the group
#pragma unroll
    for (int j = 0; j < NOSC; ++j) eo[j] = 0.f;
#pragma unroll
    for (int c = 0; c < NC; ++c) ec[c] = 0.f;
#pragma unroll 1
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, N_t, C, m.max_reco, m.n_osc);
        const EMap em = E.em[i];
        const PP nrm = E.nrm[i];
        const float *gv = ws.v;
        float ep[4] = {0.f, 0.f, 0.f, 0.f};   // d/da0, d/da1, d/da2, d/d norm
#pragma unroll 1
        for (int k = rot_tid(i, (N_t + 31) >> 5); k < N_t; k += nth) {
            float gu = 0.f;
            if (spline) {
                gu = spline_adjoint_source(gv, ws.edge, k, N_t);
                spline_adjoint_edge(ws.u, gv, m.e_edge, em, ws.edge, k, N_t, ep);
                if (k == N_t - 1) spline_adjoint_edge(ws.u, gv, m.e_edge, em, ws.edge, N_t, N_t, ep);
            } else {
                // per source k: gu = sum_t F_kt gv_t; A0 = (gu - gv(floor Y_k)) / w,
                // A1 = (gv(floor Y_k+1) - gu) / w
                const float e0 = m.e_edge[k], e1 = m.e_edge[k + 1];
                const float d0 = ws.edge.t[k], d1 = ws.edge.t[k + 1];
                const float w = 1.f + (d1 - d0), iw = 1.f / w;
                const int f0i = (int)floorf(d0), f1i = (int)floorf(d1);
                const int t0 = k + f0i, t1 = k + 1 + f1i;
#pragma unroll 1
                for (int t = max(t0, 0); t <= min(t1, N_t - 1); ++t) {
                    const float ylo = (float)(k - t) + d0, yhi = (float)(k + 1 - t) + d1;
                    const float ov = fminf(yhi, 1.f) - fmaxf(ylo, 0.f);
                    if (ov > 0.f) gu = fmaf(ov, gv[t], gu);
                }
                gu *= iw;
                const float g0 = (t0 >= 0 && t0 < N_t) ? gv[t0] : 0.f;
                const float g1 = (t1 >= 0 && t1 < N_t) ? gv[t1] : 0.f;
                const float uk = ws.u[k];   // (already per mapped width)
                const float A0 = uk * (gu - g0), A1 = uk * (g1 - gu);
                ep[0] += (A0 + A1) * em.inv_de;
                ep[1] += (A0 * e0 + A1 * e1) * em.inv_de;
                ep[2] += (A0 * e0 * e0 + A1 * e1 * e1) * em.inv_de;
            }
            const float ts = ws.ts[k], pt = ws.ptot[k];
            const float gb = pmul(nrm, gu * ts);    // d nll / d(ptot)
#pragma unroll
            for (int j = 0; j < NOSC; ++j) eo[j] = fmaf(gb, ws.dp[j * N_t + k], eo[j]);
            ep[3] = fmaf(gu * ts, pt, ep[3]);
#pragma unroll
            for (int c = 0; c < NC; ++c)
                if (c < C) ec[c] = fmaf(gb, ws.pcw[c * N_t + k], ec[c]);
            ws.dp[k] = pmul(nrm, gu * ds.t[k] * pt);    // d nll / d s for this bin (dp[0] reused)
        }
        __syncwarp();
        const float tot = warp_sum_split<4>(ep);
        if ((lane & 7) == 0) E.part[(i * kMaxWarps + warp) * 4 + (lane >> 3)] = tot;
    }
    float *pw = E.part + FIT_MAX_DATASETS * kMaxWarps * 4 + warp * 32;
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = j < NOSC ? eo[j] : (j - NOSC < NC ? ec[j - NOSC < NC ? j - NOSC : 0] : 0.f);
    const float t8 = warp_sum_split<8>(v);
    if ((lane & 3) == 0) pw[lane >> 2] = t8;
    if constexpr (NC > 8 - NOSC) {   // the cores past the first 8 - NOSC
        constexpr int c0 = 8 - NOSC;
        float w[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) w[c] = c0 + c < NC ? ec[c0 + c < NC ? c0 + c : 0] : 0.f;
        const float t16 = warp_sum_split<16>(w);
        if ((lane & 1) == 0) pw[8 + (lane >> 1)] = t16;
    }
    __syncthreads();
}

// Stage F, after stage E: its totals in double into grad, and the shape reweights: the bins of
// each distinct shape parameter (CSR) summed by sp_lanes lanes. Ends with a barrier.
template <int NOSC>
static __device__ __forceinline__ void st_adjoint_finish(const DevModel &m, EvalShared &E, float *wsb, float *grad) {
    const int tid = threadIdx.x, nw = blockDim.x >> 5, nth = blockDim.x;
    {
        // totals: four per dataset, then the survival parameters and powers; four lanes each,
        // from the last warp down (the shapes below start at the first)
        const int nmap = 4 * E.n, nv = nmap + NOSC + m.C, sub = tid & 3;
#pragma unroll 1
        for (int v0 = 0; v0 < nv; v0 += nth >> 2) {
            const int v = v0 + ((nth - 1 - tid) >> 2);
            if (v0 + (((nth - 1 - (tid | 31))) >> 2) >= nv) break;   // uniform over the warp
            const bool map = v < nmap;
            const int i = v >> 2, q = map ? (v & 3) : v - nmap;
            const float *p = map ? E.part + (int64_t)i * kMaxWarps * 4 + q
                                 : E.part + FIT_MAX_DATASETS * kMaxWarps * 4 + min(q, 31);
            const double s = quad_total(p, map ? 4 : 32, v < nv ? nw : 0, sub);
            if (sub != 0 || v >= nv) continue;
            const DevDataset &ds = m.ds[E.dl[map ? i : 0]];
            const int pi = map ? (q < 3 ? ds.esc_idx[q] : ds.norm_idx) : q < NOSC ? m.osc_idx[q] : m.core_power_idx[q - NOSC];
            const int dup = map ? ds.map_dup : m.osc_dup;
            if (pi < 0) continue;
            if ((dup >> q) & 1)
                E.dup[v] = (float)s;
            else
                grad[pi] += (float)s;
        }
    }
    if (m.any_map_dup) {
        __syncthreads();
        if (tid == 0) {
#pragma unroll 1
            for (int v = 0; v < 4 * E.n + NOSC + m.C; ++v) {
                const bool map = v < 4 * E.n;
                const int q = map ? (v & 3) : v - 4 * E.n;
                const DevDataset &ds = m.ds[E.dl[map ? v >> 2 : 0]];
                const int pi = map ? (q < 3 ? ds.esc_idx[q] : ds.norm_idx) : q < NOSC ? m.osc_idx[q] : m.core_power_idx[q - NOSC];
                if (pi >= 0 && (((map ? ds.map_dup : m.osc_dup) >> q) & 1)) grad[pi] += E.dup[v];
            }
        }
    }
    if (m.shared_roles) __syncthreads();
#pragma unroll 1
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
        const float *gs = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, m.N_t, m.C, m.max_reco, m.n_osc).dp;
        const int L = ds.sp_lanes, per = nth / L;   // lanes per parameter, parameters per pass
        const int work = ds.n_sp * L;
#pragma unroll 1
        for (int q0 = rot_tid(i, (work + 31) >> 5); q0 < ((work + 31) & ~31); q0 += per * L) {
            const int p = q0 / L, sub = q0 & (L - 1);
            const int4 sp = p < ds.n_sp ? ds.sp[p] : make_int4(0, 0, 0, 1);
            float s = 0.f;
            if (sp.w)
#pragma unroll 1
                for (int r = sub; r < sp.z; r += L) s += gs[sp.y + r];
            else
#pragma unroll 1
                for (int r = sub; r < sp.z; r += L) s += gs[ds.sp_k[sp.y + r]];
            for (int o = L >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (p < ds.n_sp && sub == 0) grad[sp.x] += s;
        }
        if (m.shared_roles) __syncthreads();
    }
    __syncthreads();
}

template <bool GEN>
static __device__ __forceinline__ void st_adjoint_rest(const DevModel &m, EvalShared &E, float *wsb, float *grad) {
    if (GEN && m.osc_mode == FIT_OSC_STERILE4) {
        if (m.C <= 2)
            st_adjoint_rest_n<2, 6, GEN>(m, E, wsb);
        else
            st_adjoint_rest_n<FIT_MAX_CORES, 6, GEN>(m, E, wsb);
        st_adjoint_finish<6>(m, E, wsb, grad);
    } else {
        if (m.C <= 2)
            st_adjoint_rest_n<2, 4, GEN>(m, E, wsb);
        else
            st_adjoint_rest_n<FIT_MAX_CORES, 4, GEN>(m, E, wsb);
        st_adjoint_finish<4>(m, E, wsb, grad);
    }
}

template <bool GEN>
static __device__ __forceinline__ int eval_setup_any(const DevModel &m, EvalShared &E, const ParVecs &q, uint32_t mask,
                                                     int first, int group) {
    if (GEN && m.osc_mode == FIT_OSC_STERILE4) return eval_setup<6>(m, E, q, mask, first, group);
    return eval_setup<4>(m, E, q, mask, first, group);
}

// The Poisson -2lnL of the datasets in `mask` and (GRAD) its theta gradient added to
// grad. wsb: ws_group dataset workspaces. Returns the -2lnL on every thread; E.status (cleared
// here) holds kSt* bits on failure. Starts and ends with a barrier.
template <bool GEN, bool GRAD>
static __device__ double eval_datasets(const DevModel &m, EvalShared &E, const ParVecs &q, uint32_t mask,
                                       const float *data, float *wsb, float *grad) {
    __syncthreads();
    if (threadIdx.x == 0) {
        E.status = 0;
        E.nll = 0.0;
    }
#pragma unroll 1
    for (int first = 0; first < m.n_ds;) {
        first = eval_setup_any<GEN>(m, E, q, mask, first, m.ws_group);
        if (E.n > 0) {
            st_signal<GRAD, GEN>(m, E, q, wsb);
            st_remap<GEN>(m, E, wsb);
            st_fold(m, E, wsb);
            st_lik<GRAD>(m, E, q, data, wsb);
        }
        if (E.status || E.bad) {   // block-uniform after the barriers
            __syncthreads();
            if (threadIdx.x == 0 && !E.status) E.status = kStEscale;
            __syncthreads();
            return INFINITY;
        }
        if (E.n == 0) continue;
        if (GRAD) {
            lik_finish<true>(m, E, grad);
            if (m.shared_roles) __syncthreads();
            st_bkg_shape(m, E, wsb, grad);
            st_adjoint_fold(m, E, wsb);
            __syncthreads();
            if (threadIdx.x == 0) lik_dups(m, E, grad);
            if (m.shared_roles) __syncthreads();
            st_adjoint_rest<GEN>(m, E, wsb, grad);
        } else {
            lik_finish<false>(m, E, nullptr);
            __syncthreads();
            if (threadIdx.x == 0) lik_dups(m, E, nullptr);
        }
    }
    __syncthreads();
    return E.nll;
}

// Expected counts of every dataset into mu (n_data floats). E.status as eval_datasets; datasets
// before an invalid energy map are written. Starts and ends with a barrier.
template <bool GEN>
static __device__ void expected_datasets(const DevModel &m, EvalShared &E, const ParVecs &q, float *wsb, float *mu) {
    __syncthreads();
    if (threadIdx.x == 0) E.status = 0;
#pragma unroll 1
    for (int first = 0; first < m.n_ds;) {
        first = eval_setup_any<GEN>(m, E, q, 0xffffffffu, first, m.ws_group);
        if (E.n > 0) {
            st_signal<false, GEN>(m, E, q, wsb);
            st_remap<GEN>(m, E, wsb);
            st_fold(m, E, wsb);
            st_mu(m, E, q, wsb, mu);
        }
        if (E.bad) {
            __syncthreads();
            if (threadIdx.x == 0) E.status = kStEscale;
            __syncthreads();
            return;
        }
    }
    __syncthreads();
}

// ------------------------------------------------------------------------------------
// Triangular matrix-vector products of the prior blocks: out_r = sum_c M(r, c) x_c over the rows
// of all blocks together, as tiles of up to 128 rows x 32 (64 for blocks of more than 512)
// columns, a warp per tile and four rows per lane: a column of a tile is one coalesced 16-byte
// load per lane and one broadcast of x, eight in flight (the factors come from L2: 0.7 MB per
// evaluation for the 400 x 400 block's two products). A tile leaves its partial sums at
// part[seg * tri_rows + row]; after a barrier tri_sum adds a row's segments in order. With
// 4-byte loads of 32-row tiles each product of that block took 13 500 cycles with 512 threads.
// x: by parameter index.
static __device__ __noinline__ void tri_apply(const DevModel &m, const TriTile *tiles, int n_tiles, const float *M,
                                                 const float *x, float *part) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
        int t = threadIdx.x >> 5;
    if (t >= n_tiles) return;
    TriTile T = tiles[t];
#pragma unroll 1
    while (true) {
        const TriTile next = tiles[min(t + nw, n_tiles - 1)];   // its latency behind this tile's
        const int p4 = T.pitch >> 2;
        const float4 *col = reinterpret_cast<const float4 *>(M + T.mat) + min(lane, p4 - 1);
        const float *xb = x + T.in0;
        const int *idx = m.blk_idx + T.idx;
        const bool seq = T.in0 >= 0;
        float4 s[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
        int c = 0;
        auto add = [](float4 &a, const float4 &r, float v) {
            a.x = fmaf(r.x, v, a.x);
            a.y = fmaf(r.y, v, a.y);
            a.z = fmaf(r.z, v, a.z);
            a.w = fmaf(r.w, v, a.w);
        };
#pragma unroll 1
        for (; c + 8 <= T.cols; c += 8, col += 8 * p4) {
            float4 r[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) r[u] = col[u * p4];
            if (seq) {
#pragma unroll
                for (int u = 0; u < 8; ++u) add(s[u & 1], r[u], xb[c + u]);
            } else {
#pragma unroll
                for (int u = 0; u < 8; ++u) add(s[u & 1], r[u], x[idx[c + u]]);
            }
        }
#pragma unroll 1
        for (; c < T.cols; ++c, col += p4) add(s[0], *col, seq ? xb[c] : x[idx[c]]);
        float *o = part + T.seg * m.tri_rows + T.out + 4 * lane;
        const float e[4] = {s[0].x + s[1].x, s[0].y + s[1].y, s[0].z + s[1].z, s[0].w + s[1].w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (4 * lane + u < T.rows) o[u] = e[u];
        t += nw;
        if (t >= n_tiles) break;
        T = next;
    }
}

__device__ __forceinline__ float tri_sum(const DevModel &m, const float *part, int row, bool upper) {
    const int x = m.tri_seg[row];
    const int s0 = upper ? (x >> 8) & 255 : 0, s1 = upper ? x >> 16 : x & 255;
    float t = part[s0 * m.tri_rows + row];
#pragma unroll 1
    for (int q = s0 + 1; q < s1; ++q) t += part[q * m.tri_rows + row];
    return t;
}

}  // namespace fitcore

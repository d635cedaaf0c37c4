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

struct DevDetector {
    int n_reco;
    int col_w;               // padded width of the column bands
    const int *row_lo;       // [N_r] first true bin of row j's band
    const int *row_len;      // [N_r] band length
    const int *row_off;      // [N_r] offset of the row's band in rrow
    const float *rrow;       // packed row bands
    const int *col_lo;       // [N_t] first reco row of column k's band
    const float *rcol;       // [col_w x N_t]: rcol[b * N_t + k] = R[col_lo[k] + b][k] (0 past the band)
    const float *rdense_hi;  // [N_r x ldt] dense response, TF32-exact high part (tensor-core fold)
    const float *rdense_lo;  // [N_r x ldt] R - rdense_hi
    const int *col_len;      // [N_t] band length of column k
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
    const int *sp_param;     // [n_sp] parameter index
    const int *sp_ptr;       // [n_sp + 1] CSR offsets into sp_k
    const int *sp_k;         // true bins of each shape parameter
    int lik_dup, map_dup;    // gradient totals whose parameter receives another total too: bits of
                             // (deviance, efficiency, rates) and of (a0, a1, a2, norm)
    int sp_lanes;            // lanes that share one shape parameter's sum (a power of two <= 32)
    float w[FIT_MAX_CORES];  // core flux shares
    float kl_hi[FIT_MAX_CORES], kl_lo[FIT_MAX_CORES];  // K L_dc / pi as a float pair (half-turns)
};

// One tile of a triangular matrix-vector product: out rows row0..row0+31 of a block (clipped to it),
// summed over `cols` <= kTriCols columns from col0.
constexpr int kTriCols = 64;
struct TriTile {
    int mat;                 // offset of the block's matrix (rows of n floats, column-major over the
                             // tile's lanes: element (out r, in c) at mat + c * n + r)
    int n;                   // block size
    int row0, col0, cols;
    int in0;                 // first input index when the block's parameters are consecutive, else -1
    int idx;                 // offset of the block's parameter indices (DevModel::blk_idx)
    int out;                 // concatenated row of the block's row 0
    int seg;                 // partial-sum slot
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
    double osc_val_d[kMaxOsc];   // the constant survival parameters in double
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
    const float *blk_L;      // lower Cholesky factor of V (row-major, dense)
    const float *blk_W;      // L^-1 (row-major, dense lower triangle)
    const double *blk_L64;   // L in double (final theta of a fit)
    const float *asimov;     // [n_data] expectation at theta0
    const int *slot_ds;      // [n_data] dataset of each data bin
    int ws_eval_floats;      // workspace of one dataset of one evaluation (a multiple of 4)
    int ws_group;            // datasets evaluated together (their workspaces are held at once)
    // matrix-vector products with the triangular prior blocks as tiles of 32 rows x kTriCols
    // columns (see tri_apply): tri_lo for L z / W d, tri_up for L^T g / W^T z
    const TriTile *tri_lo, *tri_up;
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
// Phase in half-turns: y = x / pi = (dm_hi + dm_lo) * (c_hi + c_lo), c = K L / (pi E), carried
// as a float pair. The probability depends on sin^2 x and sin 2x only, so y is reduced by
// its nearest integer, which is exact (y_hi - rint(y_hi) is representable), and sin, cos of
// pi r, |r| <= 1/2, come from sincospif. The pair keeps r accurate to ~1e-8 even at 50 km
// (y ~ 30), and no pi constant or multi-word reduction enters the arithmetic.
__device__ __forceinline__ void phase_sc(float dm, float dm_lo, float c_hi, float c_lo, float &s,
                                         float &c) {
    const float yh = dm * c_hi;
    const float yl = fmaf(dm, c_hi, -yh) + fmaf(dm, c_lo, dm_lo * c_hi);
    const float r = (yh - rintf(yh)) + yl;
    sincospif(r, &s, &c);
}

// sin^2(pi r) for |r| <= 1/2: u q(u), u = r^2, q a degree-7 polynomial fitted for the
// smallest largest absolute error (Lawson iteration; sin2pi_fit.py in this directory). Its
// FP32 evaluation is within 1.8e-7 of sin^2.
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

// sin^2 of the phase pi (dm + dm_lo)(c_hi + c_lo): the half-turn count reduced by its nearest
// integer as in the binned evaluation. Both pairs normalised (|low| <= ulp(high) / 2), so the
// reduced phase stays within 1/2 (the polynomial's range) up to rounding.
__device__ __forceinline__ float sin2_phase(float dm, float dm_lo, float c_hi, float c_lo) {
    const float yh = dm * c_hi;
    const float yl = fmaf(dm, c_hi, -yh) + fmaf(dm, c_lo, dm_lo * c_hi);
    return sin2pi((yh - rintf(yh)) + yl);
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

// P(L_dc, E_k) and dP/d(eta_i) for the four survival parameters.
//  mode FIT_OSC_EQ1:     eta = (sin^2 2th13, dm2_ee, sin^2 2th12, dm2_21), Eq. 1
//  mode FIT_OSC_VACUUM3: eta = (sin^2 th12, sin^2 th13, dm2_21, dm2_31), exact vacuum P
// eta_lo carries the low parts of the two mass splittings; dx = pi c (dx/d dm2).
__device__ __forceinline__ float survival_mode(int mode, const float (&eta)[4],
                                               const float (&eta_lo)[4], const OscCoef &k,
                                               float c_hi, float c_lo, float (&dP)[4]) {
    const float dx = 3.14159265358979f * c_hi;
    if (mode == FIT_OSC_EQ1) {
        const float S13 = eta[0], S12 = eta[2];
        const float root = sqrtf(fmaxf(1.f - S13, 1e-12f));
        const float c2 = 0.5f * (1.f + root);
        const float c4 = c2 * c2;
        float se, ce, s2, cc2;
        phase_sc(eta[1], eta_lo[1], c_hi, c_lo, se, ce);
        phase_sc(eta[3], eta_lo[3], c_hi, c_lo, s2, cc2);
        const float qe = se * se, q21 = s2 * s2;
        const float P = (1.f - cterm(k, 0, qe)) - cterm(k, 1, q21);
        const float dc4 = -c2 * 0.5f / root;
        dP[0] = -qe - dc4 * S12 * q21;
        dP[1] = -S13 * 2.f * se * ce * dx;
        dP[2] = -c4 * q21;
        dP[3] = -c4 * S12 * 2.f * s2 * cc2 * dx;
        return P;
    } else {
        const float s12 = eta[0], s13 = eta[1];
        const float c12 = 1.f - s12, c13 = 1.f - s13;
        const float S12 = 4.f * s12 * c12, S13 = 4.f * s13 * c13;
        float a21, b21, a31, b31;
        phase_sc(eta[2], eta_lo[2], c_hi, c_lo, a21, b21);
        phase_sc(eta[3], eta_lo[3], c_hi, c_lo, a31, b31);
        const float a32 = a31 * b21 - b31 * a21;   // sin(x31 - x21)
        const float b32 = b31 * b21 + a31 * a21;   // cos(x31 - x21)
        const float q21 = a21 * a21, q31 = a31 * a31, q32 = a32 * a32;
        const float d21 = 2.f * a21 * b21 * dx, d31 = 2.f * a31 * b31 * dx,
                    d32 = 2.f * a32 * b32 * dx;
        const float P = ((1.f - cterm(k, 0, q21)) - cterm(k, 1, q31)) - cterm(k, 2, q32);
        dP[0] = -c13 * c13 * 4.f * (1.f - 2.f * s12) * q21 - S13 * (q32 - q31);
        dP[1] = 2.f * c13 * S12 * q21 - 4.f * (1.f - 2.f * s13) * (c12 * q31 + s12 * q32);
        dP[2] = -c13 * c13 * S12 * d21 + S13 * s12 * d32;
        dP[3] = -S13 * (c12 * d31 + s12 * d32);
        return P;
    }
}

// The sin^2 coefficients of survival_mode from float pairs e of the exact parameter values.
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

__device__ __forceinline__ float survival(const DevModel &m, const float (&eta)[4],
                                          const float (&eta_lo)[4], const OscCoef &k,
                                          float c_hi, float c_lo, float (&dP)[4]) {
    return survival_mode(m.osc_mode, eta, eta_lo, k, c_hi, c_lo, dP);
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

// Survival of the formula with NOSC parameters: 4 (Eq. 1 or the three-flavour formula) or 6
// (the 3+1 formula).
template <int NOSC>
struct OscTraits;
template <>
struct OscTraits<4> {
    using Coef = OscCoefN<3>;
    static __device__ __forceinline__ float survival(int mode, const float (&eta)[4], const float (&eta_lo)[4],
                                                     const Coef &k, float c_hi, float c_lo, float (&dP)[4]) {
        return survival_mode(mode, eta, eta_lo, k, c_hi, c_lo, dP);
    }
    static __device__ __forceinline__ Coef coef(int mode, const F2 (&e)[4]) { return osc_coef(mode, e); }
};
template <>
struct OscTraits<6> {
    using Coef = OscCoefN<6>;
    static __device__ __forceinline__ float survival(int, const float (&eta)[6], const float (&eta_lo)[6],
                                                     const Coef &k, float c_hi, float c_lo, float (&dP)[6]) {
        return survival_sterile(eta, eta_lo, k, c_hi, c_lo, dP);
    }
    static __device__ __forceinline__ Coef coef(int, const F2 (&e)[6]) { return osc_coef_sterile(e); }
};

// Poisson deviance 2[mu - n + n ln(n/mu)] = 2 mu h(r), r = (n - mu)/mu,
// h(r) = (1+r) ln(1+r) - r, by its alternating series for |r| < 1/4.
__device__ __forceinline__ float deviance(float n, float mu) {
    if (n == 0.f) return 2.f * mu;
    const float r = (n - mu) / mu;
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
__device__ __forceinline__ float pval(const float *pv, int idx, float dflt) {
    return idx >= 0 ? pv[idx] : dflt;
}

// A parameter as the float pair h + l: h = its float value, l = the exact rounding residual
// (theta0_f - h) + delta + theta0_lo. Products x * theta are then formed as fma(x, l, x h),
// so the kernels evaluate at the caller's double-precision point, not at its float rounding
// (high-statistics normalisations have enough curvature for that rounding to show).
struct PP {
    float h, l;
};

__device__ __forceinline__ PP ppair(const DevModel &m, const float *pv, const float *pd, int p,
                                    float dflt) {
    if (p < 0) return PP{dflt, 0.f};
    const float h = pv[p];
    return PP{h, ((m.theta0_f[p] - h) + pd[p]) + m.theta0_lo[p]};
}

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
    float a0, a1m1, a2, inv_de, e_lo, de;
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

// v_j for target bin j
template <class Map>
__device__ __forceinline__ float spline_target(const float *u, const float *e_edge, const Map &em, int j, int N) {
    int k0, k1;
    float t0, t1;
    bool in0, in1;
    edge_bin(j, edge_inv_r(e_edge, em, j), N, k0, t0, in0);
    edge_bin(j + 1, edge_inv_r(e_edge, em, j + 1), N, k1, t1, in1);
    float acc = 0.f;
    for (int k = k0, it = 0; k < k1 && it < 64; ++k, ++it) acc += u[k];
    return acc + (hermite_G(u, k1, t1, N) - hermite_G(u, k0, t0, N));
}

// Adjoint of the spline remap for source bin i: d(-2lnL)/du_i. With w_e = gv_{e-1} - gv_e the
// weight of F(x_e) (gv outside the grid 0), dF(x_e)/du_i is 1 for i < k_e (the cumulative)
// plus the Hermite weights of u_i in G_{k_e}; the cumulative part sums to gv_{e*-1}, e* the
// first edge with k_e > i.
template <class Map>
__device__ __forceinline__ float spline_adjoint_source(const float *gv, const float *e_edge, const Map &em,
                                                       int i, int N) {
    auto kb = [&](int e, int &k, float &t) {
        bool in;
        edge_bin(e, edge_inv_r(e_edge, em, e), N, k, t, in);
    };
    // e*: start from the inverse shift at edge i and walk to the first edge with k_e > i
    int e = min(max(i + 1 - (int)floorf(edge_inv_r(e_edge, em, i)), 0), N + 1);
    int k;
    float t;
    for (int it = 0; it < 64 && e > 0; ++it) {   // step down while the edge before is past i
        kb(e - 1, k, t);
        if (k <= i) break;
        --e;
    }
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
    for (int ee = e - 1, it = 0; ee >= 0 && it < 64; --ee, ++it)
        if (!local(ee)) break;
    for (int ee = e, it = 0; ee <= N && it < 64; ++ee, ++it)
        if (!local(ee)) break;
    return g;
}

// Edge e's share of d(-2lnL)/d(a0, a1, a2): w_e f(x_e) dx_e/da_i, dx/da_i = -x^i / E''(x)
// (f the spline's density per MeV, 0 off the grid); added to ep[0..2].
template <class Map>
__device__ __forceinline__ void spline_adjoint_edge(const float *u, const float *gv, const float *e_edge,
                                                    const Map &em, int e, int N, float *ep) {
    const float r = edge_inv_r(e_edge, em, e);
    int k;
    float t;
    bool in;
    edge_bin(e, r, N, k, t, in);
    if (!in) return;
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
    em.e_lo = m.e_lo;
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
// Per-dataset workspace (floats), arrays of length N_t unless noted:
//   u, v (-> gv), ts = t s, ptot, dp[n_osc] (dp[0] is reused for the shape gradient),
//   pcw[C] = w_c P_c per core, f0[max_reco], gmu[max_reco]
struct DsWs {
    float *u, *v, *ts, *ptot, *dp, *pcw, *f0, *gmu;
};

__host__ __device__ inline int eval_ws_floats(int N_t, int C, int max_reco, int n_osc) {
    return ((4 + n_osc + C) * N_t + 2 * max_reco + 3) & ~3;
}

__device__ __forceinline__ DsWs carve_ds_ws(float *base, int N_t, int C, int max_reco, int n_osc) {
    DsWs w;
    w.u = base;
    w.v = w.u + N_t;
    w.ts = w.v + N_t;
    w.ptot = w.ts + N_t;
    w.dp = w.ptot + N_t;          // n_osc * N_t
    w.pcw = w.dp + n_osc * N_t;   // C * N_t
    w.f0 = w.pcw + C * N_t;       // max_reco
    w.gmu = w.f0 + max_reco;      // max_reco
    return w;
}

// Shared state of one evaluation (one per block).
struct EvalShared {
    typename OscTraits<6>::Coef kc;         // sin^2 coefficients (the first three for 4 parameters)
    float eta[kMaxOsc], eta_lo[kMaxOsc];
    PP nrm[FIT_MAX_DATASETS], eff[FIT_MAX_DATASETS];
    EMap em[FIT_MAX_DATASETS];
    PP power[FIT_MAX_CORES], rate[FIT_MAX_BACKGROUNDS];
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
            E.eta[lane] = h;
            E.eta_lo[lane] = l;
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
    } else if (warp == 1) {
        if (lane >= 16 && lane - 16 < m.C) E.power[lane - 16] = ppair(q, m.core_power_idx[lane - 16], 1.f);
    }
    if (warp == (int)(blockDim.x >> 5) - 1 && lane < m.n_bkg) E.rate[lane] = ppair(q, m.bkg[lane].rate_idx, 1.f);
    __syncthreads();
    return next;
}

// Stage A: u_k (and with DERIV the per-bin partials the adjoint needs). Ends with a barrier.
template <bool DERIV, int NOSC, int MODE>
static __device__ __forceinline__ void st_signal_mode(const DevModel &m, const EvalShared &E, const ParVecs &q,
                                                      float *wsb) {
    const int N_t = m.N_t, C = m.C, nth = blockDim.x;
    typename OscTraits<NOSC>::Coef kc;
#pragma unroll
    for (int i = 0; i < (int)(sizeof(kc.hi) / sizeof(float)); ++i) {
        kc.hi[i] = E.kc.hi[i];
        kc.lo[i] = E.kc.lo[i];
    }
    float eta[NOSC], eta_lo[NOSC];
#pragma unroll
    for (int i = 0; i < NOSC; ++i) {
        eta[i] = E.eta[i];
        eta_lo[i] = E.eta_lo[i];
    }
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, N_t, C, m.max_reco, m.n_osc);
        const PP nrm = E.nrm[i];
        for (int k = rot_tid(i, (N_t + 31) >> 5); k < N_t; k += nth) {
            const float ih = m.inv_e_hi[k], il = m.inv_e_lo[k];
            const int sp = ds.shape_idx[k];
            const float tk = ds.t[k];
            float pt = 0.f, dpt[NOSC];
#pragma unroll
            for (int j = 0; j < NOSC; ++j) dpt[j] = 0.f;
            for (int c = 0; c < C; ++c) {
                const float w = ds.w[c];
                if (w == 0.f) {
                    if (DERIV) ws.pcw[c * N_t + k] = 0.f;
                    continue;
                }
                const float ch = ds.kl_hi[c] * ih;
                const float cl = fmaf(ds.kl_hi[c], ih, -ch) + ds.kl_hi[c] * il + ds.kl_lo[c] * ih;
                float dP[NOSC];
                const float P = OscTraits<NOSC>::survival(MODE, eta, eta_lo, kc, ch, cl, dP);
                const PP pw = E.power[c];
                const float wP = w * P;
                if (DERIV) ws.pcw[c * N_t + k] = wP;
                pt += pmul(pw, wP);
                if (DERIV) {
#pragma unroll
                    for (int j = 0; j < NOSC; ++j) dpt[j] = fmaf(pw.h * w, dP[j], dpt[j]);
                }
            }
            const float ts = pmul(ppair(q, sp, 1.f), tk);
            if (DERIV) {
                ws.ts[k] = ts;
                ws.ptot[k] = pt;
#pragma unroll
                for (int j = 0; j < NOSC; ++j) ws.dp[j * N_t + k] = dpt[j];
            }
            ws.u[k] = pmul(nrm, ts * pt);
        }
    }
    __syncthreads();
}

// GEN: the general build (any formula); else Eq. 1 or the three-flavour formula.
template <bool DERIV, bool GEN>
static __device__ __forceinline__ void st_signal(const DevModel &m, const EvalShared &E, const ParVecs &q, float *wsb) {
    if (GEN && m.osc_mode == FIT_OSC_STERILE4)
        st_signal_mode<DERIV, 6, FIT_OSC_STERILE4>(m, E, q, wsb);
    else if (m.osc_mode == FIT_OSC_EQ1)
        st_signal_mode<DERIV, 4, FIT_OSC_EQ1>(m, E, q, wsb);
    else
        st_signal_mode<DERIV, 4, FIT_OSC_VACUUM3>(m, E, q, wsb);
}

// Corrected content of target bin t under the overlap rule. Source bin k covers [Y_k, Y_k+1] in
// grid units, Y_k = k + D(e_k); target t gathers the sources whose mapped interval overlaps
// [t, t+1]; overlaps are computed relative to the target (k - t is an exact small integer),
// which keeps them accurate in FP32.
__device__ __forceinline__ float overlap_target(const float *u, const float *e_edge, const EMap &em, int t, int N_t) {
    // first source whose mapped upper edge lies above t: start from the fixed point
    // k ~ t - D(k) and step until the bracket is right
    int k = t - (int)floorf(em.disp(e_edge[t]));
    k = min(max(k, 0), N_t - 1);
    k = t - (int)floorf(em.disp(e_edge[k]));
    k = min(max(k - 1, 0), N_t - 1);
    while (k > 0 && (float)(k - t) + em.disp(e_edge[k]) > 0.f) --k;
    float acc = 0.f;
    float dlo = em.disp(e_edge[k]);
    for (int it = 0; it < 64 && k < N_t; ++it, ++k) {
        const float dhi = em.disp(e_edge[k + 1]);
        const float ylo = (float)(k - t) + dlo;      // mapped edges relative to target t
        const float yhi = (float)(k + 1 - t) + dhi;
        if (ylo >= 1.f) break;
        const float ov = fminf(yhi, 1.f) - fmaxf(ylo, 0.f);
        if (ov > 0.f) acc = fmaf(u[k], ov / (1.f + (dhi - dlo)), acc);
        dlo = dhi;
    }
    return acc;
}

// Stage B: v = M(a) u. Ends with a barrier. GEN: compiled with the spline option.
template <bool GEN>
static __device__ __forceinline__ void st_remap(const DevModel &m, const EvalShared &E, float *wsb) {
    const int N_t = m.N_t, nth = blockDim.x;
    const bool spline = GEN && m.remap_mode == FIT_REMAP_SPLINE;
    for (int i = 0; i < E.n; ++i) {
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, N_t, m.C, m.max_reco, m.n_osc);
        const EMap em = E.em[i];
        for (int t = rot_tid(i, (N_t + 31) >> 5); t < N_t; t += nth)
            ws.v[t] = spline ? spline_target(ws.u, m.e_edge, em, t, N_t) : overlap_target(ws.u, m.e_edge, em, t, N_t);
    }
    __syncthreads();
}

// Stage C: fold into reco bins, f0 = R v (before the efficiency), banded rows. Each warp takes
// four rows at a time and two strides of each, so eight independent load/FMA chains per lane
// are in flight. Ends with a barrier.
static __device__ __forceinline__ void st_fold(const DevModel &m, const EvalShared &E, float *wsb) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
        const DevDetector &dt = m.det[ds.det];
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, m.N_t, m.C, m.max_reco, m.n_osc);
        const int nr = ds.n_reco;
        for (int j0 = rot_tid(i, nr) >> 5; j0 < nr; j0 += 4 * nw) {
            int lo[4], len[4];
            const float *rr[4];
            int lmax = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = j0 + u * nw;
                const bool on = j < nr;
                lo[u] = on ? dt.row_lo[j] : 0;
                len[u] = on ? dt.row_len[j] : 0;
                rr[u] = dt.rrow + (on ? dt.row_off[j] : 0);
                lmax = max(lmax, len[u]);
            }
            float s[4][2] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
            for (int b = lane; b < lmax; b += 64) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (b < len[u]) s[u][0] = fmaf(rr[u][b], ws.v[lo[u] + b], s[u][0]);
                    if (b + 32 < len[u]) s[u][1] = fmaf(rr[u][b + 32], ws.v[lo[u] + b + 32], s[u][1]);
                }
            }
            float t[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) t[u] = s[u][0] + s[u][1];
            const float tot = warp_sum_split<4>(t);
            const int j = j0 + (lane >> 3) * nw;
            if ((lane & 7) == 0 && j < nr) ws.f0[j] = tot;
        }
    }
    __syncthreads();
}

// Expected counts of one bin: efficiency x fold + backgrounds; tm / sh receive the templates and
// 1 + delta of the dataset's backgrounds (the loads of all of them in flight together).
__device__ __forceinline__ float bin_mu(const DevModel &m, const EvalShared &E, int i, const DevDataset &ds,
                                        const ParVecs &q, float f0, int j, int nb, float (&tm)[kMaxBkgDs],
                                        float (&sh)[kMaxBkgDs]) {
    int si[kMaxBkgDs];
#pragma unroll
    for (int b = 0; b < kMaxBkgDs; ++b) {
        const DevBkg &bk = m.bkg[ds.bkg_begin + min(b, max(nb - 1, 0))];
        tm[b] = b < nb ? bk.tmpl[j] : 0.f;
        si[b] = b < nb ? bk.shape_idx[j] : -1;
    }
    float mu = pmul(E.eff[i], f0);
#pragma unroll
    for (int b = 0; b < kMaxBkgDs; ++b) {
        if (b >= nb) break;
        const float del = si[b] >= 0 ? q.pv[si[b]] : 0.f;
        sh[b] = 1.f + del;
        mu += pmul(E.rate[ds.bkg_begin + b], fmaf(tm[b], del, tm[b]));
    }
    return mu;
}

// Expected counts of the group's datasets into mu (the whole data vector). Ends with a barrier.
static __device__ __forceinline__ void st_mu(const DevModel &m, const EvalShared &E, const ParVecs &q, float *wsb,
                                             float *mu) {
    const int nth = blockDim.x;
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, m.N_t, m.C, m.max_reco, m.n_osc);
        for (int j = rot_tid(i, (ds.n_reco + 31) >> 5); j < ds.n_reco; j += nth) {
            float tm[kMaxBkgDs], sh[kMaxBkgDs];
            mu[ds.data_off + j] = bin_mu(m, E, i, ds, q, ws.f0[j], j, ds.bkg_end - ds.bkg_begin, tm, sh);
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
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, m.N_t, m.C, m.max_reco, m.n_osc);
        const int nr = ds.n_reco, nb = ds.bkg_end - ds.bkg_begin;
        const int t0 = rot_tid(i, (nr + 31) >> 5);
        if ((t0 & ~31) >= nr) continue;      // this warp has no bin of this dataset
        float part[8];   // deviance, d/d eff, d/d rate_b
#pragma unroll
        for (int b = 0; b < 8; ++b) part[b] = 0.f;
        for (int j = t0; j < nr; j += nth) {
            const float n = data[ds.data_off + j], f0 = ws.f0[j];
            float tm[kMaxBkgDs], sh[kMaxBkgDs];
            const float mu = bin_mu(m, E, i, ds, q, f0, j, nb, tm, sh);
            if (!(mu > 0.f)) {
                atomicOr(&E.status, kStMuNonpos);
                continue;
            }
            part[0] += deviance(n, mu);
            const float g = 2.f * (mu - n) / mu;
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
    for (int i = 0; i < E.n; ++i) nll += E.nll_ds[i];
    E.nll = nll;
    if (grad == nullptr) return;
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
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
    for (int p = threadIdx.x; p < m.n_bs; p += blockDim.x) {
        float s = 0.f;
        for (int r = m.bs_ptr[p]; r < m.bs_ptr[p + 1]; ++r) {
            const BkgShapeRef ref = m.bs_ref[r];
            for (int i = 0; i < E.n; ++i) {
                if (E.dl[i] != ref.d) continue;
                const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, m.N_t, m.C, m.max_reco, m.n_osc);
                s += ws.gmu[ref.j] * E.rate[ref.q].h * ref.tmpl;
            }
        }
        grad[m.bs_param[p]] += s;
    }
}

// Stage D: adjoint of the fold, v <- gv = eff R^T gmu (column bands). rcol is exactly 0 past each
// column's band, so the loop runs the widest band of the warp's 32 adjacent columns (nearly
// their own widths: the resolution changes slowly with energy) with the row index clamped (no
// early exit) and four partial sums. No barrier.
static __device__ __forceinline__ void st_adjoint_fold(const DevModel &m, const EvalShared &E, float *wsb) {
    const int N_t = m.N_t, nth = blockDim.x;
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
        const DevDetector &dt = m.det[ds.det];
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, N_t, m.C, m.max_reco, m.n_osc);
        const int jmax = ds.n_reco - 1;
        const PP eff = E.eff[i];
        float *gv = ws.v;   // v is dead after the fold
        for (int k = rot_tid(i, (N_t + 31) >> 5); k < N_t; k += nth) {
            const int lo = dt.col_lo[k];
            const int cw = __reduce_max_sync(__activemask(), dt.col_len[k]);
            const float *rc = dt.rcol + k;
            float s[4] = {0.f, 0.f, 0.f, 0.f};
            int b = 0;
            for (; b + 7 < cw; b += 8) {   // eight loads in flight
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    s[u & 3] = fmaf(rc[(int64_t)(b + u) * N_t], ws.gmu[min(lo + b + u, jmax)], s[u & 3]);
            }
            for (; b < cw; ++b) s[0] = fmaf(rc[(int64_t)b * N_t], ws.gmu[min(lo + b, jmax)], s[0]);
            gv[k] = pmul(eff, (s[0] + s[1]) + (s[2] + s[3]));
        }
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
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
        const DsWs ws = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, N_t, C, m.max_reco, m.n_osc);
        const EMap em = E.em[i];
        const PP nrm = E.nrm[i];
        const float *gv = ws.v;
        float ep[4] = {0.f, 0.f, 0.f, 0.f};   // d/da0, d/da1, d/da2, d/d norm
        for (int k = rot_tid(i, (N_t + 31) >> 5); k < N_t; k += nth) {
            float gu = 0.f;
            if (spline) {
                gu = spline_adjoint_source(gv, m.e_edge, em, k, N_t);
                spline_adjoint_edge(ws.u, gv, m.e_edge, em, k, N_t, ep);
                if (k == N_t - 1) spline_adjoint_edge(ws.u, gv, m.e_edge, em, N_t, N_t, ep);
            } else {
                // per source k: gu = sum_t F_kt gv_t; A0 = (gu - gv(floor Y_k)) / w,
                // A1 = (gv(floor Y_k+1) - gu) / w
                const float e0 = m.e_edge[k], e1 = m.e_edge[k + 1];
                const float d0 = em.disp(e0), d1 = em.disp(e1);
                const float w = 1.f + (d1 - d0), iw = 1.f / w;
                const int f0i = (int)floorf(d0), f1i = (int)floorf(d1);
                const int t0 = k + f0i, t1 = k + 1 + f1i;
                for (int t = max(t0, 0); t <= min(t1, N_t - 1); ++t) {
                    const float ylo = (float)(k - t) + d0, yhi = (float)(k + 1 - t) + d1;
                    const float ov = fminf(yhi, 1.f) - fmaxf(ylo, 0.f);
                    if (ov > 0.f) gu = fmaf(ov * iw, gv[t], gu);
                }
                const float g0 = (t0 >= 0 && t0 < N_t) ? gv[t0] : 0.f;
                const float g1 = (t1 >= 0 && t1 < N_t) ? gv[t1] : 0.f;
                const float uk = ws.u[k] * iw;
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
    for (int i = 0; i < E.n; ++i) {
        const DevDataset &ds = m.ds[E.dl[i]];
        const float *gs = carve_ds_ws(wsb + (int64_t)i * m.ws_eval_floats, m.N_t, m.C, m.max_reco, m.n_osc).dp;
        const int L = ds.sp_lanes, per = nth / L;   // lanes per parameter, parameters per pass
        const int work = ds.n_sp * L;
        for (int q0 = rot_tid(i, (work + 31) >> 5); q0 < ((work + 31) & ~31); q0 += per * L) {
            const int p = q0 / L, sub = q0 & (L - 1);
            float s = 0.f;
            if (p < ds.n_sp)
                for (int r = ds.sp_ptr[p] + sub; r < ds.sp_ptr[p + 1]; r += L) s += gs[ds.sp_k[r]];
            for (int o = L >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (p < ds.n_sp && sub == 0) grad[ds.sp_param[p]] += s;
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

// The Poisson -2lnL of the datasets in `mask` and (grad != nullptr) its theta gradient added to
// grad. wsb: ws_group dataset workspaces. Returns the -2lnL on every thread; E.status (cleared
// here) holds kSt* bits on failure. Starts and ends with a barrier.
template <bool GEN>
static __device__ double eval_datasets(const DevModel &m, EvalShared &E, const ParVecs &q, uint32_t mask,
                                       const float *data, float *wsb, float *grad) {
    __syncthreads();
    if (threadIdx.x == 0) {
        E.status = 0;
        E.nll = 0.0;
    }
    for (int first = 0; first < m.n_ds;) {
        first = eval_setup_any<GEN>(m, E, q, mask, first, m.ws_group);
        if (E.n > 0) {
            if (grad != nullptr)
                st_signal<true, GEN>(m, E, q, wsb);
            else
                st_signal<false, GEN>(m, E, q, wsb);
            st_remap<GEN>(m, E, wsb);
            st_fold(m, E, wsb);
            if (grad != nullptr)
                st_lik<true>(m, E, q, data, wsb);
            else
                st_lik<false>(m, E, q, data, wsb);
        }
        if (E.status || E.bad) {   // block-uniform after the barriers
            __syncthreads();
            if (threadIdx.x == 0 && !E.status) E.status = kStEscale;
            __syncthreads();
            return INFINITY;
        }
        if (E.n == 0) continue;
        if (grad != nullptr) {
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
// of all blocks together, as tiles of 32 rows x kTriCols columns (a warp per tile, a lane per
// row: every column is one coalesced load and one broadcast of x, sixteen in flight). A tile
// leaves its partial sum at part[seg * tri_rows + row]; after a barrier tri_sum adds a row's
// segments in order. x: by parameter index.
static __device__ __forceinline__ void tri_apply(const DevModel &m, const TriTile *tiles, int n_tiles, const float *M,
                                                 const float *x, float *part) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int t = threadIdx.x >> 5; t < n_tiles; t += nw) {
        const TriTile T = tiles[t];
        const int r = min(T.row0 + lane, T.n - 1), cols = T.cols;
        const float *col = M + T.mat + (int64_t)T.col0 * T.n + r;
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        int c = 0;
        if (T.in0 >= 0) {
            const float *xb = x + T.in0 + T.col0;
            for (; c + 15 < cols; c += 16) {
#pragma unroll
                for (int u = 0; u < 16; ++u) s[u & 3] = fmaf(col[(int64_t)(c + u) * T.n], xb[c + u], s[u & 3]);
            }
            for (; c < cols; ++c) s[0] = fmaf(col[(int64_t)c * T.n], xb[c], s[0]);
        } else {
            const int *idx = m.blk_idx + T.idx + T.col0;
            for (; c + 7 < cols; c += 8) {
#pragma unroll
                for (int u = 0; u < 8; ++u) s[u & 3] = fmaf(col[(int64_t)(c + u) * T.n], x[idx[c + u]], s[u & 3]);
            }
            for (; c < cols; ++c) s[0] = fmaf(col[(int64_t)c * T.n], x[idx[c]], s[0]);
        }
        if (T.row0 + lane < T.n) part[T.seg * m.tri_rows + T.out + T.row0 + lane] = (s[0] + s[1]) + (s[2] + s[3]);
    }
}

__device__ __forceinline__ float tri_sum(const DevModel &m, const float *part, int row, bool upper) {
    const int x = m.tri_seg[row];
    const int s0 = upper ? (x >> 8) & 255 : 0, s1 = upper ? x >> 16 : x & 255;
    float t = part[s0 * m.tri_rows + row];
    for (int q = s0 + 1; q < s1; ++q) t += part[q * m.tri_rows + row];
    return t;
}

}  // namespace fitcore

// Device side of the fits: the minimiser's state machine, the transformation layer and the
// preconditioner, shared by the persistent kernel (fit_kernel_*.cu, one translation unit per
// block size so that they compile in parallel) and the lockstep engine (kernels.cu).
#pragma once
#include "kernels.cuh"

namespace fitcore {

// ------------------------------------------------------------------------------------
// shared-memory helpers
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void copy_model(DevModel *dst, const DevModel *src) {
    const int n = (int)(sizeof(DevModel) / sizeof(int));
    const int *s = reinterpret_cast<const int *>(src);
    int *d = reinterpret_cast<int *>(dst);
#pragma unroll 1
    for (int i = threadIdx.x; i < n; i += blockDim.x) d[i] = s[i];
    __syncthreads();
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// ------------------------------------------------------------------------------------
// persistent batched L-BFGS
// ------------------------------------------------------------------------------------
constexpr int kMaxHist = 32;
constexpr int kStallWindow = 100;   // iterations per stall check
constexpr int kMaxLsFresh = 30;     // line-search trials along steepest descent
constexpr int kNDots = 4 * kMaxHist + 1;

// Minimiser state of one fit between two evaluations: in shared memory while a block works on
// the fit, in global memory between the launches of the lockstep engine.
constexpr int kPhStart = 0, kPhTrial = 1, kPhDone = 2;

struct FitState {
    // L-BFGS history in scalars: SY[i][j] = s_i.y_j (needed for i older than j and i = j),
    // YY[i][j] = y_i.y_j (symmetric), rho_i = 1 / s_i.y_i, by history slot
    // (rows padded by one double: a lane per row otherwise meets one bank)
    double SY[kMaxHist][kMaxHist + 1], YY[kMaxHist][kMaxHist + 1];
    double rho[kMaxHist];
    double gamma;
    double f, edm;
    // line search on phi(alpha) = f(z + alpha d): bracket [lo, hi], kink crossing a_cr
    double alpha, dphi0, eps_f, lo, flo, dlo, hi, fhi, dhi, a_cr, f_cr;
    int hn, head, occ;
    int phase, ls_it, have_lo, pending, restarts_left, since_restart;
    int iters, n_evals, status;
    int win_it;     // stall window: iteration and value at its start
    double f_win;
};

// What one minimiser step does to the fit's vectors, decided by one warp from the scalars.
struct FitStep {
    int next;                  // kNextDirection, kNextTrial, kNextDone
    int init;                  // the trial is the start point
    int save_cr, save_lo;      // keep the trial as the kink crossing / the best lower point
    int src;                   // accepted point: 0 none, 1 the trial, 2 the kink crossing, 3 the lower point
    float alpha;               // next trial: z + alpha d
};
constexpr int kNextDirection = 0, kNextTrial = 1, kNextDone = 2;

struct alignas(16) FitSmem {
    DevModel m;
    EvalShared E;
    double red[kMaxWarps + 1];
    FitState st;
    double dots[kNDots];       // fused pass: S.y_new | Y.y_new | S.g | Y.g | g.g
    // d = -(cg g + sum_k cs_k s_slot(k) + cy_k y_slot(k)), k < n_dir
    float cs[kMaxHist], cy[kMaxHist];
    int slot[kMaxHist];
    int n_dir;
    float cg;
    FitStep step;
    int inst;
    float pre_u[kMaxPreRank];  // preconditioner scratch
};

struct FitVecs {
    float *z, *g, *d, *zt, *gt, *zlo, *glo, *zcr, *gcr, *pv, *pd, *gth, *zw, *gzw, *pl, *S, *Y;
};

// 15 P-vectors at base; the 2 hist P-vectors of the history at hbase (pitch fit_vec_pitch(P))
__device__ __forceinline__ FitVecs carve_fit_vecs(float *base, float *hbase, int P, int hist) {
    const int Pp = fit_vec_pitch(P);
    FitVecs v;
    v.z = base;
    v.g = v.z + Pp;
    v.d = v.g + Pp;
    v.zt = v.d + Pp;
    v.gt = v.zt + Pp;
    v.zlo = v.gt + Pp;
    v.glo = v.zlo + Pp;
    v.zcr = v.glo + Pp;
    v.gcr = v.zcr + Pp;
    v.pv = v.gcr + Pp;
    v.pd = v.pv + Pp;
    v.gth = v.pd + Pp;
    v.zw = v.gth + Pp;    // preconditioned fits: z of the trial point and its z-gradient
    v.gzw = v.zw + Pp;
    v.pl = v.gzw + Pp;
    v.S = hbase;
    v.Y = v.S + (int64_t)hist * Pp;
    return v;
}

// block-wide dot product of two P-vectors (double result on every thread)
__device__ __forceinline__ double bdot(const float *a, const float *b, int n, double *red) {
    float acc = 0.f;
#pragma unroll 1
    for (int i = threadIdx.x; i < n; i += blockDim.x) acc = fmaf(a[i], b[i], acc);
    return block_sum(acc, red);
}

// One pass of block-wide dot products into `out`, a warp per history slot set in `occ`: s_j.y_new,
// y_j.y_new (when ynew is given), s_j.g and y_j.g at out[type * kMaxHist + j], and g.g at
// out[4 kMaxHist]; a slot's four products share its two history vectors, so the history is read
// once. 16-byte loads, the last P mod 4 entries scalar. Ends with a barrier.
static __device__ __noinline__ void fused_dots(const float *Sv, const float *Yv, const float *ynew, const float *g, int P,
                           unsigned occ, double *out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int pitch = fit_vec_pitch(P), n4 = P >> 2, tail = (P & ~3) + lane;
    const int live = __popc(occ);
    const float *yn = ynew ? ynew : g;
#pragma unroll 1
    for (int w = warp; w <= live; w += nw) {
        if (w == live) {   // g.g
            float acc = 0.f;
#pragma unroll 1
            for (int k = lane; k < n4; k += 32) {
                const float4 x = reinterpret_cast<const float4 *>(g)[k];
                acc = fmaf(x.x, x.x, fmaf(x.y, x.y, fmaf(x.z, x.z, fmaf(x.w, x.w, acc))));
            }
            if (tail < P) acc = fmaf(g[tail], g[tail], acc);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) out[kNDots - 1] = (double)acc;
            continue;
        }
        unsigned left = occ;   // the w-th occupied slot
#pragma unroll 1
        for (int i = 0; i < w; ++i) left &= left - 1;
        const int j = __ffs(left) - 1;
        const float *s = Sv + (int64_t)j * pitch, *y = Yv + (int64_t)j * pitch;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int k = lane; k < n4; k += 32) {
            const float4 a = reinterpret_cast<const float4 *>(s)[k], b = reinterpret_cast<const float4 *>(y)[k];
            const float4 u = reinterpret_cast<const float4 *>(yn)[k], v = reinterpret_cast<const float4 *>(g)[k];
            acc[0] = fmaf(a.x, u.x, fmaf(a.y, u.y, fmaf(a.z, u.z, fmaf(a.w, u.w, acc[0]))));
            acc[1] = fmaf(b.x, u.x, fmaf(b.y, u.y, fmaf(b.z, u.z, fmaf(b.w, u.w, acc[1]))));
            acc[2] = fmaf(a.x, v.x, fmaf(a.y, v.y, fmaf(a.z, v.z, fmaf(a.w, v.w, acc[2]))));
            acc[3] = fmaf(b.x, v.x, fmaf(b.y, v.y, fmaf(b.z, v.z, fmaf(b.w, v.w, acc[3]))));
        }
        if (tail < P) {
            const float a = s[tail], b = y[tail], u = yn[tail], v = g[tail];
            acc[0] = fmaf(a, u, acc[0]);
            acc[1] = fmaf(b, u, acc[1]);
            acc[2] = fmaf(a, v, acc[2]);
            acc[3] = fmaf(b, v, acc[3]);
        }
        const float t = warp_sum_split<4>(acc);
        if ((lane & 7) == 0) out[(lane >> 3) * kMaxHist + j] = (double)t;
    }
    __syncthreads();
}

__device__ __forceinline__ void reset_history(FitState &st) {
    st.hn = 0;
    st.head = 0;
    st.occ = 0;
    st.gamma = 1.0;
}

// num / den in double: the FP32 reciprocal, two Newton-Raphson steps for 1 / den and one correction of
// the quotient by its residual (within an ulp: tests/test_quick_division.py). The library's double
// division takes 1467 cycles here, this about 450. Operands outside FP32's normal range take the
// division.
static __device__ __noinline__ double quick_div(double num, double den) {
    const float d = (float)den;
    if (!(fabsf(d) > 1e-30f && fabsf(d) < 1e30f)) return num / den;
    double r = (double)__frcp_rn(d);
    r = fma(r, fma(-den, r, 1.0), r);
    r = fma(r, fma(-den, r, 1.0), r);
    const double q = num * r;
    return fma(r, fma(-den, q, num), q);
}

// One warp: folds the pending curvature pair (slot S.st.head, if `pending`) into the scalar
// history and runs the L-BFGS two-loop recursion on scalars. Every inner product the
// recursion needs is one of s_i.g, y_i.g, s_i.y_j (i older than j) or y_i.y_j, so the
// direction is d = -(cg g + sum_j cs_j s_j + sum_j cy_j y_j) with coefficients from the
// recurrence, and g^T H g (returned, on every lane) follows from the same scalars. Lane k holds
// chronological history position k; both triangular recurrences run column by column.
//
// What bounds it: the chain of double operations, 66 cycles each, one column after another. So
// the columns' matrix entries are scaled by rho off the chain (a column costs one broadcast and
// one fma), the products with YY ride along, slots advance without a modulo, and the pending
// pair's rows are written by a lane per slot. On the three-dataset model (nine pairs on
// average) a step's direction took 38 700 cycles before.
static __device__ double lbfgs_scalars(FitSmem &S, int hist_max, bool pending) {
    const int lane = threadIdx.x & 31;
    const double *dt = S.dots;
    FitState &st = S.st;
    if (pending) {
        const int c = st.head, occ = st.occ;
        const double sy = dt[c], yy = dt[kMaxHist + c];
        if (sy > 1e-10 * yy && yy > 0.0) {
            const double q = quick_div(lane == 1 ? sy : 1.0, lane == 1 ? yy : sy);   // 1/s.y, s.y/y.y
            __syncwarp();
            if (lane < hist_max && ((occ >> lane) & 1) && lane != c) {
                st.SY[lane][c] = dt[lane];
                st.YY[lane][c] = st.YY[c][lane] = dt[kMaxHist + lane];
            }
            if (lane == 0) {
                st.SY[c][c] = sy;
                st.YY[c][c] = yy;
                st.rho[c] = q;
                st.occ = occ | (1 << c);
                st.head = c + 1 == hist_max ? 0 : c + 1;
                st.hn = min(st.hn + 1, hist_max);
            }
            if (lane == 1) st.gamma = q;
        } else if ((occ >> c) & 1) {
            // rejected pair written over the oldest one: that pair is gone as well
            __syncwarp();
            if (lane == 0) {
                st.occ = occ & ~(1 << c);
                st.hn -= 1;
            }
        }
    }
    __syncwarp();
    const int hn = st.hn;
    const int oldest = st.head >= hn ? st.head - hn : st.head - hn + hist_max;
    const double gam = st.gamma, gg = dt[kNDots - 1];
    const bool live = lane < hn;
    auto slot_of = [&](int k) { return oldest + k >= hist_max ? oldest + k - hist_max : oldest + k; };
    const int sl = live ? slot_of(lane) : 0;    // this lane's history slot
    const double sg = live ? dt[2 * kMaxHist + sl] : 0.0, yg = live ? dt[3 * kMaxHist + sl] : 0.0;
    const double rho = live ? st.rho[sl] : 0.0;
    // alpha_k = rho_k (s_k.g - sum_{l > k} alpha_l s_k.y_l), newest first; u_k = sum_l alpha_l y_k.y_l
    double a = rho * sg, alpha = 0.0, u = 0.0;
#pragma unroll 1
    for (int l = hn - 1; l >= 0; --l) {
        const int sll = slot_of(l);
        const double rs = lane < l ? rho * st.SY[sl][sll] : 0.0, yy = live ? st.YY[sl][sll] : 0.0;
        const double al = __shfl_sync(0xffffffffu, a, l);
        if (lane == l) alpha = al;
        a = fma(-al, rs, a);
        u = fma(al, yy, u);
    }
    // beta_k = rho_k (gam (y_k.g - u_k) + sum_{l < k} (alpha_l - beta_l) s_l.y_k), oldest first
    double b = rho * (gam * (yg - u)), beta = 0.0;
#pragma unroll 1
    for (int l = 0; l < hn; ++l) {
        const double rs = live && lane > l ? rho * st.SY[slot_of(l)][sl] : 0.0;
        const double al = __shfl_sync(0xffffffffu, alpha, l), bl = __shfl_sync(0xffffffffu, b, l);
        if (lane == l) beta = bl;
        b = fma(al - bl, rs, b);
    }
    const double cs = alpha - beta, cy = -gam * alpha;
    double part = live ? cs * sg + cy * yg : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    const double ghg = gam * gg + part;
    if (live) {
        S.cs[lane] = (float)cs;
        S.cy[lane] = (float)cy;
        S.slot[lane] = sl;
    }
    const bool ok = ghg > 0.0;   // else not a descent direction: drop the history, steepest descent
    __syncwarp();
    if (lane == 0) {
        S.n_dir = ok ? hn : 0;
        S.cg = ok ? (float)gam : 1.f;
        if (!ok) reset_history(st);
    }
    __syncwarp();
    return ok ? ghg : gg;
}

// theta from z (transformation layer): pd = J z, pv = theta0 + pd and its residual pl; J is the
// width or scale outside the prior blocks and the Cholesky factor L inside. part: scratch of
// tri_segs x tri_rows floats. Ends with a barrier.
static __device__ __noinline__ void theta_of_z(const DevModel &m, const float *z, FitVecs &V, float *part) {
    const int tid = threadIdx.x, nth = blockDim.x;
    auto put = [&](int i, float d) {
        const float h = m.theta0_f[i] + d;
        V.pd[i] = d;
        V.pv[i] = h;
        V.pl[i] = presid(m, h, d, i);
    };
#pragma unroll 1
    for (int i = tid; i < m.P; i += nth) {
        const float s = m.zscale[i];
        if (s > 0.f) put(i, s * z[i]);
    }
    if (m.tri_rows > 0) {
        tri_apply(m, m.tri_lo, m.n_tri_lo, m.L_lo, z, part);
        __syncthreads();
#pragma unroll 1
        for (int r = tid; r < m.tri_rows; r += nth) put(m.tri_param[r], tri_sum(m, part, r, false));
    }
    __syncthreads();
}

// Prior in z space and the chain rule back to z: gz = J^T gth + 2 z over the constrained
// coordinates (J = diag(scale) outside the prior blocks, the Cholesky factor L inside);
// returns the prior |z|^2 (all threads). part as in theta_of_z.
static __device__ double eval_z_prior(const DevModel &m, const float *z, const float *gth, float *gz, float *part,
                               double *red) {
    const int tid = threadIdx.x, nth = blockDim.x;
    float acc = 0.f;
#pragma unroll 1
    for (int i = tid; i < m.P; i += nth) {
        const float s = m.zscale[i];
        if (s > 0.f) {
            const bool con = m.prior_inv[i] > 0.f;
            gz[i] = s * gth[i] + (con ? 2.f * z[i] : 0.f);
            if (con) acc = fmaf(z[i], z[i], acc);
        }
    }
    if (m.tri_rows > 0) {
        tri_apply(m, m.tri_up, m.n_tri_up, m.L_up, gth, part);
        __syncthreads();
#pragma unroll 1
        for (int r = tid; r < m.tri_rows; r += nth) {
            const int p = m.tri_param[r];
            const float zj = z[p];
            gz[p] = tri_sum(m, part, r, true) + 2.f * zj;
            acc = fmaf(zj, zj, acc);
        }
    }
    return block_sum(acc, red);
}

// Parameters held at their start values (a profile-likelihood point): a zero z-gradient keeps
// every L-BFGS direction, and so the parameter, where it is. Only parameters outside the prior
// blocks can be held (their z coordinate is the parameter itself, scaled).
__device__ __forceinline__ void hold_fixed(const uint8_t *fixed, float *gz, int P) {
    if (fixed == nullptr) return;
#pragma unroll 1
    for (int i = threadIdx.x; i < P; i += blockDim.x)
        if (fixed[i]) gz[i] = 0.f;
}

// y = x + Q (coef o (Q^T x)) for the model's preconditioner (coef = pre_c: y = T x; coef =
// pre_c + r: y = T^-1 x). Q^T rows: a warp per row, 16-byte loads, the last P mod 4 entries
// scalar (the padding of x is never read); then a thread per entry over the r rows. x and y
// may be the same vector. u: r floats of shared scratch. Held parameters (fixed) are left out
// of Q: T then maps them to themselves and mixes them into nothing, so they stay held in w
// (T^-1 is then only approximate for the free part, which only moves the start). Ends with a
// barrier.
static __device__ __noinline__ void pre_apply(const DevModel &m, const float *coef, const float *x, float *y, float *u,
                          const uint8_t *fixed) {
    const int P = m.P, Pp = fit_vec_pitch(P), r = m.pre_r;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int nfull = P >> 2;
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    // four rows per warp and pass, so that their loads are in flight together
#pragma unroll 1
    for (int k0 = warp; k0 < r; k0 += 4 * nw) {
        const float4 *q4[4];
#pragma unroll
        for (int u4 = 0; u4 < 4; ++u4) q4[u4] = reinterpret_cast<const float4 *>(m.pre_Q + (int64_t)min(k0 + u4 * nw, r - 1) * Pp);
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
        for (int c = lane; c < nfull; c += 32) {
            float4 b = x4[c];
            if (fixed) {
                const uint8_t *f = fixed + 4 * c;
                if (f[0]) b.x = 0.f;
                if (f[1]) b.y = 0.f;
                if (f[2]) b.z = 0.f;
                if (f[3]) b.w = 0.f;
            }
#pragma unroll
            for (int u4 = 0; u4 < 4; ++u4) {
                const float4 a = __ldg(q4[u4] + c);
                acc[u4] = fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, acc[u4]))));
            }
        }
        if (lane < (P & 3) && !(fixed && fixed[4 * nfull + lane])) {
            const float b = x[4 * nfull + lane];
#pragma unroll
            for (int u4 = 0; u4 < 4; ++u4)
                acc[u4] = fmaf(__ldg(reinterpret_cast<const float *>(q4[u4]) + 4 * nfull + lane), b, acc[u4]);
        }
        const float t = warp_sum_split<4>(acc);
        const int k = k0 + (lane >> 3) * nw;
        if ((lane & 7) == 0 && k < r) u[k] = __ldg(coef + k) * t;
    }
    __syncthreads();
#pragma unroll 1
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
        float acc = x[i];
        if (!(fixed && fixed[i])) {
#pragma unroll 1
            for (int k0 = 0; k0 < r; k0 += 16) {   // sixteen rows' loads in flight
                float q[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) q[k] = __ldg(m.pre_Q + (int64_t)min(k0 + k, r - 1) * Pp + i);
#pragma unroll
                for (int k = 0; k < 16; ++k) acc = fmaf(q[k], k0 + k < r ? u[k0 + k] : 0.f, acc);
            }
        }
        y[i] = acc;
    }
    __syncthreads();
}

// -2lnL(theta(z)) and its z-gradient gz. Returns +inf on an invalid point. ws: the evaluation
// workspace (also the scratch of the prior blocks' products, before and after the datasets).
template <bool GEN>
static __device__ double eval_z(const DevModel &m, const float *z, float *gz, FitVecs &V, float *ws,
                         const float *data, uint32_t mask, FitSmem &S, const uint8_t *fixed) {
    theta_of_z(m, z, V, ws);
#pragma unroll 1
    for (int i = threadIdx.x; i < m.P; i += blockDim.x) V.gth[i] = 0.f;
    const double nll = eval_datasets<GEN, true>(m, S.E, ParVecs{V.pv, V.pd, V.pl}, mask, data, ws, V.gth);
    if (S.E.status) return INFINITY;
    const double prior = eval_z_prior(m, z, V.gth, gz, ws, S.red);
    hold_fixed(fixed, gz, m.P);
    return nll + prior;
}

// The same in the preconditioned coordinates w (z = T w): -2lnL and g_w = T^T g_z.
template <bool GEN>
static __device__ double eval_w(const DevModel &m, const float *w, float *gw, FitVecs &V, float *ws,
                         const float *data, uint32_t mask, FitSmem &S, const uint8_t *fixed) {
    pre_apply(m, m.pre_c, w, V.zw, S.pre_u, fixed);
    const double f = eval_z<GEN>(m, V.zw, V.gzw, V, ws, data, mask, S, fixed);
    __syncthreads();
    pre_apply(m, m.pre_c, V.gzw, gw, S.pre_u, fixed);   // T is symmetric; held entries stay 0
    return f;
}

// cubic minimiser through (a, fa, ga), (b, fb, gb), or the secant of the slopes when the
// values are not informative (difference within the noise allowance)
__device__ __forceinline__ double ls_interp(double a, double fa, double ga, double b, double fb,
                                            double gb, double eps_f) {
    double t;
    if (isfinite(fb) && fabs(fb - fa) > eps_f) {
        const double d1 = ga + gb - 3.0 * (fa - fb) / (a - b);
        const double disc = d1 * d1 - ga * gb;
        if (disc >= 0.0) {
            const double d2 = copysign(sqrt(disc), b - a);
            t = b - (b - a) * (gb + d2 - d1) / (gb - ga + 2.0 * d2);
        } else {
            t = 0.5 * (a + b);
        }
    } else if (isfinite(gb) && gb != ga) {
        t = a - ga * (b - a) / (gb - ga);
    } else {
        t = 0.5 * (a + b);
    }
    const double lo = fmin(a, b), hi = fmax(a, b), w = hi - lo;
    if (!(t >= lo + 0.1 * w && t <= hi - 0.1 * w)) t = 0.5 * (a + b);
    return t;
}

struct FitParams {
    int hist, max_iter, max_ls, restarts;
    double edm_tol, f_noise_rel;
    uint64_t deadline;         // %globaltimer value past which a fit stops with TIMEOUT
};

// The scalar half of a minimiser step after the evaluation (fa, slope da along the search
// direction): updates the state and decides what happens to the vectors (S.step). One warp.
static __device__ void decide_trial(FitSmem &S, double fa, double da, const FitParams &F) {
    const double c1 = 1e-4, c2 = 0.9;
    const bool first = (threadIdx.x & 31) == 0;
    FitState &st = S.st;
    FitStep q;
    q.next = kNextDirection;
    q.init = q.save_cr = q.save_lo = q.src = 0;
    q.alpha = 0.f;
    if (st.phase == kPhStart) {
        // the start point's evaluation
        q.init = 1;
        if (!isfinite(fa)) q.next = kNextDone;
        __syncwarp();
        if (first) {
            reset_history(st);
            st.f = fa;
            st.n_evals++;
            st.restarts_left = F.restarts;
            st.since_restart = F.hist;
            st.pending = 0;
            st.f_win = fa;
            st.win_it = 0;
            if (q.next == kNextDone) st.status = FIT_STATUS_NONFINITE;
        }
    } else {
        // a line-search trial at alpha came back
        const double f = st.f, dphi0 = st.dphi0, eps_f = st.eps_f;
        double alpha = st.alpha, lo = st.lo, flo = st.flo, dlo = st.dlo, hi = st.hi, fhi = st.fhi, dhi = st.dhi;
        double a_cr = st.a_cr, f_cr = st.f_cr;
        int ls_it = st.ls_it, have_lo = st.have_lo, iters = st.iters, status = st.status;
        const int hn = st.hn;
        const bool armijo = fa <= f + c1 * alpha * dphi0;
        const bool approx = fa <= f + eps_f;
        const bool val_ok = isfinite(fa) && (armijo || approx);
        bool stop = false;
        double f_acc = fa;
        if (val_ok && fabs(da) <= -c2 * dphi0) {
            q.src = 1;
        } else {
            if (val_ok && da >= c2 * dphi0 && alpha < a_cr) {   // crossed a kink
                a_cr = alpha;
                f_cr = fa;
                q.save_cr = 1;
            }
            if (!val_ok || fa > flo + eps_f || da >= 0.0) {
                hi = alpha;
                fhi = fa;
                dhi = da;
            } else {
                lo = alpha;
                flo = fa;
                dlo = da;
                have_lo = 1;
                q.save_lo = 1;
            }
            if (!isfinite(hi)) {
                alpha = 4.0 * alpha;
            } else {
                alpha = ls_interp(lo, flo, dlo, hi, fhi, dhi, eps_f);
                if (hi - lo <= 1e-7 * hi) stop = true;
            }
            // a quasi-Newton direction is well scaled (the unit step is usually right), so its
            // search stops after max_ls trials; a steepest-descent search (fresh history) has
            // to find the scale and gets kMaxLsFresh
            if (!stop && ++ls_it < (hn == 0 ? kMaxLsFresh : F.max_ls)) q.next = kNextTrial;
        }
        bool mark = false, drop = false;
        if (q.next != kNextTrial) {
            if (q.src == 0) {
                if (isfinite(a_cr)) {
                    q.src = q.save_cr ? 1 : 2;   // (the trial itself when it was just kept)
                    f_acc = f_cr;
                } else if (have_lo) {
                    q.src = q.save_lo ? 1 : 3;
                    f_acc = flo;
                }
            }
            if (q.src) {
                iters++;
                // stall: a whole window of iterations that lowered the value by no more than
                // the FP32 noise allowance (the line search then only trades noise, e.g. on a
                // crease of the energy correction)
                if (iters - st.win_it >= kStallWindow) {
                    if (st.f_win - f_acc <= 2.0 * F.f_noise_rel * (1.0 + fabs(f_acc))) {
                        status = FIT_STATUS_STALLED;
                        q.next = kNextDone;
                    }
                    mark = true;
                }
            } else if (hn > 0) {   // retry from steepest descent
                drop = true;
            } else {
                status = FIT_STATUS_LINESEARCH_FAIL;
                q.next = kNextDone;
            }
        }
        q.alpha = (float)alpha;
        __syncwarp();   // every lane has read the state
        if (first) {
            if (drop) reset_history(st);
            st.n_evals++;
            st.alpha = alpha;
            st.lo = lo;
            st.flo = flo;
            st.dlo = dlo;
            st.hi = hi;
            st.fhi = fhi;
            st.dhi = dhi;
            st.a_cr = a_cr;
            st.f_cr = f_cr;
            st.ls_it = ls_it;
            st.have_lo = have_lo;
            st.iters = iters;
            st.status = status;
            if (q.src) {   // curvature pair in the next slot; folded in by the next fused pass
                st.f = f_acc;
                st.pending = 1;
                st.since_restart++;
            }
            if (mark) {
                st.f_win = f_acc;
                st.win_it = iters;
            }
        }
    }
    if (first) {
        st.phase = q.next == kNextTrial ? kPhTrial : q.next == kNextDone ? kPhDone : st.phase;
        S.step = q;
    }
}

// After the fused dot products: folds the pending pair, runs the recursion, and either ends the
// fit (EDM, iteration limit, clock), asks for another direction after a history restart, or
// starts the line search (S.step). One warp.
static __device__ void decide_direction(FitSmem &S, const FitParams &F) {
    const bool first = (threadIdx.x & 31) == 0;
    FitState &st = S.st;
    const double ghg = lbfgs_scalars(S, F.hist, st.pending != 0);
    const double edm = 0.5 * ghg, f = st.f;
    const int hn = st.hn, restarts_left = st.restarts_left;
    int next = kNextTrial, status = st.status;
    bool again = false;
    if (edm < F.edm_tol && st.since_restart >= F.hist) {
        if (restarts_left == 0) {
            status = FIT_STATUS_CONVERGED;
            next = kNextDone;
        } else {
            again = true;
            next = kNextDirection;
        }
    } else if (st.iters >= F.max_iter) {
        status = FIT_STATUS_MAXITER;
        next = kNextDone;
    } else if (global_ns() > F.deadline) {
        status = FIT_STATUS_TIMEOUT;
        next = kNextDone;
    }
    // first trial: the unit step, or a step of length 1 along steepest descent
    double alpha = 1.0;
    if (hn == 0) {
        const double dn = (double)S.cg * sqrt(S.dots[kNDots - 1]);
        alpha = fmin(1.0, 1.0 / fmax(dn, 1e-30));
    }
    __syncwarp();   // every lane has read the state
    if (first) {
        st.edm = edm;
        st.pending = 0;
        st.status = status;
        st.phase = next == kNextTrial ? kPhTrial : kPhDone;
        S.step.next = next;
        S.step.alpha = (float)alpha;
        if (again) {
            // drop the history and rebuild it (at least hist iterations): the fresh pairs come
            // from the directions still moving, the flat ones a short history may not have seen
            st.restarts_left = restarts_left - 1;
            st.since_restart = 0;
            reset_history(st);
        }
        if (next == kNextTrial) {
            st.alpha = alpha;
            st.dphi0 = -ghg;
            st.eps_f = F.f_noise_rel * (1.0 + fabs(f));
            st.lo = 0.0;
            st.flo = f;
            st.dlo = -ghg;
            st.hi = st.fhi = st.dhi = INFINITY;
            st.a_cr = INFINITY;
            st.f_cr = 0.0;
            st.have_lo = 0;
            st.ls_it = 0;
        }
    }
}

// One step of the minimiser: consumes the evaluation (fa, V.gt) of the point V.zt and leaves
// the next point to evaluate in V.zt (returns true), or ends the fit (returns false, S.st.phase
// = kPhDone, S.st.status set).
//
// L-BFGS in whitened coordinates with the two-loop recursion on scalars (fused_dots,
// lbfgs_scalars). Line search on phi(alpha) = f(z + alpha d): accepts a strong-Wolfe point or
// the approximate-Wolfe point of Hager & Zhang (value within the noise allowance eps_f, slope
// condition), brackets with cubic / secant interpolation, and falls back to the smallest trial
// that crossed a kink (value not increased, slope risen past c2 phi'(0)) or to the best lower
// point. A failed search with a history retries from steepest descent. Stop: EDM =
// 1/2 g^T H g < edm_tol (optionally after `restarts` history rebuilds), max_iter, or the clock.
//
// The scalars are FP64 (64 times slower than FP32 here: a warp's double operation holds the
// SM's FP64 pipe for 16 cycles), so one warp computes them and the block acts on its decision.
static __device__ bool fit_decide(FitSmem &S, FitVecs &V, int P, double fa, const FitParams &F) {
    const int tid = threadIdx.x, nth = blockDim.x;
    __syncthreads();
    const double da = (S.st.phase != kPhStart && isfinite(fa)) ? bdot(V.gt, V.d, P, S.red) : (double)INFINITY;
    if (tid < 32) decide_trial(S, fa, da, F);
    __syncthreads();
    const FitStep q = S.step;
    if (q.init) {
#pragma unroll 1
        for (int i = tid; i < P; i += nth) {
            V.z[i] = V.zt[i];
            V.g[i] = V.gt[i];
        }
    }
    if (q.save_cr) {
#pragma unroll 1
        for (int i = tid; i < P; i += nth) {
            V.zcr[i] = V.zt[i];
            V.gcr[i] = V.gt[i];
        }
    }
    if (q.save_lo) {
#pragma unroll 1
        for (int i = tid; i < P; i += nth) {
            V.zlo[i] = V.zt[i];
            V.glo[i] = V.gt[i];
        }
    }
    if (q.src) {
        const float *zs = q.src == 1 ? V.zt : q.src == 2 ? V.zcr : V.zlo;
        const float *gs = q.src == 1 ? V.gt : q.src == 2 ? V.gcr : V.glo;
        const int64_t c = (int64_t)S.st.head * fit_vec_pitch(P);
#pragma unroll 1
        for (int i = tid; i < P; i += nth) {
            const float zn = zs[i], gn = gs[i];
            V.S[c + i] = zn - V.z[i];
            V.Y[c + i] = gn - V.g[i];
            V.z[i] = zn;
            V.g[i] = gn;
        }
    }
    if (q.next == kNextTrial) {   // the next point along the same direction
#pragma unroll 1
        for (int i = tid; i < P; i += nth) V.zt[i] = fmaf(q.alpha, V.d[i], V.z[i]);
        __syncthreads();
        return true;
    }
    if (q.next == kNextDone) {
        __syncthreads();
        return false;
    }
    // ---- direction d = -H g: fused dot products, scalar two-loop, one combination ------------
    int next;
    do {
        __syncthreads();
        const bool pending = S.st.pending != 0;
        fused_dots(V.S, V.Y, pending ? V.Y + (int64_t)S.st.head * fit_vec_pitch(P) : nullptr, V.g, P,
                   (unsigned)S.st.occ | (pending ? 1u << S.st.head : 0u), S.dots);
        if (tid < 32) decide_direction(S, F);
        __syncthreads();
        next = S.step.next;
    } while (next == kNextDirection);
    if (next == kNextTrial) {
        // d = -(cg g + sum cs_k s_k + sum cy_k y_k) and the first trial z + alpha d, eight pairs'
        // loads in flight per thread
        const float cg = S.cg, af = S.step.alpha;
        const int n = S.n_dir, Pp = fit_vec_pitch(P);
#pragma unroll 1
        for (int i = tid; i < P; i += nth) {
            float h = cg * V.g[i];
            int k = 0;
#pragma unroll 1
            for (; k + 7 < n; k += 8) {
                float s[8], y[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int64_t o = (int64_t)S.slot[k + u] * Pp + i;
                    s[u] = V.S[o];
                    y[u] = V.Y[o];
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) h = fmaf(S.cy[k + u], y[u], fmaf(S.cs[k + u], s[u], h));
            }
#pragma unroll 1
            for (; k < n; ++k) {
                const int64_t o = (int64_t)S.slot[k] * Pp + i;
                h = fmaf(S.cy[k], V.Y[o], fmaf(S.cs[k], V.S[o], h));
            }
            V.d[i] = -h;
            V.zt[i] = fmaf(af, -h, V.z[i]);
        }
    }
    __syncthreads();
    return next == kNextTrial;
}

__device__ __forceinline__ void init_state(FitState &st) {
    st.phase = kPhStart;
    st.f = INFINITY;
    st.edm = INFINITY;
    st.iters = 0;
    st.n_evals = 0;
    st.win_it = 0;
    st.f_win = INFINITY;
    st.status = FIT_STATUS_MAXITER;
    st.pending = 0;
    st.have_lo = 0;
    st.ls_it = 0;
    reset_history(st);
}

// Start point z0 = J^-1 (theta_start - theta0) into z (theta_start = theta0 if st == nullptr);
// pd is scratch, part as in theta_of_z. Ends with a barrier.
static __device__ void start_z(const DevModel &m, const double *st, float *z, float *pd, float *part) {
    const int tid = threadIdx.x, P = m.P, nth = blockDim.x;
#pragma unroll 1
    for (int i = tid; i < P; i += nth) {
        const float dd = st ? (float)(st[i] - m.theta0[i]) : 0.f;
        pd[i] = dd;
        const float s = m.zscale[i];
        if (s > 0.f) z[i] = dd / s;
    }
    __syncthreads();
    if (m.tri_rows > 0) {
        tri_apply(m, m.tri_lo, m.n_tri_lo, m.W_lo, pd, part);
        __syncthreads();
#pragma unroll 1
        for (int r = tid; r < m.tri_rows; r += nth) z[m.tri_param[r]] = tri_sum(m, part, r, false);
    }
    __syncthreads();
}

// Result: theta = theta0 + J z in double, and the fit's summary.
// Held parameters (fixed) are reported at their start values exactly (their z carries the
// start's FP32 rounding, ~1e-8 relative).
static __device__ void write_result(const DevModel &m, const FitState &st, const float *z, double *best,
                             fit_result *out, const double *start, const uint8_t *fixed) {
    const int tid = threadIdx.x;
#pragma unroll 1
    for (int i = tid; i < m.P; i += blockDim.x) {
        const float s = m.zscale[i];
        if (fixed && fixed[i]) best[i] = start ? start[i] : m.theta0[i];
        else if (s > 0.f) best[i] = m.theta0[i] + (double)s * (double)z[i];
    }
    for (int b = 0; b < m.n_blocks; ++b) {
        const int n = m.blk_size[b];
        const int *idx = m.blk_idx + m.blk_idx_off[b];
        // a thread per row over L^T (coalesced), four partial sums so that the products of one
        // row do not wait for one another
        const double *Lt = m.blk_L64 + m.blk_mat_off[b] + (int64_t)n * n;
#pragma unroll 1
        for (int i = tid; i < n; i += blockDim.x) {
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            int j = 0;
#pragma unroll 1
            for (; j + 3 <= i; j += 4) {
#pragma unroll
                for (int u = 0; u < 4; ++u) s[u] = fma(Lt[(int64_t)(j + u) * n + i], (double)z[idx[j + u]], s[u]);
            }
#pragma unroll 1
            for (; j <= i; ++j) s[0] = fma(Lt[(int64_t)j * n + i], (double)z[idx[j]], s[0]);
            best[idx[i]] = m.theta0[idx[i]] + ((s[0] + s[1]) + (s[2] + s[3]));
        }
    }
    if (tid == 0) {
        fit_result r;
        r.nll_min = st.f;
        r.edm = st.edm;
        r.iters = st.iters;
        r.n_evals = st.n_evals;
        r.status = st.status;
        r.pad = 0;
        *out = r;
    }
}

// At most T threads; MINB resident blocks per SM. Each block fits one instance at a time.
// GEN false: models of Eq. 1 or the three-flavour formula with the overlap-length energy
// correction; true: any model, the 3+1 formula and the spline correction included (a separate
// build, so that the common case carries none of their registers).
// PRE: the preconditioned build (fits in w, z = T w), used when the launch asks for it and every
// model of the batch has its preconditioner.
template <int T, int MINB, bool GEN, bool PRE>
__global__ void __launch_bounds__(T, MINB) fit_kernel(FitArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FitSmem &S = *reinterpret_cast<FitSmem *>(smem_raw);
    float *dyn = reinterpret_cast<float *>(smem_raw + sizeof(FitSmem));
    float *gws = A.ws_global + (int64_t)blockIdx.x * A.ws_stride;
    FitParams F;
    F.hist = A.hist;
    F.max_iter = A.max_iter;
    F.max_ls = A.max_ls;
    F.restarts = A.restarts;
    F.edm_tol = A.edm_tol;
    F.f_noise_rel = A.f_noise_rel;
    F.deadline = (A.began ? *A.began : global_ns()) + A.budget_ns;   // (the first thread's counts)
    const int tid = threadIdx.x;

    while (true) {
        if (tid == 0) S.inst = atomicAdd(A.queue, 1);
        __syncthreads();
        const int q = S.inst;
        __syncthreads();
        if (q >= A.n_inst) break;
        const int ii = A.order ? A.order[q] : q;   // queue position -> instance
        const fit_instance in = A.inst[ii];
        copy_model(&S.m, A.models + in.model);
        if (PRE && A.pre_tab) {   // the preconditioner of the datasets this instance fits
            if (tid == 0) {
                const uint32_t mk = in.mask & ((1u << S.m.n_ds) - 1u);
                const PreEntry *e = A.pre_tab + (int64_t)in.model * A.pre_per_model;
#pragma unroll 1
                for (int k = 0; k < A.pre_per_model; ++k)
                    if (e[k].Q && e[k].mask == mk) {
                        S.m.pre_Q = e[k].Q;
                        S.m.pre_c = e[k].c;
                        S.m.pre_r = e[k].r;
                        break;
                    }
            }
            __syncthreads();
        }
        const DevModel &m = S.m;
        const int P = m.P;
        // workspace: the 15 working vectors and the evaluation workspace in shared memory when
        // they fit, else in this block's global slice; the history in shared memory after them
        // unless it is placed in the global slice (hist_global)
        // (global slice: history first, then the rest)
        const int hfl = fit_hist_floats(P, F.hist), loc = fit_work_floats(P) + m.ws_floats;
        const bool loc_smem = loc + (A.hist_global ? 0 : hfl) <= A.smem_floats;
        float *base = loc_smem ? dyn : gws + (A.hist_global ? hfl : 0);
        float *hbase = A.hist_global ? gws : base + loc;
        FitVecs V = carve_fit_vecs(base, hbase, P, F.hist);
        float *ws = base + fit_work_floats(P);
        const float *data = A.data + in.data_off;
        constexpr bool pre = PRE;
        // (one thread reads the clock: the branches hold barriers, so the block must agree)
        if (tid == 0) {
            init_state(S.st);
            S.step.next = global_ns() > F.deadline ? kNextDone : kNextDirection;
        }
        __syncthreads();
        if (S.step.next == kNextDone) {
#pragma unroll 1
            for (int i = tid; i < P; i += blockDim.x) V.z[i] = 0.f;
            if (tid == 0) S.st.status = FIT_STATUS_TIMEOUT;
            __syncthreads();
        } else {
            start_z(m, A.start ? A.start + in.param_off : nullptr, V.zt, V.pd, ws);
            const uint8_t *fx = A.fixed ? A.fixed + in.param_off : nullptr;
            if (pre) pre_apply(m, m.pre_c + m.pre_r, V.zt, V.zt, S.pre_u, fx);   // w0 = T^-1 z0
            while (true) {
                const double fa = pre ? eval_w<GEN>(m, V.zt, V.gt, V, ws, data, in.mask, S, fx)
                                      : eval_z<GEN>(m, V.zt, V.gt, V, ws, data, in.mask, S, fx);
                if (!fit_decide(S, V, P, fa, F)) break;
            }
        }
        const float *zres = V.z;
        if (pre) {   // back to z = T w
            pre_apply(m, m.pre_c, V.z, V.zw, S.pre_u, A.fixed ? A.fixed + in.param_off : nullptr);
            zres = V.zw;
        }
        write_result(m, S.st, zres, A.best + in.param_off, A.results + ii,
                     A.start ? A.start + in.param_off : nullptr, A.fixed ? A.fixed + in.param_off : nullptr);
        __syncthreads();
    }
}

template <int T, int MINB>
static const void *fit_kernel_of(bool general, bool pre) {
    if (pre)
        return general ? reinterpret_cast<const void *>(&fit_kernel<T, MINB, true, true>)
                       : reinterpret_cast<const void *>(&fit_kernel<T, MINB, false, true>);
    return general ? reinterpret_cast<const void *>(&fit_kernel<T, MINB, true, false>)
                   : reinterpret_cast<const void *>(&fit_kernel<T, MINB, false, false>);
}

}  // namespace fitcore

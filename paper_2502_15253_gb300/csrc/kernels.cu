// Kernels of the forward-folding fit: batched expectation, batched -2lnL + gradient, and the
// lockstep fit engines. See dev_model.cuh for the per-block evaluation, fit_dev.cuh for the
// minimiser and the persistent fit kernel.
#include "fit_dev.cuh"

namespace fitcore {

// Prior in theta space (Eq. 6): sum ((theta-theta0)/sigma)^2 + sum_B d_B^T V_B^-1 d_B with
// V^-1 = W^T W (W = L^-1), evaluated as |W d|^2; gradient 2 W^T W d added to grad.
// zs: shared scratch of P floats; part: scratch of tri_segs x tri_rows floats. Returns the prior
// term (all threads). Starts with a barrier.
__device__ double prior_theta(const DevModel &m, const float *pd, float *grad, float *zs, float *part,
                              double *red) {
    const int tid = threadIdx.x, nth = blockDim.x;
    __syncthreads();
    float acc = 0.f;
#pragma unroll 1
    for (int i = tid; i < m.P; i += nth) {
        const float pi = m.prior_inv[i];
        if (pi > 0.f) {
            const float r = pd[i] * pi;
            acc = fmaf(r, r, acc);
            if (grad) grad[i] += 2.f * r * pi;
        }
    }
    if (m.tri_rows > 0) {
        tri_apply(m, m.tri_lo, m.n_tri_lo, m.W_lo, pd, part);
        __syncthreads();
#pragma unroll 1
        for (int r = tid; r < m.tri_rows; r += nth) {
            const float z = tri_sum(m, part, r, false);
            zs[m.tri_param[r]] = z;
            acc = fmaf(z, z, acc);
        }
        __syncthreads();
        if (grad) {
            tri_apply(m, m.tri_up, m.n_tri_up, m.W_up, zs, part);
            __syncthreads();
#pragma unroll 1
            for (int r = tid; r < m.tri_rows; r += nth) grad[m.tri_param[r]] += 2.f * tri_sum(m, part, r, true);
        }
    }
    return block_sum(acc, red);
}

// ------------------------------------------------------------------------------------
// batched expectation / evaluation in theta space: block per parameter vector
// ------------------------------------------------------------------------------------
struct alignas(16) EvalSmem {
    DevModel m;
    EvalShared E;
    double red[kMaxWarps + 1];
};

// T threads per block, MINB resident blocks per SM; GEN: any model (the 3+1 formula, the spline
// correction), else Eq. 1 and the three-flavour formula with the overlap rule. The dataset
// workspaces are in shared memory when ws_in_smem, else in this block's slice of ws_global.
template <int T, int MINB, bool GEN>
__global__ void __launch_bounds__(T, MINB) eval_kernel(EvalArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    EvalSmem &S = *reinterpret_cast<EvalSmem *>(smem_raw);
    copy_model(&S.m, A.model);
    const DevModel &m = S.m;
    const int P = m.P, Pp = fit_vec_pitch(P);
    float *pv = reinterpret_cast<float *>(smem_raw + sizeof(EvalSmem));
    float *pd = pv + Pp, *pl = pd + Pp, *grad = pl + Pp, *zs = grad + Pp;
    float *ws = A.ws_in_smem ? zs + Pp : A.ws_global + (int64_t)blockIdx.x * m.ws_floats;
    const ParVecs q{pv, pd, pl};
    const bool want_grad = A.grad != nullptr;

    for (int b = blockIdx.x; b < A.B; b += gridDim.x) {
        const double *th = A.theta + (int64_t)b * P;
#pragma unroll 1
        for (int i = threadIdx.x; i < P; i += blockDim.x) {
            const double t = th[i];
            const float h = (float)t, d = (float)(t - m.theta0[i]);
            pv[i] = h;
            pd[i] = d;
            pl[i] = presid(m, h, d, i);
            grad[i] = 0.f;
        }
        double nll = 0.0;
        if (A.mu) {
            expected_datasets<GEN>(m, S.E, q, ws, A.mu + (int64_t)b * m.n_data);
        } else {
            const float *dat = A.data ? A.data + (int64_t)b * m.n_data : m.asimov;
            const uint32_t mask = A.masks ? A.masks[b] : 0xffffffffu;
            nll = want_grad ? eval_datasets<GEN, true>(m, S.E, q, mask, dat, ws, grad)
                            : eval_datasets<GEN, false>(m, S.E, q, mask, dat, ws, nullptr);
        }
        const int st = S.E.status;
        if (A.mu == nullptr && st == 0) nll += prior_theta(m, pd, want_grad ? grad : nullptr, zs, ws, S.red);
        if (threadIdx.x == 0) {
            if (A.nll) A.nll[b] = st ? INFINITY : nll;
            if (A.status)
                A.status[b] = (st & kStEscale) ? FIT_STATUS_ESCALE_NONMONOTONE
                              : (st & kStMuNonpos) ? FIT_STATUS_MU_NONPOSITIVE : 0;
        }
        __syncthreads();
        if (want_grad)
#pragma unroll 1
            for (int i = threadIdx.x; i < P; i += blockDim.x) A.grad[(int64_t)b * P + i] = st ? NAN : grad[i];
        __syncthreads();
    }
}

size_t eval_smem_bytes(const DevModel &hm, bool ws_in_smem) {
    size_t b = sizeof(EvalSmem) + sizeof(float) * 5 * (size_t)fit_vec_pitch(hm.P);
    if (ws_in_smem) b += sizeof(float) * (size_t)hm.ws_floats;
    return (b + 15) & ~size_t(15);
}

const void *eval_kernel_func(int threads, bool general) {
    if (threads == 512)
        return general ? reinterpret_cast<const void *>(&eval_kernel<512, 1, true>)
                       : reinterpret_cast<const void *>(&eval_kernel<512, 1, false>);
    if (threads == 128)
        return general ? reinterpret_cast<const void *>(&eval_kernel<128, 4, true>)
                       : reinterpret_cast<const void *>(&eval_kernel<128, 4, false>);
    return general ? reinterpret_cast<const void *>(&eval_kernel<256, 2, true>)
                   : reinterpret_cast<const void *>(&eval_kernel<256, 2, false>);
}

// ------------------------------------------------------------------------------------
// lockstep engine
// ------------------------------------------------------------------------------------
size_t ls_state_bytes() { return sizeof(FitState); }
size_t ls_step_smem_bytes(const DevModel &hm) {
    return sizeof(FitSmem) + sizeof(float) * (size_t)hm.tri_segs * hm.tri_rows;
}

struct alignas(16) LsEvalSmem {
    DevModel m;
    EvalShared E;
};

size_t ls_eval_smem_bytes(int P, int ws_floats) {
    return sizeof(LsEvalSmem) + sizeof(float) * (3 * (size_t)fit_vec_pitch(P) + (size_t)ws_floats);
}

__device__ __forceinline__ FitVecs ls_vecs(const LsArgs &A, int g, int P) {
    float *base = A.vec + (int64_t)g * A.vec_stride;
    return carve_fit_vecs(base, base + fit_work_floats(P), P, A.hist);
}

__device__ __forceinline__ void copy_state(FitState *dst, const FitState *src) {
    const int n = (int)(sizeof(FitState) / sizeof(double));
    const double *s = reinterpret_cast<const double *>(src);
    double *d = reinterpret_cast<double *>(dst);
    for (int i = threadIdx.x; i < n; i += blockDim.x) d[i] = s[i];
}

__device__ __forceinline__ FitParams ls_params(const LsArgs &A) {
    FitParams F;
    F.hist = A.hist;
    F.max_iter = A.max_iter;
    F.max_ls = A.max_ls;
    F.restarts = A.restarts;
    F.edm_tol = A.edm_tol;
    F.f_noise_rel = A.f_noise_rel;
    F.deadline = *A.deadline;
    return F;
}

// Start points, theta of the first evaluation, state, and the first active list (all of them).
__global__ void __launch_bounds__(128) ls_init_kernel(LsArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FitSmem &S = *reinterpret_cast<FitSmem *>(smem_raw);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *A.deadline = global_ns() + A.budget_ns;
        *A.n_act_next = A.n;
    }
    copy_model(&S.m, A.model);
    float *part = reinterpret_cast<float *>(smem_raw + sizeof(FitSmem));
    const DevModel &m = S.m;
    const int P = m.P, nd = m.n_ds;
    for (int g = blockIdx.x; g < A.n; g += gridDim.x) {
        const fit_instance in = A.inst[A.group[g]];
        FitVecs V = ls_vecs(A, g, P);
        start_z(m, A.start ? A.start + in.param_off : nullptr, V.zt, V.pd, part);
        if (A.precond) {   // w0 = T^-1 z0; the trial's z = T w0 is kept in zw
            const uint8_t *fx = A.fixed ? A.fixed + in.param_off : nullptr;
            pre_apply(m, m.pre_c + m.pre_r, V.zt, V.zt, S.pre_u, fx);
            pre_apply(m, m.pre_c, V.zt, V.zw, S.pre_u, fx);
            theta_of_z(m, V.zw, V, part);
        } else {
            theta_of_z(m, V.zt, V, part);
        }
        for (int i = threadIdx.x; i < nd * P; i += blockDim.x) A.gsl[(int64_t)g * nd * P + i] = 0.f;
        if (threadIdx.x == 0) {
            init_state(S.st);
            A.stat[g] = 0;
            A.act_next[g] = g;
        }
        __syncthreads();
        copy_state(A.state + g, &S.st);
        __syncthreads();
    }
}

// Parameter vectors of group index g into shared memory (three vectors on the fit pitch).
__device__ __forceinline__ ParVecs ls_params_in(const LsArgs &A, int g, int P, float *pv) {
    const FitVecs V = ls_vecs(A, g, P);
    float *pd = pv + fit_vec_pitch(P), *pl = pd + fit_vec_pitch(P);
#pragma unroll 1
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
        pv[i] = V.pv[i];
        pd[i] = V.pd[i];
        pl[i] = V.pl[i];
    }
    return ParVecs{pv, pd, pl};
}

// Forward pass and likelihood of one (instance, dataset) per block iteration: stages A (no
// partials), B, C, C2; stores the dataset's -2lnL, dD/dmu and the efficiency / background
// gradient contributions.
template <bool GEN>
__device__ __forceinline__ void ls_forward_body(LsArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LsEvalSmem &S = *reinterpret_cast<LsEvalSmem *>(smem_raw);
    copy_model(&S.m, A.model);
    const DevModel &m = S.m;
    const int P = m.P, nd = m.n_ds, na = *A.n_act;
    float *pv = reinterpret_cast<float *>(smem_raw + sizeof(LsEvalSmem));
    float *wsb = A.ws_in_smem ? pv + 3 * fit_vec_pitch(P) : A.ws_global + (int64_t)blockIdx.x * A.ws_stride;
    const DsWs ws = carve_ds_ws(wsb, m.N_t, m.C, m.max_reco, m.n_osc);
    for (int it = blockIdx.x; it < na * nd; it += gridDim.x) {
        const int g = A.act[it / nd], d = it % nd;
        const fit_instance in = A.inst[A.group[g]];
        const int64_t gd = (int64_t)g * nd + d;
        if (!((in.mask >> d) & 1u)) {
            if (threadIdx.x == 0) A.nll_ds[gd] = 0.0;
            continue;
        }
        const ParVecs q = ls_params_in(A, g, P, pv);
        if (threadIdx.x == 0) {
            S.E.status = 0;
            S.E.nll = 0.0;
        }
        eval_setup_any<GEN>(m, S.E, q, 1u << d, 0, 1);
        if (S.E.n) {
            st_signal<false, GEN>(m, S.E, q, wsb);
            st_remap<GEN>(m, S.E, wsb);
            st_fold(m, S.E, wsb);
            st_lik<true>(m, S.E, q, A.data + in.data_off, wsb);
            if (!S.E.status) {
                lik_finish<true>(m, S.E, A.gsl + gd * P);
                __syncthreads();
                if (threadIdx.x == 0) lik_dups(m, S.E, A.gsl + gd * P);
                if (m.shared_roles) __syncthreads();
                st_bkg_shape(m, S.E, wsb, A.gsl + gd * P);
            }
            const int nr = m.ds[d].n_reco;
            float *gm = A.gmu + gd * m.max_reco;
            for (int j = threadIdx.x; j < nr; j += blockDim.x) gm[j] = ws.gmu[j];
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            const int st = S.E.bad ? kStEscale : S.E.status;
            A.nll_ds[gd] = S.E.nll;
            if (st) atomicOr(&A.stat[g], st);
        }
        __syncthreads();
    }
}

// basic build (Eq. 1 / three-flavour, overlap correction) and general build (any model)
__global__ void __launch_bounds__(128) ls_forward_kernel(LsArgs A) { ls_forward_body<false>(A); }
__global__ void __launch_bounds__(128) ls_forward_kernel6(LsArgs A) { ls_forward_body<true>(A); }

// Adjoint of one (instance, dataset) per block iteration: stage A again with the partials,
// then stages D, E, F into the dataset's gradient slice.
template <bool GEN>
__device__ __forceinline__ void ls_adjoint_body(LsArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LsEvalSmem &S = *reinterpret_cast<LsEvalSmem *>(smem_raw);
    copy_model(&S.m, A.model);
    const DevModel &m = S.m;
    const int P = m.P, nd = m.n_ds, na = *A.n_act;
    float *pv = reinterpret_cast<float *>(smem_raw + sizeof(LsEvalSmem));
    float *wsb = A.ws_in_smem ? pv + 3 * fit_vec_pitch(P) : A.ws_global + (int64_t)blockIdx.x * A.ws_stride;
    const DsWs ws = carve_ds_ws(wsb, m.N_t, m.C, m.max_reco, m.n_osc);
    for (int it = blockIdx.x; it < na * nd; it += gridDim.x) {
        const int g = A.act[it / nd], d = it % nd;
        const fit_instance in = A.inst[A.group[g]];
        if (!((in.mask >> d) & 1u) || A.stat[g] != 0) continue;
        const int64_t gd = (int64_t)g * nd + d;
        const ParVecs q = ls_params_in(A, g, P, pv);
        const int nr = m.ds[d].n_reco;
        const float *gm = A.gmu + gd * m.max_reco;
        for (int j = threadIdx.x; j < nr; j += blockDim.x) ws.gmu[j] = gm[j];
        eval_setup_any<GEN>(m, S.E, q, 1u << d, 0, 1);
        if (S.E.n) {
            st_signal<true, GEN>(m, S.E, q, wsb);
            st_adjoint_fold(m, S.E, wsb);
            __syncthreads();
            st_adjoint_rest<GEN>(m, S.E, wsb, A.gsl + gd * P);
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(128) ls_adjoint_kernel(LsArgs A) { ls_adjoint_body<false>(A); }
__global__ void __launch_bounds__(128) ls_adjoint_kernel6(LsArgs A) { ls_adjoint_body<true>(A); }

// ---- lockstep rounds with the folds on the tensor cores (engine 2) ---------------------------
// Between these kernels the library runs, per dataset d, F_d = V_d R^T and GV_d = G_d R as
// split-TF32 GEMMs over the active instances (row a of each matrix = active position a). Each
// (instance, dataset) pair keeps its own evaluation workspace for the whole round, so the
// survival partials of the forward pass serve the adjoint without being recomputed.

__device__ __forceinline__ float tf32_hi(float x) {
    uint32_t b = __float_as_uint(x);
    b = (b + 0x1000u) & 0xFFFFE000u;   // nearest value with 10 mantissa bits
    return __uint_as_float(b);
}

// Stage A (with the partials) and B per (instance, dataset); v as TF32 high part and rest.
template <bool GEN>
__device__ __forceinline__ void ls_tc_fwd_body(LsArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LsEvalSmem &S = *reinterpret_cast<LsEvalSmem *>(smem_raw);
    copy_model(&S.m, A.model);
    const DevModel &m = S.m;
    const int P = m.P, nd = m.n_ds, na = *A.n_act;
    float *pv = reinterpret_cast<float *>(smem_raw + sizeof(LsEvalSmem));
    for (int it = blockIdx.x; it < na * nd; it += gridDim.x) {
        const int a = it / nd, d = it % nd, g = A.act[a];
        const fit_instance in = A.inst[A.group[g]];
        const int64_t gd = (int64_t)g * nd + d;
        if (!((in.mask >> d) & 1u)) {
            if (threadIdx.x == 0) A.nll_ds[gd] = 0.0;
            continue;
        }
        float *wsb = A.ws_global + (int64_t)it * A.ws_stride;
        const DsWs ws = carve_ds_ws(wsb, m.N_t, m.C, m.max_reco, m.n_osc);
        const ParVecs q = ls_params_in(A, g, P, pv);
        eval_setup_any<GEN>(m, S.E, q, 1u << d, 0, 1);
        if (S.E.n) {
            st_signal<true, GEN>(m, S.E, q, wsb);
            st_remap<GEN>(m, S.E, wsb);
            float *vh = A.vhi + ((int64_t)d * A.n + a) * m.ldt, *vl = A.vlo + ((int64_t)d * A.n + a) * m.ldt;
            for (int t = threadIdx.x; t < m.ldt; t += blockDim.x) {
                const float x = t < m.N_t ? ws.v[t] : 0.f;
                const float hi = tf32_hi(x);
                vh[t] = hi;
                vl[t] = x - hi;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0 && S.E.bad) atomicOr(&A.stat[g], kStEscale);
        __syncthreads();
    }
}

__global__ void __launch_bounds__(128) ls_tc_fwd_kernel(LsArgs A) { ls_tc_fwd_body<false>(A); }
__global__ void __launch_bounds__(128) ls_tc_fwd_kernel6(LsArgs A) { ls_tc_fwd_body<true>(A); }

// Stage C2 per (instance, dataset) from the fold F = R v of the GEMM: -2lnL, dD/dmu (TF32
// high part and rest for the adjoint GEMM), efficiency and background gradients.
template <bool GEN>
__device__ __forceinline__ void ls_tc_lik_body(LsArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LsEvalSmem &S = *reinterpret_cast<LsEvalSmem *>(smem_raw);
    copy_model(&S.m, A.model);
    const DevModel &m = S.m;
    const int P = m.P, nd = m.n_ds, na = *A.n_act;
    float *pv = reinterpret_cast<float *>(smem_raw + sizeof(LsEvalSmem));
    for (int it = blockIdx.x; it < na * nd; it += gridDim.x) {
        const int a = it / nd, d = it % nd, g = A.act[a];
        const fit_instance in = A.inst[A.group[g]];
        const int64_t gd = (int64_t)g * nd + d;
        if (!((in.mask >> d) & 1u) || A.stat[g] != 0) continue;
        float *wsb = A.ws_global + (int64_t)it * A.ws_stride;
        const DsWs ws = carve_ds_ws(wsb, m.N_t, m.C, m.max_reco, m.n_osc);
        const int nr = m.ds[d].n_reco;
        const float *fr = A.fbuf + ((int64_t)d * A.n + a) * A.ldf;
        const ParVecs q = ls_params_in(A, g, P, pv);
        for (int j = threadIdx.x; j < nr; j += blockDim.x) {
            ws.f0[j] = fr[j];
            ws.gmu[j] = 0.f;   // (the fold's low part: none here)
        }
        if (threadIdx.x == 0) {
            S.E.status = 0;
            S.E.nll = 0.0;
        }
        eval_setup_any<GEN>(m, S.E, q, 1u << d, 0, 1);
        if (S.E.n) {
            st_lik<true>(m, S.E, q, A.data + in.data_off, wsb);
            if (!S.E.status) {
                lik_finish<true>(m, S.E, A.gsl + gd * P);
                __syncthreads();
                if (threadIdx.x == 0) lik_dups(m, S.E, A.gsl + gd * P);
                if (m.shared_roles) __syncthreads();
                st_bkg_shape(m, S.E, wsb, A.gsl + gd * P);
            }
            float *gh = A.ghi + ((int64_t)d * A.n + a) * A.ldr, *gl = A.glo + ((int64_t)d * A.n + a) * A.ldr;
            for (int j = threadIdx.x; j < A.ldr; j += blockDim.x) {
                const float x = j < nr ? ws.gmu[j] : 0.f;
                const float hi = tf32_hi(x);
                gh[j] = hi;
                gl[j] = x - hi;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            const int st = S.E.bad ? kStEscale : S.E.status;
            A.nll_ds[gd] = S.E.nll;
            if (st) atomicOr(&A.stat[g], st);
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(128) ls_tc_lik_kernel(LsArgs A) { ls_tc_lik_body<false>(A); }
__global__ void __launch_bounds__(128) ls_tc_lik_kernel6(LsArgs A) { ls_tc_lik_body<true>(A); }

// Stages E and F per (instance, dataset) from GV = R^T dD/dmu of the GEMM (gv = eff GV).
template <bool GEN>
__device__ __forceinline__ void ls_tc_adj_body(LsArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LsEvalSmem &S = *reinterpret_cast<LsEvalSmem *>(smem_raw);
    copy_model(&S.m, A.model);
    const DevModel &m = S.m;
    const int P = m.P, nd = m.n_ds, na = *A.n_act;
    float *pv = reinterpret_cast<float *>(smem_raw + sizeof(LsEvalSmem));
    for (int it = blockIdx.x; it < na * nd; it += gridDim.x) {
        const int a = it / nd, d = it % nd, g = A.act[a];
        const fit_instance in = A.inst[A.group[g]];
        if (!((in.mask >> d) & 1u) || A.stat[g] != 0) continue;
        const int64_t gd = (int64_t)g * nd + d;
        float *wsb = A.ws_global + (int64_t)it * A.ws_stride;
        const DsWs ws = carve_ds_ws(wsb, m.N_t, m.C, m.max_reco, m.n_osc);
        const ParVecs q = ls_params_in(A, g, P, pv);
        eval_setup_any<GEN>(m, S.E, q, 1u << d, 0, 1);
        if (S.E.n) {
            const float *gr = A.gvbuf + ((int64_t)d * A.n + a) * m.ldt;
            for (int k = threadIdx.x; k < m.N_t; k += blockDim.x) ws.v[k] = pmul(S.E.eff[0], gr[k]);
            __syncthreads();
            st_adjoint_rest<GEN>(m, S.E, wsb, A.gsl + gd * P);
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(128) ls_tc_adj_kernel(LsArgs A) { ls_tc_adj_body<false>(A); }
__global__ void __launch_bounds__(128) ls_tc_adj_kernel6(LsArgs A) { ls_tc_adj_body<true>(A); }

// Minimiser step per active instance: gathers the round's evaluation (dataset sums, prior,
// gradient in z), runs fit_decide, and either prepares theta of the next trial point and puts
// the instance on the next active list, or writes its result.
__global__ void __launch_bounds__(128) ls_step_kernel(LsArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FitSmem &S = *reinterpret_cast<FitSmem *>(smem_raw);
    copy_model(&S.m, A.model);
    float *part = reinterpret_cast<float *>(smem_raw + sizeof(FitSmem));
    const DevModel &m = S.m;
    const int P = m.P, nd = m.n_ds, na = *A.n_act;
    const FitParams F = ls_params(A);
    for (int a = blockIdx.x; a < na; a += gridDim.x) {
        const int g = A.act[a];
        const int ii = A.group[g];
        const fit_instance in = A.inst[ii];
        FitVecs V = ls_vecs(A, g, P);
        copy_state(&S.st, A.state + g);
        // theta gradient = sum of the dataset slices in a fixed order; the slices are cleared
        float *gs = A.gsl + (int64_t)g * nd * P;
#pragma unroll 1
        for (int i = threadIdx.x; i < P; i += blockDim.x) {
            float t = 0.f;
            for (int d = 0; d < nd; ++d) {
                if ((in.mask >> d) & 1u) t += gs[(int64_t)d * P + i];
                gs[(int64_t)d * P + i] = 0.f;
            }
            V.gth[i] = t;
        }
        const int st = A.stat[g];
        double fa = 0.0;
        for (int d = 0; d < nd; ++d)
            if ((in.mask >> d) & 1u) fa += A.nll_ds[(int64_t)g * nd + d];
        __syncthreads();
        const uint8_t *fx = A.fixed ? A.fixed + in.param_off : nullptr;
        if (st != 0) {
            fa = INFINITY;
        } else if (A.precond) {   // z of the trial in zw; g_w = T g_z
            fa += eval_z_prior(m, V.zw, V.gth, V.gzw, part, S.red);
            hold_fixed(fx, V.gzw, P);
            __syncthreads();
            pre_apply(m, m.pre_c, V.gzw, V.gt, S.pre_u, fx);
        } else {
            fa += eval_z_prior(m, V.zt, V.gth, V.gt, part, S.red);
            hold_fixed(fx, V.gt, P);
        }
        const bool more = fit_decide(S, V, P, fa, F);
        if (more) {
            if (A.precond) {
                pre_apply(m, m.pre_c, V.zt, V.zw, S.pre_u, fx);
                theta_of_z(m, V.zw, V, part);
            } else {
                theta_of_z(m, V.zt, V, part);
            }
            if (threadIdx.x == 0) {
                A.stat[g] = 0;
                A.act_next[atomicAdd(A.n_act_next, 1)] = g;
            }
        } else {
            const float *zres = V.z;
            if (A.precond) {   // back to z = T w
                pre_apply(m, m.pre_c, V.z, V.zw, S.pre_u, fx);
                zres = V.zw;
            }
            write_result(m, S.st, zres, A.best + in.param_off, A.results + ii,
                         A.start ? A.start + in.param_off : nullptr, fx);
        }
        __syncthreads();
        copy_state(A.state + g, &S.st);
        __syncthreads();
    }
}

__global__ void clock_kernel(uint64_t *t) { *t = global_ns(); }

const void *fit_kernel_func(int threads, int variant, bool general, bool pre) {
    if (threads > 256) return fit_kernel_512(general, pre);
    if (threads > 128) return fit_kernel_256(general, pre);
    return variant == 5 ? fit_kernel_128x5(general, pre) : fit_kernel_128x4(general, pre);
}

size_t fit_smem_bytes(int floats) { return sizeof(FitSmem) + sizeof(float) * (size_t)floats; }

}  // namespace fitcore

// Expected counts for the rows of the linearised fit and of the preconditioner (fisher_U, lin_base and
// linear_mle_rows in capi.cu): Jacobians by central differences, 0.01 apart in z.
//
// The difference of two expectations keeps few of their digits, and the rows of strongly
// correlated nuisances cancel further, so what a start point is made of includes the FP32
// rounding of these expectations: evaluated in another order they are as accurate, but start
// points then move by up to 1e-2 of a parameter (flat directions; 2.4e-4 of the vector). So the
// order of operations here is fixed - datasets one after another, a thread per bin over the
// cores, sincospif, a warp per reco row - and the faster evaluation (dev_model.cuh) is free to
// change its own. A model calls this once per geometry and dataset subset.
#include <algorithm>
#include <string>

#include "kernels.cuh"

int fitcore_fail(int code, const std::string &msg);
void fitcore_count_launch();
int fitcore_raise_eval_smem(const void *func, size_t bytes);   // capi.cu

namespace fitcore {

namespace {

namespace fixed_order {

__device__ __forceinline__ void phase_sc(float dm, float dm_lo, float c_hi, float c_lo, float &s,
                                         float &c) {
    const float yh = dm * c_hi;
    const float yl = fmaf(dm, c_hi, -yh) + fmaf(dm, c_lo, dm_lo * c_hi);
    const float r = (yh - rintf(yh)) + yl;
    sincospif(r, &s, &c);
}

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


}  // namespace fixed_order

struct RowSmem {
    DevModel m;
    int status;
};

// A dataset's expected counts; NOSC 6: the 3+1 formula.
template <int NOSC>
__device__ void expected_dataset(const DevModel &m, int d, const float *pv, const float *pd, float *u, float *v,
                                 float *f0, int *status, float *mu_out) {
    const DevDataset &ds = m.ds[d];
    const DevDetector &dt = m.det[ds.det];
    const int N_t = m.N_t, C = m.C, nr = ds.n_reco;
    const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
    auto pair = [&](int p, float dflt) { return p < 0 ? PP{dflt, 0.f} : PP{pv[p], presid(m, pv[p], pd[p], p)}; };
    float eta[NOSC], eta_lo[NOSC];
    F2 e[NOSC];
#pragma unroll
    for (int i = 0; i < NOSC; ++i) {
        const int p = m.osc_idx[i];
        if (osc_is_dm(m.osc_mode, i)) {
            eta[i] = p >= 0 ? m.theta0_f[p] : m.osc_val[i];
            eta_lo[i] = p >= 0 ? m.theta0_lo[p] + pd[p] : m.osc_val_lo[i];
        } else {
            eta[i] = p >= 0 ? pv[p] : m.osc_val[i];
            eta_lo[i] = 0.f;
        }
        e[i] = p >= 0 ? f2_norm(pv[p], presid(m, pv[p], pd[p], p)) : F2{m.osc_val[i], m.osc_val_lo[i]};
    }
    const auto kc = OscTraits<NOSC>::coef(m.osc_mode, e);
    const PP nrm = pair(ds.norm_idx, 1.f), eff = pair(ds.eff_idx, 1.f);
    const EMap em = make_emap(m, ds, pv, pd);
    {
        const float s0 = em.slope(m.e_edge[0]), s1 = em.slope(m.e_edge[N_t]);
        if (!(s0 > 0.25f && s0 < 4.f && s1 > 0.25f && s1 < 4.f)) {
            if (tid == 0) atomicOr(status, kStEscale);
            return;
        }
    }
    for (int k = tid; k < N_t; k += nth) {
        const float ih = m.inv_e_hi[k], il = m.inv_e_lo[k];
        float pt = 0.f;
        for (int cc = 0; cc < C; ++cc) {
            const float w = ds.w[cc];
            if (w == 0.f) continue;
            const float ch = ds.kl_hi[cc] * ih;
            const float cl = fmaf(ds.kl_hi[cc], ih, -ch) + ds.kl_hi[cc] * il + ds.kl_lo[cc] * ih;
            float dP[NOSC];
            float P;
            if constexpr (NOSC == 6)
                P = fixed_order::survival_sterile(eta, eta_lo, kc, ch, cl, dP);
            else
                P = fixed_order::survival_mode(m.osc_mode, eta, eta_lo, kc, ch, cl, dP);
            pt += pmul(pair(m.core_power_idx[cc], 1.f), w * P);
        }
        const float ts = pmul(pair(ds.shape_idx[k], 1.f), ds.t[k]);
        u[k] = pmul(nrm, ts * pt);
    }
    __syncthreads();
    for (int t = tid; t < N_t; t += nth) {
        if (m.remap_mode == FIT_REMAP_SPLINE) {
            v[t] = fixed_order::spline_target(u, m.e_edge, em, t, N_t);
            continue;
        }
        int k = t - (int)floorf(em.disp(m.e_edge[t]));
        k = min(max(k, 0), N_t - 1);
        k = t - (int)floorf(em.disp(m.e_edge[k]));
        k = min(max(k - 1, 0), N_t - 1);
        while (k > 0 && (float)(k - t) + em.disp(m.e_edge[k]) > 0.f) --k;
        while (k + 1 < N_t && (float)(k + 1 - t) + em.disp(m.e_edge[k + 1]) <= 0.f) ++k;
        float acc = 0.f;
        float dlo = em.disp(m.e_edge[k]);
        for (; k < N_t; ++k) {
            const float dhi = em.disp(m.e_edge[k + 1]);
            const float ylo = (float)(k - t) + dlo;
            const float yhi = (float)(k + 1 - t) + dhi;
            if (ylo >= 1.f) break;
            const float ov = fminf(yhi, 1.f) - fmaxf(ylo, 0.f);
            if (ov > 0.f) acc = fmaf(u[k], ov / (1.f + (dhi - dlo)), acc);
            dlo = dhi;
        }
        v[t] = acc;
    }
    __syncthreads();
    // a warp per row over its band, two strides of 32 bins; R = its TF32 part + the rest, exactly
    for (int j = warp; j < nr; j += nw) {
        const int2 band = dt.row_band[j];
        const float *rh = dt.rdense_hi + (int64_t)j * m.ldt + band.x, *rl = dt.rdense_lo + (int64_t)j * m.ldt + band.x;
        float s0 = 0.f, s1 = 0.f;
        for (int b = lane; b < band.y; b += 64) {
            s0 = fmaf(rh[b] + rl[b], v[band.x + b], s0);
            if (b + 32 < band.y) s1 = fmaf(rh[b + 32] + rl[b + 32], v[band.x + b + 32], s1);
        }
        float t = s0 + s1;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) f0[j] = t;
    }
    __syncthreads();
    for (int j = tid; j < nr; j += nth) {
        float mu = pmul(eff, f0[j]);
        for (int b = ds.bkg_begin; b < ds.bkg_end; ++b) {
            const DevBkg &bk = m.bkg[b];
            const float tm = bk.tmpl[j];
            const float shaped = bk.shape_idx[j] >= 0 ? fmaf(tm, pv[bk.shape_idx[j]], tm) : tm;
            mu += pmul(pair(bk.rate_idx, 1.f), shaped);
        }
        mu_out[ds.data_off + j] = mu;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(256) expected_rows_kernel(const DevModel *__restrict__ gm, int B,
                                                            const double *__restrict__ theta, float *__restrict__ mu,
                                                            int *__restrict__ status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RowSmem &S = *reinterpret_cast<RowSmem *>(smem_raw);
    {
        const int n = (int)(sizeof(DevModel) / sizeof(int));
        const int *src = reinterpret_cast<const int *>(gm);
        int *dst = reinterpret_cast<int *>(&S.m);
        for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    const DevModel &m = S.m;
    float *pv = reinterpret_cast<float *>(smem_raw + ((sizeof(RowSmem) + 15) & ~size_t(15)));
    float *pd = pv + m.P, *u = pd + m.P, *v = u + m.N_t, *f0 = v + m.N_t;
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
        const double *th = theta + (int64_t)b * m.P;
        for (int i = threadIdx.x; i < m.P; i += blockDim.x) {
            pv[i] = (float)th[i];
            pd[i] = (float)(th[i] - m.theta0[i]);
        }
        if (threadIdx.x == 0) S.status = 0;
        __syncthreads();
        for (int d = 0; d < m.n_ds; ++d) {
            if (m.osc_mode == FIT_OSC_STERILE4)
                expected_dataset<6>(m, d, pv, pd, u, v, f0, &S.status, mu + (int64_t)b * m.n_data);
            else
                expected_dataset<4>(m, d, pv, pd, u, v, f0, &S.status, mu + (int64_t)b * m.n_data);
            __syncthreads();
            const int bad = S.status;
            __syncthreads();   // every warp has read it before the next dataset can set it
            if (bad) break;
        }
        if (threadIdx.x == 0) status[b] = S.status ? FIT_STATUS_ESCALE_NONMONOTONE : 0;
        __syncthreads();
    }
}

}  // namespace

// theta [B x P], mu [B x n_data], status [B]: device buffers. Asynchronous on s.
int expected_rows(const DevModel &h, const DevModel *dev, int B, const double *theta, float *mu, int *status,
                  cudaStream_t s) {
    const size_t smem = ((sizeof(RowSmem) + 15) & ~size_t(15)) + sizeof(float) * (2 * (size_t)h.P + 2 * h.N_t + h.max_reco);
    // (raised only: the attribute is shared with other threads' calls for larger models)
    if (fitcore_raise_eval_smem(reinterpret_cast<const void *>(&expected_rows_kernel), smem) != FIT_OK) {
        cudaGetLastError();
        return FIT_ERR_CUDA;
    }
    expected_rows_kernel<<<std::min(B, 152 * 4), 256, smem, s>>>(dev, B, theta, mu, status);
    fitcore_count_launch();
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fitcore_fail(FIT_ERR_CUDA, std::string("expected rows: ") + cudaGetErrorString(e));
    return FIT_OK;
}

}  // namespace fitcore

// Batched expectation with the response fold on tensor cores: for B parameter vectors,
//   V_d[b][k] = (M(a) u)_k        energy-corrected true spectrum of dataset d (CUDA cores)
//   F_d = V_d R_d^T               fold, one GEMM per dataset (tcgen05, TF32 or split 3xTF32)
//   mu[b][d][j] = eps F + backgrounds
// The fold is the one dense contraction of the path: one response matrix times many spectra.
// Plain TF32 keeps 11 significant bits per operand (training-set generation for the warm
// start); the split form F = Vh Rh^T + Vh Rl^T + Vl Rh^T, with x = xh + xl and xh exact in TF32,
// restores FP32-level accuracy where the expectation is compared with the FP64 oracle.
#include <algorithm>
#include <cstring>
#include <string>

#include "gemm_tc.cuh"
#include "kernels.cuh"

int fitcore_fail(int code, const std::string &msg);
void fitcore_count_launch();
int fitcore_raise_eval_smem(const void *func, size_t bytes);   // capi.cu

namespace fitcore {

namespace {

// TF32-exact round-to-nearest of x (10 explicit mantissa bits), as a float
__device__ __forceinline__ float tf32_round(float x) {
    uint32_t b = __float_as_uint(x);
    b = (b + 0x1000u) & 0xFFFFE000u;
    return __uint_as_float(b);
}

// One (instance b, dataset d) at a time per block (grid.y = datasets, the instances strided over
// grid.x): survival x reweights on the true grid (the evaluation's sums over core pairs, without
// derivatives), energy correction gathered per target bin, written as V_hi / V_lo rows of length
// ldt. Blocks of dataset 0 also store the instance's parameter pairs for the epilogue.
// Bound by instruction issue in the survival sums (20 000 bin-cores per instance and dataset on
// the 53 km model); a block keeps its copy of the model's header for all its instances. 4096
// instances of that model took 700 us with a block per (instance, dataset), FP64 coefficients
// by one thread and the phase count of the formula tested per bin.
struct SignalSmem {
    DevModel m;
    EvalShared E;
};
inline size_t signal_smem_bytes(const DevModel &h) {
    const int edge = (h.N_t + 4) & ~3;
    return sizeof(SignalSmem) + sizeof(float) * (3 * (size_t)fit_vec_pitch(h.P) + ((h.N_t + 3) & ~3) +
                                                 (h.remap_mode == FIT_REMAP_SPLINE ? 3 : 1) * edge);
}

// Four blocks of 256 fit the registers (62 a thread): with 32 instead of 24 warps per SM 4096
// instances of the 53 km model (2000 bins) took 549 us instead of 567. On short rows the set-up
// and its barriers weigh more than the sums, and more, smaller blocks hide them: 128 threads
// against 256 for 4000 instances took 44 against 50 us with 200 bins, 171 against 208 with 400, 111
// against 120 with 600, but 245 against 239 with 997 and 557 against 549 with 2000 (four even
// quarters per block: 160 or 224 threads lose 6 % there).
constexpr int kSignalThreads = 256;
inline int signal_threads(int n_t) { return n_t <= 640 ? 128 : kSignalThreads; }

template <int NOSC, int MODE>
__global__ void __launch_bounds__(kSignalThreads, 4) signal_v_kernel(const DevModel *__restrict__ gm, int B,
                                                          const double *__restrict__ theta, float *__restrict__ vhi,
                                                          float *__restrict__ vlo, float *__restrict__ pv_out,
                                                          float *__restrict__ pl_out, int *__restrict__ status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SignalSmem &S = *reinterpret_cast<SignalSmem *>(smem_raw);
    {
        const int n = (int)(sizeof(DevModel) / sizeof(int));
        const int *src = reinterpret_cast<const int *>(gm);
        int *dst = reinterpret_cast<int *>(&S.m);
        for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    const DevModel &m = S.m;
    const int d = blockIdx.y, tid = threadIdx.x, nth = blockDim.x, N_t = m.N_t;
    const int Pp = fit_vec_pitch(m.P), edge = (N_t + 4) & ~3;
    float *pv = reinterpret_cast<float *>(smem_raw + sizeof(SignalSmem)), *pd = pv + Pp, *pl = pd + Pp;
    float *u = pl + Pp;
    EdgeTab T;   // (overlap rule: T.t holds the displacements of the grid edges)
    T.t = u + ((N_t + 3) & ~3);
    T.r = T.t + edge;
    T.k = reinterpret_cast<int *>(T.r + edge);
    const ParVecs q{pv, pd, pl};
    const DevDataset &ds = m.ds[d];
    const bool spline = m.remap_mode == FIT_REMAP_SPLINE;
#pragma unroll 1
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
        const double *th = theta + (int64_t)b * m.P;
        for (int i = tid; i < m.P; i += nth) {
            const double t = th[i];
            const float h = (float)t, del = (float)(t - m.theta0[i]);
            pv[i] = h;
            pd[i] = del;
            pl[i] = presid(m, h, del, i);
            if (d == 0) {
                pv_out[(int64_t)b * m.P + i] = h;
                pl_out[(int64_t)b * m.P + i] = pl[i];
            }
        }
        eval_setup<NOSC>(m, S.E, q, 1u << d, 0, 1);
        float *vh = vhi + ((int64_t)d * B + b) * m.ldt, *vl = vlo + ((int64_t)d * B + b) * m.ldt;
        if (S.E.bad) {   // (block-uniform) the energy map is not increasing on the grid
            if (tid == 0) atomicExch(&status[b], FIT_STATUS_ESCALE_NONMONOTONE);
            for (int k = tid; k < m.ldt; k += nth) vh[k] = vl[k] = 0.f;
            continue;
        }
        const PP nrm = S.E.nrm[0];
        const EMap em = S.E.em[0];
#pragma unroll 1
        for (int k = tid; k < N_t; k += nth) {
            const float ih = m.inv_e_hi[k], il = m.inv_e_lo[k], e0 = m.e_edge[k], e1 = m.e_edge[k + 1];
            const int sp = ds.shape_idx[k];
            const float tk = ds.t[k];
            float pt, corr, dpt[NOSC];
            CoreSums<false, NOSC, MODE>::run(S.E, 0, m.C, ih, il, nullptr, 0, pt, corr, dpt);
            const float ts = pmul(ppair(q, sp, 1.f), tk);
            const float x = pmul(nrm, fmaf(ts, pt, ts * corr));
            if (spline) {
                u[k] = x;
                edge_store(T, m.e_edge, em, k, N_t);
                if (k == N_t - 1) edge_store(T, m.e_edge, em, N_t, N_t);
            } else {
                const float d0 = em.disp(e0), d1 = em.disp(e1);
                u[k] = x / (1.f + (d1 - d0));
                T.t[k] = d0;
                if (k == N_t - 1) T.t[N_t] = d1;
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int t = tid; t < m.ldt; t += nth) {
            float acc = 0.f;
            if (t < N_t) acc = spline ? spline_target(u, T, t, N_t) : overlap_target(u, T.t, em.inv_slope, t, N_t);
            const float hi = tf32_round(acc);
            vh[t] = hi;
            vl[t] = acc - hi;
        }
    }
}

// mu[b][off_d + j] = eps_d F_d[b][j] + sum_b r B (1 + delta), NaN where the instance has a status; a
// block per instance at a time
__global__ void __launch_bounds__(128) mu_epilogue_kernel(const DevModel *__restrict__ gm, int B,
                                                          const float *__restrict__ F, int ldf,
                                                          const float *__restrict__ pv_all,
                                                          const float *__restrict__ pl_all, float *__restrict__ mu,
                                                          const int *__restrict__ status) {
    const DevModel &m = *gm;
    const int P = m.P, n_data = m.n_data, n_ds = m.n_ds;
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
        const ParVecs q{pv_all + (int64_t)b * P, nullptr, pl_all + (int64_t)b * P};
        const bool bad = status[b] != 0;
        for (int d = 0; d < n_ds; ++d) {
            const DevDataset &ds = m.ds[d];
            const PP eff = ppair(q, ds.eff_idx, 1.f);
            for (int j = threadIdx.x; j < ds.n_reco; j += blockDim.x) {
                float v = pmul(eff, F[((int64_t)d * B + b) * ldf + j]);
                for (int k = ds.bkg_begin; k < ds.bkg_end; ++k) {
                    const DevBkg &bk = m.bkg[k];
                    const float tm = bk.tmpl[j];
                    const float shaped = bk.shape_idx[j] >= 0 ? fmaf(tm, q.pv[bk.shape_idx[j]], tm) : tm;
                    v += pmul(ppair(q, bk.rate_idx, 1.f), shaped);
                }
                mu[(int64_t)b * n_data + ds.data_off + j] = bad ? NAN : v;
            }
        }
    }
}

}  // namespace

// theta, mu, status: device buffers. precision 0 = TF32 fold, 1 = split 3xTF32 fold.
int expected_tc(const DevModel &h, const DevModel *dev, int B, const double *theta, float *mu, int *status,
                int precision, cudaStream_t s) {
    const int nds = h.n_ds, ldt = h.ldt;
    int ldf = 0;
    for (int d = 0; d < nds; ++d) ldf = std::max(ldf, h.ds[d].n_reco);
    ldf = (ldf + 3) / 4 * 4;
    float *vhi = nullptr, *vlo = nullptr, *F = nullptr, *pv = nullptr, *pl = nullptr;
    auto cleanup = [&]() {
        for (float *p : {vhi, vlo, F, pv, pl})
            if (p) cudaFreeAsync(p, s);
    };
    if (fitcore::pool_alloc(&vhi, sizeof(float) * (size_t)nds * B * ldt, s) ||
        fitcore::pool_alloc(&vlo, sizeof(float) * (size_t)nds * B * ldt, s) ||
        fitcore::pool_alloc(&F, sizeof(float) * (size_t)nds * B * ldf, s) ||
        fitcore::pool_alloc(&pv, sizeof(float) * (size_t)B * h.P, s) ||
        fitcore::pool_alloc(&pl, sizeof(float) * (size_t)B * h.P, s)) {
        cudaGetLastError();
        cleanup();
        return fitcore_fail(FIT_ERR_OOM, "fit_model_expected_tc: workspace");
    }
    cudaMemsetAsync(status, 0, sizeof(int) * B, s);
    const size_t smem = signal_smem_bytes(h);
    const void *fn = h.osc_mode == FIT_OSC_EQ1       ? (const void *)signal_v_kernel<4, FIT_OSC_EQ1>
                     : h.osc_mode == FIT_OSC_VACUUM3 ? (const void *)signal_v_kernel<4, FIT_OSC_VACUUM3>
                                                     : (const void *)signal_v_kernel<6, FIT_OSC_STERILE4>;
    const int threads = signal_threads(h.N_t);
    int dev_id = 0, sms = 0, per_sm = 0;
    // (raised only: the attribute is shared with other threads' calls for larger models)
    if (fitcore_raise_eval_smem(fn, smem) != FIT_OK) {
        cudaGetLastError();
        cleanup();
        return FIT_ERR_CUDA;
    }
    if (cudaGetDevice(&dev_id) || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev_id) ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem) || per_sm < 1) {
        cudaGetLastError();
        cleanup();
        return fitcore_fail(FIT_ERR_CUDA, "fit_model_expected_tc: launch shape");
    }
    // one wave of resident blocks over (instance, dataset)
    const int gx = std::max(1, std::min(B, (per_sm * sms + nds - 1) / nds));
    void *args[] = {(void *)&dev, &B, &theta, &vhi, &vlo, &pv, &pl, &status};
    cudaLaunchKernel(fn, dim3(gx, nds), dim3(threads), args, smem, s);
    fitcore_count_launch();
    int rc = FIT_OK;
    for (int d = 0; d < nds && rc == FIT_OK; ++d) {
        const DevDetector &dt = h.det[h.ds[d].det];
        GemmOut o;
        o.epi = EPI_F32;
        o.C = F + (size_t)d * B * ldf;
        o.ldc = ldf;
        const float *Vh = vhi + (size_t)d * B * ldt, *Vl = vlo + (size_t)d * B * ldt;
        rc = precision == 1 ? tc_gemm_split(B, dt.n_reco, h.N_t, Vh, Vl, ldt, dt.rdense_hi, dt.rdense_lo, ldt, o, s)
                            : tc_gemm(true, B, dt.n_reco, h.N_t, Vh, ldt, dt.rdense_hi, ldt, o, s, nullptr);
    }
    if (rc == FIT_OK) {
        mu_epilogue_kernel<<<std::min(B, 152 * 16), 128, 0, s>>>(dev, B, F, ldf, pv, pl, mu, status);
        fitcore_count_launch();
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = fitcore_fail(FIT_ERR_CUDA, std::string("fit_model_expected_tc: ") + cudaGetErrorString(e));
    }
    cleanup();
    return rc;
}

}  // namespace fitcore

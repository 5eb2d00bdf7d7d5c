// molt_line.cu -- launch of the single-line time loops (molt_line.cuh).
#include <algorithm>
#include <cmath>
#include "molt_internal.h"
#include "molt_line.cuh"

namespace molt {

namespace {

struct F64LinePlan {
    int R, K, threads, nw;     // points per thread, CTAs (one cluster), threads per CTA, warps on the line
};

int f64_line_window(double nu, int R, int n, int nw)
{
    return f64_window(nu, 32 * R, nw) + (n % (32 * R) ? 1 : 0);
}

// The split with the shortest sweep, in cycles: 7 operations a point and about
// 24 of carries per thread, each 64 cycles on the quarter of the SM that the
// warp sits on (76 when all four work); two barriers (about 30 cycles in a
// CTA, 370 in a cluster, and the reads of other CTAs' slots, about 600).
// 256 points: 2 per thread, one CTA of 4 warps; 3000 points, P = 2: 4 per
// thread on 8 CTAs.
F64LinePlan f64_line_plan(int n, double nu)
{
    F64LinePlan best{0, 0, 0, 0};
    double cost = 0.0;
    for (int R = 2; R <= 8; R *= 2) {
        const int nw = (n + 32 * R - 1) / (32 * R);
        for (int K = 1; K <= 8; K *= 2) {
            const int wc = (nw + K - 1) / K;
            if (wc > 8 || (K > 1 && nw < K)) continue;
            const double ops = 7.0 * R + 24.0 + 4.0 * std::min(f64_line_window(nu, R, n, nw), nw);
            const double c = ops * ((wc + 3) / 4) * (wc >= 4 ? 76.0 : 64.0) + (K > 1 ? 1340.0 : 60.0);
            if (best.R == 0 || c < cost) {
                cost = c;
                best = F64LinePlan{R, K, 32 * wc, nw};
            }
        }
    }
    return best;
}

template <int R, int BC>
cudaError_t run_line_f64(const F64LinePlan &pl, const F64LineAxis &A, const F64LineRun &p, cudaStream_t s)
{
    if (pl.K == 1) {
        k_line_f64<R, BC, false><<<1, pl.threads, 0, s>>>(A, p);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)pl.K);
    cfg.blockDim = dim3((unsigned)pl.threads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)pl.K;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_line_f64<R, BC, true>, A, p);
}

template <int BC>
cudaError_t run_line_f64_r(const F64LinePlan &pl, const F64LineAxis &A, const F64LineRun &p, cudaStream_t s)
{
    return pl.R == 2 ? run_line_f64<2, BC>(pl, A, p, s) : pl.R == 4 ? run_line_f64<4, BC>(pl, A, p, s)
                                                                    : run_line_f64<8, BC>(pl, A, p, s);
}

template <int BC, int RPT>
cudaError_t run_line_f32(const AxisDev &A, const F32LineRun &p, cudaStream_t s)
{
    const size_t smem = sizeof(float) * 4 * 32 * (RPT + 1);
    k_line_f32<BC, RPT><<<1, 32, smem, s>>>(A, p);
    return cudaGetLastError();
}

template <int BC>
cudaError_t run_line_f32_r(int rpt, const AxisDev &A, const F32LineRun &p, cudaStream_t s)
{
    switch (rpt) {
    case 8: return run_line_f32<BC, 8>(A, p, s);
    case 16: return run_line_f32<BC, 16>(A, p, s);
    case 32: return run_line_f32<BC, 32>(A, p, s);
    case 64: return run_line_f32<BC, 64>(A, p, s);
    default: return cudaErrorInvalidValue;
    }
}

template <int BC, bool CTA>
cudaError_t run_line_smem(const AxisDev &A, const F32LineRun &p, size_t smem_max, cudaStream_t s)
{
    const bool dps = line_smem_bytes(CTA, A.ls, A.n, true) <= smem_max;
    const size_t smem = line_smem_bytes(CTA, A.ls, A.n, dps);
    k_line_f32_smem<BC, CTA><<<1, CTA ? kCtaLineThreads : 32, smem, s>>>(A, dps ? 1 : 0, p);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_line_f64(int bc, double nu, int quad, const AxisDev &ax, const F64LineRun &p, cudaStream_t s)
{
    const F64LinePlan pl = f64_line_plan(ax.n, nu);
    if (pl.R == 0) return cudaErrorInvalidValue;
    const int n = ax.n, R = pl.R;
    F64LineAxis A{};
    A.n = n;
    A.gl = (n - 1) / R;
    A.len_last = n - A.gl * R;
    A.nw = pl.nw;
    A.jw = f64_line_window(nu, R, n, pl.nw);
    A.d = ax.d;
    const double om2 = -std::expm1(-2.0 * nu), kap = f64_kappa(nu, quad);
    A.rho = quad >= 2 ? -0.5 * quad_R(nu) / kap : 0.0;
    auto pw = [&](double k) { return std::exp(-nu * k); };
    A.dR = pw(R);
    A.dRl = pw(A.len_last);
    f64_inverse_decay(A.d, om2, A.e1, A.id);
    for (int k = 0; k < 5; ++k) A.dRk[k] = pw((double)R * (1 << k));
    A.dW = pw(32.0 * R);
    A.dWl = pw(n - 32.0 * R * (A.nw - 1));
    A.mu = ax.mu;
    A.inv = ax.inv;
    for (int k = 0; k <= R; ++k) A.pw[k] = pw(k);
    f64_inflow_weights(nu, R, A.w);
    f64_inflow_weights(nu, A.len_last, A.wl);
    A.dpow = ax.dpow64;
    return bc == BC_PERIODIC ? run_line_f64_r<BC_PERIODIC>(pl, A, p, s) : run_line_f64_r<BC_DIRICHLET>(pl, A, p, s);
}

cudaError_t launch_line_f32(int bc, int rpt, const AxisDev &A, const F32LineRun &p, cudaStream_t s)
{
    return bc == BC_PERIODIC ? run_line_f32_r<BC_PERIODIC>(rpt, A, p, s) : run_line_f32_r<BC_DIRICHLET>(rpt, A, p, s);
}

cudaError_t configure_line_kernels(size_t smem_max)
{
    const void *kernels[] = {(const void *)k_line_f32_smem<BC_PERIODIC, false>, (const void *)k_line_f32_smem<BC_PERIODIC, true>,
                             (const void *)k_line_f32_smem<BC_DIRICHLET, false>,
                             (const void *)k_line_f32_smem<BC_DIRICHLET, true>};
    for (const void *k : kernels) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

bool line_smem_ok(bool cta, const AxisDev &A, size_t smem_max)
{
    return A.m <= (cta ? kLineSeg : 32) && line_smem_bytes(cta, A.ls, A.n, false) <= smem_max;
}

cudaError_t launch_line_f32_smem(int bc, bool cta, const AxisDev &A, const F32LineRun &p, size_t smem_max, cudaStream_t s)
{
    if (bc == BC_PERIODIC)
        return cta ? run_line_smem<BC_PERIODIC, true>(A, p, smem_max, s) : run_line_smem<BC_PERIODIC, false>(A, p, smem_max, s);
    return cta ? run_line_smem<BC_DIRICHLET, true>(A, p, smem_max, s) : run_line_smem<BC_DIRICHLET, false>(A, p, smem_max, s);
}

}  // namespace molt

// molt_f64.cu -- instantiation, launch shapes and constants of the float64
// line passes (molt_f64.cuh).
#include <algorithm>
#include <cmath>
#include "molt_internal.h"
#include "molt_f64.cuh"

namespace molt {

namespace {

// segments whose inflow matters: d^(R win) <= 2^-60
int f64_window(double nu, int R) { return std::max(1, (int)std::ceil(60.0 * std::log(2.0) / (nu * (double)R))); }

// The window's sums over win of G segments: steps one by one cost an operation
// each (64 cycles with few warps about), doubling one operation, a barrier and
// a trip through shared memory; blocks = steps left after dbl doublings.
void f64_window_sums(int win, int G, int *dbl, int *blocks)
{
    const int J = std::min(win, std::max(G - 1, 1));
    double best = 0.0;
    for (int k = 0; k <= 7; ++k) {
        const int b = (J + (1 << k) - 1) >> k;
        const double cost = b + 1.75 * k;
        if (k == 0 || cost < best) {
            best = cost;
            *dbl = k;
            *blocks = b;
        }
    }
}

double half_K(double nu) { return -std::expm1(-2.0 * nu) / (2.0 * nu); }

F64Axis f64_axis(double nu, int quad, int bc, int R, const AxisDev &A)
{
    F64Axis c{};
    c.n = A.n;
    c.G = (A.n + R - 1) / R;
    c.len_last = A.n - (c.G - 1) * R;
    c.win = f64_window(nu, R) + (c.len_last < R ? 1 : 0);    // a short last segment spans less than d^R
    c.R = R;
    f64_window_sums(c.win, c.G, &c.dbl, &c.blocks);
    for (int k = 0; k < 8; ++k) c.pd[k] = std::exp(-nu * (double)R * (double)(1 << k));
    c.pB = c.pd[c.dbl];
    c.d = A.d;
    const double om2 = -std::expm1(-2.0 * nu);             // 1 - d^2
    c.kappa = f64_kappa(nu, quad);
    c.rho = quad >= 2 ? -0.5 * quad_R(nu) / c.kappa : 0.0;
    c.dR = std::exp(-nu * (double)R);
    c.dRl = std::exp(-nu * (double)c.len_last);
    f64_inverse_decay(c.d, om2, c.e1, c.id);
    c.mu = A.mu;
    c.inv = A.inv;
    for (int k = 0; k <= R; ++k) c.pw[k] = std::exp(-nu * (double)k);
    f64_inflow_weights(nu, R, c.w);
    f64_inflow_weights(nu, c.len_last, c.wl);
    c.dpow = A.dpow64;
    (void)bc;
    return c;
}

template <int R, int BC, int KM>
cudaError_t run_f64(bool contig, const F64Plan &pl, const F64Axis &A, const F64Lines &L, const F64Prog &p, cudaStream_t s)
{
    const unsigned grid = (unsigned)((L.nlines + pl.C - 1) / pl.C);
    if (contig) k_f64<R, BC, KM, true><<<grid, pl.threads, pl.smem, s>>>(A, L, p);
    else k_f64<R, BC, KM, false><<<grid, pl.threads, pl.smem, s>>>(A, L, p);
    return cudaGetLastError();
}

template <int BC, int KM>
cudaError_t run_f64_r(bool contig, const F64Plan &pl, const F64Axis &A, const F64Lines &L, const F64Prog &p, cudaStream_t s)
{
    switch (pl.R) {
    case 4: return run_f64<4, BC, KM>(contig, pl, A, L, p, s);
    case 8: return run_f64<8, BC, KM>(contig, pl, A, L, p, s);
    case 16: return run_f64<16, BC, KM>(contig, pl, A, L, p, s);
    case 32: return run_f64<32, BC, KM>(contig, pl, A, L, p, s);
    default: return cudaErrorInvalidValue;
    }
}

template <int R, int BC, int KM>
cudaError_t attr_f64()
{
    cudaError_t e = cudaFuncSetAttribute(k_f64<R, BC, KM, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_f64<R, BC, KM, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

template <int BC, int KM>
cudaError_t attr_f64_r()
{
    cudaError_t e = attr_f64<4, BC, KM>();
    if (e == cudaSuccess) e = attr_f64<8, BC, KM>();
    if (e == cudaSuccess) e = attr_f64<16, BC, KM>();
    return e == cudaSuccess ? attr_f64<32, BC, KM>() : e;
}

}  // namespace

double f64_kappa(double nu, int quad)
{
    const double R2 = quad >= 2 ? quad_R(nu) : 0.0;
    return -half_K(nu) - 0.5 * R2 * -std::expm1(-2.0 * nu);
}

// (1 - d^2) / d and 1 / d carry the boundary terms past a segment's first and
// last point; where d is so small that the next point sees nothing of them,
// they drop out (the end points themselves are set)
void f64_inverse_decay(double d, double om2, double &e1, double &id)
{
    id = d > 1e-140 ? 1.0 / d : 0.0;
    e1 = om2 * id;
}

void f64_inflow_weights(double nu, int len, double *w)
{
    const double om2 = -std::expm1(-2.0 * nu);
    for (int k = 0; k < len; ++k) w[k] = std::exp(-nu * (double)(k + 1)) * (-std::expm1(-2.0 * nu * (double)(len - k)) / om2);
}

bool f64_axis_ok(int n, bool contig) { return n <= kF64MaxR * kF64Threads / (contig ? 1 : 2); }

// Segment length R and lines per CTA C: the pair whose busiest quarter of an
// SM (each issues its own warps) has the least to do.  A segment costs about 8
// operations a point and sweep (12 with a Horner step's fields), 2 per block of
// its inflow window, 3.5 per doubling, and 18 for its ends and barriers; whole
// warps are issued whether their threads are live or not; a quarter with one
// warp also waits about 0.4 of its time for the recurrences, with k warps 0.4 / k;
// runs of two columns cost 1.15 (half a sector each).  Equal choices take the
// longer runs (larger C).  Measured against other weights: 1000 x 777, P = 3: y 58
// us at R = 32, C = 8 (68 at R = 8, C = 2); 288 x 2016, P = 1: y 19 us at R = 16, C =
// 2 (27 at R = 32, C = 4); 70 x 300, P = 2: y 15 us at R = 4, C = 2 (21 at R = 16, C =
// 4); 512^2, P = 3: x 38 us at R = 8 (42 at R = 16).
bool f64_plan(int n, int64_t nlines, bool contig, bool horner, double nu, int sms, F64Plan *out)
{
    if (!f64_axis_ok(n, contig)) return false;
    double best = 0.0;
    F64Plan pl{};
    for (int R = 4; R <= kF64MaxR; R *= 2) {
        const int G = (n + R - 1) / R;
        int dbl = 0, blocks = 0;
        f64_window_sums(f64_window(nu, R), G, &dbl, &blocks);
        const double ops = (horner ? 12.0 : 8.0) * R + 2.0 * blocks + 3.5 * dbl + 18.0;
        // strided accesses in runs of 4 columns or more, except where a column fills the CTA
        const int c_min = contig ? 1 : (4 * G <= kF64Threads ? 4 : 2);
        for (int C = c_min; C <= 32 && C * G <= kF64Threads; C *= 2) {
            const int threads = (C * G + 31) / 32 * 32, warps = threads / 32;
            const size_t smem = f64_smem(threads, C, R, horner);
            const int64_t ctas = (nlines + C - 1) / C, per_sm = (ctas + sms - 1) / sms;
            const int occ = (int)std::max<size_t>(1, std::min<size_t>(512 / threads, (size_t)(227 * 1024) / (smem + 1024)));
            // warps a quarter works through; beyond one round of resident CTAs the SMs even out
            const double load = per_sm <= occ ? std::ceil(per_sm * warps / 4.0) : (double)ctas / sms * warps / 4.0 + 0.5;
            const double resident = std::min(load, std::max(1.0, occ * warps / 4.0));
            const double cost = load * ops * (1.0 + 0.4 / resident) * (!contig && C == 2 ? 1.15 : 1.0);
            if (pl.R == 0 || cost < best || (cost == best && C > pl.C)) {
                best = cost;
                pl = F64Plan{R, G, C, threads, smem};
            }
        }
    }
    if (pl.R == 0) return false;
    *out = pl;
    return true;
}

cudaError_t launch_f64(int bc, bool contig, const F64Plan &pl, double nu, int quad, const AxisDev &ax, int64_t stride,
                       int64_t inner, int64_t nlines, bool horner, F64Prog p, cudaStream_t s)
{
    if (contig && ax.n % 4 == 0) {
        uintptr_t bits = (uintptr_t)p.u | (uintptr_t)p.up | (uintptr_t)p.un;
        for (int k = 0; k < MAXG; ++k) bits |= (uintptr_t)p.g[k] | (uintptr_t)p.out[k];
        p.vec = (bits & 31) == 0;
    }
    const F64Axis A = f64_axis(nu, quad, bc, pl.R, ax);
    F64Lines L{stride, inner, nlines, pl.C, 0};
    while ((1 << L.cshift) < pl.C) ++L.cshift;
    if (bc == BC_PERIODIC)
        return horner ? run_f64_r<BC_PERIODIC, 1>(contig, pl, A, L, p, s) : run_f64_r<BC_PERIODIC, 0>(contig, pl, A, L, p, s);
    return horner ? run_f64_r<BC_DIRICHLET, 1>(contig, pl, A, L, p, s) : run_f64_r<BC_DIRICHLET, 0>(contig, pl, A, L, p, s);
}

cudaError_t configure_f64_kernels()
{
    cudaError_t e = attr_f64_r<BC_PERIODIC, 0>();
    if (e == cudaSuccess) e = attr_f64_r<BC_PERIODIC, 1>();
    if (e == cudaSuccess) e = attr_f64_r<BC_DIRICHLET, 0>();
    return e == cudaSuccess ? attr_f64_r<BC_DIRICHLET, 1>() : e;
}

}  // namespace molt

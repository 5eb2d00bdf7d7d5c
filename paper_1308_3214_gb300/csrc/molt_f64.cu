// molt_f64.cu -- instantiation, launch shapes and constants of the float64
// line passes (molt_f64.cuh).
#include <algorithm>
#include <map>
#include <cmath>
#include "molt_internal.h"
#include "molt_f64.cuh"

namespace molt {

namespace {

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

F64Axis f64_axis(double nu, int quad, int R, const AxisDev &A)
{
    F64Axis c{};
    c.n = A.n;
    c.G = (A.n + R - 1) / R;
    c.len_last = A.n - (c.G - 1) * R;
    c.win = f64_window(nu, R, c.G) + (c.len_last < R ? 1 : 0);    // a short last segment spans less than d^R
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

template <int KM, bool CONTIG, bool ADJ>
const void *batch_kernel(int R)
{
    switch (R) {
    case 4: return (const void *)k_f64_batch<4, KM, CONTIG, ADJ>;
    case 8: return (const void *)k_f64_batch<8, KM, CONTIG, ADJ>;
    case 16: return (const void *)k_f64_batch<16, KM, CONTIG, ADJ>;
    default: return (const void *)k_f64_batch<32, KM, CONTIG, ADJ>;
    }
}

const void *batch_kernel(int axis, bool adj, int R)
{
    if (axis == 0) return adj ? batch_kernel<1, true, true>(R) : batch_kernel<1, true, false>(R);
    return adj ? batch_kernel<0, false, true>(R) : batch_kernel<0, false, false>(R);
}

}  // namespace

double f64_kappa(double nu, int quad)
{
    const double R2 = quad >= 2 ? quad_R(nu) : 0.0;
    return -half_K(nu) - 0.5 * R2 * -std::expm1(-2.0 * nu);
}

int f64_window(double nu, int points, int count)
{
    const double w = std::ceil(60.0 * std::log(2.0) / (nu * (double)points));
    return (int)std::max(1.0, std::min(w, (double)count));     // (w itself may exceed an int)
}

// (1 - d^2) / d and 1 / d carry the boundary terms past a segment's first and
// last point; where d is so small that the next point sees nothing of them,
// they drop out (the end points themselves are set; the end nodes of a line
// object, which are interior, take theirs one by one, k_obj_sweep)
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
bool f64_plan(int n, int64_t nlines, bool contig, bool horner, double nu, int sms, F64Plan *out, int rmax, int tmax)
{
    if (!f64_axis_ok(n, contig)) return false;
    double best = 0.0;
    F64Plan pl{};
    for (int R = 4; R <= rmax; R *= 2) {
        const int G = (n + R - 1) / R;
        int dbl = 0, blocks = 0;
        f64_window_sums(f64_window(nu, R, G), G, &dbl, &blocks);
        const double ops = (horner ? 12.0 : 8.0) * R + 2.0 * blocks + 3.5 * dbl + 18.0;
        // strided accesses in runs of 4 columns or more, except where a column fills the CTA
        const int c_min = contig ? 1 : (4 * G <= kF64Threads ? 4 : 2);
        for (int C = c_min; C <= 32 && (C * G <= tmax || (C == c_min && C * G <= kF64Threads)); C *= 2) {
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
    const F64Axis A = f64_axis(nu, quad, pl.R, ax);
    F64Lines L{stride, inner, nlines, ax.n, pl.C, 0};
    while ((1 << L.cshift) < pl.C) ++L.cshift;
    if (bc == BC_PERIODIC)
        return horner ? run_f64_r<BC_PERIODIC, 1>(contig, pl, A, L, p, s) : run_f64_r<BC_PERIODIC, 0>(contig, pl, A, L, p, s);
    return horner ? run_f64_r<BC_DIRICHLET, 1>(contig, pl, A, L, p, s) : run_f64_r<BC_DIRICHLET, 0>(contig, pl, A, L, p, s);
}

// Tasks and work lists of a batch's passes: the shape of each problem's lines
// as f64_plan picks it with the batch's points behind it, grouped by segment
// length and CTA size (rounded up to 64 threads), the longest programs first.
// Several problems: segments of at most 16 points and CTAs of at most 128
// threads where the line allows (fewer dead lanes past the lines' ends, a
// shorter tail to every launch).  Measured, us: 100 problems of 64..256 points
// 4200 -> 2958 (R <= 16 alone 2980, T <= 128 alone 3608), 15 of 64..1024 3900 -> 2880,
// 4 of 128..512 886 -> 796; a single problem is planned as in a handle of its own
// (1024 x 1000 gradient 1504 against 1538).
void f64_batch_plan(const F64BatchGrid *probs, int nprob, int quad, int sms, F64BatchLists &out)
{
    int64_t points = 0;
    for (int i = 0; i < nprob; ++i) points += (int64_t)probs[i].ax->n * probs[i].ay->n;
    out.tasks.assign(2 * (size_t)nprob, F64Task{});
    out.items.clear();
    for (int axis = 0; axis < 2; ++axis) {
        const bool contig = axis == 0;
        std::map<std::pair<int, int>, std::vector<int>> groups;
        for (int i = 0; i < nprob; ++i) {
            const F64BatchGrid &g = probs[i];
            const AxisDev &A = contig ? *g.ax : *g.ay;
            const int64_t lines = contig ? g.ay->n : g.ax->n;
            const double nu = contig ? g.nux : g.nuy;
            F64Plan pl{};
            f64_plan(A.n, std::max(lines, points / A.n), contig, contig, nu, sms, &pl, nprob > 1 ? 16 : kF64MaxR,
                     nprob > 1 ? 128 : kF64Threads);
            F64Task &t = out.tasks[(size_t)axis * nprob + i];
            t.A = f64_axis(nu, quad, pl.R, A);
            t.L = F64Lines{contig ? 1 : (int64_t)g.pitch, lines, lines, g.pitch, pl.C, 0};
            while ((1 << t.L.cshift) < pl.C) ++t.L.cshift;
            t.off = g.off;
            t.p.P = g.P;
            t.p.vec = contig;                          // rows start on 32 bytes and are padded to 4 points
            if (contig) {
                t.p.ng = g.P;
                t.p.nout = 1;
                t.p.epi = 1;
                // in the units of the powers: kappa per application of either axis' D
                const double kx = f64_kappa(g.nux, quad), ky = f64_kappa(g.nuy, quad);
                double ux = 1.0;
                for (int q = 0; q <= g.P; ++q, ux *= kx) {
                    double ug = ky;
                    for (int k = 0; k < g.P; ++k, ug *= ky) {
                        t.p.coef[0][q][k] = g.coef[q * g.ldc + k] * ux * ug;
                        if (t.p.coef[0][q][k] != 0.0) t.p.add[0][q] |= 1u << k;
                    }
                    t.p.cu[0][q] = g.cu[q] * ux;
                    if (t.p.cu[0][q] != 0.0) t.p.ucu[0] |= 1u << q;
                }
            }
            groups[{pl.R, (pl.threads + 63) / 64 * 64}].push_back(i);
        }
        out.classes[axis].clear();
        for (auto &g : groups) {
            F64BatchClass c{g.first.first, g.first.second, 0, (int)out.items.size(), 0};
            std::stable_sort(g.second.begin(), g.second.end(), [&](int a, int b) { return probs[a].P > probs[b].P; });
            for (int i : g.second) {
                const F64Task &t = out.tasks[(size_t)axis * nprob + i];
                c.smem = std::max(c.smem, sizeof(double) * f64_task_words() + f64_smem(c.threads, t.L.C, c.R, contig));
                for (int64_t l = 0; l < t.L.nlines; l += t.L.C)
                    out.items.push_back(make_int2(axis * nprob + i, (int)(l / t.L.C)));
            }
            c.count = (int)out.items.size() - c.begin;
            out.classes[axis].push_back(c);
        }
        // the class with the most threads first (it runs on the caller's stream)
        std::sort(out.classes[axis].begin(), out.classes[axis].end(), [](const F64BatchClass &a, const F64BatchClass &b) {
            return (int64_t)a.count * a.threads > (int64_t)b.count * b.threads;
        });
    }
}

cudaError_t launch_f64_batch(int axis, bool adj, const F64BatchClass &c, F64BatchPass bp, cudaStream_t s)
{
    bp.items += c.begin;
    void *args[] = {&bp};
    return cudaLaunchKernel(batch_kernel(axis, adj, c.R), dim3((unsigned)c.count), dim3((unsigned)c.threads), args, c.smem, s);
}

cudaError_t configure_f64_batch_kernels()
{
    for (int axis = 0; axis < 2; ++axis)
        for (int adj = 0; adj < 2; ++adj)
            for (int R = 4; R <= kF64MaxR; R *= 2) {
                const cudaError_t e = cudaFuncSetAttribute(batch_kernel(axis, adj != 0, R),
                                                           cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
                if (e != cudaSuccess) return e;
            }
    return cudaSuccess;
}

cudaError_t configure_f64_kernels()
{
    cudaError_t e = attr_f64_r<BC_PERIODIC, 0>();
    if (e == cudaSuccess) e = attr_f64_r<BC_PERIODIC, 1>();
    if (e == cudaSuccess) e = attr_f64_r<BC_DIRICHLET, 0>();
    return e == cudaSuccess ? attr_f64_r<BC_DIRICHLET, 1>() : e;
}

}  // namespace molt

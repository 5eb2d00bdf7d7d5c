// molt_line.cuh -- the time loop of a single line (1D grids) as one kernel
// (sm_103a): many steps per launch, the levels on chip between them.
//
// A 1D step is a few thousand operations; launched one by one (also from a
// graph) each step pays the launch, its first loads and the way back through
// L2.  Here the line stays with its threads for the whole run:
//
//   * k_line_f64 (MOL_FP64): the sweeps of molt_f64.cuh with the line spread
//     over the threads of one CTA or of a cluster, R points per thread, both
//     levels in registers.  A float64 operation occupies a quarter of an SM
//     for 64 cycles per warp (measured; the latency is the same 64), so short
//     segments on many warps win until the carry scan (about 24 operations a
//     thread and sweep) outweighs them, and long lines take up to 8 SMs: a
//     cluster barrier costs 0.2 us.
//   * k_line_f32 (MOL_MIXED): the arithmetic of the one-step kernels, so that a
//     run gives the same bits launched either way: the warp-per-line register
//     sweep (k_contig_res) where the line splits into whole segments, else
//     the shared-memory sweeps (k_horner), by a warp or by the whole CTA.
//
// Measured, us per step, one launch per step (graph) -> here.  MOL_FP64: 256 points
// periodic, P = 1, 7.4 -> 2.7; 352 points periodic, P = 3, 25 -> 11; 3000 points, P = 2,
// 47 -> 9.6 (8 CTAs).  MOL_MIXED, P = 3: 768 points 6.0 -> 3.1 (whole segments on one
// warp); 1000 points 19 -> 15 (one warp, shared memory); 10001 points, with boundary
// data or without, 34 -> 17.4 (three sweeps by 16 warps; bound by their instructions).
//
// Boundary data (mol_solve_dirichlet) travel in the launch's parameters, up to
// kLineDataSteps steps per launch.
#pragma once
#include <cooperative_groups.h>
#include "molt_kernels.cuh"
#include "molt_regs.cuh"
#include "molt_f64.cuh"

namespace molt {

constexpr int kLineDataSteps = 24;       // steps per launch with boundary data
constexpr int kLineDataStepsF32 = 48;

// Constants of a float64 line split into segments of R points, 32 per warp.
struct F64LineAxis {
    int n, gl, len_last;       // points, last segment, its points
    int nw;                    // warps on the line
    int jw;                    // warps whose inflow matters on each side
    double d, rho;
    double dR, dRl, e1, id;    // as F64Axis
    double dRk[5];             // d^(R 2^k)
    double dW, dWl;            // d^points of a full warp and of the last one
    double mu, inv;
    double pw[9], w[8], wl[8]; // d^k and the inflow weights, as F64Axis
    const double *dpow;
};

struct F64LineRun {
    int P, steps;
    bool first;                // the first step is the start: u + F/2
    bool data;                 // end[][] holds each step's end values
    double cu[MAXP];           // kappa^t f_t
    const double *u0, *u1;     // u^{n-1}, u^n (u0 unused when first)
    double *v0, *v1;           // the last two levels
    // step k: values of the Horner step t's D at both ends (times kappa^(t-1)), then the new level's
    double end[kLineDataSteps][MAXP][2];
    double bnew[kLineDataSteps][2];
};

// shared memory of one CTA: per warp E, H, kw, first, last; then s_1, s_{n-2},
// the line's last zero-inflow y
struct F64LineSlots {
    double E[8], H[8], kw[8], first[8], last[8], s1, sn2, yl;
};

template <int R, int BC, bool CLUSTER>
__global__ void __launch_bounds__(256) k_line_f64(const __grid_constant__ F64LineAxis A,
                                                  const __grid_constant__ F64LineRun p)
{
    namespace cg = cooperative_groups;
    __shared__ F64LineSlots sl;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = CLUSTER ? (int)cl.block_rank() : 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwc = blockDim.x >> 5;
    const int gw = rank * nwc + warp, g = gw * 32 + lane;          // warp and segment on the line
    const int n = A.n, a0 = g * R;
    const bool live = g <= A.gl, lastseg = g == A.gl, wlive = gw < A.nw, lastwarp = gw == A.nw - 1;
    const int len = !live ? 0 : lastseg ? A.len_last : R;
    auto sync = [&]() {
        if (CLUSTER) cl.sync();
        else __syncthreads();
    };
    auto at = [&](int q) -> F64LineSlots * {                       // slots of the CTA of warp q
        return CLUSTER ? cl.map_shared_rank(&sl, q / nwc) : &sl;
    };
    auto multw = [&](int q) -> double { return q == A.nw - 1 ? A.dWl : A.dW; };

    // per-thread constants: d^(R lane); the response of this segment's right
    // inflow to an inflow of its warp; the way of the warp's right inflow here
    double dl = 1.0, cL = 0.0, fG = 1.0;
    for (int k = 0; k < lane; ++k) dl *= A.dR;
    if (live && !lastseg) {
        const int ll = lastwarp ? A.gl & 31 : 31;
        double pr = 1.0, dq = dl * A.dR;
        for (int q = lane + 1; q <= ll; ++q) {
            const bool tail = lastwarp && q == ll;
            cL = fma(pr * (tail ? A.wl[0] : A.w[0]), dq, cL);
            pr *= tail ? A.dRl : A.dR;
            dq *= A.dR;
        }
        fG = pr;
    }
    if (lane == 0) sl.kw[warp] = !live ? 0.0 : lastseg ? A.wl[0] : fma(A.dR, cL, A.w[0]);

    double uc[R], up[R], r[R], z[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        uc[k] = k < len ? p.u1[a0 + k] : 0.0;
        up[k] = k < len && !p.first ? p.u0[a0 + k] : 0.0;
    }

    // z <- second difference of z, the neighbours' values by shuffles and
    // through the warps' slots (one barrier)
    auto sdiff = [&](double (&v)[R]) {
        double lastv = v[R - 1];
        if (lastseg) lastv = f64_pick<R>(v, A.len_last - 1);
        __syncwarp();
        double zl = __shfl_up_sync(0xffffffffu, lastv, 1), zr = __shfl_down_sync(0xffffffffu, v[0], 1);
        if (lane == 0) sl.first[warp] = v[0];
        if ((lane == 31 && live) || lastseg) sl.last[warp] = lastv;   // the warp's last segment on the line
        sync();
        if (lane == 0 && live) zl = gw > 0 ? at(gw - 1)->last[(gw - 1) % nwc]
                                           : (BC == BC_PERIODIC ? at(A.nw - 1)->last[(A.nw - 1) % nwc] : 0.0);
        if (lastseg) zr = BC == BC_PERIODIC ? at(0)->first[0] : 0.0;
        else if (lane == 31 && live) zr = at(gw + 1)->first[(gw + 1) % nwc];
        if (lastseg && len < R) {
#pragma unroll
            for (int k = 1; k < R; ++k) v[k] = k == A.len_last ? zr : v[k];
        }
        double dm = v[0] - zl;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const double dp = (k + 1 < R ? v[k + 1] : zr) - v[k];
            v[k] = dp - dm;
            dm = dp;
        }
    };

    // z: s on entry, rho s + T^{-1} s (with the boundary terms) on exit; eL, eR:
    // the values at Dirichlet ends
    auto solve = [&](double eL, double eR) {
        double s[R];
        if (BC == BC_DIRICHLET) {
            // s_1 and s_{n-2} for the end terms; the end rows drop out
            if (a0 <= 1 && 1 < a0 + len) sl.s1 = f64_pick<R>(z, 1 - a0);
            if (a0 <= n - 2 && n - 2 < a0 + len) sl.sn2 = f64_pick<R>(z, n - 2 - a0);
            if (g == 0) z[0] = 0.0;
        }
        const int keep = BC == BC_DIRICHLET && lastseg ? len - 1 : len;
#pragma unroll
        for (int k = 0; k < R; ++k) s[k] = z[k] = k < keep ? z[k] : 0.0;
#pragma unroll
        for (int k = 1; k < R; ++k) z[k] = fma(A.d, z[k - 1], z[k]);
        double E = z[R - 1];
        if (lastseg) {                                             // y ends with the line
            E = f64_pick<R>(z, A.len_last - 1);
#pragma unroll
            for (int k = 0; k < R; ++k) z[k] = k < len ? z[k] : 0.0;
        }
#pragma unroll
        for (int k = R - 2; k >= 0; --k) z[k] = fma(A.d, z[k + 1], z[k]);
        // warp scans: y at the segment's start and g past its end, both without
        // the inflow of the warp
        __syncwarp();
        double x = E;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const double y = __shfl_up_sync(0xffffffffu, x, 1 << k);
            if (lane >= (1 << k)) x = fma(A.dRk[k], y, x);
        }
        double ex = __shfl_up_sync(0xffffffffu, x, 1);
        ex = lane == 0 ? 0.0 : ex;
        const double yl = fma(A.dRl, ex, E);                       // of the last segment: y_{n-1}
        double v = fma(lastseg ? A.wl[0] : live ? A.w[0] : 0.0, ex, z[0]);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const double y = __shfl_down_sync(0xffffffffu, v, 1 << k);
            if (lane + (1 << k) < 32) v = fma(A.dRk[k], y, v);
        }
        double hx = __shfl_down_sync(0xffffffffu, v, 1);
        hx = lane == 31 || !live || lastseg ? 0.0 : hx;
        if (lane == 0) sl.H[warp] = v;
        if (lastseg) { sl.E[warp] = yl; sl.yl = yl; }
        else if (lane == 31 && live) sl.E[warp] = x;
        sync();
        if (!wlive) return;
        // inflow of the warp from the left (c) and from the right (go)
        const int J = A.jw < A.nw ? A.jw : A.nw;
        double c = 0.0, go = 0.0;
        auto Ew = [&](int q) { return at(q)->E[q % nwc]; };
        auto Hw = [&](int q, double ci) { const F64LineSlots *t = at(q); return fma(t->kw[q % nwc], ci, t->H[q % nwc]); };
        if (BC == BC_PERIODIC) {
            int q = gw - J;
            if (q < 0) q += A.nw;
            for (int j = 0; j < J; ++j) {
                c = fma(multw(q), c, Ew(q));
                q = q + 1 == A.nw ? 0 : q + 1;
            }
            if (J == A.nw) c *= A.inv;
            double ci = fma(multw(gw), c, Ew(gw)), pr = 1.0;
            q = gw + 1 == A.nw ? 0 : gw + 1;
            for (int j = 0; j < J; ++j) {
                go = fma(pr, Hw(q, ci), go);
                ci = fma(multw(q), ci, Ew(q));
                pr *= multw(q);
                q = q + 1 == A.nw ? 0 : q + 1;
            }
            if (J == A.nw) go *= A.inv;
        } else {
            for (int q = max(gw - J, 0); q < gw; ++q) c = fma(A.dW, c, Ew(q));
            double pr = 1.0;
            if (!lastwarp) {
                double ci = fma(A.dW, c, Ew(gw));
                for (int q = gw + 1; q <= min(gw + J, A.nw - 1); ++q) {
                    go = fma(pr, Hw(q, ci), go);
                    if (q < A.nw - 1) ci = fma(A.dW, ci, Ew(q));
                    pr *= A.dW;
                }
            }
        }
        const double yin = fma(dl, c, ex), gin = fma(fG, go, fma(cL, c, hx));
        double a = yin, b = gin;
        if (BC == BC_DIRICHLET) {
            const bool all = A.jw >= A.nw, nl = all || gw < A.jw, nr = all || A.nw - 1 - gw < A.jw;
            double r0 = 0.0, r1 = 0.0;
            if (nl) {
                double ci = 0.0, pr = 1.0, g0 = 0.0;
                for (int q = 0; q <= min(J, A.nw - 1); ++q) {
                    g0 = fma(pr, Hw(q, ci), g0);
                    if (q < A.nw - 1) ci = fma(A.dW, ci, Ew(q));
                    pr *= A.dW;
                }
                r0 = fma(-A.rho, at(0)->s1, eL - g0);
            }
            if (nr) {
                double ci = 0.0;
                for (int q = max(A.nw - 1 - J, 0); q < A.nw - 1; ++q) ci = fma(A.dW, ci, Ew(q));
                // s_{n-2} sits with its owner's CTA
                const int qo = ((n - 2) / R) >> 5;
                r1 = fma(-A.rho, at(qo)->sn2, eR - fma(A.dWl, ci, at(A.nw - 1)->yl));
            }
            if (all) {
                const double t0 = (r0 - A.mu * r1) * A.inv;
                r1 = (r1 - A.mu * r0) * A.inv;
                r0 = t0;
            }
            if (nl && live) {
                const double t0 = r0 * A.dpow[a0];
                a = fma(t0, A.e1, a);
                b = fma(t0, lastseg ? A.dRl : A.dR, b);
            }
            if (nr && live) b = fma(r1 * A.dpow[n - a0 - len], A.id, b);
        }
        if (!live) return;
#pragma unroll
        for (int k = 0; k < R; ++k) z[k] = fma(A.rho, s[k], z[k]);
        if (lastseg) {
#pragma unroll
            for (int k = 0; k < R; ++k) z[k] = k < len ? fma(b, A.pw[k < len ? len - k : 0], fma(a, A.wl[k], z[k])) : 0.0;
        } else {
#pragma unroll
            for (int k = 0; k < R; ++k) z[k] = fma(b, A.pw[R - k], fma(a, A.w[k], z[k]));
        }
        if (BC == BC_DIRICHLET) {
            if (g == 0) z[0] = eL;
            if (lastseg) {
#pragma unroll
                for (int k = 0; k < R; ++k) z[k] = k == len - 1 ? eR : z[k];
            }
        }
    };

    for (int st = 0; st < p.steps; ++st) {
#pragma unroll
        for (int k = 0; k < R; ++k) r[k] = uc[k];
        sdiff(r);
        for (int t = p.P; t >= 1; --t) {
            const double w = p.cu[t];
            if (t == p.P) {
#pragma unroll
                for (int k = 0; k < R; ++k) z[k] = w * r[k];
            } else {
                sdiff(z);
#pragma unroll
                for (int k = 0; k < R; ++k) z[k] = fma(w, r[k], z[k]);
            }
            solve(p.data ? p.end[st][t][0] : 0.0, p.data ? p.end[st][t][1] : 0.0);
        }
        const bool half = p.first && st == 0;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const double nu = half ? fma(0.5, z[k], uc[k]) : fma(2.0, uc[k], z[k] - up[k]);
            up[k] = uc[k];
            uc[k] = nu;
        }
        if (p.data) {
            if (g == 0) uc[0] = p.bnew[st][0];
            if (lastseg) {
#pragma unroll
                for (int k = 0; k < R; ++k) uc[k] = k == len - 1 ? p.bnew[st][1] : uc[k];
            }
        }
    }
#pragma unroll
    for (int k = 0; k < R; ++k)
        if (k < len) {
            p.v0[a0 + k] = up[k];
            p.v1[a0 + k] = uc[k];
        }
    if (CLUSTER) cl.sync();            // no CTA leaves while its slots may be read
}

// ---------------------------------------------------------------------------
// float32 sweeps, float32-pair levels
// ---------------------------------------------------------------------------
struct F32LineRun {
    int P, steps;
    bool first, data;          // as F64LineRun
    float cu[MAXP];
    const float *h0, *l0, *h1, *l1;      // u^{n-1}, u^n
    float *vh0, *vl0, *vh1, *vl1;        // the last two levels
    float end[kLineDataStepsF32][MAXP][2];
    float bh[kLineDataStepsF32][2], bl[kLineDataStepsF32][2];   // the new level's end values as pairs
};

// Lines of whole segments (n a multiple of RPT, at most 32 RPT): one warp, the
// sweeps of k_contig_res; the levels in shared memory, lane = segment.
template <int BC, int RPT>
__global__ void __launch_bounds__(32) k_line_f32(const __grid_constant__ AxisDev A, const __grid_constant__ F32LineRun p)
{
    constexpr int SS = RPT + 1;                // odd: a lane's walk and a row's both conflict-free
    extern __shared__ __align__(16) float sm32[];
    const int lane = threadIdx.x, n = A.n;
    float *uh = sm32, *ul = uh + 32 * SS, *ph = ul + 32 * SS, *pl = ph + 32 * SS;
    auto pos = [&](int j) { return (j / RPT) * SS + j % RPT; };
    for (int j = lane; j < n; j += 32) {
        uh[pos(j)] = p.h1[j];
        ul[pos(j)] = p.l1[j];
        ph[pos(j)] = p.first ? 0.f : p.h0[j];
        pl[pos(j)] = p.first ? 0.f : p.l0[j];
    }
    __syncwarp();
    const int a = lane * RPT, Ld = n / RPT - 1;
    const bool full = lane <= Ld;
    const int jl = a > 0 ? a - 1 : (BC == BC_PERIODIC ? n - 1 : 0);
    const int jr = lane < Ld ? a + RPT : (BC == BC_PERIODIC ? 0 : n - 1);
    for (int st = 0; st < p.steps; ++st) {
        // r = accurate second difference of u (Dirichlet ends take their neighbour's)
        float r[RPT], z[RPT];
#pragma unroll
        for (int k = 0; k < RPT; ++k) r[k] = z[k] = 0.f;
        if (full) {
            const float *H = uh + lane * SS, *L = ul + lane * SS;
            float hm = uh[pos(jl)], lm = ul[pos(jl)], h0 = H[0], l0 = L[0];
            const float hr = uh[pos(jr)], lr = ul[pos(jr)];
#pragma unroll
            for (int k = 0; k < RPT; ++k) {
                const float hp = k + 1 < RPT ? H[k + 1] : hr, lp = k + 1 < RPT ? L[k + 1] : lr;
                r[k] = sdiff_pair(hm, h0, hp, lm, l0, lp);
                hm = h0; h0 = hp;
                lm = l0; l0 = lp;
            }
            if (BC == BC_DIRICHLET) {
                if (lane == 0) r[0] = r[1];
                if (lane == Ld) r[RPT - 1] = r[RPT - 2];
            }
        }
        for (int t = p.P; t >= 1; --t) warp_sweep_rreg<float, BC, RPT>(z, r, p.cu[t], A, lane);
        const bool half = p.first && st == 0;
        const float ea = half ? 1.f : 2.f, eb = half ? 0.f : -1.f, ec = half ? 0.5f : 1.f;
        __syncwarp();                              // the neighbours' reads of this level are done
        if (full) {
            float *H = uh + lane * SS, *L = ul + lane * SS, *PH = ph + lane * SS, *PL = pl + lane * SS;
#pragma unroll
            for (int k = 0; k < RPT; ++k) {
                float nh, nl;
                const float h = H[k], l = L[k];
                level_pair(h, l, PH[k], PL[k], z[k], ea, eb, ec, nh, nl);
                PH[k] = h;
                PL[k] = l;
                H[k] = nh;
                L[k] = nl;
            }
        }
        __syncwarp();
    }
    for (int j = lane; j < n; j += 32) {
        p.vh1[j] = uh[pos(j)];
        p.vl1[j] = ul[pos(j)];
        p.vh0[j] = ph[pos(j)];
        p.vl0[j] = pl[pos(j)];
    }
}

// Any other line, and lines with boundary data: the sweeps of k_horner.  CTA:
// kCtaLineThreads threads, at most kLineSeg points each (their share of
// u^{n-1} in registers); else one warp, every level in shared memory.
// Shared memory: buf, r, uh, ul [ls] (warp: ph, pl too), the table d^j (dps),
// the carry scratch.
constexpr int kLineSeg = 24;

__host__ __device__ inline size_t line_smem_bytes(bool cta, int ls, int n, bool dps)
{
    return sizeof(float) * ((size_t)(cta ? 4 : 6) * ls + (dps ? (size_t)n + 1 : 0) + 2 * (kCtaLineThreads / 32) + 4);
}

template <int BC, bool CTA>
__global__ void __launch_bounds__(CTA ? kCtaLineThreads : 32) k_line_f32_smem(const __grid_constant__ AxisDev A, int dps,
                                                                             const __grid_constant__ F32LineRun p)
{
    extern __shared__ __align__(16) float sm32[];
    const int t = threadIdx.x, T = CTA ? kCtaLineThreads : 32, n = A.n, m = A.m, ls = A.ls;
    float *buf = sm32, *r = buf + ls, *uh = r + ls, *ul = uh + ls;
    float *ph = CTA ? nullptr : ul + ls, *pl = CTA ? nullptr : ph + ls;
    float *dpt = ul + (CTA ? 1 : 3) * ls, *scr = dpt + (dps ? n + 1 : 0);
    const float *dp = dps ? dpt : A.dpow32;
    auto sync = [&]() {
        if (CTA) __syncthreads();
        else __syncwarp();
    };
    if (dps)
        for (int j = t; j <= n; j += T) dpt[j] = A.dpow32[j];
    for (int j = t; j < n; j += T) {
        const int q = spos_raw(j, m, A.ms, A.mmagic);
        uh[q] = p.h1[j];
        ul[q] = p.l1[j];
        if (!CTA) {
            ph[q] = p.first ? 0.f : p.h0[j];
            pl[q] = p.first ? 0.f : p.l0[j];
        }
    }
    const int a = t * m, cnt = a < n ? min(m, n - a) : 0, o = t * A.ms;   // this thread's points and their slots
    float qh[kLineSeg], ql[kLineSeg];
    if (CTA) {
#pragma unroll
        for (int k = 0; k < kLineSeg; ++k) {
            qh[k] = k < cnt && !p.first ? p.h0[a + k] : 0.f;
            ql[k] = k < cnt && !p.first ? p.l0[a + k] : 0.f;
        }
    }
    sync();
    for (int st = 0; st < p.steps; ++st) {
        for (int k = 0; k < cnt; ++k) {
            const int c = BC == BC_DIRICHLET ? sd_centre<BC>(a + k, n) : a + k;
            const int q0 = spos<BC>(c - 1, A), q1 = spos<BC>(c, A), q2 = spos<BC>(c + 1, A);
            r[o + k] = sdiff_pair(uh[q0], uh[q1], uh[q2], ul[q0], ul[q1], ul[q2]);
            buf[o + k] = 0.f;
        }
        sync();
        for (int q = p.P; q >= 1; --q) {
            const float gL = p.data ? p.end[st][q][0] : 0.f, gR = p.data ? p.end[st][q][1] : 0.f;
            if constexpr (CTA) sweep_D_cta<float, 2, BC>(buf, r, p.cu[q], A, dp, scr, gL, gR);
            else sweep_D<float, 2, BC>(buf, r, p.cu[q], A, dp, t, gL, gR);
            sync();
        }
        const bool half = p.first && st == 0;
        const float ea = half ? 1.f : 2.f, eb = half ? 0.f : -1.f, ec = half ? 0.5f : 1.f;
        auto level = [&](int k, float &vh, float &vl) {        // vh, vl: u^{n-1} in, u^n out
            const float h = uh[o + k], l = ul[o + k];
            float nh, nl;
            level_pair(h, l, vh, vl, buf[o + k], ea, eb, ec, nh, nl);
            if (BC == BC_DIRICHLET && p.data && (a + k == 0 || a + k == n - 1)) {
                nh = p.bh[st][a + k == 0 ? 0 : 1];
                nl = p.bl[st][a + k == 0 ? 0 : 1];
            }
            vh = h;
            vl = l;
            uh[o + k] = nh;
            ul[o + k] = nl;
        };
        if (CTA) {
#pragma unroll
            for (int k = 0; k < kLineSeg; ++k)
                if (k < cnt) level(k, qh[k], ql[k]);
        } else {
            for (int k = 0; k < cnt; ++k) level(k, ph[o + k], pl[o + k]);
        }
        sync();
    }
    for (int j = t; j < n; j += T) {
        const int q = spos_raw(j, m, A.ms, A.mmagic);
        p.vh1[j] = uh[q];
        p.vl1[j] = ul[q];
        if (!CTA) {
            p.vh0[j] = ph[q];
            p.vl0[j] = pl[q];
        }
    }
    if (CTA) {
#pragma unroll
        for (int k = 0; k < kLineSeg; ++k)
            if (k < cnt) {
                p.vh0[a + k] = qh[k];
                p.vl0[a + k] = ql[k];
            }
    }
}

}  // namespace molt

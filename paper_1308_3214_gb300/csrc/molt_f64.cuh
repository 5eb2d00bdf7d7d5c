// molt_f64.cuh -- float64 line passes (sm_103a): lines of up to 8192 points on the
// contiguous axis and 4096 on the others, whole segments or not (longer ones
// stay with the shared-memory kernels, molt_kernels.cuh).
//
// GB300 retires two float64 lane-operations per SM and clock (measured:
// 0.53 T fma/s, against 0.85 T values/s of HBM traffic), so a float64 pass is
// bound by how many float64 operations it spends on a point; everything else
// -- shared memory, barriers, integer work -- runs in the shadow of that pipe.
// These passes spend 7 on an application of D (the earlier ones 13):
//
//   * D in the form  e = kappa (rho s + g),  (1 + d^2) g_j - d (g_{j-1} + g_{j+1}) = s_j,
//     s the second difference of the input.  It is the difference form
//     q_j = c1 s_j + c2 (s_{j-1} + s_{j+1}) of molt_kernels.cuh with the part
//     of q that the solve would undo taken out: with gamma = -c2 / d,
//     c1 s_j + c2 (s_{j-1} + s_{j+1}) = gamma (T s)_j + (c1 - gamma (1 + d^2)) s_j
//     for T the operator on the left, so e = gamma s + kappa T^{-1} s, kappa =
//     c1 - gamma (1 + d^2), rho = gamma / kappa.  Forming s costs 2, the term
//     rho s 1 instead of 3 for q.
//   * kappa never touches a point: the powers leave their units to the
//     consumer's Horner weights (host: coefficients times kappa^p).
//   * each thread owns a segment of R points in registers and solves it once
//     with zero inflow (causal, then anti-causal in place: 2 operations); what
//     flows in from the other segments and the line ends adds a w_k + b d^(len-k)
//     (2 operations), w_k = d^(k+1) (1 - d^(2 (len-k))) / (1 - d^2) the response
//     to an inflow from the left, both factors constants of the launch.  (As
//     a d^k + b d^(len-1-k) the two terms would cancel at slow decay.)  The
//     earlier scheme reduced, rescanned and reduced again.
//
// Carries: each segment publishes E (its zero-inflow y at its last point); the
// causal inflow of segment m is
//   yin_m = sum_j d^(R (j-1)) E_{m-j},
// with which its g at its first point, before anything flows in from the
// right, is H_m = G_m + w_0 yin_m (G zero-inflow); published in turn, it gives
//   gin_m = sum_j d^(R (j-1)) H_{m+j};   a = yin,  b = gin.
// Either sum takes the segments that matter (d^(R win) <= 2^-60; the whole line
// where the decay is slow): one operation a segment, or, for a wide window,
// after log2 B rounds that leave in each slot the sum over a block of B
// segments, one a block.  (Both sums from one exchange cost 5 operations a
// segment, 64 cycles each where a quarter of an SM has a single warp: steps of
// 72 x 65, P = 2, CFL 3.8 took 35.7 us, now 20.8; 256^2, P = 2, 34.0 -> 23.2; 512^2,
// P = 3, 63 -> 55; 1000^2 periodic, P = 3, CFL 4, 183 -> 173.)  What the window
// leaves out is below float64 rounding of the line's largest value; far ahead of a
// point's response a value can be exactly zero.
// Dirichlet (e = 0, or given data, at the ends; s_0 := s_1, s_{n-1} := s_{n-2}):
// the rows at the ends drop out of s, and A' d^j + B' d^(n-1-j) with
//   A' + mu B' = r_0 = e_0/kappa - rho s_1 - g_0,
//   mu A' + B' = r_1 = e_{n-1}/kappa - rho s_{n-2} - g_{n-1}
// joins a and b in the segments it reaches (d^k = (1 - d^2)/d w_k + d^(2 len - k)).
// Periodic lines: what the line's last point hands to its first, all images
// through 1 / (1 - mu), joins yin in the segments it reaches, and what its first
// hands to its last joins gin.  The last segment may hold fewer than R points.
//
// One kernel serves every axis: on the contiguous one neighbouring threads hold
// neighbouring segments of a row and each reads its own segment in 32-byte
// vectors (whole sectors; the segments of a warp are not coalesced, but the
// load unit stays below a tenth of its rate beside the float64 pipe, and
// neither staging nor its barriers are needed); on the strided ones
// neighbouring threads hold neighbouring columns, so that every access is a
// run of C columns.  s waits in shared memory while its registers hold y and g.
//
// Measured, us per pass, against the earlier warp-per-row, clustered and
// shared-memory kernels: 2048^2, P = 3, y 419 -> 225, x 1470 -> 354 (22 and 41
// operations a point: 80 and 83 % of the float64 pipe's cycles); 96 x 100 x 75, P = 2,
// x 154 -> 54, y 260 -> 133, z 72 -> 31; 256^3 periodic, P = 2, x 1150 -> 771, y
// 3000 -> 2150 (87 %), z 746 -> 496.
#pragma once
#include <cstdint>
#include <vector>
#include <cuda_runtime.h>
#include "molt_kernels.cuh"

namespace molt {

constexpr int kF64MaxR = 32;
constexpr int kF64Threads = 256;       // threads per CTA at most
constexpr int kF64BatchP = 5;          // highest order of a batched problem

// Constants of one axis for segments of R points (host, molt_f64.cu).
struct F64Axis {
    int n, G, len_last;    // points, segments, points of the last one
    int R;                 // points per segment
    int win;               // segments whose inflow matters on each side,
    int dbl, blocks;       // summed as blocks of 2^dbl
    double d, rho, kappa;
    double dR, dRl;        // d^R, d^len_last
    double pB, pd[8];      // decay over a block; over 2^k segments
    double e1, id;         // (1 - d^2) / d, 1 / d
    double mu, inv;        // as AxisDev
    double pw[kF64MaxR + 1];   // d^k
    double w[kF64MaxR];    // w_k of a full segment
    double wl[kF64MaxR];   // w_k of the last one
    const double *dpow;    // d^j, j = 0..n
};

struct F64Lines {
    int64_t stride, inner, nlines;
    int64_t pitch;         // contiguous axis: from one line to the next
    int C, cshift;         // lines per CTA; log2 C (strided axes)
};

// The program of a pass: powers (P applications to u, out[p-1] = scale[p-1]
// D^p u / kappa^p) or the Horner pass of HornerParams with its weights times
// kappa^t.  Zero weights, unit scales and the level's weights are flagged by
// the host (a comparison would cost the float64 pipe an operation).
// NO, NF: outputs and fields it has room for.
template <int NO, int NF>
struct F64ProgT {
    int P, ng, nout, epi;
    unsigned add[NO][MAXP];    // [o][t]: bit k set where field k has a weight
    unsigned ucu[NO];          // [o]: bit t set where u has a weight in step t
    unsigned scaled;           // bit p-1: scale[p-1] != 1
    bool hea, heb, hec;        // ea, eb != 0, ec != 1
    bool vec;                  // contiguous axis: every segment starts on 32 bytes
    const double *g[NF];
    double *out[NF];
    double scale[NF];
    double coef[NO][MAXP][NF];
    double cu[NO][MAXP];
    double ea, eb, ec;
    const double *u, *up;
    double *un;
};
struct F64Prog : F64ProgT<MAXP, MAXG> {};

// this thread's place on its line
struct F64Seg {
    double *E, *G, *first, *ends;   // slots [threads] and [4][C]
    double *s;                 // this segment's s: s[k ss]
    int ss;
    int t, st, t0;             // slot, distance to the next segment's slot, slot of segment 0
    int seg, line, C, a;       // a: its first point
    bool live, last, tail;     // on the line; its last segment; shorter than R
};

template <int R>
__device__ __forceinline__ double f64_pick(const double (&z)[R], int k)
{
    double v = z[0];
#pragma unroll
    for (int i = 1; i < R; ++i) v = (i == k) ? z[i] : v;
    return v;
}

// Inflow of this segment, a w_k + b d^(len-k), and the right sides r_0, r_1 of
// the boundary terms, from the segments' e (its zero-inflow y at its last
// point, already in E) and g0 (zero-inflow g at its first).  Sums over a wide
// window first double the block each slot holds (A.dbl times), then run over
// the blocks.  Every thread of the CTA calls it.
template <int BC, bool ADJ>
__device__ __forceinline__ void f64_inflow(const F64Axis &A, const F64Seg &c, double e, double g0, double &a, double &b,
                                           double &r0, double &r1)
{
    const int G = A.G, m = c.seg, t = c.t;
    const double *cur = c.E;
    double *nxt = c.first;
    double yin = 0.0, gin = 0.0, h = 0.0;
    for (int k = 0; k < A.dbl; ++k) {
        if (c.live) nxt[t] = m >= 1 << k ? fma(A.pd[k], cur[t - (c.st << k)], cur[t]) : cur[t];
        __syncthreads();
        cur = nxt;
        nxt = nxt == c.E ? c.first : c.E;
    }
    if (c.live)
        for (int j = min(A.blocks - 1, (m - 1) >> A.dbl); j >= 0; --j)
            yin = fma(A.pB, yin, cur[t - (1 + (j << A.dbl)) * c.st]);
    if (BC == BC_PERIODIC) {
        // what the line's last point hands to its first, all images
        if (c.live && c.last) c.ends[c.line] = A.inv * fma(A.dRl, yin, e);
        __syncthreads();
        if (c.live && m < A.win) yin = fma(c.ends[c.line], A.dpow[c.a], yin);
    }
    if (c.live) {
        h = fma(c.last ? A.wl[0] : A.w[0], yin, g0);
        c.G[t] = h;
    }
    __syncthreads();
    cur = c.G;
    nxt = c.E;
    for (int k = 0; k < A.dbl; ++k) {
        if (c.live) nxt[t] = m + (1 << k) < G ? fma(A.pd[k], cur[t + (c.st << k)], cur[t]) : cur[t];
        __syncthreads();
        cur = nxt;
        nxt = nxt == c.E ? c.G : c.E;
    }
    if (c.live)
        for (int j = min(A.blocks - 1, (G - 2 - m) >> A.dbl); j >= 0; --j)
            gin = fma(A.pB, gin, cur[t + (1 + (j << A.dbl)) * c.st]);
    if (BC == BC_PERIODIC) {
        if (c.live && m == 0) c.ends[c.C + c.line] = A.inv * fma(c.last ? A.dRl : A.dR, gin, h);
        __syncthreads();
        if (c.live && G - 1 - m < A.win) gin = fma(c.ends[c.C + c.line], A.dpow[c.last ? 0 : A.n - c.a - A.R], gin);
    } else {
        double *v = c.ends + 2 * c.C + c.line;
        if (c.live && m == 0) {
            const double g = fma(c.last ? A.dRl : A.dR, gin, h);
            v[0] = ADJ ? -g : fma(-A.rho, c.ends[c.line], -g);
        }
        if (c.live && c.last) {
            const double g = fma(A.dRl, yin, e);
            v[c.C] = ADJ ? -g : fma(-A.rho, c.ends[c.C + c.line], -g);
        }
        __syncthreads();
        if (c.live) {
            r0 = v[0];
            r1 = v[c.C];
        }
    }
    a = yin;
    b = gin;
}

// z: s on entry, rho s + T^{-1} s (with the boundary terms) on exit.  Every
// thread of the CTA calls it.
// ADJ (Dirichlet): on the interior points the operator is D = kappa (rho +
// S M) Delta, S the solve with zero ends, M = 1 but 1 - rho d at each of the
// two points next to the ends (what s_0 := s_1 and s_{n-1} := s_{n-2} put
// into rows 1 and n-2).  S is symmetric, so D^T = kappa Delta^T (rho + M S):
// here z becomes rho z + M S z for z with its end values dropped, and Delta^T,
// the second difference with zeros past the interior, follows at the caller.
template <int R, int BC, bool ADJ>
__device__ __forceinline__ void f64_solve(double (&z)[R], const F64Axis &A, const F64Seg &c)
{
    const double d = A.d;
    const int L = A.len_last;
    double e = 0.0;
    if (c.live) {
        if (BC == BC_DIRICHLET) {
            if (c.seg == 0) {
                if (!ADJ) c.ends[c.line] = z[1];
                z[0] = 0.0;
            }
            // s_{n-2}: the last segment's, or the end of the one before it
            if (!ADJ && (L >= 2 ? c.last : c.seg == A.G - 2)) c.ends[c.C + c.line] = f64_pick<R>(z, L >= 2 ? L - 2 : R - 1);
        }
        if (c.last) {
            const int keep = BC == BC_DIRICHLET ? L - 1 : L;
#pragma unroll
            for (int k = 0; k < R; ++k) z[k] = k < keep ? z[k] : 0.0;
        }
#pragma unroll
        for (int k = 0; k < R; ++k) c.s[k * c.ss] = z[k];
#pragma unroll
        for (int k = 1; k < R; ++k) z[k] = fma(d, z[k - 1], z[k]);
        e = z[R - 1];
        if (c.tail) {                                  // y ends with the line
            e = f64_pick<R>(z, L - 1);
#pragma unroll
            for (int k = 0; k < R; ++k) z[k] = k < L ? z[k] : 0.0;
        }
#pragma unroll
        for (int k = R - 2; k >= 0; --k) z[k] = fma(d, z[k + 1], z[k]);
        c.E[c.t] = e;
    }
    __syncthreads();
    double a = 0.0, b = 0.0, r0 = 0.0, r1 = 0.0;
    f64_inflow<BC, ADJ>(A, c, e, z[0], a, b, r0, r1);
    if (c.live) {
        if (BC == BC_DIRICHLET) {
            // the boundary terms in the segments they reach: of both ends
            // where the window covers the line, else of the nearer end alone
            const bool all = A.win >= A.G;
            if (all) {
                const double t0 = (r0 - A.mu * r1) * A.inv;
                r1 = (r1 - A.mu * r0) * A.inv;
                r0 = t0;
            }
            if (all || c.seg < A.win) {
                const double t0 = r0 * A.dpow[c.a];
                a = fma(t0, A.e1, a);
                b = fma(t0, c.last ? A.dRl : A.dR, b);
            }
            if (all || A.G - 1 - c.seg < A.win) b = fma(r1 * A.dpow[A.n - c.a - (c.last ? L : R)], A.id, b);
        }
#pragma unroll
        for (int k = 0; k < R; ++k) z[k] = fma(A.rho, c.s[k * c.ss], z[k]);
        if (c.tail) {
#pragma unroll
            for (int k = 0; k < R; ++k) z[k] = k < L ? fma(b, A.pw[k < L ? L - k : 0], fma(a, A.wl[k], z[k])) : 0.0;
        } else {
#pragma unroll
            for (int k = 0; k < R; ++k) z[k] = fma(b, A.pw[R - k], fma(a, A.w[k], z[k]));
        }
        if constexpr (ADJ) {
            const int km = L >= 2 ? L - 2 : R - 1;     // point n - 2 and its segment
            const bool hm = L >= 2 ? c.last : c.seg == A.G - 2;
            double g1 = 0.0, gm = 0.0;
            if (c.seg == 0) g1 = fma(-A.rho, c.s[c.ss], z[1]);
            if (hm) gm = fma(-A.rho, c.s[km * c.ss], f64_pick<R>(z, km));
            if (c.seg == 0) z[1] = fma(-A.rho * A.d, g1, z[1]);
            if (hm) {
                const double v = fma(-A.rho * A.d, gm, f64_pick<R>(z, km));
#pragma unroll
                for (int k = 0; k < R; ++k) z[k] = k == km ? v : z[k];
            }
        }
        if (BC == BC_DIRICHLET) {
            if (c.seg == 0) z[0] = 0.0;
            if (c.last) {
#pragma unroll
                for (int k = 0; k < R; ++k) z[k] = k == L - 1 ? 0.0 : z[k];
            }
        }
    }
}

// z <- second difference of z (+ cu r), zl and zr the neighbours' values; the
// last segment's right neighbour enters at its own length
template <int R>
__device__ __forceinline__ void f64_sdiff(double (&z)[R], double zl, double zr, const F64Axis &A, const F64Seg &c)
{
    if (c.tail) {
#pragma unroll
        for (int k = 1; k < R; ++k) z[k] = k == A.len_last ? zr : z[k];
    }
    double dm = z[0] - zl;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const double dp = (k + 1 < R ? z[k + 1] : zr) - z[k];
        z[k] = dp - dm;
        dm = dp;
    }
}

// f(k, v) for this segment's points k < len of a field, v = q[k st].  (Plain
// loads: u^{n-1}, which the next level may be written over, is one of the fields.)
// vec: in 32-byte vectors (contiguous axis; len is a multiple of 4 then).
template <int R, bool CONTIG, class F>
__device__ __forceinline__ void f64_each(const double *q, int64_t st, int len, bool vec, F &&f)
{
    if (CONTIG && vec) {
#pragma unroll
        for (int k = 0; k < R; k += 4)
            if (k < len) {
                const double4_32a v = *reinterpret_cast<const double4_32a *>(q + k);
                f(k, v.x);
                f(k + 1, v.y);
                f(k + 2, v.z);
                f(k + 3, v.w);
            }
    } else if (CONTIG) {
#pragma unroll
        for (int k = 0; k < R; ++k)
            if (k < len) f(k, q[k]);
    } else {
#pragma unroll
        for (int k = 0; k < R; ++k) {
            if (k < len) f(k, *q);
            q += st;
        }
    }
}

template <int R, bool CONTIG>
__device__ __forceinline__ void f64_store(double *q, int64_t st, int len, bool vec, const double (&z)[R])
{
    if (CONTIG && vec) {
#pragma unroll
        for (int k = 0; k < R; k += 4)
            if (k < len) {
                double4_32a v;
                v.x = z[k];
                v.y = z[k + 1];
                v.z = z[k + 2];
                v.w = z[k + 3];
                *reinterpret_cast<double4_32a *>(q + k) = v;
            }
    } else {
        const int64_t s1 = CONTIG ? 1 : st;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            if (k < len) *q = z[k];
            q += s1;
        }
    }
}

// KM 0: powers; 1: Horner with nout outputs (or the next level).  Dynamic
// shared memory: slots [4][threads] (E, G, first, last), ends [4][C], s [R]
// [threads], (KM 1) r [R][threads].
__host__ __device__ inline size_t f64_smem(int threads, int C, int R, bool horner)
{
    return sizeof(double) * ((size_t)threads * 4 + 4 * C + (size_t)R * threads * (horner ? 2 : 1));
}

// One CTA's lines, from block * C on.  ADJ: the transposed operators (the
// adjoint step; Dirichlet, one output).  PAD: lines end in padding (zeros) up
// to a multiple of 4 points, which vectors may read and write back as zeros.
template <int R, int BC, int KM, bool CONTIG, bool ADJ, bool PAD, class Prog>
__device__ __forceinline__ void f64_pass(const F64Axis &A, const F64Lines &LS, const Prog &p, int block, double *sm64)
{
    const int T = blockDim.x, t = threadIdx.x, n = A.n, G = A.G;
    double *first = sm64 + 2 * T, *last = sm64 + 3 * T, *sbuf = sm64 + 4 * T + 4 * LS.C;
    F64Seg c;
    c.first = first;
    c.E = sm64;
    c.G = sm64 + T;
    c.ends = sm64 + 4 * T;
    c.s = sbuf + t;
    c.ss = T;
    c.t = t;
    c.C = LS.C;
    if (CONTIG) {
        c.line = t / G;
        c.seg = t - c.line * G;
        c.t0 = c.line * G;
        c.st = 1;
        c.live = c.line < LS.C;
    } else {
        c.line = t & (LS.C - 1);
        c.seg = t >> LS.cshift;
        c.t0 = c.line;
        c.st = LS.C;
        c.live = c.seg < G;
    }
    c.last = c.seg == G - 1;
    c.tail = c.last && A.len_last < R;
    const int a = c.a = c.seg * R, len = c.last ? A.len_last : R;
    const int64_t line = (int64_t)block * LS.C + c.line;
    const bool io = c.live && line < LS.nlines;
    const int64_t st = CONTIG ? 1 : LS.stride;
    const int64_t lbase = !io ? 0 : CONTIG ? line * LS.pitch : (line % LS.inner) + (line / LS.inner) * LS.inner * (int64_t)n;
    const int64_t at = lbase + (int64_t)a * st;        // this segment's first point

    double z[R];
#pragma unroll
    for (int k = 0; k < R; ++k) z[k] = 0.0;
    // s of u: points a-1 .. a+len (wrapped or clamped)
    if (io) {
        auto row = [&](int j) -> int64_t {
            if (BC == BC_PERIODIC) return j < 0 ? j + n : (j >= n ? j - n : j);
            return j < 0 ? 0 : (j > n - 1 ? n - 1 : j);
        };
        const double zl = ADJ ? 0.0 : p.u[lbase + row(a - 1) * st], zr = ADJ ? 0.0 : p.u[lbase + row(a + len) * st];
        f64_each<R, CONTIG>(p.u + at, st, len, p.vec, [&](int k, double v) { z[k] = v; });
        if (!ADJ) f64_sdiff<R>(z, zl, zr, A, c);
    }
    // neighbours' values through shared memory, then the second difference
    auto exchange_sdiff = [&]() {
        if (c.live) {
            first[t] = z[0];
            last[t] = c.tail ? f64_pick<R>(z, A.len_last - 1) : z[R - 1];
        }
        __syncthreads();
        if (c.live) {
            double zl = 0.0, zr = 0.0;
            const int sl = c.seg > 0 ? c.seg - 1 : (BC == BC_PERIODIC ? G - 1 : -1);
            const int sr = c.last ? (BC == BC_PERIODIC ? 0 : -1) : c.seg + 1;
            if (sl >= 0) zl = last[c.t0 + sl * c.st];
            if (sr >= 0) zr = first[c.t0 + sr * c.st];
            f64_sdiff<R>(z, zl, zr, A, c);
        }
    };

    auto apply = [&]() {                               // ADJ: D^T / kappa of z
        f64_solve<R, BC, ADJ>(z, A, c);
        if (ADJ) exchange_sdiff();
    };
    auto pad = [&]() {                                 // points past the line's end, before they are stored
        if (PAD && CONTIG && c.tail) {
#pragma unroll
            for (int k = 0; k < R; ++k) z[k] = k < len ? z[k] : 0.0;
        }
    };

    if (KM == 0) {
        for (int q = 0; q < p.P; ++q) {
            if (!ADJ && q > 0) exchange_sdiff();
            apply();
            if (ADJ) pad();
            if (p.out[q] != nullptr && io) {
                if (p.scaled >> q & 1u) {              // the last power of mol_apply_D
                    const double sc = p.scale[q];
                    double w[R];
#pragma unroll
                    for (int k = 0; k < R; ++k) w[k] = sc * z[k];
                    f64_store<R, CONTIG>(p.out[q] + at, st, len, p.vec, w);
                } else {
                    f64_store<R, CONTIG>(p.out[q] + at, st, len, p.vec, z);
                }
            }
        }
        return;
    }
    // Horner: r = s of u stays in shared memory
    double *r = sbuf + (size_t)R * T + t;
#pragma unroll
    for (int k = 0; k < R; ++k) r[k * T] = z[k];
    for (int o = 0; o < p.nout; ++o) {
#pragma unroll
        for (int k = 0; k < R; ++k) z[k] = 0.0;
        bool zero = true;
        for (int q = p.P; q >= 0; --q) {
            const unsigned add = p.add[o][q];
            if (io)
                for (int f = 0; f < p.ng; ++f)
                    if (add >> f & 1u) {
                        const double w = p.coef[o][q][f];
                        f64_each<R, CONTIG>(p.g[f] + at, st, len, p.vec, [&](int k, double v) { z[k] = fma(w, v, z[k]); });
                    }
            zero = zero && add == 0;
            if (q == 0) break;
            const double w = p.cu[o][q];
            if (zero) {
                if (!(p.ucu[o] >> q & 1u)) continue;
                if (!ADJ) __syncthreads();         // the slots' last readers are done
#pragma unroll
                for (int k = 0; k < R; ++k) z[k] = w * r[k * T];
            } else {
                if (!ADJ) exchange_sdiff();
                if (p.ucu[o] >> q & 1u) {
#pragma unroll
                    for (int k = 0; k < R; ++k) z[k] = fma(w, r[k * T], z[k]);
                }
            }
            apply();
            zero = false;
        }
        if (!io) continue;
        if (p.epi) {
            // next level: ea u + eb u_prev + ec F
            if (p.hec) {
#pragma unroll
                for (int k = 0; k < R; ++k) z[k] *= p.ec;
            }
            if (p.hea) f64_each<R, CONTIG>(p.u + at, st, len, p.vec, [&](int k, double v) { z[k] = fma(p.ea, v, z[k]); });
            if (p.heb) f64_each<R, CONTIG>(p.up + at, st, len, p.vec, [&](int k, double v) { z[k] = fma(p.eb, v, z[k]); });
        }
        pad();
        f64_store<R, CONTIG>((p.epi ? p.un : p.out[o]) + at, st, len, p.vec, z);
    }
}

template <int R, int BC, int KM, bool CONTIG>
__global__ void __launch_bounds__(kF64Threads, 2) k_f64(const __grid_constant__ F64Axis A, F64Lines LS,
                                                       const __grid_constant__ F64Prog p)
{
    extern __shared__ __align__(16) double sm64[];
    f64_pass<R, BC, KM, CONTIG, false, false>(A, LS, p, (int)blockIdx.x, sm64);
}

// The same passes over the problems of a batch (Dirichlet): a CTA looks its
// problem up in the work list and copies the problem's constants (1.5 KB) to
// shared memory in front of the pass's own; one launch per segment length and
// CTA size.  The constants cost shared-memory loads instead of constant operands,
// which the float64 pipe hides.  Warps beyond the problem's lines leave.
// Measured against the earlier batch passes (13 operations an application, a warp
// per row, three exchanges per column): 100 problems of 64..256 points, 9 steps,
// 5379 -> 2958 us; 4 problems, 1337 -> 796; gradient on 131 x 160, P = 2 (one problem,
// 80 steps), 6861 -> 2912, on 500 x 301 3074 -> 1972.
struct F64Task {
    F64Axis A;
    F64Lines L;
    F64ProgT<1, kF64BatchP> p;  // its pointers: from the launch, off elements on
    long long off;
};

struct F64BatchPass {
    const F64Task *tasks;
    const int2 *items;          // (task, group of C lines)
    const double *u, *up, *g[kF64BatchP];
    double *un, *out[kF64BatchP];
    double ea, eb, ec;
};

// A problem of a batch as the plan needs it; coef rows are ldc apart.
struct F64BatchGrid {
    const AxisDev *ax, *ay;
    double nux, nuy;
    int P, pitch, ldc;
    long long off;
    const double *cu, *coef;
};
struct F64BatchClass {
    int R, threads;
    size_t smem;
    int begin, count;           // of the work list
};
struct F64BatchLists {
    std::vector<F64Task> tasks; // x passes, then y passes
    std::vector<int2> items;
    std::vector<F64BatchClass> classes[2];
};
void f64_batch_plan(const F64BatchGrid *probs, int nprob, int quad, int sms, F64BatchLists &out);
cudaError_t launch_f64_batch(int axis, bool adj, const F64BatchClass &c, F64BatchPass bp, cudaStream_t s);
cudaError_t configure_f64_batch_kernels();

__host__ __device__ constexpr int f64_task_words() { return (int)((sizeof(F64Task) + 15) / 16 * 2); }

template <int R, int KM, bool CONTIG, bool ADJ>
__global__ void __launch_bounds__(kF64Threads, 2) k_f64_batch(const __grid_constant__ F64BatchPass bp)
{
    extern __shared__ __align__(16) double sm64[];
    static_assert(sizeof(F64Task) % 8 == 0, "copied in words");
    F64Task &k = *reinterpret_cast<F64Task *>(sm64);
    const int2 item = bp.items[blockIdx.x];
    {
        const unsigned long long *src = reinterpret_cast<const unsigned long long *>(bp.tasks + item.x);
        unsigned long long *dst = reinterpret_cast<unsigned long long *>(sm64);
        for (int i = threadIdx.x; i < (int)(sizeof(F64Task) / 8); i += blockDim.x) dst[i] = __ldg(src + i);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        k.p.u = bp.u + k.off;
        k.p.up = bp.up + k.off;
        k.p.un = bp.un + k.off;
        for (int q = 0; q < k.p.P; ++q) {
            k.p.g[q] = bp.g[q] + k.off;
            k.p.out[q] = bp.out[q] + k.off;
        }
        k.p.ea = bp.ea; k.p.eb = bp.eb; k.p.ec = bp.ec;
        k.p.hea = bp.ea != 0.0; k.p.heb = bp.eb != 0.0; k.p.hec = bp.ec != 1.0;
    }
    __syncthreads();
    // (strided axes pad the threads of a line's C columns only: C G threads work)
    if ((int)(threadIdx.x & ~31u) >= k.L.C * k.A.G) return;
    f64_pass<R, BC_DIRICHLET, KM, CONTIG, ADJ, true>(k.A, k.L, k.p, item.y, sm64 + f64_task_words());
}

}  // namespace molt

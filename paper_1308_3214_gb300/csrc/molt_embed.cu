// molt_embed.cu -- embedded boundaries (Sec. 4.3): the 2D scheme on a domain
// cut out of a grid, its lines being "line objects" (the interior grid nodes
// of a grid line plus a boundary point at each end, off the grid).
//
// L^{-1} on a line object of m interior nodes: nodes x_0 = a, x_1..x_m (spacing
// h, x_1 = a + ga), x_{m+1} = b = x_m + gb; the data at a and b are zero.
//   J^L_k = (alpha/2) int_{x_{k-1}}^{x_k} e^{-alpha (x_k - y)} p(y) dy,
//   J^R_k = (alpha/2) int_{x_k}^{x_{k+1}} e^{-alpha (y - x_k)} p(y) dy,
// p the quadratic through x_{k-1}, x_k, x_{k+1} (moved one node inward where
// that node does not exist), integrated exactly; I^L_k = e^{-alpha(x_k -
// x_{k-1})} I^L_{k-1} + J^L_k from I^L_0 = 0, I^R likewise from the right;
// w = I^L + I^R + A e^{-alpha (x - a)} + B e^{-alpha (b - x)} with w(a) = w(b)
// = 0.  Both precisions evaluate D = 1 - L^{-1} in a difference form on the
// line object (the kernels' comments); a line is read and written in place in
// the caller's layout: x lines with stride 1, y lines with stride nx.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "molt.h"
#include "molt_internal.h"

namespace {

constexpr int kObjMaxM = 2046;             // interior nodes of a line object at most
constexpr int kObjThreads32 = 128;         // threads per line object in the float32 sweep
constexpr int kObjCpb[2] = {1, 4};         // float32 sweep: line objects per CTA, contiguous / strided axis

// Float64 line objects: the difference form of the float32 sweeps (below) with
// the chain of molt_f64.cuh.  With e = D v and T' = (1 - d^2) T the recurrences
// read T'_k = q_k + d T'_{k+1} (from b to a) and e_k = d e_{k-1} + T'_k (from a to
// b), all cells decaying by d: the short end cells enter only as factors, e_1 =
// lam T'_1 (lam = (1 - dA^2)/(1 - d^2)), and in the boundary terms.  q_k combines
// second differences as in the float32 sweeps (weights times 1 - d^2).
struct ObjLine {
    long long base;     // element index of the first interior node
    int m;              // interior nodes
    int pad_;
    double dA, dB;      // e^{-alpha ga}, e^{-alpha gb}
    double lam;
    double mu, inv;     // e^{-alpha (b - a)}, 1 / (1 - mu^2)
    double g11, g12;    // q_1 = g11 s_1 + g12 s_2
    double gNa, gNb;    // q_m = gNa s_{m-1} + gNb s_m
    double p1, q1;      // s_1 = p1 (v_2 - v_1) - q1 v_1 (v_2 = 0 when m = 1)
    double pm, qm;      // s_m = pm (0 - v_m) - qm (v_m - v_{m-1})
};

constexpr int kObjR = 16;                  // points per thread at most

struct ObjAxis {
    long long stride;   // element stride along the lines (1 for x, nx for y)
    int threads, ctas;  // launch shape
    const int4 *items;  // [ctas][threads]: line (-1: none), segment, slot of the line's segment 0,
                        // slots to the next segment
    int win;            // segments whose inflow matters
    int direct;         // d too small to divide by: e1 = id = 0
    double d, e1, id;   // e^{-alpha h}, (1 - d^2)/d, 1/d
    double gc, ge;      // uniform rows
    const double *dpow; // d^k, k = 0..kObjMaxM
    double pw[kObjR + 1];
    double w[kObjR + 1][kObjR];   // inflow weights of a segment of len points (molt_f64.cuh)
};

enum : int { OBJ_D = 0, OBJ_LINV = 1, OBJ_BOTH = 2 };

constexpr int kCombMax = 8;
// out = sum_t c_t x_t (+ cw times a sweep's result)
struct CombTerms {
    int n;
    double cw;
    double c[kCombMax];
    const double *x[kCombMax];
    double *out;        // nullptr: none
};

template <bool FWD>
__device__ __forceinline__ void affine_scan32(float &p, float &q, int lane)
{
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        const float pp = FWD ? __shfl_up_sync(0xffffffffu, p, k) : __shfl_down_sync(0xffffffffu, p, k);
        const float qq = FWD ? __shfl_up_sync(0xffffffffu, q, k) : __shfl_down_sync(0xffffffffu, q, k);
        const bool take = FWD ? lane >= k : lane + k < 32;
        if (take) {
            q = qq * p + q;
            p = pp * p;
        }
    }
}

// OBJ_D: out = D v; OBJ_LINV: out = v - D v (= L^{-1} v); OBJ_BOTH: out = D v, out2 =
// v - D v (and out3 = D v when given).  accum adds to out.  cb.out: the result is
// not stored but combined, cb.out = cw result + sum c_t x_t (the level update
// rides on the last sweep of F).
//
// A thread owns R consecutive nodes of a line, counted from the line's far end
// (index 0 = node m), so that the first chain runs forward.  Which segment of
// which line is a table made with the handle: whole lines packed into the CTAs
// whatever their lengths, the segments of a row on neighbouring threads, those
// of (up to) 4 neighbouring columns interleaved.  The sweep reads its nodes and two halo nodes on each side straight from the
// field; one barrier carries the segments' E and G, a second the line's two
// end values (T'_1 is large where the first gap is small: lam multiplies it
// before it is added to anything).  Bound by float64 latency on grids of a few hundred nodes per
// line (64 cycles an operation and a warp per SM quarter), by the float64 pipe
// above: 10 operations a node instead of 18 (14 to 16 issued, with the ends of
// segments and lines), spread over a line's worth of threads instead of one warp.
// us per step of the ellipse at P = 2, 10 sweeps and a combination before, 9 sweeps
// now: 129^2 89 -> 78, 400^2 137 -> 97, 777^2 217 -> 142, 2048^2 647 -> 564 (73 % of the
// float64 pipe).
template <int R>
__global__ void __launch_bounds__(512) k_obj_sweep(const __grid_constant__ ObjAxis ax, const ObjLine *__restrict__ lines,
                                                   const double *__restrict__ in, double *out, double *out2, double *out3,
                                                   int mode, int accum, const __grid_constant__ CombTerms cb)
{
    extern __shared__ __align__(16) double smo[];
    const int T = blockDim.x, t = threadIdx.x;
    double *E = smo, *G = smo + T, *ends = smo + 2 * T;          // [2][T], at the line's slot 0: its
    const int4 it = ax.items[blockIdx.x * T + t];                // zero-inflow e_m and inflow to T'_1
    const int seg = it.y, t0 = it.z, st = it.w;
    const bool on = it.x >= 0;
    const ObjLine &ln = lines[on ? it.x : 0];
    const int m = ln.m, a = seg * R;
    // the tables are constant; the fields are the work of the kernels before
    molt::pdl_enter();
    const bool live = on, last = live && a + R >= m;
    const int len = live ? min(R, m - a) : 0;
    // node of index j (0 = node m): field element top - j stride
    const long long top = ln.base + (long long)(m - 1 - a) * ax.stride;
    double v[R], z[R];
    if (live) {
        const double *q = in + top;
        auto val = [&](int j) -> double { return a + j >= 0 && a + j < m ? q[-(long long)j * ax.stride] : 0.0; };
        double f[R + 4];                                          // v at j = -2 .. R + 1
#pragma unroll
        for (int j = -2; j < R + 2; ++j) f[j + 2] = val(j);
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = f[j + 2];
        // second differences at j = -1 .. R; the end triples with their spacings
        // (only the threads that hold them: a predicated operation costs the
        // float64 pipe as much as an executed one)
        double sd[R + 2];
        double dm = f[1] - f[0];
#pragma unroll
        for (int j = -1; j <= R; ++j) {
            const double dp = f[j + 3] - f[j + 2];
            sd[j + 1] = dp - dm;
            dm = dp;
        }
        const int k1 = m - 1 - a;                                 // node 1
        if (seg == 0) sd[1] = ln.qm * (f[3] - f[2]) - ln.pm * (f[2] - f[1]);      // node m
        if (k1 <= R) {
            double c0 = 0.0, c1 = 0.0, c2 = 0.0;
#pragma unroll
            for (int j = 0; j <= R; ++j) {
                c0 = j == k1 ? f[j + 1] : c0;
                c1 = j == k1 ? f[j + 2] : c1;
                c2 = j == k1 && j < R ? f[j < R ? j + 3 : 0] : c2;    // (the boundary's zero at j = R)
            }
            const double s1 = ln.q1 * (c2 - c1) - ln.p1 * (c1 - c0);
#pragma unroll
            for (int j = 0; j <= R; ++j) sd[j + 1] = j == k1 ? s1 : sd[j + 1];
        }
#pragma unroll
        for (int j = 0; j < R; ++j) z[j] = fma(ax.ge, sd[j] + sd[j + 2], ax.gc * sd[j + 1]);
        if (seg == 0) z[0] = fma(ln.gNb, sd[1], ln.gNa * sd[2]);
        if (last) {
            double s1 = 0.0, s2 = 0.0;
#pragma unroll
            for (int j = 0; j < R; ++j) {
                s1 = j == k1 ? sd[j + 1] : s1;
                s2 = j == k1 ? sd[j] : s2;
            }
            const double q1 = fma(ln.g11, s1, ln.g12 * s2);
#pragma unroll
            for (int j = 0; j < R; ++j) z[j] = j < k1 ? z[j] : (j == k1 ? q1 : 0.0);
        }
#pragma unroll
        for (int j = 1; j < R; ++j) z[j] = fma(ax.d, z[j - 1], z[j]);
        const double e = z[R - 1];
        if (last) {                                               // T'_1 enters e_1 times lam
            double e1 = z[0];
#pragma unroll
            for (int j = 1; j < R; ++j) e1 = j == len - 1 ? z[j] : e1;
            e1 *= ln.lam;
#pragma unroll
            for (int j = 0; j < R; ++j) z[j] = j < len - 1 ? z[j] : (j == len - 1 ? e1 : 0.0);
        }
#pragma unroll
        for (int j = R - 2; j >= 0; --j) z[j] = fma(ax.d, z[j + 1], z[j]);
        E[t] = e;
        G[t] = z[0];
    }
    // what the result is added to, and the decays of the boundary terms: on
    // their way while the carries are
    const int ns = (m + R - 1) / R;
    double add[R], d1 = 0.0, da = 0.0, db = 0.0;
#pragma unroll
    for (int j = 0; j < R; ++j) add[j] = 0.0;
    if (live) {
        d1 = __ldg(ax.dpow + m - 1);
        da = __ldg(ax.dpow + a);
        db = __ldg(ax.dpow + m - a - len);
        if (accum) {
#pragma unroll
            for (int j = 0; j < R; ++j)
                if (j < len) add[j] = out[top - (long long)j * ax.stride];
        }
        if (cb.out) {
            if (accum) {
#pragma unroll
                for (int j = 0; j < R; ++j) add[j] *= cb.cw;
            }
            for (int k = 0; k < cb.n; ++k) {
                const double *x = cb.x[k] + top;
                const double c = cb.c[k];
#pragma unroll
                for (int j = 0; j < R; ++j)
                    if (j < len) add[j] = fma(c, x[-(long long)j * ax.stride], add[j]);
            }
        }
    }
    __syncthreads();
    double yin = 0.0, gin = 0.0;
    if (live) {
        const int J = min(ax.win, ns);
        const double dR = ax.pw[R], dl = ax.pw[m - (ns - 1) * R], w0 = ax.w[R][0], wl = ax.w[m - (ns - 1) * R][0];
        for (int l = max(seg - J, 0); l < seg; ++l) yin = fma(dR, yin, E[t0 + l * st]);
        double Y = fma(dR, yin, E[t]), pr = 1.0;
        for (int l = seg + 1; l <= min(seg + J, ns - 1); ++l) {
            gin = fma(pr, fma(l == ns - 1 ? wl : w0, Y, G[t0 + l * st]), gin);
            Y = fma(dR, Y, E[t0 + l * st]);
            pr *= dR;
        }
        if (seg == 0) ends[t0] = fma(last ? dl : dR, gin, G[t]);
        if (last) ends[T + t0] = dl * yin;
    }
    __syncthreads();
    if (!live) return;
    // boundary terms: what the inflow's part of e_1 lacks (lam - 1) and e = 0 at b
    {
        const bool all = ax.win + 1 >= ns, nl = all || seg < ax.win, nr = all || ns - 1 - seg <= ax.win;
        if (nl || nr) {
            const double y1 = (ln.lam - 1.0) * ends[T + t0];
            const double em = fma(y1, d1, ends[t0]);
            const double B = -ln.dB * em * ln.inv;
            if (nl) {
                const double ca = B * ln.dB * da;
                yin = fma(ca, ax.e1, yin);
                gin = fma(ca, ax.pw[len], gin);
            }
            if (nr) gin = fma(fma(-B * ln.mu, ln.dA, y1) * db, ax.id, gin);
            // a decay too small to divide by (f64_inverse_decay) carries nothing
            // past the end nodes m and 1, but these stand a gap away from the boundary
            // points, whatever its length, and have their terms
            if (ax.direct) {
                if (seg == 0) z[0] = fma(B, ln.dB, z[0]);
                if (last) {
#pragma unroll
                    for (int j = 0; j < R; ++j) z[j] = j == len - 1 ? z[j] + fma(-B * ln.mu, ln.dA, y1) : z[j];
                }
            }
        }
    }
    // e, then the result
#pragma unroll
    for (int j = 0; j < R; ++j)
        if (j < len) z[j] = fma(gin, ax.pw[len - j], fma(yin, ax.w[len][j], z[j]));
    double *o = (cb.out ? cb.out : out) + top;
#pragma unroll
    for (int j = 0; j < R; ++j)
        if (j < len) {
            const long long at = -(long long)j * ax.stride;
            if (mode == OBJ_BOTH) {
                out2[top + at] = v[j] - z[j];
                if (out3) out3[top + at] = z[j];
            }
            double r = mode == OBJ_LINV ? v[j] - z[j] : z[j];
            if (cb.out) r = fma(cb.cw, r, add[j]);
            else if (accum) r += add[j];
            o[at] = r;
        }
}

// out = sum_t c_t x_t at the interior nodes (out may be one of the x_t)
__global__ void __launch_bounds__(256) k_obj_combine(CombTerms t, const ObjLine *rows, int nrows)
{
    for (int li = blockIdx.x; li < nrows; li += gridDim.x) {
        const long long base = rows[li].base;
        for (int k = threadIdx.x; k < rows[li].m; k += blockDim.x) {
            double v = 0.0;
            for (int j = 0; j < t.n; ++j) v += t.c[j] * t.x[j][base + k];
            t.out[base + k] = v;
        }
    }
}

// ---------------------------------------------------------------------------
// float32 sweeps: the difference form of D on a line object
// ---------------------------------------------------------------------------
// With g_k the decay of cell k (between x_{k-1} and x_k) and e = D v, the two
// recurrences and the boundary terms give, at every interior node k = 1..N-1,
//   T_k - g_{k+1} T_{k+1} = q_k,   T_k = (e_k - g_k e_{k-1}) / (1 - g_k^2),
// with e = 0 at both boundary points; q_k is local in v and vanishes on
// linear data, so it is a combination of second divided differences:
//   q_k = ge s_{k-1} + gc s_k + ge s_{k+1} on the uniform interior
//   (s_t = v_{t-1} - 2 v_t + v_{t+1}, the divided difference times h^2), and
//   two per-line coefficients on rows 1 and N-1, whose end triples (a, x_1,
//   x_2) and (x_{m-1}, x_m, b) have their own spacings.
// The anti-causal recurrence gives T from T_N = 0, the causal one e from
// e_0 = 0, and the homogeneous solutions A' e^{-alpha (x - a)} + B'
// e^{-alpha (b - x)} restore e_N = 0.  D v then never subtracts two nearly
// equal numbers, so float32 sweeps keep their accuracy (D v << v for smooth
// fields); the input's second differences come from float32 pairs when the
// input is a time level.
struct ObjLineF {
    long long base;     // element index of the first interior node
    int m, pad_;
    float dA, dB;       // decays of the end cells
    float rA, rB;       // dA / d, dB / d (d as in the table d^k, obj_decay_floor32)
    float cA, cB;       // 1 - dA^2, 1 - dB^2
    float mu, inv;      // e^{-alpha (b - a)}, 1 / (1 - mu^2)
    float g11, g12;     // row 1: q_1 = g11 s_1 + g12 s_2
    float gNa, gNb;     // row N-1: q_m = gNa s_{m-1} + gNb s_m
    float p1, q1;       // s_1 = p1 (v_2 - v_1) - q1 v_1 (v_2 = 0 when m = 1)
    float pm, qm;       // s_m = pm (0 - v_m) - qm (v_m - v_{m-1})
};

struct ObjAxisF {
    long long stride;
    float d, c;         // e^{-alpha h}, 1 - d^2
    float gc, ge;       // uniform rows
    const float *dpow;  // d^k
};

enum : int { OBJF_D = 0, OBJF_LINV = 1, OBJF_BOTH = 2 };

// out = sum_t c_t x_t in float32 (the partial sums of F)
struct CombTermsF {
    int n;
    float c[kCombMax];
    const float *x[kCombMax];
};

// The level update that rides on F's last sweep: (nh, nl) = a u + b up + c
// sum_t c_t x_t in pair arithmetic, term own being the sweep's result, which
// is not stored.  (A pass of its own read every term again, 20 us at 2048^2.)
// With that and the small sweeps overlapping their launches, us per step of
// the ellipse at P = 2: 257^2 61 -> 50, 400^2 75 -> 61, 777^2 85 -> 79, 1025^2
// 104 -> 98, 2048^2 190 -> 181.
struct LevelF {
    CombTermsF t;
    int own;
    float a, b, c;
    const float *uh, *ul, *ph, *pl;
    float *nh, *nl;       // nullptr: none
};

__device__ __forceinline__ void obj_level32(const LevelF &lv, long long i, float own)
{
    const float uh = lv.uh[i], ul = lv.ul[i];
    const float ph = lv.b != 0.f ? lv.ph[i] : 0.f, pl = lv.b != 0.f ? lv.pl[i] : 0.f;
    float F = 0.f;
    for (int j = 0; j < lv.t.n; ++j) F += lv.t.c[j] * (j == lv.own ? own : lv.t.x[j][i]);
    float h, l;
    molt::level_pair(uh, ul, ph, pl, F, lv.a, lv.b, lv.c, h, l);
    lv.nh[i] = h;
    lv.nl[i] = l;
}

// MODE OBJF_D: out = D v; OBJF_LINV: out = v - D v (= L^{-1} v); OBJF_BOTH:
// out = D v and out2 = v - D v (and out3 = D v when given).  accum adds to
// out.  PAIR: v is a float32 pair level (in = hi, lo = lo plane), else a
// float32 field.
// A CTA takes CPB consecutive line objects at a time, kObjThreads32 threads
// per line.  Loads and stores run over grid positions along the lines, the
// CPB lines interleaved, so that on the strided axis (consecutive lines =
// adjacent columns) a row's CPB values are read and written together.  In the
// recurrences each thread reduces a chunk of its group's line, the chunk maps
// are composed over the lanes of a warp (shuffles) and over the group's warps
// (their totals in shared memory), and each chunk is re-run from its carry.
// slot: elements per line array (> obj_slot(m + 1)), four arrays per line.  lv.nh: the
// result is not stored but combined into the next level.
// one word of padding per 32: threads that walk chunks of 4 or 8 nodes start
// on different banks
__host__ __device__ __forceinline__ int obj_slot(int k) { return k + (k >> 5); }

template <bool PAIR, int CPB>
__global__ void __launch_bounds__(kObjThreads32 * CPB) k_obj_sweep32(ObjAxisF ax, const ObjLineF *lines, int nlines,
                                                                    const float *__restrict__ in,
                                                                    const float *__restrict__ lo, float *out,
                                                                    float *out2, float *out3, int mode, int accum,
                                                                    int slot, const __grid_constant__ LevelF lv)
{
    constexpr int NW = kObjThreads32 / 32, NT = kObjThreads32 * CPB;
    extern __shared__ __align__(16) float smf[];
    __shared__ float2 totA[CPB][NW], totC[CPB][NW];   // warp totals of the two recurrences
    __shared__ long long l_base[CPB], l_pos[CPB];      // first interior node: element, position on the line's axis
    __shared__ int l_m[CPB];
    __shared__ float l_Ad[CPB], l_Bd[CPB];
    const int tid = threadIdx.x;
    const int grp = tid / kObjThreads32, gt = tid % kObjThreads32, warp = gt >> 5, lane = gt & 31;
    const int ij = tid % CPB, ii = tid / CPB;           // interleaved load/store mapping: line, position
    const long long st = ax.stride;
    const float d = ax.d, c = ax.c;
    molt::pdl_enter();
    for (int gb = blockIdx.x * CPB; gb < nlines; gb += gridDim.x * CPB) {
        __syncthreads();
        if (tid < CPB) {
            const int li = gb + tid;
            const bool ok = li < nlines;
            l_m[tid] = ok ? lines[li].m : 0;
            l_base[tid] = ok ? lines[li].base : 0;
            l_pos[tid] = (ok && CPB > 1) ? lines[li].base / st : 0;
        }
        __syncthreads();
        long long p_lo = l_pos[0], p_hi = l_pos[0] + l_m[0] - 1;
#pragma unroll
        for (int j = 1; j < CPB; ++j)
            if (l_m[j] > 0) {
                p_lo = min(p_lo, l_pos[j]);
                p_hi = max(p_hi, l_pos[j] + l_m[j] - 1);
            }
        {
            const int mj = l_m[ij];
            const long long bj = l_base[ij], pj = l_pos[ij];
            float *Hj = smf + (size_t)ij * 4 * slot, *Lj = Hj + slot;
            for (long long r = p_lo + ii; r <= p_hi; r += NT / CPB) {
                const long long k = r - pj + 1;
                if (k >= 1 && k <= mj) {
                    Hj[k] = in[bj + (k - 1) * st];
                    Lj[k] = PAIR ? lo[bj + (k - 1) * st] : 0.f;
                }
            }
            if (ii == 0) { Hj[0] = 0.f; Lj[0] = 0.f; Hj[mj + 1] = 0.f; Lj[mj + 1] = 0.f; }
        }
        __syncthreads();
        // the recurrences of line grp
        const int li = gb + grp;
        const int m = l_m[grp], N = m + 1;
        float *H = smf + (size_t)grp * 4 * slot;
        float *Lo = H + slot;        // lo plane (PAIR)
        float *S = Lo + slot;        // second differences s_t
        float *Q = S + slot;         // q_k, then T_k, then e_k (obj_slot)
        const ObjLineF &ln = lines[li < nlines ? li : 0];
        // second differences s_t, t = 1..m (end triples with their spacings)
        for (int t = 1 + gt; t <= m; t += kObjThreads32) {
            float sv;
            if (t == 1 || t == m) {
                // differences of the pair values, then the end triple's weights
                const float v1h = H[t], v1l = Lo[t];
                const float dn = __fadd_rn(__fsub_rn(H[t + 1], v1h), __fsub_rn(Lo[t + 1], v1l));   // v_{t+1} - v_t
                const float dp = __fadd_rn(__fsub_rn(v1h, H[t - 1]), __fsub_rn(v1l, Lo[t - 1]));   // v_t - v_{t-1}
                if (t == 1) sv = ln.p1 * dn - ln.q1 * dp;
                else sv = ln.pm * dn - ln.qm * dp;
            } else {
                sv = PAIR ? molt::sdiff_pair(H[t - 1], H[t], H[t + 1], Lo[t - 1], Lo[t], Lo[t + 1])
                          : (H[t + 1] - H[t]) - (H[t] - H[t - 1]);
            }
            S[t] = sv;
        }
        __syncthreads();
        for (int k = 1 + gt; k <= m; k += kObjThreads32) {
            float q;
            if (k == 1) q = ln.g11 * S[1] + (m >= 2 ? ln.g12 * S[2] : 0.f);
            else if (k == m) q = ln.gNa * S[m - 1] + ln.gNb * S[m];
            else q = ax.ge * (S[k - 1] + S[k + 1]) + ax.gc * S[k];
            Q[obj_slot(k)] = q;
        }
        if (gt == 0) { Q[0] = 0.f; Q[obj_slot(N)] = 0.f; }
        __syncthreads();
        const int s = (N + kObjThreads32) / kObjThreads32;      // ceil((N + 1) / threads)
        const int k0 = m > 0 ? min(gt * s, N + 1) : 0, k1 = m > 0 ? min(k0 + s, N + 1) : 0;
        // anti-causal: T_k = q_k + g_{k+1} T_{k+1}, T_N = 0 (g_N = dB); a
        // thread's chunk reads and writes only its own entries of Q
        {
            float qq = 0.f;
            for (int k = k1 - 1; k >= k0; --k) {
                const float g = (k == N - 1) ? ln.dB : d;
                qq = (k == N) ? 0.f : g * qq + Q[obj_slot(k)];
            }
            float p = ax.dpow[k1 - k0];
            if (k0 <= N - 1 && N - 1 < k1) p *= ln.rB;
            affine_scan32<false>(p, qq, lane);
            if (lane == 0) totA[grp][warp] = make_float2(p, qq);
            __syncthreads();
            float yin = 0.f;                                     // carry from the warps to the right
            for (int w = NW - 1; w > warp; --w) yin = totA[grp][w].x * yin + totA[grp][w].y;
            const float pn = __shfl_down_sync(0xffffffffu, p, 1), qn = __shfl_down_sync(0xffffffffu, qq, 1);
            float y = (lane == 31) ? yin : pn * yin + qn;
            for (int k = k1 - 1; k >= k0; --k) {
                const float g = (k == N - 1) ? ln.dB : d;
                y = (k == N) ? 0.f : g * y + Q[obj_slot(k)];
                Q[obj_slot(k)] = y;
            }
        }
        // causal: e_k = g_k e_{k-1} + (1 - g_k^2) T_k, e_0 = 0 (g_1 = dA, g_N = dB)
        {
            float qq = 0.f;
            for (int k = k0; k < k1; ++k) {
                const float g = (k == 1) ? ln.dA : (k == N ? ln.dB : d);
                const float cg = (k == 1) ? ln.cA : (k == N ? ln.cB : c);
                qq = (k == 0) ? 0.f : g * qq + cg * Q[obj_slot(k)];
            }
            float p = ax.dpow[k1 - k0];
            if (k0 <= 1 && 1 < k1) p *= ln.rA;
            if (k0 <= N && N < k1) p *= ln.rB;
            affine_scan32<true>(p, qq, lane);
            if (lane == 31) totC[grp][warp] = make_float2(p, qq);
            __syncthreads();
            float yin = 0.f;                                     // carry from the warps to the left
            for (int w = 0; w < warp; ++w) yin = totC[grp][w].x * yin + totC[grp][w].y;
            const float pp = __shfl_up_sync(0xffffffffu, p, 1), qp = __shfl_up_sync(0xffffffffu, qq, 1);
            float y = (lane == 0) ? yin : pp * yin + qp;
            for (int k = k0; k < k1; ++k) {
                const float g = (k == 1) ? ln.dA : (k == N ? ln.dB : d);
                const float cg = (k == 1) ? ln.cA : (k == N ? ln.cB : c);
                y = (k == 0) ? 0.f : g * y + cg * Q[obj_slot(k)];
                Q[obj_slot(k)] = y;
            }
        }
        __syncthreads();
        // e += A' e^{-alpha (x - a)} + B' e^{-alpha (b - x)} with e_0 = e_N = 0
        if (gt == 0 && m > 0) {
            const float Bp = -Q[obj_slot(N)] * ln.inv, Ap = -Bp * ln.mu;
            l_Ad[grp] = Ap * ln.dA;
            l_Bd[grp] = Bp * ln.dB;
        }
        __syncthreads();
        {
            const int mj = l_m[ij];
            const long long bj = l_base[ij], pj = l_pos[ij];
            const float *Hj = smf + (size_t)ij * 4 * slot, *Lj = Hj + slot, *Qj = Hj + 3 * slot;
            const float Ad = l_Ad[ij], Bd = l_Bd[ij];
            for (long long r = p_lo + ii; r <= p_hi; r += NT / CPB) {
                const long long kk = r - pj + 1;
                if (kk >= 1 && kk <= mj) {
                    const int k = (int)kk;
                    const float e = Qj[obj_slot(k)] + Ad * ax.dpow[k - 1] + Bd * ax.dpow[mj - k];
                    const float v = Hj[k] + Lj[k];
                    const long long at = bj + (k - 1) * st;
                    float rr = (mode == OBJF_LINV) ? v - e : e;
                    if (accum) rr = out[at] + rr;
                    if (lv.nh) {
                        obj_level32(lv, at, rr);
                        continue;
                    }
                    out[at] = rr;
                    if (mode == OBJF_BOTH) {
                        out2[at] = v - e;
                        if (out3) out3[at] = e;
                    }
                }
            }
        }
    }
}

// the sweep of axis a, from a pair level or a float32 field
auto sweep32_kernel(bool pair, int a)
{
    return a == 0 ? (pair ? k_obj_sweep32<true, kObjCpb[0]> : k_obj_sweep32<false, kObjCpb[0]>)
                  : (pair ? k_obj_sweep32<true, kObjCpb[1]> : k_obj_sweep32<false, kObjCpb[1]>);
}

// out = sum_t c_t x_t at the interior nodes, row by row (the line objects of
// the contiguous axis): outside the domain every field stays zero.
__global__ void __launch_bounds__(256) k_obj_combine32(CombTermsF t, const ObjLineF *rows, int nrows, float *out)
{
    for (int li = blockIdx.x; li < nrows; li += gridDim.x) {
        const long long base = rows[li].base;
        const int m = rows[li].m;
        for (int k = threadIdx.x; k < m; k += blockDim.x) {
            const long long i = base + k;
            float v = 0.f;
            for (int j = 0; j < t.n; ++j) v += t.c[j] * t.x[j][i];
            out[i] = v;
        }
    }
}

// ---------------------------------------------------------------------------
// host constants
// ---------------------------------------------------------------------------
// int_0^nu t^k e^{-t} dt, k = 0, 1, 2: the power series below 1 (the closed
// forms cancel for short cells), the closed forms above
double exp_moment(int k, double nu)
{
    if (nu < 1.0) {
        double term = std::pow(nu, k + 1), sum = 0.0;   // term = (-1)^i nu^{k+1+i} / i!
        for (int i = 0; i < 60; ++i) {
            const double t = term / (double)(k + 1 + i);
            sum += t;
            if (std::fabs(t) < 1e-18 * std::fabs(sum)) break;
            term *= -nu / (double)(i + 1);
        }
        return sum;
    }
    const double e = std::exp(-nu);
    if (k == 0) return -std::expm1(-nu);
    if (k == 1) return 1.0 - (1.0 + nu) * e;
    return 2.0 - (2.0 + nu * (2.0 + nu)) * e;
}

// w[i] = (alpha/2) int_0^len e^{-alpha s} l_i(s) ds, l_i the Lagrange basis of
// the nodes s_0, s_1, s_2 (s measured from the destination node into the cell).
// With t = alpha s: l_i = (t^2 - alpha (sa + sb) t + alpha^2 sa sb) / (alpha^2
// (s_i - sa)(s_i - sb)) and ds = dt / alpha.
void obj_cell_weights(const double s[3], double len, double alpha, double w[3])
{
    const double nu = alpha * len;
    const double M0 = exp_moment(0, nu), M1 = exp_moment(1, nu), M2 = exp_moment(2, nu);
    for (int i = 0; i < 3; ++i) {
        const double sa = s[(i + 1) % 3], sb = s[(i + 2) % 3];
        const double num = M2 - alpha * (sa + sb) * M1 + alpha * alpha * sa * sb * M0;
        w[i] = num / (2.0 * alpha * alpha * (s[i] - sa) * (s[i] - sb));
    }
}

// H(l) = Q / (2 alpha^2 (1 - e^{-2 alpha l})), Q = t M_1 - M_2 at t = alpha l: what
// the quadratic part of the increments of a cell of length l adds to q
double obj_cell_H(double l, double alpha)
{
    const double t = alpha * l;
    return (t * exp_moment(1, t) - exp_moment(2, t)) / (2.0 * alpha * alpha * -std::expm1(-2.0 * t));
}

// The float64 constants of a line object.  With D_k the second divided
// difference at node k and H as above, inserting the increments (Newton form
// on each cell) into q_k = T_k - g_{k+1} T_{k+1} leaves
//   q_k = D_k (H_k + H_{k+1} - (x_{k+1} - x_{k-1}) / (2 alpha))
//         - g_k H_k D_{k-1} - g_{k+1} H_{k+1} D_{k+1},
// the one-sided interpolants of the end cells putting D_1 for D_0 and D_m for
// D_{m+1}; no term cancels where a gap is small.  Scaled by 1 - d^2 and by
// h^2 = s_k / (2 D_k).
ObjLine make_line(long long base, int m, double h, double ga, double gb, double alpha)
{
    ObjLine L{};
    L.base = base;
    L.m = m;
    const double b = ga + (double)(m - 1) * h + gb, c = -std::expm1(-2.0 * alpha * h);
    const double d = std::exp(-alpha * h), sc = c / (2.0 * h * h);
    L.dA = std::exp(-alpha * ga);
    L.dB = std::exp(-alpha * gb);
    L.lam = -std::expm1(-2.0 * alpha * ga) / c;
    L.mu = std::exp(-alpha * b);
    L.inv = 1.0 / (-std::expm1(-2.0 * alpha * b));
    const double Ha = obj_cell_H(ga, alpha), Hb = obj_cell_H(gb, alpha), H = obj_cell_H(h, alpha);
    const double ca = -std::expm1(-alpha * ga), cb = -std::expm1(-alpha * gb);       // 1 - g of the end cells
    const double nx = m >= 2 ? h : gb, pv = m >= 2 ? h : ga;       // cell after node 1, cell before node m
    const double h2 = 2.0 * h * h;
    L.p1 = h2 / ((ga + nx) * nx);
    L.q1 = h2 / ((ga + nx) * ga);
    L.pm = h2 / ((pv + gb) * gb);
    L.qm = h2 / ((pv + gb) * pv);
    if (m >= 2) {
        L.g11 = sc * (ca * Ha + H - (ga + h) / (2.0 * alpha));
        L.gNb = sc * (cb * Hb + H - (gb + h) / (2.0 * alpha));
        L.g12 = L.gNa = -sc * d * H;
    } else {
        L.g11 = L.gNb = sc * (ca * Ha + cb * Hb - (ga + gb) / (2.0 * alpha));
    }
    return L;
}


// Row k (1 <= k <= N-1) of the difference form as weights on the node
// values v_0..v_N (beta, a dense vector): (v_k - g_k v_{k-1})/(1 - g_k^2) -
// g_{k+1}(v_{k+1} - g_{k+1} v_k)/(1 - g_{k+1}^2) minus the same combination of
// the increments, J^L_k - g_k J^R_{k-1} over (1 - g_k^2), ..., + J^R_k.  x: node
// positions x_0..x_N; the increments use the quadrature rule of the line.
std::vector<double> diff_row(const std::vector<double> &x, int k, double alpha)
{
    const int N = (int)x.size() - 1;
    std::vector<double> b(N + 1, 0.0);
    auto g = [&](int j) { return std::exp(-alpha * (x[j] - x[j - 1])); };   // decay of cell j
    auto add_JL = [&](int j, double c) {   // c J^L_j: cell [x_{j-1}, x_j], destination x_j
        const int c0 = (j + 1 <= N) ? j - 1 : j - 2;
        double ts[3], w[3];
        for (int i = 0; i < 3; ++i) ts[i] = x[j] - x[c0 + i];
        obj_cell_weights(ts, x[j] - x[j - 1], alpha, w);
        for (int i = 0; i < 3; ++i) b[c0 + i] += c * w[i];
    };
    auto add_JR = [&](int j, double c) {   // c J^R_j: cell [x_j, x_{j+1}], destination x_j
        const int c0 = (j - 1 >= 0) ? j - 1 : j;
        double ts[3], w[3];
        for (int i = 0; i < 3; ++i) ts[i] = x[c0 + i] - x[j];
        obj_cell_weights(ts, x[j + 1] - x[j], alpha, w);
        for (int i = 0; i < 3; ++i) b[c0 + i] += c * w[i];
    };
    const double gk = g(k), gk1 = g(k + 1), ik = 1.0 / (1.0 - gk * gk), ik1 = 1.0 / (1.0 - gk1 * gk1);
    b[k] += ik + gk1 * gk1 * ik1;
    b[k - 1] -= gk * ik;
    b[k + 1] -= gk1 * ik1;
    add_JL(k, -ik);
    add_JR(k - 1, gk * ik);
    add_JL(k + 1, gk1 * ik1);
    add_JR(k, -gk1 * gk1 * ik1);
    add_JR(k, -1.0);
    return b;
}

// weight of v_j in the second divided difference over the nodes t-1, t, t+1
double ddiff_w(const std::vector<double> &x, int t, int j)
{
    const double a = x[t - 1], c = x[t], e = x[t + 1];
    if (j == t - 1) return 2.0 / ((a - c) * (a - e));
    if (j == t) return 2.0 / ((c - a) * (c - e));
    return 2.0 / ((e - a) * (e - c));
}

// node positions of a line object (x_0 = a = 0)
std::vector<double> obj_positions(int m, double h, double ga, double gb)
{
    std::vector<double> x(m + 2);
    x[0] = 0.0;
    for (int j = 1; j <= m; ++j) x[j] = ga + (double)(j - 1) * h;
    x[m + 1] = x[m] + gb;
    return x;
}

// The table's d^1 is at least this (alpha h up to 83), so that dA / d times it stays
// dA in float32, whose range both leave at alpha h of 88 and 104 (0 times infinity).
// What crosses a whole cell is then 2^-120 of what enters instead of less.
constexpr double obj_decay_floor32 = 7.52316384526264e-37;       // 2^-120

// the float32 constants of a line object.  The rows 1 and N-1 of the
// difference form are computed in float64 from the increments and written
// as weights on the second divided differences (scaled by h^2): a row
// vanishes on linear data, so node 0 (node N) carries only s_1 (s_m), node
// 3 (node N-3) only s_2 (s_{m-1}).
ObjLineF make_line32(long long base, int m, double h, double ga, double gb, double alpha)
{
    ObjLineF L{};
    L.base = base;
    L.m = m;
    const std::vector<double> x = obj_positions(m, h, ga, gb);
    const int N = m + 1;
    const double b = x[N];
    L.dA = (float)std::exp(-alpha * ga);
    L.dB = (float)std::exp(-alpha * gb);
    const bool fast = std::exp(-alpha * h) < obj_decay_floor32;
    L.rA = (float)(fast ? std::exp(-alpha * ga) / obj_decay_floor32 : std::exp(-alpha * (ga - h)));
    L.rB = (float)(fast ? std::exp(-alpha * gb) / obj_decay_floor32 : std::exp(-alpha * (gb - h)));
    L.cA = (float)(-std::expm1(-2.0 * alpha * ga));
    L.cB = (float)(-std::expm1(-2.0 * alpha * gb));
    L.mu = (float)std::exp(-alpha * b);
    L.inv = (float)(1.0 / (-std::expm1(-2.0 * alpha * b)));
    const double h2 = h * h;
    // s_1 = h^2 divided difference over (x_0, x_1, x_2) = p1 (v_2 - v_1) - q1 (v_1 - v_0)
    L.p1 = (float)(2.0 * h2 / ((x[2] - x[0]) * (x[2] - x[1])));
    L.q1 = (float)(2.0 * h2 / ((x[2] - x[0]) * (x[1] - x[0])));
    L.pm = (float)(2.0 * h2 / ((x[N] - x[m - 1]) * (x[N] - x[m])));
    L.qm = (float)(2.0 * h2 / ((x[N] - x[m - 1]) * (x[m] - x[m - 1])));
    const std::vector<double> b1 = diff_row(x, 1, alpha);
    L.g11 = (float)(b1[0] / ddiff_w(x, 1, 0) / h2);
    L.g12 = m >= 2 ? (float)(b1[3] / ddiff_w(x, 2, 3) / h2) : 0.f;
    const std::vector<double> bm = diff_row(x, m, alpha);
    L.gNb = (float)(bm[N] / ddiff_w(x, m, N) / h2);
    L.gNa = m >= 2 ? (float)(bm[N - 3] / ddiff_w(x, m - 1, N - 3) / h2) : 0.f;
    return L;
}

// the uniform rows: ge s_{k-1} + gc s_k + ge s_{k+1}, from a uniform line
void uniform_rows32(double h, double alpha, float &gc, float &ge)
{
    const int m = 9, k = 5;
    const std::vector<double> x = obj_positions(m, h, h, h);
    const std::vector<double> bk = diff_row(x, k, alpha);
    const double e = bk[k - 2] / ddiff_w(x, k - 1, k - 2);
    const double c = (bk[k - 1] - e * ddiff_w(x, k - 1, k - 1)) / ddiff_w(x, k, k - 1);
    ge = (float)(e / (h * h));
    gc = (float)(c / (h * h));
}

}  // namespace

using namespace molt;

struct mol_embed_ctx {
    int64_t nx = 0, ny = 0, N = 0;
    double hx = 0, hy = 0, alpha = 0, beta = 0;
    int P = 1;
    std::vector<double> tw;             // weights of C^m D^{p-m}: tw[p * 8 + m]
    ObjAxis ax[2]{};                    // x lines (rows), y lines (columns)
    ObjLine *lines[2] = {nullptr, nullptr};
    int nlines[2] = {0, 0};
    double *dpow[2] = {nullptr, nullptr};
    double *V[kMaxP + 1] = {};          // V[1..P]: the Table 3 auxiliaries
    double *tmp = nullptr, *t1 = nullptr, *t2 = nullptr, *t3 = nullptr, *lev = nullptr, *Fb = nullptr;
    double *io[2] = {nullptr, nullptr}; // device copies of mol_embed_solve_host
    std::vector<void *> allocs;
    int seg = 8;                          // float64 sweeps: points per thread
    int sms = 152;
    int slot = 2;                         // float32 sweeps: elements per line array
    int smem32[2] = {0, 0}, grid32[2] = {1, 1};   // float32 sweep launch per axis
    int64_t launches = 0;
    std::string err;
    bool timing = false;                // per-kind CUDA events (0 x sweeps, 1 y sweeps, 2 combinations)
    int prec = 0;                       // MOL_FP64 or MOL_MIXED (float32 sweeps, float32-pair levels)
    ObjAxisF ax32[2]{};
    ObjLineF *lines32[2] = {nullptr, nullptr};
    float *dpow32[2] = {nullptr, nullptr};
    float *V32[kMaxP + 1] = {};
    float *tmp32 = nullptr, *t132 = nullptr, *t232 = nullptr, *t332 = nullptr, *Fb32 = nullptr;
    float *lh[3] = {nullptr, nullptr, nullptr}, *ll[3] = {nullptr, nullptr, nullptr};   // pair levels
    std::vector<cudaEvent_t> ev_pool;
    struct Rec { int kind; cudaEvent_t a, b; };
    std::vector<Rec> recs;
};

namespace {

mol_status efail(mol_embed_ctx *e, mol_status st, const std::string &msg)
{
    if (e) e->err = msg;
    else set_global_error(msg);
    return st;
}

#define ECK(expr, what)                                                                   \
    do {                                                                                  \
        cudaError_t e_ = (expr);                                                          \
        if (e_ != cudaSuccess) return efail(e, MOL_ECUDA, std::string(what) + ": " + cudaGetErrorString(e_)); \
    } while (0)

mol_status ealloc(mol_embed_ctx *e, void **p, size_t bytes)
{
    if (alloc_injected_failure())
        return efail(e, MOL_ENOMEM, "device allocation of " + std::to_string(bytes) + " bytes failed (injected)");
    cudaError_t r = cudaMalloc(p, bytes);
    if (r != cudaSuccess) {
        cudaGetLastError();
        return efail(e, MOL_ENOMEM, "device allocation of " + std::to_string(bytes) + " bytes failed");
    }
    e->allocs.push_back(*p);
    return MOL_OK;
}

void efree_all(mol_embed_ctx *e)
{
    for (auto &r : e->recs) { e->ev_pool.push_back(r.a); e->ev_pool.push_back(r.b); }
    e->recs.clear();
    for (cudaEvent_t v : e->ev_pool) cudaEventDestroy(v);
    e->ev_pool.clear();
    for (void *p : e->allocs) cudaFree(p);
    e->allocs.clear();
}

cudaEvent_t take_event(mol_embed_ctx *e)
{
    if (!e->ev_pool.empty()) {
        cudaEvent_t v = e->ev_pool.back();
        e->ev_pool.pop_back();
        return v;
    }
    cudaEvent_t v = nullptr;
    return cudaEventCreate(&v) == cudaSuccess ? v : nullptr;
}

// events around one launch of the given kind while pass timing is on
struct Timed {
    mol_embed_ctx *e;
    int kind;
    cudaStream_t s;
    cudaEvent_t a = nullptr, b = nullptr;
    Timed(mol_embed_ctx *e_, int k, cudaStream_t s_) : e(e_), kind(k), s(s_)
    {
        if (!e->timing) return;
        a = take_event(e);
        b = take_event(e);
        if (a) cudaEventRecord(a, s);
    }
    ~Timed()
    {
        if (!a || !b) return;
        cudaEventRecord(b, s);
        e->recs.push_back({kind, a, b});
    }
};

// one sweep along axis a (0: the rows, 1: the columns of the field)
mol_status sweep(mol_embed_ctx *e, int a, const double *in, double *out, double *out2, int mode, int accum, cudaStream_t s,
                 double *out3 = nullptr, const CombTerms *cb = nullptr)
{
    if (e->nlines[a] == 0) return MOL_OK;
    const CombTerms none{};
    const ObjAxis &X = e->ax[a];
    const size_t smem = sizeof(double) * 4 * (size_t)X.threads;
    Timed t(e, a, s);
    // a sweep that leaves SMs free lets the next one start while it ends (the
    // next one's threads fetch their tables and wait): 9 launches a step, each
    // as short as its latencies on small grids
    ECK(launch_kernel(e->seg == 4 ? k_obj_sweep<4> : e->seg == 8 ? k_obj_sweep<8> : e->seg == 12 ? k_obj_sweep<12>
                                                                                                  : k_obj_sweep<16>,
                      dim3(X.ctas), dim3(X.threads), smem, s, X.ctas <= e->sms && !e->timing, 1, X,
                      (const ObjLine *)e->lines[a], in, out, out2, out3, mode, accum, cb ? *cb : none),
        "line-object sweep");
    ++e->launches;
    ECK(cudaGetLastError(), "line-object sweep");
    return MOL_OK;
}

// The work table of axis a (k_obj_sweep): m = the interior nodes of its lines.
// Rows one by one, columns in groups of 4 (fewer where a group would not fit a
// CTA), the longest first, each into the first CTA with room for it.
mol_status obj_items(mol_embed_ctx *e, int a, const std::vector<int> &m)
{
    ObjAxis &X = e->ax[a];
    const int R = e->seg, n = (int)m.size();
    auto segs = [&](int l) { return (m[l] + R - 1) / R; };
    int gmax = 1;
    for (int l = 0; l < n; ++l) gmax = std::max(gmax, segs(l));
    const int T = X.threads = gmax <= 128 ? 128 : gmax <= 256 ? 256 : 512;
    const double nu = e->alpha * (a == 0 ? e->hx : e->hy);
    X.win = f64_window(nu, R, gmax);
    struct Group { int line, count, len; };              // len: segments of its longest line
    std::vector<Group> gr;
    for (int l = 0; l < n;) {
        int c = a == 0 ? 1 : std::min(4, n - l), g = 1;
        for (;; c = c > 2 ? 2 : 1) {
            g = 1;
            for (int q = 0; q < c; ++q) g = std::max(g, segs(l + q));
            if (c == 1 || c * g <= T) break;
        }
        gr.push_back({l, c, g});
        l += c;
    }
    std::stable_sort(gr.begin(), gr.end(), [](const Group &x, const Group &y) { return x.count * x.len > y.count * y.len; });
    std::vector<int> used;                               // slots taken, per CTA
    std::vector<int4> items;
    size_t open = 0;                                     // CTAs before it have no room for anything more
    for (const Group &g : gr) {
        const int need = g.count * g.len;
        size_t c = open;
        while (c < used.size() && used[c] + need > T) ++c;
        if (c == used.size()) {
            used.push_back(0);
            items.resize(items.size() + T, int4{-1, 0, 0, 0});
        }
        const int base = used[c];
        for (int k = 0; k < g.len; ++k)
            for (int q = 0; q < g.count; ++q)
                if (k * R < m[g.line + q]) items[c * T + base + k * g.count + q] = int4{g.line + q, k, base + q, g.count};
        used[c] += need;
        while (open < used.size() && used[open] == T) ++open;
    }
    X.ctas = (int)used.size();
    if (items.empty()) return MOL_OK;
    int4 *d = nullptr;
    mol_status st = ealloc(e, (void **)&d, sizeof(int4) * items.size());
    if (st != MOL_OK) return st;
    if (cudaMemcpy(d, items.data(), sizeof(int4) * items.size(), cudaMemcpyHostToDevice) != cudaSuccess)
        return efail(e, MOL_ECUDA, "work table upload");
    X.items = d;
    return MOL_OK;
}

mol_status combine(mol_embed_ctx *e, const CombTerms &t, cudaStream_t s)
{
    if (e->nlines[0] == 0) return MOL_OK;
    Timed tm(e, 2, s);
    k_obj_combine<<<e->nlines[0], 256, 0, s>>>(t, e->lines[0], e->nlines[0]);
    ++e->launches;
    ECK(cudaGetLastError(), "combine");
    return MOL_OK;
}

#define EST(expr)                              \
    do {                                       \
        mol_status st_ = (expr);               \
        if (st_ != MOL_OK) return st_;         \
    } while (0)

// out = C v (eq. C_def_ADI) with L^{-1} = 1 - D: L_y^{-1} D_x v + L_x^{-1} D_y v.  dyv:
// D_y v when an earlier sweep has formed it, else null.  cb: combined instead
// of stored (out then holds L_y^{-1} D_x v only).
mol_status apply_C(mol_embed_ctx *e, const double *v, double *out, cudaStream_t s, const double *dyv = nullptr,
                   const CombTerms *cb = nullptr)
{
    EST(sweep(e, 0, v, e->t1, nullptr, OBJ_D, 0, s));                   // t1 = D_x v
    EST(sweep(e, 1, e->t1, out, nullptr, OBJ_LINV, 0, s));              // out = L_y^{-1} t1
    if (!dyv) {
        EST(sweep(e, 1, v, e->t1, nullptr, OBJ_D, 0, s));               // t1 = D_y v
        dyv = e->t1;
    }
    return sweep(e, 0, dyv, out, nullptr, OBJ_LINV, 1, s, nullptr, cb);   // out += L_x^{-1} D_y v
}

// out = D v (eq. D_def_ADI) = v - L_x^{-1} L_y^{-1} v = D_y v + D_x (L_y^{-1} v); dyv
// receives D_y v as well
mol_status apply_Dadi(mol_embed_ctx *e, const double *v, double *out, cudaStream_t s, double *dyv)
{
    EST(sweep(e, 1, v, out, e->t2, OBJ_BOTH, 0, s, dyv));               // out = D_y v, t2 = L_y^{-1} v
    return sweep(e, 0, e->t2, out, nullptr, OBJ_D, 1, s);               // out += D_x t2
}

// out = ea u + eb up + ec F[u] at the interior nodes (eq. Full_2D, terms in
// Table 3 order: after stage p, V[k] = C^{p-k+1} D^{k-1} u).  The last stage's
// last C is combined with the other terms by its own last sweep.
mol_status run_update(mol_embed_ctx *e, const double *u, const double *up, double *out, double ea, double eb,
                      double ec, cudaStream_t s)
{
    const int P = e->P;
    for (int p = 1; p <= P; ++p) {
        const bool last = p == P;
        // terms of F's sum: those of earlier stages, then c_{p,p-k+1} V[k]
        CombTerms t{};
        t.out = last ? out : e->Fb;
        const double f = last ? ec : 1.0;
        auto add = [&](double c, const double *x) { t.c[t.n] = c; t.x[t.n++] = x; };
        if (last && ea != 0.0) add(ea, u);
        if (last && eb != 0.0) add(eb, up);
        auto weight = [&](int k) { return f * e->tw[p * 8 + (p - k + 1)]; };
        if (p == 1) {
            t.cw = weight(1);
            EST(apply_C(e, u, e->V[1], s, nullptr, last ? &t : nullptr));
            continue;                                   // C u joins stage 2's sum
        }
        if (p > 2) add(f, e->Fb);
        // D_y V_{p-1} serves both D V_{p-1} and C V_{p-1}: formed once
        EST(apply_Dadi(e, e->V[p - 1], e->V[p], s, e->t3));
        add(weight(p), e->V[p]);
        for (int k = 1; k < p; ++k) {
            const bool end = last && k == p - 1;
            if (k == p - 1) {
                // V[1] is still C u here when p = 2; the other stages' C are done
                if (p == 2) add(f * e->tw[1 * 8 + 1], e->V[1]);
                for (int q = 1; q < k; ++q) add(weight(q), e->V[q]);
                t.cw = weight(k);
            }
            EST(apply_C(e, e->V[k], e->tmp, s, k == p - 1 ? e->t3 : nullptr, end ? &t : nullptr));
            if (!end) std::swap(e->V[k], e->tmp);
        }
        if (last) continue;
        // not the last stage: its own sum
        add(t.cw, e->V[p - 1]);
        EST(combine(e, t, s));
    }
    return MOL_OK;
}

// ---- float32 sweeps (MOL_MIXED) ----
// one difference-form sweep along axis a; lo: the lo plane when in is a pair level
mol_status sweep32(mol_embed_ctx *e, int a, const float *in, const float *lo, float *out, float *out2, int mode,
                   int accum, cudaStream_t s, float *out3 = nullptr, const LevelF *lv = nullptr)
{
    if (e->nlines[a] == 0) return MOL_OK;
    const int cpb = kObjCpb[a];
    const int grid = std::min(e->grid32[a], (e->nlines[a] + cpb - 1) / cpb);
    Timed t(e, a, s);
    ECK(launch_kernel(sweep32_kernel(lo != nullptr, a), dim3(grid), dim3(kObjThreads32 * cpb), (size_t)e->smem32[a], s,
                      grid <= e->sms && !e->timing, 1, e->ax32[a], (const ObjLineF *)e->lines32[a], e->nlines[a], in, lo,
                      out, out2, out3, mode, accum, e->slot, lv ? *lv : LevelF{}),
        "line-object sweep (float32)");
    ++e->launches;
    ECK(cudaGetLastError(), "line-object sweep (float32)");
    return MOL_OK;
}

// out = C v (eq. C_def_ADI) with L^{-1} = 1 - D: D_x v - D_y D_x v + D_y v - D_x D_y v.
// dyv: D_y v when an earlier sweep has formed it, else null.  lv: the level
// update that takes C v in its last sweep (out then holds a partial sum).
mol_status apply_C32(mol_embed_ctx *e, const float *v, const float *vlo, float *out, cudaStream_t s,
                     const float *dyv = nullptr, const LevelF *lv = nullptr)
{
    EST(sweep32(e, 0, v, vlo, e->t132, nullptr, OBJF_D, 0, s));               // t1 = D_x v
    EST(sweep32(e, 1, e->t132, nullptr, out, nullptr, OBJF_LINV, 0, s));      // out = L_y^{-1} t1
    if (!dyv) {
        EST(sweep32(e, 1, v, vlo, e->t132, nullptr, OBJF_D, 0, s));           // t1 = D_y v
        dyv = e->t132;
    }
    return sweep32(e, 0, dyv, nullptr, out, nullptr, OBJF_LINV, 1, s, nullptr, lv);   // out += L_x^{-1} D_y v
}

// out = D v (eq. D_def_ADI) = v - L_x^{-1} L_y^{-1} v = D_y v + D_x (L_y^{-1} v); dyv, when
// given, receives D_y v as well
mol_status apply_D32(mol_embed_ctx *e, const float *v, float *out, cudaStream_t s, float *dyv = nullptr)
{
    EST(sweep32(e, 1, v, nullptr, out, e->t232, OBJF_BOTH, 0, s, dyv));       // out = D_y v, t2 = L_y^{-1} v
    return sweep32(e, 0, e->t232, nullptr, out, nullptr, OBJF_D, 1, s);       // out += D_x t2
}

mol_status combine32(mol_embed_ctx *e, const CombTermsF &t, float *out, cudaStream_t s)
{
    if (e->nlines[0] == 0) return MOL_OK;
    Timed tm(e, 2, s);
    k_obj_combine32<<<std::min(e->nlines[0], 8 * e->sms), 256, 0, s>>>(t, e->lines32[0], e->nlines[0], out);
    ++e->launches;
    ECK(cudaGetLastError(), "combine (float32)");
    return MOL_OK;
}

// F[u] of the pair level (uh, ul), Table 3 order as run_update.  With nh
// set: (nh, nl) = ea u + eb up + ec F in pair arithmetic, in F's last sweep;
// else F (float32) into F32.
mol_status run_update32(mol_embed_ctx *e, const float *uh, const float *ul, const float *ph, const float *pl,
                        float *nh, float *nl, float *F32, float ea, float eb, float ec, cudaStream_t s)
{
    const int P = e->P;
    LevelF lv{};
    lv.a = ea; lv.b = eb; lv.c = ec;
    lv.uh = uh; lv.ul = ul; lv.ph = ph; lv.pl = pl;
    lv.nh = nh; lv.nl = nl;
    for (int p = 1; p <= P; ++p) {
        // F's partial sum.  The terms of stage 1 are tw_11 C u alone, and C u
        // is still in tmp32 after stage 2 (whose only C swaps V_1 out), so
        // with P > 1 they join the sum of stage 2 instead of a pass of their own
        const bool fuse = p == P && nh;
        CombTermsF &t = lv.t;
        t.n = 0;
        auto add = [&](double c, const float *x) { t.c[t.n] = (float)c; t.x[t.n++] = x; };
        if (p == 1) {
            add(e->tw[1 * 8 + 1], e->V32[1]);
            lv.own = 0;
            EST(apply_C32(e, uh, ul, e->V32[1], s, nullptr, fuse ? &lv : nullptr));
            if (P > 1) continue;
        } else {
            // D_y V_{p-1} serves both D V_{p-1} and C V_{p-1}: formed once
            EST(apply_D32(e, e->V32[p - 1], e->V32[p], s, e->t332));
            for (int k = 1; k < p; ++k) {
                if (k == p - 1) {
                    // (the last C V_k, of k = p - 1, goes to tmp32: then V_{p-1})
                    if (p == 2) add(e->tw[1 * 8 + 1], e->V32[1]);
                    else add(1.0, e->Fb32);
                    for (int q = 1; q <= p; ++q) {
                        if (q == k) lv.own = t.n;
                        add(e->tw[p * 8 + (p - q + 1)], q == k ? e->tmp32 : e->V32[q]);
                    }
                }
                EST(apply_C32(e, e->V32[k], nullptr, e->tmp32, s, k == p - 1 ? e->t332 : nullptr,
                              fuse && k == p - 1 ? &lv : nullptr));
                std::swap(e->V32[k], e->tmp32);
            }
        }
        if (!fuse) EST(combine32(e, t, p < P ? e->Fb32 : F32, s));
    }
    return MOL_OK;
}

mol_status to_pair(mol_embed_ctx *e, const double *x, int k, cudaStream_t s)
{
    ECK(launch_to_pair(x, e->lh[k], e->ll[k], e->N, s), "level conversion");
    ++e->launches;
    return MOL_OK;
}

mol_status from_pair(mol_embed_ctx *e, int k, double *x, cudaStream_t s)
{
    ECK(launch_from_pair(e->lh[k], e->ll[k], x, e->N, s), "level conversion");
    ++e->launches;
    return MOL_OK;
}

mol_status check_dev(mol_embed_ctx *e, const void *p, const char *name)
{
    if (!p) return efail(e, MOL_EINVAL, std::string(name) + " is NULL");
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return efail(e, MOL_EINVAL, std::string(name) + ": not a CUDA pointer");
    }
    if (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged)
        return efail(e, MOL_EINVAL, std::string(name) + " must be device memory");
    return MOL_OK;
}

}  // namespace

extern "C" {

mol_status mol_embed_create(const mol_embed_geom *g, double c, double dt, double beta, int P, mol_prec prec,
                            mol_embed *out)
{
    if (!out) return efail(nullptr, MOL_EINVAL, "out is NULL");
    *out = nullptr;
    if (!g) return efail(nullptr, MOL_EINVAL, "geometry is NULL");
    if (g->nx < 3 || g->ny < 3 || g->nx > (1 << 15) || g->ny > (1 << 15))
        return efail(nullptr, MOL_EINVAL, "nx and ny must be in 3..32768");
    if (!(g->hx > 0) || !(g->hy > 0) || !std::isfinite(g->hx) || !std::isfinite(g->hy))
        return efail(nullptr, MOL_EINVAL, "hx and hy must be positive");
    if (!g->row_lo || !g->row_hi || !g->row_gap_lo || !g->row_gap_hi || !g->col_lo || !g->col_hi ||
        !g->col_gap_lo || !g->col_gap_hi)
        return efail(nullptr, MOL_EINVAL, "geometry arrays must not be NULL");
    if (P < 1 || P > kMaxP) return efail(nullptr, MOL_EINVAL, "P must be in 1..5");
    if (prec != MOL_FP64 && prec != MOL_MIXED) return efail(nullptr, MOL_EINVAL, "unknown precision");
    if (!(c > 0) || !(dt > 0) || !std::isfinite(c) || !std::isfinite(dt))
        return efail(nullptr, MOL_EINVAL, "c and dt must be positive");
    const double bmax = beta_max_of(P);
    if (beta <= 0) beta = bmax;
    if (beta > bmax * (1.0 + 1e-12))
        return efail(nullptr, MOL_EUNSTABLE, "beta above beta_max(P): the scheme is not A-stable");

    const int64_t nx = g->nx, ny = g->ny;
    // lines, and the agreement of rows and columns on the interior nodes
    std::vector<int> seen((size_t)(nx * ny), 0);
    int64_t maxm = 1;
    for (int a = 0; a < 2; ++a) {
        const int64_t nl = a == 0 ? ny : nx, len = a == 0 ? nx : ny;
        const int64_t *lo = a == 0 ? g->row_lo : g->col_lo, *hi = a == 0 ? g->row_hi : g->col_hi;
        const double *ga = a == 0 ? g->row_gap_lo : g->col_gap_lo, *gb = a == 0 ? g->row_gap_hi : g->col_gap_hi;
        for (int64_t l = 0; l < nl; ++l) {
            if (lo[l] > hi[l]) continue;
            const std::string who = std::string(a == 0 ? "row " : "column ") + std::to_string(l) + ": ";
            if (lo[l] < 0 || hi[l] >= len) return efail(nullptr, MOL_EINVAL, who + "interior nodes outside the grid");
            if (hi[l] - lo[l] + 1 > kObjMaxM)
                return efail(nullptr, MOL_EINVAL, who + "more than " + std::to_string(kObjMaxM) + " interior nodes");
            if (!(ga[l] > 0) || !(gb[l] > 0) || !std::isfinite(ga[l]) || !std::isfinite(gb[l]))
                return efail(nullptr, MOL_EINVAL, who + "gaps must be positive and finite");
            for (int64_t k = lo[l]; k <= hi[l]; ++k) seen[(size_t)(a == 0 ? l * nx + k : k * nx + l)] |= 1 << a;
            maxm = std::max<int64_t>(maxm, hi[l] - lo[l] + 1);
        }
    }
    for (int v : seen)
        if (v == 1 || v == 2)
            return efail(nullptr, MOL_EINVAL, "rows and columns disagree on which nodes are interior");

    mol_embed_ctx *e = new mol_embed_ctx();
    e->nx = nx;
    e->ny = ny;
    e->N = nx * ny;
    e->hx = g->hx;
    e->hy = g->hy;
    e->P = P;
    e->prec = prec;
    e->beta = beta;
    e->alpha = beta / (c * dt);                          // eq. L_def
    e->tw.assign(8 * 8, 0.0);
    for (int p = 1; p <= P; ++p)
        for (int m = 1; m <= p; ++m) e->tw[p * 8 + m] = term_weight(p, m, beta);
    mol_status st = MOL_OK;
    cudaError_t ce;
    std::vector<int> msz[2];                             // interior nodes of the lines
    for (int a = 0; a < 2 && st == MOL_OK; ++a) {
        const double h = a == 0 ? e->hx : e->hy, alpha = e->alpha;
        ObjAxis &X = e->ax[a];
        X.stride = a == 0 ? 1 : nx;
        X.d = std::exp(-alpha * h);
        {
            const double c = -std::expm1(-2.0 * alpha * h), sc = c / (2.0 * h * h), H = obj_cell_H(h, alpha);
            X.gc = sc * (2.0 * H - h / alpha);
            X.ge = -sc * X.d * H;
            f64_inverse_decay(X.d, c, X.e1, X.id);
            X.direct = X.id == 0.0;
            for (int k = 0; k <= kObjR; ++k) X.pw[k] = std::exp(-alpha * h * (double)k);
            for (int k = 1; k <= kObjR; ++k) f64_inflow_weights(alpha * h, k, X.w[k]);
        }
        std::vector<double> tab(kObjMaxM + 1);
        for (int k = 0; k <= kObjMaxM; ++k) tab[k] = std::exp(-alpha * h * (double)k);
        std::vector<ObjLine> ls;
        const int64_t nl = a == 0 ? ny : nx;
        const int64_t *lo = a == 0 ? g->row_lo : g->col_lo, *hi = a == 0 ? g->row_hi : g->col_hi;
        const double *ga = a == 0 ? g->row_gap_lo : g->col_gap_lo, *gb = a == 0 ? g->row_gap_hi : g->col_gap_hi;
        for (int64_t l = 0; l < nl; ++l) {
            if (lo[l] > hi[l]) continue;
            const long long base = a == 0 ? l * nx + lo[l] : lo[l] * nx + l;   // first interior node
            ls.push_back(make_line(base, (int)(hi[l] - lo[l] + 1), h, ga[l], gb[l], alpha));
            msz[a].push_back(ls.back().m);
        }
        e->nlines[a] = (int)ls.size();
        if ((st = ealloc(e, (void **)&e->dpow[a], sizeof(double) * tab.size())) != MOL_OK) break;
        if ((ce = cudaMemcpy(e->dpow[a], tab.data(), sizeof(double) * tab.size(), cudaMemcpyHostToDevice)) != cudaSuccess) {
            st = efail(e, MOL_ECUDA, "table upload");
            break;
        }
        X.dpow = e->dpow[a];
        if (!ls.empty()) {
            if ((st = ealloc(e, (void **)&e->lines[a], sizeof(ObjLine) * ls.size())) != MOL_OK) break;
            if ((ce = cudaMemcpy(e->lines[a], ls.data(), sizeof(ObjLine) * ls.size(), cudaMemcpyHostToDevice)) !=
                cudaSuccess) {
                st = efail(e, MOL_ECUDA, "line table upload");
                break;
            }
        }
        if (prec == MOL_MIXED) {
            // float32 constants of the difference form
            ObjAxisF &Y = e->ax32[a];
            Y.stride = X.stride;
            Y.d = (float)X.d;
            Y.c = (float)(-std::expm1(-2.0 * alpha * h));
            uniform_rows32(h, alpha, Y.gc, Y.ge);
            std::vector<float> tab32(tab.begin(), tab.end());
            tab32[1] = std::max(tab32[1], (float)obj_decay_floor32);
            std::vector<ObjLineF> ls32;
            for (int64_t l = 0; l < nl; ++l) {
                if (lo[l] > hi[l]) continue;
                const long long base = a == 0 ? l * nx + lo[l] : lo[l] * nx + l;
                ls32.push_back(make_line32(base, (int)(hi[l] - lo[l] + 1), h, ga[l], gb[l], alpha));
            }
            if ((st = ealloc(e, (void **)&e->dpow32[a], sizeof(float) * tab32.size())) != MOL_OK) break;
            if ((ce = cudaMemcpy(e->dpow32[a], tab32.data(), sizeof(float) * tab32.size(), cudaMemcpyHostToDevice)) !=
                cudaSuccess) {
                st = efail(e, MOL_ECUDA, "table upload");
                break;
            }
            Y.dpow = e->dpow32[a];
            if (!ls32.empty()) {
                if ((st = ealloc(e, (void **)&e->lines32[a], sizeof(ObjLineF) * ls32.size())) != MOL_OK) break;
                if ((ce = cudaMemcpy(e->lines32[a], ls32.data(), sizeof(ObjLineF) * ls32.size(),
                                     cudaMemcpyHostToDevice)) != cudaSuccess) {
                    st = efail(e, MOL_ECUDA, "line table upload");
                    break;
                }
            }
        }
    }
    // work fields; every sweep writes only interior nodes, so they start at zero
    std::vector<std::pair<void **, size_t>> work;
    const size_t plane = sizeof(double) * (size_t)e->N, plane32 = sizeof(float) * (size_t)e->N;
    if (prec == MOL_FP64) {
        for (double **b : {&e->tmp, &e->t1, &e->t2, &e->t3, &e->lev, &e->Fb}) work.push_back({(void **)b, plane});
        for (int k = 1; k <= P; ++k) work.push_back({(void **)&e->V[k], plane});
    } else {
        for (float **b : {&e->tmp32, &e->t132, &e->t232, &e->t332, &e->Fb32}) work.push_back({(void **)b, plane32});
        for (int k = 1; k <= P; ++k) work.push_back({(void **)&e->V32[k], plane32});
        for (int k = 0; k < 3; ++k) {
            work.push_back({(void **)&e->lh[k], plane32});
            work.push_back({(void **)&e->ll[k], plane32});
        }
    }
    for (auto &w : work) {
        if (st != MOL_OK) break;
        if ((st = ealloc(e, w.first, w.second)) != MOL_OK) break;
        if ((ce = cudaMemset(*w.first, 0, w.second)) != cudaSuccess) st = efail(e, MOL_ECUDA, "memset");
    }
    if (st == MOL_OK) {
        // line arrays sized for the longest line (even, for 16-byte alignment)
        e->slot = (obj_slot((int)maxm + 1) + 2) & ~1;
        // (float32: four arrays per line)
        int dev = 0, sms = 152;
        if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        e->sms = sms;
        if (prec == MOL_FP64) {
            // points per thread: about 12 operations each and 48 of inflow and
            // line ends per thread, whole warps over the SMs' quarters
            int64_t nodes = 0;
            for (int v : msz[0]) nodes += v;
            double best = 0.0;
            for (int R : {4, 8, 12, 16}) {
                if (maxm > (int64_t)R * 512) continue;
                const double w = 1.08 * (double)nodes / (32.0 * R) / (4.0 * sms);
                const double cost = (12.0 * R + 48.0) * (w <= 8.0 ? std::ceil(w) : w + 0.5);
                if (best == 0.0 || cost < best) {
                    best = cost;
                    e->seg = R;
                }
            }
            for (int a = 0; a < 2 && st == MOL_OK; ++a) st = obj_items(e, a, msz[a]);
        } else {
            for (int a = 0; a < 2 && st == MOL_OK; ++a) {
                e->smem32[a] = (int)(sizeof(float) * 4 * (size_t)e->slot * kObjCpb[a]);
                for (int v = 0; v < 2 && st == MOL_OK; ++v)
                    if ((ce = cudaFuncSetAttribute((const void *)sweep32_kernel(v == 0, a),
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   e->smem32[a])) != cudaSuccess)
                        st = efail(e, MOL_ECUDA, std::string("kernel attributes: ") + cudaGetErrorString(ce));
                int ps = 1;
                if (st == MOL_OK &&
                    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, (const void *)sweep32_kernel(true, a),
                                                                  kObjThreads32 * kObjCpb[a], e->smem32[a]) !=
                        cudaSuccess) {
                    cudaGetLastError();
                    ps = 1;
                }
                e->grid32[a] = std::max(1, sms) * std::max(1, ps);
            }
        }
    }
    if (st != MOL_OK) {
        set_global_error(e->err);
        efree_all(e);
        delete e;
        return st;
    }
    *out = e;
    return MOL_OK;
}

mol_status mol_embed_destroy(mol_embed e)
{
    if (!e) return MOL_OK;
    efree_all(e);
    delete e;
    return MOL_OK;
}

const char *mol_embed_last_error(mol_embed e) { return e ? e->err.c_str() : mol_last_error(nullptr); }

mol_status mol_embed_linv(mol_embed e, const double *v, double *w, int axis, void *stream)
{
    if (!e) return efail(nullptr, MOL_EINVAL, "handle is NULL");
    EST(check_dev(e, v, "v"));
    EST(check_dev(e, w, "w"));
    if (axis != 0 && axis != 1) return efail(e, MOL_EINVAL, "axis must be 0 (x) or 1 (y)");
    if (v == w) return efail(e, MOL_EINVAL, "v and w must not overlap");
    cudaStream_t s = (cudaStream_t)stream;
    if (e->prec == MOL_MIXED) {
        EST(to_pair(e, v, 0, s));
        ECK(cudaMemsetAsync(e->t132, 0, sizeof(float) * (size_t)e->N, s), "memset");
        EST(sweep32(e, axis, e->lh[0], e->ll[0], e->t132, nullptr, OBJF_LINV, 0, s));
        ECK(launch_from_f32(e->t132, w, e->N, s), "conversion");
        ++e->launches;
        return MOL_OK;
    }
    ECK(cudaMemsetAsync(w, 0, sizeof(double) * (size_t)e->N, s), "memset");
    return sweep(e, axis, v, w, nullptr, OBJ_LINV, 0, s);
}

mol_status mol_embed_apply_F(mol_embed e, const double *u, double *F, void *stream)
{
    if (!e) return efail(nullptr, MOL_EINVAL, "handle is NULL");
    EST(check_dev(e, u, "u"));
    EST(check_dev(e, F, "F"));
    if (u == F) return efail(e, MOL_EINVAL, "u and F must not overlap");
    cudaStream_t s = (cudaStream_t)stream;
    if (e->prec == MOL_MIXED) {
        EST(to_pair(e, u, 0, s));
        EST(run_update32(e, e->lh[0], e->ll[0], nullptr, nullptr, nullptr, nullptr, e->t232, 0.f, 0.f, 1.f, s));
        ECK(launch_from_f32(e->t232, F, e->N, s), "conversion");
        ++e->launches;
        return MOL_OK;
    }
    ECK(cudaMemsetAsync(F, 0, sizeof(double) * (size_t)e->N, s), "memset");      // (the update writes the interior)
    return run_update(e, u, nullptr, F, 0.0, 0.0, 1.0, s);
}

mol_status mol_embed_start(mol_embed e, const double *u0, double *u1, void *stream)
{
    if (!e) return efail(nullptr, MOL_EINVAL, "handle is NULL");
    EST(check_dev(e, u0, "u0"));
    EST(check_dev(e, u1, "u1"));
    if (u0 == u1) return efail(e, MOL_EINVAL, "u0 and u1 must not overlap");
    cudaStream_t s = (cudaStream_t)stream;
    if (e->prec == MOL_MIXED) {
        EST(to_pair(e, u0, 0, s));
        EST(run_update32(e, e->lh[0], e->ll[0], nullptr, nullptr, e->lh[1], e->ll[1], nullptr, 1.f, 0.f, 0.5f, s));
        return from_pair(e, 1, u1, s);
    }
    ECK(cudaMemsetAsync(u1, 0, sizeof(double) * (size_t)e->N, s), "memset");
    return run_update(e, u0, nullptr, u1, 1.0, 0.0, 0.5, s);
}

mol_status mol_embed_step(mol_embed e, double *u_prev, double *u_cur, int64_t nsteps, void *stream)
{
    if (!e) return efail(nullptr, MOL_EINVAL, "handle is NULL");
    EST(check_dev(e, u_prev, "u_prev"));
    EST(check_dev(e, u_cur, "u_cur"));
    if (u_prev == u_cur) return efail(e, MOL_EINVAL, "u_prev and u_cur must not overlap");
    if (nsteps < 0) return efail(e, MOL_EINVAL, "nsteps must be >= 0");
    cudaStream_t s = (cudaStream_t)stream;
    if (e->prec == MOL_MIXED) {
        if (nsteps == 0) return MOL_OK;
        // the levels as float32 pairs for the whole call (rotating through
        // three internal pair levels), converted back at the end
        EST(to_pair(e, u_prev, 0, s));
        EST(to_pair(e, u_cur, 1, s));
        int r[3] = {0, 1, 2};
        for (int64_t k = 0; k < nsteps; ++k) {
            EST(run_update32(e, e->lh[r[1]], e->ll[r[1]], e->lh[r[0]], e->ll[r[0]], e->lh[r[2]], e->ll[r[2]], nullptr,
                             2.f, -1.f, 1.f, s));
            const int t = r[0];
            r[0] = r[1];
            r[1] = r[2];
            r[2] = t;
        }
        EST(from_pair(e, r[0], u_prev, s));
        return from_pair(e, r[1], u_cur, s);
    }
    double *b[3] = {u_prev, u_cur, e->lev};
    for (int64_t k = 0; k < nsteps; ++k) {
        EST(run_update(e, b[1], b[0], b[2], 2.0, -1.0, 1.0, s));
        double *t = b[0];
        b[0] = b[1];
        b[1] = b[2];
        b[2] = t;
    }
    // the levels back into the caller's buffers: after k steps the roles
    // (previous, current, spare) have rotated k times through (u_prev, u_cur, lev)
    const size_t bytes = sizeof(double) * (size_t)e->N;
    if (b[1] == e->lev) {                 // (u_cur, lev, u_prev)
        ECK(cudaMemcpyAsync(u_prev, u_cur, bytes, cudaMemcpyDeviceToDevice, s), "level copy");
        ECK(cudaMemcpyAsync(u_cur, e->lev, bytes, cudaMemcpyDeviceToDevice, s), "level copy");
    } else if (b[0] == e->lev) {          // (lev, u_prev, u_cur)
        ECK(cudaMemcpyAsync(u_cur, u_prev, bytes, cudaMemcpyDeviceToDevice, s), "level copy");
        ECK(cudaMemcpyAsync(u_prev, e->lev, bytes, cudaMemcpyDeviceToDevice, s), "level copy");
    }
    return MOL_OK;
}

mol_status mol_embed_solve_host(mol_embed e, const double *u0, double *u_out, int64_t nsteps, void *stream)
{
    if (!e) return efail(nullptr, MOL_EINVAL, "handle is NULL");
    if (!u0 || !u_out) return efail(e, MOL_EINVAL, "u0 and u_out must not be NULL");
    if (nsteps < 0) return efail(e, MOL_EINVAL, "nsteps must be >= 0");
    cudaStream_t s = (cudaStream_t)stream;
    const size_t bytes = sizeof(double) * (size_t)e->N;
    for (int k = 0; k < 2; ++k)
        if (!e->io[k]) EST(ealloc(e, (void **)&e->io[k], bytes));
    ECK(cudaMemcpyAsync(e->io[0], u0, bytes, cudaMemcpyHostToDevice, s), "copy in");
    if (nsteps > 0) {
        EST(mol_embed_start(e, e->io[0], e->io[1], stream));
        EST(mol_embed_step(e, e->io[0], e->io[1], nsteps - 1, stream));
        ECK(cudaMemcpyAsync(u_out, e->io[1], bytes, cudaMemcpyDeviceToHost, s), "copy out");
    } else {
        ECK(cudaMemcpyAsync(u_out, e->io[0], bytes, cudaMemcpyDeviceToHost, s), "copy out");
    }
    ECK(cudaStreamSynchronize(s), "synchronize");
    return MOL_OK;
}

mol_status mol_embed_sync(mol_embed e, void *stream)
{
    if (!e) return efail(nullptr, MOL_EINVAL, "handle is NULL");
    ECK(cudaStreamSynchronize((cudaStream_t)stream), "synchronize");
    return MOL_OK;
}

int64_t mol_embed_launch_count(mol_embed e) { return e ? e->launches : 0; }

mol_status mol_embed_set_pass_timing(mol_embed e, int enable)
{
    if (!e) return efail(nullptr, MOL_EINVAL, "handle is NULL");
    e->timing = enable != 0;
    return MOL_OK;
}

mol_status mol_embed_pass_times(mol_embed e, double total_ms[3], int64_t launches[3])
{
    if (!e) return efail(nullptr, MOL_EINVAL, "handle is NULL");
    if (!total_ms || !launches) return efail(e, MOL_EINVAL, "output arrays must not be NULL");
    for (int k = 0; k < 3; ++k) { total_ms[k] = 0.0; launches[k] = 0; }
    for (auto &r : e->recs) {
        float ms = 0.f;
        cudaError_t ce = cudaEventSynchronize(r.b);
        if (ce == cudaSuccess) ce = cudaEventElapsedTime(&ms, r.a, r.b);
        if (ce != cudaSuccess) return efail(e, MOL_ECUDA, std::string("pass timing: ") + cudaGetErrorString(ce));
        total_ms[r.kind] += ms;
        launches[r.kind] += 1;
        e->ev_pool.push_back(r.a);
        e->ev_pool.push_back(r.b);
    }
    e->recs.clear();
    return MOL_OK;
}

}  // extern "C"

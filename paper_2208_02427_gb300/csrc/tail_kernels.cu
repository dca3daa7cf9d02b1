// tail_kernels.cu -- the small levels of a V-cycle in shared memory, on one CTA or a cluster.
//
// Below some size a level's launches cost more than its work. This kernel runs the V-cycle from
// level `first` of one problem down to its coarsest level and back with every level's u and q in
// shared memory: one CTA, with a CTA barrier between phases, or a thread-block cluster that splits
// the larger levels by rows. In a cluster each CTA owns a block of rows of every split level and
// keeps a copy of the row on either side; whoever updates a border row stores it in the
// neighbour's copy as well (distributed shared memory), so that all reads but those of one
// residual row are local, and a cluster barrier (about 450 cycles, measured) stands where the
// launches were. Levels too small for that run on the first CTA alone.
//
// What bounds it: in FP64 the pipe of the SMs it runs on (about 18 operations a point and cycle at
// 2 per clock and SM), in FP32 the phases' latency. The per-point arithmetic is that of the other
// kernels, so the tail changes the launch structure and nothing else.
//
// Layout: a row keeps its even columns in one half and its odd ones in the other (hs elements
// each), so a colour's points in a row are contiguous (no bank conflicts). A thread keeps its place
// c in the half rows of a level and steps over rows, so that a phase is little more than its loads,
// its arithmetic and a barrier: with the mapping worked out anew in every phase, or four points a
// thread, a phase of a 17 x 17 level took 900 cycles.
//
// Work left out because its result is known or never read:
//  - the first red pass of a level that starts from zero needs no neighbours and is done by the
//    restriction that makes its source;
//  - with Gauss-Seidel the red points' values before a sweep are never read, so only the black
//    points are interpolated;
//  - with Gauss-Seidel and 1/d = 2^-k (FP64) a black point's residual after its update is exactly 0:
//    psi = s 2^-k is exact unless it underflows, and r = fma(-d, psi, s). Points whose value is zero,
//    subnormal or not finite are computed.
#include <cooperative_groups.h>

#include <algorithm>

#include "vcycle_arith.cuh"

namespace lap {

namespace {

namespace cg = cooperative_groups;

constexpr int TAIL_LEVELS = 30;
constexpr int SMEM_TAIL_LOG = 9;
static_assert(SMEM_TAIL_THREADS == 1 << SMEM_TAIL_LOG, "the threads are a power of two");
constexpr int TAIL_HEAD = 1024;  // bytes of shared memory before the arrays: the levels' geometry
constexpr int TAIL_STAGED = 32;  // coarsest unknowns up to which the inverse is staged (8 KB)

// One level in a CTA's shared memory. Rows b0 - 1 .. b0 + rows are held, in slots 0 .. rows + 1.
struct TailLevel {
    int m, n, hs;    // points, elements per half row
    int b0, b1;      // the rows this CTA owns
    int u, q;        // element offsets of slot 0
    int gl;          // log2 of the threads side by side on a half row
};

static_assert(TAIL_LEVELS * sizeof(TailLevel) <= TAIL_HEAD, "the geometry fits its place");

__host__ __device__ inline int tail_half(int m) { return ((m + 1) / 2 + 1) & ~1; }
// Rows per CTA of a split level (all but the last CTA, which also has the ring row).
__host__ __device__ inline int tail_rows(int n, int nc, int ncl)
{
    const int quantum = 1 << ncl, blocks = (n - 1 + quantum - 1) / quantum;
    return quantum * ((blocks + nc - 1) / nc);
}
// Slots of level l: a split level's rows (and the ring row) with a row on either side, else all rows.
__host__ __device__ inline int tail_slots(int n, int l, int nc, int ncl, int rows0)
{
    return (nc > 1 && l < ncl ? (rows0 >> l) + 1 : n) + 2;
}

__device__ __forceinline__ int log2_up(int v) { return v <= 1 ? 0 : 32 - __clz(v - 1); }

// What the phases share. sm: this CTA's arrays; lo, hi: the same arrays of the CTAs below and above
// (null without one), root: of the cluster's first CTA.
template <class T>
struct Tail {
    T *sm, *lo, *hi, *root;
    int rank, rows0;
    Arith<T> A;
    T b2, d, inv_d, w, omw;
    int shift;  // 1/d = 2^-shift (POW2)

    // s / d. (In FP32 the factor is converted once: a conversion from FP64 in every phase costs the
    // FP64 pipe 64 cycles a warp.)
    template <bool POW2>
    __device__ __forceinline__ T over_d(T s) const
    {
        if constexpr (sizeof(T) == 4) return __fmul_rn(s, inv_d);
        else return times_inv_d<POW2>(A.o, s, inv_d, shift);
    }

    // Row slot of row j (u or q array at offset off) of level g, for j within a row of the own ones.
    __device__ __forceinline__ T* row(const TailLevel& g, int off, int j) const
    {
        return sm + off + (j - g.b0 + 1) * 2 * g.hs;
    }
    // Stores v, an element of row j of u (in_row: its place in the row), and in the neighbours' copies
    // of a border row.
    template <bool CL>
    __device__ __forceinline__ void put(const TailLevel& g, int l, int j, T* at, int in_row, T v) const
    {
        *at = v;
        if (CL) {
            if (lo && j == g.b0) lo[g.u + ((rows0 >> l) + 1) * 2 * g.hs + in_row] = v;
            if (hi && j == g.b1 - 1) hi[g.u + in_row] = v;
        }
    }
};

// This thread's points of one colour (0, 1: points with (i + j) % 2 == colour) of a level: one place c
// of a half row, in rows j, j + step, ... (n of them). The threads side by side on a half row are a
// power of two, at most half the CTA, so step is even and every row has the same half.
struct Walk {
    int at;    // offset of the first one from row b0 - 1
    int oth;   // from a point to its west neighbour (the east one is next to it)
    int n, j, c, odd;
};
struct Place {
    Walk w[2];
    int stride, step;  // offsets and rows between a thread's points
};
__device__ __forceinline__ Place place(const TailLevel& g)
{
    Place p;
    const int c = threadIdx.x & ((1 << g.gl) - 1), rs = 2 * g.hs;
    const int jl = max(1, g.b0), jh = min(g.n - 2, g.b1 - 1), j = jl + (threadIdx.x >> g.gl);
    p.step = SMEM_TAIL_THREADS >> g.gl;
    p.stride = p.step * rs;
    const int rows = j <= jh ? ((jh - j) >> (SMEM_TAIL_LOG - g.gl)) + 1 : 0;
#pragma unroll
    for (int colour = 0; colour < 2; ++colour) {
        Walk& w = p.w[colour];
        w.odd = (j + colour) & 1;
        w.c = c;
        w.j = j;
        w.at = (j - g.b0 + 1) * rs + (w.odd ? g.hs : 0) + c;
        w.oth = (w.odd ? -g.hs : g.hs) - 1 + w.odd;
        w.n = c + w.odd >= 1 && 2 * c + w.odd <= g.m - 2 ? rows : 0;
    }
    return p;
}

// One colour pass of Eq. 6 (GS) or Eq. 7. BATCH points' operands are loaded before the first is
// stored (a colour's points do not read one another).
template <class T, bool CL, bool UNIT, bool POW2, bool GS, bool HQ>
__device__ __forceinline__ void tail_pass(const Tail<T>& t, const TailLevel& g, const Place& p, const Walk& w, int l)
{
    constexpr int BATCH = sizeof(T) == 4 ? 4 : 2;
    const int rs = 2 * g.hs, in_row = (w.odd ? g.hs : 0) + w.c;
    T* u = t.sm + g.u + w.at;
    const T* q = t.sm + g.q + w.at;
    auto value = [&](const T* c, const T* qc) {
        T s = t.A.template nsum<UNIT>(c[w.oth], c[w.oth + 1], c[-rs], c[rs], t.b2);
        if (HQ) s = t.A.add(s, *qc);
        s = t.template over_d<POW2>(s);
        return GS ? s : t.A.fma(t.w, s, t.A.mul(t.omw, c[0]));
    };
    int k = 0, j = w.j;
#pragma unroll 1
    for (; k + BATCH <= w.n; k += BATCH) {
        T x[BATCH];
#pragma unroll
        for (int b = 0; b < BATCH; ++b) x[b] = value(u + b * p.stride, q + b * p.stride);
#pragma unroll
        for (int b = 0; b < BATCH; ++b) t.template put<CL>(g, l, j + b * p.step, u + b * p.stride, in_row, x[b]);
        u += BATCH * p.stride;
        q += BATCH * p.stride;
        j += BATCH * p.step;
    }
#pragma unroll 1
    for (; k < w.n; ++k) {
        t.template put<CL>(g, l, j, u, in_row, value(u, q));
        u += p.stride;
        q += p.stride;
        j += p.step;
    }
}

// Takes the restricted residual v of coarse point (I, J): C.q, and the first red pass there (the
// correction starts at zero: s = 0 + q) for a red point. dst: the arrays that hold the coarse level,
// cb0 the row of their slot 1. first: there is a red pass to do.
template <class T, bool CL, bool POW2, bool GS>
__device__ __forceinline__ void coarse_put(const Tail<T>& t, const TailLevel& C, int lc, T* dst, int cb0, bool away,
                                           bool first, int I, int J, T v)
{
    const int in_row = (I & 1) * C.hs + (I >> 1), at = (J - cb0 + 1) * 2 * C.hs + in_row;
    dst[C.q + at] = v;
    if (first && ((I + J) & 1) == 0) {
        T x = t.template over_d<POW2>(t.A.add((T)0, v));
        if (!GS) x = t.A.fma(t.w, x, t.A.mul(t.omw, (T)0));
        if (CL && !away) t.template put<true>(C, lc, J, dst + C.u + at, in_row, x);
        else dst[C.u + at] = x;
    }
}

// The residual's stencil at an element of u (oth: to its west neighbour), and the full-weighting
// edges, out of line for the points whose black residual is not known to be zero: inline, the
// compiler evaluates them for every point and selects.
template <bool UNIT, bool HQ>
__device__ __noinline__ double black_residual(Arith<double> A, const double* c, int oth, const double* s, const double* n,
                                              const double* q, double b2, double d)
{
    double x = A.template nsum<UNIT>(c[oth], c[oth + 1], *s, *n, b2);
    if (HQ) x = A.add(x, *q);
    return A.fma(-d, *c, x);
}
__device__ __noinline__ double edge_sum(Arith<double> A, double w, double e, double s, double n)
{
    return A.add(A.add(w, e), A.add(s, n));
}

// The residual of the CTA's interior rows, and of the row below them where it is another CTA's, to
// the scratch array r. BZ: the black residuals are zero where the value is regular.
template <class T, bool CL, bool UNIT, bool HQ, bool BZ>
__device__ __forceinline__ void tail_residual(const Tail<T>& t, const TailLevel& g, const Place& p, int l, T* r)
{
    const int rs = 2 * g.hs;
    const T *u0 = t.sm + g.u, *q0 = t.sm + g.q;
#pragma unroll
    for (int colour = 0; colour < 2; ++colour) {
        const Walk w = p.w[colour];
#pragma unroll 1
        for (int k = 0, at = w.at; k < w.n; ++k, at += p.stride) {
            const T* c = u0 + at;
            if constexpr (BZ) {
                if (colour == 1) {
                    T v = (T)0;
                    if (irregular(*c)) v = black_residual<UNIT, HQ>(t.A, c, w.oth, c - rs, c + rs, q0 + at, t.b2, t.d);
                    r[at] = v;
                    continue;
                }
            }
            T x = t.A.template nsum<UNIT>(c[w.oth], c[w.oth + 1], c[-rs], c[rs], t.b2);
            if (HQ) x = t.A.add(x, q0[at]);
            r[at] = t.A.fma(-t.d, *c, x);
        }
    }
    if (CL && t.lo) {  // row b0 - 1 (odd): its u is in the copy, the row below it and its q in the CTA below
        const T* below = t.lo + g.u + ((t.rows0 >> l) - 1) * rs;  // row b0 - 2
        const T* ql = t.lo + g.q + (t.rows0 >> l) * rs;           // row b0 - 1
        for (int k = threadIdx.x; k < 2 * (g.m / 2); k += blockDim.x) {
            const int odd = k & 1, c = k >> 1, i = 2 * c + odd, at = (odd ? g.hs : 0) + c;
            if (i < 1 || i > g.m - 2) continue;
            const int oth = (odd ? -g.hs : g.hs) - 1 + odd;
            const T* v = u0 + at;
            if constexpr (BZ) {
                if (odd == 0) {
                    T z = (T)0;
                    if (irregular(*v)) z = black_residual<UNIT, HQ>(t.A, v, oth, below + at, v + rs, ql + at, t.b2, t.d);
                    r[at] = z;
                    continue;
                }
            }
            T x = t.A.template nsum<UNIT>(v[oth], v[oth + 1], below[at], v[rs], t.b2);
            if (HQ) x = t.A.add(x, ql[at]);
            r[at] = t.A.fma(-t.d, *v, x);
        }
    }
}

// C.q = 0.25 ((4 r + 2 edges) + corners) at the coarse rows J with 2 J among the CTA's rows.
template <class T, bool CL, bool POW2, bool GS, bool BZ>
__device__ __forceinline__ void tail_restrict(const Tail<T>& t, const TailLevel& g, const TailLevel& C, int l,
                                              const T* r, T* dst, int cb0, bool away, bool first)
{
    const int rs = 2 * g.hs, Ja = max(1, (g.b0 + 1) >> 1), Jb = min(C.n - 2, (g.b1 - 1) >> 1);
    const T two = t.A.two();
    // coarse column I at the fine level's half-row place I
    const int I = threadIdx.x & ((1 << g.gl) - 1), step = SMEM_TAIL_THREADS >> g.gl;
    if (I < 1 || I > C.m - 2) return;
#pragma unroll 1
    for (int J = Ja + (threadIdx.x >> g.gl); J <= Jb; J += step) {
        const T* c = r + (2 * J - g.b0 + 1) * rs + I;
        const T* o = c + g.hs - 1;  // the odd columns left and right
        T edges = (T)0;
        const T W = o[0], E = o[1], S = c[-rs], N = c[rs];
        if constexpr (BZ) {
            if (!(W == 0.0 && E == 0.0 && S == 0.0 && N == 0.0)) edges = edge_sum(t.A, W, E, S, N);
        } else {
            edges = t.A.add(t.A.add(W, E), t.A.add(S, N));
        }
        const T corners = t.A.add(t.A.add(o[-rs], o[-rs + 1]), t.A.add(o[rs], o[rs + 1]));
        coarse_put<T, CL, POW2, GS>(t, C, l + 1, dst, cb0, away, first, I, J,
                                    t.A.quarter(t.A.fma(two, t.A.fma(two, c[0], edges), corners)));
    }
}

// u += bilinear interpolation of the coarse correction (src: the arrays that hold it, cb0: the row
// of their slot 1) on the CTA's interior rows; black points only, or both colours.
template <class T, bool CL, bool GSONLY>
__device__ __forceinline__ void tail_prolong(const Tail<T>& t, const TailLevel& g, const TailLevel& C, const Place& p,
                                             int l, const T* src, int cb0)
{
#pragma unroll
    for (int colour = GSONLY ? 1 : 0; colour < 2; ++colour) {
        const Walk w = p.w[colour];
        // coarse columns c and c + 1 of rows j / 2 and j / 2 + 1
        const int i0 = (w.c & 1) * C.hs + (w.c >> 1), i1 = ((w.c + 1) & 1) * C.hs + ((w.c + 1) >> 1), up = 2 * C.hs;
        const T* a = src + C.u + ((w.j >> 1) - cb0 + 1) * up;
        T* u = t.sm + g.u + w.at;
#pragma unroll 1
        for (int k = 0; k < w.n; ++k, u += p.stride, a += (p.step >> 1) * up) {
            T e;
            if (GSONLY) e = t.A.half(t.A.add(a[i0], a[w.odd ? i1 : up + i0]));  // black: odd on even rows, even on odd ones
            else if ((w.j & 1) == 0) e = w.odd ? t.A.half(t.A.add(a[i0], a[i1])) : a[i0];
            else
                e = w.odd ? t.A.quarter(t.A.add(t.A.add(a[i0], a[i1]), t.A.add(a[up + i0], a[up + i1])))
                          : t.A.half(t.A.add(a[i0], a[up + i0]));
            t.template put<CL>(g, l, w.j + k * p.step, u, (w.odd ? g.hs : 0) + w.c, t.A.add(*u, e));
        }
    }
}

// The coarsest level: u = A^-1 b, b = q + ring terms in FP64 (the expressions of coarse_cta; a
// correction's ring is zero and adds nothing). ainv: the transposed inverse. Up to 32 unknowns are
// one warp's: lane k holds b_k and the rows' products meet by shuffle; ainv is in shared memory then
// (from global memory its loads are a chain).
template <class T>
__device__ __forceinline__ void tail_coarse(const Tail<T>& t, const TailLevel& g, bool hasq, bool ring, double b2,
                                            const double* ainv, double* b)
{
    const int mi = g.m - 2, N = mi * (g.n - 2), rs = 2 * g.hs;
    auto at = [&](int off, int i, int j) -> T& { return t.sm[off + (j - g.b0 + 1) * rs + (i & 1) * g.hs + (i >> 1)]; };
    auto rhs = [&](int i, int j) {
        double v = hasq ? (double)at(g.q, i, j) : 0.0;
        if (!ring) return v;
        if (i == 1) v = __dadd_rn(v, (double)at(g.u, i - 1, j));
        if (i == g.m - 2) v = __dadd_rn(v, (double)at(g.u, i + 1, j));
        if (j == 1) v = __fma_rn(b2, (double)at(g.u, i, j - 1), v);
        if (j == g.n - 2) v = __fma_rn(b2, (double)at(g.u, i, j + 1), v);
        return v;
    };
    if (N <= TAIL_STAGED) {
        if (threadIdx.x >= 32) return;
        const int k = min((int)threadIdx.x, N - 1), j0 = k / mi, i = 1 + k - j0 * mi, j = 1 + j0;
        const double v = rhs(i, j);
        double x = 0.0;
#pragma unroll 4
        for (int l = 0; l < N; ++l) x = __fma_rn(ainv[l * N + k], __shfl_sync(0xffffffffu, v, l), x);
        if (threadIdx.x < N) at(g.u, i, j) = (T)x;
        return;
    }
    for (int k = threadIdx.x; k < N; k += blockDim.x) b[k] = rhs(1 + k % mi, 1 + k / mi);
    __syncthreads();
#pragma unroll 1
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        double x = 0.0;
#pragma unroll 4
        for (int l = 0; l < N; ++l) x = __fma_rn(ainv[(int64_t)l * N + k], b[l], x);
        at(g.u, 1 + k % mi, 1 + k / mi) = (T)x;
    }
}

// The V-cycle of one job, nc CTAs splitting its first ncl levels. One function per combination of
// flags, out of line: inlined side by side, their loop invariants were all kept in registers at once
// and spilled. The dynamic shared memory holds the levels' geometry, then the arrays.
template <class T, bool CL, bool UNIT, bool POW2, bool GS>
__device__ __noinline__ void tail_cycle(TailJob jb, const BatchLevel<T>* __restrict__ lv, int nu1, int nu2, T w,
                                        T omw, int nc, int ncl)
{
    extern __shared__ uint4 smem4[];
    TailLevel* const G = reinterpret_cast<TailLevel*>(smem4);
    T* const smem = reinterpret_cast<T*>(smem4 + TAIL_HEAD / 16);
    const int nl = jb.last - jb.first + 1;
    const BatchLevel<T> F = lv[jb.first];
    Tail<T> t;
    t.A = arith<T>();
    t.rank = CL ? (int)cg::this_cluster().block_rank() : 0;
    t.rows0 = CL ? tail_rows(F.n, nc, ncl) : 0;
    t.sm = smem;
    t.shift = F.inv_d_shift;
    if constexpr (sizeof(T) == 8) {
        t.b2 = in_reg(t.A.o, (T)F.b2);
        t.d = in_reg(t.A.o, (T)F.d);
        t.w = in_reg(t.A.o, w);
        t.omw = in_reg(t.A.o, omw);
        t.inv_d = in_reg(t.A.o, (T)F.inv_d);
    } else {
        t.b2 = (T)F.b2;
        t.d = (T)F.d;
        t.inv_d = (T)F.inv_d;
        t.w = w;
        t.omw = omw;
    }
    // geometry, one thread per level
    if (threadIdx.x < nl) {
        int m = F.m, n = F.n, at = 0;
        TailLevel g{};
        for (int l = 0; l <= (int)threadIdx.x; ++l) {
            const int hs = tail_half(m), size = tail_slots(n, l, nc, ncl, t.rows0) * 2 * hs;
            const bool split = CL && l < ncl;
            g.m = m;
            g.n = n;
            g.hs = hs;
            if (split) {
                const int r = t.rows0 >> l;
                g.b0 = min(t.rank * r, n);
                g.b1 = (t.rank + 1) * r >= n - 1 ? n : (t.rank + 1) * r;
                if (t.rank * r >= n - 1) g.b0 = g.b1 = n;  // nothing left for this CTA
            } else {
                g.b0 = 0;
                g.b1 = n;
            }
            g.gl = min(8, log2_up(m / 2));
            g.u = at;
            g.q = at + size;
            at += 2 * size;
            m = (m - 1) / 2 + 1;
            n = (n - 1) / 2 + 1;
        }
        G[threadIdx.x] = g;
    }
    __syncthreads();
    const TailLevel g0 = G[0];
    const int slots0 = tail_slots(F.n, 0, nc, ncl, t.rows0), first_elems = 2 * slots0 * 2 * g0.hs;
    const TailLevel gl = G[nl - 1];
    const int all = gl.q + tail_slots(gl.n, nl - 1, nc, ncl, t.rows0) * 2 * gl.hs;
    // behind the levels: the residual (as large as the largest u held here: in a cluster a level
    // of the first CTA alone may be larger than its rows of a split one), then the coarsest level's
    // right-hand side
    T* const r = t.sm + all;
    int r_elems = 0;
    for (int l = 0; l < nl; ++l) r_elems = max(r_elems, G[l].q - G[l].u);
    double* const b = reinterpret_cast<double*>(r + r_elems);
    const int N = (gl.m - 2) * (gl.n - 2);
    const double* ainv = lv[jb.last].ainv_t;
    if (N <= TAIL_STAGED) {  // behind b
        for (int k = threadIdx.x; k < N * N; k += blockDim.x) b[N + k] = ainv[k];
        ainv = b + N;
    }
    t.lo = t.hi = nullptr;
    t.root = t.sm;
    if (CL) {
        cg::cluster_group cl = cg::this_cluster();
        t.root = cl.map_shared_rank(t.sm, 0);
        if (t.rank > 0 && g0.b0 < g0.b1) t.lo = cl.map_shared_rank(t.sm, t.rank - 1);
        if (t.rank + 1 < nc && g0.b1 < g0.n) t.hi = cl.map_shared_rank(t.sm, t.rank + 1);
    }
    // the first level's rows with the copies around them, the others zero
    {
        const int r0 = max(0, g0.b0 - 1), r1 = min(F.n - 1, g0.b1), rows = g0.b0 < g0.b1 ? r1 - r0 + 1 : 0;
        for (int r = threadIdx.x >> 5; r < rows; r += blockDim.x >> 5) {
            const int j = r0 + r;
            const T* gu = F.u + (int64_t)j * F.pitch;
            const T* gq = F.q ? F.q + (int64_t)j * F.pitch : nullptr;
            T *su = t.row(g0, g0.u, j), *sq = t.row(g0, g0.q, j);
            for (int i = threadIdx.x & 31; i < F.m; i += 32) {
                const int at = (i & 1) * g0.hs + (i >> 1);
                su[at] = gu[i];
                if (gq) sq[at] = gq[i];
            }
        }
        for (int k = first_elems + threadIdx.x; k < all; k += blockDim.x) t.sm[k] = (T)0;
    }
    auto barrier = [&](int l) {
        if (CL && l < ncl) cg::this_cluster().sync();
        else __syncthreads();
    };
    barrier(0);
    auto mine = [&](int l) { return !CL || l < ncl || t.rank == 0; };
    // the sweeps of level l, the first red pass left out when `red_done`
    auto smooth = [&](const TailLevel& g, const Place& p, int l, int sweeps, bool red_done) {
        on_flag(l > 0 || F.q, [&](auto HQ) {
#pragma unroll 1
            for (int k = 0; k < sweeps; ++k) {
                if (k > 0 || !red_done) {
                    tail_pass<T, CL, UNIT, POW2, GS, HQ.value>(t, g, p, p.w[0], l);
                    barrier(l);
                }
                tail_pass<T, CL, UNIT, POW2, GS, HQ.value>(t, g, p, p.w[1], l);
                barrier(l);
            }
        });
    };
    auto restrict = [&](auto HQ, const TailLevel& g, const Place& p, int l, T* dst,
                        int cb0, bool away, bool first) {
        constexpr bool BZ = sizeof(T) == 8 && POW2 && GS;
        const TailLevel C = G[l + 1];
        on_flag(BZ && nu1 > 0, [&](auto Z) {
            tail_residual<T, CL, UNIT, HQ.value, BZ && Z.value>(t, g, p, l, r);
            __syncthreads();
            tail_restrict<T, CL, POW2, GS, BZ && Z.value>(t, g, C, l, r, dst, cb0, away, first);
        });
        barrier(l);
    };
#pragma unroll 1
    for (int l = 0; l < nl - 1; ++l) {
        if (!mine(l)) break;
        const TailLevel g = G[l];
        const Place p = place(g);
        smooth(g, p, l, nu1, l > 0);
        const bool away = CL && l == ncl - 1;  // the coarse level is the first CTA's alone
        T* dst = away ? t.root : t.sm;
        const int cb0 = away ? 0 : G[l + 1].b0;
        const bool first = nu1 > 0 && l + 1 < nl - 1;
        if (l == 0 && !F.q) restrict(std::false_type{}, g, p, l, dst, cb0, away, first);
        else restrict(std::true_type{}, g, p, l, dst, cb0, away, first);
    }
    if (mine(nl - 1)) {
        tail_coarse(t, G[nl - 1], nl > 1 || F.q, nl == 1, F.b2, ainv, b);
        __syncthreads();
    }
#pragma unroll 1
    for (int l = nl - 2; l >= 0; --l) {
        if (CL && l == ncl - 1) cg::this_cluster().sync();  // the first CTA has the levels below ready
        if (!mine(l)) continue;
        const bool away = CL && l == ncl - 1;
        const T* src = away ? t.root : t.sm;
        const int cb0 = away ? 0 : G[l + 1].b0;
        const TailLevel g = G[l];
        const Place p = place(g);
        if (GS && nu2 > 0) tail_prolong<T, CL, true>(t, g, G[l + 1], p, l, src, cb0);
        else tail_prolong<T, CL, false>(t, g, G[l + 1], p, l, src, cb0);
        barrier(l);
        smooth(g, p, l, nu2, false);
    }
    // interior rows of the first level back to memory
    for (int j = max(1, g0.b0) + (threadIdx.x >> 5); j <= min(F.n - 2, g0.b1 - 1); j += blockDim.x >> 5) {
        T* gu = F.u + (int64_t)j * F.pitch;
        const T* su = t.row(g0, g0.u, j);
        for (int i = 1 + (threadIdx.x & 31); i <= F.m - 2; i += 32) gu[i] = su[(i & 1) * g0.hs + (i >> 1)];
    }
    if (CL) cg::this_cluster().sync();  // no CTA leaves while another may still read its memory
}

template <class T, bool CL>
__device__ __forceinline__ void tail_dispatch(const TailJob& jb, const BatchLevel<T>* __restrict__ lv, int nu1, int nu2,
                                              bool gs, T w, T omw, int nc, int ncl)
{
    const bool unit = lv[jb.first].unit_beta != 0, pow2 = sizeof(T) == 8 && lv[jb.first].inv_d_shift > 0;
    on_flag(gs, [&](auto GS) {
        constexpr bool D = sizeof(T) == 8;
        if (unit) tail_cycle<T, CL, true, D, GS.value>(jb, lv, nu1, nu2, w, omw, nc, ncl);  // d = 4
        else if (pow2) tail_cycle<T, CL, false, D, GS.value>(jb, lv, nu1, nu2, w, omw, nc, ncl);
        else tail_cycle<T, CL, false, false, GS.value>(jb, lv, nu1, nu2, w, omw, nc, ncl);
    });
}

template <class T, bool CL>
__global__ void __launch_bounds__(SMEM_TAIL_THREADS, 1)
    smem_tail_kernel(const TailJob* __restrict__ jobs, int count, unsigned* claim, const BatchLevel<T>* __restrict__ lv,
                     const int* __restrict__ active, int nu1, int nu2, int gs, T w, T omw, int nc, int ncl)
{
    after_prior();
    if (CL) {
        tail_dispatch<T, true>(jobs[0], lv, nu1, nu2, gs != 0, w, omw, nc, ncl);
        return;
    }
    const ItemClaim ic{claim, count};
    for (int k = ic.take(-1); k < count; k = ic.take(k)) {
        const TailJob jb = jobs[k];
        if (active && !active[lv[jb.first].problem]) continue;
        tail_dispatch<T, false>(jb, lv, nu1, nu2, gs != 0, w, omw, 1, 0);
        __syncthreads();  // shared memory is reused by the next job
    }
    ic.finish();
}

constexpr size_t SMEM_MAX = 227 * 1024 - 2048;  // dynamic shared memory left beside the static

template <class T, bool CL>
cudaError_t tail_attributes(size_t smem)
{
    static std::atomic<size_t> set[ATTR_DEVICES];
    auto kern = smem_tail_kernel<T, CL>;
    const int dev = attr_slot();
    if (dev >= 0 && set[dev].load() >= smem + 1) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess && CL) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) attr_record(set, dev, smem + 1);
    return e;
}

// The largest cluster of at most 16 CTAs with `smem` bytes each that the current device can hold.
template <class T>
int cluster_size(size_t smem)
{
    static std::atomic<int> known[ATTR_DEVICES];
    const int dev = attr_slot();
    if (dev >= 0 && known[dev].load() > 0) return known[dev].load();
    int best = 1;
    for (int nc = 16; nc > 1 && best == 1; nc /= 2) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = nc;
        cfg.blockDim = SMEM_TAIL_THREADS;
        cfg.dynamicSmemBytes = SMEM_MAX;
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = nc;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int n = 0;
        if (tail_attributes<T, true>(SMEM_MAX) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, smem_tail_kernel<T, true>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        if (n > 0) best = nc;
    }
    if (dev >= 0) known[dev].store(best);
    return best;
}

template <class T>
size_t tail_bytes(int m, int n, int nl, int nc, int ncl)
{
    const int rows0 = nc > 1 ? tail_rows(n, nc, ncl) : 0;
    size_t elems = 0, largest = 0;
    for (int l = 0; l < nl; ++l) {
        const size_t size = (size_t)tail_slots(n, l, nc, ncl, rows0) * 2 * tail_half(m);
        elems += 2 * size;
        largest = std::max(largest, size);
        if (l == nl - 1) break;
        m = (m - 1) / 2 + 1;
        n = (n - 1) / 2 + 1;
    }
    const size_t N = (size_t)(m - 2) * (n - 2);
    return TAIL_HEAD + (elems + largest) * sizeof(T) + (N + (N <= TAIL_STAGED ? N * N : 0)) * sizeof(double);
}

}  // namespace

template <class T>
SmemTail plan_smem_tail(int m, int n, int nl, bool cluster)
{
    SmemTail p;
    if (nl < 1 || nl > TAIL_LEVELS || m > SMEM_TAIL_THREADS) return p;  // two half rows per CTA width
    // a level is worth splitting while its phases last longer than a cluster barrier: about 1000
    // points in FP64, 4000 in FP32; every CTA keeps at least two rows
    if (cluster && nl > 1) {
        const int nc = cluster_size<T>(SMEM_MAX);
        int ncl = 0, a = m, b = n;
        while (nc > 1 && ncl < nl - 1 && (int64_t)a * b >= (sizeof(T) == 8 ? 1000 : 4000) &&
               (tail_rows(n, nc, ncl + 1) >> ncl) >= 2) {
            // an uneven cut that leaves half the CTAs without rows is not worth another split level
            if ((n - 1 + tail_rows(n, nc, ncl + 1) - 1) / tail_rows(n, nc, ncl + 1) < std::max(2, nc / 2)) break;
            ++ncl;
            a = (a - 1) / 2 + 1;
            b = (b - 1) / 2 + 1;
        }
        if (ncl > 0) {
            const size_t bytes = tail_bytes<T>(m, n, nl, nc, ncl);
            if (bytes <= SMEM_MAX) {
                p.nc = nc;
                p.ncl = ncl;
                p.bytes = bytes;
                return p;
            }
        }
    }
    const size_t bytes = tail_bytes<T>(m, n, nl, 1, 0);
    if (bytes <= SMEM_MAX) {
        p.nc = 1;
        p.bytes = bytes;
    }
    return p;
}
template SmemTail plan_smem_tail<double>(int, int, int, bool);
template SmemTail plan_smem_tail<float>(int, int, int, bool);

template <class T>
cudaError_t launch_smem_tail(const TailJob* jobs, int count, const BatchLevel<T>* lv, const int* active, int nu1,
                             int nu2, bool gs, double w, const SmemTail& plan, cudaStream_t s, unsigned* claim)
{
    if (count == 0) return cudaSuccess;
    const int g = gs ? 1 : 0;
    const T wt = (T)w, omw = (T)(1.0 - w);
    if (plan.nc > 1) {
        cudaError_t e = tail_attributes<T, true>(SMEM_MAX);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = plan.nc;
        cfg.blockDim = SMEM_TAIL_THREADS;
        cfg.dynamicSmemBytes = plan.bytes;
        cfg.stream = s;
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = plan.nc;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_after
        at[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = 2;
        e = cudaLaunchKernelEx(&cfg, smem_tail_kernel<T, true>, jobs, count, (unsigned*)nullptr, lv, active, nu1, nu2,
                               g, wt, omw, plan.nc, plan.ncl);
        note_launch();
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    const cudaError_t e = tail_attributes<T, false>(SMEM_MAX);
    if (e != cudaSuccess) return e;
    const int grid = batch_grid((const void*)smem_tail_kernel<T, false>, SMEM_TAIL_THREADS, plan.bytes, count,
                                claim != nullptr);
    launch_after(smem_tail_kernel<T, false>, grid, SMEM_TAIL_THREADS, plan.bytes, s, jobs, count, claim, lv, active, nu1, nu2, g,
                                                                           wt, omw, 1, 0);
    note_launch();
    return cudaGetLastError();
}
template cudaError_t launch_smem_tail<double>(const TailJob*, int, const BatchLevel<double>*, const int*, int, int, bool, double, const SmemTail&, cudaStream_t, unsigned*);
template cudaError_t launch_smem_tail<float>(const TailJob*, int, const BatchLevel<float>*, const int*, int, int, bool, double, const SmemTail&, cudaStream_t, unsigned*);

}  // namespace lap

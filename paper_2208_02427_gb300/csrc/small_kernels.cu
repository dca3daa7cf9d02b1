// small_kernels.cu -- a whole solve in one CTA: small grids with the paper's stopping rule.
//
// On a grid of a few thousand points (the paper's chamber is 25 x 17) a sweep is shorter than a
// launch. These kernels hold the field in shared memory and run check periods (check_every
// iterations, the last shortened to max_iter) until max |psi^{k+1} - psi^k| (Eq. 16) over the
// period's last iteration is <= tol or not finite. They take the initial and the final residual
// norm too and write their report straight to the host's pinned block, so a solve is one launch
// and one wait.
//
// What bounds them is the FP64 pipe of one SM. A warp's FP64 instruction occupies its scheduler's
// unit for 64 cycles however many lanes are active (measured: 1, 8, 16 and 32 active lanes all
// take 64 cycles a dependent fma, 16 SM cycles with the four schedulers busy), so the cost is the
// number of warp instructions and lanes are packed as full as the work allows. Everything else
// (addresses, the stopping test) is kept off the path: a thread owns the same points in every
// sweep, keeps their offsets and last values in registers, and the stopping test is a flag that
// rides on the sweep's own barrier.
// Measured on the chamber with the paper's rule (whole solves through the binding, the field's copy
// included), against one CTA with an index division per point, three barriers and two reductions
// per test, and one Thomas chain per thread: SOR(1.75) 235 -> 122 us (1.1 us an iteration, 45 us of
// it outside the loop), ADI(1.3, form B) 2362 -> 644 us (6.3 us an iteration).
#include <algorithm>

#include "lap_device.cuh"
#include "lap_internal.cuh"

namespace lap {

namespace {

constexpr int SP_THREADS = 512;
constexpr int SP_MAX_POINTS = 4096;
static_assert(SP_MAX_POINTS / 2 <= 4 * SP_THREADS, "four points of a colour per thread at most");
constexpr unsigned long long INF_BITS = 0x7ff0000000000000ull;

// ||r||_2 of the dense m x n field u, all threads taking part: bit for bit the sum that
// defect_sumsq_kernel and sum_partials_kernel give for a grid this small, where thread g of block
// g / 256 holds the one point g (a tree over each warp, over a block's eight warps, then over the
// blocks). red: 8 doubles per 256 interior points.
template <bool UNIT_BETA>
__device__ double cta_residual_norm(const FmaOps& o, const double* u, int m, int n, double b2, double d,
                                    double* red)
{
    const int mi = m - 2, total = mi * (n - 2), blocks = (total + 255) / 256;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    for (int v = wid; v < 8 * blocks; v += nw) {
        const int k = 32 * v + lane;
        double acc = 0.0;
        if (k < total) {
            const double* c = u + (1 + k / mi) * m + 1 + k % mi;
            const double s = neighbour_sum<UNIT_BETA>(o, c[-1], c[1], c[-m], c[m], b2);
            const double r = __fma_rn(-d, *c, s);
            acc = __fma_rn(r, r, 0.0);
        }
        acc = warp_sum(acc);
        if (lane == 0) red[v] = acc;
    }
    __syncthreads();
    if (wid == 0) {
        double part = 0.0;
        for (int b = 0; b < blocks; ++b) {
            const double v = warp_sum(lane < 8 ? red[8 * b + lane] : 0.0);
            if (lane == b) part = v;
        }
        part = warp_sum(part);
        if (lane == 0) red[0] = sqrt(part);
    }
    __syncthreads();
    const double r = red[0];
    __syncthreads();
    return r;
}

// The stopping test of a period, given each thread's largest |change| of its last iteration (as
// ordered bits) and called just before the iteration's own barrier: flags set f says whether some
// change exceeds tol and whether some is not finite. Three sets in turn: set (f + 2) % 3 is
// cleared after the barrier of set f, when every thread has read it and none can write it yet.
struct StopFlags {
    int over[3], bad[3];
};
__device__ __forceinline__ void stop_vote(StopFlags* s, int f, unsigned long long dl,
                                          unsigned long long tol_bits)
{
    if (dl > tol_bits) s->over[f] = 1;
    if (dl >= INF_BITS) s->bad[f] = 1;
}
// After the barrier: whether the solve stops here.
__device__ __forceinline__ bool stop_read(StopFlags* s, int f, int* status)
{
    const int over = s->over[f], bad = s->bad[f];
    if (threadIdx.x == 0) {
        const int z = f == 0 ? 2 : f - 1;
        s->over[z] = s->bad[z] = 0;
    }
    *status = bad ? 2 : (over ? 1 : 0);
    return *status != 1;
}

// The largest of the threads' values (ordered bits).
__device__ unsigned long long cta_max(unsigned long long v, unsigned long long* red)
{
    v = warp_max_u64(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    unsigned long long best = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) best = red[k] > best ? red[k] : best;
    return best;
}

// ---- point methods: Jacobi and red-black Gauss-Seidel / SOR --------------------------------
// One pass over the points off[0 .. count) of this thread (Eqs. 5-7), from a to b (the same
// buffer for the red-black methods); cur[] are their last values. All points' operands are
// loaded before the first is stored (a colour's points do not read one another).
template <bool UNIT_BETA, bool POW2, bool GS, int N>
__device__ __forceinline__ unsigned long long point_pass(const FmaOps& o, const double* a, double* b,
                                                         int m, const int (&off)[N], double (&cur)[N],
                                                         int count, double b2, double inv_d, int shift,
                                                         double w, double omw, bool track,
                                                         unsigned long long dl)
{
    double nv[N];
#pragma unroll
    for (int p = 0; p < N; ++p) {
        if (p >= count) continue;
        const double* c = a + off[p];
        const double s = neighbour_sum<UNIT_BETA>(o, c[-1], c[1], c[-m], c[m], b2);
        const double g = times_inv_d<POW2>(o, s, inv_d, shift);
        nv[p] = GS ? g : __fma_rn(w, g, fmul(o, omw, cur[p]));
    }
#pragma unroll
    for (int p = 0; p < N; ++p)
        if (p < count) b[off[p]] = nv[p];
    if (track) {
#pragma unroll
        for (int p = 0; p < N; ++p) {
            if (p >= count) continue;
            const unsigned long long v = abs_bits(fadd(o, nv[p], -cur[p]));
            dl = v > dl ? v : dl;
        }
    }
#pragma unroll
    for (int p = 0; p < N; ++p)
        if (p < count) cur[p] = nv[p];
    return dl;
}

// N: points of one colour (Jacobi: of one half of the interior) per thread, at most.
template <int N, bool JACOBI, bool UNIT_BETA, bool POW2, bool GS>
__global__ void __launch_bounds__(SP_THREADS)
    small_point_kernel(double* __restrict__ psi, int m, int n, int64_t pitch, double b2, double d,
                       double inv_d, int shift, double w, double omw, long long every,
                       long long max_iter, double tol, SmallReport* __restrict__ rep)
{
    const FmaOps o = load_fma_ops();
    b2 = in_reg(o, b2);
    d = in_reg(o, d);
    inv_d = in_reg(o, inv_d);
    w = in_reg(o, w);
    omw = in_reg(o, omw);
    extern __shared__ double u[];
    __shared__ double red[8 * SP_MAX_POINTS / 256];
    __shared__ unsigned long long red64[SP_THREADS / 32];
    __shared__ StopFlags flags;
    const int tid = threadIdx.x, nt = blockDim.x;
    double* a = u;
    double* b = JACOBI ? u + m * n : u;
    for (int k = tid; k < m * n; k += nt) {
        const double v = psi[(int64_t)(k / m) * pitch + k % m];
        a[k] = v;
        if (JACOBI) b[k] = v;
    }
    if (tid < 3) flags.over[tid] = flags.bad[tid] = 0;
    const double r0 = cta_residual_norm<UNIT_BETA>(o, a, m, n, b2, d, red);
    // this thread's points: list 0 the red ones, list 1 the black ones (Jacobi: the two halves of
    // the interior in row order, one pass after the other without a barrier between)
    int off[2][N], count[2];
    double cur[2][N];
    const int mi = m - 2, half_w = (mi + 1) / 2, rows = n - 2, total = mi * rows;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        count[c] = 0;
        if (JACOBI) {
            const int lo = c == 0 ? 0 : total / 2, hi = c == 0 ? total / 2 : total;
#pragma unroll
            for (int p = 0; p < N; ++p) {
                const int k = lo + tid + p * nt;
                if (k < hi) {
                    off[c][p] = (1 + k / mi) * m + 1 + k % mi;
                    cur[c][p] = a[off[c][p]];
                    count[c] = p + 1;
                }
            }
        } else {
            // same-colour points in row order, rows alternating between per[0] and per[1] points
            const int first = c == 0 ? half_w : mi / 2, second = mi - first;  // in rows 1, 2
            const int colour_total = (rows + 1) / 2 * first + rows / 2 * second;
#pragma unroll
            for (int p = 0; p < N; ++p) {
                const int k = tid + p * nt;
                if (k < colour_total) {
                    const int pair = k / mi, in = k - pair * mi;  // two rows hold mi of a colour
                    const int j = 1 + 2 * pair + (in >= first);
                    const int t = in >= first ? in - first : in;
                    off[c][p] = j * m + 1 + ((1 + j + c) & 1) + 2 * t;
                    cur[c][p] = a[off[c][p]];
                    count[c] = p + 1;
                }
            }
        }
    }
    const unsigned long long tol_bits = abs_bits(tol);
    unsigned long long dl = 0;
    long long k = 0;
    int status = isfinite(r0) ? 1 : 2, f = 0;
    bool tested = false;
    while (status == 1 && k < max_iter) {
        const long long rest = max_iter - k, nst = every < rest ? every : rest;
        for (long long s = 0; s < nst; ++s) {
            const bool track = s == nst - 1;
            dl = point_pass<UNIT_BETA, POW2, GS>(o, a, b, m, off[0], cur[0], count[0], b2, inv_d, shift, w,
                                                 omw, track, 0ull);
            if (!JACOBI) __syncthreads();
            dl = point_pass<UNIT_BETA, POW2, GS>(o, a, b, m, off[1], cur[1], count[1], b2, inv_d, shift, w,
                                                 omw, track, dl);
            if (track) stop_vote(&flags, f, dl, tol_bits);
            __syncthreads();
            if (JACOBI) {
                double* t = a;
                a = b;
                b = t;
            }
        }
        k += nst;
        tested = true;
        if (stop_read(&flags, f, &status)) break;
        f = f == 2 ? 0 : f + 1;
    }
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int p = 0; p < N; ++p)
            if (p < count[c]) {
                const int j = off[c][p] / m, i = off[c][p] - j * m;
                psi[(int64_t)j * pitch + i] = cur[c][p];
            }
    const unsigned long long worst = cta_max(dl, red64);
    const double rn = k > 0 ? cta_residual_norm<UNIT_BETA>(o, a, m, n, b2, d, red) : r0;
    if (tid == 0) {
        rep->k = k;
        rep->status = status;
        rep->last_check = tested ? __longlong_as_double((long long)worst) : __longlong_as_double(-1ll);
        rep->r0 = r0;
        rep->r_final = rn;
    }
}

// ---- line methods: zebra SLOR (x-lines) and ADI (x-lines, then y-lines) ---------------------
// The chunked algorithm of line_kernels.cu, with the SW lanes of a warp segment on one line:
// lane p holds chunk p (L unknowns) and the separator behind it; the separators' tridiagonal
// system is solved by parallel cyclic reduction across the segment (shuffles), so a colour of
// lines needs one CTA barrier. SW is chosen so that a colour's lines fill about one warp per
// scheduler: more lanes per line shorten the serial recurrences but add reduction levels and, past
// one warp per scheduler, queue for the FP64 units. L = 0 (as many lanes as unknowns) is plain
// cyclic reduction. Chamber, x-lines (23 unknowns, 12 lines a colour), FP64 instructions on the
// busiest scheduler per half sweep: 48 at SW = 32 (L = 0), 30 at SW = 8 (L = 2), 50 at SW = 4.
constexpr int SL_THREADS = 512;

// A direction's tables rebased into shared memory.
struct CtaLines {
    int N, L, P, Ll, K0, levels, maxp, sw_log;
    double alpha, wc, bnd, c1;
    const double *e, *inv_den, *sc, *F, *gln, *glnl, *k1, *k2, *invb;
};

__device__ __forceinline__ CtaLines cta_lines(const FmaOps& o, const LineTables& t, double bnd,
                                              double c1, int sw_log, double* sm)
{
    // sm: e and alpha behind it, then the rest of the tables in their order
    const int len = small_line_table_doubles(t);
    for (int k = threadIdx.x; k < len; k += blockDim.x) sm[k < t.L ? k : k + 1] = t.e[k];
    if (threadIdx.x == 0) sm[t.L] = t.alpha;
    CtaLines c;
    c.N = t.N;
    c.L = t.L;
    c.P = t.P;
    c.Ll = t.Ll;
    c.K0 = t.K0;
    c.levels = t.levels;
    c.maxp = t.maxp;
    c.sw_log = sw_log;
    c.alpha = in_reg(o, t.alpha);
    c.wc = in_reg(o, t.wc);
    c.bnd = in_reg(o, bnd);
    c.c1 = in_reg(o, c1);
    c.e = sm;
    c.inv_den = sm + 1 + (t.inv_den - t.e);
    c.sc = sm + 1 + (t.sc - t.e);
    c.F = sm + 1 + (t.F - t.e);
    c.gln = sm + 1 + (t.gln - t.e);
    c.glnl = sm + 1 + (t.glnl - t.e);
    c.k1 = sm + 1 + (t.k1 - t.e);
    c.k2 = sm + 1 + (t.k2 - t.e);
    c.invb = sm + 1 + (t.invb - t.e);
    return c;
}

// Relaxes the lines `first`, first + 2, ... <= lines: element k (0 .. N + 1) of line l at
// u[l * sx + k * sa]. G: work space, one slot per unknown of a line and lines of a colour.
// TRACK: the largest |new - prev| of the points written, which also go to prev.
template <int FORM, bool TRACK>
__device__ __forceinline__ unsigned long long cta_colour(const FmaOps& o, const CtaLines& t, double* u,
                                                         double* prev, int sx, int sa, int lines,
                                                         int first, double omw, double* G,
                                                         unsigned long long dl)
{
    const int SW = 1 << t.sw_log, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int p = lane & (SW - 1), per_warp = 32 >> t.sw_log, nw = blockDim.x >> 5;
    const int count = (lines - first) / 2 + 1;  // lines >= first
    const int L = t.L, S = t.P - 1, N = t.N;
    const unsigned full = 0xffffffffu;
    for (int g = wid; g * per_warp < count; g += nw) {
        const int li = g * per_warp + (lane >> t.sw_log);
        const bool act = li < count;
        double* line = u + (first + 2 * (act ? li : 0)) * sx;
        double* pl = prev + (first + 2 * (act ? li : 0)) * sx;
        // G of chunk position q at q * gs: lanes in consecutive words
        double* gw = G + g * 32 * (L > 0 ? L : 1) + lane;
        const int len = !act || p >= t.P ? 0 : (p == t.P - 1 ? t.Ll : L);
        const bool sep = act && p < S;
        const int k0 = 1 + p * (L + 1);
        const double* gl = p == t.P - 1 ? t.glnl : t.gln;
        auto rhs = [&](int k) {
            const double* c = line + k * sa;
            const double b = fadd(o, c[-sx], c[sx]);
            return FORM == 1 ? __fma_rn(t.c1, c[0], b) : b;
        };
        // The Dirichlet ends enter b~_1 and b~_N. They are added outside the loops (as a test per
        // position the compiler issues their fma at every position).
        double Gq = 0.0, D = 0.0;
        if (len > 0) {
            Gq = rhs(k0);
            if (p == 0) Gq = __fma_rn(t.bnd, line[0], Gq);
            gw[0] = Gq;
            D = fmul(o, gl[0], Gq);
        }
        int q = 1;
        for (; q < min(len, t.K0); ++q) {
            const double b = rhs(k0 + q);
            Gq = __fma_rn(t.e[q - 1], Gq, b);
            D = __fma_rn(gl[q], b, D);
            gw[32 * q] = Gq;
        }
        for (; q < len; ++q) {
            Gq = __fma_rn(t.e[q - 1], Gq, rhs(k0 + q));
            gw[32 * q] = Gq;
        }
        if (len > 0 && p == t.P - 1) {  // the far end, linear in G and D
            const double far = fmul(o, t.bnd, line[(N + 1) * sa]);
            Gq = fadd(o, Gq, far);
            gw[32 * (len - 1)] = Gq;
            if (len <= t.K0) D = __fma_rn(gl[len - 1], far, D);
        }
        double rho = 0.0;
        if (sep) rho = rhs(k0 + L);
        if (L > 0) {
            const double ylast = len > 0 ? fmul(o, t.inv_den[len - 1], Gq) : 0.0;
            const double ynext = __shfl_down_sync(full, D, 1, SW);
            if (sep) rho = __fma_rn(t.alpha, fadd(o, ylast, ynext), rho);
        } else {
            if (sep && p == 0) rho = __fma_rn(t.bnd, line[0], rho);
            if (sep && p == N - 1) rho = __fma_rn(t.bnd, line[(N + 1) * sa], rho);
        }
        for (int lev = 0, s = 1; lev < t.levels; ++lev, s <<= 1) {
            // the multipliers are 0 where a neighbour is missing (and the shuffle returns rho)
            const double lo = __shfl_up_sync(full, rho, s, SW), hi = __shfl_down_sync(full, rho, s, SW);
            const int at = lev * t.maxp + min(p, S - 1);
            rho = __fma_rn(t.k2[at], hi, __fma_rn(t.k1[at], lo, rho));
            if (!sep) rho = 0.0;
        }
        const double xs = sep ? fmul(o, rho, t.invb[p]) : 0.0;
        const double xup = __shfl_up_sync(full, xs, 1, SW);
        const double xl = p > 0 ? xup : 0.0;
        auto out = [&](int k, double scale, double Z) {
            double* c = line + k * sa;
            const double v = FORM == 0 ? __fma_rn(scale, Z, fmul(o, omw, *c)) : fmul(o, scale, Z);
            *c = v;
            if (TRACK) {
                double* q = pl + k * sa;
                const unsigned long long b = abs_bits(fadd(o, v, -*q));
                dl = b > dl ? b : dl;
                *q = v;
            }
        };
        if (sep) out(k0 + L, t.wc, xs);
        // e[L] is alpha: the position before a separator couples to it with alpha, and the last
        // chunk, possibly shorter, has no separator behind it (xs = 0)
        double Z = xs;
        q = len - 1;
        for (; q >= t.K0; --q) {
            Z = __fma_rn(t.e[q + 1], Z, gw[32 * q]);
            out(k0 + q, t.sc[q], Z);
        }
        for (; q >= 0; --q) {
            Z = __fma_rn(t.e[q + 1], Z, __fma_rn(xl, t.F[q], gw[32 * q]));
            out(k0 + q, t.sc[q], Z);
        }
    }
    return dl;
}

template <bool ADI, int FORM>
__global__ void __launch_bounds__(SL_THREADS)
    small_line_kernel(double* __restrict__ psi, int m, int n, int64_t pitch, double b2, double d,
                      const LineTables tx, double bndx, double c1x, int swx, const LineTables ty,
                      double bndy, double c1y, int swy, double omw, int unit_beta, long long every,
                      long long max_iter, double tol, SmallReport* __restrict__ rep)
{
    extern __shared__ double u[];
    const FmaOps o = load_fma_ops();
    __shared__ double red[8 * SP_MAX_POINTS / 256];
    __shared__ unsigned long long red64[SL_THREADS / 32];
    __shared__ StopFlags flags;
    double* prev = u + m * n;
    double* G = prev + m * n;
    double* tabs = G + small_line_work_doubles(m, n, tx, swx, ty, swy, ADI);
    const int tid = threadIdx.x;
    b2 = in_reg(o, b2);
    d = in_reg(o, d);
    omw = in_reg(o, omw);
    const CtaLines X = cta_lines(o, tx, bndx, c1x, swx, tabs);
    const CtaLines Y = ADI ? cta_lines(o, ty, bndy, c1y, swy, tabs + small_line_table_doubles(tx) + 1) : X;
    for (int k = tid; k < m * n; k += blockDim.x) u[k] = prev[k] = psi[(int64_t)(k / m) * pitch + k % m];
    if (tid < 3) flags.over[tid] = flags.bad[tid] = 0;
    const double r0 = unit_beta ? cta_residual_norm<true>(o, u, m, n, b2, d, red)
                                : cta_residual_norm<false>(o, u, m, n, b2, d, red);
    const unsigned long long tol_bits = abs_bits(tol);
    unsigned long long dl = 0;
    long long k = 0;
    int status = isfinite(r0) ? 1 : 2, f = 0;
    bool tested = false;
    while (status == 1 && k < max_iter) {
        const long long rest = max_iter - k, nst = every < rest ? every : rest;
        for (long long s = 0; s < nst; ++s) {
            // the iteration's last half sweep keeps prev, the field before the next iteration
            dl = 0;
            for (int first = 1; first <= 2; ++first) {
                if (first <= n - 2) dl = cta_colour<FORM, !ADI>(o, X, u, prev, m, 1, n - 2, first, omw, G, dl);
                if (!ADI && first == 2 && s == nst - 1) stop_vote(&flags, f, dl, tol_bits);
                __syncthreads();
            }
            if (ADI)
                for (int first = 1; first <= 2; ++first) {
                    if (first <= m - 2) dl = cta_colour<FORM, true>(o, Y, u, prev, 1, m, m - 2, first, omw, G, dl);
                    if (first == 2 && s == nst - 1) stop_vote(&flags, f, dl, tol_bits);
                    __syncthreads();
                }
        }
        k += nst;
        tested = true;
        if (stop_read(&flags, f, &status)) break;
        f = f == 2 ? 0 : f + 1;
    }
    const int mi = m - 2;
    for (int q = tid; q < mi * (n - 2); q += blockDim.x) {
        const int i = 1 + q % mi, j = 1 + q / mi;
        psi[(int64_t)j * pitch + i] = u[j * m + i];
    }
    const unsigned long long worst = cta_max(dl, red64);
    double rn = r0;
    if (k > 0)
        rn = unit_beta ? cta_residual_norm<true>(o, u, m, n, b2, d, red)
                       : cta_residual_norm<false>(o, u, m, n, b2, d, red);
    if (tid == 0) {
        rep->k = k;
        rep->status = status;
        rep->last_check = tested ? __longlong_as_double((long long)worst) : __longlong_as_double(-1ll);
        rep->r0 = r0;
        rep->r_final = rn;
    }
}

// Raises the dynamic shared-memory limit of kernel `f` to smem on the current device.
template <class F>
cudaError_t raise_smem(F* f, std::atomic<size_t>* set, size_t smem)
{
    const int dev = attr_slot();
    if (smem <= SMEM_UNASKED || (dev >= 0 && smem <= set[dev].load())) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) attr_record(set, dev, smem);
    return e;
}

}  // namespace

bool small_points_ok(int m, int n) { return (int64_t)m * n <= SP_MAX_POINTS; }

cudaError_t launch_small_point(const Field& f, const Coef& c, bool jacobi, bool gs, double w,
                               int64_t every, int64_t max_iter, double tol, SmallReport* rep,
                               cudaStream_t s)
{
    static std::atomic<size_t> set[36][ATTR_DEVICES];
    // as many warps as one colour fills with 1, 2 or 4 points per thread (at least 2): a warp with
    // idle lanes, or a point per thread too many, costs the FP64 pipe as much as a full one
    const int per_pass = ((f.m - 2) * (f.n - 2) + 1) / 2;
    const int each = per_pass <= SP_THREADS ? 1 : (per_pass <= 2 * SP_THREADS ? 2 : 4);
    const int threads = std::max(64, ((per_pass + each - 1) / each + 31) / 32 * 32);
    const size_t smem = (jacobi ? 2 : 1) * sizeof(double) * (size_t)f.m * f.n;
    const bool p2 = c.inv_d_shift > 0;
    cudaError_t e = cudaSuccess;
    auto go = [&](auto* kern, int slot) {
        e = raise_smem(kern, set[slot], smem);
        if (e != cudaSuccess) return;
        kern<<<1, threads, smem, s>>>(f.p, f.m, f.n, f.pitch, c.b2, c.d, c.inv_d, c.inv_d_shift, w, 1.0 - w,
                                      (long long)every, (long long)max_iter, tol, rep);
    };
#define LAP_SP(N, U, P, SLOT)                                                            \
    do {                                                                                 \
        if (jacobi) go(small_point_kernel<N, true, U, P, true>, SLOT);                   \
        else if (gs) go(small_point_kernel<N, false, U, P, true>, SLOT + 1);             \
        else go(small_point_kernel<N, false, U, P, false>, SLOT + 2);                    \
    } while (0)
#define LAP_SPN(N, SLOT)                                                                 \
    do {                                                                                 \
        if (c.unit_beta) {                                                               \
            if (p2) LAP_SP(N, true, true, SLOT); else LAP_SP(N, true, false, SLOT + 3);  \
        } else {                                                                         \
            if (p2) LAP_SP(N, false, true, SLOT + 6); else LAP_SP(N, false, false, SLOT + 9); \
        }                                                                                \
    } while (0)
    if (each == 1) LAP_SPN(1, 0);
    else if (each == 2) LAP_SPN(2, 12);
    else LAP_SPN(4, 24);
#undef LAP_SPN
#undef LAP_SP
    note_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

int small_line_lanes_log(int count, int N)
{
    // lanes per line: the largest power of two that keeps a colour's `count` lines within one warp
    // per scheduler (128 lanes), and no more than the line's unknowns need
    int k = 0;
    while (k < 5 && (count << (k + 1)) <= 128 && (1 << k) < N) ++k;
    return k;
}

size_t small_line_smem(int m, int n, const LineTables& tx, int swx, const LineTables& ty, int swy, bool adi)
{
    return sizeof(double) * ((size_t)2 * m * n + small_line_work_doubles(m, n, tx, swx, ty, swy, adi) +
                             small_line_table_doubles(tx) + 1 + (adi ? small_line_table_doubles(ty) + 1 : 0));
}

cudaError_t launch_small_line(const Field& f, const Coef& c, bool adi, int form, const LineTables& tx,
                              const LineCoefs& kx, int swx, const LineTables& ty, const LineCoefs& ky,
                              int swy, int64_t every, int64_t max_iter, double tol, SmallReport* rep,
                              cudaStream_t s)
{
    static std::atomic<size_t> set[4][ATTR_DEVICES];
    const size_t smem = small_line_smem(f.m, f.n, tx, swx, ty, swy, adi);
    cudaError_t e = cudaSuccess;
    auto go = [&](auto* kern, int slot) {
        e = raise_smem(kern, set[slot], smem);
        if (e != cudaSuccess) return;
        // as many warps as a colour's lines fill (at least 4: one per scheduler)
        auto warps = [](int lines, int sw) { return ((lines + 1) / 2 + (32 >> sw) - 1) / (32 >> sw); };
        int nw = std::max(4, warps(f.n - 2, swx));
        if (adi) nw = std::max(nw, warps(f.m - 2, swy));
        const int threads = 32 * std::min(nw, SL_THREADS / 32);
        kern<<<1, threads, smem, s>>>(f.p, f.m, f.n, f.pitch, c.b2, c.d, tx, kx.bnd, kx.c1, swx, ty, ky.bnd,
                                      ky.c1, swy, kx.omw, c.unit_beta ? 1 : 0, (long long)every,
                                      (long long)max_iter, tol, rep);
    };
    if (adi) {
        if (form == 0) go(small_line_kernel<true, 0>, 0); else go(small_line_kernel<true, 1>, 1);
    } else {
        if (form == 0) go(small_line_kernel<false, 0>, 2); else go(small_line_kernel<false, 1>, 3);
    }
    note_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace lap

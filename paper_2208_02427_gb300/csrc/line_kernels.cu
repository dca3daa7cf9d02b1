// line_kernels.cu -- zebra line relaxation (SLOR / ADI half sweeps, Eqs. 8-10).
//
// Every line of one zebra colour is an independent tridiagonal system with constant
// coefficients, -alpha x_{k-1} + delta x_k - alpha x_{k+1} = b_k (k = 1..N). The kernels solve
// it scaled: with nb_k the sum of the two neighbouring lines' values, the right-hand side is
//   form A (Eqs. 8-9):  b~_k = nb_k                       and  x = cross x~,
//   form B (Eq. 10):    b~_k = fma(c1, psi_k, nb_k)       and  x = w cross x~,
// c1 = d (1 - w) / (w cross), the Dirichlet ends adding (off / cross) psi_end to b~_1 and b~_N
// (off, cross: the along-line and across-line coefficients, 1 and beta^2 for x-lines). The line
// is cut into P <= 32 chunks of L unknowns (the last holds Ll), each but the last followed by
// one separator unknown. Per chunk, with den_q the Thomas pivots of the zero-end chunk matrix
// and e_q = alpha / den_q:
//   forward    G_q = fma(e_{q-1}, G_{q-1}, b~_q)             (G_q = den_q y'_q, unnormalised)
//   separators  the chunks' zero-end solutions end in y_last = G_{L-1} / den_{L-1} and start in
//              y_first = sum_q (T^-1)_{0q} b~_q; with them the separators satisfy a small
//              tridiagonal system, solved exactly by parallel cyclic reduction over one warp;
//   back       Z_q = fma(e_{q+1}, Z_{q+1}, G_q + xl F_q),  Z_{L-1} = G_{L-1} + xl F_{L-1} + alpha xr
//              (Z_q = den_q x~_q; xl, xr the separators around the chunk; F_q the forward
//              elimination of alpha at the chunk's left end),
//   output     form A: psi = fma(sc_q, Z_q, (1 - w) psi),  form B: psi = sc_q Z_q,
//              sc_q = w cross / den_q (w cross for a separator).
// (T^-1)_{0q} and F_q decay geometrically away from the chunk's left end; from the position K0
// on, where both are below 2^-64 of their first value, their terms are left out. Per unknown
// this is 5 FP64 operations (1 add + 0-1 fma for b~, 1 forward, 1 back, 1-2 for the output)
// plus 2 within K0 of a chunk's start. All tables depend on the line length and coefficients
// only and are computed once on the host.
//
// x-lines (rows, contiguous): a CTA works on one line at a time; b~ is built into shared memory
// with coalesced loads, one or two warps run the chunk recurrences (thread = chunk) and the separator
// solve, and the CTA writes the line back coalesced. The
// CTAs stay resident and take the lines of both zebra colours in order from a counter, so a
// half sweep is one launch (line_x_kernel). On GB300 each of
// an SM's four schedulers has its own FP64 unit (0.5 fma per clock; measured), and one warp's
// dependent fma chain alone keeps it busy, so the six line CTAs that fit an SM's shared memory
// are enough recurrence warps; the CTA's other warps shorten the load and store phases.
// y-lines (columns, strided by the pitch), and rows of up to 1024 unknowns: a thread per (line,
// chunk), one launch per colour, no transposed copy of the field (line_y_kernel).
#include "lap_device.cuh"
#include "lap_internal.cuh"

namespace lap {

namespace {

constexpr unsigned FULL = 0xffffffffu;
// x-lines: threads of the CTA that builds and writes a line (measured at 4097^2: 128, 160,
// 224, 256, 288, 320 threads gave 288, 285, 269, 266, 262, 255 us per form-A half sweep, the
// form-B ones 293, 282, 258, 265, 242, 272 us), the unrolling of its load and store loops,
// and the positions per batch of the chunk recurrences
constexpr int LX_THREADS = 256;
constexpr int LX_UNROLL = 8;
constexpr int XB = 8;

// ---- x-lines --------------------------------------------------------------------------
// x-lines are cut into up to LINE_MAX_CHUNKS_X = 64 chunks, run by the CTA's first two warps
// (thread p = chunk p): the recurrences, the serial part of a line, take half the steps of a
// 32-chunk cut on two schedulers, for about a tenth more FP64 operations (the chunks' boundary
// layers cover a larger share of the shorter chunks). Values passed between neighbouring
// chunks go through ex[] in shared memory, ordered by a 64-thread barrier.
__device__ __forceinline__ void bar_chunks() { asm volatile("bar.sync 1, 64;" ::: "memory"); }

// separator_solve across the two warps: level by level, each separator's value through ex[].
__device__ __forceinline__ double separator_solve_x(const LineTables& t, int p, int S, double rho,
                                                   double* ex)
{
    double r = p < S ? rho : 0.0;
    for (int lev = 0, s = 1; lev < t.levels; ++lev, s <<= 1) {
        ex[p] = r;
        bar_chunks();
        const double up = p >= s ? ex[p - s] : 0.0;
        const double dn = p + s < LINE_MAX_CHUNKS_X ? ex[p + s] : 0.0;
        bar_chunks();
        double v = r;
        if (p < S && p >= s) v = __fma_rn(t.k1[lev * t.maxp + p], up, v);
        if (p + s < S) v = __fma_rn(t.k2[lev * t.maxp + p], dn, v);
        r = v;
    }
    return p < S ? r * t.invb[p] : 0.0;
}

// The recurrences of one line held in shared memory in chunk layout (chunk p at sm[p * Ls],
// its separator at sm[p * Ls + L]), thread p = chunk p (p < 64): b~ in, the output values' Z
// (chunk positions) and x~ (separators) out. ex: 64 doubles of shared memory.
__device__ __forceinline__ void line_recurrences(const FmaOps& o, const LineTables& t,
                                                 double* sm, int p, double* ex)
{
    const int L = t.L, P = t.P, Ls = t.stride, K0 = t.K0;
    {
        const int S = P - 1;
        const bool act = p < P;
        const int len = p == P - 1 ? t.Ll : L;
        double* y = sm + p * Ls;
        const double* __restrict__ gl = p == P - 1 ? t.glnl : t.gln;
        const double alpha = in_reg(o, t.alpha);
        double G = 0.0, D = 0.0;
        const double* __restrict__ te = t.e;
        if (act) {
            // operands of a step are loaded in the step before, ahead of its store, which waits for the
            // fma (a half sweep at 3001 x 2050 105 -> 93 us)
            const int kb = min(len, K0);
            G = y[0];
            D = fmul(o, __ldg(gl), G);
            int q = 1;
            double b = y[min(1, len - 1)], e = __ldg(te), gv = __ldg(gl + min(1, len - 1));
            for (; q < kb; ++q) {
                const int nx = min(q + 1, len - 1);
                const double nb = y[nx], ne = __ldg(te + q), ng = __ldg(gl + nx);
                D = __fma_rn(gv, b, D);
                G = __fma_rn(e, G, b);
                y[q] = G;
                b = nb;
                e = ne;
                gv = ng;
            }
            // the bulk in batches: operands of XB positions loaded before the chain uses them
            for (; q + XB <= len; q += XB) {
                double bv[XB], ev[XB];
#pragma unroll
                for (int u = 0; u < XB; ++u) {
                    bv[u] = y[q + u];
                    ev[u] = __ldg(te + q + u - 1);
                }
#pragma unroll
                for (int u = 0; u < XB; ++u) {
                    G = __fma_rn(ev[u], G, bv[u]);
                    y[q + u] = G;
                }
            }
            if (q < len) {
                b = y[q];
                e = __ldg(te + q - 1);
                for (; q < len; ++q) {
                    const double nb = y[min(q + 1, len - 1)], ne = __ldg(te + q);
                    G = __fma_rn(e, G, b);
                    y[q] = G;
                    b = nb;
                    e = ne;
                }
            }
        }
        const double ylast = act ? fmul(o, t.inv_den[len - 1], G) : 0.0;
        ex[p] = D;
        bar_chunks();
        const double yfirst_next = p + 1 < LINE_MAX_CHUNKS_X ? ex[p + 1] : 0.0;
        bar_chunks();
        double rho = 0.0;
        if (p < S) rho = __fma_rn(alpha, fadd(o, ylast, yfirst_next), y[L]);
        const double xs = separator_solve_x(t, p, S, rho, ex);
        ex[p] = xs;
        bar_chunks();
        const double xl_ = p > 0 ? ex[p - 1] : 0.0;
        if (act) {
            const double xl = p > 0 ? xl_ : 0.0;
            const double xr = p < S ? xs : 0.0;
            int q = len - 1;
            double Gq = y[q];
            if (q < K0) Gq = __fma_rn(xl, t.F[q], Gq);
            double Z = __fma_rn(alpha, xr, Gq);
            y[q] = Z;
            --q;
            for (; q - XB + 1 >= K0; q -= XB) {
                double gv[XB], ev[XB];
#pragma unroll
                for (int u = 0; u < XB; ++u) {
                    gv[u] = y[q - u];
                    ev[u] = __ldg(te + q - u + 1);
                }
#pragma unroll
                for (int u = 0; u < XB; ++u) {
                    Z = __fma_rn(ev[u], Z, gv[u]);
                    y[q - u] = Z;
                }
            }
            if (q >= 0) {
                double gv = y[q], e = __ldg(te + q + 1), f = __ldg(t.F + q);
                for (; q >= K0; --q) {
                    const int nx = max(q - 1, 0);
                    const double ng = y[nx], ne = __ldg(te + nx + 1), nf = __ldg(t.F + nx);
                    Z = __fma_rn(e, Z, gv);
                    y[q] = Z;
                    gv = ng;
                    e = ne;
                    f = nf;
                }
                for (; q >= 0; --q) {
                    const int nx = max(q - 1, 0);
                    const double ng = y[nx], ne = __ldg(te + nx + 1), nf = __ldg(t.F + nx);
                    Z = __fma_rn(e, Z, __fma_rn(xl, f, gv));
                    y[q] = Z;
                    gv = ng;
                    e = ne;
                    f = nf;
                }
            }
            if (p < S) y[L] = xs;
        }
    }
}

// Phase 1 of an x-line: b~ of the row into shared memory in chunk layout, by threads tid =
// 0..nthr-1 (coalesced); each thread also adds the Dirichlet end terms of the entries it wrote.
// Loads go to L2 (ld.global.cg): rows of the first colour are written by other CTAs of the same
// launch, and L1 is not coherent between SMs.
template <int FORM>
__device__ __forceinline__ void line_x_load(const FmaOps& o, const LineTables& t, double* sm,
                                            const double* row, int64_t pitch, double bnd, double c1,
                                            int tid, int nthr)
{
    const int N = t.N, L = t.L, Ls = t.stride;
    const double* up = row - pitch;
    const double* dn = row + pitch;
#pragma unroll LX_UNROLL
    for (int k = 1 + tid; k <= N; k += nthr) {
        const double nb = fadd(o, __ldcg(up + k), __ldcg(dn + k));
        const double b = FORM == 1 ? __fma_rn(c1, __ldcg(row + k), nb) : nb;
        const int g = k - 1, p = g / (L + 1);
        sm[p * Ls + (g - p * (L + 1))] = b;
    }
    if (tid == 0) sm[0] = __fma_rn(bnd, __ldcg(row), sm[0]);
    if (tid == (N - 1) % nthr) {
        const int g = N - 1, p = g / (L + 1);
        double* e = sm + p * Ls + (g - p * (L + 1));
        *e = __fma_rn(bnd, __ldcg(row + N + 1), *e);
    }
}

// Phase 3 of an x-line: the output values written to the row (coalesced), by the same
// thread-to-element mapping as line_x_load.
template <int FORM>
__device__ __forceinline__ void line_x_store(const FmaOps& o, const LineTables& t, const double* sm,
                                             double* row, double omw, int tid, int nthr)
{
    const int N = t.N, L = t.L, Ls = t.stride;
#pragma unroll LX_UNROLL
    for (int k = 1 + tid; k <= N; k += nthr) {
        const int g = k - 1, p = g / (L + 1), q = g - p * (L + 1);
        const double v = sm[p * Ls + q];
        if (FORM == 0)
            row[k] = __fma_rn(t.sc[q], v, fmul(o, omw, __ldcg(row + k)));
        else
            row[k] = fmul(o, t.sc[q], v);
    }
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(unsigned* p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Wait until *flag != 0, at most LX_SPIN_LIMIT polls (seconds); after that the error word is
// set and the caller goes on: the host reports the error, nothing hangs.
constexpr unsigned LX_SPIN_LIMIT = 1u << 24;
__device__ __forceinline__ void wait_flag(const unsigned* flag, unsigned* err)
{
    for (unsigned it = 0; it < LX_SPIN_LIMIT; ++it) {
        if (ld_acquire(flag) != 0u) return;
        __nanosleep(128);
    }
    atomicExch(err, 1u);
}

// A whole x-line half sweep (both zebra colours) in one launch of resident CTAs. Work item
// i < nodd is row 1 + 2i (first colour), item nodd + i is row 2 + 2i (second colour); a CTA
// claims items from a counter in that order and runs the three phases on each, separated by
// CTA barriers. A second-colour row needs its two first-colour neighbours finished: they were
// claimed a colour earlier by CTAs that are running, so the wait ends (almost always at once).
// A first-colour row is published by a release store of its flag after the CTA's barrier.
// Against one launch per colour this removes the second launch's wait for the first's last
// CTAs (2048 lines on 912 CTA slots at 4097^2 left a third of the last wave idle) and lets
// CTAs at different phases overlap. sync: [0] error word (kept until the host reads it),
// [1] item counter, [2 + r] flag of row r; [1 ..] zeroed before each launch.
template <int FORM>
__global__ void __launch_bounds__(LX_THREADS, 6)
    line_x_kernel(double* __restrict__ psi, int64_t pitch, int nlines, const LineTables t,
                  double bnd, double c1, double omw, unsigned* __restrict__ sync)
{
    const FmaOps o = load_fma_ops();
    extern __shared__ double sm[];
    __shared__ int s_item;
    __shared__ double ex[LINE_MAX_CHUNKS_X];
    const int nodd = (nlines + 1) / 2;
    c1 = in_reg(o, c1);
    omw = in_reg(o, omw);
    unsigned* const done = sync + 2;
    for (;;) {
        if (threadIdx.x == 0) {
            const int item = (int)atomicAdd(sync + 1, 1u);
            if (item >= nodd && item < nlines) {
                const int r = 2 + 2 * (item - nodd);
                wait_flag(done + r - 1, sync);
                if (r + 1 <= nlines) wait_flag(done + r + 1, sync);
            }
            s_item = item;
        }
        __syncthreads();
        const int item = s_item;
        if (item >= nlines) return;
        const int r = item < nodd ? 1 + 2 * item : 2 + 2 * (item - nodd);
        double* row = psi + (int64_t)r * pitch;
        line_x_load<FORM>(o, t, sm, row, pitch, bnd, c1, threadIdx.x, LX_THREADS);
        __syncthreads();
        if (threadIdx.x < LINE_MAX_CHUNKS_X) line_recurrences(o, t, sm, threadIdx.x, ex);
        __syncthreads();
        line_x_store<FORM>(o, t, sm, row, omw, threadIdx.x, LX_THREADS);
        __syncthreads();
        if (threadIdx.x == 0 && item < nodd) {
            __threadfence();
            st_release(done + r, 1u);
        }
    }
}

// ---- y-lines: lines across the threads ----------------------------------------------
// A zebra colour is one launch. A CTA takes `nl` neighbouring lines of the colour whole: thread (line l,
// chunk c) runs its chunk's forward recurrence (G to a scratch array laid out [position][line]; it reads
// it back itself), the CTA solves its lines' separators in shared memory, and the threads run back and
// write. Element k of line l lies at psi + (first_line + 2 l) sx + k sa, its neighbouring lines at +-sx (sa =
// pitch, sx = 1: neighbouring lines share the sectors of a row). With two warps' lines and chunks in CTAs of
// their own the separators took a launch between forward and back, three launches a colour; one
// launch gives every multiprocessor the same number of lines and no waits between them. Half sweeps, three
// launches a colour / one: 300^2 27 / 14 us, 1000^2 41 / 28, 2050 x 3001 102 / 86, 500 x 4000 99 / 72, 4097^2
// 197 / 193 (ADI less SLOR iterations), 3001 x 2050 92 / 77 (launch times).
// What bounds it is the recurrence: a dependent fma takes 71 clocks, one warp on each scheduler nearly
// fills the FP64 pipe, and everything else has to be out of the way: a step's field values and table
// entries are loaded PIPE positions ahead, into registers (a table entry loaded in its step waited for the
// store of the step before, which waits for that step's fma).
constexpr int PIPE = 4;  // 8 needs 200 registers, and fewer warps hide less: 79 us against 75 at 3001 x 2050

template <int FORM>
__global__ void __launch_bounds__(LY_THREADS)
    line_y_kernel(double* __restrict__ psi, int64_t sa, int64_t sx, int first_line, int count, int nl, const LineTables t,
                  double bnd, double c1, double omw, double wc, double* __restrict__ G, int64_t gp)
{
    after_prior();
    extern __shared__ double sm[];
    const FmaOps o = load_fma_ops();
    const int l0 = blockIdx.x * nl, lines = min(nl, count - l0);
    const int c = (int)threadIdx.x / nl, l = (int)threadIdx.x - c * nl;
    const bool act = c < t.P && l < lines;
    const int L = t.L, len = c == t.P - 1 ? t.Ll : L, K0 = t.K0, S = t.P - 1;
    const int k0 = 1 + c * (L + 1);
    const double* __restrict__ te = t.e;
    double* __restrict__ line = psi + (int64_t)(first_line + 2 * (l0 + l)) * sx;
    double* __restrict__ g = G + (l0 + l) + (int64_t)(k0 - 1) * gp;
    double* const yl = sm;                  // [chunk][line] the last value of a chunk's zero-end solution,
    double* const yf = sm + t.P * nl;       // its first,
    double* const bs = sm + 2 * t.P * nl;   // and the right-hand side of the separator behind it
    const double alpha = in_reg(o, t.alpha);
    c1 = in_reg(o, c1);
    omw = in_reg(o, omw);
    wc = in_reg(o, wc);

    if (act) {
        const double* __restrict__ gl = c == t.P - 1 ? t.glnl : t.gln;
        // the field values and table entries of chunk positions q0 .. (loads only; the adds come with the
        // recurrence)
        double ra[PIPE], rb[PIPE], rc[PIPE], re[PIPE];
        auto load = [&](int q0, double* a, double* b_, double* cc, double* ee) {
#pragma unroll
            for (int u = 0; u < PIPE; ++u)
                if (q0 + u < len) {
                    const double* at = line + (int64_t)(k0 + q0 + u) * sa;
                    a[u] = at[-sx];
                    b_[u] = at[sx];
                    if (FORM == 1) cc[u] = at[0];
                    ee[u] = __ldg(te + q0 + u - 1);
                }
        };
        load(1, ra, rb, rc, re);
        // position 0 (peeled: a per-step test inside the batches would issue both sides' FP64
        // operations on every step)
        double b0;
        {
            const double* at = line + (int64_t)k0 * sa;
            b0 = fadd(o, at[-sx], at[sx]);
            if (FORM == 1) b0 = __fma_rn(c1, at[0], b0);
            if (c == 0) b0 = __fma_rn(bnd, line[0], b0);  // the near Dirichlet end
        }
        double G_ = b0;
        double D = fmul(o, __ldg(gl), b0);
        g[0] = G_;
        // positions 1.., PIPE at a time; batches that reach into the boundary layer also carry the
        // y_first sum, the others only the recurrence
        auto step = [&](int q, double a_, double b_, double c_, double e_) {
            const double nbv = fadd(o, a_, b_);
            const double b = FORM == 1 ? __fma_rn(c1, c_, nbv) : nbv;
            G_ = __fma_rn(e_, G_, b);
            g[(int64_t)q * gp] = G_;
            return b;
        };
        for (int q0 = 1; q0 < len; q0 += PIPE) {
            double na[PIPE], nb_[PIPE], nc[PIPE], ne[PIPE];
            if (q0 + PIPE < len) load(q0 + PIPE, na, nb_, nc, ne);
            if (q0 < K0) {
                double gv[PIPE];
#pragma unroll
                for (int u = 0; u < PIPE; ++u)
                    if (q0 + u < len) gv[u] = __ldg(gl + q0 + u);
#pragma unroll
                for (int u = 0; u < PIPE; ++u) {
                    const int q = q0 + u;
                    if (q < len) {
                        const double b = step(q, ra[u], rb[u], rc[u], re[u]);
                        if (q < K0) D = __fma_rn(gv[u], b, D);
                    }
                }
            } else if (q0 + PIPE <= len) {
#pragma unroll
                for (int u = 0; u < PIPE; ++u) step(q0 + u, ra[u], rb[u], rc[u], re[u]);
            } else {
#pragma unroll
                for (int u = 0; u < PIPE; ++u)
                    if (q0 + u < len) step(q0 + u, ra[u], rb[u], rc[u], re[u]);
            }
#pragma unroll
            for (int u = 0; u < PIPE; ++u) {
                ra[u] = na[u];
                rb[u] = nb_[u];
                if (FORM == 1) rc[u] = nc[u];
                re[u] = ne[u];
            }
        }
        if (c == t.P - 1) {  // the far Dirichlet end enters b~_N with coefficient 1
            const double extra = fmul(o, bnd, line[(int64_t)(t.N + 1) * sa]);
            G_ = fadd(o, G_, extra);
            g[(int64_t)(len - 1) * gp] = G_;
            if (len - 1 < K0) D = __fma_rn(gl[len - 1], extra, D);
        }
        if (c < S) {
            const double* at = line + (int64_t)(k0 + len) * sa;
            const double nb = fadd(o, at[-sx], at[sx]);
            bs[c * nl + l] = FORM == 1 ? __fma_rn(c1, at[0], nb) : nb;
        }
        yl[c * nl + l] = fmul(o, t.inv_den[len - 1], G_);
        yf[c * nl + l] = D;
    }
    __syncthreads();
    // separator c of the line: thread (l, c); its solution into bs
    double r = 0.0;
    if (act && c < S)
        r = __fma_rn(alpha, fadd(o, yl[c * nl + l], yf[(c + 1) * nl + l]), bs[c * nl + l]);
    for (int lev = 0, d = 1; lev < t.levels; ++lev, d <<= 1) {  // cyclic reduction (line_tables)
        __syncthreads();
        if (act && c < S) yl[c * nl + l] = r;
        __syncthreads();
        if (act && c < S) {
            double v = r;
            if (c >= d) v = __fma_rn(t.k1[lev * t.maxp + c], yl[(c - d) * nl + l], v);
            if (c + d < S) v = __fma_rn(t.k2[lev * t.maxp + c], yl[(c + d) * nl + l], v);
            r = v;
        }
    }
    if (act && c < S) bs[c * nl + l] = r = r * t.invb[c];
    __syncthreads();
    if (!act) return;

    const double xl = c > 0 ? bs[(c - 1) * nl + l] : 0.0;
    const double xr = c < S ? r : 0.0;
    line += (int64_t)k0 * sa;
    // positions run backwards: batch j holds q = top - u, u = 0..PIPE-1
    const double* __restrict__ tsc = t.sc;
    double gv[PIPE], ov[PIPE], ev[PIPE], sv[PIPE];
    auto load = [&](int top, double* gg, double* oo, double* ee, double* ss) {
#pragma unroll
        for (int u = 0; u < PIPE; ++u)
            if (top - u >= 0) {
                gg[u] = g[(int64_t)(top - u) * gp];
                if (FORM == 0) oo[u] = line[(int64_t)(top - u) * sa];
                ee[u] = __ldg(te + top - u + 1);
                ss[u] = __ldg(tsc + top - u);
            }
    };
    // position len - 1 (peeled), then len - 2 .. 0, PIPE at a time; batches wholly past the
    // boundary layer skip its term
    auto out = [&](int q, double Z, double old, double sc) {
        line[(int64_t)q * sa] = FORM == 0 ? __fma_rn(sc, Z, fmul(o, omw, old)) : fmul(o, sc, Z);
    };
    load(len - 2, gv, ov, ev, sv);
    if (c < S) {  // the separator behind the chunk
        double* at = line + (int64_t)len * sa;
        *at = FORM == 0 ? __fma_rn(wc, xr, fmul(o, omw, *at)) : fmul(o, wc, xr);
    }
    double Z;
    {
        const int q = len - 1;
        double Gq = g[(int64_t)q * gp];
        if (q < K0) Gq = __fma_rn(xl, t.F[q], Gq);
        Z = __fma_rn(alpha, xr, Gq);
        out(q, Z, FORM == 0 ? line[(int64_t)q * sa] : 0.0, __ldg(tsc + q));
    }
    for (int top = len - 2; top >= 0; top -= PIPE) {
        double ng[PIPE], no[PIPE], ne[PIPE], ns[PIPE];
        if (top - PIPE >= 0) load(top - PIPE, ng, no, ne, ns);
        if (top - PIPE + 1 >= K0) {
#pragma unroll
            for (int u = 0; u < PIPE; ++u) {
                Z = __fma_rn(ev[u], Z, gv[u]);
                out(top - u, Z, ov[u], sv[u]);
            }
        } else {
            double fv[PIPE];
#pragma unroll
            for (int u = 0; u < PIPE; ++u)
                if (top - u >= 0) fv[u] = __ldg(t.F + top - u);
#pragma unroll
            for (int u = 0; u < PIPE; ++u) {
                const int q = top - u;
                if (q >= 0) {
                    double Gq = gv[u];
                    if (q < K0) Gq = __fma_rn(xl, fv[u], Gq);
                    Z = __fma_rn(ev[u], Z, Gq);
                    out(q, Z, ov[u], sv[u]);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < PIPE; ++u) {
            gv[u] = ng[u];
            if (FORM == 0) ov[u] = no[u];
            ev[u] = ne[u];
            sv[u] = ns[u];
        }
    }
}

}  // namespace

size_t line_smem_bytes(const LineTables& t) { return sizeof(double) * (size_t)t.P * t.stride; }

// Raise the dynamic shared-memory limit of the x-line kernels to `smem` on the current device
// (done outside stream capture; later launches only repeat it when a longer line comes). Lines of 5952 .. 6079
// unknowns pass 48 KB by the kernels' static arrays.
static std::atomic<size_t> g_line_smem_set[ATTR_DEVICES];

cudaError_t prepare_line_kernels(size_t smem)
{
    const int dev = attr_slot();
    if (smem <= SMEM_UNASKED || (dev >= 0 && smem <= g_line_smem_set[dev].load()))
        return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(line_x_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(line_x_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem);
    if (e == cudaSuccess) attr_record(g_line_smem_set, dev, smem);
    return e;
}

size_t line_x_sync_words(int nlines) { return (size_t)nlines + 4; }

cudaError_t launch_line_x(double* psi, int64_t pitch, int nlines, const LineTables& t, int form,
                          const LineCoefs& k, unsigned* sync, cudaStream_t s)
{
    if (nlines <= 0) return cudaSuccess;
    const size_t smem = line_smem_bytes(t);
    cudaError_t e = prepare_line_kernels(smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, form == 0 ? line_x_kernel<0> : line_x_kernel<1>, LX_THREADS, smem);
    if (e != cudaSuccess) return e;
    const int grid = std::min(nlines, std::max(1, per_sm) * device_sms());
    e = cudaMemsetAsync(sync + 1, 0, (line_x_sync_words(nlines) - 1) * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    if (form == 0)
        line_x_kernel<0><<<grid, LX_THREADS, smem, s>>>(psi, pitch, nlines, t, k.bnd, k.c1, k.omw, sync);
    else
        line_x_kernel<1><<<grid, LX_THREADS, smem, s>>>(psi, pitch, nlines, t, k.bnd, k.c1, k.omw, sync);
    note_launch();
    return cudaGetLastError();
}

size_t line_y_scratch_doubles(const LineTables& t, int64_t gp) { return (size_t)gp * (size_t)t.N; }

cudaError_t launch_line_y(double* psi, int64_t sa, int64_t sx, int first_line, int count, const LineTables& t, int form,
                          const LineCoefs& k, double* scratch, int64_t gp, cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    const int nl = std::min(LY_THREADS / t.P, line_y_lines(count, device_sms()));
    const int grid = (count + nl - 1) / nl, threads = (nl * t.P + 31) / 32 * 32;
    const size_t smem = (size_t)3 * t.P * nl * sizeof(double);
    if (form == 0)
        launch_after(line_y_kernel<0>, grid, threads, smem, s, psi, sa, sx, first_line, count, nl, t, k.bnd, k.c1, k.omw, k.wc, scratch, gp);
    else
        launch_after(line_y_kernel<1>, grid, threads, smem, s, psi, sa, sx, first_line, count, nl, t, k.bnd, k.c1, k.omw, k.wc, scratch, gp);
    note_launch();
    return cudaGetLastError();
}

}  // namespace lap

// gs_restrict.cuh -- residual and restriction after a Gauss-Seidel black pass, for one grid and batches.
#pragma once

#include "lap_device.cuh"

namespace lap {

// ---- V-cycle steps 2, 3 after Gauss-Seidel smoothing, beta = 1: residual and restriction in one ----
// After a black pass a black point's residual is exactly 0: psi = s / 4 is exact unless it underflows,
// and fma(-4, psi, s) = 0. So only the red residuals are computed, half of all, and the edges of
// the full weighting (all black) are 0: qc = 0.25 (4 c + corners). A black neighbour that is zero,
// subnormal or not finite (its psi may be inexact) sends its coarse point to edges_out_of_line.
// A warp takes 31 coarse columns (lane 0 the odd column to their left) and runs up `rows` coarse rows:
// lane I holds the corner residual at (2 I + 1, 2 J + 1), gets the one at 2 I - 1 by shuffle, and
// carries the pair's sum to the next row. FP64 operations per fine point (the bound): 2.9 against 6
// for a full residual pass and a restriction pass, and the residual never goes to memory.
// 4097^2, level 0: 172 us (114 + 58) -> 101 us.
// (W + E) + (S + N) of the black residuals around `c`; 0 without arithmetic where a black point and
// everything in its equation is zero (a correction or a field that nothing has reached yet).
template <bool HQ>
__device__ __noinline__ double edges_out_of_line(const double* c, const double* q, int64_t p, double one, double nzero)
{
    const FmaOps o{one, nzero};
    auto residual = [&](int64_t d) {
        const double *x = c + d;
        const double W = x[-1], E = x[1], S = x[-p], N = x[p], C = *x, Q = HQ ? q[d] : 0.0;
        unsigned long long any = abs_bits(W) | abs_bits(E) | abs_bits(S) | abs_bits(N) | abs_bits(C);
        if (HQ) any |= abs_bits(Q);
        if (any == 0) return 0.0;
        if (!irregular(C)) return 0.0;
        double s = neighbour_sum<true>(o, W, E, S, N, 1.0);
        if (HQ) s = fadd(o, s, Q);
        return __fma_rn(-4.0, C, s);
    };
    const double W = residual(-1), E = residual(1), S = residual(-p), N = residual(p);
    return fadd(o, fadd(o, W, E), fadd(o, S, N));
}

// acc plus the square of the residual of black point c (beta = 1, no source), out of line: rare, or
// all zero.
static __device__ __noinline__ double black_square(const double* c, int64_t p, double one, double nzero, double acc)
{
    const FmaOps o{one, nzero};
    const unsigned long long any = abs_bits(c[-1]) | abs_bits(c[1]) | abs_bits(c[-p]) | abs_bits(c[p]) | abs_bits(*c);
    if (any == 0) return acc;
    const double r = __fma_rn(-4.0, *c, neighbour_sum<true>(o, c[-1], c[1], c[-p], c[p], 1.0));
    return __fma_rn(r, r, acc);
}

// Coarse column I = 31 seg + lane, coarse rows J0 .. J1 - 1 (1 <= J0, J1 <= nc - 1; the whole warp
// takes part). red: the coarse level's first red pass from zero, ec := (0 + q) / 4 at its red points
// (the black ones untouched); else ec := 0.
template <bool HQ>
__device__ __forceinline__ void gs_restrict_run(const FmaOps& o, const double* __restrict__ u,
                                                const double* __restrict__ q, int mf, int64_t pf,
                                                double* __restrict__ qc, double* __restrict__ ec, int64_t pc, int seg,
                                                int J0, int J1, bool red)
{
    const double four = in_reg(o, 4.0), two = in_reg(o, 2.0);
    const int mc = (mf - 1) / 2 + 1, lane = threadIdx.x & 31, I = 31 * seg + lane;
    if (J0 >= J1) return;  // warp-uniform
    const bool in = I <= mc - 2, out = in && lane > 0;
    // row 2 J at column 2 I of the fine level
    const double* a = u + (int64_t)(2 * J0) * pf + 2 * (in ? I : 1);
    const double* b = HQ ? q + (int64_t)(2 * J0) * pf + 2 * (in ? I : 1) : nullptr;
    // red residual at c, given its south neighbour
    auto residual = [&](const double* c, const double* qq, double W, double S) {
        double s = neighbour_sum<true>(o, W, c[1], S, c[pf], 1.0);
        if (HQ) s = fadd(o, s, *qq);
        return __fma_rn(-four, *c, s);
    };
    // the odd row below the first coarse row; its north neighbours are the row's east ones
    double S = a[-pf];
    double corner = residual(a - pf + 1, b - pf + 1, S, a[-2 * pf + 1]);
    double pair = fadd(o, __shfl_up_sync(0xffffffffu, corner, 1), corner);
    for (int J = J0; J < J1; ++J) {
        const double E = a[1], N = a[pf], W = lane > 0 ? a[-1] : 0.0;
        corner = residual(a + pf + 1, b + pf + 1, N, E);
        const double up = fadd(o, __shfl_up_sync(0xffffffffu, corner, 1), corner);
        if (out) {
            double s = fadd(o, fadd(o, W, E), fadd(o, S, N));
            if (HQ) s = fadd(o, s, *b);
            const double c = __fma_rn(-four, *a, s);
            const double corners = fadd(o, pair, up);
            double v;
            if (irregular(W) || irregular(E) || irregular(S) || irregular(N)) {
                const double e = edges_out_of_line<HQ>(a, b, pf, o.one, o.nzero);
                v = __fma_rn(two, __fma_rn(two, c, e), corners);
            } else {
                v = __fma_rn(four, c, corners);
            }
            v = scale_down_pow2(o, v, 2, 0.25);
            const int64_t at = (int64_t)J * pc + I;
            qc[at] = v;
            if (!red) ec[at] = 0.0;
            else if (((I + J) & 1) == 0) ec[at] = scale_down_pow2(o, plus_zero(v), 2, 0.25);
        }
        S = N;
        pair = up;
        a += 2 * pf;
        if (HQ) b += 2 * pf;
    }
}

}  // namespace lap

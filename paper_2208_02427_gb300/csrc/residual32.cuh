// residual32.cuh -- the mixed solver's residual of FP64 values on the integer pipe (beta = 1).
//
// r = (E + W) + (N + S) - 4 C is four FP64 operations a point, 428 us of FP64 pipe at 8193^2 where the
// field's bytes take 118 us. The sum needs no floating point: a run of RUN_ROWS rows by RUN_COLS columns
// takes the largest exponent of its values (neighbours included), brings each value to 56-bit fixed
// point at that exponent, adds integers, and rounds the sum once to FP32. A value within 2^-3 of the run's
// largest is exact and a smaller one is cut at 2^-55 of the largest, M, so the error before the rounding to FP32 is
// at most 8 2^-55 M = 2^-52 M. The bound of the FP64 expression, which rounds three sums of up to 2 M, 2 M
// and 4 M, is 2^-50 M.
// Runs lie at fixed places of the grid, so a point's residual depends on the field alone, not on the
// launch: the same value from the single-grid and the batched kernels.
// Infinities and NaN, and runs whose largest value is outside about 1e-18 .. 1e35 (FP32 results would leave
// its normal range), take the FP64 expression.
#pragma once

#include "lap_device.cuh"
#include "lap_internal.cuh"

namespace lap {

constexpr int RUN_COLS = 62;  // two columns a lane, the first and the last of the warp's 64 as neighbours

__host__ __device__ inline int run_strips(int m) { return (m - 2 + RUN_COLS - 1) / RUN_COLS; }
__host__ __device__ inline int run_blocks(int n) { return (n - 2 + RUN_ROWS - 1) / RUN_ROWS; }

struct ResidualRuns {
    const double* psi;
    int64_t pitch;
    float* r32;
    float* e32;  // nullable: set to zero
    int64_t pitch32;
    int m, n;
    bool vec;  // rows of psi start on 16-byte boundaries
};

// 56-bit fixed point as two signed parts, h 2^28 + l: sums of parts need no carries, and signs and factors
// go to the multiply pipe. |h|, |l| < 2^28.
struct Fixed {
    int h, l;
};
__device__ __forceinline__ unsigned shr32(unsigned x, int n)  // 0 for n > 31
{
    unsigned r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
    return r;
}
__device__ __forceinline__ unsigned long long shr64(unsigned long long x, int n)  // 0 for n > 63
{
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
}
__device__ __forceinline__ long long shl64(long long x, int n)  // 0 for n > 63
{
    long long r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
}

// x 2^(1078 - E) rounded towards zero, E the run's largest biased exponent.
__device__ __forceinline__ Fixed to_fixed(double x, int E)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int n = E + 4 - (int)((hi >> 20) & 0x7ffu);  // >= 4; a zero's or a subnormal's shifts all out
    const unsigned mh = __funnelshift_l(lo, hi, 11) | 0x80000000u;  // the mantissa, top-aligned in 64 bits
    const unsigned long long mant = ((unsigned long long)mh << 32) | (lo << 11);
    const int sign = ((int)hi >> 31) | 1;
    return Fixed{(int)shr32(mh, n) * sign, (int)((unsigned)shr64(mant, n + 4) & 0xfffffffu) * sign};
}

// 4 neighbours - 4 c, times 2^(E - 1078), rounded once to FP32 (to nearest, ties to even);
// scale = 2^(E - 1046), 963 <= E <= 1140.
__device__ __forceinline__ float from_fixed(const Fixed& w, const Fixed& e, const Fixed& s, const Fixed& n, const Fixed& c,
                                            float scale)
{
    int vh = w.h + e.h + n.h + (s.h - 4 * c.h), vl = w.l + e.l + n.l + (s.l - 4 * c.l);
    // balanced, |vl| <= 2^27: parts that nearly cancel (vl up to 2^31, rounded to FP32) would lose a sum of up to
    // 64 units in its estimate, and with it the whole residual of a field close to its solution
    const int carry = (vl + (1 << 27)) >> 28;
    vh += carry;
    vl -= carry * (1 << 28);
    const long long v = (long long)vh * (1 << 28) + vl;
    // |v| < 2^(k + 2), k the exponent of its FP32 estimate: shifted by 61 - k it fills 29 bits or more of the
    // upper word, and what is below only has to break ties
    const float g = fmaf((float)vh, 268435456.0f, (float)vl);
    const unsigned ex = (unsigned)__float_as_int(g) & 0x7f800000u;  // 0 for v = 0: all shifts out
    const long long t = shl64(v, 188 - (int)(ex >> 23));
    const int top = (int)(t >> 32) | ((unsigned)t != 0u ? 1 : 0);
    return __int2float_rn(top) * __int_as_float((int)ex - (61 << 23)) * scale;
}

// The run of strip s and row block b by the FP64 expression.
static __device__ __noinline__ float residual_run_fp64(const ResidualRuns& R, int s, int b, float scale, float acc)
{
    const FmaOps o = load_fma_ops();
    const double d = in_reg(o, 4.0);
    const int lane = threadIdx.x & 31, y1 = min(1 + RUN_ROWS * (b + 1), R.n - 1);
    for (int j = 1 + RUN_ROWS * b; j < y1; ++j)
        for (int c = lane; c < RUN_COLS; c += 32) {
            const int i = 1 + RUN_COLS * s + c;
            if (i > R.m - 2) continue;
            const double* x = R.psi + (int64_t)j * R.pitch + i;
            const float rf = to_float_rn(__fma_rn(-d, x[0], neighbour_sum<true>(o, x[-1], x[1], x[-R.pitch], x[R.pitch], 1.0)));
            const float rs = __fmul_rn(rf, scale);
            acc = __fmaf_rn(rs, rs, acc);
            R.r32[(int64_t)j * R.pitch32 + i] = rf;
            if (R.e32) R.e32[(int64_t)j * R.pitch32 + i] = 0.0f;
        }
    return acc;
}

// The residuals of the run of strip s and row block b by one warp, into r32; returns acc + the lane's sum of
// (scale r)^2. All of the run's loads are issued before the first is used.
__device__ __forceinline__ float residual_run(const ResidualRuns& R, int s, int b, float scale, float acc)
{
    const int lane = threadIdx.x & 31;
    const int y0 = 1 + RUN_ROWS * b;                 // first row of the run
    const int ca = RUN_COLS * s + 2 * lane, cb = ca + 1;  // the lane's columns
    double xa[RUN_ROWS + 2], xb[RUN_ROWS + 2];
    const double* p = R.psi + (int64_t)(y0 - 1) * R.pitch + ca;
    const bool inside = ca > 0 && cb < R.m - 1;  // both columns off the ring: no corner
#pragma unroll
    for (int k = 0; k < RUN_ROWS + 2; ++k) {
        const int j = y0 - 1 + k;
        xa[k] = xb[k] = 0.0;
        if (j < R.n) {
            if (inside && R.vec) {
                const double2 v = *reinterpret_cast<const double2*>(p + k * R.pitch);
                xa[k] = v.x;
                xb[k] = v.y;
            } else {
                const bool edge = j == 0 || j == R.n - 1;  // corners belong to no stencil
                if (ca < R.m && !(edge && (ca == 0 || ca == R.m - 1))) xa[k] = p[k * R.pitch];
                if (cb < R.m && !(edge && cb == R.m - 1)) xb[k] = p[k * R.pitch + 1];
            }
        }
    }
    // the largest |x| by its upper word, compared as FP32 (the same order; an upper word that is an FP32 NaN,
    // values from about 2^1017 on, infinities and NaN, gives the FP32 NaN)
    float mx = 0.0f;
    auto larger = [&](double x) {
        asm("max.NaN.f32 %0, %0, %1;" : "+f"(mx) : "f"(fabsf(__int_as_float(__double2hiint(x)))));
    };
#pragma unroll
    for (int k = 0; k < RUN_ROWS + 2; ++k) {
        larger(xa[k]);
        larger(xb[k]);
    }
    const int E = (int)(__reduce_max_sync(0xffffffffu, (unsigned)__float_as_int(mx)) >> 20);
    if (E < 963 || E > 1140) return residual_run_fp64(R, s, b, scale, acc);
    const float unit = __int_as_float((E - 1046 + 127) << 23);
    Fixed sa = to_fixed(xa[0], E), sb = to_fixed(xb[0], E);
    Fixed a = to_fixed(xa[1], E), c = to_fixed(xb[1], E);
    const bool outa = lane > 0 && ca <= R.m - 2, outb = lane < 31 && cb <= R.m - 2;
    const float scale_a = outa ? scale : 0.0f, scale_b = outb ? scale : 0.0f;
    float* q = R.r32 + (int64_t)y0 * R.pitch32 + ca;
    const int rows = min(RUN_ROWS, R.n - 1 - y0);
#pragma unroll
    for (int k = 1; k <= RUN_ROWS; ++k) {
        if (k > rows) break;
        const Fixed na = to_fixed(xa[k + 1], E), nb = to_fixed(xb[k + 1], E);
        const Fixed w{__shfl_up_sync(0xffffffffu, c.h, 1), __shfl_up_sync(0xffffffffu, c.l, 1)};
        const Fixed e{__shfl_down_sync(0xffffffffu, a.h, 1), __shfl_down_sync(0xffffffffu, a.l, 1)};
        const float ra = from_fixed(w, c, sa, na, a, unit), rb = from_fixed(a, e, sb, nb, c, unit);
        if (outa && outb) {
            *reinterpret_cast<float2*>(q) = make_float2(ra, rb);
        } else {
            if (outa) q[0] = ra;
            if (outb) q[1] = rb;
        }
        q += R.pitch32;
        const float fa = __fmul_rn(ra, scale_a), fb = __fmul_rn(rb, scale_b);
        acc = __fmaf_rn(fa, fa, acc);
        acc = __fmaf_rn(fb, fb, acc);
        if (R.e32) {
            float* z = R.e32 + (int64_t)(y0 + k - 1) * R.pitch32 + ca;
            if (outa) z[0] = 0.0f;
            if (outb) z[1] = 0.0f;
        }
        sa = a;
        sb = c;
        a = na;
        c = nb;
    }
    return acc;
}

}  // namespace lap

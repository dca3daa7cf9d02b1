// residual32.cuh -- the mixed solver's residual of FP64 values on the integer pipe (beta = 1).
//
// r = (E + W) + (N + S) - 4 C is four FP64 operations a point, 428 us of FP64 pipe at 8193^2 where the
// field's bytes take 118 us. The sum needs no floating point: a run of RUN_ROWS rows by RUN_COLS columns
// takes the largest exponent of its values (neighbours included), brings each value to fixed point at that
// exponent, adds integers, and rounds the sum once to FP32. 60 bits hold every value down to 2^-7 of the
// run's largest whole, 84 bits every value down to 2^-31; a run takes the short form where that cuts none of its
// values (zeros need no bits), else the long one, so the result is the exact residual rounded once, at every point,
// whatever the other values of its run are. (Cut at 2^-55 of the run's largest value instead, a point far below
// that had an error of up to 2^-52 of it, where the FP64 expression rounds relative to the point's own neighbours.)
// Runs with a wider range take the FP64 expression. Share of the runs in the long form: 2% at 4097^2 and 7% at
// 1537 x 1025 of a solved sine ring (where the field changes sign), 3% in a batch of 1024 grids with U[0, 1] rings;
// in the FP64 expression at most 0.1%. (With 56 bits, 2^-3, for the short form the batch had 25% in the long one:
// 7.66 ms a solve against 7.29.)
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

__device__ __forceinline__ long long shl64(long long x, int n)  // 0 for n > 63
{
    long long r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
}

// The short form, x 2^(1082 - E) with E the run's largest biased exponent, |.| < 2^60; and the long one,
// x 2^(1106 - E), in three signed parts (h 2^28 + l) 2^28 + t of less than 2^28, whose sums need no carries.
using Short = long long;
struct Long {
    int h, l, t;
};

// x in fixed point: exact for an exponent from E - 7 (short), E - 31 (long) on, and for zeros.
// (The 1 in front of the fraction by a sign, the lower word's shift as a product: the integer pipe is what bounds
// the kernel.)
__device__ __forceinline__ void to_fixed(double x, int E, Short& f)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int n = E + 4 - (int)((hi >> 20) & 0x7ffu);  // 4 .. 11, more for a zero
    // the mantissa, top-aligned in 64 bits: mh 2^32 + ml
    const unsigned mh = __funnelshift_l(lo, hi, 11) | ((unsigned)(n - 12) & 0x80000000u), ml = lo * 2048u;
    const long long v = (long long)(((unsigned long long)(mh >> (n & 31)) << 32) | __funnelshift_r(ml, mh, n));
    f = (int)hi < 0 ? -v : v;
}
__device__ __forceinline__ void to_fixed(double x, int E, Long& f)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int n = E + 4 - (int)((hi >> 20) & 0x7ffu);  // 4 .. 35, more for a zero
    const unsigned mh = __funnelshift_l(lo, hi, 11) | ((unsigned)(n - 36) & 0x80000000u), ml = lo * 2048u;
    // shifted right by n - 4: 96 bits, of which the upper 84 are the three parts
    const unsigned w2 = mh >> ((n - 4) & 31), w1 = __funnelshift_r(ml, mh, n - 4), w0 = __funnelshift_r(0u, ml, n - 4);
    const int sign = ((int)hi >> 31) | 1;
    f = Long{(int)(w2 >> 4) * sign, (int)(__funnelshift_r(w1, w2, 8) & 0xfffffffu) * sign,
             (int)(__funnelshift_r(w0, w1, 12) & 0xfffffffu) * sign};
}

// 4 neighbours - 4 c, rounded once to FP32 (to nearest, ties to even); unit = 2^(E - 1082), 963 <= E <= 1140.
__device__ __forceinline__ float from_fixed(Short w, Short e, Short s, Short n, Short c, float unit)
{
    const long long v = (w + e) + n + (s - 4 * c);
    // An FP32 estimate g of v for its exponent k. The lower word is taken signed, so that where the words nearly
    // cancel (a residual close to 0) it is v itself. g does not fall where v rises, and powers of two are exact, so
    // |v| < 2^(k + 1): shifted by 62 - k it fills 30 bits or more of the upper word, and what is below only has to
    // break ties. (g rounds up to 2^63 at most: no shift. v = 0: all shifts out.)
    const int lo = (int)v;
    const float g = fmaf((float)((int)(v >> 32) + (int)((unsigned)lo >> 31)), 4294967296.0f, (float)lo);
    const int sh = max(0, 127 + 62 - ((__float_as_int(g) >> 23) & 0xff));
    const long long t = shl64(v, sh);
    const int top = (int)(t >> 32) | ((unsigned)t != 0u ? 1 : 0);
    return __int2float_rn(top) * __uint_as_float((unsigned)(127 + 32 - sh) << 23) * unit;
}
// The same from the long form; 982 <= E <= 1140.
__device__ __forceinline__ float from_fixed(const Long& w, const Long& e, const Long& s, const Long& n, const Long& c,
                                            float unit)
{
    const int vh = w.h + e.h + n.h + (s.h - 4 * c.h), vl = w.l + e.l + n.l + (s.l - 4 * c.l),
              vt = w.t + e.t + n.t + (s.t - 4 * c.t);
    const long long v = (long long)vh * (1 << 28) + vl + (vt >> 28);  // and 28 bits below, low
    const int low = vt & 0xfffffff;
    // all of it where it is short, else what is below only has to break ties
    const bool all = v + (1ll << 34) >= 0 && v < 1ll << 34;
    const long long x = all ? v * (1 << 28) + low : 2 * v + (low ? 1 : 0);
    return __ll2float_rn(x) * (unit * (all ? 0x1p-24f : 0x1p3f));
}

// The neighbouring lane's value (up: of the lane below).
__device__ __forceinline__ Short from_lane(Short f, bool up)
{
    return up ? __shfl_up_sync(0xffffffffu, f, 1) : __shfl_down_sync(0xffffffffu, f, 1);
}
__device__ __forceinline__ Long from_lane(const Long& f, bool up)
{
    auto shfl = [&](int v) { return up ? __shfl_up_sync(0xffffffffu, v, 1) : __shfl_down_sync(0xffffffffu, v, 1); };
    return Long{shfl(f.h), shfl(f.l), shfl(f.t)};
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

// The lane's two values (columns ca, ca + 1) of row j, at p; zeros outside the grid. inside: both columns off the
// ring: no corner.
__device__ __forceinline__ double2 run_values(const ResidualRuns& R, const double* p, int j, int ca, bool inside)
{
    if (j >= R.n) return make_double2(0.0, 0.0);
    if (inside && R.vec) return *reinterpret_cast<const double2*>(p);
    const bool edge = j == 0 || j == R.n - 1;  // corners belong to no stencil
    double2 v = make_double2(0.0, 0.0);
    if (ca < R.m && !(edge && (ca == 0 || ca == R.m - 1))) v.x = p[0];
    if (ca + 1 < R.m && !(edge && ca + 1 == R.m - 1)) v.y = p[1];
    return v;
}

// Residuals ra, rb of the lane's columns into r32 at q (and zeros into e32 at z); returns acc + the sum of
// (scale r)^2 over those that are the lane's own.
__device__ __forceinline__ float put_residuals(float ra, float rb, bool outa, bool outb, float* q, float* z, float scale_a,
                                               float scale_b, float acc)
{
    if (outa && outb) {
        *reinterpret_cast<float2*>(q) = make_float2(ra, rb);
    } else {
        if (outa) q[0] = ra;
        if (outb) q[1] = rb;
    }
    if (z) {
        if (outa) z[0] = 0.0f;
        if (outb) z[1] = 0.0f;
    }
    const float fa = __fmul_rn(ra, scale_a), fb = __fmul_rn(rb, scale_b);
    acc = __fmaf_rn(fa, fa, acc);
    return __fmaf_rn(fb, fb, acc);
}

// The lane's values (columns ca, ca + 1) of the run whose first row is y0, all loads issued before the first is used.
__device__ __forceinline__ void load_run(const ResidualRuns& R, int y0, int ca, double (&xa)[RUN_ROWS + 2],
                                         double (&xb)[RUN_ROWS + 2])
{
    const double* p = R.psi + (int64_t)(y0 - 1) * R.pitch + ca;
    const bool inside = ca > 0 && ca + 1 < R.m - 1;
#pragma unroll
    for (int k = 0; k < RUN_ROWS + 2; ++k) {
        const double2 v = run_values(R, p + k * R.pitch, y0 - 1 + k, ca, inside);
        xa[k] = v.x;
        xb[k] = v.y;
    }
}

// residual_run from the values and their largest exponent, in one of the forms.
template <class F>
__device__ __forceinline__ float residual_rows(const ResidualRuns& R, const double (&xa)[RUN_ROWS + 2],
                                               const double (&xb)[RUN_ROWS + 2], int E, int y0, int ca, float scale, float acc)
{
    const int lane = threadIdx.x & 31, cb = ca + 1;
    const float unit = __int_as_float((E - 1082 + 127) << 23);
    F sa, sb, a, c, na, nb;
    to_fixed(xa[0], E, sa);
    to_fixed(xb[0], E, sb);
    to_fixed(xa[1], E, a);
    to_fixed(xb[1], E, c);
    const bool outa = lane > 0 && ca <= R.m - 2, outb = lane < 31 && cb <= R.m - 2;
    const float scale_a = outa ? scale : 0.0f, scale_b = outb ? scale : 0.0f;
    const int64_t at = (int64_t)y0 * R.pitch32 + ca;
    float* q = R.r32 + at;
    const int rows = min(RUN_ROWS, R.n - 1 - y0);
#pragma unroll
    for (int k = 1; k <= RUN_ROWS; ++k) {
        if (k > rows) break;
        to_fixed(xa[k + 1], E, na);
        to_fixed(xb[k + 1], E, nb);
        const F w = from_lane(c, true), e = from_lane(a, false);
        float* z = R.e32 ? R.e32 + at + (int64_t)(k - 1) * R.pitch32 : nullptr;
        acc = put_residuals(from_fixed(w, c, sa, na, a, unit), from_fixed(a, e, sb, nb, c, unit), outa, outb, q, z, scale_a,
                            scale_b, acc);
        q += R.pitch32;
        sa = a;
        sb = c;
        a = na;
        c = nb;
    }
    return acc;
}

// The residuals of the run of strip s and row block b by one warp, into r32; returns acc + the lane's sum of
// (scale r)^2.
__device__ __forceinline__ float residual_run(const ResidualRuns& R, int s, int b, float scale, float acc)
{
    const int y0 = 1 + RUN_ROWS * b, ca = RUN_COLS * s + 2 * (threadIdx.x & 31);
    double xa[RUN_ROWS + 2], xb[RUN_ROWS + 2];
    load_run(R, y0, ca, xa, xb);
    // the largest |x| by its upper word, compared as FP32 (the same order; an upper word that is an FP32 NaN,
    // values from about 2^1017 on, infinities and NaN, gives the FP32 NaN), and the smallest
    float mx = 0.0f, mn = __int_as_float(0x7f800000);
#pragma unroll
    for (int k = 0; k < RUN_ROWS + 2; ++k) {
        const float fa = fabsf(__int_as_float(__double2hiint(xa[k]))), fb = fabsf(__int_as_float(__double2hiint(xb[k])));
        asm("max.NaN.f32 %0, %0, %1, %2;" : "+f"(mx) : "f"(fa), "f"(fb));
        asm("min.f32 %0, %0, %1, %2;" : "+f"(mn) : "f"(fa), "f"(fb));
    }
    const int E = (int)(__reduce_max_sync(0xffffffffu, (unsigned)__float_as_int(mx)) >> 20);
    if (E < 963 || E > 1140) return residual_run_fp64(R, s, b, scale, acc);
    if ((int)(__reduce_min_sync(0xffffffffu, (unsigned)__float_as_int(mn)) >> 20) < E - 7) {
        // zeros aside: less 1, a zero's upper word is the largest
        unsigned nz = ~0u;
        auto smaller = [&](double x) {
            nz = min(nz, (((unsigned)__double2hiint(x) & 0x7fffffffu) | (__double2loint(x) ? 1u : 0u)) - 1u);
        };
#pragma unroll
        for (int k = 0; k < RUN_ROWS + 2; ++k) {
            smaller(xa[k]);
            smaller(xb[k]);
        }
        const int least = (int)(__reduce_min_sync(0xffffffffu, nz) >> 20);
        if (least < E - 31 || (least < E - 7 && E < 982)) return residual_run_fp64(R, s, b, scale, acc);
        if (least < E - 7) return residual_rows<Long>(R, xa, xb, E, y0, ca, scale, acc);
    }
    return residual_rows<Short>(R, xa, xb, E, y0, ca, scale, acc);
}

}  // namespace lap

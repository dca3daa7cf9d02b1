// loop_kernels.cu -- the device-side stopping test of a solve loop, and a self-check.
//
// loop_decide_kernel runs inside the body of a conditional CUDA graph node: after each check
// period it applies the host loop's stopping rule of Eq. 16 and sets the loop's condition.
// setup_kernel puts a solve's small state on the device. check_rounding_kernel compares the residual kernels' integer-pipe
// FP64 -> FP32 rounding with the conversion instruction. fp64_rate_kernel measures the FP64
// fused multiply-add issue rate, the peak that the FP64-bound kernels are measured against.
#include <algorithm>

#include "lap_device.cuh"
#include "lap_internal.cuh"
#include "norm_end.cuh"

namespace lap {

namespace {

// The stopping test of Eq. 16 in a device-resident solve loop, after each period inside the body of a
// conditional CUDA graph (the L2 rules are taken at the end of the norm kernels, norm_end.cuh).
__global__ void loop_decide_kernel(LoopState* st, const unsigned long long* __restrict__ maxd,
                                   cudaGraphConditionalHandle h)
{
    if (threadIdx.x != 0) return;
    const bool on = loop_test(st, st->last_nr, __longlong_as_double((long long)*maxd));
    cudaGraphSetConditional(h, on ? 1u : 0u);
}

// SolveSetup: block row l takes the ring of level l (row 0, row n - 1, columns 0 and m - 1).
template <class T>
__global__ void setup_kernel(const SolveSetup<T> a)
{
    if (blockIdx.x == 0 && blockIdx.y == 0) {
        if (threadIdx.x == 0) {
            a.wslot[0] = a.w;
            a.wslot[1] = a.omw;
            *a.loop = a.state;
            *a.done = 0u;
        }
        for (int l = threadIdx.x; l < a.levels; l += blockDim.x) {
            a.lv[l] = a.level[l];
            a.jobs[l] = TailJob{l, a.levels - 1};
        }
    }
    const int l = blockIdx.y;
    if (l >= a.levels || l < a.rings) return;
    const BatchLevel<T>& V = a.level[l];
    const int m = V.m, n = V.n;
    for (int64_t k = blockIdx.x * blockDim.x + threadIdx.x; k < 2 * ((int64_t)m + n); k += gridDim.x * blockDim.x) {
        int64_t at;
        if (k < m) at = k;
        else if (k < 2 * (int64_t)m) at = (int64_t)(n - 1) * V.pitch + (k - m);
        else if (k < 2 * (int64_t)m + n) at = (k - 2 * (int64_t)m) * V.pitch;
        else at = (k - 2 * (int64_t)m - n) * V.pitch + (m - 1);
        V.u[at] = (T)0;
        if (V.q) V.q[at] = (T)0;
        if (V.r) V.r[at] = (T)0;
    }
}

// The loop test of a device-resident batched solve, run before the loop (first) and after each cycle
// inside the body of a conditional CUDA graph: st[0] counts the cycles, st[1] is the cap; the loop goes
// on while some problem is still running (the convergence kernel counts them down) and the cap is not
// reached.
__global__ void batch_loop_decide_kernel(long long* st, const int* __restrict__ remaining,
                                         cudaGraphConditionalHandle h, int first)
{
    if (threadIdx.x != 0) return;
    const long long k = st[0] + (first ? 0 : 1);
    st[0] = k;
    cudaGraphSetConditional(h, *remaining > 0 && k < st[1] ? 1u : 0u);
}

// dst's ring := src's.
__global__ void copy_ring_kernel(double* __restrict__ dst, const double* __restrict__ src, int m, int n, int64_t pitch)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= 2 * ((int64_t)m + n)) return;
    int64_t at;
    if (k < m) at = k;
    else if (k < 2 * (int64_t)m) at = (n - 1) * pitch + (k - m);
    else if (k < 2 * (int64_t)m + n) at = (k - 2 * (int64_t)m) * pitch;
    else at = (k - 2 * (int64_t)m - n) * pitch + (m - 1);
    dst[at] = src[at];
}

// The rings of the u, q and r buffers of a batch's levels set to zero, a block per level (level 0 of
// an FP64 problem, the caller's field, has no q and is left alone).
template <class T>
__global__ void zero_rings_kernel(const BatchLevel<T>* __restrict__ lv)
{
    const BatchLevel<T> V = lv[blockIdx.x];
    if (!V.q) return;
    const int64_t m = V.m, n = V.n;
    for (int64_t k = threadIdx.x; k < 2 * (m + n); k += blockDim.x) {
        int64_t at;
        if (k < m) at = k;
        else if (k < 2 * m) at = (n - 1) * V.pitch + (k - m);
        else if (k < 2 * m + n) at = (k - 2 * m) * V.pitch;
        else at = (k - 2 * m - n) * V.pitch + (m - 1);
        V.u[at] = (T)0;
        V.q[at] = (T)0;
        if (V.r) V.r[at] = (T)0;
    }
}

}  // namespace

namespace {

__device__ __forceinline__ unsigned long long mix64(unsigned long long x)
{
    x += 0x9e3779b97f4a7c15ull;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
    return x ^ (x >> 31);
}

// to_float_rn against the conversion instruction, and scale_down_pow2 against the FP64
// multiply by 2^-s (s = 1..4), on `count` doubles drawn from seed: random bit patterns,
// exponents near the FP32 range's ends, exact ties, all-ones fractions, +-0 and FP64
// subnormals, and exponents within a few of zero, in turn; and to_double_exact against the
// conversion on random FP32 bit patterns, every eighth one with a zero exponent (+-0 or
// an FP32 subnormal).
__global__ void check_rounding_kernel(long long count, unsigned long long seed,
                                      unsigned long long* bad)
{
    const FmaOps o = load_fma_ops();
    unsigned long long local = 0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < count;
         k += (long long)gridDim.x * blockDim.x) {
        const unsigned long long r = mix64(seed ^ (unsigned long long)k), r2 = mix64(r);
        const unsigned long long sign_frac = r & 0x800fffffffffffffull;
        unsigned long long b;
        switch (k % 6) {
        case 0: b = r; break;
        case 1: b = sign_frac | ((unsigned long long)(1023 - 130 + (r2 % 270)) << 52); break;
        case 2: b = (r & 0x800fffffe0000000ull) | 0x10000000ull | ((unsigned long long)(1023 + (int)(r2 % 60) - 30) << 52); break;
        case 3: b = (r & 0xfff0000000000000ull) | 0x000fffffffffffffull; break;
        case 4: b = (r2 & 3) ? (r & 0x8000000000000000ull) : sign_frac; break;  // +-0, subnormal
        default: b = sign_frac | ((r2 % 8) << 52); break;
        }
        const double x = __longlong_as_double((long long)b);
        const float want = __double2float_rn(x), got = to_float_rn(x);
        if (__float_as_uint(want) != __float_as_uint(got) && !(want != want && got != got)) ++local;
        const float f = __uint_as_float((unsigned int)(k & 7 ? r2 >> 32 : (r2 >> 32) & 0x807fffffu));
        const double fw = (double)f, fg = to_double_exact(f);
        if (__double_as_longlong(fw) != __double_as_longlong(fg) && !(fw != fw && fg != fg))
            ++local;
        const int s = 1 + (int)((r2 >> 8) & 3);
        const double p = __hiloint2double((1023 - s) << 20, 0);  // 2^-s
        const double wd = __dmul_rn(x, p), gd = scale_down_pow2(o, x, s, p);
        if (__double_as_longlong(wd) != __double_as_longlong(gd) && !(wd != wd && gd != gd))
            ++local;
    }
    if (local) atomicAdd(bad, local);
}

// FP64 issue-rate probe: every thread runs CHAINS independent recurrences x = fma(x, a, b)
// for `iters` steps, with a and b in registers (in_reg; constant-bank operands issue slower,
// see lap_device.cuh), so the FP64 pipe never waits on a dependency once a few warps per SM
// are resident. fmas issued = threads * CHAINS * iters. The result is stored only when it
// equals an impossible value, which keeps the chains live.
constexpr int RATE_CHAINS = 8;
__global__ void __launch_bounds__(256)
    fp64_rate_kernel(long long iters, double a, double b, double* __restrict__ sink)
{
    const FmaOps o = load_fma_ops();
    a = in_reg(o, a);
    b = in_reg(o, b);
    double x[RATE_CHAINS];
#pragma unroll
    for (int k = 0; k < RATE_CHAINS; ++k) x[k] = (double)(threadIdx.x + 32 * k) * 1e-3;
    for (long long t = 0; t < iters; ++t) {
#pragma unroll
        for (int k = 0; k < RATE_CHAINS; ++k) x[k] = __fma_rn(x[k], a, b);
    }
    double acc = x[0];
#pragma unroll
    for (int k = 1; k < RATE_CHAINS; ++k) acc = fmax(acc, x[k]);
    if (acc == -1.0) sink[blockIdx.x] = acc;
}

}  // namespace

int64_t launch_fp64_rate(int blocks, long long iters, double* sink, cudaStream_t s)
{
    // a < 1, b > 0: every chain tends to b / (1 - a) = 1, no overflow or subnormals
    fp64_rate_kernel<<<blocks, 256, 0, s>>>(iters, 0.999999, 1e-6, sink);
    note_launch();
    if (cudaGetLastError() != cudaSuccess) return -1;
    return (int64_t)blocks * 256 * RATE_CHAINS * iters;
}

cudaError_t launch_check_rounding(long long count, unsigned long long seed, unsigned long long* bad,
                                  cudaStream_t s)
{
    check_rounding_kernel<<<152 * 8, 256, 0, s>>>(count, seed, bad);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_batch_loop_decide(long long* st, const int* remaining, cudaGraphConditionalHandle h,
                                     bool first, cudaStream_t s)
{
    batch_loop_decide_kernel<<<1, 32, 0, s>>>(st, remaining, h, first ? 1 : 0);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_copy_ring(double* dst, const Field& src, cudaStream_t s)
{
    const int64_t points = 2 * ((int64_t)src.m + src.n);
    copy_ring_kernel<<<(unsigned)((points + 255) / 256), 256, 0, s>>>(dst, src.p, src.m, src.n, src.pitch);
    note_launch();
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_zero_rings(const BatchLevel<T>* lv, int count, cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    zero_rings_kernel<T><<<count, 256, 0, s>>>(lv);
    note_launch();
    return cudaGetLastError();
}
template cudaError_t launch_zero_rings<double>(const BatchLevel<double>*, int, cudaStream_t);
template cudaError_t launch_zero_rings<float>(const BatchLevel<float>*, int, cudaStream_t);

cudaError_t launch_loop_decide(LoopState* st, const unsigned long long* maxd, cudaGraphConditionalHandle h,
                               cudaStream_t s)
{
    loop_decide_kernel<<<1, 32, 0, s>>>(st, maxd, h);
    note_launch();
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_setup(const SolveSetup<T>& a, cudaStream_t s)
{
    int64_t side = 0;
    for (int l = a.rings; l < a.levels; ++l) side = std::max<int64_t>(side, (int64_t)a.level[l].m + a.level[l].n);
    const int x = (int)std::min<int64_t>(64, std::max<int64_t>(1, (2 * side + 255) / 256));
    setup_kernel<T><<<dim3(x, std::max(1, a.levels)), 256, 0, s>>>(a);
    note_launch();
    return cudaGetLastError();
}
template cudaError_t launch_setup<double>(const SolveSetup<double>&, cudaStream_t);
template cudaError_t launch_setup<float>(const SolveSetup<float>&, cudaStream_t);

}  // namespace lap

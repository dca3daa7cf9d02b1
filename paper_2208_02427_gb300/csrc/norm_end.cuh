// norm_end.cuh -- the end of a norm kernel: the last block to finish sums the blocks' partial sums of
// squares and, in a device-resident solve loop, takes the stopping test.
//
// The sum and the test each had a launch of their own. On small grids a launch costs more than they do
// (about 3.5 us a kernel in the body of a conditional graph), so the block that finishes last takes
// them over. It sums in sum_partials_kernel's order (256 threads, the same trees), so the norm is the
// same bit for bit.
#pragma once

#include "lap_device.cuh"
#include "lap_internal.cuh"

namespace lap {

// The sum of partials[0 .. count) by 256 threads, valid in thread 0.
__device__ __forceinline__ double sum_partials_256(const double* partials, int count, double* red)
{
    double acc = 0.0;
    for (int k = threadIdx.x; k < count; k += 256) acc = __dadd_rn(acc, __ldcg(partials + k));
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    double v = 0.0;
    if (threadIdx.x < 32) v = warp_sum(threadIdx.x < 8 ? red[threadIdx.x] : 0.0);
    return v;
}

// The stopping test after a period (Eq. 16 when mode is 2, else the L2 rules on the norm nr): the host
// loop's arithmetic. Returns whether the loop goes on.
__device__ __forceinline__ bool loop_test(LoopState* st, double nr, double maxd)
{
    st->k += st->steps;
    const double val = st->mode == 2 ? maxd : (st->mode == 0 ? nr / st->r0 : nr);
    const bool conv = st->mode == 0 ? nr <= st->tol * st->r0 : val <= st->tol;
    st->last_check = val;
    st->last_nr = nr;
    const int status = !isfinite(val) ? 2 : (conv ? 0 : 1);  // LAP_DIVERGED, LAP_CONVERGED, LAP_MAXITER
    st->status = status;
    return status == 1 && st->k + st->steps <= st->max_iter;
}

// The first residual of a solve: r0, the solves that end there, and the mixed solver's norm scale
// (2^-e with r0 = f 2^e). An r0 out of the scale's range ends the loop with status LOOP_NO_SCALE: the
// host goes on with FP64 sums.
__device__ __forceinline__ bool loop_first(LoopState* st, double r0, float* scale)
{
    st->r0 = st->last_nr = r0;
    int status = 1;
    if (!isfinite(r0)) status = 2;
    else if ((st->mode == 0 && r0 == 0.0) || (st->mode == 1 && r0 <= st->tol)) status = 0;
    if (scale && status == 1) {
        const int e = ilogb(r0);
        if (r0 > 0.0 && e >= -100 && e <= 100) *scale = ldexpf(1.0f, -e);
        else status = LOOP_NO_SCALE;
    }
    st->status = status;
    return status == 1 && st->k + st->steps <= st->max_iter;
}

// v: this block's sum of squares (thread 0). Blocks of 256 threads; red: 8 doubles of shared memory
// that the block no longer needs.
__device__ __forceinline__ void norm_end(const NormEnd& e, double v, double* partials, double* red)
{
    if (threadIdx.x == 0) partials[blockIdx.x] = v;
    if (!e.done) return;
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(e.done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const double s = sum_partials_256(partials, gridDim.x, red);
    if (threadIdx.x != 0) return;
    *e.done = 0u;  // for the next norm on the stream
    const double nr = sqrt(s);
    e.nrm[0] = s;
    e.nrm[1] = nr;
    if (!e.loop) return;
    bool on;
    if (e.first) on = loop_first(e.loop, nr, e.scale_out);
    else on = loop_test(e.loop, e.scale ? nr / (double)*e.scale : nr, 0.0);
    cudaGraphSetConditional(e.handle, on ? 1u : 0u);
}

}  // namespace lap

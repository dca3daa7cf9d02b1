// vcycle_arith.cuh -- the V-cycle's arithmetic in one precision, shared by the kernels that run the
// cycle over many grids and the small-level tail: the single-grid kernels' expressions.
#pragma once

#include <type_traits>

#include "lap_device.cuh"
#include "lap_internal.cuh"

namespace lap {

// Arithmetic of one precision, matching the single-grid kernels of that precision.
template <class T> struct Arith;
template <> struct Arith<double> {
    FmaOps o;
    __device__ double add(double a, double b) const { return fadd(o, a, b); }
    __device__ double mul(double a, double b) const { return fmul(o, a, b); }
    __device__ double fma(double a, double b, double c) const { return __fma_rn(a, b, c); }
    template <bool UNIT>
    __device__ double nsum(double w, double e, double s, double n, double b2) const
    {
        return neighbour_sum<UNIT>(o, w, e, s, n, b2);
    }
    template <bool POW2>
    __device__ double inv_d(double s, const BatchLevel<double>& L) const
    {
        return times_inv_d<POW2>(o, s, L.inv_d, L.inv_d_shift);
    }
    __device__ double half(double x) const { return scale_down_pow2(o, x, 1, 0.5); }
    __device__ double quarter(double x) const { return scale_down_pow2(o, x, 2, 0.25); }
    __device__ double two() const { return in_reg(o, 2.0); }
};
template <> struct Arith<float> {
    __device__ float add(float a, float b) const { return __fadd_rn(a, b); }
    __device__ float mul(float a, float b) const { return __fmul_rn(a, b); }
    __device__ float fma(float a, float b, float c) const { return __fmaf_rn(a, b, c); }
    template <bool UNIT>
    __device__ float nsum(float w, float e, float s, float n, float b2) const
    {
        const float ew = __fadd_rn(w, e), ns = __fadd_rn(s, n);
        return UNIT ? __fadd_rn(ns, ew) : __fmaf_rn(b2, ns, ew);
    }
    template <bool POW2>
    __device__ float inv_d(float s, const BatchLevel<float>& L) const
    {
        return __fmul_rn(s, (float)L.inv_d);
    }
    __device__ float half(float x) const { return __fmul_rn(0.5f, x); }
    __device__ float quarter(float x) const { return __fmul_rn(0.25f, x); }
    __device__ float two() const { return 2.0f; }
};

template <class T>
__device__ __forceinline__ Arith<T> arith();
template <>
__device__ __forceinline__ Arith<double> arith<double>() { return Arith<double>{load_fma_ops()}; }
template <>
__device__ __forceinline__ Arith<float> arith<float>() { return Arith<float>{}; }

// A flag that is uniform over a block (a level's beta == 1, 1/d a power of two, a source
// term, GS or SOR) becomes a template argument: the loop is compiled once per value. Left a
// run-time choice inside the per-point code, the compiler evaluates both sides of the short
// FP64 branch and selects, one FP64 operation more per point (measured: the batched FP64
// residual norm at 89% FP64-pipe occupancy for half its useful throughput).
template <class F>
__device__ __forceinline__ void on_flag(bool a, F&& f)
{
    if (a) f(std::true_type{});
    else f(std::false_type{});
}

}  // namespace lap

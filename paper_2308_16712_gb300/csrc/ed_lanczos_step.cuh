// ed_lanczos_step.cuh -- the vector part of a Lanczos step over a short vector in
// one block: alpha = Re<v, w>, w -= alpha v + beta vp, beta' = |w|, vn = w / beta',
// shared by the single- and many-sector solvers.
//
// A step of separate kernels (dot, update with norm, normalise, counter) over a
// few thousand elements takes three launches and their reductions' latency --
// compensated merges are chains of fp64 additions of some 80 cycles each --
// three times over: 34 us at 2518 states, 110 us for 100 sectors of 9000.  One
// block of 1024 threads per vector takes the two reductions back to back.
// Up to kFusedMax elements; beyond, one SM's load bandwidth is the bound.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

namespace edk {

constexpr int kFusedThreads = 1024;
constexpr unsigned long long kFusedMax = 16384;

struct StepSum {
    double s, c;
};

__device__ __forceinline__ StepSum step_two_sum(double a, double b)
{
    const double s = a + b, bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ StepSum step_merge(StepSum a, StepSum b)
{
    StepSum r = step_two_sum(a.s, b.s);
    r.c += a.c + b.c;
    return r;
}

// the compensated sum over the block, in every thread (fixed tree)
__device__ __forceinline__ double step_block_sum(StepSum k)
{
    __shared__ StepSum part[kFusedThreads / 32];
    __shared__ double total;
    for (int o = 16; o > 0; o >>= 1)
        k = step_merge(k, StepSum{__shfl_down_sync(0xffffffffu, k.s, o), __shfl_down_sync(0xffffffffu, k.c, o)});
    if ((threadIdx.x & 31) == 0)
        part[threadIdx.x >> 5] = k;
    __syncthreads();
    if (threadIdx.x < 32) {
        k = part[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1)
            k = step_merge(k, StepSum{__shfl_down_sync(0xffffffffu, k.s, o), __shfl_down_sync(0xffffffffu, k.c, o)});
        if (threadIdx.x == 0)
            total = k.s + k.c;
    }
    __syncthreads();
    return total;
}

__device__ __forceinline__ double step_re_dot(double a, double b) { return a * b; }
__device__ __forceinline__ double step_re_dot(double2 a, double2 b) { return fma(a.x, b.x, a.y * b.y); }
__device__ __forceinline__ double step_up(double a) { return a; }
__device__ __forceinline__ double step_up(float a) { return (double)a; }
__device__ __forceinline__ double2 step_up(double2 a) { return a; }
__device__ __forceinline__ double2 step_up(float2 a) { return make_double2(a.x, a.y); }
__device__ __forceinline__ double step_axpby(double w, double a, double v, double b, double p)
{
    return fma(-b, p, fma(-a, v, w));
}
__device__ __forceinline__ double2 step_axpby(double2 w, double a, double2 v, double b, double2 p)
{
    return make_double2(step_axpby(w.x, a, v.x, b, p.x), step_axpby(w.y, a, v.y, b, p.y));
}
__device__ __forceinline__ double step_scale(double w, double s) { return w * s; }
__device__ __forceinline__ double2 step_scale(double2 w, double s) { return make_double2(w.x * s, w.y * s); }
__device__ __forceinline__ void step_down(float *o, double a) { *o = (float)a; }
__device__ __forceinline__ void step_down(float2 *o, double2 a) { *o = make_float2((float)a.x, (float)a.y); }

// One step of n elements by one block of kFusedThreads.  vp null: first step
// (beta[0] unused).  alpha[0], beta[1] and vn are written; x32, keep64, keep32
// get copies of vn where given.  w may be w_in.
template <typename D, typename F, typename WI>
__device__ __forceinline__ void lanczos_step(unsigned long long n, const WI *w_in, D *w, const D *v, const D *vp, D *vn,
                                             F *x32, D *keep64, F *keep32, double *alpha, double *beta)
{
    double s0 = 0.0, s1 = 0.0;
    unsigned long long i = threadIdx.x;
    for (; i + kFusedThreads < n; i += 2 * kFusedThreads) {
        const D a0 = v[i], a1 = v[i + kFusedThreads];
        const D b0 = step_up(w_in[i]), b1 = step_up(w_in[i + kFusedThreads]);
        s0 += step_re_dot(a0, b0);
        s1 += step_re_dot(a1, b1);
    }
    if (i < n)
        s0 += step_re_dot(v[i], step_up(w_in[i]));
    const double a = step_block_sum(step_two_sum(s0, s1));
    const double b = vp ? beta[0] : 0.0;
    s0 = s1 = 0.0;
    for (i = threadIdx.x; i < n; i += 2 * kFusedThreads) {
        const unsigned long long j = i + kFusedThreads;
        const D r = step_axpby(step_up(w_in[i]), a, v[i], b, vp ? vp[i] : D{});
        w[i] = r;
        s0 += step_re_dot(r, r);
        if (j < n) {
            const D q = step_axpby(step_up(w_in[j]), a, v[j], b, vp ? vp[j] : D{});
            w[j] = q;
            s1 += step_re_dot(q, q);
        }
    }
    const double nrm = sqrt(fmax(step_block_sum(step_two_sum(s0, s1)), 0.0));
    const double sc = nrm > 0.0 ? 1.0 / nrm : 0.0;
    for (i = threadIdx.x; i < n; i += kFusedThreads) {
        const D r = step_scale(w[i], sc);
        vn[i] = r;  // may be vp's buffer: read above by this thread only
        if (x32)
            step_down(x32 + i, r);
        if (keep64)
            keep64[i] = r;
        if (keep32)
            step_down(keep32 + i, r);
    }
    if (threadIdx.x == 0) {
        alpha[0] = a;
        beta[1] = nrm;
    }
}

}  // namespace edk

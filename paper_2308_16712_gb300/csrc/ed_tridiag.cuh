// ed_tridiag.cuh -- eigenvalues of small symmetric tridiagonal matrices by
// multisection with Sturm counts, and the lowest eigenvector by inverse
// iteration, one block per matrix: shared by the single- and many-sector Lanczos
// solvers.
//
// Bound by chains of fp64 operations (a division takes some 900 cycles on this
// GPU, a multiply-add some 80, and an SM sub-partition starts one for a warp
// every 75), not by work: a count is one block-wide evaluation with one warp per
// sub-partition, so a round brackets an eigenvalue 129 times more narrowly
// instead of 33 times; the counts use the division-free form of the sequence;
// the pivots of the inverse iteration are divided out once instead of in each of
// its passes; and its chains run on shared memory.  Matrices of 50 and of 6 steps
// together: 0.65 -> 0.21 ms (0.29 with 256 threads and the chains in memory).
#pragma once

#include <cuda_runtime.h>

namespace edk {

constexpr int kTriThreads = 128;
constexpr int kTriShared = 768;  // matrices up to this size are worked on in shared memory

// Number of eigenvalues below x: sign changes of p_0 = 1, p_1 = a_0 - x,
// p_{i+1} = (a_i - x) p_i - b_i^2 p_{i-1} (b2[i] = b_i^2 couples i-1 and i),
// rescaled every fourth step; a vanishing p_i takes the sign that counts.  The
// computed sequence is the exact one of a matrix whose entries differ by a few
// roundings, as for the quotients p_i / p_{i-1}.  The entries are to be of order
// one, or four steps leave the range of a double: a[i] f is the diagonal, and b2
// and x are scaled alike by the caller.
__device__ __forceinline__ int tri_count(const double *a, double f, const double *b2, int m, double x)
{
    double p0 = 1.0, p1 = fma(a[0], f, -x);
    bool neg = p1 <= 0.0;
    int cnt = neg ? 1 : 0;
    for (int i = 1; i < m; ++i) {
        const double t = b2[i] * p0;
        const double p2 = fma(fma(a[i], f, -x), p1, -t);
        p0 = p1;
        p1 = p2;
        const bool s = p1 == 0.0 ? !neg : p1 < 0.0;
        cnt += s != neg ? 1 : 0;
        neg = s;
        if ((i & 3) == 0) {  // divide both by the power of two of the larger
            const int e = (int)((max((unsigned)__double2hiint(fabs(p0)), (unsigned)__double2hiint(fabs(p1))) >> 20) & 0x7ffu);
            const double r = __hiloint2double(max(1, min(2045, 2046 - e)) << 20, 0);
            p0 *= r;
            p1 *= r;
        }
    }
    return cnt;
}

// Bracket of eigenvalue number k (0 = lowest) of the leading m x m matrix, by
// the whole block; a, f and b2 as in tri_count, lo and hi scaled like them.  Ends
// when it is a few units in the last place wide.
__device__ __forceinline__ double tri_eigenvalue(const double *a, double f, const double *b2, int m, int k, double lo,
                                                 double hi)
{
    __shared__ int first;
    for (int it = 0; it < 24; ++it) {
        const double width = hi - lo;
        if (!(width > 2e-16 * fmax(fabs(lo), fabs(hi))))
            break;
        if (threadIdx.x == 0)
            first = kTriThreads;
        __syncthreads();
        const double x = lo + width * (double)(threadIdx.x + 1) / (double)(kTriThreads + 1);
        if (tri_count(a, f, b2, m, x) > k)
            atomicMin(&first, (int)threadIdx.x);
        __syncthreads();
        const int at = first;
        __syncthreads();
        const double nlo = at == 0 ? lo : lo + width * (double)at / (double)(kTriThreads + 1);
        const double nhi = at == kTriThreads ? hi : lo + width * (double)(at + 1) / (double)(kTriThreads + 1);
        if (!(nhi - nlo < width))
            break;
        lo = nlo;
        hi = nhi;
    }
    return 0.5 * (lo + hi);
}

// min / max / sum over the block (fixed tree)
template <typename F>
__device__ __forceinline__ double tri_reduce(double v, F op)
{
    __shared__ double part[kTriThreads / 32];
    for (int o = 16; o > 0; o >>= 1)
        v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0)
        part[threadIdx.x >> 5] = v;
    __syncthreads();
    v = part[0];
    for (int w = 1; w < kTriThreads / 32; ++w)
        v = op(v, part[w]);
    return v;
}

// a[0..m), b[0..m]: b[j] couples j-1 and j (b[0] unused).  The size at which the
// first vanishing coupling cuts the matrix, and the scale of its entries.
__device__ __forceinline__ int tri_effective_size(const double *a, const double *b, int m, double &scale)
{
    double s = 0.0;
    for (int i = threadIdx.x; i < m; i += kTriThreads)
        s = fmax(s, fabs(a[i]) + fabs(b[i + 1]));
    scale = tri_reduce(s, [](double u, double v) { return fmax(u, v); });
    double cut = (double)m;
    for (int i = 1 + (int)threadIdx.x; i < m; i += kTriThreads)
        if (!(b[i] > 1e-13 * fmax(scale, 1e-300))) {
            cut = (double)i;
            break;
        }
    return (int)tri_reduce(cut, [](double u, double v) { return fmin(u, v); });
}

// Gershgorin interval of the leading me x me matrix
__device__ __forceinline__ void tri_interval(const double *a, const double *b, int me, double &lo, double &hi)
{
    lo = 1e300;
    hi = -1e300;
    for (int i = threadIdx.x; i < me; i += kTriThreads) {
        const double r = (i ? fabs(b[i]) : 0.0) + (i + 1 < me ? fabs(b[i + 1]) : 0.0);
        lo = fmin(lo, a[i] - r);
        hi = fmax(hi, a[i] + r);
    }
    lo = tri_reduce(lo, [](double u, double v) { return fmin(u, v); });
    hi = tri_reduce(hi, [](double u, double v) { return fmax(u, v); });
}

struct TriShared {
    double a[kTriShared], b2[kTriShared];
    double b[kTriShared], y[kTriShared], l[kTriShared], rd[kTriShared];
};

// Eigenvalue k of the leading me x me matrix; sm holds its entries when they fit
// (filled here), b2 is global work space of me doubles otherwise.
__device__ __forceinline__ double tri_solve(const double *a, const double *b, int me, int k, TriShared &sm, double *b2)
{
    const bool fits = me <= kTriShared;
    double *q = fits ? sm.b2 : b2;
    double lo, hi;
    tri_interval(a, b, me, lo, hi);
    // the power of two that brings the largest entry near one: every step of the
    // bisection is the same up to it, in every bit
    const double top = fmax(fabs(lo), fabs(hi));
    const int e = top > 0.0 && top < 1e300 ? max(-1000, min(1000, ilogb(top))) : 0;
    const double f = scalbn(1.0, -e);
    for (int i = threadIdx.x; i < me; i += kTriThreads) {
        const double c = b[i] * f;
        q[i] = c * c;
        if (fits)
            sm.a[i] = a[i];
    }
    __syncthreads();
    return scalbn(tri_eigenvalue(fits ? sm.a : a, f, q, me, k, lo * f, hi * f), e);
}

// y_out[0..me) = normalised eigenvector for the eigenvalue lam by inverse iteration
// (four passes from the all-ones vector; LU without pivoting, guarded pivots);
// work: 2 me doubles, used when sm has no room.  The chains run in one thread.
__device__ __forceinline__ void tri_vector(const double *a, const double *b_in, int me, double lam, double scale,
                                           double *y_out, TriShared &sm, double *work)
{
    const bool fits = me <= kTriShared;
    double *rd = fits ? sm.rd : work, *l = fits ? sm.l : work + me;  // reciprocal pivots, multipliers
    double *y = fits ? sm.y : y_out;
    const double *b = fits ? sm.b : b_in;
    if (fits)
        for (int i = threadIdx.x; i < me; i += kTriThreads)
            sm.b[i] = b_in[i];
    __syncthreads();
    const double eps = 1e-15 * fmax(scale, 1e-300);
    if (threadIdx.x == 0) {
        double piv = a[0] - lam;
        for (int i = 0; i < me; ++i) {
            if (fabs(piv) < eps)
                piv = eps;
            const double r = 1.0 / piv;
            rd[i] = r;
            if (i + 1 < me) {
                const double m = b[i + 1] * r;
                l[i + 1] = m;
                piv = fma(-m, b[i + 1], a[i + 1] - lam);
            }
        }
    }
    for (int i = threadIdx.x; i < me; i += kTriThreads)
        y[i] = 1.0;
    __syncthreads();
    for (int iter = 0; iter < 4; ++iter) {
        if (threadIdx.x == 0) {
            double v = y[0];
            for (int i = 1; i < me; ++i) {
                v = fma(-l[i], v, y[i]);
                y[i] = v;
            }
            v *= rd[me - 1];
            y[me - 1] = v;
            for (int i = me - 2; i >= 0; --i) {
                v = fma(-b[i + 1], v, y[i]) * rd[i];
                y[i] = v;
            }
        }
        __syncthreads();
        double s = 0.0;
        for (int i = threadIdx.x; i < me; i += kTriThreads)
            s = fma(y[i], y[i], s);
        const double r = 1.0 / sqrt(tri_reduce(s, [](double u, double v) { return u + v; }));
        for (int i = threadIdx.x; i < me; i += kTriThreads)
            y[i] *= r;
        __syncthreads();
    }
    if (fits)
        for (int i = threadIdx.x; i < me; i += kTriThreads)
            y_out[i] = y[i];
}

}  // namespace edk

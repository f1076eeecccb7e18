// FP64 block reductions and the scalar steps of conjugate gradients, shared
// by the single-problem and the batched solvers.
//
// CG on (P^T M P + lambda D^T D) x = P^T M y (Eq. criterion, normal
// equations), textbook Hestenes-Stiefel form:
//   alpha = r.r / p.q;  x += alpha p;  r -= alpha q;
//   beta = r'.r' / r.r; p = r' + beta p.
// The criterion is reported through J = y^T M y - x^T (r + b), exact for
// every CG iterate (b = P^T M y, r = b - A x).
#pragma once

#include <math.h>

#include "tomo_internal.cuh"

namespace tomo {

// A per-thread partial sum kept as a compensated pair of floats.  A product
// of two floats is split exactly into p + e (p = fl(a b) with an unfused
// multiply, e = fmaf(a, b, -p): the FMA-based TwoProduct), and every term
// is added with Knuth's TwoSum, whose rounding error goes to the second
// float.  For the few dozen terms of one thread this is as accurate as FP64
// accumulation of the exact products (the error is of order u^2 times the
// sum of magnitudes), and it runs on the FP32 pipes: GB300 issues FP64 at a
// small fraction of its FP32 rate, and converting every element to FP64
// made the CG vector passes FP64-bound at a third of their memory rate.
// The pairs are summed across threads in FP64.
struct SumF2 {
    float hi = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void add(float a)
    {
        const float s = __fadd_rn(hi, a);
        const float bb = __fsub_rn(s, hi);
        const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)),
                                  __fsub_rn(a, bb));
        hi = s;
        lo = __fadd_rn(lo, e);
    }
    __device__ __forceinline__ void add_prod(float a, float b)
    {
        const float p = __fmul_rn(a, b);
        const float e = fmaf(a, b, -p);
        add(p);
        lo = __fadd_rn(lo, e);
    }
    // adds a (b + c), with b + c split exactly by TwoSum first
    __device__ __forceinline__ void add_prod_sum(float a, float b, float c)
    {
        const float s = __fadd_rn(b, c);
        const float bb = __fsub_rn(s, b);
        const float es = __fadd_rn(__fsub_rn(b, __fsub_rn(s, bb)),
                                   __fsub_rn(c, bb));
        add_prod(a, s);
        lo = __fadd_rn(lo, __fmul_rn(a, es));
    }
    __device__ __forceinline__ double value() const
    {
        return (double)hi + (double)lo;
    }
};

// A CG scalar (alpha or beta) as a pair of floats, hi + lo, good to 2^-48.
// Rounded to one float, its relative error of up to 2^-24 is the same in every
// element: an error along p as a whole, not noise that averages out over the
// voxels.  CG amplifies it once a Ritz value has converged on the largest
// eigenvalue, and which float alpha rounds to changes with the order of the
// transpose's float additions: x of 20 iterations (128^3, 60 views of 256^2)
// was 6e-6 to 3e-4 off its 64-bit value and two runs differed by up to 5e-4;
// with the pair 6e-6 to 2e-5 and 4e-6 to 2e-5.  The scalar step splits it once
// and keeps the two floats' bits in the CG slot: split by every thread of the
// update passes, a batch of 8 problems (31^3 to 96^3, 10 iterations) took 2.88
// ms in place of 2.82.
struct StepF2 {
    float hi, lo;
};

__device__ __forceinline__ double step_slot(double v)
{
    const float hi = (float)v;
    const float lo = (float)(v - (double)hi);
    return __hiloint2double(__float_as_int(hi), __float_as_int(lo));
}

__device__ __forceinline__ StepF2 step_of(double slot)
{
    return { __int_as_float(__double2hiint(slot)),
             __int_as_float(__double2loint(slot)) };
}

// x + a v, rounded once but for terms of order 2^-48: the product and the sum
// are split exactly (TwoProduct, TwoSum).  Where these give NaN (overflow,
// non-finite operands) the plain multiply-add's value stands.
__device__ __forceinline__ float axpy(const StepF2 &a, float v, float x)
{
    const float p = __fmul_rn(a.hi, v);
    const float e = fmaf(a.lo, v, fmaf(a.hi, v, -p));
    const float s = __fadd_rn(x, p);
    const float bb = __fsub_rn(s, x);
    const float es = __fadd_rn(__fsub_rn(x, __fsub_rn(s, bb)),
                               __fsub_rn(p, bb));
    const float y = __fadd_rn(s, __fadd_rn(es, e));
    return y == y ? y : fmaf(a.hi, v, x);
}

__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sums of K values per thread over the CTA of 256 threads; total[] is valid in
// thread 0.  GB300 completes about two FP64 operations per clock per SM, so a
// warp-wide addition holds that pipe for 16 clocks: the CTA's values go
// through shared memory and warp k adds up value k of all threads (7 + 5
// warp-wide additions instead of 5 in each of 8 warps and 5 more).  Ends with
// a barrier so `sm` can be reused by the next call.
constexpr int kSumThreads = 256;

template <int K>
__device__ __forceinline__ void block_sums(const double (&v)[K], double (&total)[K],
                                           double (*sm)[kSumThreads])
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) sm[k][threadIdx.x] = v[k];
    __syncthreads();
    if (w < K) {
        double s = sm[w][lane];
#pragma unroll
        for (int i = 1; i < kSumThreads / 32; ++i) s += sm[w][lane + 32 * i];
        s = warp_sum(s);
        __syncwarp();
        if (lane == 0) sm[w][0] = s;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) total[k] = sm[k][0];
    __syncthreads();
}

// Scalar steps; called by one thread with the grid-wide sums.

__device__ __forceinline__ void cg_finalize_init(double *S, double *report,
                                                 double rr, double xrb,
                                                 double tol2)
{
    S[S_RR] = rr;
    S[S_RR0] = rr;
    S[S_TOL2] = tol2;
    S[S_ITERS] = 0.0;
    S[S_ERR] = 0.0;
    S[S_DONE] = (rr == 0.0) ? 1.0 : 0.0;
    if (report != nullptr) {
        report[0] = S[S_YMY] - xrb;
        report[1] = rr;
    }
}

__device__ __forceinline__ void cg_finalize_pq(double *S, double pq)
{
    S[S_PQ] = pq;
    if (!(pq > 0.0) || !isfinite(pq)) {
        S[S_DONE] = 1.0;
        S[S_ERR] = 1.0;
    } else {
        S[S_ALPHA] = step_slot(S[S_RR] / pq);
    }
}

__device__ __forceinline__ void cg_finalize_update(double *S, double *report,
                                                   double rr_new, double xrb)
{
    const int k = (int)S[S_ITERS];
    S[S_BETA] = step_slot(rr_new / S[S_RR]);
    S[S_RR] = rr_new;
    S[S_ITERS] = k + 1;
    if (report != nullptr) {
        report[2 * (k + 1)] = S[S_YMY] - xrb;
        report[2 * (k + 1) + 1] = rr_new;
    }
    if (!isfinite(rr_new)) {
        S[S_DONE] = 1.0;
        S[S_ERR] = 1.0;
    } else if (rr_new <= S[S_TOL2] * S[S_RR0]) {
        S[S_DONE] = 1.0;
    }
}

// The 7-point stencil of lambda D^T D at voxel (i, j, k) of x, or with a
// diagonal weight w (nullable) the stencil of lambda R D^T D R, R = diag(w)
// (the height-weighted prior ||D R x||^2 of Eq. srt_inversion): the
// differences are taken of w x and the result is scaled by w at (i, j, k).
__device__ __forceinline__ float prior_at(const float *__restrict__ x,
                                          const float *__restrict__ w,
                                          int64_t v, int i, int j, int k,
                                          int nx, int ny, int nz, float lam)
{
    const int64_t sy = nx, sz = (int64_t)nx * ny;
    if (w == nullptr) {
        const float xc = x[v];
        float s = 0.0f;
        if (i > 0) s += xc - x[v - 1];
        if (i < nx - 1) s += xc - x[v + 1];
        if (j > 0) s += xc - x[v - sy];
        if (j < ny - 1) s += xc - x[v + sy];
        if (k > 0) s += xc - x[v - sz];
        if (k < nz - 1) s += xc - x[v + sz];
        return lam * s;
    }
    const float wc = w[v];
    const float xc = wc * x[v];
    float s = 0.0f;
    if (i > 0) s += xc - w[v - 1] * x[v - 1];
    if (i < nx - 1) s += xc - w[v + 1] * x[v + 1];
    if (j > 0) s += xc - w[v - sy] * x[v - sy];
    if (j < ny - 1) s += xc - w[v + sy] * x[v + sy];
    if (k > 0) s += xc - w[v - sz] * x[v - sz];
    if (k < nz - 1) s += xc - w[v + sz] * x[v + sz];
    return lam * wc * s;
}

}  // namespace tomo

// Vector steps of conjugate gradients on (E'E + lam I) x = b (the linear solves of Sec. II-F), for
// complex vectors of n elements.  One iteration around the normal product q = E'E p is three
// launches:
//   k_cg_dot     partial sums of <p, q + lam p>
//   k_cg_update  alpha = <r,r> / <p, F p>;  x += alpha p;  r -= alpha (q + lam p);  partial sums of <r,r>
//   k_cg_dir     p = r + (<r,r>_new / <r,r>_old) p
// The scalars stay on the device: every block adds the partial sums of the kernel before it by
// itself, in block order, so that a solve never waits for the host and, on a deterministic plan, repeats
// bit by bit.  The vectors are read and written once per step (7 reads, 3 writes an iteration), which is all these
// kernels do; they are launch-bound up to a few hundred thousand elements.  The same algebra as
// about twenty tensor operations per iteration kept the host busy for 340 us beside 115 us of
// normal product (320^2, 16 coils); a solve of 10 iterations and its gradient went from 6732 to
// 2736 us, with errors against FP64 of 6e-7 to 7e-7 (6e-7 to 1.6e-6 before).  Products and sums of the
// scalars are FP64: the square of any FP32 number is then above zero, so <r,r> is zero only where r is,
// and the iteration then stays where it is (alpha = beta = 0) instead of dividing zero by zero.
#include <algorithm>

#include "internal.h"

namespace nj {

constexpr int kCgThreads = 256;

// Sum over the block.  One warp adds 8 values a lane and then across its lanes: FP64 adds run at a low rate, and with
// every thread shuffling five times and adding eight warp sums they took longer than the vectors (the solve and
// gradient above: 2970 us, now 2736).
__device__ __forceinline__ double cg_block_sum(double v) {
    __shared__ double sh[kCgThreads], total;
    const int t = threadIdx.x;
    __syncthreads();   // a previous sum may still be read
    sh[t] = v;
    __syncthreads();
    if (t < 32) {
        double s = sh[t];
#pragma unroll
        for (int k = 32; k < kCgThreads; k += 32) s += sh[t + k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (t == 0) total = s;
    }
    __syncthreads();
    return total;
}

// Sum of one kernel's block partials, the same bits in every block.
__device__ __forceinline__ double cg_total(const double* part, int nb) {
    double v = 0.0;
    for (int k = threadIdx.x; k < nb; k += kCgThreads) v += part[k];
    return cg_block_sum(v);
}

// s + |v|^2 and s + Re{conj(a) b}, exact products.
__device__ __forceinline__ double cg_add_sqr(double s, float2 v) {
    return fma((double)v.x, (double)v.x, fma((double)v.y, (double)v.y, s));
}
__device__ __forceinline__ double cg_add_dot(double s, float2 a, float2 b) {
    return fma((double)a.x, (double)b.x, fma((double)a.y, (double)b.y, s));
}

__global__ void __launch_bounds__(kCgThreads) k_cg_start(CgArgs a) {
    pdl_wait();
    double s = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * kCgThreads + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * kCgThreads) {
        const float2 b = a.b[i];
        a.x[i] = make_float2(0.f, 0.f);
        a.r[i] = b;
        a.p[i] = b;
        s = cg_add_sqr(s, b);
    }
    const double t = cg_block_sum(s);
    if (threadIdx.x == 0) a.rr[blockIdx.x] = t;
}

__global__ void __launch_bounds__(kCgThreads) k_cg_dot(CgArgs a) {
    pdl_wait();
    double s = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * kCgThreads + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * kCgThreads) {
        const float2 p = a.p[i], q = a.q[i];
        s = cg_add_dot(s, p, make_float2(fmaf(a.lam, p.x, q.x), fmaf(a.lam, p.y, q.y)));
    }
    const double t = cg_block_sum(s);
    if (threadIdx.x == 0) a.pq[blockIdx.x] = t;
}

__global__ void __launch_bounds__(kCgThreads) k_cg_update(CgArgs a) {
    pdl_wait();
    const double rr = cg_total(a.rr, gridDim.x), pq = cg_total(a.pq, gridDim.x);
    const float alpha = pq == 0.0 ? 0.f : (float)(rr / pq);   // p = 0 (or F p = 0): no step left
    double s = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * kCgThreads + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * kCgThreads) {
        const float2 p = a.p[i], q = a.q[i];
        float2 x = a.x[i], r = a.r[i];
        x.x = fmaf(alpha, p.x, x.x);
        x.y = fmaf(alpha, p.y, x.y);
        r.x = fmaf(-alpha, fmaf(a.lam, p.x, q.x), r.x);
        r.y = fmaf(-alpha, fmaf(a.lam, p.y, q.y), r.y);
        a.x[i] = x;
        a.r[i] = r;
        s = cg_add_sqr(s, r);
    }
    const double t = cg_block_sum(s);
    if (threadIdx.x == 0) a.rr_new[blockIdx.x] = t;
}

__global__ void __launch_bounds__(kCgThreads) k_cg_dir(CgArgs a) {
    pdl_wait();
    const double rn = cg_total(a.rr_new, gridDim.x), rr = cg_total(a.rr, gridDim.x);
    const float beta = rr == 0.0 ? 0.f : (float)(rn / rr);
    for (int64_t i = (int64_t)blockIdx.x * kCgThreads + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * kCgThreads) {
        const float2 r = a.r[i], p = a.p[i];
        a.p[i] = make_float2(fmaf(beta, p.x, r.x), fmaf(beta, p.y, r.y));
    }
}

cudaError_t launch_cg(CgStep step, const CgArgs& a, cudaStream_t s) {
    const unsigned nb = (unsigned)std::max<int64_t>(1, std::min<int64_t>(kCgBlocks, (a.n + kCgThreads - 1) / kCgThreads));
    switch (step) {
        case CG_START: (void)launch_pdl(k_cg_start, nb, kCgThreads, 0, s, a); break;
        case CG_DOT: (void)launch_pdl(k_cg_dot, nb, kCgThreads, 0, s, a); break;
        case CG_UPDATE: (void)launch_pdl(k_cg_update, nb, kCgThreads, 0, s, a); break;
        default: (void)launch_pdl(k_cg_dir, nb, kCgThreads, 0, s, a); break;
    }
    return cudaGetLastError();
}

}  // namespace nj

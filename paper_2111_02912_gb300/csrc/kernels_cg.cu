// Vector steps of conjugate gradients on (E'E + lam I) x = b (the linear solves of Sec. II-F), for
// complex vectors of n elements.  One iteration around the normal product q = E'E p is three
// launches:
//   k_cg_dot     partial sums of <p, q + lam p>
//   k_cg_update  alpha = <r,r> / <p, F p>;  x += alpha p;  r -= alpha (q + lam p);  partial sums of <r,r>
//   k_cg_dir     p = r + (<r,r>_new / <r,r>_old) p
// The scalars stay on the device: every block adds the partial sums of the kernel before it by
// itself, in block order, so that a solve never waits for the host and repeats bit by bit.  The
// vectors are read and written once per step (7 reads, 3 writes an iteration), which is all these
// kernels do; they are launch-bound up to a few hundred thousand elements.  The same algebra as
// about twenty tensor operations per iteration kept the host busy for 340 us beside 115 us of
// normal product (320^2, 16 coils); a solve of 10 iterations and its gradient went from 6732 to
// 2957 us, with an error against FP64 of 5.4e-7 instead of 9.5e-7.  Sums run in FP32 within
// a thread (a few dozen terms at most) and in FP64 across threads and blocks.
#include <algorithm>

#include "internal.h"

namespace nj {

constexpr int kCgThreads = 256;

__device__ __forceinline__ double cg_block_sum(double v) {
    __shared__ double sh[kCgThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();   // sh may still be read from a previous sum
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double t = 0.0;
#pragma unroll
    for (int k = 0; k < kCgThreads / 32; ++k) t += sh[k];
    return t;
}

// Sum of one kernel's block partials, the same bits in every block.
__device__ __forceinline__ double cg_total(const double* part, int nb) {
    double v = 0.0;
    for (int k = threadIdx.x; k < nb; k += kCgThreads) v += part[k];
    return cg_block_sum(v);
}

__global__ void __launch_bounds__(kCgThreads) k_cg_start(CgArgs a) {
    pdl_wait();
    float s = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * kCgThreads + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * kCgThreads) {
        const float2 b = a.b[i];
        a.x[i] = make_float2(0.f, 0.f);
        a.r[i] = b;
        a.p[i] = b;
        s = fmaf(b.x, b.x, fmaf(b.y, b.y, s));
    }
    const double t = cg_block_sum((double)s);
    if (threadIdx.x == 0) a.rr[blockIdx.x] = t;
}

__global__ void __launch_bounds__(kCgThreads) k_cg_dot(CgArgs a) {
    pdl_wait();
    float s = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * kCgThreads + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * kCgThreads) {
        const float2 p = a.p[i], q = a.q[i];
        const float fx = fmaf(a.lam, p.x, q.x), fy = fmaf(a.lam, p.y, q.y);
        s = fmaf(p.x, fx, fmaf(p.y, fy, s));
    }
    const double t = cg_block_sum((double)s);
    if (threadIdx.x == 0) a.pq[blockIdx.x] = t;
}

__global__ void __launch_bounds__(kCgThreads) k_cg_update(CgArgs a) {
    pdl_wait();
    const double rr = cg_total(a.rr, gridDim.x), pq = cg_total(a.pq, gridDim.x);
    const float alpha = (float)(rr / pq);
    float s = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * kCgThreads + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * kCgThreads) {
        const float2 p = a.p[i], q = a.q[i];
        float2 x = a.x[i], r = a.r[i];
        x.x = fmaf(alpha, p.x, x.x);
        x.y = fmaf(alpha, p.y, x.y);
        r.x = fmaf(-alpha, fmaf(a.lam, p.x, q.x), r.x);
        r.y = fmaf(-alpha, fmaf(a.lam, p.y, q.y), r.y);
        a.x[i] = x;
        a.r[i] = r;
        s = fmaf(r.x, r.x, fmaf(r.y, r.y, s));
    }
    const double t = cg_block_sum((double)s);
    if (threadIdx.x == 0) a.rr_new[blockIdx.x] = t;
}

__global__ void __launch_bounds__(kCgThreads) k_cg_dir(CgArgs a) {
    pdl_wait();
    const double rn = cg_total(a.rr_new, gridDim.x), rr = cg_total(a.rr, gridDim.x);
    const float beta = (float)(rn / rr);
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

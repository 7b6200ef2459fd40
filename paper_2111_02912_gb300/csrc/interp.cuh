// Interpolation (gather) kernel template, instantiated per dimension in
// kernels_gather_d{1,2,3}.cu.
//
// Gather, step (3) of the Appendix: y_i = sum over the J^D window taps of
// prod_d psi(u_d) G[k mod K].  A group of G lanes (a power of two) handles one
// sample; lane l owns coils l, l+G, ...  The J*D kernel weights of the sample
// are evaluated once by the group (one psi per lane) and reused for every
// channel of every coil: the unweighted grid and the D coordinate-weighted
// grids x . r^[d] of Eq. (e,Ax).  Epilogues:
//   FWD  y_c = g_c0 (FWD_SORTED: in the sorted order that the strip spread reads, 2-D and 3-D)
//   JVP  dy_c = -i sum_d domega^[d] g_cd  (and y_c when the plain channel is present)
//   VJP  grad^[d] = sum_c Re{conj(v_c) (-i) g_cd} = sum_c Im{conj(v_c) g_cd}   (Eq. (e,jac,Ax,v))
// so the D interpolated channels per coil never leave registers.
#pragma once
#include "internal.h"

namespace nj {

// Weights of one sample into w[d * J + j] (shared, per group), copied from the
// sort's per-point weights (at d * wd + j): lane q of the group loads q, q + G, ...
template <int D, int J>
__device__ __forceinline__ void group_weights(float* w, const float* pw, int wd, int lane_g, int G) {
    for (int q = lane_g; q < D * J; q += G) {
        const int d = q / J;
        w[q] = __ldg(pw + d * wd + (q - d * J));
    }
}

// 32-byte read-only load (four complex coil values), one instruction.
__device__ __forceinline__ void ldg_v8(const float2* p, float4& lo, float4& hi) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(lo.x), "=f"(lo.y), "=f"(lo.z), "=f"(lo.w), "=f"(hi.x), "=f"(hi.y), "=f"(hi.z), "=f"(hi.w)
        : "l"(p));
}

// W coils per lane slot: lane l owns coils W (l + k G) .. W (l + k G) + W - 1, read as one load of
// 8 W bytes (W = 2: a 16-byte load, C even; W = 4: a 32-byte load, C a multiple of 4; W = 1: one
// coil).
template <int D, int J, int ND, int CPL, int MODE, int W>
__device__ __forceinline__ void gather_body(const GatherArgs& a) {
    extern __shared__ float wsm[];   // [groups][D * J]
    const int tid = threadIdx.x;

    const int G = a.G;
    const int lane_g = tid & (G - 1);
    const int grp = tid >> a.lgG;
    const int gpb = blockDim.x >> a.lgG;
    const int64_t pt = (int64_t)blockIdx.x * gpb + grp;
    const bool valid = pt < a.pts.m;
    float* w = wsm + grp * (D * J);
    int4 ix = make_int4(0, 0, 0, 0);
    if (valid) {
        ix = a.pts.idx[pt];
        group_weights<D, J>(w, a.pts.w + pt * a.pts.ws, a.pts.wd, lane_g, G);
    }
    __syncwarp();
    if (!valid) return;

    const int C = a.C;
    const int chs = ND * C;   // channel stride of one grid cell
    bool ok[CPL];
    int lofs[CPL];   // coil offset of slot k; slots past the last coil read coil 0 (never stored)
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        ok[k] = W * (lane_g + k * G) < C;
        lofs[k] = ok[k] ? W * (lane_g + k * G) : 0;
    }
    float2 acc[ND][CPL][W];
#pragma unroll
    for (int q = 0; q < ND; ++q)
#pragma unroll
        for (int k = 0; k < CPL; ++k)
#pragma unroll
            for (int i = 0; i < W; ++i) acc[q][k][i] = make_float2(0.f, 0.f);

    // innermost axis: column offsets and weights in registers
    const int Kl = a.K[D - 1];
    const int kl0 = D == 1 ? ix.x : (D == 2 ? ix.y : ix.z);
    int coff[J];
    float wl[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
        int k = kl0 + j;
        if (k >= Kl) k -= Kl;
        coff[j] = k * chs;
        wl[j] = w[(D - 1) * J + j];
    }
    const float2* g0 = a.grid;

    auto row = [&](const float2* rp, float wr) {
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const float wt = wr * wl[j];
            const float2* gp = rp + coff[j];
#pragma unroll
            for (int q = 0; q < ND; ++q)
#pragma unroll
                for (int k = 0; k < CPL; ++k) {   // unconditional loads: all taps in flight together
                        if constexpr (W == 4) {
                            float4 g, h;
                            ldg_v8(gp + q * C + lofs[k], g, h);
                            acc[q][k][0].x = fmaf(wt, g.x, acc[q][k][0].x);
                            acc[q][k][0].y = fmaf(wt, g.y, acc[q][k][0].y);
                            acc[q][k][1].x = fmaf(wt, g.z, acc[q][k][1].x);
                            acc[q][k][1].y = fmaf(wt, g.w, acc[q][k][1].y);
                            acc[q][k][2].x = fmaf(wt, h.x, acc[q][k][2].x);
                            acc[q][k][2].y = fmaf(wt, h.y, acc[q][k][2].y);
                            acc[q][k][W - 1].x = fmaf(wt, h.z, acc[q][k][W - 1].x);
                            acc[q][k][W - 1].y = fmaf(wt, h.w, acc[q][k][W - 1].y);
                        } else if constexpr (W == 2) {
                            const float4 g = __ldg((const float4*)(gp + q * C + lofs[k]));
                            acc[q][k][0].x = fmaf(wt, g.x, acc[q][k][0].x);
                            acc[q][k][0].y = fmaf(wt, g.y, acc[q][k][0].y);
                            acc[q][k][W - 1].x = fmaf(wt, g.z, acc[q][k][W - 1].x);
                            acc[q][k][W - 1].y = fmaf(wt, g.w, acc[q][k][W - 1].y);
                        } else {
                            const float2 g = __ldg(gp + q * C + lofs[k]);
                            acc[q][k][0].x = fmaf(wt, g.x, acc[q][k][0].x);
                            acc[q][k][0].y = fmaf(wt, g.y, acc[q][k][0].y);
                        }
                    }
        }
    };

    if (D == 1) {
        row(g0, 1.f);
    } else if (D == 2) {
        const int K0 = a.K[0];
        const int64_t rstride = (int64_t)a.K[1] * chs;
#pragma unroll
        for (int j0 = 0; j0 < J; ++j0) {
            int k0 = ix.x + j0;
            if (k0 >= K0) k0 -= K0;
            row(g0 + k0 * rstride, w[j0]);
        }
    } else {
        const int K0 = a.K[0], K1 = a.K[1];
        const int64_t pstride = (int64_t)a.K[1] * a.K[2] * chs, rstride = (int64_t)a.K[2] * chs;
#pragma unroll 1
        for (int j0 = 0; j0 < J; ++j0) {
            int k0 = ix.x + j0;
            if (k0 >= K0) k0 -= K0;
            const float2* pp = g0 + k0 * pstride;
            const float w0 = w[j0];
#pragma unroll
            for (int j1 = 0; j1 < J; ++j1) {
                int k1 = ix.y + j1;
                if (k1 >= K1) k1 -= K1;
                row(pp + k1 * rstride, w0 * w[J + j1]);
            }
        }
    }

    const int64_t orig = ix.w;
    const int64_t M = a.M;
    if (MODE == GM_FWD) {
#pragma unroll
        for (int k = 0; k < CPL; ++k)
#pragma unroll
            for (int i = 0; i < W; ++i)
                if (ok[k]) a.y[(int64_t)(W * (lane_g + k * G) + i) * M + orig] = acc[0][k][i];
    } else if (MODE == GM_FWD_SORTED) {   // for the adjoint spread of the same points
#pragma unroll
        for (int k = 0; k < CPL; ++k)
#pragma unroll
            for (int i = 0; i < W; ++i) {
                const int c = W * (lane_g + k * G) + i, cg = c / a.v_sorted_cpt;
                if (ok[k]) a.v_sorted[((int64_t)cg * M + pt) * a.v_sorted_cpt + (c - cg * a.v_sorted_cpt)] = acc[0][k][i];
            }
    } else if (MODE == GM_JVP) {
        float dom[D];
#pragma unroll
        for (int d = 0; d < D; ++d) dom[d] = a.domega[(int64_t)d * M + orig];
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            if (!ok[k]) continue;
#pragma unroll
            for (int i = 0; i < W; ++i) {
                const int64_t c = W * (lane_g + k * G) + i;
                float2 s = make_float2(0.f, 0.f);
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    const float2 g = acc[(ND > D ? 1 : 0) + d][k][i];
                    s.x = fmaf(dom[d], g.y, s.x);    // -i * g = (g.y, -g.x)
                    s.y = fmaf(-dom[d], g.x, s.y);
                }
                a.dy[c * M + orig] = s;
                if (ND > D) a.y[c * M + orig] = acc[0][k][i];
            }
        }
    } else {   // GM_VJP
        float gsum[D];
#pragma unroll
        for (int d = 0; d < D; ++d) gsum[d] = 0.f;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            if (!ok[k]) continue;
#pragma unroll
            for (int i = 0; i < W; ++i) {
                const int64_t cv = W * (lane_g + k * G) + i;
                const float2 v = __ldg(a.v + cv * M + orig);
                if (a.v_sorted) {   // for the adjoint spread of the same v
                    if (a.v_sorted_cpt) {
                        const int64_t cg = cv / a.v_sorted_cpt;
                        a.v_sorted[(cg * M + pt) * a.v_sorted_cpt + (cv - cg * a.v_sorted_cpt)] = v;
                    } else {
                        a.v_sorted[cv * M + pt] = v;
                    }
                }
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    const float2 g = acc[d][k][i];
                    gsum[d] += v.x * g.y - v.y * g.x;   // Im{conj(v) g}
                }
            }
        }
        const unsigned mask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << ((tid & 31) & ~(G - 1)));
#pragma unroll
        for (int d = 0; d < D; ++d)
            for (int off = G >> 1; off > 0; off >>= 1) gsum[d] += __shfl_xor_sync(mask, gsum[d], off, G);
        if (lane_g == 0) {
#pragma unroll
            for (int d = 0; d < D; ++d) a.grad[(int64_t)d * M + orig] = gsum[d];
        }
    }
}

// Block size and resident blocks per SM that the registers are held to (0: no limit).  The gathers wait
// on their tap loads, so warps count, as long as nothing of weight spills.
// Single coils, narrow: 64-thread blocks, 64 registers for one and two channel blocks, 80 for more, 128 for four
// slots per lane.  Faster in 2-D (VJP 150 x 218, 5 coils, 30,011 points: 20.7 -> 15.0 us; 128^2, 9 coils, 30,000: forward
// 15.4 -> 14.1, VJP 30.3 -> 20.4; three coils with J >= 6 and values lose: 16.6 -> 17.5) and with four slots (128^2, 33 to 128
// coils, 20,000 points: forward 1.0 to 2.2 times as fast, JVP 1.3 to 2.5, VJP 1.15 to 1.4; 40 x 36 x 32, 96 coils: forward
// 2.2, VJP 2.9, JVP with values 0.97).  In 3-D (40 x 36 x 32, 30,000 points) the VJP and most JVPs gain (J = 6, 9 coils: VJP
// 178 -> 166 us, JVP 162 -> 129); the forward gains at J = 4 and 8 (9 coils: 30.7 -> 22.5, 179 -> 171) but loses
// between (J = 7: 85.9 -> 104.5), as does the JVP with values at J = 6 (182 -> 191), and so do one to three coils at
// J = 6 and 7 in the VJP (1 coil, J = 7: 65.8 -> 73.2) and one at J = 8 in the forward (47.4 -> 55.8).  1-D loses (200 cells,
// 9 coils, forward: 7.7 -> 10.2 us).  All of these keep 256 threads and no limit.
// Pairs and quads: 256 threads; the 2-D VJP and JVP pairs are held to four and three blocks
// (VJP 40.3 -> 39.1 us on the 640^2, 16-coil case; JVP with values, 192 x 256, 12 coils, 99,999 points:
// 69.6 -> 65.5 us).  The forward at 40 or 48 registers spills and gains nothing.
constexpr bool gather_narrow(int D, int J, int ND, int mode, int CPL, int W) {
    const bool fwd = mode == GM_FWD || mode == GM_FWD_SORTED;
    return W == 1 && (CPL > 1 || D == 2 || (D == 3 && !(fwd && J >= 5 && J <= 7) && !(ND == 4 && J == 6)));
}
constexpr int gather_threads(bool narrow) { return narrow ? 64 : 256; }
constexpr int gather_blocks(int D, int mode, int ND, int CPL, int W, bool narrow) {
    return narrow ? (CPL > 1 ? 8 : ND <= 2 ? 16 : 12)
           : D == 2 && W == 2 && mode == GM_VJP ? 4
           : D == 2 && W == 2 && mode == GM_JVP ? 3 : 0;
}
template <int D, int J, int ND, int CPL, int MODE, int W, bool NARROW>
__global__ void __launch_bounds__(gather_threads(NARROW), gather_blocks(D, MODE, ND, CPL, W, NARROW)) k_gather(GatherArgs a) {
    pdl_wait();
    gather_body<D, J, ND, CPL, MODE, W>(a);
}

// Whole-line gather for eight coils.  With 64-byte channel blocks the pair lanes above read eight
// half lines per warp load, and the L1 data pipe, which serves one line per wavefront, bounds the
// 3-D gathers (81-83% of its peak at half its bytes).  Here a point has eight lanes, 16 bytes each, and
// a load covers whole 128-byte lines of the row's cells; lane l always holds coil pair l mod 4.
//   ND even: a cell is ND / 2 lines; load s of a column reads blocks 2 s (lanes 0-3) and 2 s + 1.
//   ND odd: two cells, of an even column E and the odd column after it, are ND lines.  The window's
//   even and odd columns are matched so (one match per row is of two pairs when it starts at an odd
//   column), and the lines of a match are, for ND = 1: {E0 O0}, and for ND = 3: {E0 E1} {E2 O0} {O1 O2}
//   (E2 = block 2 of the even column).
// A load of a match belongs to one channel block and one column per half of the lanes, so each has
// its own accumulators and its own column weight; the epilogues are linear in the channel blocks, so
// the halves' partial sums meet only there.  Addresses are 32-bit byte offsets from the grid (the host
// takes this kernel for grids below 4 GB).
template <int D, int J, int ND, int MODE>
__device__ __forceinline__ void gather_lines_body(const GatherArgs& a) {
    constexpr int CELL = ND * 64;                        // bytes of one cell's channels
    constexpr bool ODD = ND % 2 == 1;
    constexpr int S = ODD ? ND : ND / 2;                 // loads per match or column
    constexpr int NT = ODD ? (J + 1) / 2 : J;            // matches or columns per row
    extern __shared__ float wsm[];   // [points][D * J]
    const int tid = threadIdx.x, l = tid & 7;
    const bool up = l >= 4;          // the upper half of the point's lanes
    const int64_t pt = (int64_t)blockIdx.x * (blockDim.x >> 3) + (tid >> 3);
    const bool valid = pt < a.pts.m;
    float* w = wsm + (tid >> 3) * (D * J);
    int4 ix = make_int4(0, 0, 0, 0);
    if (valid) {
        ix = a.pts.idx[pt];
        group_weights<D, J>(w, a.pts.w + pt * a.pts.ws, a.pts.wd, l, 8);
    }
    __syncwarp();
    if (!valid) return;

    const int Kl = a.K[D - 1];
    const int kl0 = D == 2 ? ix.y : ix.z;
    const float* wc = w + (D - 1) * J;
    uint32_t off[NT][S];   // byte offset of the lane's 16 bytes within the row
    float wl[NT][S];       // column weight
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        if (ODD) {
            // window positions of the match's even and odd columns; -1: none (J odd)
            int je = 2 * t, jo = 2 * t + 1 < J ? 2 * t + 1 : -1;
            if (kl0 & 1) {
                jo = 2 * t;
                je = t > 0 ? 2 * t - 1 : (J % 2 == 0 ? J - 1 : -1);
            }
            int ce = kl0 + max(je, 0), co = kl0 + max(jo, 0);
            if (ce >= Kl) ce -= Kl;
            if (co >= Kl) co -= Kl;
            const float we = je >= 0 ? wc[max(je, 0)] : 0.f, wo = jo >= 0 ? wc[max(jo, 0)] : 0.f;
            if (ND == 1) {
                off[t][0] = (uint32_t)((up ? co : ce) * CELL + (l & 3) * 16);
                wl[t][0] = up ? wo : we;
            } else {
                off[t][0] = (uint32_t)(ce * CELL + l * 16);
                wl[t][0] = we;
                off[t][S > 1 ? 1 : 0] = (uint32_t)(up ? co * CELL + (l & 3) * 16 : ce * CELL + 128 + l * 16);
                wl[t][S > 1 ? 1 : 0] = up ? wo : we;
                off[t][S - 1] = (uint32_t)(co * CELL + 64 + l * 16);
                wl[t][S - 1] = wo;
            }
        } else {
            int c = kl0 + t;
            if (c >= Kl) c -= Kl;
#pragma unroll
            for (int i = 0; i < S; ++i) {
                off[t][i] = (uint32_t)(c * CELL + 128 * i + l * 16);
                wl[t][i] = wc[t];
            }
        }
    }
    float4 acc[S];
#pragma unroll
    for (int i = 0; i < S; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);

    const char* base = (const char*)a.grid;
    auto row = [&](uint32_t rb, float wr) {
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int i = 0; i < S; ++i) {
                const float wt = wr * wl[t][i];
                float4 g;
                if (ODD && J % 2 == 1 && (t == 0 || t == NT - 1)) {   // the one column that may be missing
                    g = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (wl[t][i] != 0.f) g = __ldg((const float4*)(base + (rb + off[t][i])));
                } else {
                    g = __ldg((const float4*)(base + (rb + off[t][i])));
                }
                acc[i].x = fmaf(wt, g.x, acc[i].x);
                acc[i].y = fmaf(wt, g.y, acc[i].y);
                acc[i].z = fmaf(wt, g.z, acc[i].z);
                acc[i].w = fmaf(wt, g.w, acc[i].w);
            }
    };
    const int K0 = a.K[0];
    if (D == 2) {
        const uint32_t rstride = (uint32_t)a.K[1] * CELL;
#pragma unroll
        for (int j0 = 0; j0 < J; ++j0) {
            int k0 = ix.x + j0;
            if (k0 >= K0) k0 -= K0;
            row((uint32_t)k0 * rstride, w[j0]);
        }
    } else {
        const int K1 = a.K[1];
        const uint32_t rstride = (uint32_t)a.K[2] * CELL;
#pragma unroll 1
        for (int j0 = 0; j0 < J; ++j0) {
            int k0 = ix.x + j0;
            if (k0 >= K0) k0 -= K0;
            const float w0 = w[j0];
#pragma unroll
            for (int j1 = 0; j1 < J; ++j1) {
                int k1 = ix.y + j1;
                if (k1 >= K1) k1 -= K1;
                row((uint32_t)(k0 * K1 + k1) * rstride, w0 * w[J + j1]);
            }
        }
    }

    const int64_t orig = ix.w, M = a.M;
    const unsigned mask = 0xffu << ((tid & 31) & ~7);   // the point's lanes
    const int c0 = 2 * (l & 3);                         // this lane's coil pair
    auto block_of = [&](int i) {                        // channel block of load i
        if (ND == 1) return 0;
        if (!ODD) return 2 * i + (up ? 1 : 0);
        return i == 0 ? (up ? 1 : 0) : (i == 1 ? (up ? 0 : 2) : (up ? 2 : 1));
    };
    // Sum of what the point's two lanes of a coil pair hold; the lower lane gets the first coil.
    auto meet = [&](float4 v) {
        v.x += __shfl_xor_sync(mask, v.x, 4);
        v.y += __shfl_xor_sync(mask, v.y, 4);
        v.z += __shfl_xor_sync(mask, v.z, 4);
        v.w += __shfl_xor_sync(mask, v.w, 4);
        return up ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
    };
    const int c = c0 + (up ? 1 : 0);   // the coil this lane writes
    if (MODE == GM_FWD || MODE == GM_FWD_SORTED || (MODE == GM_JVP && ND > D)) {   // the plain image's values
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < S; ++i)
            if (block_of(i) == 0) {
                v.x += acc[i].x;
                v.y += acc[i].y;
                v.z += acc[i].z;
                v.w += acc[i].w;
            }
        const float2 y = meet(v);
        if (MODE == GM_FWD_SORTED) {   // for the adjoint spread of the same points
            const int cg = c / a.v_sorted_cpt;
            a.v_sorted[((int64_t)cg * M + pt) * a.v_sorted_cpt + (c - cg * a.v_sorted_cpt)] = y;
        } else {
            a.y[(int64_t)c * M + orig] = y;
        }
    }
    if (MODE == GM_JVP) {   // dy = -i sum_d domega^[d] g_d, the d-th weighted block at d + (plain ? 1 : 0)
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < S; ++i) {
            const int d = block_of(i) - (ND > D ? 1 : 0);
            if (d < 0) continue;
            const float dom = __ldg(a.domega + (int64_t)d * M + orig);
            v.x = fmaf(dom, acc[i].y, v.x);
            v.y = fmaf(-dom, acc[i].x, v.y);
            v.z = fmaf(dom, acc[i].w, v.z);
            v.w = fmaf(-dom, acc[i].z, v.w);
        }
        a.dy[(int64_t)c * M + orig] = meet(v);
    }
    if (MODE == GM_VJP) {
        const float2 v0 = __ldg(a.v + (int64_t)c0 * M + orig), v1 = __ldg(a.v + (int64_t)(c0 + 1) * M + orig);
        if (a.v_sorted) {   // for the adjoint spread of the same v
            const float2 v = up ? v1 : v0;
            if (a.v_sorted_cpt) {
                const int cg = c / a.v_sorted_cpt;
                a.v_sorted[((int64_t)cg * M + pt) * a.v_sorted_cpt + (c - cg * a.v_sorted_cpt)] = v;
            } else {
                a.v_sorted[(int64_t)c * M + pt] = v;
            }
        }
        float gsum[D];
#pragma unroll
        for (int d = 0; d < D; ++d) gsum[d] = 0.f;
#pragma unroll
        for (int i = 0; i < S; ++i) {   // Im{conj(v) g}
            const float t = (v0.x * acc[i].y - v0.y * acc[i].x) + (v1.x * acc[i].w - v1.y * acc[i].z);
#pragma unroll
            for (int d = 0; d < D; ++d) gsum[d] += block_of(i) == d ? t : 0.f;
        }
#pragma unroll
        for (int d = 0; d < D; ++d)
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) gsum[d] += __shfl_xor_sync(mask, gsum[d], o);
        if (l == 0) {
#pragma unroll
            for (int d = 0; d < D; ++d) a.grad[(int64_t)d * M + orig] = gsum[d];
        }
    }
}

// 64-thread blocks (eight points): a block ends as soon as its own points have their taps.  Registers:
// 96 for three and four channel blocks (20 warps per SM), else 64 (32 warps).
// 128^2 x 96, 8 coils, 2 M points: VJP 4570 -> 3600 us, forward 1350 -> 1230 us; 128-, 256-, 320- and
// 640-thread blocks took 3713, 3758, 3761 and 3933 us for the VJP, 80 and 128 registers the same as 96.
// (32-byte loads by four lanes per point ran no faster than half lines: 5130 us.)  What bounds it now
// is the latency of the taps' L2 reads: at 64^2 x 48, 250,000 points (VJP 458 us, pairs 573) 61% of the
// sectors miss L1, 5.9 GB come from L2 (12.9 TB/s) and the LSU data pipe runs at 62% of its peak, with
// 9.8 cycles of long-scoreboard stalls to an issue at 19 warps per SM.
constexpr int kLinesThreads = 64;
template <int D, int J, int ND, int MODE>
__global__ void __launch_bounds__(kLinesThreads, ND >= 3 ? 10 : 16) k_gather_lines(GatherArgs a) {
    pdl_wait();
    gather_lines_body<D, J, ND, MODE>(a);
}

template <int D, int J, int ND, int MODE>
static cudaError_t gather_cpl(const GatherArgs& a, int cpl, cudaStream_t s) {
    if (a.pts.m == 0) return cudaSuccess;
    constexpr bool fwd = MODE == GM_FWD || MODE == GM_FWD_SORTED;
    auto go = [&](auto kernel, bool narrow) {
        const int threads = gather_threads(narrow), gpb = threads / a.G;
        (void)launch_pdl(kernel, (unsigned)((a.pts.m + gpb - 1) / gpb), threads, (size_t)gpb * D * J * sizeof(float), s, a);
    };
    if constexpr (D > 1) {
        if (cpl == kGatherLines) {
            const int pts = kLinesThreads / 8;
            (void)launch_pdl(k_gather_lines<D, J, ND, MODE>, (unsigned)((a.pts.m + pts - 1) / pts), kLinesThreads,
                             (size_t)pts * D * J * sizeof(float), s, a);
            return cudaGetLastError();
        }
    }
    if (cpl == kGatherQuads) {   // coil quads (forward only)
        if constexpr (fwd) go(k_gather<D, J, ND, 1, MODE, 4, false>, false);
        else return cudaErrorInvalidValue;
    } else if (cpl == 0) {   // coil pairs
        go(k_gather<D, J, ND, 1, MODE, 2, false>, false);
    } else if (cpl == 1) {
        constexpr bool narrow = gather_narrow(D, J, ND, MODE, 1, 1);
        constexpr int few = D == 3 && narrow ? (MODE == GM_VJP && (J == 6 || J == 7) ? 3 : (fwd && J == 8 ? 1 : 0)) : 0;
        if constexpr (few > 0) {   // up to so many coils: the other blocks
            if (a.C <= few) {
                go(k_gather<D, J, ND, 1, MODE, 1, false>, false);
                return cudaGetLastError();
            }
        }
        go(k_gather<D, J, ND, 1, MODE, 1, narrow>, narrow);
    } else {
        go(k_gather<D, J, ND, 4, MODE, 1, true>, true);   // C up to 4 G = 128
    }
    return cudaGetLastError();
}

template <int D, int J>
static cudaError_t gather_mode(GatherMode mode, const GatherArgs& a, int cpl, cudaStream_t s) {
    if (mode == GM_FWD) return gather_cpl<D, J, 1, GM_FWD>(a, cpl, s);
    if constexpr (D > 1) {
        if (mode == GM_FWD_SORTED) return gather_cpl<D, J, 1, GM_FWD_SORTED>(a, cpl, s);
    }
    if (mode == GM_VJP) return gather_cpl<D, J, D, GM_VJP>(a, cpl, s);
    if (a.nd == D) return gather_cpl<D, J, D, GM_JVP>(a, cpl, s);
    return gather_cpl<D, J, D + 1, GM_JVP>(a, cpl, s);
}

template <int D>
cudaError_t gather_dim(GatherMode mode, const GatherArgs& a, int cpl, cudaStream_t s) {
    switch (a.J) {
        case 4: return gather_mode<D, 4>(mode, a, cpl, s);
        case 5: return gather_mode<D, 5>(mode, a, cpl, s);
        case 6: return gather_mode<D, 6>(mode, a, cpl, s);
        case 7: return gather_mode<D, 7>(mode, a, cpl, s);
        default: return gather_mode<D, 8>(mode, a, cpl, s);
    }
}

}  // namespace nj

// Device side of af_patch_step: one Active Flux time step (Section 2 of
// arXiv 2205.07572) on GB300 (sm_103a).  Included by af_step_f32.cu,
// af_step_f64.cu, af_step_f32_n16.cu and af_step_f32_n32.cu, which
// instantiate the launchers (per precision; FP32 also per patch size).
//
// One CTA advances one tile (<= TMX x TMY cells) of one patch:
//   stage  - the tile's degrees of freedom plus a one-cell halo are copied to
//            shared memory: a tile spanning the patch's interior columns by
//            one bulk (TMA) copy of its window rows per plane completing on
//            an mbarrier, other tiles element by element with cp.async; halo
//            entries in a direction with a same-level neighbour are read
//            straight from that neighbour's interior (the same-level ghost
//            copy of Section 3.1 fused into the load), other directions from
//            the patch's own ghost ring;
//   nodes  - one thread per node-cell evolves the corner, left-edge midpoint
//            and bottom-edge midpoint of its cell to t^{n+1/2} and t^{n+1}
//            (Eq. advection-update / Eq. ERFormula) as constant-weight
//            stencils, keeps T = Q^n + 4 Q^{n+1/2} + Q^{n+1} in shared memory
//            and writes Q^{n+1} to the output (FP32 acoustics: T and Q^{n+1}
//            accumulated together by packed FP32x2 multiply-adds);
//   update - one thread per cell forms the four face fluxes by the space-time
//            Simpson rule (Eq. Simpson-2d: f is linear, so the 3 x 3 sum is
//            f((T_lo + 4 T_mid + T_hi) / 36)) and applies Eq. 2dfv; a
//            bulk-staged tile also writes its rows' ghost columns, so whole
//            lattice rows go out.
// No tensor cores: the stencil is not a dense contraction.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "af_internal.h"
#include "af_launch.cuh"

namespace af {

template <typename T>
struct StepArgs {
    const af_work *work;
    const T *in;
    T *out;
    double *freg;
    int64_t plane;   // plane stride (elements)
    int n, ncomp;
    T dtdx, dtdy;    // dt/dx and dt/dy (the same on every level)
    T fx, fy;        // flux scale: advection a/36, b/36; acoustics c/36
    double dt0;      // level-0 time step (flux registers)
    uint32_t swap;   // bit l set: level l reads `out` and writes `in`
};

// Buffers of a work item of level l: read the current values, write the new.
template <typename T>
__device__ __forceinline__ const T *src_buf(const StepArgs<T> &A, int level) {
    return ((A.swap >> level) & 1u) ? A.out : A.in;
}
template <typename T>
__device__ __forceinline__ T *dst_buf(const StepArgs<T> &A, int level) {
    return ((A.swap >> level) & 1u) ? const_cast<T *>(A.in) : A.out;
}

template <typename T, int EQ>
struct WeightsOf;
template <typename T>
struct WeightsOf<T, AF_ACOUSTICS> { using type = AcousticSymWeights<T>; };
template <>
struct WeightsOf<float, AF_ACOUSTICS> { using type = AcousticPairWeights; };
template <typename T>
struct WeightsOf<T, AF_ADVECTION> { using type = AdvectionPairWeights<T>; };

// Launch one af_patch_step with compiled tiling k (host; af_step_f32/f64.cu).
template <typename T, int EQ>
af_status launch_step(int k, const StepArgs<T> &A, const typename WeightsOf<T, EQ>::type &W, int nwork,
                      cudaStream_t stream);

namespace dev {

__device__ __forceinline__ int dir_index(int sx, int sy) {
    if (sy == 0) return sx < 0 ? 0 : 1;
    if (sx == 0) return sy < 0 ? 2 : 3;
    return 4 + (sx > 0 ? 1 : 0) + (sy > 0 ? 2 : 0);
}

__device__ __forceinline__ void cp_async(float *smem, const float *gmem) {
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async(double *smem, const double *gmem) {
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Issue (without waiting) the copies of the window of node lines
// [x0-1, x1+1] x [y0-1, y1+1] of every plane of work item wk into Sin
// (row pitch WX, plane size WSZ).
// NC, NN: components and patch size when known at compile time (0: read
// them from A), so plane offsets become immediates.
template <typename T, int NT, int WX, int WSZ, int NC = 0, int NN = 0>
__device__ __forceinline__ void stage_issue(const StepArgs<T> &A, const af_work &wk, T *Sin) {
    const int patch = wk.patch, x0 = wk.x0, y0 = wk.y0;
    const T *const in = src_buf(A, wk.level);
    const int ww = wk.x1 - x0 + 3, wh = wk.y1 - y0 + 3;
    int nb[8];
#pragma unroll
    for (int d = 0; d < 8; ++d) nb[d] = wk.nbr[d];
    const int n = NN > 0 ? NN : A.n, W = n + 2 * kGhost + 1;
    const int plane = NN > 0 ? (int)plane_stride(NN) : (int)A.plane;
    const int ncp = (NC > 0 ? NC : A.ncomp) * kPlanes;
    const int64_t pw = (int64_t)ncp * plane;
    // positions enumerated with the compile-time window pitch WX (cheap
    // division); columns beyond the tile's window width are skipped
    for (int pos = threadIdx.x; pos < WX * wh; pos += NT) {
        const int row = pos / WX, col = pos - row * WX;
        if (col >= ww) continue;
        const int li = x0 - 1 + col, lj = y0 - 1 + row;
        const int sx = li < 0 ? -1 : (li >= n ? 1 : 0);
        const int sy = lj < 0 ? -1 : (lj >= n ? 1 : 0);
        int src = patch, si = li, sj = lj;
        if (sx | sy) {
            const int d = dir_index(sx, sy);
            int q = nb[0];
#pragma unroll
            for (int e = 1; e < 8; ++e) q = (d == e) ? nb[e] : q;
            if (q >= 0) {
                src = q;
                si = li - sx * n;
                sj = lj - sy * n;
            }
        }
        const T *g = in + (int64_t)src * pw + ((sj + kGhost) * W + (si + kGhost));
        T *sp = Sin + row * WX + col;
#pragma unroll 4
        for (int cp = 0; cp < ncp; ++cp) {
            cp_async(sp, g);
            sp += WSZ;
            g += plane;
        }
    }
}

// For a patch that advances its ghost layer, write the staged entries of the
// tile's share of the patch lattice to the output, so the output holds a
// complete patch: the entries the step does not write (the outer ghost ring
// and the lines beyond the advanced ones).
template <typename T, int NT, int WX, int WSZ, int NC = 0, int NN = 0>
__device__ __forceinline__ void stage_copy_out(const StepArgs<T> &A, const af_work &wk, const T *Sin) {
    T *const out = dst_buf(A, wk.level);
    const int patch = wk.patch, x0 = wk.x0, y0 = wk.y0, x1 = wk.x1, y1 = wk.y1;
    const int ww = x1 - x0 + 3, wh = y1 - y0 + 3;
    const int n = NN > 0 ? NN : A.n, W = n + 2 * kGhost + 1;
    const int plane = NN > 0 ? (int)plane_stride(NN) : (int)A.plane;
    const int ncp = (NC > 0 ? NC : A.ncomp) * kPlanes;
    const int64_t pw = (int64_t)ncp * plane;
    const int cxlo = x0 == -1 ? -2 : x0, cxhi = x1 == n + 1 ? n + 3 : x1;
    const int cylo = y0 == -1 ? -2 : y0, cyhi = y1 == n + 1 ? n + 3 : y1;
    // the node lines the step stores (as in tile_nodes)
    const int sxhi = x1 == n + 1 ? x1 : x1 - 1, syhi = y1 == n + 1 ? y1 : y1 - 1;
    for (int pos = threadIdx.x; pos < ww * wh; pos += NT) {
        const int row = pos / ww, col = pos - row * ww;
        const int li = x0 - 1 + col, lj = y0 - 1 + row;
        if (li >= cxlo && li < cxhi && lj >= cylo && lj < cyhi) {
            // planes whose entry here the step writes afterwards are skipped:
            // averages of the tile's cells, corners on the stored node lines,
            // left-edge midpoints on stored lines i beside the tile's rows,
            // bottom-edge midpoints on stored lines j below its columns
            const bool cx = li >= x0 && li < x1, cy = lj >= y0 && lj < y1;
            const bool nx = li >= x0 && li <= sxhi, ny = lj >= y0 && lj <= syhi;
            const unsigned written = (cx && cy ? 1u << kAvg : 0u) | (nx && cy ? 1u << kXmid : 0u) |
                                     (nx && ny ? 1u << kCorner : 0u) | (cx && ny ? 1u << kYmid : 0u);
            if (written == 0xFu) continue;
            T *o = out + (int64_t)patch * pw + (int64_t)(lj + kGhost) * W + (li + kGhost);
            const T *sp = Sin + row * WX + col;
            for (int cp = 0; cp < ncp; ++cp)
                if (!((written >> (cp % kPlanes)) & 1u)) o[cp * plane] = sp[cp * WSZ];
        }
    }
}

// Position of block entry k (see af_internal.h) relative to (i-1, j-1).
__host__ __device__ constexpr int blk_plane(int k) {
    return k < 4 ? kAvg : (k < 13 ? kCorner : (k < 19 ? kXmid : kYmid));
}
__host__ __device__ constexpr int blk_a(int k) {
    return k < 4 ? (k & 1) : (k < 13 ? (k - 4) % 3 : (k < 19 ? (k - 13) % 3 : (k - 19) % 2));
}
__host__ __device__ constexpr int blk_b(int k) {
    return k < 4 ? (k >> 1) : (k < 13 ? (k - 4) / 3 : (k < 19 ? (k - 13) / 3 : (k - 19) / 2));
}

// Orbit sums of a quad (++, +-, -+, --): symmetric, x-antisymmetric,
// y-antisymmetric parts.
template <typename T>
__device__ __forceinline__ void quad(T pp, T pm, T mp, T mm, T &ss, T &as, T &sa) {
    const T a = pp + pm, b = mp + mm;
    ss = a + b;
    as = a - b;
    sa = (pp - pm) + (mp - mm);
}

// A product rounded on its own (never contracted into a sum).
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// acc += w . v as one chain of fused multiply-adds
template <int N, typename T>
__device__ __forceinline__ void dot(T &acc, const T *w, const T *v) {
#pragma unroll
    for (int k = 0; k < N; ++k) acc = fma(w[k], v[k], acc);
}

// Acoustic node evaluation of one node-cell item (window coords qi, rj of
// node line (i, j)) with the mirror-folded weights: the 25 block values of
// each input component are combined into the orbit sums of the three nodes,
// then p += A.SS_p + Dx.AS_u + Dy.SA_v, u += A.SS_u + Dx.AS_p,
// v += A.SS_v + Dy.SA_p (the evolution operators of Eq. ERFormula).
// out: T and Q^{n+1} of corner (tc, nc), left-edge mid (tx, nx) and
// bottom-edge mid (ty, ny) for p, u, v.
template <typename T, int WX, int WSZ, bool PK = true>
__device__ __forceinline__ void acoustic_item(const AcousticSymWeights<T> &W, const T *Sin, int qi, int rj,
                                              T tc[3], T nc[3], T tx[3], T nx[3], T ty[3], T ny[3]) {
#pragma unroll
    for (int o = 0; o < 3; ++o) tc[o] = nc[o] = tx[o] = nx[o] = ty[o] = ny[o] = T(0);
    const T *base = Sin + (rj - 1) * WX + (qi - 1);
#pragma unroll
    for (int ci = 0; ci < 3; ++ci) {
        T b[25];
#pragma unroll
        for (int k = 0; k < 25; ++k) b[k] = base[(ci * kPlanes + blk_plane(k)) * WSZ + blk_b(k) * WX + blk_a(k)];
        // ---- corner node
        T css[9], cas[6], csa[6];
        quad(b[3], b[1], b[2], b[0], css[0], cas[0], csa[0]);
        quad(b[12], b[6], b[10], b[4], css[1], cas[1], csa[1]);
        quad(b[18], b[15], b[16], b[13], css[2], cas[2], csa[2]);
        quad(b[24], b[20], b[23], b[19], css[3], cas[3], csa[3]);
        css[4] = b[9] + b[7];   cas[4] = b[9] - b[7];
        css[5] = b[22] + b[21]; cas[5] = b[22] - b[21];
        css[6] = b[11] + b[5];  csa[4] = b[11] - b[5];
        css[7] = b[17] + b[14]; csa[5] = b[17] - b[14];
        css[8] = b[8];
        // ---- left-edge midpoint
        T xss[6], xas[4], xsa[3];
        quad(b[12], b[9], b[10], b[7], xss[0], xas[0], xsa[0]);
        quad(b[24], b[22], b[23], b[21], xss[1], xas[1], xsa[1]);
        xss[2] = b[3] + b[2];   xas[2] = b[3] - b[2];
        xss[3] = b[18] + b[16]; xas[3] = b[18] - b[16];
        xss[4] = b[11] + b[8];  xsa[2] = b[11] - b[8];
        xss[5] = b[17];
        // ---- bottom-edge midpoint
        T yss[6], yas[3], ysa[4];
        quad(b[12], b[6], b[11], b[5], yss[0], yas[0], ysa[0]);
        quad(b[18], b[15], b[17], b[14], yss[1], yas[1], ysa[1]);
        yss[2] = b[9] + b[8];   yas[2] = b[9] - b[8];
        yss[3] = b[3] + b[1];   ysa[2] = b[3] - b[1];
        yss[4] = b[24] + b[20]; ysa[3] = b[24] - b[20];
        yss[5] = b[22];
        if (ci == 0) {  // p: A on p; Dx.AS_p -> u; Dy.SA_p -> v
            dot<9>(tc[0], W.cA[0], css); dot<9>(nc[0], W.cA[1], css);
            dot<6>(tx[0], W.xA[0], xss); dot<6>(nx[0], W.xA[1], xss);
            dot<6>(ty[0], W.yA[0], yss); dot<6>(ny[0], W.yA[1], yss);
            dot<6>(tc[1], W.cDx[0], cas); dot<6>(nc[1], W.cDx[1], cas);
            dot<4>(tx[1], W.xDx[0], xas); dot<4>(nx[1], W.xDx[1], xas);
            dot<3>(ty[1], W.yDx[0], yas); dot<3>(ny[1], W.yDx[1], yas);
            dot<6>(tc[2], W.cDy[0], csa); dot<6>(nc[2], W.cDy[1], csa);
            dot<3>(tx[2], W.xDy[0], xsa); dot<3>(nx[2], W.xDy[1], xsa);
            dot<4>(ty[2], W.yDy[0], ysa); dot<4>(ny[2], W.yDy[1], ysa);
        } else if (ci == 1) {  // u: A on u; Dx.AS_u -> p
            dot<9>(tc[1], W.cA[0], css); dot<9>(nc[1], W.cA[1], css);
            dot<6>(tx[1], W.xA[0], xss); dot<6>(nx[1], W.xA[1], xss);
            dot<6>(ty[1], W.yA[0], yss); dot<6>(ny[1], W.yA[1], yss);
            dot<6>(tc[0], W.cDx[0], cas); dot<6>(nc[0], W.cDx[1], cas);
            dot<4>(tx[0], W.xDx[0], xas); dot<4>(nx[0], W.xDx[1], xas);
            dot<3>(ty[0], W.yDx[0], yas); dot<3>(ny[0], W.yDx[1], yas);
        } else {  // v: A on v; Dy.SA_v -> p
            dot<9>(tc[2], W.cA[0], css); dot<9>(nc[2], W.cA[1], css);
            dot<6>(tx[2], W.xA[0], xss); dot<6>(nx[2], W.xA[1], xss);
            dot<6>(ty[2], W.yA[0], yss); dot<6>(ny[2], W.yA[1], yss);
            dot<6>(tc[0], W.cDy[0], csa); dot<6>(nc[0], W.cDy[1], csa);
            dot<3>(tx[0], W.xDy[0], xsa); dot<3>(nx[0], W.xDy[1], xsa);
            dot<4>(ty[0], W.yDy[0], ysa); dot<4>(ny[0], W.yDy[1], ysa);
        }
    }
}

// acc += (w[k][0], w[k][1]) * v[k] over k, both lanes at once (packed FP32x2
// multiply-add; each lane rounds like the scalar fma chain).
template <int N>
__device__ __forceinline__ void dot2(float2 &acc, const float (*w)[2], const float *v) {
#pragma unroll
    for (int k = 0; k < N; ++k) acc = __ffma2_rn(make_float2(w[k][0], w[k][1]), make_float2(v[k], v[k]), acc);
}

// quad() in FP32 with its two partial sums as one packed add: the lanes
// (pp, mp) and (pm, mm) give a = pp + pm and b = mp + mm together, and
// (pp, mp) - (pm, mm) (a multiply-add by -1, exact before its one rounding)
// gives pp - pm and mp - mm together.  Every result is rounded as in quad().
__device__ __forceinline__ void quad2(float pp, float pm, float mp, float mm, float &ss, float &as, float &sa) {
    const float2 s = __fadd2_rn(make_float2(pp, mp), make_float2(pm, mm));
    ss = s.x + s.y;
    as = s.x - s.y;
    const float2 d = __ffma2_rn(make_float2(pm, mm), make_float2(-1.f, -1.f), make_float2(pp, mp));
    sa = d.x + d.y;
}

// FP32 acoustic node evaluation: as acoustic_item, with the T and Q^{n+1}
// accumulators of every node value packed in one float2.  The corner node's
// four quads take quad2, with the lane pairs (b3, b2), (b1, b0), (b12, b10),
// (b6, b4), (b18, b16), (b15, b13), (b24, b23), (b20, b19).  The edge
// midpoints' quads stay scalar: with them too the kernel no longer fits its
// register budget (measured slower), and the bottom-edge quads would pair b12,
// b6, b18 and b15 with other partners.  PK = false keeps all quads scalar
// (whole-patch tiles, which spill with the pairs).
template <typename T, int WX, int WSZ, bool PK = true>
__device__ __forceinline__ void acoustic_item(const AcousticPairWeights &W, const float *Sin, int qi, int rj,
                                              float tc[3], float nc[3], float tx[3], float nx[3], float ty[3],
                                              float ny[3]) {
    float2 c2[3], x2[3], y2[3];
#pragma unroll
    for (int o = 0; o < 3; ++o) c2[o] = x2[o] = y2[o] = make_float2(0.f, 0.f);
    const float *base = Sin + (rj - 1) * WX + (qi - 1);
#pragma unroll
    for (int ci = 0; ci < 3; ++ci) {
        float b[25];
#pragma unroll
        for (int k = 0; k < 25; ++k) b[k] = base[(ci * kPlanes + blk_plane(k)) * WSZ + blk_b(k) * WX + blk_a(k)];
        float css[9], cas[6], csa[6];
        if constexpr (PK) {
            quad2(b[3], b[1], b[2], b[0], css[0], cas[0], csa[0]);
            quad2(b[12], b[6], b[10], b[4], css[1], cas[1], csa[1]);
            quad2(b[18], b[15], b[16], b[13], css[2], cas[2], csa[2]);
            quad2(b[24], b[20], b[23], b[19], css[3], cas[3], csa[3]);
        } else {
            quad(b[3], b[1], b[2], b[0], css[0], cas[0], csa[0]);
            quad(b[12], b[6], b[10], b[4], css[1], cas[1], csa[1]);
            quad(b[18], b[15], b[16], b[13], css[2], cas[2], csa[2]);
            quad(b[24], b[20], b[23], b[19], css[3], cas[3], csa[3]);
        }
        css[4] = b[9] + b[7];   cas[4] = b[9] - b[7];
        css[5] = b[22] + b[21]; cas[5] = b[22] - b[21];
        css[6] = b[11] + b[5];  csa[4] = b[11] - b[5];
        css[7] = b[17] + b[14]; csa[5] = b[17] - b[14];
        css[8] = b[8];
        float xss[6], xas[4], xsa[3];
        quad(b[12], b[9], b[10], b[7], xss[0], xas[0], xsa[0]);
        quad(b[24], b[22], b[23], b[21], xss[1], xas[1], xsa[1]);
        xss[2] = b[3] + b[2];   xas[2] = b[3] - b[2];
        xss[3] = b[18] + b[16]; xas[3] = b[18] - b[16];
        xss[4] = b[11] + b[8];  xsa[2] = b[11] - b[8];
        xss[5] = b[17];
        float yss[6], yas[3], ysa[4];
        quad(b[12], b[6], b[11], b[5], yss[0], yas[0], ysa[0]);
        quad(b[18], b[15], b[17], b[14], yss[1], yas[1], ysa[1]);
        yss[2] = b[9] + b[8];   yas[2] = b[9] - b[8];
        yss[3] = b[3] + b[1];   ysa[2] = b[3] - b[1];
        yss[4] = b[24] + b[20]; ysa[3] = b[24] - b[20];
        yss[5] = b[22];
        if (ci == 0) {
            dot2<9>(c2[0], W.cA, css);  dot2<6>(x2[0], W.xA, xss);  dot2<6>(y2[0], W.yA, yss);
            dot2<6>(c2[1], W.cDx, cas); dot2<4>(x2[1], W.xDx, xas); dot2<3>(y2[1], W.yDx, yas);
            dot2<6>(c2[2], W.cDy, csa); dot2<3>(x2[2], W.xDy, xsa); dot2<4>(y2[2], W.yDy, ysa);
        } else if (ci == 1) {
            dot2<9>(c2[1], W.cA, css);  dot2<6>(x2[1], W.xA, xss);  dot2<6>(y2[1], W.yA, yss);
            dot2<6>(c2[0], W.cDx, cas); dot2<4>(x2[0], W.xDx, xas); dot2<3>(y2[0], W.yDx, yas);
        } else {
            dot2<9>(c2[2], W.cA, css);  dot2<6>(x2[2], W.xA, xss);  dot2<6>(y2[2], W.yA, yss);
            dot2<6>(c2[0], W.cDy, csa); dot2<3>(x2[0], W.xDy, xsa); dot2<4>(y2[0], W.yDy, ysa);
        }
    }
#pragma unroll
    for (int o = 0; o < 3; ++o) {
        tc[o] = c2[o].x; nc[o] = c2[o].y;
        tx[o] = x2[o].x; nx[o] = x2[o].y;
        ty[o] = y2[o].x; ny[o] = y2[o].y;
    }
}

// Advection: the nine degrees of freedom of window cell (cq, cr) in the order
// of the weights, and combinations of them.
template <typename T, int WX, int WSZ>
__device__ __forceinline__ void adv_cell(const T *Sin, int cq, int cr, T d[9]) {
    const int o = cr * WX + cq;
    const T *A = Sin + kAvg * WSZ, *C = Sin + kCorner * WSZ, *X = Sin + kXmid * WSZ, *Y = Sin + kYmid * WSZ;
    d[0] = A[o];
    d[1] = C[o];
    d[2] = C[o + 1];
    d[3] = C[o + WX];
    d[4] = C[o + WX + 1];
    d[5] = X[o];
    d[6] = X[o + 1];
    d[7] = Y[o];
    d[8] = Y[o + WX];
}
// Combination s of one cell's values.
template <typename T, int WX, int WSZ>
__device__ __forceinline__ T adv_eval(const T (*w)[2], int s, const T *Sin, int cq, int cr) {
    T d[9];
    adv_cell<T, WX, WSZ>(Sin, cq, cr, d);
    T v = w[0][s] * d[0];
#pragma unroll
    for (int k = 1; k < 9; ++k) v = fma(w[k][s], d[k], v);
    return v;
}
// Both combinations of one cell's values (FP32: packed, each lane rounded as
// alone).
template <int WX, int WSZ>
__device__ __forceinline__ void adv_eval2(const float (*w)[2], const float *Sin, int cq, int cr, float &v0, float &v1) {
    float d[9];
    adv_cell<float, WX, WSZ>(Sin, cq, cr, d);
    float2 v = __fmul2_rn(make_float2(w[0][0], w[0][1]), make_float2(d[0], d[0]));
#pragma unroll
    for (int k = 1; k < 9; ++k) v = __ffma2_rn(make_float2(w[k][0], w[k][1]), make_float2(d[k], d[k]), v);
    v0 = v.x;
    v1 = v.y;
}
template <int WX, int WSZ>
__device__ __forceinline__ void adv_eval2(const double (*w)[2], const double *Sin, int cq, int cr, double &v0,
                                          double &v1) {
    double d[9];
    adv_cell<double, WX, WSZ>(Sin, cq, cr, d);
    v0 = w[0][0] * d[0];
    v1 = w[0][1] * d[0];
#pragma unroll
    for (int k = 1; k < 9; ++k) {
        v0 = fma(w[k][0], d[k], v0);
        v1 = fma(w[k][1], d[k], v1);
    }
}

// T and Q^{n+1} of a node of type t at window entry (qi, rj), lattice plane
// `plane` (see AdvectionPairWeights): with the weights folded, nine values and
// two combinations, for eighteen values, two combinations and the time sum.
// FP32 is bound by its shared-memory loads and issue slots, FP64 by its pipe
// (20 operations a node before, 18 now): FP32 4096^2 cells in 16 x 16 patches
// 333 -> 241 us, FP64 1024^2 194 -> 162 us.
template <typename T, int WX, int WSZ>
__device__ __forceinline__ void adv_node(const AdvectionPairWeights<T> &W, int t, int plane, const T *Sin, int qi, int rj,
                                         T &sum, T &q1) {
    if (W.fold) {
        adv_eval2<WX, WSZ>(W.v[t], Sin, qi + W.off[t][1][0], rj + W.off[t][1][1], sum, q1);
    } else {
        const T qh = adv_eval<T, WX, WSZ>(W.v[t], 0, Sin, qi + W.off[t][0][0], rj + W.off[t][0][1]);
        q1 = adv_eval<T, WX, WSZ>(W.v[t], 1, Sin, qi + W.off[t][1][0], rj + W.off[t][1][1]);
        sum = fma(T(4), qh, Sin[plane * WSZ + rj * WX + qi]) + q1;
    }
}

// The T arrays of a tile in shared memory: T of the corner, left-edge and
// bottom-edge node (0, 1, 2) of component c at node-cell s.  FP32 acoustics
// keeps a node's components together -- (p, u, v) of the corner in 16 bytes, (p,
// u) of the left-edge and (p, v) of the bottom-edge node in 8; the other two
// enter no flux -- so that a node-cell is written by three stores and a cell
// reads its faces by eight loads, for nine and twenty: the step is bound by
// issue slots (4096^2 cells in 32 x 8 tiles 470 -> 466 us, 2048^2 in 16 x 16
// tiles 174 -> 164, adaptive acoustics on 5436 leaves 1240 -> 1201).
template <typename T, int EQ, int TSZ>
struct TArrays {
    static constexpr bool packed = EQ == AF_ACOUSTICS && sizeof(T) == 4;
    static __device__ __forceinline__ T get(const T *ST, int node, int c, int s) {
        if constexpr (packed)
            return node == 0 ? ST[4 * s + c] : ST[(2 + 2 * node) * TSZ + 2 * s + (c == 0 ? 0 : 1)];
        else
            return ST[(c * 3 + node) * TSZ + s];
    }
};

// Tile width whose node and cell items are enumerated with a compile-time
// pitch (tile_nodes, tile_fluxes).
template <int TMX, int NN>
__host__ __device__ constexpr int fast_width() {
    return (NN > 0 && TMX == NN + 2) ? NN : TMX;
}

// Point values of one staged tile (Eq. advection-update / Eq. ERFormula):
// Q^{n+1} of every node the tile owns to the output, T = Q^n + 4 Q^{n+1/2}
// + Q^{n+1} to ST.  Sin: window (pitch WX, plane size WSZ); ST: T arrays
// (pitch TX, size TSZ).  The caller synchronises before tile_fluxes.
template <typename T, int EQ, int NT, int WX, int WSZ, int TX, int TSZ, int TMX = TX - 1, int NN = 0>
__device__ __forceinline__ void tile_nodes(const StepArgs<T> &A, const typename WeightsOf<T, EQ>::type &W,
                                           const T *Sin, T *ST, int patch, int level, int x0, int x1, int y0,
                                           int y1) {
    constexpr int ncomp = (EQ == AF_ACOUSTICS) ? 3 : 1;
    const int tw = x1 - x0, th = y1 - y0;
    const int n = NN > 0 ? NN : A.n, W_ = n + 2 * kGhost + 1;
    const int plane = NN > 0 ? (int)plane_stride(NN) : (int)A.plane;
    const int64_t pw = (int64_t)ncomp * kPlanes * plane;
    T *outp = dst_buf(A, level) + (int64_t)patch * pw;
    // node lines stored by this tile: [x0, x1) plus x1 itself when the tile
    // ends on the outer edge of the advanced first ghost layer
    const int sxhi = (x1 == n + 1) ? x1 : x1 - 1;
    const int syhi = (y1 == n + 1) ? y1 : y1 - 1;

    // ---- point values.  Node-cells (ii, jj), ii in [0, tw], jj in [0, th].
    // A tile of the fast width FW (tw == FW) enumerates columns [0, FW) with
    // the compile-time pitch FW -- one warp covers consecutive words of one
    // row, so the block loads are free of bank conflicts -- and its last node
    // column (ii = FW) as a short list after them; other tiles use the pitch
    // tw + 1.  FW is the tiling's width, except in a tiling two cells wider
    // than patches of a compile-time size NN (built for whole patches with
    // their first ghost layer), where it is NN: the tiles of patches that
    // advance only their interior.
    constexpr int FW = fast_width<TMX, NN>();
    const bool full = (tw == FW);
    const int pitch = full ? FW : tw + 1;
    const int nmain = pitch * (th + 1);
    const int nitems = nmain + (full ? th + 1 : 0);
    for (int it = threadIdx.x; it < nitems; it += NT) {
        int jj, ii;
        if (it < nmain) {
            if (full) {
                jj = it / FW;
                ii = it - jj * FW;
            } else {
                jj = it / pitch;
                ii = it - jj * pitch;
            }
        } else {
            jj = it - nmain;
            ii = FW;
        }
        const int i = x0 + ii, j = y0 + jj;
        const int qi = ii + 1, rj = jj + 1;
        const bool hx = j < y1, hy = i < x1;            // edge midpoints that exist
        const bool st_x = i <= sxhi, st_y = j <= syhi;  // stored lines
        T *const ob = outp + ((j + kGhost) * W_ + (i + kGhost));  // this node-cell in plane 0 of comp 0
        const int so = jj * TX + ii;
        if constexpr (EQ == AF_ACOUSTICS) {
            T tc[3], nc[3], tx[3], nx[3], ty[3], ny[3];
            acoustic_item<T, WX, WSZ, TMX != NN + 2>(W, Sin, qi, rj, tc, nc, tx, nx, ty, ny);
            if constexpr (TArrays<T, EQ, TSZ>::packed) {
                *reinterpret_cast<float4 *>(ST + 4 * so) = make_float4(tc[0], tc[1], tc[2], 0.f);
                *reinterpret_cast<float2 *>(ST + 4 * TSZ + 2 * so) = make_float2(tx[0], tx[1]);
                *reinterpret_cast<float2 *>(ST + 6 * TSZ + 2 * so) = make_float2(ty[0], ty[2]);
            }
#pragma unroll
            for (int o = 0; o < 3; ++o) {
                if constexpr (!TArrays<T, EQ, TSZ>::packed) {
                    ST[(o * 3 + 0) * TSZ + so] = tc[o];
                    ST[(o * 3 + 1) * TSZ + so] = tx[o];
                    ST[(o * 3 + 2) * TSZ + so] = ty[o];
                }
                T *po = ob + o * kPlanes * plane;
                if (st_x && st_y) __stcs(po + kCorner * plane, nc[o]);
                if (st_x && hx) __stcs(po + kXmid * plane, nx[o]);
                if (hy && st_y) __stcs(po + kYmid * plane, ny[o]);
            }
        } else {
            T sum, q1;
            adv_node<T, WX, WSZ>(W, 0, kCorner, Sin, qi, rj, sum, q1);
            ST[0 * TSZ + so] = sum;
            if (st_x && st_y) ob[kCorner * plane] = q1;
            if (hx) {
                adv_node<T, WX, WSZ>(W, 1, kXmid, Sin, qi, rj, sum, q1);
                ST[1 * TSZ + so] = sum;
                if (st_x) ob[kXmid * plane] = q1;
            }
            if (hy) {
                adv_node<T, WX, WSZ>(W, 2, kYmid, Sin, qi, rj, sum, q1);
                ST[2 * TSZ + so] = sum;
                if (st_y) ob[kYmid * plane] = q1;
            }
        }
    }
}

// Fluxes (Eq. Simpson-2d) and the update (Eq. 2dfv) of one tile whose T
// arrays tile_nodes has written; reads the cell averages from the window.
// FREG: adaptive runs, whose flux registers take the rounded face fluxes: in
// FP32 the update takes the same ones, rounded before their difference (uniform
// runs and FP64 leave one product in the difference's multiply-add).
template <typename T, int EQ, int NT, int WX, int WSZ, int TX, int TSZ, int TMX, int NN, bool FREG>
__device__ __forceinline__ void tile_fluxes(const StepArgs<T> &A, const T *Sin, const T *ST, int patch, int level,
                                            int x0, int x1, int y0, int y1) {
    constexpr int ncomp = (EQ == AF_ACOUSTICS) ? 3 : 1;
    const int tw = x1 - x0, th = y1 - y0;
    const int n = NN > 0 ? NN : A.n, W_ = n + 2 * kGhost + 1;
    const int plane = NN > 0 ? (int)plane_stride(NN) : (int)A.plane;
    const int64_t pw = (int64_t)ncomp * kPlanes * plane;
    T *outp = dst_buf(A, level) + (int64_t)patch * pw;
    constexpr int FW = fast_width<TMX, NN>();  // as in tile_nodes
    const bool full = (tw == FW);
    for (int it = threadIdx.x; it < tw * th; it += NT) {
        int jj, ii;
        if (full) {
            jj = it / FW;
            ii = it - jj * FW;
        } else {
            jj = it / tw;
            ii = it - jj * tw;
        }
        const int i = x0 + ii, j = y0 + jj;
        const int s00 = jj * TX + ii;
        T Fl[3], Fr[3], Gb[3], Gt[3];
        if constexpr (TArrays<T, EQ, TSZ>::packed) {
            auto corner = [&](int s) { return *reinterpret_cast<const float4 *>(ST + 4 * s); };
            auto mid = [&](int node, int s) { return *reinterpret_cast<const float2 *>(ST + (2 + 2 * node) * TSZ + 2 * s); };
            const float4 c00 = corner(s00), c10 = corner(s00 + 1), c01 = corner(s00 + TX), c11 = corner(s00 + TX + 1);
            const float2 xl = mid(1, s00), xr = mid(1, s00 + 1), yb = mid(2, s00), yt = mid(2, s00 + TX);
            // time-Simpson sums, as below
            Fl[0] = fma(4.f, xl.x, c00.x) + c01.x;
            Fl[1] = fma(4.f, xl.y, c00.y) + c01.y;
            Fr[0] = fma(4.f, xr.x, c10.x) + c11.x;
            Fr[1] = fma(4.f, xr.y, c10.y) + c11.y;
            Gb[0] = fma(4.f, yb.x, c00.x) + c10.x;
            Gb[2] = fma(4.f, yb.y, c00.z) + c10.z;
            Gt[0] = fma(4.f, yt.x, c01.x) + c11.x;
            Gt[2] = fma(4.f, yt.y, c01.z) + c11.z;
        } else
#pragma unroll
        for (int c = 0; c < ncomp; ++c) {
            const T *Tc = ST + (c * 3 + 0) * TSZ, *Tx = ST + (c * 3 + 1) * TSZ, *Ty = ST + (c * 3 + 2) * TSZ;
            // time-Simpson sums at the three points of each face (the
            // multiply-adds written out, as in the update below)
            Fl[c] = fma(T(4), Tx[s00], Tc[s00]) + Tc[s00 + TX];
            Fr[c] = fma(T(4), Tx[s00 + 1], Tc[s00 + 1]) + Tc[s00 + TX + 1];
            Gb[c] = fma(T(4), Ty[s00], Tc[s00]) + Tc[s00 + 1];
            Gt[c] = fma(T(4), Ty[s00 + TX], Tc[s00 + TX]) + Tc[s00 + TX + 1];
        }
        T fl[3], fr[3], gb[3], gt[3];
        auto flux = [](T k, T s) { return FREG && sizeof(T) == 4 ? mul_rn(k, s) : k * s; };
        if constexpr (EQ == AF_ACOUSTICS) {
            // f = c (u, p, 0), g = c (v, 0, p)
            fl[0] = flux(A.fx, Fl[1]); fl[1] = flux(A.fx, Fl[0]); fl[2] = T(0);
            fr[0] = flux(A.fx, Fr[1]); fr[1] = flux(A.fx, Fr[0]); fr[2] = T(0);
            gb[0] = flux(A.fy, Gb[2]); gb[1] = T(0); gb[2] = flux(A.fy, Gb[0]);
            gt[0] = flux(A.fy, Gt[2]); gt[1] = T(0); gt[2] = flux(A.fy, Gt[0]);
        } else {
            fl[0] = flux(A.fx, Fl[0]); fr[0] = flux(A.fx, Fr[0]);
            gb[0] = flux(A.fy, Gb[0]); gt[0] = flux(A.fy, Gt[0]);
        }
        T *const ob = outp + ((j + kGhost) * W_ + (i + kGhost));
        const int sa = (jj + 1) * WX + (ii + 1);
#pragma unroll
        for (int c = 0; c < ncomp; ++c) {
            // Q - dt/dx (F_r - F_l) - dt/dy (G_t - G_b), the multiply-adds
            // written out so every instantiation rounds alike
            const T q = Sin[(c * kPlanes + kAvg) * WSZ + sa];
            __stcs(ob + c * kPlanes * plane, fma(-A.dtdy, gt[c] - gb[c], fma(-A.dtdx, fr[c] - fl[c], q)));
        }
    }
}

// Adaptive runs: dt_l F of the tile's faces on the patch boundary, added to the
// FP64 flux registers.  One value per thread and turn -- the components whose
// flux is not identically zero, along each side -- read before the flux loop
// and stored after it, so that the registers' latency hides behind the loop.
// (In the loop itself, two lanes of every warp took all warps through the FP64
// multiply-adds of both x sides: 60 warp instructions of that pipe for a
// 16 x 16 tile, 8 now.  Adaptive acoustics on 5436 leaves 1317 -> 1237 us a
// coarse step.)
template <typename T, int EQ, int NT, int TX, int TSZ, int NN>
struct BoundaryFluxes {
    static constexpr int ncomp = (EQ == AF_ACOUSTICS) ? 3 : 1, nz = (EQ == AF_ACOUSTICS) ? 2 : 1;
    static constexpr int kHeld = 2;  // values a thread holds over the flux loop (a 32 x 32 patch on 128 threads)
    double *reg[kHeld];
    double old[kHeld];
    T flux[kHeld];

    // Value t of the tile: its register, and its flux from the T arrays; null
    // if the face is not in the tile.
    static __device__ __forceinline__ double *value(const StepArgs<T> &A, const T *ST, int patch, int x0, int x1, int y0,
                                                    int y1, int t, T &f) {
        const int n = NN > 0 ? NN : A.n;
        const int q = nz * n, side = (t >= q) + (t >= 2 * q) + (t >= 3 * q), r = t - side * q;
        const int z = nz == 2 && r >= n ? 1 : 0, k = r - z * n;
        const bool xs = side < 2;
        const int line = (side & 1) ? n : 0, cell = (side & 1) ? n - 1 : 0;  // the face's node line, its cell inside
        const int lo = xs ? x0 : y0, hi = xs ? x1 : y1, klo = xs ? y0 : x0, khi = xs ? y1 : x1;
        if (cell < lo || cell >= hi || k < klo || k >= khi) return nullptr;
        // f = c (u, p, 0), g = c (v, 0, p): component c of the flux is value v
        const int c = EQ == AF_ACOUSTICS ? (xs ? z : 2 * z) : 0;
        const int v = EQ == AF_ACOUSTICS ? (xs ? 1 - z : 2 - 2 * z) : 0;
        const int s = xs ? (k - y0) * TX + (line - x0) : (line - y0) * TX + (k - x0);
        using TA = TArrays<T, EQ, TSZ>;
        f = mul_rn(xs ? A.fx : A.fy, fma(T(4), TA::get(ST, xs ? 1 : 2, v, s), TA::get(ST, 0, v, s)) +
                                         TA::get(ST, 0, v, s + (xs ? TX : 1)));
        return A.freg + ((int64_t)patch * 4 + side) * ncomp * n + c * n + k;
    }
    __device__ __forceinline__ void begin(const StepArgs<T> &A, const T *ST, int patch, int x0, int x1, int y0, int y1) {
#pragma unroll
        for (int h = 0; h < kHeld; ++h) {
            const int t = threadIdx.x + h * NT, total = 4 * nz * (NN > 0 ? NN : A.n);
            reg[h] = t < total ? value(A, ST, patch, x0, x1, y0, y1, t, flux[h]) : nullptr;
            if (reg[h]) old[h] = *reg[h];
        }
    }
    __device__ __forceinline__ void end(const StepArgs<T> &A, const T *ST, int patch, int level, int x0, int x1, int y0,
                                        int y1) {
        // dt_l = dt0 / 2^level, scaled exactly by the power of two
        const double dtl = A.dt0 * __longlong_as_double((long long)(1023 - level) << 52);
        const int total = 4 * nz * (NN > 0 ? NN : A.n);
#pragma unroll
        for (int h = 0; h < kHeld; ++h)
            if (reg[h]) *reg[h] = old[h] + dtl * (double)flux[h];
        for (int t = threadIdx.x + kHeld * NT; t < total; t += NT) {
            T f;
            double *const p = value(A, ST, patch, x0, x1, y0, y1, t, f);
            if (p) *p += dtl * (double)f;
        }
    }
};

// Point values, then fluxes and update, of one staged tile.
template <typename T, int EQ, int NT, int WX, int WSZ, int TX, int TSZ, int TMX = TX - 1, int NN = 0>
__device__ __forceinline__ void tile_compute(const StepArgs<T> &A, const typename WeightsOf<T, EQ>::type &W,
                                             const T *Sin, T *ST, int patch, int level, int x0, int x1, int y0,
                                             int y1) {
    tile_nodes<T, EQ, NT, WX, WSZ, TX, TSZ, TMX, NN>(A, W, Sin, ST, patch, level, x0, x1, y0, y1);
    __syncthreads();
    // flux registers (adaptive runs) or none: two instantiations, so the
    // uniform grid's loop carries nothing of them
    if (A.freg != nullptr) {
        BoundaryFluxes<T, EQ, NT, TX, TSZ, NN> B;
        B.begin(A, ST, patch, x0, x1, y0, y1);
        tile_fluxes<T, EQ, NT, WX, WSZ, TX, TSZ, TMX, NN, true>(A, Sin, ST, patch, level, x0, x1, y0, y1);
        B.end(A, ST, patch, level, x0, x1, y0, y1);
    } else {
        tile_fluxes<T, EQ, NT, WX, WSZ, TX, TSZ, TMX, NN, false>(A, Sin, ST, patch, level, x0, x1, y0, y1);
    }
}

// Resident CTAs per SM the register allocation must allow: FP32 acoustics
// is issue-bound and needs about 24 warps per SM to hide its shared-memory
// and staging latency (80 registers at 128 threads).
template <typename T, int EQ, int NT>
__host__ __device__ constexpr int min_ctas() {
    return (EQ == AF_ACOUSTICS && sizeof(T) == 4) ? (768 / NT > 0 ? 768 / NT : 1) : 1;
}

// Shared-memory geometry of a TMX x TMY tile.  The window is TMX + 3 node
// columns wide; its pitch is two more, the lattice width of TMX-cell patches,
// so that their full-width tiles can be staged in bulk -- except for a tile
// two cells wider than patches of a compile-time size NN (the whole patch
// with its first ghost layer), whose pitch is the lattice width of NN-cell
// patches: its window is then the whole patch lattice, staged in bulk too.
// Each plane has room for the window origin's offset and the bulk copies'
// rounding to 16 bytes (12 elements), and a size that keeps every plane
// 16-byte aligned.
template <int TMX, int TMY, int NN = 0>
struct Geo {
    static constexpr int WX = (NN > 0 && TMX == NN + 2) ? NN + 2 * kGhost + 1 : TMX + 2 * kGhost + 1;
    static constexpr int WY = TMY + 3, WSZ = (WX * WY + 12 + 3) / 4 * 4;  // window
    static constexpr int TX = TMX + 1, TY = TMY + 1, TSZ = TX * TY;  // T arrays
};

// ---------------------------------------------------------------------------
// Bulk staging.  When the window pitch equals the lattice width (WX = n + 5)
// and the tile spans the patch's interior columns (x0 = 0, x1 = n), the
// window rows y0-1 .. y1+1 of each plane -- ghost columns included -- are one
// contiguous span of the patch lattice, and one bulk (TMA) copy per plane
// stages them, signalling an mbarrier.  Entries in a direction with a
// same-level neighbour are then overwritten with that neighbour's values (the
// fused same-level ghost copy of Section 3.1), exactly the entries the
// element-wise staging takes from the neighbour; the staged window is the same.

// Limit of a wait on a bulk copy: 2^31 SM cycles (about a second), far
// beyond any real copy, and an iteration cap behind it.
constexpr long long kWaitCycles = 1ll << 31;
constexpr unsigned kWaitIters = 1u << 26;

// Tiles whose wait gave up, one counter per translation unit that
// instantiates step kernels (read by wait_timeouts_here).
static __device__ unsigned int g_wait_timeouts;

__device__ __forceinline__ unsigned smem_addr(const void *p) {
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
// One bulk copy global -> shared of `bytes` (both addresses 16-byte aligned,
// bytes a multiple of 16) completing on `bar`.
__device__ __forceinline__ void bulk_copy_g2s(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
// Wait for phase `parity` of `bar`; false if the iteration limit ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity) {
    const unsigned a = smem_addr(bar);
    const long long t0 = clock64();
    for (unsigned it = 0; it < kWaitIters; ++it) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
        if (clock64() - t0 > kWaitCycles) break;
    }
    return false;
}

// A work item read as four 16-byte loads (the work list is 16-byte
// aligned: af_patch_step refuses it otherwise).
__device__ __forceinline__ af_work load_work(const af_work *w) {
    union {
        af_work w;
        int4 v[4];
    } u;
    const int4 *src = reinterpret_cast<const int4 *>(w);
#pragma unroll
    for (int q = 0; q < 4; ++q) u.v[q] = __ldg(src + q);
    return u.w;
}

// Work items prefetched into L2 this many items ahead of the CTA that reads
// them: about one wave of resident CTAs of the 32 x 8 tiling (6 CTAs on each
// of 152 SMs), so the item is in L2 when its CTA starts and the bulk copies
// of its window go out one DRAM round trip earlier.
constexpr int kWorkPrefetch = 912;
__device__ __forceinline__ void prefetch_work(const af_work *w, unsigned idx, unsigned nwork) {
    if (threadIdx.x == 0 && idx < nwork) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(w + idx));
}

// The patch's flux registers (4 sides x ncomp x n doubles), prefetched into
// L2 while the tile is staged: the flux phase reads them back.
template <typename T, int NT>
__device__ __forceinline__ void prefetch_freg(const StepArgs<T> &A, int patch, int ncomp, int n) {
    if (A.freg == nullptr) return;
    const double *p = A.freg + (int64_t)patch * 4 * ncomp * n;
    const int lines = (4 * ncomp * n * 8 + 127) / 128;
    for (int t = threadIdx.x; t < lines; t += NT) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p + 16 * t));
}

// Offset (elements) of the window origin from the start of the shared
// window buffer: room for the rounding of a bulk copy's start down to 16
// bytes, plus the 16-byte phase of the window origin of a tile with y0 = 0.
template <typename T, int WX>
__host__ __device__ constexpr int win_off() {
    return 16 / (int)sizeof(T) + ((kGhost - 1) * WX + kGhost - 1) % (16 / (int)sizeof(T));
}

// True if work item wk is staged in bulk by a kernel with window pitch WX:
// the pitch is the lattice width, the tile spans the interior columns, and
// its window origin has the 16-byte phase win_off assumes (y0 * WX a
// multiple of 16 bytes: every tile of the compiled tilings).
template <typename T, int WX>
__device__ __forceinline__ bool bulk_tile(const StepArgs<T> &A, const af_work &wk) {
    constexpr int E = 16 / (int)sizeof(T);
    return A.n + 2 * kGhost + 1 == WX && wk.x0 == 0 && wk.x1 == A.n && wk.y0 >= 0 && wk.y1 <= A.n &&
           (wk.y0 * WX) % E == 0;
}

// Issue (thread 0) the bulk copies of work item wk (bulk_tile true) into the
// window at Sin (= window buffer + win_off, so that every plane's copy
// starts on a 16-byte boundary), completing on bar.  Nothing is issued for
// an item carrying AF_WORK_SKIP_BULK_COPY, so a wait on bar runs out.
template <typename T, int WX, int WSZ, int NC>
__device__ __forceinline__ void bulk_issue(const StepArgs<T> &A, const af_work &wk, T *Sin, uint64_t *bar) {
    constexpr int n = WX - 2 * kGhost - 1;
    constexpr int E = 16 / (int)sizeof(T);
    constexpr int ncp = NC * kPlanes;
    constexpr int64_t plane = plane_stride(n), pw = ncp * plane;
    if (wk.flags & AF_WORK_SKIP_BULK_COPY) return;
    const int y0 = wk.y0, wh = wk.y1 - y0 + 3;
    const int g_org = (y0 - 1 + kGhost) * WX + (kGhost - 1);  // lattice offset of window entry (0, 0)
    const int g_lo = (g_org - 1) / E * E;                     // row start (lattice column 0), rounded down
    const int g_hi = (g_org - 1 + wh * WX + E - 1) / E * E;    // end of the last row, rounded up
    const unsigned bytes = (unsigned)((g_hi - g_lo) * (int)sizeof(T));
    mbar_expect_tx(bar, bytes * ncp);
    const T *src = src_buf(A, wk.level) + (int64_t)wk.patch * pw + g_lo;
    T *dst = Sin + (g_lo - g_org);
#pragma unroll
    for (int cp = 0; cp < ncp; ++cp) bulk_copy_g2s(dst + cp * WSZ, src + cp * plane, bytes, bar);
}

// Halo list of a bulk-staged tile of n-cell patches: the window entries
// outside the patch interior -- columns -1, n, n+1 of every window row, and
// rows -1 (y0 = 0) and n .. y1+1 of columns 0 .. n-1.  Entry t gets its node
// (li, lj) and returns the same-level neighbour it is read from (*src: the
// lattice offset there), or -1: no such neighbour, the patch's own ghost
// value (staged by the bulk copy) stays.
template <int n>
struct HaloList {
    int y0, wh, nlo, ncol, count;
    __device__ __forceinline__ HaloList(int y0_, int y1) : y0(y0_), wh(y1 - y0_ + 3) {
        nlo = y0 == 0 ? 1 : 0;
        const int nhi = y1 + 2 > n ? y1 + 2 - n : 0;
        ncol = 3 * wh;
        count = ncol + (nlo + nhi) * n;
    }
    __device__ __forceinline__ int entry(const int nb[8], int t, int &li, int &lj, int &src) const {
        if (t < ncol) {
            const int c = t / wh;
            li = c == 0 ? -1 : n - 1 + c;
            lj = y0 - 1 + (t - c * wh);
        } else {
            const int u = t - ncol, r = u / n;
            li = u - r * n;
            lj = r < nlo ? -1 : n + r - nlo;
        }
        const int sx = li < 0 ? -1 : (li >= n ? 1 : 0);
        const int sy = lj < 0 ? -1 : (lj >= n ? 1 : 0);
        const int d = dir_index(sx, sy);
        int q = nb[0];
#pragma unroll
        for (int e = 1; e < 8; ++e) q = (d == e) ? nb[e] : q;
        src = (lj - sy * n + kGhost) * (n + 2 * kGhost + 1) + (li - sx * n + kGhost);
        return q;
    }
};

// Stage work item wk (bulk_tile true) into the window at Sin: bulk copies,
// then the halo entries read with plain loads (issued before the wait) and
// stored once the copies have landed.  Returns false (in every thread) if a
// wait gave up; g_wait_timeouts is then incremented.  Ends with a CTA
// barrier.
template <typename T, int NT, int WX, int WSZ, int NC>
__device__ __forceinline__ bool stage_bulk(const StepArgs<T> &A, const af_work &wk, T *Sin, uint64_t *bar) {
    constexpr int n = WX - 2 * kGhost - 1;
    constexpr int ncp = NC * kPlanes;
    constexpr int64_t plane = plane_stride(n), pw = ncp * plane;
    const T *const in = src_buf(A, wk.level);
    if (threadIdx.x == 0) mbar_init(bar, 1);
    __syncthreads();
    if (threadIdx.x == 0) bulk_issue<T, WX, WSZ, NC>(A, wk, Sin, bar);
    int nb[8];
#pragma unroll
    for (int d = 0; d < 8; ++d) nb[d] = wk.nbr[d];
    const HaloList<n> H(wk.y0, wk.y1);
    bool waited = false, ok = true;
    for (int t = threadIdx.x; t < H.count; t += NT) {
        int li, lj, so;
        const int q = H.entry(nb, t, li, lj, so);
        if (q < 0) continue;
        const T *g = in + (int64_t)q * pw + so;
        T v[ncp];
#pragma unroll
        for (int cp = 0; cp < ncp; ++cp) v[cp] = __ldg(g + cp * plane);
        if (!waited) {  // the bulk copy must land before its entries are overwritten
            ok = mbar_wait(bar, 0);
            waited = true;
        }
        T *sp = Sin + (lj - H.y0 + 1) * WX + (li + 1);
#pragma unroll
        for (int cp = 0; cp < ncp; ++cp) sp[cp * WSZ] = v[cp];
    }
    if (!waited) ok = mbar_wait(bar, 0);
    if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) {
            atomicAdd(&g_wait_timeouts, 1u);
            mbar_wait(bar, 0);  // bounded: give the copies in flight a second chance to land
        }
        return false;
    }
    return true;
}

// True if work item wk is a whole patch with its first ghost layer ([-1,
// n+1)^2) and the window (pitch WX, WY rows) is exactly the patch lattice:
// the window is then one contiguous span of each plane from lattice offset 0.
template <typename T, int WX, int WY>
__device__ __forceinline__ bool ext_bulk_tile(const StepArgs<T> &A, const af_work &wk) {
    return A.n + 2 * kGhost + 1 == WX && WY == WX && wk.x0 == -1 && wk.x1 == A.n + 1 && wk.y0 == -1 &&
           wk.y1 == A.n + 1;
}

// Stage work item wk (ext_bulk_tile true) into the window at Sx (16-byte
// aligned): one bulk copy of each whole plane lattice, then the entries
// outside the patch interior in a direction with a same-level neighbour
// overwritten with that neighbour's values (read with plain loads before the
// wait, stored after it).  Returns false (in every thread) if the wait gave
// up; g_wait_timeouts is then incremented.  Ends with a CTA barrier.
template <typename T, int NT, int WX, int WSZ, int NC>
__device__ __forceinline__ bool stage_bulk_ext(const StepArgs<T> &A, const af_work &wk, T *Sx, uint64_t *bar) {
    constexpr int n = WX - 2 * kGhost - 1;
    constexpr int E = 16 / (int)sizeof(T);
    constexpr int ncp = NC * kPlanes;
    constexpr int64_t plane = plane_stride(n), pw = ncp * plane;
    constexpr unsigned bytes = (unsigned)((WX * WX + E - 1) / E * E * (int)sizeof(T));
    static_assert((WX * WX + E - 1) / E * E <= plane, "the copy stays inside the plane");
    static_assert(E + (WX * WX + E - 1) / E * E <= WSZ, "the copy stays inside the window slot");
    const T *const in = src_buf(A, wk.level);
    if (threadIdx.x == 0) mbar_init(bar, 1);
    __syncthreads();
    if (threadIdx.x == 0 && !(wk.flags & AF_WORK_SKIP_BULK_COPY)) {
        mbar_expect_tx(bar, bytes * ncp);
        const T *src = in + (int64_t)wk.patch * pw;
#pragma unroll
        for (int cp = 0; cp < ncp; ++cp) bulk_copy_g2s(Sx + cp * WSZ, src + cp * plane, bytes, bar);
    }
    int nb[8];
#pragma unroll
    for (int d = 0; d < 8; ++d) nb[d] = wk.nbr[d];
    bool waited = false, ok = true;
    for (int t = threadIdx.x; t < WX * WX; t += NT) {
        const int lj = t / WX - kGhost, li = t - (lj + kGhost) * WX - kGhost;
        const int sx = li < 0 ? -1 : (li >= n ? 1 : 0);
        const int sy = lj < 0 ? -1 : (lj >= n ? 1 : 0);
        if (!(sx | sy)) continue;
        const int d = dir_index(sx, sy);
        int q = nb[0];
#pragma unroll
        for (int e = 1; e < 8; ++e) q = (d == e) ? nb[e] : q;
        if (q < 0) continue;
        const T *g = in + (int64_t)q * pw + ((lj - sy * n + kGhost) * WX + (li - sx * n + kGhost));
        T v[ncp];
#pragma unroll
        for (int cp = 0; cp < ncp; ++cp) v[cp] = __ldg(g + cp * plane);
        if (!waited) {  // the bulk copy must land before its entries are overwritten
            ok = mbar_wait(bar, 0);
            waited = true;
        }
#pragma unroll
        for (int cp = 0; cp < ncp; ++cp) Sx[cp * WSZ + t] = v[cp];
    }
    if (!waited) ok = mbar_wait(bar, 0);
    if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) {
            atomicAdd(&g_wait_timeouts, 1u);
            mbar_wait(bar, 0);  // bounded: give the copies in flight a second chance to land
        }
        return false;
    }
    return true;
}

// For a bulk-staged tile: write the ghost columns (-2, -1, n, n+1, n+2) of
// the lattice rows y0 .. y1-1 the tile writes, in every plane, with the
// staged t^n values.  The tile's rows then go out whole, so consecutive rows
// fill their shared 32-byte sectors and no partial sector needs a
// read-modify-write in DRAM.  No other entry of a patch without a
// non-same-level neighbour is read, so these values are never used.
template <typename T, int NT, int WX, int WSZ, int NC>
__device__ __forceinline__ void write_ghost_columns(const StepArgs<T> &A, const af_work &wk, const T *Sin) {
    constexpr int n = WX - 2 * kGhost - 1;
    constexpr int ncp = NC * kPlanes;
    constexpr int64_t plane = plane_stride(n), pw = ncp * plane;
    static_assert(NT % 8 == 0, "threads in groups of eight: five ghost columns each");
    T *const out = dst_buf(A, wk.level) + (int64_t)wk.patch * pw;
    const int y0 = wk.y0, rows = wk.y1 - y0;
    const int k = threadIdx.x & 7;  // ghost column -2, -1, n, n+1, n+2 (k < 5)
    if (k >= 5) return;
    const int li = k < 2 ? k - kGhost : n + (k - 2);
    for (int row = threadIdx.x >> 3; row < rows; row += NT / 8) {
        T *o = out + (int64_t)(y0 + row + kGhost) * WX + (li + kGhost);
        const T *sp = Sin + (row + 1) * WX + (li + 1);
#pragma unroll
        for (int cp = 0; cp < ncp; ++cp) __stcs(o + cp * plane, sp[cp * WSZ]);
    }
}

// One tile per CTA.  SPLIT: gridDim.y CTAs share a tile, each a band of its
// rows, as if the tile had been built that way (few_tiles).
template <typename T, int EQ, int NT, int TMX, int TMY, int NN = 0, bool SPLIT = false>
__global__ void __launch_bounds__(NT, (min_ctas<T, EQ, NT>())) step_kernel(const __grid_constant__ StepArgs<T> A,
                                                  const __grid_constant__ typename WeightsOf<T, EQ>::type W) {
    using Gm = Geo<TMX, TMY, NN>;
    constexpr int ncomp = (EQ == AF_ACOUSTICS) ? 3 : 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *const Sbase = reinterpret_cast<T *>(smem_raw);
    T *Sin = Sbase + win_off<T, Gm::WX>();
    T *ST = Sbase + ncomp * kPlanes * Gm::WSZ;
    const unsigned block = chain_begin();
    prefetch_work(A.work, block + kWorkPrefetch, gridDim.x);
    af_work wk = load_work(A.work + block);
    if (wk.x1 - wk.x0 > TMX || wk.y1 - wk.y0 > TMY) return;  // built for another tiling
    if constexpr (SPLIT) {
        // (a tile whose copies are made to fail stays whole: one wait runs out)
        const bool whole = wk.flags & AF_WORK_SKIP_BULK_COPY;
        const int h = wk.y1 - wk.y0, y0 = wk.y0, part = whole ? 1 : (int)gridDim.y;
        if ((int)blockIdx.y >= part) return;
        wk.y0 = (int16_t)(y0 + h * (int)blockIdx.y / part);
        wk.y1 = (int16_t)(y0 + h * ((int)blockIdx.y + 1) / part);
        if (wk.y0 == wk.y1) return;
    }
    prefetch_freg<T, NT>(A, wk.patch, ncomp, NN > 0 ? NN : A.n);
    __shared__ __align__(8) uint64_t bar;
    bool staged = false;
    if (bulk_tile<T, Gm::WX>(A, wk)) {
        if (!stage_bulk<T, NT, Gm::WX, Gm::WSZ, ncomp>(A, wk, Sin, &bar)) return;  // counted in g_wait_timeouts
        staged = true;
    }
    if constexpr (NN > 0 && TMX == NN + 2 && TMY == NN + 2) {
        if (!staged && ext_bulk_tile<T, Gm::WX, Gm::WY>(A, wk)) {
            Sin = Sbase + 16 / (int)sizeof(T);  // the window origin is lattice offset 0: 16-byte aligned
            if (!stage_bulk_ext<T, NT, Gm::WX, Gm::WSZ, ncomp>(A, wk, Sin, &bar)) return;
            staged = true;
        }
    }
    if (!staged) {
        stage_issue<T, NT, Gm::WX, Gm::WSZ, ncomp, NN>(A, wk, Sin);
        cp_async_commit();
        cp_async_wait_all();
        __syncthreads();
    }
    if (wk.flags & 1) {
        stage_copy_out<T, NT, Gm::WX, Gm::WSZ, ncomp, NN>(A, wk, Sin);
        __syncthreads();  // copies land before the computed values overwrite them
    }
    tile_compute<T, EQ, NT, Gm::WX, Gm::WSZ, Gm::TX, Gm::TSZ, TMX, NN>(A, W, Sin, ST, wk.patch, wk.level, wk.x0,
                                                                      wk.x1, wk.y0, wk.y1);
    if (bulk_tile<T, Gm::WX>(A, wk)) write_ghost_columns<T, NT, Gm::WX, Gm::WSZ, ncomp>(A, wk, Sin);
}

}  // namespace dev

template <typename Kern>
inline cudaError_t ensure_smem(Kern k, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Launch of a step kernel, chained to the one before it (launch_chained) unless
// that unbalances the SMs (chain_even).  FP32 steps, which take 4 to 15 us where
// it does, are shorter chained all the same where a stream's launch gap counts
// (0.65 to 1.12 of the unchained time, mostly below 1); two large tiles an SM
// gain nothing from it in a graph (256 tiles of 32 x 32 cells 13.6 us, 14.5
// chained).  FP64 advection of an adaptive run: chain_even_mixed (coarse step of
// 1144 leaves of 8 x 8 cells 103 us, 126 all chained).
template <auto Kern, int NT, typename T, typename Wt>
af_status launch_tiles(const StepArgs<T> &A, const Wt &W, int nwork, int split, size_t smem, cudaStream_t stream) {
    constexpr bool f64 = sizeof(T) == 8, acoustics = !std::is_same<Wt, AdvectionPairWeights<T>>::value;
    if (ensure_smem(Kern, smem) != cudaSuccess) return AF_ERR_CUDA;
    bool chain = !(f64 && acoustics);
    const int64_t grid = (int64_t)nwork * split;
    if (chain && grid > kSMs) {
        const int r = resident_ctas<Kern>(NT, smem);
        const bool even = chain_even(grid, r);
        if (f64)
            chain = A.freg == nullptr ? even : chain_even_mixed(grid, r);
        else if (!even || r <= 2)
            chain = !recording(stream);
    }
    return launch_chained(chain, Kern, dim3(nwork, split), NT, smem, stream, A, W) == cudaSuccess ? AF_OK : AF_ERR_CUDA;
}

template <typename T, int EQ, int NT, int TMX, int TMY, int PIPE, int NN>
af_status launch_tiling(const StepArgs<T> &A, const typename WeightsOf<T, EQ>::type &W, int nwork,
                        cudaStream_t stream) {
    using Gm = dev::Geo<TMX, TMY, NN>;
    constexpr int ncomp = (EQ == AF_ACOUSTICS) ? 3 : 1;
    const size_t win = sizeof(T) * (size_t)ncomp * kPlanes * Gm::WSZ;
    const size_t tarr = sizeof(T) * (size_t)ncomp * 3 * Gm::TSZ;
    if constexpr (PIPE) {
        // There is no persistent (two-window) kernel: in two experimental
        // builds a launch of it on 48 x 48 patches ended in an unspecified
        // launch failure whose cause was not found, and it was the slower one.
        (void)win;
        (void)tarr;
        return AF_ERR_UNIMPLEMENTED;
    } else {
        // (8 TSZ words are used of the 9 where the T arrays are packed)
        const size_t smem = win + tarr;
        if (smem > 227 * 1024) return AF_ERR_UNIMPLEMENTED;
        if constexpr (NN == 0) {
            const int split = few_tiles(sizeof(T) == 8, EQ == AF_ACOUSTICS, {TMX, TMY, NT, 0}, nwork, A.n, A.freg != nullptr);
            if (split > 1) return launch_tiles<dev::step_kernel<T, EQ, NT, TMX, TMY, 0, true>, NT>(A, W, nwork, split, smem, stream);
        }
        return launch_tiles<dev::step_kernel<T, EQ, NT, TMX, TMY, NN>, NT>(A, W, nwork, 1, smem, stream);
    }
}

#define AF_TILING_CASE(K)                                                                                 \
    case K:                                                                                               \
        return launch_tiling<T, EQ, tiling(K).threads, tiling(K).tmx, tiling(K).tmy, tiling(K).persistent, NN>( \
            A, W, nwork, stream);

// All tilings for patches of NN x NN cells (NN = 0: any size, read at run time).
template <typename T, int EQ, int NN>
af_status launch_step_nn(int k, const StepArgs<T> &A, const typename WeightsOf<T, EQ>::type &W, int nwork,
                         cudaStream_t stream) {
    static_assert(kNumTilings == 10, "one case per compiled tiling");
    switch (k) {
        AF_TILING_CASE(0)
        AF_TILING_CASE(1)
        AF_TILING_CASE(2)
        AF_TILING_CASE(3)
        AF_TILING_CASE(4)
        AF_TILING_CASE(5)
        AF_TILING_CASE(6)
        AF_TILING_CASE(7)
        AF_TILING_CASE(8)
        AF_TILING_CASE(9)
    }
    return AF_ERR_ARG;
}

// FP32 kernels are also compiled for 16 x 16-cell patches (the adaptive
// workloads) and 32 x 32-cell patches, with lattice widths and plane offsets
// as constants: 13 % faster on the adaptive advection step, 3 % on the
// 16.8M-cell acoustics step.  The instantiations live in translation units
// of their own (af_step_f32_n16.cu, af_step_f32_n32.cu).
extern template af_status launch_step_nn<float, AF_ACOUSTICS, 16>(int, const StepArgs<float> &,
                                                                  const WeightsOf<float, AF_ACOUSTICS>::type &, int,
                                                                  cudaStream_t);
extern template af_status launch_step_nn<float, AF_ADVECTION, 16>(int, const StepArgs<float> &,
                                                                  const WeightsOf<float, AF_ADVECTION>::type &, int,
                                                                  cudaStream_t);
extern template af_status launch_step_nn<float, AF_ACOUSTICS, 32>(int, const StepArgs<float> &,
                                                                  const WeightsOf<float, AF_ACOUSTICS>::type &, int,
                                                                  cudaStream_t);
extern template af_status launch_step_nn<float, AF_ADVECTION, 32>(int, const StepArgs<float> &,
                                                                  const WeightsOf<float, AF_ADVECTION>::type &, int,
                                                                  cudaStream_t);

template <typename T, int EQ>
af_status launch_step(int k, const StepArgs<T> &A, const typename WeightsOf<T, EQ>::type &W, int nwork,
                      cudaStream_t stream) {
    // (few tiles are split further, by the kernels for any size)
    if constexpr (sizeof(T) == 4) if (few_tiles(false, EQ == AF_ACOUSTICS, tiling(k), nwork, A.n, A.freg != nullptr) == 1) {
        if (A.n == 16) return launch_step_nn<T, EQ, 16>(k, A, W, nwork, stream);
        if (A.n == 32) return launch_step_nn<T, EQ, 32>(k, A, W, nwork, stream);
    }
    return launch_step_nn<T, EQ, 0>(k, A, W, nwork, stream);
}

// Reads (and, if reset, clears) this translation unit's g_wait_timeouts;
// each translation unit that instantiates step kernels exports it under its
// own name (af_step_f32.cu, af_step_f64.cu, af_step_f32_n16.cu,
// af_step_f32_n32.cu, af_step_var.cu).
static inline af_status wait_timeouts_here(unsigned int *count, bool reset) {
    unsigned int v = 0;
    if (cudaMemcpyFromSymbol(&v, dev::g_wait_timeouts, sizeof(v)) != cudaSuccess) return AF_ERR_CUDA;
    *count = v;
    if (reset && v != 0) {
        const unsigned int zero = 0;
        if (cudaMemcpyToSymbol(dev::g_wait_timeouts, &zero, sizeof(zero)) != cudaSuccess) return AF_ERR_CUDA;
    }
    return AF_OK;
}
af_status wait_timeouts_f32(unsigned int *count, bool reset);
af_status wait_timeouts_f64(unsigned int *count, bool reset);
af_status wait_timeouts_f32_n16(unsigned int *count, bool reset);
af_status wait_timeouts_f32_n32(unsigned int *count, bool reset);
af_status wait_timeouts_var(unsigned int *count, bool reset);
af_status wait_timeouts_cnn(unsigned int *count, bool reset);

// Instantiated once each, in af_step_f32.cu and af_step_f64.cu.
extern template af_status launch_step<float, AF_ACOUSTICS>(int, const StepArgs<float> &,
                                                           const WeightsOf<float, AF_ACOUSTICS>::type &, int,
                                                           cudaStream_t);
extern template af_status launch_step<float, AF_ADVECTION>(int, const StepArgs<float> &,
                                                           const WeightsOf<float, AF_ADVECTION>::type &, int,
                                                           cudaStream_t);
extern template af_status launch_step<double, AF_ACOUSTICS>(int, const StepArgs<double> &,
                                                            const WeightsOf<double, AF_ACOUSTICS>::type &, int,
                                                            cudaStream_t);
extern template af_status launch_step<double, AF_ADVECTION>(int, const StepArgs<double> &,
                                                            const WeightsOf<double, AF_ADVECTION>::type &, int,
                                                            cudaStream_t);

}  // namespace af

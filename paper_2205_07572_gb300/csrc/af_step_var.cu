// af_patch_step_var: one Active Flux step of variable-velocity advection
// (Sections 4.2 and 4.3 of arXiv 2205.07572) on GB300.
//
// The tile staging, the same-level halo and the whole-patch copy of patches
// that advance their ghost layer are those of the constant-velocity kernel
// (af_step_kernels.cuh).  The velocity depends on position (and, for the
// swirl, on time), so the evolved point values are no longer fixed stencils:
// every node traces its characteristic back to t^n -- an exact rotation for
// solid-body rotation, one classical Runge-Kutta step for the swirl -- and
// evaluates the reconstruction (Eq. poly) of the cell holding the foot.  The
// fluxes take the velocity at their quadrature points (solid body) or at the
// face centre for each time level (Eqs. swirlF, swirlG).
//
// These kernels are bound by arithmetic, so it is kept small:
//  - the foot is traced as a displacement from its node: the sines and cosines
//    at the node come from a table over the tile's lines (as do those at the
//    face centres), and a Runge-Kutta stage turns them by the small angle of
//    its displacement (angle addition, a short series: turn()).  Two sincospi
//    per velocity, 56 per cell, were most of the kernel.  A displacement also
//    keeps the digits that a foot's absolute position loses;
//  - both fields' time dependence separates from the face's values, so a node
//    keeps one time-Simpson sum for the fluxes, not its two new values;
//  - what depends on the level only comes from the host (FP64 arithmetic in
//    every thread's preamble cost an FP32 tile a third of its time).
// FP32 swirl, 4096^2 cells in 16 x 16 patches: 1740 -> 701 us (FMA pipe; the
// displacements, tables and series 1.7x, both feet packed and one node per
// thread and turn 1.2x, 128 threads a tile and half the multiplications 1.2x).
// FP64 swirl, 512^2: 1286 -> 498 us; FP32 solid body, 2048^2: 261 -> 135 us.
#include <cuda_runtime.h>

#include <cmath>

#include "af_step_kernels.cuh"

namespace af {
namespace dev {

// The values of one quantity for the two feet of a node, at t^n + dt/2 (x)
// and t^n + dt (y).  In FP32 every operation on them is one packed FP32x2
// instruction: both feet for the issue slots of one.
template <typename T>
struct Two {
    T x, y;
};
__device__ __forceinline__ float2 f2(Two<float> a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ Two<float> two(float2 a) { return {a.x, a.y}; }
__device__ __forceinline__ Two<float> mul(Two<float> a, Two<float> b) { return two(__fmul2_rn(f2(a), f2(b))); }
__device__ __forceinline__ Two<float> add(Two<float> a, Two<float> b) { return two(__fadd2_rn(f2(a), f2(b))); }
__device__ __forceinline__ Two<float> fma(Two<float> a, Two<float> b, Two<float> c) {
    return two(__ffma2_rn(f2(a), f2(b), f2(c)));
}
__device__ __forceinline__ Two<double> mul(Two<double> a, Two<double> b) { return {a.x * b.x, a.y * b.y}; }
__device__ __forceinline__ Two<double> add(Two<double> a, Two<double> b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Two<double> fma(Two<double> a, Two<double> b, Two<double> c) {
    return {::fma(a.x, b.x, c.x), ::fma(a.y, b.y, c.y)};
}
template <typename T>
__device__ __forceinline__ Two<T> both(T a) {
    return {a, a};
}

// Constants of one level, rounded once on the host.
template <typename T>
struct VarLevel {
    T rdx, rdy;    // reciprocal mesh widths (swirl: over 12 pi, what swirl_feet leaves out)
    T dtdx, dtdy;  // dt / dx, dt / dy
    T hx, hy;      // mesh widths
    T e[3];        // weights of q^n, q^{n+1/2}, q^{n+1} in a face's time-Simpson sum
    T kx, ky;      // swirl: the face velocities' constants, over 36
    // swirl: factor of each Runge-Kutta stage's displacement (tau/2, tau/2,
    // tau, tau backwards, times the velocity's constants, cos(pi t) and the
    // 2 pi of an angle), x and y; solid body: sin(pi tau), cos(pi tau) - 1
    Two<T> a[4], b[4];
};

template <typename T>
struct VarArgs {
    StepArgs<T> s;      // work list, buffers, flux registers, layout
    double x_lo, y_lo;  // node line 0 of patch (0, 0)
    double dx0, dy0;    // level-0 mesh widths
    VarLevel<T> lev[AF_MAX_LEVEL + 1];
};

__device__ __forceinline__ void scpi(float x, float &s, float &c) { sincospif(x, &s, &c); }
__device__ __forceinline__ void scpi(double x, double &s, double &c) { sincospi(x, &s, &c); }

// Of an angle z = 2 pi x: sin z, cos z and cos z - 1 (= -2 sin^2 pi x, without
// cancellation); solid body: x itself in .s.
template <typename T>
struct SC {
    T s, c, n;
};

// How a displacement's angle z = 2 pi d is turned into sin z and cos z: by their
// Taylor series up to |z| <= 0.02 (kTiny), 0.25 (kSmall) -- the terms left out are
// below 5e-8 of sin z and 1e-8 in cos z (FP32; 1e-17, 1e-18 in
// FP64), 1e-9 and 7e-9 for kTiny -- and by sincospi beyond.  The host picks by
// the time step, which bounds d: a 4096-cell run turns by at most 7e-4, a
// 64-cell run by 0.04.
enum Turn { kAny = 0, kSmall = 1, kTiny = 2 };
constexpr double kTurnMax[3] = {1e300, 0.25, 0.02};

template <typename T, int MODE>
__device__ __forceinline__ void turn(Two<T> u, Two<T> &s, Two<T> &c) {
    if constexpr (MODE == kAny) {
        scpi(u.x * T(1.0 / M_PI), s.x, c.x);
        scpi(u.y * T(1.0 / M_PI), s.y, c.y);
    } else {
        const Two<T> w = mul(u, u);
        auto step = [&](Two<T> p, double k) { return fma(w, p, both(T(k))); };
        if constexpr (sizeof(T) == 4 && MODE == kTiny) {
            s = mul(u, step(both(T(-1.0 / 6.0)), 1.0));
            c = step(both(T(-0.5)), 1.0);
        } else if constexpr (sizeof(T) == 4) {
            s = mul(u, step(step(both(T(1.0 / 120.0)), -1.0 / 6.0), 1.0));
            c = step(step(step(both(T(-1.0 / 720.0)), 1.0 / 24.0), -0.5), 1.0);
        } else if constexpr (MODE == kTiny) {
            s = mul(u, step(step(step(both(T(-1.0 / 5040.0)), 1.0 / 120.0), -1.0 / 6.0), 1.0));
            c = step(step(step(both(T(-1.0 / 720.0)), 1.0 / 24.0), -0.5), 1.0);
        } else {
            s = step(step(both(T(-1.0 / 39916800.0)), 1.0 / 362880.0), -1.0 / 5040.0);
            s = mul(u, step(step(step(s, 1.0 / 120.0), -1.0 / 6.0), 1.0));
            c = step(step(both(T(1.0 / 479001600.0)), -1.0 / 3628800.0), 1.0 / 40320.0);
            c = step(step(step(step(c, -1.0 / 720.0), 1.0 / 24.0), -0.5), 1.0);
        }
    }
}

// Swirl: displacements (as angles 2 pi d) of the feet at t^n of the
// characteristics through the node with angles (x, y) at t^n + dt/2 and
// t^n + dt, one classical Runge-Kutta step backwards each.  The velocity is
// (the centred differences of Eq. swirlODE)
//   a = -sin^2(pi x) sin(2 pi y) cos(pi t) sin(pi dy) / (pi dy)
//     = (cos 2 pi x - 1) sin 2 pi y times constants of the stage, in L.a[q],
// and its mirror; the addition theorems turn the node's angles by a stage's.
template <typename T, int MODE>
__device__ __forceinline__ void swirl_feet(const VarLevel<T> &L, const SC<T> &x, const SC<T> &y, Two<T> &dx,
                                           Two<T> &dy) {
    Two<T> da = mul(both(x.n * y.s), L.a[0]), db = mul(both(y.n * x.s), L.b[0]);
    // h (k1 + 2 k2 + 2 k3 + k4) / 6 from h/2 k1, h/2 k2, h k3, h k4: summed as
    // 2 h/2 k1 + 4 h/2 k2 + 2 h k3 + h k4, the 1/6 left to the caller
    dx = add(da, da), dy = add(db, db);
    constexpr double w[4] = {2, 4, 2, 1};
#pragma unroll
    for (int q = 1; q < 4; ++q) {
        Two<T> s, c;
        turn<T, MODE>(da, s, c);
        const Two<T> xs = fma(both(x.s), c, mul(both(x.c), s));                  // sin
        const Two<T> xn = fma(both(x.c), c, fma(both(-x.s), s, both(T(-1))));    // cos - 1
        turn<T, MODE>(db, s, c);
        const Two<T> ys = fma(both(y.s), c, mul(both(y.c), s));
        const Two<T> yn = fma(both(y.c), c, fma(both(-y.s), s, both(T(-1))));
        da = mul(mul(xn, ys), L.a[q]);
        db = mul(mul(yn, xs), L.b[q]);
        if (q < 3)
            dx = fma(both(T(w[q])), da, dx), dy = fma(both(T(w[q])), db, dy);
        else
            dx = add(dx, da), dy = add(dy, db);
    }
}

// Cell of a point f in cells from a node line (0): -1, 0 or, for a point from
// a midpoint (hi = 1), 1.  A foot is at most one mesh width from its node, so
// these are all, and all of them are in the tile's window.
template <typename T>
__device__ __forceinline__ int cell_of(T f, int hi) {
    return f < T(0) ? -1 : (f > T(1) ? hi : 0);
}

// Reconstruction of the staged cells holding the two points (fx, fy), in cells
// from node lines (i, j) at window entry o.
template <typename T, int WX, int WSZ>
__device__ __forceinline__ Two<T> eval_near(const T *Sin, int o, int hx, int hy, Two<T> fx, Two<T> fy) {
    const int ix = cell_of(fx.x, hx), iy = cell_of(fy.x, hy), jx = cell_of(fx.y, hx), jy = cell_of(fy.y, hy);
    const T *const P = Sin + o + iy * WX + ix, *const Q = Sin + o + jy * WX + jx;
    auto at = [&](int plane, int k) -> Two<T> { return {P[plane * WSZ + k], Q[plane * WSZ + k]}; };
    const Two<T> c00 = at(kCorner, 0), c10 = at(kCorner, 1), c01 = at(kCorner, WX), c11 = at(kCorner, WX + 1);
    const Two<T> xl = at(kXmid, 0), xr = at(kXmid, 1), yb = at(kYmid, 0), yt = at(kYmid, WX), av = at(kAvg, 0);
    const Two<T> cen = fma(both(T(-0.25)), add(add(xl, xr), add(yb, yt)),
                           fma(both(T(-0.0625)), add(add(c00, c10), add(c01, c11)), mul(both(T(2.25)), av)));
    // the three Lagrange polynomials at z = 2 h, h = f - cell - 1/2
    auto basis = [&](Two<T> h, Two<T> l[3]) {
        const Two<T> s = mul(h, add(h, h));  // z^2 / 2
        l[0] = fma(both(T(-1)), h, s);
        l[1] = fma(both(T(-2)), s, both(T(1)));
        l[2] = add(s, h);
    };
    Two<T> lx[3], ly[3];
    basis(add(fx, Two<T>{T(-0.5) - T(ix), T(-0.5) - T(jx)}), lx);
    basis(add(fy, Two<T>{T(-0.5) - T(iy), T(-0.5) - T(jy)}), ly);
    const Two<T> r0 = fma(lx[2], c10, fma(lx[1], yb, mul(lx[0], c00)));
    const Two<T> r1 = fma(lx[2], xr, fma(lx[1], cen, mul(lx[0], xl)));
    const Two<T> r2 = fma(lx[2], c11, fma(lx[1], yt, mul(lx[0], c01)));
    return fma(ly[2], r2, fma(ly[1], r1, mul(ly[0], r0)));
}

// NN: the patch size of a tiling two cells wider, if known when compiled: its
// tiles then have the pitch of the patch lattice and are staged in bulk.
template <typename T, int FIELD, int MODE, int NT, int TMX, int TMY, int NN>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? 768 / NT : 1) step_var_kernel(const __grid_constant__ VarArgs<T> V) {
    using Gm = Geo<TMX, TMY, NN>;
    constexpr int WX = Gm::WX, WSZ = Gm::WSZ, TX = Gm::TX, TSZ = Gm::TSZ;
    constexpr bool SWIRL = FIELD == AF_FIELD_SWIRL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *const Sbase = reinterpret_cast<T *>(smem_raw);
    T *Sin = Sbase + win_off<T, WX>();
    T *ST = Sbase + kPlanes * WSZ;  // [node type][TSZ]: the time-Simpson sums of the node values
    // the tile's node lines (0) and the midpoints after them (1), per axis:
    // the sine and cosine of 2 pi x (swirl), or x itself in .s (solid body)
    __shared__ SC<T> tx[2][TMX + 1], ty[2][TMY + 1];
    const StepArgs<T> &A = V.s;
    const af_work wk = load_work(A.work + chain_begin());
    if (wk.x1 - wk.x0 > TMX || wk.y1 - wk.y0 > TMY) return;
    const int n = NN > 0 ? NN : A.n, W_ = n + 2 * kGhost + 1, level = wk.level;
    const int plane = NN > 0 ? (int)plane_stride(NN) : (int)A.plane;
    const int x0 = wk.x0, x1 = wk.x1, y0 = wk.y0, y1 = wk.y1, tw = x1 - x0, th = y1 - y0;
    const VarLevel<T> &L = V.lev[level];
    for (int e = threadIdx.x; e < 2 * (tw + th + 2); e += NT) {
        const bool ax = e < 2 * (tw + 1);
        const int r = ax ? e : e - 2 * (tw + 1), len = ax ? tw + 1 : th + 1, m = r >= len ? 1 : 0, k = r - m * len;
        const double h = (ax ? V.dx0 : V.dy0) * __longlong_as_double((long long)(1023 - level) << 52);
        const T org = (T)((ax ? V.x_lo : V.y_lo) + (double)((long long)(ax ? wk.ix : wk.iy) * n) * h);
        const T x = org + ((T)((ax ? x0 : y0) + k) + (m ? T(0.5) : T(0))) * (ax ? L.hx : L.hy);
        SC<T> v{x, T(0), T(0)};
        if constexpr (SWIRL) {
            T sp, cp;
            scpi(x, sp, cp);
            v.s = T(2) * sp * cp;
            v.n = T(-2) * sp * sp;
            v.c = T(1) + v.n;
        }
        if (ax)
            tx[m][k] = v;
        else
            ty[m][k] = v;
    }
    // the staging below ends with a barrier, which the tables need too
    __shared__ __align__(8) uint64_t bar;
    const bool bulk = bulk_tile<T, WX>(A, wk);
    bool staged = bulk;
    if (bulk) {  // bulk (TMA) copies of the window rows, as in the constant-velocity step
        if (!stage_bulk<T, NT, WX, WSZ, 1>(A, wk, Sin, &bar)) return;  // counted in g_wait_timeouts
    }
    if constexpr (NN > 0 && TMX == NN + 2 && TMY == NN + 2) {
        if (!staged && ext_bulk_tile<T, WX, Gm::WY>(A, wk)) {
            Sin = Sbase + 16 / (int)sizeof(T);
            if (!stage_bulk_ext<T, NT, WX, WSZ, 1>(A, wk, Sin, &bar)) return;
            staged = true;
        }
    }
    if (!staged) {
        stage_issue<T, NT, WX, WSZ, 1, NN>(A, wk, Sin);
        cp_async_commit();
        cp_async_wait_all();
        __syncthreads();
    }
    if (wk.flags & 1) {
        stage_copy_out<T, NT, WX, WSZ, 1, NN>(A, wk, Sin);
        __syncthreads();
    }
    T *outp = dst_buf(A, level) + (int64_t)wk.patch * kPlanes * plane;
    const int sxhi = (x1 == n + 1) ? x1 : x1 - 1;
    const int syhi = (y1 == n + 1) ? y1 : y1 - 1;
    // ---- point values at t^{n+1/2}, t^{n+1}: corners (i, j), left-edge and
    // bottom-edge midpoints, one node per thread and turn and type after type:
    // a third of a node-cell's work each, so a tile's last, partial turn is
    // short (289 node-cells on 256 threads took two turns for 1.13)
    const int nc = (tw + 1) * (th + 1), nx = (tw + 1) * th, ny = tw * (th + 1);
    // r / w = r m >> 16 for r < 1089 and w <= 33 (m = 2^16 / w rounded up is
    // at most 1/w of 2^16 / r too large)
    const unsigned m0 = (65536u + tw) / (tw + 1), m1 = (65536u + tw - 1) / tw;
    for (int it = threadIdx.x; it < nc + nx + ny; it += NT) {
        const int ntype = it < nc ? 0 : (it < nc + nx ? 1 : 2);
        const int r = it - (ntype == 0 ? 0 : (ntype == 1 ? nc : nc + nx)), w = ntype == 2 ? tw : tw + 1;
        const int jj = (int)((unsigned)r * (ntype == 2 ? m1 : m0) >> 16), ii = r - jj * w;
        const int i = x0 + ii, j = y0 + jj;
        const bool st_x = i <= sxhi, st_y = j <= syhi;
        const int so = jj * TX + ii, sw = (jj + 1) * WX + (ii + 1);
        const SC<T> x = tx[ntype == 2][ii], y = ty[ntype == 1][jj];
        const T ox = ntype == 2 ? T(0.5) : T(0), oy = ntype == 1 ? T(0.5) : T(0);
        Two<T> dx, dy;  // the feet, less the node
        if constexpr (SWIRL) {
            swirl_feet<T, MODE>(L, x, y, dx, dy);
        } else {  // the rotation back by pi tau, less the identity
            dx = fma(both(y.s), L.a[0], mul(both(x.s), L.a[1]));
            dy = fma(both(-x.s), L.a[0], mul(both(y.s), L.a[1]));
        }
        const Two<T> v = eval_near<T, WX, WSZ>(Sin, sw, ntype == 2, ntype == 1, fma(dx, both(L.rdx), both(ox)),
                                               fma(dy, both(L.rdy), both(oy)));
        const int pl = ntype == 0 ? kCorner : (ntype == 1 ? kXmid : kYmid);
        ST[ntype * TSZ + so] = ::fma(L.e[0], Sin[pl * WSZ + sw], ::fma(L.e[1], v.x, L.e[2] * v.y));
        if ((st_x || ntype == 2) && (st_y || ntype == 1))
            outp[pl * plane + (j + kGhost) * W_ + (i + kGhost)] = v.y;
    }
    __syncthreads();

    // ---- fluxes and update of cells [x0, x1) x [y0, y1)
    const T *const Tc = ST, *const Tx = ST + TSZ, *const Ty = ST + 2 * TSZ;
    for (int it = threadIdx.x; it < tw * th; it += NT) {
        const int jj = it / tw, ii = it - jj * tw;
        const int i = x0 + ii, j = y0 + jj;
        const int so = jj * TX + ii, sw = (jj + 1) * WX + (ii + 1);
        // x-face on node line ii + di (di = 0 left, 1 right); y-face on jj + dj
        auto xflux = [&](int di) -> T {
            const T tl = Tc[so + di], tm = Tx[so + di], tu = Tc[so + di + TX];
            if constexpr (SWIRL)
                return tx[0][ii + di].n * ty[1][jj].s * L.ky * (::fma(T(4), tm, tl) + tu);
            else
                return T(-M_PI / 36.0) *
                       ::fma(ty[0][jj].s, tl, ::fma(T(4) * ty[1][jj].s, tm, ty[0][jj + 1].s * tu));
        };
        auto yflux = [&](int dj) -> T {
            const T tl = Tc[so + dj * TX], tm = Ty[so + dj * TX], tr = Tc[so + dj * TX + 1];
            if constexpr (SWIRL)
                return ty[0][jj + dj].n * tx[1][ii].s * L.kx * (::fma(T(4), tm, tl) + tr);
            else
                return T(M_PI / 36.0) * ::fma(tx[0][ii].s, tl, ::fma(T(4) * tx[1][ii].s, tm, tx[0][ii + 1].s * tr));
        };
        const T fl = xflux(0), fr = xflux(1), gb = yflux(0), gt = yflux(1);
        const T q = Sin[kAvg * WSZ + sw];
        outp[(j + kGhost) * W_ + (i + kGhost)] = ::fma(-L.dtdy, gt - gb, ::fma(-L.dtdx, fr - fl, q));
        if (A.freg != nullptr) {
            const double dtl = A.dt0 * __longlong_as_double((long long)(1023 - level) << 52);
            double *fr_p = A.freg + (int64_t)wk.patch * 4 * n;
            const bool iny = (j >= 0 && j < n), inx = (i >= 0 && i < n);
            if (iny && i == 0) fr_p[0 * n + j] += dtl * (double)fl;
            if (iny && i == n - 1) fr_p[1 * n + j] += dtl * (double)fr;
            if (inx && j == 0) fr_p[2 * n + i] += dtl * (double)gb;
            if (inx && j == n - 1) fr_p[3 * n + i] += dtl * (double)gt;
        }
    }
    if (bulk) write_ghost_columns<T, NT, WX, WSZ, 1>(A, wk, Sin);
}

template <typename T, int FIELD, int MODE, int NT, int TMX, int TMY, int NN>
af_status launch_var_kernel(const VarArgs<T> &V, int nwork, cudaStream_t stream) {
    using Gm = Geo<TMX, TMY, NN>;
    const size_t smem = sizeof(T) * ((size_t)kPlanes * Gm::WSZ + 3 * (size_t)Gm::TSZ);
    if (smem > 227 * 1024) return AF_ERR_UNIMPLEMENTED;
    constexpr auto kern = step_var_kernel<T, FIELD, MODE, NT, TMX, TMY, NN>;
    if (ensure_smem(kern, smem) != cudaSuccess) return AF_ERR_CUDA;
    // (in a stream, FP32 tiles of up to 18 x 18 cells gain from it in any case;
    // larger ones, and FP64, lose up to 1.2x and 1.5x where it is uneven)
    const bool chain = chain_even(nwork, resident_ctas<kern>(NT, smem)) || (sizeof(T) == 4 && TMX <= 18 && !recording(stream));
    return launch_chained(chain, kern, nwork, NT, smem, stream, V) == cudaSuccess ? AF_OK : AF_ERR_CUDA;
}

// A tiling two cells wider than a patch (8 x 8 and 16 x 16 patches with their
// ghost layer) takes the kernel compiled for that size.
template <typename T, int FIELD, int MODE, int NT, int TMX, int TMY>
af_status launch_var_tiling(const VarArgs<T> &V, int nwork, cudaStream_t stream) {
    if constexpr (MODE != kAny && (TMX == 10 || TMX == 18))
        if (V.s.n == TMX - 2) return launch_var_kernel<T, FIELD, MODE, NT, TMX, TMY, TMX - 2>(V, nwork, stream);
    return launch_var_kernel<T, FIELD, MODE, NT, TMX, TMY, 0>(V, nwork, stream);
}

// The persistent tiling (a CTA looping over tiles) runs here as one tile per
// CTA, and every tiling on at most 128 threads: an FP32 SM then holds six tiles
// instead of three, whose barriers and staging overlap better (4096^2 cells,
// 18 x 18 tiles on 256, 192, 128 threads: 997, 951, 855 us at one stage of this
// kernel); FP64, bound by its pipe, does not care.
#define AF_VAR_CASE(K)                                                                                       \
    case K:                                                                                                  \
        return launch_var_tiling<T, FIELD, MODE, (tiling(K).threads < 128 ? tiling(K).threads : 128),        \
                                 tiling(K).tmx, tiling(K).tmy>(V, nwork, stream);

template <typename T, int FIELD, int MODE>
af_status launch_var(int k, const VarArgs<T> &V, int nwork, cudaStream_t stream) {
    static_assert(kNumTilings == 10, "one case per compiled tiling");
    switch (k) {
        AF_VAR_CASE(0)
        AF_VAR_CASE(1)
        AF_VAR_CASE(2)
        AF_VAR_CASE(3)
        AF_VAR_CASE(4)
        AF_VAR_CASE(5)
        AF_VAR_CASE(6)
        AF_VAR_CASE(7)
        AF_VAR_CASE(8)
        AF_VAR_CASE(9)
    }
    return AF_ERR_ARG;
}

}  // namespace dev
}  // namespace af

extern "C" af_status af_patch_step_var(const af_config *cfg, int32_t tiling_index, int32_t nwork,
                                       const af_work *d_work, const af_state_pair *state, const af_velocity *vel,
                                       double dt0, double dx0, double dy0, double *d_flux_reg, void *stream) {
    using namespace af;
    if (cfg == nullptr || state == nullptr || vel == nullptr || nwork < 0) return AF_ERR_ARG;
    if (tiling_index < 0 || tiling_index >= kNumTilings) return AF_ERR_ARG;
    if (cfg->eq != AF_ADVECTION || cfg->ncomp != 1 || cfg->n < 2 || cfg->n > 64) return AF_ERR_ARG;
    if (cfg->prec != AF_F64 && cfg->prec != AF_F32) return AF_ERR_ARG;
    if (vel->field != AF_FIELD_SOLID_BODY && vel->field != AF_FIELD_SWIRL) return AF_ERR_ARG;
    if (!(dt0 > 0.0) || !(dx0 > 0.0) || !(dy0 > 0.0)) return AF_ERR_ARG;
    if (!(vel->x_hi > vel->x_lo) || !(vel->y_hi > vel->y_lo)) return AF_ERR_ARG;
    if (nwork == 0) return AF_OK;
    void *b0 = state->buf[0], *b1 = state->buf[1];
    if (d_work == nullptr || b0 == nullptr || b1 == nullptr || b0 == b1) return AF_ERR_ARG;
    if ((reinterpret_cast<uintptr_t>(b0) | reinterpret_cast<uintptr_t>(b1)) & 31u) return AF_ERR_LAYOUT;
    if (reinterpret_cast<uintptr_t>(d_work) & 15u) return AF_ERR_LAYOUT;
    if (reinterpret_cast<uintptr_t>(d_flux_reg) & 7u) return AF_ERR_LAYOUT;
    // speed bound over the domain and its two ghost layers at level 0
    double vmax;
    if (vel->field == AF_FIELD_SOLID_BODY) {
        const double ex = 3.0 * dx0, ey = 3.0 * dy0;
        const double mx = std::fmax(std::fabs(vel->x_lo - ex), std::fabs(vel->x_hi + ex));
        const double my = std::fmax(std::fabs(vel->y_lo - ey), std::fabs(vel->y_hi + ey));
        vmax = M_PI * std::fmax(mx, my);
    } else {
        vmax = 1.0;  // |sin^2 sin| <= 1 and sin(pi h) / (pi h) <= 1
    }
    if (!(vmax * dt0 <= std::fmin(dx0, dy0))) return AF_ERR_CFL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int k = tiling_index;
    auto fill = [&](auto &V, auto one) {
        using T = decltype(one);
        V.s.work = d_work;
        V.s.freg = d_flux_reg;
        V.s.plane = plane_stride(cfg->n);
        V.s.n = cfg->n;
        V.s.ncomp = 1;
        V.s.dt0 = dt0;
        V.s.swap = state->parity;
        V.s.in = static_cast<const T *>(b0);
        V.s.out = static_cast<T *>(b1);
        V.x_lo = vel->x_lo;
        V.y_lo = vel->y_lo;
        V.dx0 = dx0;
        V.dy0 = dy0;
        // at t + dt_l, + dt_l/2, + dt_l/4 level l needs entries l, l + 1, l + 2 of
        // the cosines (swirl; the rotation: the sines) at t + dt0 / 2^k: a third
        // of the calls, which an in-cache step would wait for
        const bool swirl = vel->field == AF_FIELD_SWIRL;
        double at[AF_MAX_LEVEL + 3];
        for (int k = 0; k < AF_MAX_LEVEL + 3; ++k)
            at[k] = swirl ? std::cos(M_PI * (vel->t + std::ldexp(dt0, -k))) : std::sin(M_PI * std::ldexp(dt0, -k));
        const double now = swirl ? std::cos(M_PI * vel->t) : 0.0;
        for (int l = 0; l <= AF_MAX_LEVEL; ++l) {
            const double dtl = std::ldexp(dt0, -l), hx = std::ldexp(dx0, -l), hy = std::ldexp(dy0, -l);
            dev::VarLevel<T> &v = V.lev[l];
            v.hx = (T)hx;
            v.hy = (T)hy;
            v.dtdx = (T)dtl / v.hx;
            v.dtdy = (T)dtl / v.hy;
            if (swirl) {
                const double kx = std::sin(M_PI * hx) / (M_PI * hx);
                const double ky = dy0 == dx0 ? kx : std::sin(M_PI * hy) / (M_PI * hy);
                v.e[0] = (T)now;
                v.e[1] = (T)(4.0 * at[l + 1]);
                v.e[2] = (T)at[l];
                v.kx = (T)(-0.5 * kx / 36.0);
                v.ky = (T)(0.5 * ky / 36.0);
                v.rdx = (T)(1.0 / (12.0 * M_PI * hx));
                v.rdy = (T)(1.0 / (12.0 * M_PI * hy));
                // stage times t^n + tau, + tau/2, + tau/2, + 0
                const double half[4] = {at[l + 1], at[l + 2], at[l + 2], now}, full[4] = {at[l], at[l + 1], at[l + 1], now};
                for (int q = 0; q < 4; ++q) {
                    const double tau = (q < 2 ? -0.5 : -1.0) * dtl;
                    v.a[q] = {(T)(M_PI * ky * 0.5 * tau * half[q]), (T)(M_PI * ky * tau * full[q])};
                    v.b[q] = {(T)(-M_PI * kx * 0.5 * tau * half[q]), (T)(-M_PI * kx * tau * full[q])};
                }
            } else {
                v.rdx = (T)(1.0 / hx);
                v.rdy = (T)(1.0 / hy);
                v.e[0] = v.e[2] = T(1);
                v.e[1] = T(4);
                v.a[0] = {(T)at[l + 1], (T)at[l]};
                // cos - 1 without cancellation
                v.a[1] = {(T)(-2.0 * at[l + 2] * at[l + 2]), (T)(-2.0 * at[l + 1] * at[l + 1])};
            }
        }
    };
    // a stage is displaced by at most dt0 times the speed (1)
    const double z = 2.0 * M_PI * dt0;
    auto launch = [&](auto &V, auto one) {
        using T = decltype(one);
        fill(V, one);
        if (vel->field == AF_FIELD_SOLID_BODY) return dev::launch_var<T, AF_FIELD_SOLID_BODY, dev::kTiny>(k, V, nwork, s);
        if (z <= dev::kTurnMax[dev::kTiny]) return dev::launch_var<T, AF_FIELD_SWIRL, dev::kTiny>(k, V, nwork, s);
        return z <= dev::kTurnMax[dev::kSmall] ? dev::launch_var<T, AF_FIELD_SWIRL, dev::kSmall>(k, V, nwork, s)
                                               : dev::launch_var<T, AF_FIELD_SWIRL, dev::kAny>(k, V, nwork, s);
    };
    if (cfg->prec == AF_F64) {
        dev::VarArgs<double> V{};
        return launch(V, 0.0);
    }
    dev::VarArgs<float> V{};
    return launch(V, 0.0f);
}

namespace af {
af_status wait_timeouts_var(unsigned int *count, bool reset) { return wait_timeouts_here(count, reset); }
}  // namespace af

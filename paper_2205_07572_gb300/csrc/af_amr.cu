// Adaptive-mesh kernels of libaf.so (Section 3 of arXiv 2205.07572):
// ghost exchange, regrid transfer, conservative fix, tagging, mass totals.
//
// Positions are exact integers: one unit is half the cell width of level
// lmax, so a level-l cell is 2^(lmax-l+1) units wide and every node, cell
// centre and Simpson point is a lattice point of that unit.  The forest is
// located through per-level region maps (af_forest.d_map), which stay in L2.
// They are 32-bit: the domain is (B << lmax) 2n units wide, and a map of
// (B << lmax)^2 entries that fits the GPU keeps that below 2^25.  (With 64-bit
// positions the divisions by a region's width were most of the kernels that
// look owners up: on 2100 leaves a ghost plan took 209 us, now 69.)
#include <cuda_runtime.h>

#include <cstring>

#include "af_internal.h"
#include "af_launch.cuh"

namespace af {
namespace {

struct DevForest {
    int nleaf, B, lmax, n;
    const int32_t *level, *ix, *iy, *map;
    int D;           // domain width in units
    uint32_t rcp;    // 2^32 / (2n) rounded up: region() divides by 2n with it
};

DevForest make_dev(const af_forest &f, int n) {
    DevForest d;
    d.nleaf = f.nleaf;
    d.B = f.B;
    d.lmax = f.lmax;
    d.n = n;
    d.level = f.d_level;
    d.ix = f.d_ix;
    d.iy = f.d_iy;
    d.map = f.d_map;
    d.D = (int)((long long)f.B * n * (2LL << f.lmax));
    d.rcp = (uint32_t)(((1ull << 32) + 2 * n - 1) / (2 * n));
    return d;
}

__host__ __device__ inline long long map_offset(int B, int l) {
    // sum_{m<l} (B << m)^2 = B^2 (4^l - 1) / 3
    return (long long)B * B * (((1LL << (2 * l)) - 1) / 3);
}

// Width of a level-l cell in units.
__device__ __forceinline__ int hwid(const DevForest &F, int l) { return 2 << (F.lmax - l); }

__device__ __forceinline__ int wrapd(const DevForest &F, int x) {
    // positions are at most one domain width outside [0, D)
    if (x < 0) x += F.D;
    if (x >= F.D) x -= F.D;
    if ((unsigned)x >= (unsigned)F.D) {
        x %= F.D;
        return x < 0 ? x + F.D : x;
    }
    return x;
}

// Finest-level region (column or row) of position x >= 0: x / (2n).  The
// product with the rounded-up reciprocal is too large by at most one.
__device__ __forceinline__ int region(const DevForest &F, int x) {
    const int q = (int)__umulhi((uint32_t)x, F.rcp);
    return q * 2 * F.n > x ? q - 1 : q;
}

// Leaf whose half-open extent contains (x, y).  A region of the finest level
// lmax is a leaf (entry q >= 0) or lies inside the coarser leaf -2 - entry
// (af_forest_build_map), so one load finds it; a map without that second
// kind of entry is searched level by level.
__device__ __forceinline__ int lookup(const DevForest &F, int x, int y) {
    const int rx = region(F, wrapd(F, x)), ry = region(F, wrapd(F, y));
#pragma unroll 1
    for (int l = F.lmax; l >= 0; --l) {
        const int sh = F.lmax - l;
        const int q = __ldg(F.map + map_offset(F.B, l) + (int64_t)(ry >> sh) * (F.B << l) + (rx >> sh));
        if (q >= 0) return q < F.nleaf ? q : -1;
        if (q <= -2 && l == F.lmax) return -2 - q < F.nleaf ? -2 - q : -1;
    }
    return -1;
}

// Owner of a point value: the finest leaf touching the point, ties in the
// order above-right, above-left, below-right, below-left.
__device__ __forceinline__ int entry_owner(const DevForest &F, int plane, int x, int y) {
    const int touching = plane == kAvg ? 1 : 4;  // an average's owner is the leaf around it
    int best = -1, bl = -1;
    // a loop, not four copies of lookup(): the callers' code has to stay small
    // (unrolled everywhere, a regrid's transfer spent 25 of 32 cycles per
    // instruction waiting for the instruction cache)
#pragma unroll 1
    for (int k = 0; k < touching; ++k) {
        const int q = lookup(F, x - (k & 1), y - (k >> 1));
        if (q >= 0) {
            const int lq = __ldg(F.level + q);
            if (lq > bl) {
                best = q;
                bl = lq;
            }
        }
    }
    return best;
}

__device__ __forceinline__ int leaf_x0(const DevForest &F, int q) {
    return __ldg(F.ix + q) * F.n * hwid(F, __ldg(F.level + q));
}
__device__ __forceinline__ int leaf_y0(const DevForest &F, int q) {
    return __ldg(F.iy + q) * F.n * hwid(F, __ldg(F.level + q));
}

// x - x0 unwrapped across the periodic box
__device__ __forceinline__ int reld(const DevForest &F, int x, int x0) {
    const int d = wrapd(F, x - x0);
    return d > F.D / 2 ? d - F.D : d;
}

// State of all leaves: one array, or two with a per-level choice of the
// current one (af_state_pair).
template <typename T>
struct StateView {
    using value = T;
    T *base0, *base1;
    const int32_t *level;  // leaf levels (read only when parity != 0)
    uint32_t parity;       // bit l: level l is current in base1
    int64_t plane;         // plane stride
    int ncomp, W;          // components, lattice width
    __device__ __forceinline__ T *patch(int q) const {
        T *b = (parity != 0u && ((parity >> __ldg(level + q)) & 1u)) ? base1 : base0;
        return b + (int64_t)q * ncomp * kPlanes * plane;
    }
    __device__ __forceinline__ T *patch_at_level(int q, int l) const {
        return (((parity >> l) & 1u) ? base1 : base0) + (int64_t)q * ncomp * kPlanes * plane;
    }
    __device__ __forceinline__ T *at(int q, int c, int k, int i, int j) const {
        return patch(q) + (int64_t)(c * kPlanes + k) * plane + (int64_t)(j + kGhost) * W + (i + kGhost);
    }
};

// Lattice indices (i, j) of point (x, y) in plane k of leaf q.
__device__ __forceinline__ void lattice_of(const DevForest &F, int q, int k, int x, int y, int &i, int &j) {
    const int sh = F.lmax - __ldg(F.level + q) + 1;  // hw = 2^sh
    const int hw = 1 << sh;
    int dx = reld(F, x, leaf_x0(F, q)), dy = reld(F, y, leaf_y0(F, q));
    if (k == kAvg || k == kYmid) dx -= hw / 2;
    if (k == kAvg || k == kXmid) dy -= hw / 2;
    i = dx >> sh;  // floor division (arithmetic shift)
    j = dy >> sh;
    // owners are always within two cells of the lattice; clamp defensively
    const int lo = -kGhost, hi = F.n + kGhost;
    i = i < lo ? lo : (i > hi ? hi : i);
    j = j < lo ? lo : (j > hi ? hi : j);
}

// Explicitly rounded operations: the reconstruction below is evaluated in
// one fixed order of roundings wherever it is inlined, so the direct and the
// planned ghost exchange (and the regrid transfer) agree bit for bit.
__device__ __forceinline__ float r_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double r_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float r_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double r_sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float r_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double r_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float r_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double r_fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// sum_a w_a row_a of the three rows of nodal values with weights (l0, l1, l2)
// in x and (m0, m1, m2) in y.
template <typename R>
__device__ __forceinline__ R recon_combine(R c00, R c10, R c01, R c11, R xl, R xr, R yb, R yt, R cen, R l0, R l1,
                                           R l2, R m0, R m1, R m2) {
    const R r0 = r_fma(l2, c10, r_fma(l1, yb, r_mul(l0, c00)));
    const R r1 = r_fma(l2, xr, r_fma(l1, cen, r_mul(l0, xl)));
    const R r2 = r_fma(l2, c11, r_fma(l1, yt, r_mul(l0, c01)));
    return r_fma(m2, r2, r_fma(m1, r1, r_mul(m0, r0)));
}

// The centre value of the biquadratic from its average and boundary nodes:
// (9/4) Q - (1/16) sum(corners) - (1/4) sum(edge midpoints).
template <typename R>
__device__ __forceinline__ R recon_centre(R c00, R c10, R c01, R c11, R xl, R xr, R yb, R yt, R avg) {
    const R sc = r_add(r_add(c00, c10), r_add(c01, c11)), se = r_add(r_add(xl, xr), r_add(yb, yt));
    return r_sub(r_sub(r_mul(R(2.25), avg), r_mul(R(0.0625), sc)), r_mul(R(0.25), se));
}

// The reconstruction (Eq. poly) of one cell at (xi, eta) in [-1, 1]^2 from
// its corners c.., edge midpoints x./y. and average: the tensor Lagrange
// interpolant on {-1,0,1}^2 whose centre value follows from the average.
// Evaluated in the state's precision R (FP32 for an FP32 state: GB300's
// FP64 rate is a small fraction of its FP32 rate).
template <typename R>
__device__ __forceinline__ R recon_eval(R c00, R c10, R c01, R c11, R xl, R xr, R yb, R yt, R avg, R xi, R eta) {
    const R cen = recon_centre<R>(c00, c10, c01, c11, xl, xr, yb, yt, avg);
    const R lx0 = r_mul(r_mul(R(0.5), xi), r_sub(xi, R(1))), lx1 = r_sub(R(1), r_mul(xi, xi));
    const R lx2 = r_mul(r_mul(R(0.5), xi), r_add(xi, R(1)));
    const R ly0 = r_mul(r_mul(R(0.5), eta), r_sub(eta, R(1))), ly1 = r_sub(R(1), r_mul(eta, eta));
    const R ly2 = r_mul(r_mul(R(0.5), eta), r_add(eta, R(1)));
    return recon_combine<R>(c00, c10, c01, c11, xl, xr, yb, yt, cen, lx0, lx1, lx2, ly0, ly1, ly2);
}

// Mean of the biquadratic reconstruction of a cell (nodal values as for
// recon_eval) over one of its four quarters: qx, qy = 0 for the lower half
// (xi or eta in [-1, 0]), 1 for the upper half.  The mean of each 1D
// Lagrange basis function over a half interval replaces its point value:
// over [-1, 0] the three functions average 5/12, 2/3, -1/12, over [0, 1]
// -1/12, 2/3, 5/12.  This is exactly the Simpson rule over the quarter
// (exact for quadratics), in 9 multiply-adds instead of 9 evaluations.
template <typename R>
__device__ __forceinline__ R recon_quarter_mean(R c00, R c10, R c01, R c11, R xl, R xr, R yb, R yt, R avg, int qx,
                                                int qy) {
    const R cen = recon_centre<R>(c00, c10, c01, c11, xl, xr, yb, yt, avg);
    const R lo = R(5) / R(12), mid = R(2) / R(3), hi = R(-1) / R(12);
    return recon_combine<R>(c00, c10, c01, c11, xl, xr, yb, yt, cen, qx ? hi : lo, mid, qx ? lo : hi,
                            qy ? hi : lo, mid, qy ? lo : hi);
}

// Simpson's rule over a cell from the values f(a, b) at its 3 x 3 points
// (a, b in {0, 1, 2}): exact for the biquadratic reconstruction.
template <typename R, typename Fn>
__device__ __forceinline__ R simpson9(Fn f) {
    const R w[3] = {R(1) / R(6), R(2) / R(3), R(1) / R(6)};
    R s = R(0);
#pragma unroll 1
    for (int e = 0; e < 9; ++e) s = r_fma(r_mul(w[e % 3], w[e / 3]), f(e % 3, e / 3), s);
    return s;
}

// 2^-sh (exact)
__device__ __forceinline__ void pow2_neg(int sh, float &r) { r = __int_as_float((127 - sh) << 23); }
__device__ __forceinline__ void pow2_neg(int sh, double &r) { r = __longlong_as_double((long long)(1023 - sh) << 52); }

// The nine values the reconstruction of one cell of leaf q combines at
// (x, y) (component 0; component c is cstride entries further), and where
// (x, y) lies in the cell.
template <typename T>
struct ReconSite {
    const T *v[9];  // c00, c10, c01, c11, xl, xr, yb, yt, avg
    T xi, eta;      // position in [-1, 1]^2
    int qx, qy;     // quarter holding (x, y)
};

// Point value (plane k, lattice entry (ii, jj)) of leaf q, whose cells are hw
// wide and whose corner is (x0, y0), component 0.  Point values on the leaf's
// boundary lines are read from their owner: a leaf whose neighbours are all
// same-level does not keep the copies in its ghost ring current (its step
// reads the neighbours directly).
template <typename T>
__device__ __forceinline__ const T *node_value(const DevForest &F, const StateView<T> &S, int q, int lq, int x0, int y0,
                                               int hw, int k, int ii, int jj) {
    if (ii > 0 && ii < F.n && jj > 0 && jj < F.n) return S.at(q, 0, k, ii, jj);
    const int nx = x0 + ii * hw + (k == kYmid ? hw / 2 : 0);
    const int ny = y0 + jj * hw + (k == kXmid ? hw / 2 : 0);
    const int o = entry_owner(F, k, nx, ny);
    if (o < 0 || o == q) return S.at(q, 0, k, ii, jj);
    const int lo = __ldg(F.level + o);
    const int ko = lo == lq ? k : kCorner;
    int oi, oj;
    lattice_of(F, o, ko, nx, ny, oi, oj);
    return S.at(o, 0, ko, oi, oj);
}

template <typename T>
__device__ void recon_locate(const DevForest &F, const StateView<T> &S, int q, int x, int y, ReconSite<T> &r) {
    const int lq = __ldg(F.level + q), sh = F.lmax - lq + 1;  // hw = 2^sh
    const int hw = 1 << sh;
    const int x0 = __ldg(F.ix + q) * F.n * hw, y0 = __ldg(F.iy + q) * F.n * hw;
    const int dx = reld(F, x, x0), dy = reld(F, y, y0);
    int i = dx >= 0 ? (dx >> sh) : 0, j = dy >= 0 ? (dy >> sh) : 0;
    i = i > F.n - 1 ? F.n - 1 : i;
    j = j > F.n - 1 ? F.n - 1 : j;
    T rhw;
    pow2_neg(sh, rhw);
    r.xi = (T)(2 * (dx - i * hw) - hw) * rhw;  // exact: a multiple of 1/2 (of 2^-sh, below 2^24 units)
    r.eta = (T)(2 * (dy - j * hw) - hw) * rhw;
    r.qx = 2 * (dx - i * hw) >= hw;
    r.qy = 2 * (dy - j * hw) >= hw;
    auto node = [&](int k, int ii, int jj) { return node_value<T>(F, S, q, lq, x0, y0, hw, k, ii, jj); };
#pragma unroll 1
    for (int e = 0; e < 8; ++e)  // four corners, xl, xr, yb, yt
        r.v[e] = node(e < 4 ? kCorner : (e < 6 ? kXmid : kYmid), i + (e < 6 ? e & 1 : 0), j + (e < 4 ? e >> 1 : (e == 7)));
    r.v[8] = S.at(q, 0, kAvg, i, j);
}

// The reconstruction at a located site (quarter: its mean over the quarter
// of the cell holding the site instead), component offset coff.
template <typename T>
__device__ __forceinline__ T recon_value(const ReconSite<T> &r, int64_t coff, bool quarter) {
    T v[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) v[e] = r.v[e][coff];
    if (quarter) return recon_quarter_mean<T>(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], r.qx, r.qy);
    return recon_eval<T>(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], r.xi, r.eta);
}

// Value of the reconstruction of leaf q, component c, at (x, y); with
// quarter set instead the mean of the reconstruction over the quarter of the
// cell holding (x, y) that (x, y) lies in (the centre of a finer cell).
template <typename T>
__device__ T recon_at(const DevForest &F, const StateView<T> &S, int q, int c, int x, int y, bool quarter = false) {
    ReconSite<T> r;
    recon_locate<T>(F, S, q, x, y, r);
    return recon_value<T>(r, (int64_t)c * kPlanes * S.plane, quarter);
}

// Values of every component c < nc for an entry of plane k of a destination at
// level lp from owner q (Section 3.1: copy, fine -> coarse, coarse -> fine).
// Averages from finer cells are summed in FP64; what is copied or interpolated
// stays in the state's precision.
template <typename T>
__device__ void transfer_all(const DevForest &F, const StateView<T> &S, int lp, int q, int k, int x, int y, int nc,
                             T out[3]) {
    const int lq = __ldg(F.level + q);
    const int64_t cs = (int64_t)kPlanes * S.plane;
    int i, j;
    if (lq == lp || (lq > lp && k != kAvg)) {
        const int ko = lq == lp ? k : kCorner;
        lattice_of(F, q, ko, x, y, i, j);
        const T *v = S.at(q, 0, ko, i, j);
        for (int c = 0; c < nc; ++c) out[c] = v[c * cs];
        return;
    }
    if (lq > lp) {  // an average from a finer owner: the mean of its four cells
        const int h = hwid(F, lq) / 2;
        const T *v[4];
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                lattice_of(F, q, kAvg, x + (2 * a - 1) * h, y + (2 * b - 1) * h, i, j);
                v[2 * b + a] = S.at(q, 0, kAvg, i, j);
            }
        for (int c = 0; c < nc; ++c) {
            double s = 0.0;
            s += (double)v[0][c * cs];
            s += (double)v[1][c * cs];
            s += (double)v[2][c * cs];
            s += (double)v[3][c * cs];
            out[c] = (T)(0.25 * s);
        }
        return;
    }
    if (k != kAvg || lq == lp - 1) {  // a coarser owner: its reconstruction (quarter mean for an average)
        ReconSite<T> r;
        recon_locate<T>(F, S, q, x, y, r);
        for (int c = 0; c < nc; ++c) out[c] = recon_value<T>(r, c * cs, k == kAvg);
        return;
    }
    // an average from an owner two or more levels coarser (a forest that is
    // not 2:1 balanced): Simpson's rule over the destination cell
    const int h = hwid(F, lp) / 2;
    for (int c = 0; c < nc; ++c)
        out[c] = simpson9<T>([&](int a, int b) { return recon_at<T>(F, S, q, c, x + (a - 1) * h, y + (b - 1) * h); });
}

// transfer_all out of line: for the few entries of a leaf that need it.
template <typename T>
__device__ __noinline__ void transfer_entry(const DevForest &F, const StateView<T> &S, int lp, int q, int k, int x, int y,
                                            T out[3]) {
    transfer_all<T>(F, S, lp, q, k, x, y, S.ncomp, out);
}

__device__ __forceinline__ void entry_xy(const DevForest &F, int p, int k, int i, int j, int &x, int &y) {
    const int hw = hwid(F, __ldg(F.level + p));
    x = leaf_x0(F, p) + i * hw + ((k == kAvg || k == kYmid) ? hw / 2 : 0);
    y = leaf_y0(F, p) + j * hw + ((k == kAvg || k == kXmid) ? hw / 2 : 0);
}

// True if some neighbour region of leaf p at its own level is not a leaf.
__device__ bool has_other_level_neighbour(const DevForest &F, int p) {
    const int l = __ldg(F.level + p);
    const int side = F.B << l;
    const int px = __ldg(F.ix + p), py = __ldg(F.iy + p);
    const int32_t *const map = F.map + map_offset(F.B, l);
    bool other = false;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        if (e == 4) continue;
        int nx = px + e % 3 - 1, ny = py + e / 3 - 1;
        nx = nx < 0 ? nx + side : (nx >= side ? nx - side : nx);
        ny = ny < 0 ? ny + side : (ny >= side ? ny - side : ny);
        other |= __ldg(map + (int64_t)ny * side + nx) < 0;
    }
    return other;
}

// One pass of the exchange: pass 0 = finer owners, 1 = same level, 2 = coarser.
template <typename T>
__global__ void fill_kernel(const __grid_constant__ DevForest F, StateView<T> S, uint32_t dst, uint32_t src, int flags, int pass) {
    const int p = blockIdx.x;
    const int lp = __ldg(F.level + p);
    if (!((dst >> lp) & 1u)) return;
    __shared__ int s_skip;
    if (threadIdx.x == 0) s_skip = !(flags & AF_FILL_ALL_PATCHES) && !has_other_level_neighbour(F, p);
    __syncthreads();
    if (s_skip) return;
    const int n = F.n, W = n + 2 * kGhost + 1;
    const int total = kPlanes * W * W;
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int k = e / (W * W), r = e - k * W * W;
        const int j = r / W - kGhost, i = r % W - kGhost;
        if (i > 0 && i < n && j > 0 && j < n) continue;  // strictly inside: the leaf's own
        if (i == n + kGhost && (k == kAvg || k == kYmid)) continue;  // never read by the step
        if (j == n + kGhost && (k == kAvg || k == kXmid)) continue;
        int x, y;
        entry_xy(F, p, k, i, j, x, y);
        const int q = entry_owner(F, k, x, y);
        if (q < 0 || q == p) continue;
        const int lq = __ldg(F.level + q);
        const int rel_pass = lq > lp ? 0 : (lq == lp ? 1 : 2);
        if (rel_pass != pass || !((src >> lq) & 1u)) continue;
        if ((flags & AF_FILL_SAME_LEVEL_ONLY) && lq != lp) continue;
        T v[3];
        transfer_all<T>(F, S, lp, q, k, x, y, S.ncomp, v);
        for (int c = 0; c < S.ncomp; ++c) *S.at(p, c, k, i, j) = v[c];
    }
}

// ---------------------------------------------------------------------------
// Ghost plan: the owner of every ghost entry resolved once per forest, so an
// exchange is two flat passes over a list instead of per-entry searches.
// Pass A (kinds copy / mean of four finer averages) writes only entries the
// destination does not own and reads only owned ones, so its entries are
// independent; among them are the boundary-line point values of every leaf
// with a coarser-or-finer neighbour.  Pass B (coarse -> fine) then reads the
// coarse leaf's whole cell -- boundary-line nodes included -- from that
// leaf's own lattice, which pass A has just made current.
struct GhostEntry {
    int32_t dst, src;
    uint16_t dst_off;  // plane * plane_stride + lattice index (component 0)
    uint8_t kind, levels;  // levels: dst level | src level << 4
    uint32_t aux;      // kinds 0, 1: source offset; kinds 2, 3: u | v << 16 (quarter cells of the source)
};
static_assert(sizeof(GhostEntry) == AF_GHOST_ENTRY_BYTES, "ghost plan entry layout");
enum : uint8_t { kGCopy = 0, kGMean4 = 1, kGPoint = 2, kGSimpson = 3 };

// Classify ghost entry (k, i, j) of leaf p; false if it is not exchanged.
__device__ bool ghost_entry(const DevForest &F, int64_t plane, int p, int lp, int k, int i, int j, GhostEntry &g) {
    const int n = F.n, W = n + 2 * kGhost + 1;
    if (i > 0 && i < n && j > 0 && j < n) return false;
    if (i == n + kGhost && (k == kAvg || k == kYmid)) return false;
    if (j == n + kGhost && (k == kAvg || k == kXmid)) return false;
    int x, y;
    entry_xy(F, p, k, i, j, x, y);
    const int q = entry_owner(F, k, x, y);
    if (q < 0 || q == p) return false;
    const int lq = __ldg(F.level + q);
    g.dst = p;
    g.src = q;
    g.dst_off = (uint16_t)(k * plane + (int64_t)(j + kGhost) * W + (i + kGhost));
    g.levels = (uint8_t)(lp | (lq << 4));
    int si, sj;
    if (lq == lp) {
        lattice_of(F, q, k, x, y, si, sj);
        g.kind = kGCopy;
        g.aux = (uint32_t)(k * plane + (int64_t)(sj + kGhost) * W + (si + kGhost));
    } else if (lq > lp) {
        if (k == kAvg) {
            const int h = hwid(F, lq) / 2;  // the four finer cells: (si, sj) .. (si + 1, sj + 1)
            lattice_of(F, q, kAvg, x - h, y - h, si, sj);
            g.kind = kGMean4;
            g.aux = (uint32_t)(kAvg * plane + (int64_t)(sj + kGhost) * W + (si + kGhost));
        } else {
            lattice_of(F, q, kCorner, x, y, si, sj);
            g.kind = kGCopy;
            g.aux = (uint32_t)(kCorner * plane + (int64_t)(sj + kGhost) * W + (si + kGhost));
        }
    } else {
        // in quarter cells of the source (2^sh units, sh >= 0 for a
        // leaf coarser than another)
        const int sh = F.lmax - lq - 1;
        int u = reld(F, x, leaf_x0(F, q)) >> sh, v = reld(F, y, leaf_y0(F, q)) >> sh;
        u = u < 0 ? 0 : (u > 4 * n ? 4 * n : u);
        v = v < 0 ? 0 : (v > 4 * n ? 4 * n : v);
        g.kind = k == kAvg ? kGSimpson : kGPoint;
        g.aux = (uint32_t)u | ((uint32_t)v << 16);
    }
    return true;
}

__device__ __forceinline__ bool plan_leaf(const DevForest &F, int p, int flags) {
    return (flags & AF_FILL_ALL_PATCHES) || has_other_level_neighbour(F, p);
}

// The lattice entries a leaf does not hold strictly inside, numbered in
// lattice order (plane, row, column): rows -2 .. 0 whole, six columns of rows
// 1 .. n-1 (-2 .. 0, n .. n+2), rows n .. n+2 whole.
__host__ __device__ constexpr int ring_count(int n) { return 6 * (n + 2 * kGhost + 1) + 6 * (n - 1); }
__device__ __forceinline__ void ring_entry(int n, int e, int &k, int &i, int &j) {
    const int W = n + 2 * kGhost + 1, per = ring_count(n), lo = 3 * W, mid = lo + 6 * (n - 1);
    k = e / per;
    const int r = e - k * per;
    if (r < lo) {
        j = r / W;
        i = r - j * W - kGhost;
        j -= kGhost;
    } else if (r < mid) {
        const int m = (r - lo) / 6, c = r - lo - 6 * m;
        j = m + 1;
        i = c < 3 ? c - kGhost : n + c - 3;
    } else {
        const int m = (r - mid) / W;
        i = r - mid - m * W - kGhost;
        j = n + m;
    }
}

// counts[0]: pass-A entries, counts[1]: pass-B entries.
__global__ void __launch_bounds__(256) plan_count_kernel(const __grid_constant__ DevForest F, int64_t plane, int flags,
                                                         unsigned long long *counts) {
    const int p = blockIdx.x;
    __shared__ unsigned int s_cnt[2];
    if (threadIdx.x < 2) s_cnt[threadIdx.x] = 0;
    if (!plan_leaf(F, p, flags)) return;  // the same for the whole CTA
    __syncthreads();
    const int lp = __ldg(F.level + p), total = kPlanes * ring_count(F.n);
    unsigned int c0 = 0, c1 = 0;
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        int k, i, j;
        ring_entry(F.n, e, k, i, j);
        GhostEntry g;
        if (ghost_entry(F, plane, p, lp, k, i, j, g)) (g.kind >= kGPoint ? c1 : c0) += 1;
    }
    c0 = __reduce_add_sync(0xffffffffu, c0);
    c1 = __reduce_add_sync(0xffffffffu, c1);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&s_cnt[0], c0);
        atomicAdd(&s_cnt[1], c1);
    }
    __syncthreads();
    if (threadIdx.x < 2 && s_cnt[threadIdx.x]) atomicAdd(counts + threadIdx.x, (unsigned long long)s_cnt[threadIdx.x]);
}

// Pass-A entries fill [0, na), pass-B entries [na, na + nb); cursor[2] starts at 0.
// Each leaf reserves one contiguous range per pass and writes its entries
// there in lattice order (plane, row, column), so the threads of an
// executing warp touch consecutive destination entries (and, for copies,
// consecutive source entries): the exchange's accesses coalesce.  The order
// of the leaves' ranges is whatever order the CTAs reserve them in; each
// destination entry appears once, so the order does not change the result.
// The entries are found once and kept in shared memory (pass A from the
// front, pass B from the back) until their ranges are known.
__global__ void __launch_bounds__(256) plan_build_kernel(const __grid_constant__ DevForest F, int64_t plane, int flags, GhostEntry *plan,
                                                         long long na, long long nb, unsigned long long *cursor,
                                                         int *overflow) {
    const int p = blockIdx.x;
    extern __shared__ __align__(16) unsigned char plan_smem[];
    GhostEntry *const held = reinterpret_cast<GhostEntry *>(plan_smem);  // [kPlanes * ring_count(n)]
    __shared__ unsigned long long s_base[2];
    __shared__ unsigned int s_warp[2][32];
    if (!plan_leaf(F, p, flags)) return;  // the same for the whole CTA
    const int lp = __ldg(F.level + p), total = kPlanes * ring_count(F.n);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = (blockDim.x + 31) >> 5;
    const unsigned below = (1u << lane) - 1u;
    unsigned run0 = 0, run1 = 0;
    for (int e0 = 0; e0 < total; e0 += blockDim.x) {
        const int e = e0 + threadIdx.x;
        GhostEntry g;
        bool v = false;
        if (e < total) {
            int k, i, j;
            ring_entry(F.n, e, k, i, j);
            v = ghost_entry(F, plane, p, lp, k, i, j, g);
        }
        const int b = v ? (g.kind >= kGPoint) : 0;
        const unsigned m0 = __ballot_sync(0xffffffffu, v && b == 0), m1 = __ballot_sync(0xffffffffu, v && b == 1);
        if (lane == 0) {
            s_warp[0][warp] = __popc(m0);
            s_warp[1][warp] = __popc(m1);
        }
        __syncthreads();
        unsigned off0 = 0, off1 = 0, tot0 = 0, tot1 = 0;
        for (int w = 0; w < nwarp; ++w) {
            if (w < warp) {
                off0 += s_warp[0][w];
                off1 += s_warp[1][w];
            }
            tot0 += s_warp[0][w];
            tot1 += s_warp[1][w];
        }
        if (v) held[b ? total - 1 - (int)(run1 + off1 + __popc(m1 & below)) : (int)(run0 + off0 + __popc(m0 & below))] = g;
        run0 += tot0;
        run1 += tot1;
        __syncthreads();
    }
    if (threadIdx.x < 2) {
        const unsigned c = threadIdx.x ? run1 : run0;
        s_base[threadIdx.x] = c ? atomicAdd(cursor + threadIdx.x, (unsigned long long)c) : 0ull;
    }
    __syncthreads();
    for (unsigned e = threadIdx.x; e < run0 + run1; e += blockDim.x) {
        const int b = e >= run0;
        const unsigned r = b ? e - run0 : e;
        const long long slot = (long long)(s_base[b] + r);
        if (slot >= (b ? nb : na))
            atomicExch(overflow, 1);
        else
            plan[(b ? na : 0) + slot] = held[b ? total - 1 - (int)r : (int)r];
    }
}

// Pass A for one component (advection): one entry per thread and turn.
template <typename T>
__global__ void plan_exec_a1(StateView<T> S, const GhostEntry *__restrict__ plan, long long na, uint32_t levels,
                            int same_only) {
    const unsigned block = chain_begin();
    for (long long t = block * (long long)blockDim.x + threadIdx.x; t < na; t += (long long)gridDim.x * blockDim.x) {
        const GhostEntry g = plan[t];
        const int ld = g.levels & 15, ls = g.levels >> 4;
        if (!((levels >> ld) & 1u) || !((levels >> ls) & 1u) || (same_only && ld != ls)) continue;
        const T *src = S.patch_at_level(g.src, ls) + g.aux;
        T *dst = S.patch_at_level(g.dst, ld) + g.dst_off;
        const int64_t cs = (int64_t)kPlanes * S.plane;
        for (int c = 0; c < S.ncomp; ++c) {
            if (g.kind == kGCopy) {
                dst[c * cs] = src[c * cs];
            } else {
                const T *a = src + c * cs;
                const double sum = (double)a[0] + (double)a[1] + (double)a[S.W] + (double)a[S.W + 1];
                dst[c * cs] = (T)(0.25 * sum);
            }
        }
    }
}

// Pass A for three components (acoustics).  A thread's work is a chain of
// dependent reads from L2 (31 of 33 cycles per instruction were spent waiting),
// so what counts is how many reads are in flight: all components are read before
// any is written (a store may alias the next load, as far as the compiler knows)
// and the next entry before this one's values, in few enough registers for 48
// warps on an SM.  Adaptive acoustics on 5436 leaves 1201 -> 1162 us a coarse
// step; with one component there is nothing to overlap, and plan_exec_a1 is the
// faster one (2944 leaves 178 us, 196 this way).
template <typename T>
__global__ void __launch_bounds__(256, 6) plan_exec_a3(StateView<T> S, const GhostEntry *__restrict__ plan, long long na,
                                                       uint32_t levels, int same_only) {
    const unsigned block = chain_begin();
    const long long stride = (long long)gridDim.x * blockDim.x;
    const int64_t cs = (int64_t)kPlanes * S.plane;
    long long t = block * (long long)blockDim.x + threadIdx.x;
    if (t >= na) return;
    GhostEntry g = plan[t];
    for (;;) {
        t += stride;
        const bool more = t < na;
        const GhostEntry next = plan[more ? t : 0];
        const int ld = g.levels & 15, ls = g.levels >> 4;
        if (((levels >> ld) & 1u) && ((levels >> ls) & 1u) && (!same_only || ld == ls)) {
            const T *src = S.patch_at_level(g.src, ls) + g.aux;
            T *dst = S.patch_at_level(g.dst, ld) + g.dst_off;
            T v[3];
            if (g.kind == kGCopy) {
#pragma unroll
                for (int c = 0; c < 3; ++c) v[c] = src[c * cs];
            } else {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const T *a = src + c * cs;
                    const double sum = (double)a[0] + (double)a[1] + (double)a[S.W] + (double)a[S.W + 1];
                    v[c] = (T)(0.25 * sum);
                }
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) dst[c * cs] = v[c];
        }
        if (!more) break;
        g = next;
    }
}

// Pass B in FP32.  Few entries, each a chain: the entry, then nine values of the
// coarser leaf per component.  All NC components' values are read before one is
// written, and nothing is computed in FP64 (positions in a cell are multiples of
// a half: exact in either).  Adaptive acoustics on 5436 leaves 1157 -> 1135 us a
// coarse step, advection on 2944 leaves 184 -> 179.
template <int NC>
__global__ void __launch_bounds__(256) plan_exec_b(StateView<float> S, int n, const GhostEntry *__restrict__ plan, long long nb,
                                                   uint32_t levels) {
    using T = float;
    const unsigned block = chain_begin();
    for (long long t = block * (long long)blockDim.x + threadIdx.x; t < nb; t += (long long)gridDim.x * blockDim.x) {
        const GhostEntry g = plan[t];
        const int ld = g.levels & 15, ls = g.levels >> 4;
        if (!((levels >> ld) & 1u) || !((levels >> ls) & 1u)) continue;
        T *dst = S.patch_at_level(g.dst, ld) + g.dst_off;
        const int u = (int)(g.aux & 0xffffu), v = (int)(g.aux >> 16);
        const int64_t cs = (int64_t)kPlanes * S.plane;
        const int W = S.W;
        // the cell holding the quarter-cell position (u, v) of the source leaf,
        // chosen as the direct exchange chooses it
        int ci = u / 4, cj = v / 4;
        ci = ci > n - 1 ? n - 1 : ci;
        cj = cj > n - 1 ? n - 1 : cj;
        const T *cell = S.patch_at_level(g.src, ls) + (int64_t)(cj + kGhost) * W + (ci + kGhost);
        T w[NC][9], r[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const T *cr = cell + c * cs + kCorner * S.plane, *xm = cell + c * cs + kXmid * S.plane;
            const T *ym = cell + c * cs + kYmid * S.plane, *av = cell + c * cs + kAvg * S.plane;
            w[c][0] = cr[0], w[c][1] = cr[1], w[c][2] = cr[W], w[c][3] = cr[W + 1];
            w[c][4] = xm[0], w[c][5] = xm[1], w[c][6] = ym[0], w[c][7] = ym[W], w[c][8] = av[0];
        }
        if (g.kind != kGPoint) {
            // the mean over the quarter of the cell that (u, v), the centre of a
            // cell one level finer, lies in
#pragma unroll
            for (int c = 0; c < NC; ++c)
                r[c] = recon_quarter_mean<T>(w[c][0], w[c][1], w[c][2], w[c][3], w[c][4], w[c][5], w[c][6], w[c][7], w[c][8],
                                             u - 4 * ci >= 2, v - 4 * cj >= 2);
        } else {
            const T xi = (T)0.5 * (T)(u - 4 * ci) - (T)1, eta = (T)0.5 * (T)(v - 4 * cj) - (T)1;
#pragma unroll
            for (int c = 0; c < NC; ++c)
                r[c] = recon_eval<T>(w[c][0], w[c][1], w[c][2], w[c][3], w[c][4], w[c][5], w[c][6], w[c][7], w[c][8], xi, eta);
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) dst[c * cs] = r[c];
    }
}

// Pass B in FP64, component by component: read ahead as above, acoustics were no
// faster (levels 2-5, 671 us a coarse step either way) and advection slower (2944
// leaves 1000 us, 1014).
__global__ void plan_exec_b_f64(StateView<double> S, int n, const GhostEntry *__restrict__ plan, long long nb, uint32_t levels) {
    using T = double;
    const unsigned block = chain_begin();
    for (long long t = block * (long long)blockDim.x + threadIdx.x; t < nb; t += (long long)gridDim.x * blockDim.x) {
        const GhostEntry g = plan[t];
        const int ld = g.levels & 15, ls = g.levels >> 4;
        if (!((levels >> ld) & 1u) || !((levels >> ls) & 1u)) continue;
        const T *q = S.patch_at_level(g.src, ls);
        T *dst = S.patch_at_level(g.dst, ld) + g.dst_off;
        const int u0 = (int)(g.aux & 0xffffu), v0 = (int)(g.aux >> 16);
        const int64_t cs = (int64_t)kPlanes * S.plane;
        const int W = S.W;
        // value at quarter-cell position (u, v) of the source leaf, with the
        // cell chosen as the direct exchange chooses it
        // quarter: the mean over the quarter of the cell holding (u, v) that
        // (u, v), the centre of a cell one level finer, lies in
        auto at = [&](const T *b, int u, int v, bool quarter) -> T {
            int ci = u / 4, cj = v / 4;
            ci = ci > n - 1 ? n - 1 : ci;
            cj = cj > n - 1 ? n - 1 : cj;
            const T xi = (T)(0.5 * (double)(u - 4 * ci) - 1.0), eta = (T)(0.5 * (double)(v - 4 * cj) - 1.0);
            const T *cr = b + kCorner * S.plane + (int64_t)(cj + kGhost) * W + (ci + kGhost);
            const T *xm = b + kXmid * S.plane + (int64_t)(cj + kGhost) * W + (ci + kGhost);
            const T *ym = b + kYmid * S.plane + (int64_t)(cj + kGhost) * W + (ci + kGhost);
            const T *av = b + kAvg * S.plane + (int64_t)(cj + kGhost) * W + (ci + kGhost);
            if (quarter)
                return recon_quarter_mean<T>(cr[0], cr[1], cr[W], cr[W + 1], xm[0], xm[1], ym[0], ym[W], av[0],
                                             u - 4 * ci >= 2, v - 4 * cj >= 2);
            return recon_eval<T>(cr[0], cr[1], cr[W], cr[W + 1], xm[0], xm[1], ym[0], ym[W], av[0], xi, eta);
        };
        for (int c = 0; c < S.ncomp; ++c) {
            const T *b = q + c * cs;
            dst[c * cs] = at(b, u0, v0, g.kind != kGPoint);
        }
    }
}

// Sites of a quarter of a leaf that a refinement reads: the corners, left-edge
// and bottom-edge midpoints and averages of its m x m cells, closed.
__host__ __device__ constexpr int quarter_sites(int m) { return (m + 1) * (m + 1) + 2 * m * (m + 1) + m * m; }
constexpr int kStagedMax = 32;  // largest patch whose quarter is staged (26 KB in FP64)

// The state of every leaf of the new forest from the old one.
//  - A leaf of both forests is copied (16-byte words).
//  - A child of an old leaf is interpolated: its 4 (n+1)^2 entries use each of
//    the quarter's sites up to a dozen times, so the CTA first gathers them in
//    shared memory, looking the owner of a boundary site up once.  Only entries
//    on the old leaf's own boundary may belong to another leaf and are looked
//    up one by one.  (Looked up per entry and site, in 64 bits, the transfer
//    between 2100 and 2700 leaves averaged 721 us; with the quarters staged and
//    the look-ups kept out of line, 94.  The copies alone would take 17 us at
//    the HBM rate; latency of the few CTAs that refine bounds the rest.)
//  - A merged leaf is averaged from its children, the owner of everything
//    strictly inside known from four lookups.
template <typename T>
__global__ void __launch_bounds__(256, 3) transfer_kernel(
    const __grid_constant__ DevForest Fo, const __grid_constant__ StateView<T> So, const __grid_constant__ DevForest Fn,
    const __grid_constant__ StateView<T> Sn) {
    const int p = blockIdx.x;
    const int l = __ldg(Fn.level + p), px = __ldg(Fn.ix + p), py = __ldg(Fn.iy + p);
    const int64_t words = (int64_t)Sn.ncomp * kPlanes * Sn.plane;
    T *dst = Sn.patch(p);
    int same = -1;
    if (l <= Fo.lmax) {
        const long long side = (long long)Fo.B << l;
        same = __ldg(Fo.map + map_offset(Fo.B, l) + (long long)py * side + px);
    }
    const int n = Fn.n, m = n + 1;
    const int hwn = 2 << (Fn.lmax - l);
    const int x0 = px * n * hwn, y0 = py * n * hwn;
    if (same >= 0) {
        const T *srcp = So.patch(same);
        constexpr int V = 16 / (int)sizeof(T);  // elements per 16-byte load
        if (words % V == 0 && ((reinterpret_cast<uintptr_t>(srcp) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0) {
            const int4 *s4 = reinterpret_cast<const int4 *>(srcp);
            int4 *d4 = reinterpret_cast<int4 *>(dst);
            for (int64_t e = threadIdx.x; e < words / V; e += blockDim.x) d4[e] = __ldg(s4 + e);
        } else {
            for (int64_t e = threadIdx.x; e < words; e += blockDim.x) dst[e] = srcp[e];
        }
        __syncthreads();
        // The point values on the right (i = n) and top (j = n) faces: where the
        // neighbour across was the owner in the old forest (same level, or
        // finer) the leaf's own copy is not kept current -- a step of a leaf
        // with eight same-level neighbours stores node lines 0 .. n-1 only --
        // yet the leaf owns them in the new forest if that neighbour became
        // coarser.  Take them from their old owner.
        for (int e = threadIdx.x; e < 4 * m; e += blockDim.x) {
            const int side = e / m, r = e - side * m;  // 0, 1: corner / left-mid on line i = n; 2, 3: on j = n
            const int k = side == 0 || side == 2 ? kCorner : (side == 1 ? kXmid : kYmid);
            const int i = side < 2 ? n : r, j = side < 2 ? r : n;
            if ((k == kXmid && j == n) || (k == kYmid && i == n)) continue;
            const int x = x0 + i * hwn + (k == kYmid ? hwn / 2 : 0);
            const int y = y0 + j * hwn + (k == kXmid ? hwn / 2 : 0);
            const int q = entry_owner(Fo, k, x, y);
            if (q < 0 || q == same) continue;
            T v[3];
            transfer_entry<T>(Fo, So, l, q, k, x, y, v);
            for (int c = 0; c < Sn.ncomp; ++c) *Sn.at(p, c, k, i, j) = v[c];
        }
        return;
    }
    for (int64_t e = threadIdx.x; e < words; e += blockDim.x) dst[e] = T(0);
    // the old leaves of the new leaf's four quarters (the same one for a child)
    extern __shared__ __align__(16) unsigned char site_smem[];
    T *const site = reinterpret_cast<T *>(site_smem);
    __shared__ int s_q[4];
    if (threadIdx.x < 4) {
        const int w = n * hwn;
        s_q[threadIdx.x] = lookup(Fo, x0 + (threadIdx.x & 1 ? w - 1 : 0), y0 + (threadIdx.x & 2 ? w - 1 : 0));
    }
    __syncthreads();
    const int q0 = s_q[0], nc = Sn.ncomp;
    const bool child = q0 >= 0 && __ldg(Fo.level + q0) == l - 1 && n % 2 == 0 && n <= kStagedMax;
    // every quarter one leaf: then those own what lies strictly inside
    bool four = q0 >= 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) four = four && s_q[e] >= 0 && __ldg(Fo.level + (s_q[e] < 0 ? 0 : s_q[e])) <= l + 1;
    const int mq = n / 2, cx = (px & 1) * mq, cy = (py & 1) * mq, sites = quarter_sites(mq);
    const int qhw = 2 * hwn, qx0 = x0 - cx * qhw, qy0 = y0 - cy * qhw;  // the old leaf's cells and corner (child)
    const int b1 = (mq + 1) * (mq + 1), b2 = b1 + (mq + 1) * mq, b3 = b2 + mq * (mq + 1);
    if (child) {
        for (int e = threadIdx.x; e < sites; e += blockDim.x) {
            const int k = e < b1 ? kCorner : (e < b2 ? kXmid : (e < b3 ? kYmid : kAvg));
            const int r = e - (e < b1 ? 0 : (e < b2 ? b1 : (e < b3 ? b2 : b3)));
            const int w = (k == kCorner || k == kXmid) ? mq + 1 : mq, j = r / w, i = r - j * w;
            const T *v = k == kAvg ? So.at(q0, 0, kAvg, cx + i, cy + j)
                                   : node_value<T>(Fo, So, q0, l - 1, qx0, qy0, qhw, k, cx + i, cy + j);
            for (int c = 0; c < nc; ++c) site[c * sites + e] = v[c * kPlanes * So.plane];
        }
    }
    __syncthreads();
    // The cells' averages and the point values on their boundaries: node
    // lines 0 .. n, the right (i = n) and top (j = n) lines included -- a leaf
    // finer than its neighbour across that face owns those nodes (the finer
    // grid's values are used at coarse-fine faces), and nothing else writes
    // them.  Entries owned by another leaf are overwritten by the exchange
    // that follows a regrid.
    for (int e = threadIdx.x; e < kPlanes * m * m; e += blockDim.x) {
        const int k = e / (m * m), r = e - k * m * m, j = r / m, i = r - j * m;
        if ((i == n && (k == kAvg || k == kYmid)) || (j == n && (k == kAvg || k == kXmid))) continue;
        const int x = x0 + i * hwn + ((k == kAvg || k == kYmid) ? hwn / 2 : 0);
        const int y = y0 + j * hwn + ((k == kAvg || k == kXmid) ? hwn / 2 : 0);
        const bool inside = k == kAvg || (i > 0 && i < n && j > 0 && j < n) ||
                            (k == kXmid && i > 0 && i < n) || (k == kYmid && j > 0 && j < n);
        const int nx = cx * 2 + i, ny = cy * 2 + j;  // in half cells of the old leaf (child)
        const bool in = k == kAvg || ((k == kYmid || (nx > 0 && nx < 2 * n)) && (k == kXmid || (ny > 0 && ny < 2 * n)));
        int q;
        if (child ? in : inside && four)
            q = child ? q0 : s_q[(2 * i + (k == kAvg || k == kYmid) >= n) + 2 * (2 * j + (k == kAvg || k == kXmid) >= n)];
        else
            q = entry_owner(Fo, k, x, y);
        if (q < 0) continue;
        T v[3];
        if (child && q == q0) {
            // cell (ci, cj) of the quarter; the last line is the last cell's far edge
            const int ux = 2 * i + (k == kAvg || k == kYmid), uy = 2 * j + (k == kAvg || k == kXmid);  // quarter cells
            const int ci = min(ux >> 2, mq - 1), cj = min(uy >> 2, mq - 1);
            const T xi = T(0.5) * (T)(ux - 4 * ci) - T(1), eta = T(0.5) * (T)(uy - 4 * cj) - T(1);
            const int c0 = cj * (mq + 1) + ci, xo = b1 + cj * (mq + 1) + ci, yo = b2 + cj * mq + ci, ao = b3 + cj * mq + ci;
            for (int c = 0; c < nc; ++c) {
                const T *w = site + c * sites;
                const T c00 = w[c0], c10 = w[c0 + 1], c01 = w[c0 + mq + 1], c11 = w[c0 + mq + 2];
                const T xl = w[xo], xr = w[xo + 1], yb = w[yo], yt = w[yo + mq], av = w[ao];
                v[c] = k == kAvg ? recon_quarter_mean<T>(c00, c10, c01, c11, xl, xr, yb, yt, av, ux - 4 * ci >= 2, uy - 4 * cj >= 2)
                                 : recon_eval<T>(c00, c10, c01, c11, xl, xr, yb, yt, av, xi, eta);
            }
        } else {
            // an average comes from at most one level finer (the four children's
            // mean); a point value is the coinciding vertex of any finer owner
            if (k == kAvg && __ldg(Fo.level + q) > l + 1) continue;
            transfer_entry<T>(Fo, So, l, q, k, x, y, v);
        }
        for (int c = 0; c < nc; ++c) *Sn.at(p, c, k, i, j) = v[c];
    }
}

template <typename T>
__device__ __forceinline__ void atomic_add_state(T *p, double v);
template <>
__device__ __forceinline__ void atomic_add_state<double>(double *p, double v) { atomicAdd(p, v); }
template <>
__device__ __forceinline__ void atomic_add_state<float>(float *p, double v) { atomicAdd(p, (float)v); }

// A chain of loads per thread -- the leaf, its neighbour, the registers of both
// -- on few threads, so its time is that chain's latency: the registers of all
// NC components are read before any is written, which the compiler cannot
// arrange itself (they may be the same as far as it knows).  Adaptive acoustics on
// 5436 leaves 1161 -> 1157 us a coarse step, levels 3-7 with a ring per tree
// 3996 -> 3980.
template <typename T, int NC>
__global__ void reflux_kernel(const __grid_constant__ DevForest F, StateView<T> S, uint32_t sync, double dx0, double dy0, double *freg) {
    const int n = F.n;
    const int64_t total = (int64_t)F.nleaf * 4 * n;
    const unsigned block = chain_begin();
    for (int64_t t = block * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        int p, side, k;
        face_entry(t, n, p, side, k);
        const int l = __ldg(F.level + p);
        if (l >= AF_MAX_LEVEL || !((sync >> l) & 1u) || !((sync >> (l + 1)) & 1u)) continue;
        const int hw = hwid(F, l), x0 = leaf_x0(F, p), y0 = leaf_y0(F, p);
        const int x1 = x0 + n * hw, y1 = y0 + n * hw;
        int px, py;
        if (side == 0) { px = x0 - 1; py = y0 + k * hw + hw / 2; }
        else if (side == 1) { px = x1; py = y0 + k * hw + hw / 2; }
        else if (side == 2) { px = x0 + k * hw + hw / 2; py = y0 - 1; }
        else { px = x0 + k * hw + hw / 2; py = y1; }
        const int q = lookup(F, px, py);
        if (q < 0 || __ldg(F.level + q) != l + 1) continue;
        const int hf = hwid(F, l + 1);
        const int fside = side ^ 1;
        const int start = side < 2 ? reld(F, y0 + k * hw, leaf_y0(F, q)) : reld(F, x0 + k * hw, leaf_x0(F, q));
        const int kf = start / hf;
        if (kf < 0 || kf + 1 >= n) continue;
        const int ci = side == 0 ? 0 : (side == 1 ? n - 1 : k);
        const int cj = side == 2 ? 0 : (side == 3 ? n - 1 : k);
        const double h = (side < 2 ? dx0 : dy0) * __hiloint2double((1023 - l) << 20, 0);  // / 2^l, exactly
        const int64_t rw = 4LL * NC * n;
        double *rc = freg + p * rw + (int64_t)side * NC * n + k, *rf = freg + q * rw + (int64_t)fside * NC * n + kf;
        double coarse[NC], f0[NC], f1[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            coarse[c] = rc[c * n];
            f0[c] = rf[c * n];
            f1[c] = rf[c * n + 1];
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const double fine = 0.5 * (f0[c] + f1[c]);
            const double d = (side == 1 || side == 3) ? (coarse[c] - fine) / h : (fine - coarse[c]) / h;
            atomic_add_state<T>(S.at(p, c, kAvg, ci, cj), d);
            rc[c * n] = 0.0;
            rf[c * n] = 0.0;
            rf[c * n + 1] = 0.0;
        }
    }
}

template <typename T>
__global__ void tag_kernel(const __grid_constant__ DevForest F, StateView<T> S, int comp, int kind, double dx0, double dy0, double rthr,
                           double cthr, int8_t *tags, double *ind) {
    const int p = blockIdx.x, n = F.n;
    const int l = __ldg(F.level + p);
    // kind 0: largest value and largest negated one; kind 1: largest centred
    // differences in x, y
    double a = -INFINITY, b = -INFINITY;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        const int j = e / n, i = e % n;
        if (kind == 0) {
            const double q = *S.at(p, comp, kAvg, i, j);
            a = fmax(a, q);
            b = fmax(b, -q);
        } else if (i >= 1 && i < n - 1 && j >= 1 && j < n - 1) {
            // the largest differences; divided by the widths once below (division
            // by a positive number is monotonic, rounding included)
            a = fmax(a, fabs((double)*S.at(p, comp, kAvg, i + 1, j) - (double)*S.at(p, comp, kAvg, i - 1, j)));
            b = fmax(b, fabs((double)*S.at(p, comp, kAvg, i, j + 1) - (double)*S.at(p, comp, kAvg, i, j - 1)));
        }
    }
    __shared__ double sa[256], sb[256];
    sa[threadIdx.x] = a;
    sb[threadIdx.x] = b;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) {
            sa[threadIdx.x] = fmax(sa[threadIdx.x], sa[threadIdx.x + s]);
            sb[threadIdx.x] = fmax(sb[threadIdx.x], sb[threadIdx.x + s]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double v = sa[0] + sb[0];
        if (kind != 0) {
            // mesh widths of level l, exactly (their FP64 divisions, needed by kind
            // 1 only, stood at the start of every thread: 82 leaves 4.7 -> 5.05 us)
            const double half = __hiloint2double((1023 + 1 - l) << 20, 0);  // 2 / 2^l
            v = fmax(fmax(sa[0] / (half * dx0), sb[0] / (half * dy0)), 0.0);
        }
        if (ind) ind[p] = v;
        tags[p] = (int8_t)(v >= rthr ? 1 : (v < cthr ? -1 : 0));
    }
}

constexpr int kMassBlocks = 256;
constexpr int kMassThreads = 256;

// Pass 1: block b sums leaves [b * chunk, (b+1) * chunk) in a fixed order.
template <typename T>
__global__ void mass_partial(DevForest F, StateView<T> S, double dx0, double dy0, int chunk, double *part) {
    const int n = F.n, nc = S.ncomp;
    __shared__ double sm[kMassThreads];
    for (int c = 0; c < nc; ++c) {
        double acc = 0.0;
        const int p0 = blockIdx.x * chunk, p1 = min(F.nleaf, p0 + chunk);
        for (int p = p0; p < p1; ++p) {
            const int l = __ldg(F.level + p);
            const double area = (dx0 / (double)(1LL << l)) * (dy0 / (double)(1LL << l));
            double s = 0.0;
            for (int e = threadIdx.x; e < n * n; e += blockDim.x) s += (double)*S.at(p, c, kAvg, e % n, e / n);
            acc += s * area;
        }
        sm[threadIdx.x] = acc;
        __syncthreads();
        for (int s = blockDim.x / 2; s > 0; s >>= 1) {
            if ((int)threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
            __syncthreads();
        }
        if (threadIdx.x == 0) part[blockIdx.x * nc + c] = sm[0];
        __syncthreads();
    }
}

__global__ void mass_final(const double *part, int nblocks, int nc, double *out) {
    __shared__ double sm[kMassThreads];
    for (int c = 0; c < nc; ++c) {
        double acc = 0.0;
        for (int b = threadIdx.x; b < nblocks; b += blockDim.x) acc += part[b * nc + c];
        sm[threadIdx.x] = acc;
        __syncthreads();
        for (int s = blockDim.x / 2; s > 0; s >>= 1) {
            if ((int)threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
            __syncthreads();
        }
        if (threadIdx.x == 0) out[c] = sm[0];
        __syncthreads();
    }
}

bool check_cfg(const af_config *cfg) {
    return cfg && cfg->n >= 2 && cfg->n <= 64 && (cfg->eq == AF_ADVECTION || cfg->eq == AF_ACOUSTICS) &&
           (cfg->prec == AF_F64 || cfg->prec == AF_F32) && cfg->ncomp == (cfg->eq == AF_ADVECTION ? 1 : 3);
}

bool check_forest(const af_forest *f) {
    return f && f->nleaf >= 0 && f->B >= 1 && f->lmax >= 0 && f->lmax <= AF_MAX_LEVEL &&
           (f->nleaf == 0 || (f->d_level && f->d_ix && f->d_iy && f->d_map));
}

template <typename T>
StateView<T> view(const af_config &cfg, const af_forest &f, const af_state_pair &st) {
    StateView<T> s;
    s.base0 = static_cast<T *>(st.buf[0]);
    s.base1 = static_cast<T *>(st.buf[1]);
    s.level = f.d_level;
    s.parity = st.parity;
    s.plane = plane_stride(cfg.n);
    s.ncomp = cfg.ncomp;
    s.W = cfg.n + 2 * kGhost + 1;
    return s;
}

af_state_pair single(const void *d_state) {
    af_state_pair p;
    p.buf[0] = p.buf[1] = const_cast<void *>(d_state);
    p.parity = 0u;
    p.pad_ = 0u;
    return p;
}

// A pair is usable if its current arrays exist and are aligned; a pair whose
// parity is zero may leave buf[1] NULL.
af_status check_pair(const af_state_pair *st) {
    if (!st || !st->buf[0] || (st->parity != 0u && !st->buf[1])) return AF_ERR_ARG;
    if ((reinterpret_cast<uintptr_t>(st->buf[0]) | reinterpret_cast<uintptr_t>(st->buf[1])) & 31u)
        return AF_ERR_LAYOUT;
    return AF_OK;
}

// Launch of a kernel of 256-thread CTAs over a list, chained to the one before
// it unless that unbalances the SMs of a graph (in a stream the launch gap saved
// is more).
template <auto Kern, typename... Args>
cudaError_t launch_list(bool chain, int grid, cudaStream_t s, const Args &...args) {
    if (chain && !chain_even(grid, resident_ctas<Kern>(256, 0))) chain = !recording(s);
    return launch_chained(chain, Kern, grid, 256, 0, s, args...);
}

inline af_status launched() { return cudaGetLastError() == cudaSuccess ? AF_OK : AF_ERR_CUDA; }

int mass_blocks(int nleaf) { return nleaf < kMassBlocks ? (nleaf < 1 ? 1 : nleaf) : kMassBlocks; }

}  // namespace
}  // namespace af

using namespace af;

extern "C" int64_t af_forest_map_offset(int32_t B, int32_t level) {
    if (B < 1 || level < 0 || level > AF_MAX_LEVEL + 1) return -1;
    return map_offset(B, level);
}

extern "C" af_status af_forest_build_map(int32_t nleaf, int32_t B, int32_t lmax, const int32_t *h_level,
                                         const int32_t *h_ix, const int32_t *h_iy, int32_t *h_map) {
    if (nleaf < 0 || B < 1 || lmax < 0 || lmax > AF_MAX_LEVEL || !h_map) return AF_ERR_ARG;
    if (nleaf > 0 && (!h_level || !h_ix || !h_iy)) return AF_ERR_ARG;
    const long long total = map_offset(B, lmax + 1);
    for (long long e = 0; e < total; ++e) h_map[e] = -1;
    for (int p = 0; p < nleaf; ++p) {
        const int l = h_level[p];
        if (l < 0 || l > lmax) return AF_ERR_ARG;
        const long long side = (long long)B << l;
        if (h_ix[p] < 0 || h_ix[p] >= side || h_iy[p] < 0 || h_iy[p] >= side) return AF_ERR_ARG;
        int32_t &slot = h_map[map_offset(B, l) + (long long)h_iy[p] * side + h_ix[p]];
        if (slot >= 0) return AF_ERR_ARG;
        slot = p;
    }
    // regions inside a leaf, at every finer level: -2 - (the leaf)
    for (int p = 0; p < nleaf; ++p) {
        const int l = h_level[p];
        for (int m = l + 1; m <= lmax; ++m) {
            const long long side = (long long)B << m, w = 1LL << (m - l);
            const long long x0 = (long long)h_ix[p] * w, y0 = (long long)h_iy[p] * w;
            int32_t *row = h_map + map_offset(B, m);
            for (long long y = y0; y < y0 + w; ++y)
                for (long long x = x0; x < x0 + w; ++x) {
                    int32_t &slot = row[y * side + x];
                    if (slot != -1) return AF_ERR_ARG;  // overlapping leaves
                    slot = -2 - p;
                }
        }
    }
    return AF_OK;
}

extern "C" af_status af_fill_ghosts_pair(const af_config *cfg, const af_forest *forest, uint32_t dst_levels,
                                         uint32_t src_levels, int32_t flags, const af_state_pair *state,
                                         void *stream) {
    if (!check_cfg(cfg) || !check_forest(forest)) return AF_ERR_ARG;
    if (forest->nleaf == 0) return AF_OK;
    if (const af_status e = check_pair(state)) return e;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const DevForest F = make_dev(*forest, cfg->n);
    for (int pass = 0; pass < 3; ++pass) {
        if ((flags & AF_FILL_SAME_LEVEL_ONLY) && pass != 1) continue;
        if (cfg->prec == AF_F64)
            fill_kernel<double><<<forest->nleaf, 256, 0, s>>>(F, view<double>(*cfg, *forest, *state), dst_levels,
                                                              src_levels, flags, pass);
        else
            fill_kernel<float><<<forest->nleaf, 256, 0, s>>>(F, view<float>(*cfg, *forest, *state), dst_levels,
                                                             src_levels, flags, pass);
        if (launched() != AF_OK) return AF_ERR_CUDA;
    }
    return AF_OK;
}

extern "C" af_status af_fill_ghosts(const af_config *cfg, const af_forest *forest, uint32_t dst_levels,
                                    uint32_t src_levels, int32_t flags, void *d_state, void *stream) {
    const af_state_pair st = single(d_state);
    return af_fill_ghosts_pair(cfg, forest, dst_levels, src_levels, flags, &st, stream);
}

// Upward-closed level set: with its lowest level it holds every level up to lmax.
static bool upward_closed(uint32_t levels, int lmax) {
    if (levels == 0u) return true;
    const int lo = __builtin_ctz(levels);
    const uint32_t want = (lmax >= 31 ? 0xffffffffu : ((1u << (lmax + 1)) - 1u)) & ~((1u << lo) - 1u);
    return (levels & want) == want;
}

extern "C" af_status af_ghost_plan_count(const af_config *cfg, const af_forest *forest, int32_t flags,
                                         int64_t *d_counts, void *stream) {
    if (!check_cfg(cfg) || !check_forest(forest) || !d_counts) return AF_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(d_counts) & 7u) return AF_ERR_LAYOUT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(d_counts, 0, 2 * sizeof(int64_t), s) != cudaSuccess) return AF_ERR_CUDA;
    if (forest->nleaf == 0) return AF_OK;
    plan_count_kernel<<<forest->nleaf, 256, 0, s>>>(make_dev(*forest, cfg->n), plane_stride(cfg->n), flags,
                                                     reinterpret_cast<unsigned long long *>(d_counts));
    return launched();
}

extern "C" af_status af_ghost_plan_build(const af_config *cfg, const af_forest *forest, int32_t flags, void *d_plan,
                                         int64_t n_a, int64_t n_b, int64_t *d_scratch, void *stream) {
    if (!check_cfg(cfg) || !check_forest(forest) || !d_scratch || n_a < 0 || n_b < 0) return AF_ERR_ARG;
    if (n_a + n_b > 0 && !d_plan) return AF_ERR_ARG;
    if ((reinterpret_cast<uintptr_t>(d_plan) | reinterpret_cast<uintptr_t>(d_scratch)) & 15u) return AF_ERR_LAYOUT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // scratch: two slot cursors and an overflow flag
    if (cudaMemsetAsync(d_scratch, 0, 3 * sizeof(int64_t), s) != cudaSuccess) return AF_ERR_CUDA;
    if (forest->nleaf == 0) return AF_OK;
    const size_t held = (size_t)kPlanes * ring_count(cfg->n) * sizeof(GhostEntry);
    // the limit of the largest patches (51 KB), whatever this call's: it belongs to
    // the kernel, and another thread may be about to launch it for larger patches
    constexpr int limit = kPlanes * ring_count(64) * (int)sizeof(GhostEntry);
    if (cudaFuncSetAttribute(plan_build_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, limit) != cudaSuccess)
        return AF_ERR_CUDA;
    plan_build_kernel<<<forest->nleaf, 256, held, s>>>(
        make_dev(*forest, cfg->n), plane_stride(cfg->n), flags, static_cast<GhostEntry *>(d_plan), n_a, n_b,
        reinterpret_cast<unsigned long long *>(d_scratch), reinterpret_cast<int *>(d_scratch + 2));
    return launched();
}

extern "C" af_status af_fill_ghosts_planned(const af_config *cfg, const af_forest *forest, uint32_t levels,
                                            int32_t flags, const void *d_plan, int64_t n_a, int64_t n_b,
                                            const af_state_pair *state, void *stream) {
    if (!check_cfg(cfg) || !check_forest(forest) || n_a < 0 || n_b < 0) return AF_ERR_ARG;
    if (!upward_closed(levels, forest->lmax)) return AF_ERR_ARG;
    if (n_a + n_b == 0 || levels == 0u) return AF_OK;
    if (!d_plan) return AF_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(d_plan) & 15u) return AF_ERR_LAYOUT;
    if (const af_status e = check_pair(state)) return e;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const GhostEntry *plan = static_cast<const GhostEntry *>(d_plan);
    const int same = (flags & AF_FILL_SAME_LEVEL_ONLY) ? 1 : 0;
    auto grid = [](int64_t m) { return (int)(m / 256 + 1 < 152 * 16 ? m / 256 + 1 : 152 * 16); };
    // as the step between two exchanges; FP64 passes in a graph (all of this are
    // advection's) only if both are even (319 leaves of 20 cells 9.1 us, 11.5 chained)
    bool chain = cfg->prec == AF_F32 || cfg->eq == AF_ADVECTION;
    if (chain && cfg->prec == AF_F64 &&
        !(chain_even_mixed(grid(n_a), resident_ctas<plan_exec_a1<double>>(256, 0)) &&
          chain_even_mixed(grid(n_b), resident_ctas<plan_exec_b_f64>(256, 0))))
        chain = !recording(s);
    cudaError_t e = cudaSuccess;
    auto pass_a = [&](auto one) {
        using T = decltype(one);
        const StateView<T> v = view<T>(*cfg, *forest, *state);
        return cfg->ncomp == 3 ? launch_list<plan_exec_a3<T>>(chain, grid(n_a), s, v, plan, n_a, levels, same)
                               : launch_list<plan_exec_a1<T>>(chain, grid(n_a), s, v, plan, n_a, levels, same);
    };
    if (n_a > 0) e = cfg->prec == AF_F64 ? pass_a(0.0) : pass_a(0.0f);
    if (e != cudaSuccess) return AF_ERR_CUDA;
    if (n_b > 0 && !same) {
        if (cfg->prec == AF_F64) {
            e = launch_list<plan_exec_b_f64>(chain, grid(n_b), s, view<double>(*cfg, *forest, *state), cfg->n, plan + n_a, n_b, levels);
        } else {
            const StateView<float> v = view<float>(*cfg, *forest, *state);
            e = cfg->ncomp == 3 ? launch_list<plan_exec_b<3>>(chain, grid(n_b), s, v, cfg->n, plan + n_a, n_b, levels)
                                : launch_list<plan_exec_b<1>>(chain, grid(n_b), s, v, cfg->n, plan + n_a, n_b, levels);
        }
        if (e != cudaSuccess) return AF_ERR_CUDA;
    }
    return AF_OK;
}

extern "C" af_status af_transfer_pair(const af_config *cfg, const af_forest *old_forest,
                                      const af_state_pair *old_state, const af_forest *new_forest, void *d_new,
                                      void *stream) {
    if (!check_cfg(cfg) || !check_forest(old_forest) || !check_forest(new_forest)) return AF_ERR_ARG;
    if (old_forest->B != new_forest->B || old_forest->lmax != new_forest->lmax) return AF_ERR_ARG;
    if (new_forest->nleaf == 0) return AF_OK;
    if (const af_status e = check_pair(old_state)) return e;
    if (!d_new || d_new == old_state->buf[0] || d_new == old_state->buf[1]) return AF_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(d_new) & 31u) return AF_ERR_LAYOUT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const DevForest Fo = make_dev(*old_forest, cfg->n), Fn = make_dev(*new_forest, cfg->n);
    const af_state_pair sn = single(d_new);
    const size_t held = cfg->n <= kStagedMax ? (size_t)quarter_sites(cfg->n / 2) * cfg->ncomp * (cfg->prec == AF_F64 ? 8 : 4) : 0;
    if (cfg->prec == AF_F64)
        transfer_kernel<double><<<new_forest->nleaf, 256, held, s>>>(Fo, view<double>(*cfg, *old_forest, *old_state), Fn,
                                                                    view<double>(*cfg, *new_forest, sn));
    else
        transfer_kernel<float><<<new_forest->nleaf, 256, held, s>>>(Fo, view<float>(*cfg, *old_forest, *old_state), Fn,
                                                                   view<float>(*cfg, *new_forest, sn));
    return launched();
}

extern "C" af_status af_transfer(const af_config *cfg, const af_forest *old_forest, const void *d_old,
                                 const af_forest *new_forest, void *d_new, void *stream) {
    if (!d_old) return AF_ERR_ARG;
    const af_state_pair so = single(d_old);
    return af_transfer_pair(cfg, old_forest, &so, new_forest, d_new, stream);
}

extern "C" af_status af_reflux_pair(const af_config *cfg, const af_forest *forest, uint32_t sync_levels, double dx0,
                                    double dy0, double *d_flux_reg, const af_state_pair *state, void *stream) {
    if (!check_cfg(cfg) || !check_forest(forest)) return AF_ERR_ARG;
    if (!(dx0 > 0.0) || !(dy0 > 0.0)) return AF_ERR_ARG;
    if (forest->nleaf == 0) return AF_OK;
    if (!d_flux_reg) return AF_ERR_ARG;
    if (const af_status e = check_pair(state)) return e;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const DevForest F = make_dev(*forest, cfg->n);
    const long long total = (long long)forest->nleaf * 4 * cfg->n;
    const int blocks = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
    const bool chain = cfg->prec == AF_F32 || cfg->eq == AF_ADVECTION;  // as the step before the fix
    const auto run = [&](auto state_view) {
        using T = typename decltype(state_view)::value;
        return cfg->eq == AF_ADVECTION
                   ? launch_list<reflux_kernel<T, 1>>(chain, blocks, s, F, state_view, sync_levels, dx0, dy0, d_flux_reg)
                   : launch_list<reflux_kernel<T, 3>>(chain, blocks, s, F, state_view, sync_levels, dx0, dy0, d_flux_reg);
    };
    const cudaError_t e = cfg->prec == AF_F64 ? run(view<double>(*cfg, *forest, *state)) : run(view<float>(*cfg, *forest, *state));
    return e == cudaSuccess ? AF_OK : AF_ERR_CUDA;
}

extern "C" af_status af_reflux(const af_config *cfg, const af_forest *forest, uint32_t sync_levels, double dx0,
                               double dy0, double *d_flux_reg, void *d_state, void *stream) {
    const af_state_pair st = single(d_state);
    return af_reflux_pair(cfg, forest, sync_levels, dx0, dy0, d_flux_reg, &st, stream);
}

extern "C" af_status af_tag_pair(const af_config *cfg, const af_forest *forest, const af_state_pair *state,
                                 int32_t comp, int32_t kind, double dx0, double dy0, double refine_thr,
                                 double coarsen_thr, int8_t *d_tags, double *d_indicator, void *stream) {
    if (!check_cfg(cfg) || !check_forest(forest)) return AF_ERR_ARG;
    if (comp < 0 || comp >= cfg->ncomp || (kind != 0 && kind != 1)) return AF_ERR_ARG;
    if (!(dx0 > 0.0) || !(dy0 > 0.0)) return AF_ERR_ARG;
    if (forest->nleaf == 0) return AF_OK;
    if (!d_tags) return AF_ERR_ARG;
    if (const af_status e = check_pair(state)) return e;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const DevForest F = make_dev(*forest, cfg->n);
    if (cfg->prec == AF_F64)
        tag_kernel<double><<<forest->nleaf, 256, 0, s>>>(F, view<double>(*cfg, *forest, *state), comp, kind, dx0, dy0,
                                                        refine_thr, coarsen_thr, d_tags, d_indicator);
    else
        tag_kernel<float><<<forest->nleaf, 256, 0, s>>>(F, view<float>(*cfg, *forest, *state), comp, kind, dx0, dy0,
                                                       refine_thr, coarsen_thr, d_tags, d_indicator);
    return launched();
}

extern "C" af_status af_tag(const af_config *cfg, const af_forest *forest, const void *d_state, int32_t comp,
                            int32_t kind, double dx0, double dy0, double refine_thr, double coarsen_thr,
                            int8_t *d_tags, double *d_indicator, void *stream) {
    const af_state_pair st = single(d_state);
    return af_tag_pair(cfg, forest, &st, comp, kind, dx0, dy0, refine_thr, coarsen_thr, d_tags, d_indicator, stream);
}

extern "C" int64_t af_mass_scratch_bytes(int32_t nleaf, int32_t ncomp) {
    if (nleaf < 0 || ncomp < 1) return 0;
    return (int64_t)mass_blocks(nleaf) * ncomp * (int64_t)sizeof(double);
}

namespace af {
namespace {
// Both passes of the deterministic mass reduction into `part`.
af_status launch_mass(const af_config &cfg, const af_forest &forest, const af_state_pair &st, double dx0, double dy0,
                      double *part, double *d_mass, cudaStream_t s) {
    const DevForest F = make_dev(forest, cfg.n);
    const int nb = mass_blocks(forest.nleaf);
    const int chunk = (forest.nleaf + nb - 1) / nb;
    if (cfg.prec == AF_F64)
        mass_partial<double><<<nb, kMassThreads, 0, s>>>(F, view<double>(cfg, forest, st), dx0, dy0, chunk, part);
    else
        mass_partial<float><<<nb, kMassThreads, 0, s>>>(F, view<float>(cfg, forest, st), dx0, dy0, chunk, part);
    if (launched() != AF_OK) return AF_ERR_CUDA;
    mass_final<<<1, kMassThreads, 0, s>>>(part, nb, cfg.ncomp, d_mass);
    return launched();
}
}  // namespace
}  // namespace af

extern "C" af_status af_mass_pair(const af_config *cfg, const af_forest *forest, const af_state_pair *state,
                                  double dx0, double dy0, void *d_scratch, double *d_mass, void *stream) {
    if (!check_cfg(cfg) || !check_forest(forest)) return AF_ERR_ARG;
    if (!(dx0 > 0.0) || !(dy0 > 0.0) || !d_mass || !d_scratch) return AF_ERR_ARG;
    if ((reinterpret_cast<uintptr_t>(d_scratch) | reinterpret_cast<uintptr_t>(d_mass)) & 7u) return AF_ERR_LAYOUT;
    if (forest->nleaf > 0)
        if (const af_status e = check_pair(state)) return e;
    af_state_pair st = state ? *state : single(nullptr);
    return launch_mass(*cfg, *forest, st, dx0, dy0, static_cast<double *>(d_scratch), d_mass,
                       static_cast<cudaStream_t>(stream));
}

extern "C" af_status af_mass(const af_config *cfg, const af_forest *forest, const void *d_state, double dx0,
                             double dy0, void *d_scratch, double *d_mass, void *stream) {
    const af_state_pair st = single(d_state);
    return af_mass_pair(cfg, forest, &st, dx0, dy0, d_scratch, d_mass, stream);
}

// ---------------------------------------------------------------------------
// af_mass_noalloc: af_mass for callers that cannot allocate device memory.
// The per-block partial sums live in a fixed array compiled into the
// library instead of a caller-provided scratch buffer.  Every device that
// loads the library keeps this array (8 KB) until the process exits.
static __device__ __align__(256) double g_mass_partials[256 * 4];  // kMassBlocks partial sums x up to 4 components

extern "C" af_status af_mass_noalloc(const af_config *cfg, const af_forest *forest, const void *d_state, double dx0,
                                     double dy0, double *d_mass, void *stream) {
    if (!check_cfg(cfg) || !check_forest(forest)) return AF_ERR_ARG;
    if (!(dx0 > 0.0) || !(dy0 > 0.0) || !d_mass) return AF_ERR_ARG;
    if (forest->nleaf > 0 && !d_state) return AF_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(d_mass) & 7u) return AF_ERR_LAYOUT;
    const af_state_pair st = single(d_state);
    if (forest->nleaf > 0)
        if (const af_status e = check_pair(&st)) return e;  // the alignment af_mass requires
    const int nb = mass_blocks(forest->nleaf);
    // capacity check: partial sums needed vs. the fixed array
    if ((int64_t)nb * cfg->ncomp > (int64_t)(sizeof(g_mass_partials) / sizeof(double))) return AF_ERR_ARG;
    // In host code g_mass_partials names a host-side stand-in, not device
    // memory.  Its device address is looked up on every call, with the
    // caller's device current, so that it always belongs to the current
    // context (a cached address would go stale after a device reset).  The
    // lookup enqueues no work and allocates nothing.
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_mass_partials) != cudaSuccess || p == nullptr) return AF_ERR_CUDA;
    // every partial sum read by mass_final is written by mass_partial first,
    // so nothing left in the array by an earlier call is used
    return launch_mass(*cfg, *forest, st, dx0, dy0, static_cast<double *>(p), d_mass,
                       static_cast<cudaStream_t>(stream));
}

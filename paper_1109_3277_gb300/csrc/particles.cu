// Particle kernels (§2 of Günther et al., arXiv:1109.3277): moving
// bounce-back correction and momentum exchange (Eq. 4-5), anisotropic
// Hertz / Berne–Pechukas and lubrication pair forces (Eq. 6-9), the
// Newton–Euler update, and the node coverage with fill and empty.
//
// The coverage kernels run a CTA per particle over the rows of its bounding
// box, the shell fill one or more tiles of that box, the update four lanes and
// the pair forces eight lanes per particle.  Sums are 64-bit fixed point or
// FP64 in an order that does not depend on the split of the work, so results
// are bit-reproducible run to run, alone and in a batch.
#include <algorithm>
#include <cmath>

#include "lbe_internal.cuh"

namespace lbe {

namespace {

constexpr int PT = 128;  // threads per per-particle CTA
// Threads per particle of the claim, the transition and the reset: with fewer
// particles than SMs a particle's rows spread over 16 warps (one ellipsoid
// (12, 6): 5.3, 5.2 and 4.8 us against 9.0, 8.6 and 7.6 with four).
constexpr int PT_WIDE = 512;
static int cover_threads(int np) { return np < 152 ? PT_WIDE : PT; }

// Tiles of a particle's box in the shell fill: nx x ny x nz of them, of 30 x
// tyi x tzi nodes; a tile's link entries are filled up to a multiple of pad.
struct ShellGrid {
    int nx, ny, nz, tyi, tzi, pad;
};

// The particles [first, first + parts) whose tiles a launch of the shell fill
// takes.
struct ShellRange {
    int first, parts;
};

// ---------------------------------------------------------- geometry (FP64)
// The inside test is written with explicit round-to-nearest intrinsics so
// that no multiply-add is contracted: the quadric is evaluated in a fixed
// operation order.

__device__ __forceinline__ double m_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double a_(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double s_(double a, double b) { return __dsub_rn(a, b); }

__device__ void rotmat(const double *q, double R[3][3])
{
    double w = q[0], x = q[1], y = q[2], z = q[3];
    R[0][0] = s_(1.0, m_(2.0, a_(m_(y, y), m_(z, z))));
    R[0][1] = m_(2.0, s_(m_(x, y), m_(w, z)));
    R[0][2] = m_(2.0, a_(m_(x, z), m_(w, y)));
    R[1][0] = m_(2.0, a_(m_(x, y), m_(w, z)));
    R[1][1] = s_(1.0, m_(2.0, a_(m_(x, x), m_(z, z))));
    R[1][2] = m_(2.0, s_(m_(y, z), m_(w, x)));
    R[2][0] = m_(2.0, s_(m_(x, z), m_(w, y)));
    R[2][1] = m_(2.0, a_(m_(y, z), m_(w, x)));
    R[2][2] = s_(1.0, m_(2.0, a_(m_(x, x), m_(y, y))));
}

__device__ __forceinline__ bool periodic_dim(const Lat &L, int k) { return k < 2 || !L.walls; }
__device__ __forceinline__ int ext_of(const Lat &L, int k) { return k == 0 ? L.nx : (k == 1 ? L.ny : L.nz); }

// Displacement of node coordinate xi from particle coordinate X: nearest
// periodic image, shifting the integer first and subtracting once.
__device__ __forceinline__ double node_disp(const Lat &L, int k, int xi, double X)
{
    if (periodic_dim(L, k)) {
        int n = ext_of(L, k);
        const double d = s_((double)xi, X);
        if (fabs(d) < 0.49 * n) return d;  // no shift: the same value without the division
        double s = rint(__ddiv_rn(d, (double)n));
        return s_((double)((long long)xi - (long long)s * n), X);
    }
    return s_((double)xi, X);
}

__device__ __forceinline__ double pair_disp(const Lat &L, int k, double a, double b)
{
    double r = s_(b, a);
    if (periodic_dim(L, k)) {
        double n = (double)ext_of(L, k);
        if (fabs(r) < 0.49 * n) return r;  // no shift: the same value without the division
        r = s_(r, m_(n, rint(__ddiv_rn(r, n))));
    }
    return r;
}

struct Geo {
    double R[3][3];
    float R32[3][3];
    double ip2, io2;
    float ip2f, io2f;
};

// Inside test: an FP32 evaluation decides unless it lies within 1e-3 of the
// surface, where the exact FP64 evaluation (oracle operation order) decides.
// d32 is the displacement in FP32 (error ~1e-7 lattice units); dx the exact
// FP64 displacement, formed only when needed.
__device__ __forceinline__ bool inside_q32(const Geo &g, const float d[3], float &q32)
{
    float e[3];
#pragma unroll
    for (int k = 0; k < 3; k++) e[k] = g.R32[0][k] * d[0] + g.R32[1][k] * d[1] + g.R32[2][k] * d[2];
    q32 = e[0] * e[0] * g.ip2f + (e[1] * e[1] + e[2] * e[2]) * g.io2f;
    return q32 < 0.999f;
}

__device__ __forceinline__ bool inside_exact(const Geo &g, const double dx[3])
{
    double d[3];
#pragma unroll
    for (int k = 0; k < 3; k++)
        d[k] = a_(a_(m_(g.R[0][k], dx[0]), m_(g.R[1][k], dx[1])), m_(g.R[2][k], dx[2]));
    double qv = a_(a_(m_(m_(d[0], d[0]), g.ip2), m_(m_(d[1], d[1]), g.io2)), m_(m_(d[2], d[2]), g.io2));
    return qv <= 1.0;
}

struct Box {
    int lo[3], ext[3];  // lower corner in unwrapped coordinates, extents
    int full[3];        // the axis spans a whole period (nearest image taken per node)
    int count;
};

// Axis-aligned box containing the ellipsoid at X (not necessarily wrapped),
// widened by one node, as doubles: lo[k] = floor(X - h) - 1, hi[k] =
// ceil(X + h) + 1 with h the half-extent of the rotated ellipsoid along k.
// Non-finite geometry, or a centre further than 1e9 from the origin (a
// particle that has left any lattice), gives lo > hi: an empty box.
__device__ void box_of(const Lat &L, const double *X, const double R[3][3], double rp, double ro,
                       double lo[3], double hi[3])
{
    for (int k = 0; k < 3; k++) {
        double h = sqrt(rp * rp * R[k][0] * R[k][0] + ro * ro * (R[k][1] * R[k][1] + R[k][2] * R[k][2]));
        lo[k] = floor(X[k] - h) - 1.0;
        hi[k] = ceil(X[k] + h) + 1.0;
        if (!(lo[k] <= hi[k]) || !(fabs(X[k]) < 1e9) || !(h < 1e9)) {
            lo[k] = 1.0;
            hi[k] = 0.0;
        }
    }
}

__device__ __forceinline__ bool box_empty(const double lo[3], const double hi[3])
{
    return !(lo[0] <= hi[0] && lo[1] <= hi[1] && lo[2] <= hi[2]);
}

// Integer box over lattice nodes: along walls clamped to [0, n-1]; along
// periodic axes at most one period.  Coordinates stay unwrapped (relative to
// the particle, as the box was formed around it), so a node's displacement
// from the particle is one exact subtraction; an axis clamped to a whole
// period is flagged and takes the nearest image per node instead.  All
// arithmetic before the conversion to int is in double and |lo|, |hi| are
// below ~1e9 (box_of), so no int overflows.
__device__ void finish_box(const Lat &L, const double *lo_in, const double *hi_in, Box &b)
{
    bool empty = box_empty(lo_in, hi_in);
    for (int k = 0; k < 3; k++) {
        double n = (double)ext_of(L, k);
        double lo = lo_in[k], hi = hi_in[k];
        b.full[k] = 0;
        if (empty) {
            lo = 0.0;
            hi = -1.0;
        } else if (!periodic_dim(L, k)) {
            lo = fmax(lo, 0.0);
            hi = fmin(hi, n - 1.0);
        } else if (hi - lo + 1.0 > n) {
            lo = 0.0;
            hi = n - 1.0;
            b.full[k] = 1;
        }
        b.lo[k] = hi >= lo ? (int)lo : 0;
        b.ext[k] = hi >= lo ? (int)(hi - lo + 1.0) : 0;
    }
    b.count = b.ext[0] * b.ext[1] * b.ext[2];
}

__device__ __forceinline__ int wrapi(int v, int n)
{
    v %= n;
    return v < 0 ? v + n : v;
}

// Box entry k: unwrapped coordinates u[3] and the wrapped node (x, y, z).
__device__ __forceinline__ void box_node(const Lat &L, const Box &b, int k, int u[3], int &x, int &y,
                                         int &z)
{
    int bx = k % b.ext[0];
    int t = k / b.ext[0];
    int by = t % b.ext[1];
    int bz = t / b.ext[1];
    u[0] = b.lo[0] + bx;
    u[1] = b.lo[1] + by;
    u[2] = b.lo[2] + bz;
    x = wrapi(u[0], L.nx);
    y = wrapi(u[1], L.ny);
    z = wrapi(u[2], L.nz);
}

// Displacement of a box node from the particle centre X (the centre the box
// was formed around), equal to the nearest-image displacement.
__device__ __forceinline__ double box_disp(const Lat &L, const Box &b, int k, int u, int w, double X)
{
    return b.full[k] ? node_disp(L, k, w, X) : s_((double)u, X);
}

__device__ __forceinline__ bool is_wall_z(const Lat &L, int z) { return L.walls && (z == 0 || z == L.nz - 1); }

// ---- candidate rows -------------------------------------------------------
// Along a row of the box (fixed unwrapped y, z) the nodes the inside test
// can accept lie in one x interval: where the quadric of the ellipsoid is
// at most 1.  The interval of the quadric at most QSPAN, widened by a node
// on each side, holds all of them whatever the FP32 rounding of its
// computation (relative errors ~1e-6 against a margin of ~1% of the radii),
// so only those candidates are looked at.  Boxes that span a whole period use
// the plain box loop.
constexpr float QSPAN = 1.02f;

// x interval [xa, xb] (unwrapped, clamped to the box) of row (u1, u2) for
// the ellipsoid g at Xi + Xf (integer and fraction, so that FP32 displacements
// carry no cancellation); xa > xb when the row misses it.  All in FP32: with
// the conversions in FP64, whose rate is 1/64 of FP32's, they bounded the
// coverage kernels.
__device__ __forceinline__ void row_span(const Geo &g, const int Xi[3], const float Xf[3], const Box &b, int u1, int u2,
                                         int &xa, int &xb)
{
    const float dy = (float)(u1 - Xi[1]) - Xf[1], dz = (float)(u2 - Xi[2]) - Xf[2];
    const float w[3] = {g.ip2f, g.io2f, g.io2f};
    float A = 0.f, B = 0.f, C = -QSPAN;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float r0 = g.R32[0][k], ck = __fmaf_rn(g.R32[1][k], dy, __fmul_rn(g.R32[2][k], dz));
        A = __fmaf_rn(w[k] * r0, r0, A);
        B = __fmaf_rn(2.f * w[k] * r0, ck, B);
        C = __fmaf_rn(w[k] * ck, ck, C);
    }
    const float D = __fmaf_rn(B, B, -4.f * A * C);
    xa = 1;
    xb = 0;
    if (!(D >= 0.f) || !(A > 0.f)) return;
    const float sq = sqrtf(D), ia = 0.5f / A;
    const float lo = Xf[0] + (-B - sq) * ia, hi = Xf[0] + (-B + sq) * ia;
    if (!(lo >= -1e6f && hi <= 1e6f)) {  // beyond any lattice: the whole box row
        xa = b.lo[0];
        xb = b.lo[0] + b.ext[0] - 1;
        return;
    }
    xa = max(Xi[0] + (int)floorf(lo) - 1, b.lo[0]);
    xb = min(Xi[0] + (int)ceilf(hi) + 1, b.lo[0] + b.ext[0] - 1);
}

__device__ __forceinline__ bool box_full(const Box &b) { return b.full[0] || b.full[1] || b.full[2]; }

// The nodes of a row that the inside test accepts form one interval (the
// quadric is convex along x; three neighbouring nodes on its level 1 would
// need radii beyond 1e6).  Two bounds of it from FP32 quadrics, whose error
// (below 1e-5) is far inside the margins: outer [oa, ob] holds every
// accepted node, inner [ia, ib] only accepted ones.  They differ in the few
// nodes within 1e-3 of the surface, which alone need the FP64 test.  Empty
// intervals have a > b.
struct RowSpan {
    int oa, ob, ia, ib;
};

struct RowEval {  // the FP32 quadric along a row
    float bx[3], R0[3], w1, w2;
    int Xi;
    float Xf;
    __device__ __forceinline__ float operator()(int ux) const
    {
        const float d = (float)(ux - Xi) - Xf;
        float e[3];
#pragma unroll
        for (int k = 0; k < 3; k++) e[k] = __fmaf_rn(R0[k], d, bx[k]);
        return __fmaf_rn(e[0] * e[0], w1, __fmaf_rn(e[1], e[1], e[2] * e[2]) * w2);
    }
};

__device__ __forceinline__ RowSpan span_of(const Geo &g, const int Xi[3], const float Xf[3], const Box &b, int u1,
                                           int u2)
{
    RowSpan r;
    row_span(g, Xi, Xf, b, u1, u2, r.oa, r.ob);
    RowEval q;
    const float dy = (float)(u1 - Xi[1]) - Xf[1], dz = (float)(u2 - Xi[2]) - Xf[2];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        q.R0[k] = g.R32[0][k];
        q.bx[k] = __fmaf_rn(g.R32[1][k], dy, g.R32[2][k] * dz);
    }
    q.w1 = g.ip2f;
    q.w2 = g.io2f;
    q.Xi = Xi[0];
    q.Xf = Xf[0];
    while (r.oa <= r.ob && q(r.oa) > 1.001f) r.oa++;
    while (r.oa <= r.ob && q(r.ob) > 1.001f) r.ob--;
    r.ia = r.oa;
    r.ib = r.ob;
    while (r.ia <= r.ib && !(q(r.ia) < 0.999f)) r.ia++;
    while (r.ia <= r.ib && !(q(r.ib) < 0.999f)) r.ib--;
    return r;
}

// Rows of a box that is no whole period along any axis, 32 at a time per
// warp (one a lane): f(chunk, valid, u1, u2) is called by whole warps, chunk
// counting the 32s.
template <class F>
__device__ __forceinline__ void for_rows(const Box &b, F f)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int rows = b.ext[1] * b.ext[2];
    for (int c = warp; c * 32 < rows; c += nw) {
        const int r = c * 32 + lane;
        const bool valid = r < rows;
        f(c, valid, b.lo[1] + (valid ? r % b.ext[1] : 0), b.lo[2] + (valid ? r / b.ext[1] : 0));
    }
}

// Every node of the intervals [a, b] of the warp's 32 rows (u1, u2): f(node)
// by groups of eight lanes along x, so that a row's accesses stay together.
template <class F>
__device__ __forceinline__ void fill_rows(const Lat &L, int a, int b, int u1, int u2, F f)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int xw = wrapi(a, L.nx), row = L.nx * (wrapi(u1, L.ny) + L.ny * wrapi(u2, L.nz));
    const int len = max(0, b - a + 1);
    if (!__any_sync(full, len > 0)) return;
#pragma unroll
    for (int it = 0; it < 8; it++) {
        const int src = it * 4 + (lane >> 3);
        const int x0 = __shfl_sync(full, xw, src), n0 = __shfl_sync(full, row, src), ln = __shfl_sync(full, len, src);
        for (int k = lane & 7; k < ln; k += 8) {
            int x = x0 + k;
            if (x >= L.nx) x -= L.nx;  // len <= nx
            f(n0 + x);
        }
    }
}

// Every node of a box that spans a whole period along some axis, once each.
template <class F>
__device__ __forceinline__ void for_box(const Box &b, F f)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int c = warp; c * 32 < b.count; c += nw) {
        const int k = c * 32 + lane;
        const bool valid = k < b.count;
        const int kk = valid ? k : 0;
        const int t = kk / b.ext[0];
        f(c, valid, b.lo[0] + kk % b.ext[0], b.lo[1] + t % b.ext[1], b.lo[2] + t / b.ext[1]);
    }
}

// ---- coverage geometry ----------------------------------------------------
// The geometry the coverage kernels and the shell fill need of a particle,
// computed once per update by the particle's four lanes (in the update's
// kernel; at placement and in batches in one of its own) instead of by every
// CTA: the rotation and inverse squared radii, the centre the box was formed
// around with its integer and FP32 parts, and the box.
struct PGeom {
    Geo g;
    double X[3];
    double lo[3], hi[3];  // the box as box_of gives it, before finish_box
    int Xi[3];
    float Xf[3];
    Box box;
};

// Old geometry (the last coverage update's) and new geometry, and for the
// transition the new centre unwrapped next to the old one and the union of
// the two boxes.
struct PGeom2 {
    PGeom old_, now;
    int Xui[3];    // the new centre next to the old one: integer and fraction
    float Xuf[3];
    Box uni;
};

// ---- four lanes per particle ------------------------------------------------
// The Newton-Euler update and the geometry are chains of FP64 operations,
// and this part issues a warp's FP64 instruction over many cycles whether
// one lane or 32 are active: what counts is the number of warp
// instructions.  Four neighbouring lanes therefore share a particle: lane k
// = 0..2 carries axis k of every vector and lane l = 0..3 component l of
// the quaternion, so the three (four) like operations of a vector
// (quaternion) are one instruction.  Every operation and its order are those
// of the scalar formulas.  With one thread per particle the update and the
// geometry took 19 + 23 us for a single particle and 39 + 45 us for 25,033;
// as one kernel of quads 12 and 50 us.
__device__ __forceinline__ double quad(double v, int l) { return __shfl_sync(0xffffffffu, v, l, 4); }

// A vector given around axis k (its components k, k+1, k+2 cyclically) in
// the order 0, 1, 2.
__device__ __forceinline__ void order3(int k, double d, double n, double p, double o[3])
{
    o[0] = k == 0 ? d : (k == 1 ? p : n);
    o[1] = k == 0 ? n : (k == 1 ? d : p);
    o[2] = k == 0 ? p : (k == 1 ? n : d);
}

// Row and column k of the rotation matrix of q (rotmat's operations).
__device__ __forceinline__ void quad_rot(int k, const double q[4], double row[3], double col[3])
{
    const double w = q[0];
    const double a = k == 0 ? q[1] : (k == 1 ? q[2] : q[3]);
    const double b = k == 0 ? q[2] : (k == 1 ? q[3] : q[1]);
    const double c = k == 0 ? q[3] : (k == 1 ? q[1] : q[2]);
    const double d = s_(1.0, m_(2.0, a_(m_(b, b), m_(c, c))));
    const double ab = m_(a, b), ac = m_(a, c), wc = m_(w, c), wb = m_(w, b);
    order3(k, d, m_(2.0, s_(ab, wc)), m_(2.0, a_(ac, wb)), row);
    order3(k, d, m_(2.0, a_(ab, wc)), m_(2.0, s_(ac, wb)), col);
}

// Axis k of box_of for centre Xi + Xf and half-extent h, in FP32 (the box is
// a node wider than the ellipsoid on each side; the FP32 error is below 1e-3
// of a node up to half-extents of 1e4).
__device__ __forceinline__ void box_axis(double X, float h, double &fl, double &lo, double &hi)
{
    fl = floor(X);
    const float Xf = (float)(X - fl);
    lo = fl + (double)(floorf(Xf - h) - 1.f);
    hi = fl + (double)(ceilf(Xf + h) + 1.f);
    if (!(lo <= hi) || !(fabs(X) < 1e9) || !(h < 1e9f)) {
        lo = 1.0;
        hi = 0.0;
    }
}

// Whether the box whose axis k this lane holds is empty on any axis.
__device__ __forceinline__ bool quad_empty(double lo, double hi)
{
    const unsigned bad = __ballot_sync(0xffffffffu, !(lo <= hi));
    return ((bad >> (threadIdx.x & 28)) & 7u) != 0;
}

// finish_box for axis k (lanes 0..2 of a quad write their axis, lane 0 the
// count).
__device__ __forceinline__ void quad_box(const Lat &L, int k, bool wr, bool empty, double lo, double hi, Box &b)
{
    const double n = (double)ext_of(L, k);
    int fullp = 0;
    if (empty) {
        lo = 0.0;
        hi = -1.0;
    } else if (!periodic_dim(L, k)) {
        lo = fmax(lo, 0.0);
        hi = fmin(hi, n - 1.0);
    } else if (hi - lo + 1.0 > n) {
        lo = 0.0;
        hi = n - 1.0;
        fullp = 1;
    }
    const int ext = hi >= lo ? (int)(hi - lo + 1.0) : 0;
    const int count = __shfl_sync(0xffffffffu, ext, 0, 4) * __shfl_sync(0xffffffffu, ext, 1, 4) *
                      __shfl_sync(0xffffffffu, ext, 2, 4);
    if (wr) {
        b.lo[k] = hi >= lo ? (int)lo : 0;
        b.ext[k] = ext;
        b.full[k] = fullp;
        if (k == 0) b.count = count;
    }
}

// Geometry of particle p after an update: the last geometry becomes the old
// one and the new one is formed from this lane's X (axis k) and q.  first:
// placement, the old geometry is the new one.  Called by whole warps; act:
// the quad has a particle.
__device__ __forceinline__ void geom_quad(const Lat &L, const Parts &P, int p, bool act, bool first, double X,
                                          double Xold, const double q[4])
{
    const int lane = threadIdx.x & 3, k = lane == 3 ? 0 : lane;
    const bool wr = act && lane < 3;
    PGeom2 &G = reinterpret_cast<PGeom2 *>(P.geo)[p];
    constexpr int GW = (int)(sizeof(PGeom) / 8);
    static_assert(sizeof(PGeom) % 8 == 0, "PGeom is copied in 8-byte words");
    // old_ = now: all loads, then all stores (a load after a store that may
    // alias it waits: one round trip to memory instead of eleven)
    auto copy_now = [&] {
        const double *src = reinterpret_cast<const double *>(&G.now);
        double *dst = reinterpret_cast<double *>(&G.old_);
        double v[(GW + 3) / 4];
#pragma unroll
        for (int w = 0; w < (GW + 3) / 4; w++) v[w] = lane + 4 * w < GW ? src[lane + 4 * w] : 0.0;
        __syncwarp();
        if (act)
#pragma unroll
            for (int w = 0; w < (GW + 3) / 4; w++)
                if (lane + 4 * w < GW) dst[lane + 4 * w] = v[w];
        __syncwarp();
    };
    const double rp = P.rp[p], ro = P.ro[p], lo_was = G.now.lo[k], hi_was = G.now.hi[k];
    if (!first) copy_now();
    double row[3], col[3];
    quad_rot(k, q, row, col);
    const float r0 = (float)row[0], r1 = (float)row[1], r2 = (float)row[2], rpf = (float)rp, rof = (float)ro;
    // a little wide, for the FP32 rounding
    const float h = 1.00001f * sqrtf(rpf * rpf * r0 * r0 + rof * rof * (r1 * r1 + r2 * r2));
    double fl, flu, lo, hi;
    box_axis(X, h, fl, lo, hi);
    const bool empty = quad_empty(lo, hi);
    quad_box(L, k, wr, empty, lo, hi, G.now.box);
    if (wr) {
        for (int j = 0; j < 3; j++) {
            G.now.g.R[k][j] = row[j];
            G.now.g.R32[k][j] = (float)row[j];
        }
        G.now.X[k] = X;
        G.now.lo[k] = lo;
        G.now.hi[k] = hi;
        // X = Xi + Xf, Xi integral: the FP32 displacement (u - Xi) - Xf
        // carries no large cancellation (box_axis bounds |X| < 1e9); NaN,
        // which no row meets, for geometry without a box
        G.now.Xi[k] = empty ? 0 : (int)fl;
        G.now.Xf[k] = empty ? NAN : (float)(X - fl);
    }
    if (first && act && lane < 2) {  // the radii never change
        const double inv = __ddiv_rn(1.0, lane == 0 ? m_(rp, rp) : m_(ro, ro));
        (lane == 0 ? G.now.g.ip2 : G.now.g.io2) = inv;
        (lane == 0 ? G.now.g.ip2f : G.now.g.io2f) = (float)inv;
    }
    // the new centre next to the old one, and the union of the two boxes
    const double Xu = Xold + pair_disp(L, k, Xold, X);
    double lu, hu;
    box_axis(Xu, h, flu, lu, hu);
    const bool eu = quad_empty(lu, hu);
    double lo0 = first ? lo : lo_was, hi0 = first ? hi : hi_was;
    const bool e0 = quad_empty(lo0, hi0);
    if (e0) {
        lo0 = lu;
        hi0 = hu;
    } else if (!eu) {
        lo0 = fmin(lo0, lu);
        hi0 = fmax(hi0, hu);
    }
    quad_box(L, k, wr, e0 && eu, lo0, hi0, G.uni);
    if (wr) {
        G.Xui[k] = eu ? 0 : (int)flu;
        G.Xuf[k] = eu ? NAN : (float)(Xu - flu);
    }
    __syncwarp();
    if (first) copy_now();
}

// Geometry from the particle's state in memory.
__device__ __forceinline__ void geom_body(const Lat &L, const Parts &P, int p, bool act, bool first)
{
    const int lane = threadIdx.x & 3, k = lane == 3 ? 0 : lane;
    double q[4];
#pragma unroll
    for (int j = 0; j < 4; j++) q[j] = P.q[4 * p + j];
    geom_quad(L, P, p, act, first, P.X[3 * p + k], P.Xold[3 * p + k], q);
}

// The particle of this quad in a launch of four lanes per particle: quads
// past the end work on the last particle and write nothing.
__device__ __forceinline__ int quad_particle(int n, bool &act)
{
    const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 2;
    act = g < n;
    return act ? g : n - 1;
}

__global__ void k_geom(Lat L, Parts P)
{
    bool act;
    const int p = quad_particle(P.n, act);
    geom_body(L, P, p, act, true);
}

// Fixed-order block reduction of K doubles (PT threads).
template <int K>
__device__ void block_sum(double (&v)[K], double (*sh)[PT / 32])
{
#pragma unroll
    for (int k = 0; k < K; k++) {
        double a = v[k];
        for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
        if ((threadIdx.x & 31) == 0) sh[k][threadIdx.x >> 5] = a;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < K; k++) {
            double a = 0.0;
            for (int w = 0; w < PT / 32; w++) a += sh[k][w];
            v[k] = a;
        }
    }
}

__device__ __forceinline__ int nbr_node(const Lat &L, int x, int y, int z, int i)
{
    int xx = x + cx(i), yy = y + cy(i), zz = z + cz(i);
    xx = xx < 0 ? xx + L.nx : (xx >= L.nx ? xx - L.nx : xx);
    yy = yy < 0 ? yy + L.ny : (yy >= L.ny ? yy - L.ny : yy);
    if (L.walls) {
        if (zz < 0 || zz >= L.nz) return -1;
    } else {
        zz = zz < 0 ? zz + L.nz : (zz >= L.nz ? zz - L.nz : zz);
    }
    return xx + L.nx * (yy + L.ny * zz);
}

// ------------------------------------------------------------ links
// For every link between a solid node x of particle p and a fluid node
// y = x + c_i: the population leaving y towards x was reflected into slot i
// of y by the streaming kernel (f*_ī(y)); add C = 6 w_i ρ^c(y) u_surf·c_i
// with u_surf = V + ω × r_b at the link midpoint (Eq. 4), and give the
// particle F = (2 f*_ī + C) c_ī and r_b × F (Eq. 5).

template <class S>
__global__ void __launch_bounds__(PT) k_links(Lat L, Parts P, typename S::P *__restrict__ fnew,
                                              const float *__restrict__ rho,
                                              const uint8_t *__restrict__ type,
                                              const uint32_t *__restrict__ owner)
{
    const int p = blockIdx.x;
    __shared__ Box box;
    __shared__ double sX[3];
    __shared__ float sV[3], sW[3];
    __shared__ double red[6][PT / 32];
    if (threadIdx.x == 0) {
        double R[3][3];
        rotmat(P.q + 4 * p, R);
        double lo[3], hi[3];
        box_of(L, P.X + 3 * p, R, P.rp[p], P.ro[p], lo, hi);
        finish_box(L, lo, hi, box);
        for (int k = 0; k < 3; k++) {
            sX[k] = P.X[3 * p + k];
            sV[k] = (float)P.V[3 * p + k];
            sW[k] = (float)P.W[3 * p + k];
        }
    }
    __syncthreads();
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int k = threadIdx.x; k < box.count; k += PT) {
        int x, y, z, u[3];
        box_node(L, box, k, u, x, y, z);
        int n = x + L.nx * (y + L.ny * z);
        if (!idx_ok(L, n, L.N, 2)) continue;
        if (owner[n] != (uint32_t)p) continue;
        float dn[3] = {(float)box_disp(L, box, 0, u[0], x, sX[0]), (float)box_disp(L, box, 1, u[1], y, sX[1]),
                       (float)box_disp(L, box, 2, u[2], z, sX[2])};
        float aF[3] = {0.f, 0.f, 0.f}, aT[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 1; i < Q; i++) {
            int m = nbr_node(L, x, y, z, i);
            if (m < 0 || !idx_ok(L, m, L.N, 3) || type[m] != FLUID) continue;
            float rb[3] = {dn[0] + 0.5f * cx(i), dn[1] + 0.5f * cy(i), dn[2] + 0.5f * cz(i)};
            float us[3] = {sV[0] + sW[1] * rb[2] - sW[2] * rb[1], sV[1] + sW[2] * rb[0] - sW[0] * rb[2],
                           sV[2] + sW[0] * rb[1] - sW[1] * rb[0]};
            float uc = us[0] * cx(i) + us[1] * cy(i) + us[2] * cz(i);
            const float2 fr2 = ld2f<S>(fnew, L, i, m);
            float2 out2;
#pragma unroll
            for (int c = 0; c < 2; c++) {
                float fr = c ? fr2.y : fr2.x;
                const float2 rm = ld_pair(rho, m);
                float C = 6.f * wgt(i) * (c ? rm.y : rm.x) * uc;
                (c ? out2.y : out2.x) = fr + C;
                float a = -(2.f * fr + C);  // F = (2 f* + C) c_ī, c_ī = -c_i
                float F[3] = {a * cx(i), a * cy(i), a * cz(i)};
                aF[0] += F[0];
                aF[1] += F[1];
                aF[2] += F[2];
                aT[0] += rb[1] * F[2] - rb[2] * F[1];
                aT[1] += rb[2] * F[0] - rb[0] * F[2];
                aT[2] += rb[0] * F[1] - rb[1] * F[0];
            }
            st2f<S>(fnew, L, i, m, out2);
        }
        for (int k2 = 0; k2 < 3; k2++) {
            acc[k2] += (double)aF[k2];
            acc[3 + k2] += (double)aT[k2];
        }
    }
    block_sum<6>(acc, red);
    if (threadIdx.x == 0) {
        for (int k = 0; k < 3; k++) {
            P.Flink[3 * p + k] = acc[k];
            P.Tlink[3 * p + k] = acc[3 + k];
        }
    }
}

// ------------------------------------------------------------ link nodes
// For every particle node s of the step's link list and every direction j
// whose neighbour y = s + c_j is a fluid node (the link runs from y along
// c_i = -c_j into s): the fluid kernel reflected the post-collision
// f*_i(y) into slot j of y; add C = -6 w_i ρ^c(y) (u_surf·c_i) with u_surf =
// V + ω × r_b at the link midpoint r_b = s + c_j/2 - X (Eq. 4), and give
// the particle (2 f*_i + C) c_i and r_b × that (Eq. 5).  ρ^c(y) is the
// density kernel's, this step.  Force and torque are summed in 64-bit fixed
// point (2^-40 units): each FP32 link term is rounded once to an integer and
// integer additions are exact, so the totals do not depend on the order of
// the links.

// FP32 value to 64-bit fixed point in units of 2^-40 (two's complement in an
// unsigned word, so that wrap-around addition is exact); |v| is clamped to
// 2^22, far beyond any link term.
__device__ __forceinline__ unsigned long long to_fixed(float v)
{
    v = fminf(fmaxf(v, -4194304.f), 4194304.f);
    return (unsigned long long)__float2ll_rn(v * 1099511627776.f);
}

// Sum over the lanes of grp of 64-bit two's complement words (exact, by
// 16/16/32-bit limbs).  Called by the lanes of grp.
__device__ __forceinline__ unsigned long long reduce_fix(unsigned grp, unsigned long long v)
{
    const unsigned lo = (unsigned)v, hi = (unsigned)(v >> 32);
    const unsigned s0 = __reduce_add_sync(grp, lo & 0xffffu);
    const unsigned s1 = __reduce_add_sync(grp, lo >> 16);
    const unsigned s2 = __reduce_add_sync(grp, hi);
    return ((unsigned long long)s2 << 32) + ((unsigned long long)s1 << 16) + (unsigned long long)s0;
}

// Add this lane's sums v[6] for particle p (nothing for p < 0) to the
// particle's totals: lanes of the warp with the same particle are combined
// first and one lane per particle does the atomics.  Called by all 32 lanes.
__device__ __forceinline__ void warp_add_fix(int p, const unsigned long long v[6], unsigned long long *fix)
{
    const unsigned grp = __match_any_sync(0xffffffffu, p);
    const bool leader = (int)(threadIdx.x & 31) == __ffs(grp) - 1;
    unsigned long long tot[6];
#pragma unroll
    for (int k = 0; k < 6; k++) tot[k] = reduce_fix(grp, v[k]);
    if (p < 0 || !leader) return;
#pragma unroll
    for (int k = 0; k < 6; k++) atomicAdd(&fix[6 * p + k], tot[k]);
}

// c_j for a direction j known only at run time (a lane's link): 2-bit
// fields c + 1 of the components, j = 0..18.
constexpr unsigned long long pack_dir(int axis)
{
    unsigned long long v = 0;
    for (int j = 0; j < Q; j++)
        v |= (unsigned long long)((axis == 0 ? cx(j) : (axis == 1 ? cy(j) : cz(j))) + 1) << (2 * j);
    return v;
}
constexpr unsigned long long CXP = pack_dir(0), CYP = pack_dir(1), CZP = pack_dir(2);
__device__ __forceinline__ int cdir(unsigned long long pack, int j) { return (int)((pack >> (2 * j)) & 3ull) - 1; }

// Per warp of the link kernels: the links of its list entries in
// direction-major order, (entry lane, direction) per link.
struct LinkWarp {
    uint16_t desc[32 * (Q - 1)];
    unsigned bal[Q];
    int pre[Q];
};

// The links of up to 32 list entries (e = (node, mask of fluid neighbours)
// per lane; mask 0 for a lane without an entry).  The entries' links are
// laid out direction by direction, so that lanes taking neighbouring links
// touch the same slot array at neighbouring nodes, and handed out 64 at a
// time: every lane carries two links per round, and the loads of a round are
// all in flight together.  What belongs to the entry (its place, the arm from
// the particle) is formed once by the entry's lane.  Where all entries are of
// one particle (most warps), each lane adds up its own terms over the rounds
// and the warp combines them once.  Called by all 32 lanes.
template <class S>
__device__ __forceinline__ void link_entries(const Lat &L, uint2 e, const float *__restrict__ rho,
                                             const uint32_t *__restrict__ owner, const float4 *__restrict__ X32,
                                             const float4 *__restrict__ K32, unsigned long long *fix,
                                             typename S::P *fout, LinkWarp &w)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    uint32_t fm = e.y;
    const int s = (int)e.x;
    int p = -1;
    if (fm) {
        p = (int)owner[s];
        if ((unsigned)p >= (unsigned)L.np) {  // a particle node is always owned
            idx_ok(L, p, L.np, 20);
            p = -1;
            fm = 0;
        }
    }
    const unsigned have = __ballot_sync(full, fm != 0);
    if (!have) return;
    // direction j's links: the lanes of ballot j, after those of 1 .. j-1
    int total = 0;
#pragma unroll
    for (int j = 1; j < Q; j++) {
        const unsigned b = __ballot_sync(full, (fm >> j) & 1u);
        if (lane == j) {
            w.bal[j] = b;
            w.pre[j] = total;
        }
        total += __popc(b);
    }
    __syncwarp();
    for (uint32_t m = fm; m; m &= m - 1) {
        const int j = __ffs(m) - 1;
        const int k = w.pre[j] + __popc(w.bal[j] & ((1u << lane) - 1u));
        w.desc[k] = (uint16_t)(lane | (j << 5));
    }
    const int p0 = __shfl_sync(full, p, __ffs(have) - 1);
    const bool uniform = __all_sync(full, !fm || p == p0);
    // the entry's node: s - X, nearest image, and the lattice faces it lies on
    float dx = 0.f, dy = 0.f, dz = 0.f;
    unsigned face = 0;
    if (fm) {
        const float4 X = X32[p];
        const int x = s % L.nx, t = s / L.nx, y = t % L.ny, z = t / L.ny;
        dx = (float)x - X.x;
        dy = (float)y - X.y;
        dz = (float)z - X.z;
        if (dx > 0.5f * L.nx) dx -= L.nx;
        if (dx < -0.5f * L.nx) dx += L.nx;
        if (dy > 0.5f * L.ny) dy -= L.ny;
        if (dy < -0.5f * L.ny) dy += L.ny;
        if (!L.walls) {
            if (dz > 0.5f * L.nz) dz -= L.nz;
            if (dz < -0.5f * L.nz) dz += L.nz;
        }
        face = (x == L.nx - 1 ? 1u : 0u) | (x == 0 ? 2u : 0u) | (y == L.ny - 1 ? 4u : 0u) | (y == 0 ? 8u : 0u) |
               (z == L.nz - 1 ? 16u : 0u) | (z == 0 ? 32u : 0u);
    }
    float4 V = K32[2 * p0], W = K32[2 * p0 + 1];
    unsigned long long sum[6] = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
    __syncwarp();
    // two links a lane per round: the loads of both are in flight together
    constexpr int U = 2;
    for (int k0 = 0; k0 < total; k0 += 32 * U) {
        int j[U], pn[U];
        float rx[U], ry[U], rz[U];
        typename S::P *q[U], raw[U];
        float2 rho_y[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int k = k0 + 32 * u + lane;
            const int d = k < total ? w.desc[k] : 0;
            const int src = d & 31;
            j[u] = d >> 5;  // 0: no link
            const int sn = __shfl_sync(full, s, src);
            pn[u] = __shfl_sync(full, p, src);
            const float ex = __shfl_sync(full, dx, src), ey = __shfl_sync(full, dy, src),
                        ez = __shfl_sync(full, dz, src);
            const unsigned fc = __shfl_sync(full, face, src);
            if (!j[u]) continue;
            const int cxj = cdir(CXP, j[u]), cyj = cdir(CYP, j[u]), czj = cdir(CZP, j[u]);
            // the fluid node s + c_j, around the periodic faces
            int yf = sn + cxj + L.nx * (cyj + L.ny * czj);
            if (cxj > 0 && (fc & 1u)) yf -= L.nx;
            if (cxj < 0 && (fc & 2u)) yf += L.nx;
            if (cyj > 0 && (fc & 4u)) yf -= L.nx * L.ny;
            if (cyj < 0 && (fc & 8u)) yf += L.nx * L.ny;
            if (czj > 0 && (fc & 16u)) yf -= L.N;
            if (czj < 0 && (fc & 32u)) yf += L.N;
            rx[u] = ex + 0.5f * (float)cxj;
            ry[u] = ey + 0.5f * (float)cyj;
            rz[u] = ez + 0.5f * (float)czj;
            // both components of slot j of the fluid node: one pair access
            q[u] = fout + pidx(L, j[u], yf);
            raw[u] = *q[u];
            rho_y[u] = __ldg(reinterpret_cast<const float2 *>(rho) + yf);
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            unsigned long long acc[6] = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
            if (j[u]) {
                if (!uniform) {
                    V = K32[2 * pn[u]];
                    W = K32[2 * pn[u] + 1];
                }
                const float fcx = (float)cdir(CXP, j[u]), fcy = (float)cdir(CYP, j[u]), fcz = (float)cdir(CZP, j[u]);
                // surface velocity V + ω × r_b at the link midpoint
                const float usx = __fsub_rn(__fmaf_rn(W.y, rz[u], V.x), __fmul_rn(W.z, ry[u]));
                const float usy = __fsub_rn(__fmaf_rn(W.z, rx[u], V.y), __fmul_rn(W.x, rz[u]));
                const float usz = __fsub_rn(__fmaf_rn(W.x, ry[u], V.z), __fmul_rn(W.y, rx[u]));
                // u_surf·c_i with c_i = -c_j
                const float uci = -__fadd_rn(__fadd_rn(usx * fcx, usy * fcy), usz * fcz);
                const float w6 = j[u] < 7 ? -6.f / 18.f : -6.f / 36.f;
                const float2 base = make_float2(L.base[0][j[u]], L.base[1][j[u]]), st = S::raw2(raw[u]);
                const float2 fs = make_float2(base.x + st.x, base.y + st.y);
                const float C0 = __fmul_rn(__fmul_rn(w6, rho_y[u].x), uci);
                const float C1 = __fmul_rn(__fmul_rn(w6, rho_y[u].y), uci);
                *q[u] = S::enc2(make_float2(__fadd_rn(fs.x, C0) - base.x, __fadd_rn(fs.y, C1) - base.y));
                float a = 0.f;
                a = __fadd_rn(a, __fmaf_rn(2.f, fs.x, C0));
                a = __fadd_rn(a, __fmaf_rn(2.f, fs.y, C1));
                // F = a c_i = -a c_j
                const float Fx = -a * fcx, Fy = -a * fcy, Fz = -a * fcz;
                acc[0] = to_fixed(Fx);
                acc[1] = to_fixed(Fy);
                acc[2] = to_fixed(Fz);
                acc[3] = to_fixed(__fsub_rn(__fmul_rn(ry[u], Fz), __fmul_rn(rz[u], Fy)));
                acc[4] = to_fixed(__fsub_rn(__fmul_rn(rz[u], Fx), __fmul_rn(rx[u], Fz)));
                acc[5] = to_fixed(__fsub_rn(__fmul_rn(rx[u], Fy), __fmul_rn(ry[u], Fx)));
            }
            if (uniform) {
#pragma unroll
                for (int c = 0; c < 6; c++) sum[c] += acc[c];
            } else {
                warp_add_fix(j[u] ? pn[u] : -1, acc, fix);
            }
        }
    }
    if (uniform) {
        unsigned long long t = 0ull;
#pragma unroll
        for (int c = 0; c < 6; c++) {
            const unsigned long long v = reduce_fix(full, sum[c]);
            if (lane == c) t = v;
        }
        if (lane < 6) atomicAdd(&fix[6 * p0 + lane], t);
    }
    __syncwarp();
}

// A warp takes group entries of the list at a time: 32, or 8 where the list
// is short (lists of small tiles, whose groups of 8 are of one particle), so
// that the links of one particle spread over many warps.  One ellipsoid (6,
// 3): 18.6 us with 32 and a reduction per round, 8.1 with 8; 40 dragged
// ellipsoids: 86 and 8.5 us.
template <class S>
__device__ __forceinline__ void link_list(const Lat &L, const LinkList &ll, const float *rho, const uint32_t *owner,
                                          const Parts &P, typename S::P *fout, int group, LinkWarp &w)
{
    const int count = min(*ll.count, ll.cap), lane = threadIdx.x & 31;
    const int nw = gridDim.x * (blockDim.x >> 5), w0 = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    for (int e0 = w0 * group; e0 < count; e0 += nw * group) {
        const bool valid = lane < group && e0 + lane < count;
        link_entries<S>(L, valid ? ll.ent[e0 + lane] : make_uint2(0u, 0u), rho, owner, P.X32, P.K32, P.fix, fout, w);
    }
}

template <class S>
__global__ void __launch_bounds__(256) k_link(Lat L, LinkList ll, const float *rho, const uint32_t *owner, Parts P,
                                              typename S::P *fout, int group)
{
    __shared__ LinkWarp w[256 / 32];
    link_list<S>(L, ll, rho, owner, P, fout, group, w[threadIdx.x >> 5]);
}

// Batched: blockIdx.y is the box; LINK_BATCH_CTAS CTAs per box.  With 4, 8, 16
// and 32 a step of 7 boxes of one sphere (48 x 48 x 40 f32) takes 135, 131, 131
// and 131 us, of 64 boxes of 32^3 307, 306, 311 and 314; only boxes of many
// particles would gain from more (four of 96^3 with 100 each: 558, 461, 409, 394).
constexpr int LINK_BATCH_CTAS = 8;

template <class S>
__global__ void __launch_bounds__(256) k_link_batch(BatchIndex B, int group)
{
    const int b = blockIdx.y;
    const BoxDev &bx = B.box[b];
    if (!bx.links.ent || bx.P.n == 0) return;
    const int cur = B.par[2 * b], ocur = B.par[2 * b + 1];
    __shared__ LinkWarp w[256 / 32];
    link_list<S>(bx.L, bx.links, bx.rho, bx.owner[ocur], bx.P, (typename S::P *)bx.f[1 - cur],
                 group, w[threadIdx.x >> 5]);
}

// --------------------------------------------------------- pair forces

__device__ __forceinline__ double dot3(const double *a, const double *b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }
__device__ __forceinline__ void cross3(const double *a, const double *b, double *o)
{
    o[0] = a[1] * b[2] - a[2] * b[1];
    o[1] = a[2] * b[0] - a[0] * b[2];
    o[2] = a[0] * b[1] - a[1] * b[0];
}

// Anisotropic Hertz interaction (Eq. 6-8): φ = ε(ô_i,ô_j) (1 - r/σ)^{5/2}
// for r < σ with ε = ε̄ / sqrt(1 - χ^2 (ô_i·ô_j)^2), ε̄ = K_H σ̄^{5/2},
// σ̄ = 2 r_perp, and the Berne–Pechukas σ(ô_i, ô_j, r̂).  Returns σ; fills
// the force on j and the torques on i and j (minus the analytic gradients).
__device__ double hertz_bp(double K, double rp, double ro, const double r[3], const double oi[3],
                           const double oj[3], double fj[3], double ti[3], double tj[3])
{
    for (int k = 0; k < 3; k++) fj[k] = ti[k] = tj[k] = 0.0;
    double chi = (rp * rp - ro * ro) / (rp * rp + ro * ro);
    double sbar = 2.0 * ro;
    double rl = sqrt(dot3(r, r));
    if (!(rl > 0)) return sbar;
    double rh[3] = {r[0] / rl, r[1] / rl, r[2] / rl};
    double a = dot3(rh, oi), b = dot3(rh, oj), c = dot3(oi, oj);
    double ep = 1.0 + chi * c, em = 1.0 - chi * c;
    double S = (a + b) * (a + b) / ep + (a - b) * (a - b) / em;
    double D = 1.0 - 0.5 * chi * S;
    double sigma = sbar / sqrt(D);
    double s = rl / sigma;
    if (s >= 1.0) return sigma;
    double ebar = K * sbar * sbar * sqrt(sbar);
    double Ed = 1.0 - chi * chi * c * c;
    double eps = ebar / sqrt(Ed);
    double om = 1.0 - s;
    double phit = om * om * sqrt(om);
    double dphit = -2.5 * om * sqrt(om);
    double dsig_dS = 0.25 * chi * sbar / (D * sqrt(D));
    double dS_da = 2.0 * (a + b) / ep + 2.0 * (a - b) / em;
    double dS_db = 2.0 * (a + b) / ep - 2.0 * (a - b) / em;
    double dS_dc = -chi * (a + b) * (a + b) / (ep * ep) + chi * (a - b) * (a - b) / (em * em);
    double deps_dc = ebar * chi * chi * c / (Ed * sqrt(Ed));
    double gs = eps * dphit * (-rl / (sigma * sigma)) * dsig_dS;
    double dphi_drl = eps * dphit / sigma;
    double gi[3], gj[3];
    for (int k = 0; k < 3; k++) {
        double grad = dphi_drl * rh[k] + gs * (dS_da * (oi[k] - a * rh[k]) / rl + dS_db * (oj[k] - b * rh[k]) / rl);
        fj[k] = -grad;
        gi[k] = phit * deps_dc * oj[k] + gs * (dS_da * rh[k] + dS_dc * oj[k]);
        gj[k] = phit * deps_dc * oi[k] + gs * (dS_db * rh[k] + dS_dc * oi[k]);
    }
    double u[3];
    cross3(oi, gi, u);
    for (int k = 0; k < 3; k++) ti[k] = -u[k];
    cross3(oj, gj, u);
    for (int k = 0; k < 3; k++) tj[k] = -u[k];
    return sigma;
}

// FP32 prefilter of a pair (centres and reaches in xyzw): nearest-image
// distance within reach_i + reach_j + extra.  Pairs it drops contribute
// exactly zero, so it decides nothing but the work done.
__device__ __forceinline__ bool near_pair(float4 me, float4 o, const float nl[3], const float inv[3], bool per_z,
                                          float extra)
{
    float dx = o.x - me.x, dy = o.y - me.y, dz = o.z - me.z;
    dx = __fmaf_rn(-nl[0], rintf(dx * inv[0]), dx);
    dy = __fmaf_rn(-nl[1], rintf(dy * inv[1]), dy);
    if (per_z) dz = __fmaf_rn(-nl[2], rintf(dz * inv[2]), dz);
    const float reach = me.w + o.w + extra;
    return __fmaf_rn(dx, dx, __fmaf_rn(dy, dy, dz * dz)) <= reach * reach;
}

// ---- eight lanes per particle ------------------------------------------------
// A particle's pair terms are long FP64 chains (divisions, square roots)
// and few (about 4 partners pass the prefilter in a dense emulsion), and a
// warp instruction costs the same for one active lane as for 32: eight lanes
// share a particle, test eight partners at a time and evaluate up to eight
// terms at once.  The terms are then added one after the other in the order
// of the partners' indices, one component per lane, which gives the sums of
// a plain loop bit for bit.  525
// particles (150 x 141 x 133, 10 %): 81 us with one lane per particle, 34
// now; 25,033: 127 us with one lane, 105 now.
//
// Up to PAIRS_SCAN_MAX particles the loop over all partners replaces the
// cell lists: at 10 % volume fraction it takes 15 us for 60 particles, 20 for
// 130 and 26 for 250, against 31 + 3 for 300 with the lists and a memset.
constexpr int PAIRS_SCAN_MAX = 256;
constexpr int PG = 8;                  // lanes per particle
constexpr int PAIR_GROUPS = 128 / PG;  // particles per CTA
constexpr int CAND_MAX = 96;           // candidates held per particle; beyond that a full scan

struct PairGroup {
    int cand[CAND_MAX];    // partners waiting for evaluation
    int sorted[CAND_MAX];
    double term[PG][9];    // Hertz force and torque, lubrication force
    int count;
};

// The Hertz and lubrication (Eq. 9 with 2R -> σ, R^2 -> (σ/2)^2, only for
// gaps 0 < r - σ < Δc, opposing the normal approach) contribution of
// partner j to particle i.  The lubrication coefficient K (1/h - 1/Δc) is
// capped at the pair's reduced mass M_i M_j / (M_i + M_j): at the cap one
// update (Δt = 1) removes the normal approach speed; above it the explicit
// update would reverse the approach with growing speed as h -> 0.  A pair
// is evaluated in FP64 only when the FP32 distance of the centres is within
// reach_i + reach_j + Δc (+0.05 for the FP32 error).
// t gets the Hertz force and torque and, with lub set, the lubrication force.
__device__ void pair_parts(const Lat &L, const Parts &P, const Pair &pp, int i, int j, const double oi[3],
                           double *t, bool &lub)
{
    int a = i < j ? i : j, b = i < j ? j : i;  // the pair is taken as (a, b), a < b
    double r[3];
    for (int k = 0; k < 3; k++) r[k] = pair_disp(L, k, P.X[3 * a + k], P.X[3 * b + k]);
    double Rj[3][3];
    rotmat(P.q + 4 * j, Rj);
    double oj[3] = {Rj[0][0], Rj[1][0], Rj[2][0]};
    const double *oa = i < j ? oi : oj, *ob = i < j ? oj : oi;
    double rp = 0.5 * (P.rp[a] + P.rp[b]), ro = 0.5 * (P.ro[a] + P.ro[b]);
    double fb[3], ta[3], tb[3];
    double sigma = hertz_bp(pp.k_hertz, rp, ro, r, oa, ob, fb, ta, tb);
    for (int k = 0; k < 3; k++) {
        t[k] = i == b ? fb[k] : -fb[k];
        t[3 + k] = i == a ? ta[k] : tb[k];
    }
    double rl = sqrt(dot3(r, r));
    double h = rl - sigma;
    lub = pp.lub_cut > 0 && h > 0 && h < pp.lub_cut;
    if (lub) {
        double rh[3] = {r[0] / rl, r[1] / rl, r[2] / rl};
        double du[3] = {P.V[3 * a] - P.V[3 * b], P.V[3 * a + 1] - P.V[3 * b + 1], P.V[3 * a + 2] - P.V[3 * b + 2]};
        double K = 3.0 * M_PI * pp.mu * sigma * sigma / 8.0;
        double gam = K * (1.0 / h - 1.0 / pp.lub_cut);
        const double mred = P.M[a] * P.M[b] / (P.M[a] + P.M[b]);
        if (gam > mred) gam = mred;
        double s = gam * dot3(rh, du);
        for (int k = 0; k < 3; k++) t[6 + k] = i == a ? -s * rh[k] : s * rh[k];
    }
}

// Evaluate the n <= 8 partners list[0..n) and add their terms in list order
// to acc, which is component l of (force, torque) on lane l < 6.  Called by
// the eight lanes of a group (mask m).
__device__ __forceinline__ void pair_flush(const Lat &L, const Parts &P, const Pair &pp, int i, const int *list, int n,
                                           const double oi[3], PairGroup &g, unsigned m, double &acc)
{
    const int l = threadIdx.x & (PG - 1);
    bool lub = false;
    if (l < n) pair_parts(L, P, pp, i, list[l], oi, g.term[l], lub);
    const unsigned bl = __ballot_sync(m, lub) >> (threadIdx.x & 24);
    __syncwarp(m);
    if (l < 6)
        for (int k = 0; k < n; k++) {
            acc += g.term[k][l];
            if (l < 3 && ((bl >> k) & 1u)) acc += g.term[k][6 + l];
        }
    __syncwarp(m);
}

// Pair sums of particle i over all partners in index order: eight at a
// time through the prefilter, those that pass queued and evaluated eight at
// a time.  Returns component l of (force, torque) on lane l < 6.
__device__ __forceinline__ double pairs_scan(const Lat &L, const Parts &P, const Pair &pp, int i, float4 me,
                                             const double oi[3], PairGroup &g, unsigned m)
{
    const int l = threadIdx.x & (PG - 1);
    const float nl[3] = {(float)L.nx, (float)L.ny, (float)L.nz};
    const float inv[3] = {1.f / nl[0], 1.f / nl[1], 1.f / nl[2]};
    const float extra = (float)pp.lub_cut + 0.05f;
    double acc = 0.0;
    int n = 0;
    for (int j0 = 0; j0 < P.n; j0 += PG) {
        const int j = j0 + l;
        const bool near = j < P.n && j != i && near_pair(me, P.X32[j], nl, inv, !L.walls, extra);
        const unsigned b = (__ballot_sync(m, near) >> (threadIdx.x & 24)) & 0xFFu;
        if (near) g.cand[n + __popc(b & ((1u << l) - 1u))] = j;
        n += __popc(b);
        __syncwarp(m);
        if (n >= PG) {
            pair_flush(L, P, pp, i, g.cand, PG, oi, g, m, acc);
            const int v = l < n - PG ? g.cand[PG + l] : 0;
            __syncwarp(m);
            if (l < n - PG) g.cand[l] = v;
            n -= PG;
            __syncwarp(m);
        }
    }
    if (n > 0) pair_flush(L, P, pp, i, g.cand, n, oi, g, m, acc);
    return acc;
}

__device__ __forceinline__ void pairs_store(const Parts &P, int i, double acc)
{
    const int l = threadIdx.x & (PG - 1);
    if (l < 6) P.ppart[(size_t)l * P.n + i] = acc;
}

// ---------------------------------------------------------------- cells
// Per step every particle enters the list of its cell (head[c], then next[i];
// the order does not matter).  A particle's lanes then walk the lists of the
// 27 cells around its own (each cell once when an axis has fewer than 3
// cells), one cell a lane, keep the partners the FP32 prefilter passes, sort
// them, and sum the pair terms in increasing partner index: the same terms in
// the same order as a loop over all partners.  Lattices of at most
// PAIRS_SCAN_MAX particles take that loop instead.  A compact list (count,
// prefix over the cells, fill) took three kernels, 45 us with 38 in the prefix
// at 24,389 cells, and 167 us for a walk one cell after the other; the lists
// take 4 and 105 (25,033 particles; 2,344: 12 + 34 -> 4 + 24).

__device__ __forceinline__ int cell_axis(float x, float n, float inv, int nc, bool periodic)
{
    if (periodic) x -= n * floorf(x / n);
    int c = (int)(x * inv);
    return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
}

__global__ void k_cell_lists(Lat L, Parts P, Cells C)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.n) return;
    const float4 x = P.X32[i];
    const int cx_ = cell_axis(x.x, (float)L.nx, C.inv[0], C.n[0], true);
    const int cy_ = cell_axis(x.y, (float)L.ny, C.inv[1], C.n[1], true);
    const int cz_ = cell_axis(x.z, (float)L.nz, C.inv[2], C.n[2], !L.walls);
    const int c = cx_ + C.n[0] * (cy_ + C.n[1] * cz_);
    C.cid[i] = c;
    C.next[i] = atomicExch(&C.head[c], i);
}

__device__ __forceinline__ double pairs_cells(const Lat &L, const Parts &P, const Pair &pp, const Cells &C, int i,
                                              float4 me, const double oi[3], PairGroup &g, unsigned m)
{
    const int l = threadIdx.x & (PG - 1);
    const float nl[3] = {(float)L.nx, (float)L.ny, (float)L.nz};
    const float inv[3] = {1.f / nl[0], 1.f / nl[1], 1.f / nl[2]};
    const bool per_z = !L.walls;
    const float extra = (float)pp.lub_cut + 0.05f;
    const int c0 = C.cid[i];
    const int ci[3] = {c0 % C.n[0], (c0 / C.n[0]) % C.n[1], c0 / (C.n[0] * C.n[1])};
    int lo[3], ext[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        lo[k] = C.n[k] < 3 ? 0 : ci[k] - 1;  // every cell of a short axis once
        ext[k] = C.n[k] < 3 ? C.n[k] : 3;
    }
    if (l == 0) g.count = 0;
    __syncwarp(m);
    // up to four lists a lane, walked side by side so that their loads are in
    // flight together
    constexpr int NQ = (27 + PG - 1) / PG;
    int jq[NQ];
#pragma unroll
    for (int u = 0; u < NQ; u++) {
        const int q = l + PG * u;
        int x = lo[0] + q % ext[0], y = lo[1] + q / ext[0] % ext[1], z = lo[2] + q / (ext[0] * ext[1]);
        x = x < 0 ? x + C.n[0] : (x >= C.n[0] ? x - C.n[0] : x);
        y = y < 0 ? y + C.n[1] : (y >= C.n[1] ? y - C.n[1] : y);
        if (per_z) z = z < 0 ? z + C.n[2] : (z >= C.n[2] ? z - C.n[2] : z);
        const bool in = q < ext[0] * ext[1] * ext[2] && z >= 0 && z < C.n[2];
        jq[u] = in ? C.head[x + C.n[0] * (y + C.n[1] * z)] : -1;
    }
    for (;;) {
        float4 o[NQ];
        int nx[NQ];
        bool any = false;
#pragma unroll
        for (int u = 0; u < NQ; u++) {
            const int j = max(jq[u], 0);
            any = any || jq[u] >= 0;
            o[u] = P.X32[j];
            nx[u] = C.next[j];
        }
        if (!any) break;
#pragma unroll
        for (int u = 0; u < NQ; u++) {
            if (jq[u] < 0) continue;
            if (jq[u] != i && near_pair(me, o[u], nl, inv, per_z, extra)) {
                const int at = atomicAdd(&g.count, 1);
                if (at < CAND_MAX) g.cand[at] = jq[u];
            }
            jq[u] = nx[u];
        }
    }
    __syncwarp(m);
    const int nc = g.count;
    if (nc > CAND_MAX) return pairs_scan(L, P, pp, i, me, oi, g, m);  // very dense
    __syncwarp(m);
    for (int a = l; a < nc; a += PG) {  // by increasing partner index (all distinct)
        int r = 0;
        for (int b = 0; b < nc; b++) r += g.cand[b] < g.cand[a];
        g.sorted[r] = g.cand[a];
    }
    __syncwarp(m);
    double acc = 0.0;
    for (int a = 0; a < nc; a += PG) pair_flush(L, P, pp, i, g.sorted + a, min(PG, nc - a), oi, g, m, acc);
    return acc;
}

// Pair sums of particle i by its group of eight lanes; cells null: over all
// partners.
__device__ __forceinline__ void pairs_body(const Lat &L, const Parts &P, const Pair &pp, const Cells *C, int i,
                                           PairGroup &g)
{
    const unsigned m = 0xFFu << (threadIdx.x & 24);
    const float4 me = P.X32[i];
    double Ri[3][3];
    rotmat(P.q + 4 * i, Ri);
    const double oi[3] = {Ri[0][0], Ri[1][0], Ri[2][0]};
    const double acc = C ? pairs_cells(L, P, pp, *C, i, me, oi, g, m) : pairs_scan(L, P, pp, i, me, oi, g, m);
    pairs_store(P, i, acc);
}

template <bool CELLS>
__global__ void __launch_bounds__(128) k_pairs(Lat L, Parts P, Pair pp, Cells C)
{
    __shared__ PairGroup g[PAIR_GROUPS];
    const int i = (blockIdx.x * 128 + threadIdx.x) / PG;
    if (i >= P.n) return;  // whole groups
    pairs_body(L, P, pp, CELLS ? &C : nullptr, i, g[threadIdx.x / PG]);
}

// ------------------------------------------------------------ integrate
// Leapfrog translation (V += F/M, X += V), explicit Euler of the body-frame
// Euler equations, q <- normalise(q ⊗ exp(ω_body/2)).  The total force is
// momentum exchange + pair forces + the fill/empty momentum of the last
// coverage update.

// One update of particle p by its quad; X and q get the new centre (axis k)
// and orientation, Xold the old centre.  The quads of a warp may differ in
// mode (boxes of a batch), so all take part in every exchange between lanes.
__device__ __forceinline__ void integrate_quad(const Lat &L, const Parts &P, int mode, int p, bool act, double &X,
                                               double &Xold, double q[4])
{
    const int lane = threadIdx.x & 3, k = lane == 3 ? 0 : lane;
    const bool wr = act && lane < 3;
    const int e = 3 * p + k;
    // link sums: FP64 from the two-pass link kernel, or 2^-40 fixed point
    // from the fused kernel (the other one is zero)
    const double fl = P.Flink[e] + (double)(long long)P.fix[6 * p + k] * FIXED_UNIT;
    const double tl = P.Tlink[e] + (double)(long long)P.fix[6 * p + 3 + k] * FIXED_UNIT;
    double fp = 0.0, tp = 0.0;
    for (int sp = 0; sp < P.nsplit; sp++) {
        fp += P.ppart[((size_t)sp * 6 + k) * P.n + p];
        tp += P.ppart[((size_t)sp * 6 + 3 + k) * P.n + p];
    }
    const double F = fl + fp + P.Fpend[e], T = tl + tp + P.Tpend[e];
    Xold = X = P.X[e];
    double V = P.V[e], W = P.W[e];
    const double qc = P.q[4 * p + lane];
    __syncwarp();  // every lane has read before any writes
    if (wr) {
        P.fix[6 * p + k] = 0ull;
        P.fix[6 * p + 3 + k] = 0ull;
        P.Fpair[e] = fp;
        P.Tpair[e] = tp;
        P.F[e] = F;
        P.T[e] = T;
        P.Fpend[e] = 0.0;
        P.Tpend[e] = 0.0;
        P.Flink[e] = 0.0;
        P.Tlink[e] = 0.0;
        P.Xold[e] = X;
    }
#pragma unroll
    for (int j = 0; j < 4; j++) q[j] = quad(qc, j);
    if (__all_sync(0xffffffffu, mode == LBE_PARTICLES_STATIC)) return;
    const bool moves = act && mode != LBE_PARTICLES_STATIC, free_ = mode == LBE_PARTICLES_FREE;
    double row[3], col[3];
    quad_rot(k, q, row, col);
    double wb = col[0] * quad(W, 0) + col[1] * quad(W, 1) + col[2] * quad(W, 2);
    {
        const double tb = col[0] * quad(T, 0) + col[1] * quad(T, 1) + col[2] * quad(T, 2);
        const double I = k == 0 ? P.Ipar[p] : P.Iperp[p];
        const double Lb = I * wb;
        const int k1 = k == 2 ? 0 : k + 1, k2 = k == 0 ? 2 : k - 1;
        const double wl = quad(wb, k1) * quad(Lb, k2) - quad(wb, k2) * quad(Lb, k1);
        if (free_) {
            V += F / P.M[p];
            wb += (tb - wl) / I;
        }
        X += V;
    }
    // q <- normalise(q (x) exp(ω_body / 2)): component l of the product is
    // a0 b_l ± a1 b_{l^1} ± a2 b_{l^2} ± a3 b_{l^3}
    {
        const double h = 0.5 * wb;
        const double h0 = quad(h, 0), h1 = quad(h, 1), h2 = quad(h, 2);
        const double x = h0 * h0 + h1 * h1 + h2 * h2;
        double c, s;  // cos |h|, sin |h| / |h|
        if (x < 1.0 / 256.0) {
            // Taylor series in x = |h|^2: the first terms left out are below
            // x^6 / 12! < 1e-23, so only rounding remains, and the square
            // root, the division and the general sine and cosine go
            c = 1.0 + x * (-1.0 / 2 + x * (1.0 / 24 + x * (-1.0 / 720 + x * (1.0 / 40320 + x * (-1.0 / 3628800)))));
            s = 1.0 + x * (-1.0 / 6 + x * (1.0 / 120 + x * (-1.0 / 5040 + x * (1.0 / 362880 + x * (-1.0 / 39916800)))));
        } else {
            const double hn = sqrt(x);
            s = hn > 0 ? sin(hn) / hn : 0.0;
            c = hn > 0 ? cos(hn) : 1.0;
        }
        const double b = lane == 0 ? c : (x > 0 ? s * (lane == 1 ? h0 : (lane == 2 ? h1 : h2)) : 0.0);
        const double b1 = quad(b, lane ^ 1), b2 = quad(b, lane ^ 2), b3 = quad(b, lane ^ 3);
        const double t1 = q[1] * b1, t2 = q[2] * b2, t3 = q[3] * b3;
        double o = q[0] * b;
        o += (lane & 1) ? t1 : -t1;
        o += lane == 1 || lane == 2 ? t2 : -t2;
        o += lane >= 2 ? t3 : -t3;
        const double o0 = quad(o, 0), o1 = quad(o, 1), o2 = quad(o, 2), o3 = quad(o, 3);
        // o / |o|: the product of two unit quaternions is off by rounding only,
        // and 1.5 - x / 2 is 1 / sqrt(x) to 3/8 (x - 1)^2
        const double n2 = o0 * o0 + o1 * o1 + o2 * o2 + o3 * o3;
        const double qn = fabs(n2 - 1.0) < 1e-9 ? o * (1.5 - 0.5 * n2) : o / sqrt(n2);
        if (moves) P.q[4 * p + lane] = qn;
#pragma unroll
        for (int j = 0; j < 4; j++) q[j] = quad(qn, j);
    }
    quad_rot(k, q, row, col);
    const double Wn = row[0] * quad(wb, 0) + row[1] * quad(wb, 1) + row[2] * quad(wb, 2);
    if (free_) W = Wn;
    if (periodic_dim(L, k)) {
        const double n = (double)ext_of(L, k);
        if (X < 0) X += n;
        if (X >= n) X -= n;
    }
    if (wr && moves) {
        P.X[e] = X;
        P.V[e] = V;
        P.W[e] = W;
        reinterpret_cast<float *>(P.X32 + p)[k] = (float)X;
        reinterpret_cast<float *>(P.K32 + 2 * p)[k] = (float)V;
        reinterpret_cast<float *>(P.K32 + 2 * p + 1)[k] = (float)W;
    }
}

// The update and, for particles that move, the geometry of their new
// coverage, in one launch; it also empties the step's link list.
__global__ void __launch_bounds__(128) k_integrate(Lat L, Parts P, int mode, int *links)
{
    if (links && blockIdx.x == 0 && threadIdx.x == 0) *links = 0;  // ready for the next step's list
    bool act;
    const int p = quad_particle(P.n, act);
    double X, Xold, q[4];
    integrate_quad(L, P, mode, p, act, X, Xold, q);
    if (mode != LBE_PARTICLES_STATIC) geom_quad(L, P, p, act, false, X, Xold, q);
}

// ---------------------------------------------------------------- claim
// Every non-wall node inside a particle is claimed with atomicMin, so a
// node inside several particles goes to the lowest index.

__device__ __forceinline__ void claim_body(const Lat &L, const Parts &P, int p, uint32_t *__restrict__ owner_new)
{
    const PGeom &G = reinterpret_cast<const PGeom2 *>(P.geo)[p].now;
    const Box &box = G.box;
    if (box_full(box)) {
        for_box(box, [&](int, bool valid, int ux, int u1, int u2) {
            if (!valid) return;
            const int u[3] = {ux, u1, u2};
            const int x = wrapi(ux, L.nx), y = wrapi(u1, L.ny), z = wrapi(u2, L.nz);
            if (is_wall_z(L, z)) return;
            float d32[3];
#pragma unroll
            for (int a = 0; a < 3; a++)
                d32[a] = box.full[a] ? (float)node_disp(L, a, a == 0 ? x : (a == 1 ? y : z), G.X[a])
                                     : (float)(u[a] - G.Xi[a]) - G.Xf[a];
            float q32;
            bool in = inside_q32(G.g, d32, q32);
            if (!in && q32 <= 1.001f) {
                double dx[3] = {box_disp(L, box, 0, u[0], x, G.X[0]), box_disp(L, box, 1, u[1], y, G.X[1]),
                                box_disp(L, box, 2, u[2], z, G.X[2])};
                in = inside_exact(G.g, dx);
            }
            int n = x + L.nx * (y + L.ny * z);
            if (in && idx_ok(L, n, L.N, 4)) atomicMin(owner_new + n, (uint32_t)p);
        });
        return;
    }
    for_rows(box, [&](int, bool valid, int u1, int u2) {
        int a = 1, b = 0;
        if (valid && !is_wall_z(L, wrapi(u2, L.nz))) {
            const RowSpan r = span_of(G.g, G.Xi, G.Xf, box, u1, u2);
            // the FP64 test for the nodes between the two bounds
            auto in = [&](int ux) {
                const double dx[3] = {s_((double)ux, G.X[0]), s_((double)u1, G.X[1]), s_((double)u2, G.X[2])};
                return inside_exact(G.g, dx);
            };
            const bool core = r.ia <= r.ib;
            a = r.oa;
            b = r.ob;
            while (a <= b && !(core && a >= r.ia) && !in(a)) a++;
            while (a <= b && !(core && b <= r.ib) && !in(b)) b--;
        }
        fill_rows(L, a, b, u1, u2, [&](int n) {
            if (idx_ok(L, n, L.N, 4)) atomicMin(owner_new + n, (uint32_t)p);
        });
    });
}

__global__ void __launch_bounds__(PT_WIDE) k_claim(Lat L, Parts P, uint32_t *__restrict__ owner_new)
{
    claim_body(L, P, blockIdx.x, owner_new);
}

// ------------------------------------------------------------ transition
// Compare the old and new ownership.  A node whose owner changed is handled
// by exactly one CTA: that of the lower of its old and new owner.
//  - newly covered: its fluid (mass and momentum Σ f c) goes to the particle;
//  - newly uncovered: f = f^eq(ρ̄^c, u_surf) with ρ̄^c the mean over
//    neighbours fluid before and after (ρ_ref if none); the particle loses
//    that momentum;  both through the pending force/torque.
// With placement != 0 (particles just added) nodes only change type.
//
// A node whose owner changes with p the lower of the two owners is inside
// the particle's old ellipsoid or its new one but not both, so it lies in
// the outer bound of one and outside the inner bound of the other: only
// those few nodes of each row are looked at, and their two owners decide.
// The fill or empty of a changed node is the work of a whole warp (one
// direction, or one neighbour's populations, per lane).  512^3 Pickering:
// 731 us when every candidate's two owners were read and one lane did each
// change, 198 now; 40 dragged particles, of which some change every step:
// 67 and 17 us.

// What a particle takes over with (o == NONE, covered) or gives to (w ==
// NONE, uncovered) node (x, y, z): momentum mom.  Called by a whole warp.
template <class S>
__device__ __forceinline__ void change_node(const Lat &L, const Parts &P, int p, typename S::P *f, int x, int y, int z,
                                            bool covered, const uint32_t *own_old, const uint32_t *own_new,
                                            double acc[6])
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int n = x + L.nx * (y + L.ny * z);
    const double r[3] = {node_disp(L, 0, x, P.X[3 * p]), node_disp(L, 1, y, P.X[3 * p + 1]),
                         node_disp(L, 2, z, P.X[3 * p + 2])};
    const int i = lane < Q ? lane : 0;
    const int c[3] = {cdir(CXP, i), cdir(CYP, i), cdir(CZP, i)};
    float2 v = make_float2(0.f, 0.f);  // this lane's direction, both components
    if (covered) {
        v = ld2f<S>(f, L, i, n);
    } else {
        // lane i: ρ of neighbour i, if it is fluid before and after
        float a0 = 0.f, a1 = 0.f;
        bool ok = false;
        if (lane >= 1 && lane < Q) {
            int xx = x + c[0], yy = y + c[1], zz = z + c[2];
            xx = xx < 0 ? xx + L.nx : (xx >= L.nx ? xx - L.nx : xx);
            yy = yy < 0 ? yy + L.ny : (yy >= L.ny ? yy - L.ny : yy);
            ok = !L.walls || (zz > 0 && zz < L.nz - 1);
            if (!L.walls) zz = zz < 0 ? zz + L.nz : (zz >= L.nz ? zz - L.nz : zz);
            const int m = xx + L.nx * (yy + L.ny * zz);
            ok = ok && idx_ok(L, m, L.N, 6) && own_old[m] == NONE && own_new[m] == NONE;
            if (ok) {
#pragma unroll
                for (int j = 0; j < Q; j++) {
                    const float2 v2 = ld2f<S>(f, L, j, m);
                    a0 += v2.x;
                    a1 += v2.y;
                }
            }
        }
        const unsigned have = __ballot_sync(full, ok);
        float sr0 = 0.f, sr1 = 0.f;
        for (unsigned m = have; m; m &= m - 1) {  // in the order of the directions
            sr0 += __shfl_sync(full, a0, __ffs(m) - 1);
            sr1 += __shfl_sync(full, a1, __ffs(m) - 1);
        }
        const int cnt = __popc(have);
        const float rb0 = cnt ? sr0 / cnt : (float)L.rho_ref[0], rb1 = cnt ? sr1 / cnt : (float)L.rho_ref[1];
        const double V[3] = {P.V[3 * p], P.V[3 * p + 1], P.V[3 * p + 2]};
        const double W[3] = {P.W[3 * p], P.W[3 * p + 1], P.W[3 * p + 2]};
        const float us[3] = {(float)(V[0] + W[1] * r[2] - W[2] * r[1]), (float)(V[1] + W[2] * r[0] - W[0] * r[2]),
                             (float)(V[2] + W[0] * r[1] - W[1] * r[0])};
        const float uu = us[0] * us[0] + us[1] * us[1] + us[2] * us[2];
        const float wi = i == 0 ? wgt(0) : (i < 7 ? wgt(1) : wgt(7));
        const float cu = c[0] * us[0] + c[1] * us[1] + c[2] * us[2];
        v.x = wi * rb0 * (1.f + 3.f * cu + 4.5f * cu * cu - 1.5f * uu);
        v.y = wi * rb1 * (1.f + 3.f * cu + 4.5f * cu * cu - 1.5f * uu);
        __syncwarp();
        if (lane < Q)
            f[pidx(L, i, n)] = S::enc2(make_float2(v.x - L.base[0][i], v.y - L.base[1][i]));
    }
    // Σ f c: every term is an FP32 value, whose sums over a node are exact
    // in FP64 (or differ in the last place) whatever the order
    const double both = lane < Q ? (double)v.x + (double)v.y : 0.0;
    double mom[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        double a = c[k] * both;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(full, a, o);
        mom[k] = a;
    }
    double t[3];
    cross3(r, mom, t);
    for (int k = 0; k < 3; k++) {
        acc[k] += covered ? mom[k] : -mom[k];
        acc[3 + k] += covered ? t[k] : -t[k];
    }
}

template <class S>
__device__ __forceinline__ void transition_body(const Lat &L, const Parts &P, int p, typename S::P *f, uint8_t *type,
                                                const uint32_t *__restrict__ own_old,
                                                const uint32_t *__restrict__ own_new, int placement)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    // the sums of the chunks c = k mod CHUNKS, each in the order of its chunks,
    // whatever warp takes them: the totals do not depend on the threads
    constexpr int CHUNKS = PT_WIDE / 32;
    __shared__ double part[CHUNKS][6];
    for (int k = threadIdx.x; k < CHUNKS * 6; k += blockDim.x) part[k / 6][k % 6] = 0.0;
    __syncthreads();
    const PGeom2 &G2 = reinterpret_cast<const PGeom2 *>(P.geo)[p];
    const Box &box = G2.uni;
    bool any = false;
    // one node a lane (cand: it has one): the changed ones go through
    // change_node one after the other
    auto visit = [&](int chunk, bool cand, int ux, int u1, int u2) {
        int x = 0, y = 0, z = 0;
        uint32_t o = NONE, w = NONE;
        if (cand) {
            x = wrapi(ux, L.nx);
            y = wrapi(u1, L.ny);
            z = wrapi(u2, L.nz);
            const int n = x + L.nx * (y + L.ny * z);
            if (idx_ok(L, n, L.N, 5)) {
                o = own_old[n];
                w = own_new[n];
                if (o != w && min(o, w) == (uint32_t)p && (o == NONE || w == NONE))
                    type[n] = o == NONE ? PART : FLUID;
                else
                    o = w;
            }
        }
        unsigned m = __ballot_sync(full, o != w);
        if (placement) return;
        if (!m) return;
        any = true;
        double acc[6];  // the same on every lane
        for (int k = 0; k < 6; k++) acc[k] = part[chunk % CHUNKS][k];
        for (; m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            change_node<S>(L, P, p, f, __shfl_sync(full, x, src), __shfl_sync(full, y, src), __shfl_sync(full, z, src),
                           __shfl_sync(full, (int)(o == NONE), src) != 0, own_old, own_new, acc);
        }
        __syncwarp();
        if (lane == 0)
            for (int k = 0; k < 6; k++) part[chunk % CHUNKS][k] = acc[k];
        __syncwarp();
    };
    if (box_full(box)) {
        for_box(box, visit);
    } else {
        for_rows(box, [&](int chunk, bool valid, int u1, int u2) {
            int a = 1, b = 0, ca = 1, cb = 0;  // nodes [a, b] but for [ca, cb]
            if (valid) {
                const RowSpan s0 = span_of(G2.old_.g, G2.old_.Xi, G2.old_.Xf, box, u1, u2);
                const RowSpan s1 = span_of(G2.now.g, G2.Xui, G2.Xuf, box, u1, u2);
                if (s0.oa > s0.ob) {
                    a = s1.oa;
                    b = s1.ob;
                } else if (s1.oa > s1.ob) {
                    a = s0.oa;
                    b = s0.ob;
                } else {
                    a = min(s0.oa, s1.oa);
                    b = max(s0.ob, s1.ob);
                    if (!placement && s0.ia <= s0.ib && s1.ia <= s1.ib) {
                        ca = max(s0.ia, s1.ia);
                        cb = min(s0.ib, s1.ib);
                    }
                }
            }
            if (a == ca && ca <= cb) a = cb + 1;
            while (__any_sync(full, a <= b)) {
                visit(chunk, a <= b, a, u1, u2);
                if (++a == ca && ca <= cb) a = cb + 1;
            }
        });
    }
    if (placement) return;
    any = __syncthreads_or(any);
    if (threadIdx.x < 6) {
        double a = 0.0;
        if (any)
            for (int c = 0; c < CHUNKS; c++) a += part[c][threadIdx.x];
        (threadIdx.x < 3 ? P.Fpend + 3 * p + threadIdx.x : P.Tpend + 3 * p + threadIdx.x - 3)[0] = a;
    }
}

// T threads per CTA.  With many particles eight CTAs per SM (64 registers)
// hide the latency of the row bounds (25,033: 198 us against 281 with 96
// registers); the rare changes spill.
template <class S, int T>
__global__ void __launch_bounds__(T, T == PT ? 8 : 1) k_transition(Lat L, Parts P, typename S::P *f, uint8_t *type,
                                                   const uint32_t *__restrict__ own_old,
                                                   const uint32_t *__restrict__ own_new, int placement)
{
    transition_body<S>(L, P, blockIdx.x, f, type, own_old, own_new, placement);
}

// ---------------------------------------------------------------- reset
// Clear an ownership map over every particle's box (old geometry when
// use_old), so the map is all NONE again for the next claim.

__device__ __forceinline__ void reset_body(const Lat &L, const Parts &P, int p, int use_old,
                                           uint32_t *__restrict__ owner)
{
    // The map holds, over this particle's box, only nodes inside its
    // ellipsoid (its own) or inside other particles' (cleared by them), so
    // clearing the outer bound of its own rows empties the map.
    const PGeom2 &G2 = reinterpret_cast<const PGeom2 *>(P.geo)[p];
    const PGeom &G = use_old ? G2.old_ : G2.now;
    if (box_full(G.box)) {
        for_box(G.box, [&](int, bool valid, int ux, int u1, int u2) {
            if (!valid) return;
            const int n = wrapi(ux, L.nx) + L.nx * (wrapi(u1, L.ny) + L.ny * wrapi(u2, L.nz));
            if (idx_ok(L, n, L.N, 7)) owner[n] = NONE;
        });
        return;
    }
    for_rows(G.box, [&](int, bool valid, int u1, int u2) {
        int a = 1, b = 0;
        if (valid) row_span(G.g, G.Xi, G.Xf, G.box, u1, u2, a, b);
        fill_rows(L, a, b, u1, u2, [&](int n) {
            if (idx_ok(L, n, L.N, 7)) owner[n] = NONE;
        });
    });
}

__global__ void __launch_bounds__(PT_WIDE) k_reset(Lat L, Parts P, int use_old, uint32_t *__restrict__ owner)
{
    reset_body(L, P, blockIdx.x, use_old, owner);
}

// ---------------------------------------------------------------- shell
// Shell fill (Eq. 10 and the colour rule) of the nodes particle p owns and of
// the wall planes: all the solid nodes a fluid node can see.  The particle
// nodes with fluid neighbours enter the link list.
//
// A CTA takes one tile of a particle's box (30 x TYI x TZI nodes).  The node
// types of the tile and a one-node halo become one 32-bit mask per row of x
// (fluid nodes), so that finding the shell nodes (a candidate next to a
// fluid node) and the fluid nodes next to them is a few shifts per row
// instead of 18 byte loads per node.  The density of each such fluid node
// goes into shared memory once, and every shell node takes the mean over its
// neighbours from there.  The densities are read from rho (DENSE: a density
// pass over the whole lattice ran before), or summed here from the
// populations and stored to rho for the link kernel.  The latter needs no
// pass but gathers 19 scattered 32-byte sectors per node (about 450 nodes per
// (8, 4, 4) ellipsoid): at 15 % oblate ellipsoids in 256^3 (f16) that was 1.5
// GB of DRAM traffic, more than the 1.3 GB of the pass, and 479 us against
// the pass's 225; it pays where particles are few (the host decides by their
// surface, fused_self).
//
// Tiles: with many particles 22 x 22 rows (an ellipsoid of reach 8 is one
// tile); with few, 10 x 5 rows, and with fewer than 64 such tiles 8 x 2, so
// that one particle spreads over many SMs (the halo rows are then 68 % or 150
// % more rows, which costs less than idle SMs).  Results do not depend on the tiling.
//
// A tile's link entries go into the list as one contiguous segment in row
// order (one reservation, while the densities come in), so that the link
// kernel, which walks the list in order, handles neighbouring links together:
// their slots share cache lines.  With the small tiles a segment is filled up
// to a multiple of 8 with empty entries, so that the link kernel's groups of
// 8 belong to one particle.
//
// The kernel is bound by instruction issue: rows are handled by (plane: warp,
// row: lane) without a division, and node lists are written out once instead
// of a search per node.  512^3 Pickering, DENSE: 965 us with a search per node
// and divisions, 700 now; before the masks 1,420.
constexpr int SHELL_ITEMS = 1024;  // nodes of a list held at once, and densities held per tile
constexpr int SHELL_X = 30;        // nodes of a tile along x: a mask word less the halo
constexpr int SHELL_MAX = 22;      // rows of a tile along y and z
constexpr int RS = SHELL_MAX + 4;  // rows with the halo, and an empty row on each side
constexpr int SHELL_PLANES = (SHELL_MAX + 2 + PT / 32 - 1) / (PT / 32);  // planes of rows per warp

struct ShellTile {
    uint32_t S[RS * RS];     // candidate nodes (bit b: x = x0 - 1 + b), then shell nodes
    uint32_t F[RS * RS];     // fluid nodes
    uint32_t M[RS * RS];     // particle nodes, then fluid nodes next to a shell node
    int base[RS * RS];       // node index of the row's x = 0, -1 beyond a wall
    uint16_t start[RS * RS];  // fluid nodes of M in the rows before
    uint16_t fl[SHELL_ITEMS], sl[SHELL_ITEMS];  // lists of fluid and shell nodes: row << 5 | bit
    float2 rho[SHELL_ITEMS];
    uint32_t plane[SHELL_MAX + 2];  // fluid nodes | shell nodes << 16 of a plane of rows
    int owned, next, lbase;
};

// Bits of row r that have a neighbour (one of the 18) in the mask rows a.
__device__ __forceinline__ uint32_t dilate18(const uint32_t *a, int r)
{
    const uint32_t e = a[r - 1] | a[r + 1] | a[r - RS] | a[r + RS], c = a[r];
    return a[r - RS - 1] | a[r - RS + 1] | a[r + RS - 1] | a[r + RS + 1] | e | ((c | e) << 1) | ((c | e) >> 1);
}

template <class S, bool DENSE>
__device__ void shell_tile(const Lat &L, const Parts &P, int p, int tile, ShellGrid sg, const typename S::P *__restrict__ f,
                           float *rho, float *__restrict__ psi, const uint8_t *__restrict__ type,
                           const uint32_t *__restrict__ owner, const LinkList &ll, ShellTile &sm)
{
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const PGeom &G = reinterpret_cast<const PGeom2 *>(P.geo)[p].now;
    const Box &box = G.box;
    const int tx = tile % sg.nx, ty = (tile / sg.nx) % sg.ny, tz = tile / (sg.nx * sg.ny);
    const int ox = tx * SHELL_X, oy = ty * sg.tyi, oz = tz * sg.tzi;
    if (ox >= box.ext[0] || oy >= box.ext[1] || oz >= box.ext[2]) return;
    const int ex = min(SHELL_X, box.ext[0] - ox), ey = min(sg.tyi, box.ext[1] - oy), ez = min(sg.tzi, box.ext[2] - oz);
    const int x0 = box.lo[0] + ox, y0 = box.lo[1] + oy, z0 = box.lo[2] + oz;
    const int xs = wrapi(x0 - 1, L.nx);
    auto xnode = [&](int bit) {
        const int x = xs + bit;
        return x < L.nx ? x : (L.nx >= 32 ? x - L.nx : x % L.nx);
    };
    // Rows: lane ry = 0 .. ey + 1 of plane rz = 0 .. ez + 1 (the halo first and
    // last), plane rz by warp rz mod 4; row index r.
    auto row = [&](int ry, int rz) { return ry + 1 + RS * (rz + 1); };
    for (int r = tid; r < RS * RS; r += PT) sm.S[r] = sm.F[r] = 0u;
    if (tid == 0) sm.owned = sm.next = 0;
    __syncthreads();
    // candidates of each row
    for (int rz = warp; rz < ez + 2; rz += PT / 32) {
        if (lane >= ey + 2) continue;
        const int u1 = y0 - 1 + lane, u2 = z0 - 1 + rz;
        uint32_t c = 0;
        if (lane >= 1 && lane <= ey && rz >= 1 && rz <= ez) {
            int a = x0, b = x0 + ex - 1;
            if (!box_full(box)) {
                row_span(G.g, G.Xi, G.Xf, box, u1, u2, a, b);
                a = max(a, x0);
                b = min(b, x0 + ex - 1);
            }
            if (a <= b) c = (0xFFFFFFFFu << (a - x0 + 1)) & (0xFFFFFFFFu >> (30 - (b - x0)));
        }
        const bool out = L.walls && (u2 < 0 || u2 >= L.nz);
        sm.S[row(lane, rz)] = c;
        sm.base[row(lane, rz)] = out ? -1 : L.nx * (wrapi(u1, L.ny) + L.ny * wrapi(u2, L.nz));
    }
    __syncthreads();
    // fluid and particle nodes of the rows that a candidate can see: a row's
    // 32 types by one load of the warp, eight rows in flight
    const int xl = xnode(lane);
    for (int rz = warp; rz < ez + 2; rz += PT / 32) {
        const int r = row(min(lane, ey + 1), rz);
        const int mybase = sm.base[r];
        uint32_t near = 0;
#pragma unroll
        for (int k = 0; k < 9; k++) near |= sm.S[r + k % 3 - 1 + RS * (k / 3 - 1)];
        unsigned todo = __ballot_sync(full, lane < ey + 2 && near != 0 && mybase >= 0);
        uint32_t fl = 0, pt = 0;
        while (todo) {
            uint8_t t[8];
            int rr[8];
#pragma unroll
            for (int q = 0; q < 8; q++) {
                rr[q] = todo ? __ffs(todo) - 1 : -1;
                todo &= todo - 1;
                const int b = __shfl_sync(full, mybase, max(rr[q], 0));
                t[q] = rr[q] >= 0 ? type[b + xl] : WALL;
            }
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const uint32_t bf = __ballot_sync(full, t[q] == FLUID), bp = __ballot_sync(full, t[q] == PART);
                if (lane == rr[q]) {
                    fl = bf;
                    pt = bp;
                }
            }
        }
        if (lane < ey + 2) {
            sm.F[r] = fl;
            sm.M[r] = pt;
        }
    }
    __syncthreads();
    for (int rz = warp; rz < ez + 2; rz += PT / 32) {  // shell nodes
        if (lane >= ey + 2) continue;
        const int r = row(lane, rz);
        const uint32_t c = sm.S[r] & sm.M[r];
        sm.S[r] = c ? c & dilate18(sm.F, r) : 0u;
    }
    __syncthreads();
    // fluid nodes next to them, and the counts of both per plane
    uint32_t excl[SHELL_PLANES];
#pragma unroll
    for (int q = 0; q < SHELL_PLANES; q++) {
        const int rz = warp + q * (PT / 32);
        excl[q] = 0;
        if (rz >= ez + 2) continue;  // the same for the whole warp
        uint32_t v = 0;
        if (lane < ey + 2) {
            const int r = row(lane, rz);
            const uint32_t n = sm.F[r] & dilate18(sm.S, r);
            sm.M[r] = n;
            v = (uint32_t)__popc(n) | ((uint32_t)__popc(sm.S[r]) << 16);
        }
        uint32_t incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(full, incl, o);
            if (lane >= o) incl += u;
        }
        excl[q] = incl - v;
        if (lane == 31) sm.plane[rz] = incl;
    }
    __syncthreads();
    uint32_t pl = lane < ez + 2 ? sm.plane[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(full, pl, o);
        if (lane >= o) pl += u;
    }
    const uint32_t total = __shfl_sync(full, pl, 31);
    const int nf = (int)(total & 0xFFFFu), ns = (int)(total >> 16);
#pragma unroll
    for (int q = 0; q < SHELL_PLANES; q++) {  // prefix over all rows
        const int rz = warp + q * (PT / 32);
        const uint32_t before = __shfl_sync(full, pl, max(rz - 1, 0) & 31);
        if (rz > 0) excl[q] += before;
        if (rz < ez + 2 && lane < ey + 2) sm.start[row(lane, rz)] = (uint16_t)(excl[q] & 0xFFFFu);
    }
    // items [w, w + SHELL_ITEMS) of the fluid (sh = 0) or shell (16) nodes
    auto expand = [&](const uint32_t *mask, int sh, int w, uint16_t *list) {
#pragma unroll
        for (int q = 0; q < SHELL_PLANES; q++) {
            const int rz = warp + q * (PT / 32);
            if (rz >= ez + 2 || lane >= ey + 2) continue;
            const int r = row(lane, rz);
            int k = (int)((excl[q] >> sh) & 0xFFFFu) - w;
            for (uint32_t m = mask[r]; m; m &= m - 1, k++)
                if (k >= 0 && k < SHELL_ITEMS) list[k] = (uint16_t)(r << 5 | (__ffs(m) - 1));
        }
    };
    auto node = [&](int it) { return sm.base[it >> 5] + xnode(it & 31); };
    const float dr = (float)P.drho[p];
    expand(sm.M, 0, 0, sm.fl);
    for (int ws = 0; ws < ns; ws += SHELL_ITEMS) {
        const int cs = min(ns - ws, SHELL_ITEMS);
        if (ws) {
            __syncthreads();
            if (tid == 0) sm.owned = sm.next = 0;
        }
        expand(sm.S, 16, ws, sm.sl);
        __syncthreads();
        // nodes of another particle (overlaps) drop out; the link list's
        // segment is reserved while the densities come in
        int mine = 0;
        for (int k = tid; k < cs; k += PT) {
            const int n = node(sm.sl[k]);
            if (idx_ok(L, n, L.N, 9) && owner[n] == (uint32_t)p)
                mine++;
            else
                sm.sl[k] = 0xFFFFu;
        }
        mine = __reduce_add_sync(full, mine);
        if (lane == 0 && mine) atomicAdd(&sm.owned, mine);
        __syncthreads();
        const int owned = sm.owned, padded = (owned + sg.pad - 1) / sg.pad * sg.pad;
        int reserved = 0;
        if (tid == 0 && ll.ent && owned) reserved = atomicAdd(ll.count, padded);
        if (ws == 0)
            for (int wf = 0; wf < nf; wf += SHELL_ITEMS) {
                if (wf) {
                    __syncthreads();
                    expand(sm.M, 0, wf, sm.fl);
                    __syncthreads();
                }
                for (int k = tid; k < min(nf - wf, SHELL_ITEMS); k += PT) {
                    const int n = node(sm.fl[k]);
                    if (!idx_ok(L, n, L.N, 8)) continue;
                    const float2 v = DENSE ? ld_pair(rho, n) : node_rho2<S>(f, L, n);
                    if (wf == 0) sm.rho[k] = v;
                    if (!DENSE) st_pair(rho, n, v);
                }
            }
        if (tid == 0) sm.lbase = reserved;
        __syncthreads();
        for (int k0 = 0; k0 < cs; k0 += PT) {  // whole warps: positions by vote
            const int k = k0 + tid;
            const int it = k < cs ? sm.sl[k] : 0xFFFFu;
            const bool have = it != 0xFFFFu;
            int n = 0;
            uint32_t fm = 0;
            if (have) {
                n = node(it);
                const int r = it >> 5, bit = it & 31;
                float s0 = 0.f, s1 = 0.f;
                // the neighbour rows' masks and starts, then the 18 in order;
                // a neighbour that is no fluid node adds zero
                uint32_t m[9];
                int st[9];
#pragma unroll
                for (int q = 0; q < 9; q++) {
                    m[q] = sm.M[r + q % 3 - 1 + RS * (q / 3 - 1)];
                    st[q] = sm.start[r + q % 3 - 1 + RS * (q / 3 - 1)];
                }
#pragma unroll
                for (int i = 1; i < Q; i++) {
                    const int q = cy(i) + 1 + 3 * (cz(i) + 1), b = bit + cx(i);
                    const bool on = (m[q] >> b) & 1u;
                    const int idx = st[q] + __popc(m[q] & ((1u << b) - 1u));
                    float2 v = make_float2(0.f, 0.f);
                    if (on) v = idx < SHELL_ITEMS ? sm.rho[idx] : ld_pair(rho, sm.base[r + cy(i) + RS * cz(i)] + xnode(b));
                    s0 += v.x;
                    s1 += v.y;
                    fm |= on ? 1u << i : 0u;
                }
                shell_psi(L, psi, n, dr, s0, s1, __popc(fm));
            }
            if (!ll.ent) continue;
            int at = k;
            if (owned != cs) {  // a segment without gaps
                const unsigned want = __ballot_sync(full, have);
                int first = 0;
                if (want && lane == __ffs(want) - 1) first = atomicAdd(&sm.next, __popc(want));
                if (want) first = __shfl_sync(full, first, __ffs(want) - 1);
                at = first + __popc(want & ((1u << lane) - 1u));
            }
            if (have && sm.lbase + at < ll.cap) ll.ent[sm.lbase + at] = make_uint2((unsigned)n, fm);
        }
        if (ll.ent)
            for (int k = owned + tid; k < padded; k += PT)
                if (sm.lbase + k < ll.cap) ll.ent[sm.lbase + k] = make_uint2(0u, 0u);
    }
}

// Shell fill of a 32 x 8 tile of a wall plane (z = 0 or nz - 1, Δρ = 0): the
// densities of the adjacent plane's tile and a one-node halo are summed once
// into shared memory; each wall node has five neighbours there.
constexpr int WALL_X = 32, WALL_Y = 8;
__host__ __device__ inline int wall_tiles(const Lat &L)
{
    return L.walls ? 2 * ((L.nx + WALL_X - 1) / WALL_X) * ((L.ny + WALL_Y - 1) / WALL_Y) : 0;
}

template <class S>
__device__ void wall_tile(const Lat &L, int tile, const typename S::P *__restrict__ f, float *__restrict__ psi,
                          const uint8_t *__restrict__ type, ShellTile &sm)
{
    constexpr int HX = WALL_X + 2, HN = HX * (WALL_Y + 2);
    static_assert(HN <= SHELL_ITEMS && HN <= RS * RS, "wall tile fits the particle tile's arrays");
    const int ntx = (L.nx + WALL_X - 1) / WALL_X, nty = (L.ny + WALL_Y - 1) / WALL_Y;
    const int side = tile / (ntx * nty), t = tile % (ntx * nty);
    const int x0 = (t % ntx) * WALL_X, y0 = (t / ntx) * WALL_Y;
    const int zw = side ? L.nz - 1 : 0, zf = side ? L.nz - 2 : 1;
    for (int e = threadIdx.x; e < HN; e += PT) {
        const int n = wrapi(x0 - 1 + e % HX, L.nx) + L.nx * (wrapi(y0 - 1 + e / HX, L.ny) + L.ny * zf);
        const bool fl = type[n] == FLUID;
        sm.F[e] = fl;
        if (fl) sm.rho[e] = node_rho2<S>(f, L, n);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < WALL_X * WALL_Y; k += PT) {
        const int x = x0 + k % WALL_X, y = y0 + k / WALL_X;
        if (x >= L.nx || y >= L.ny) continue;
        const int n = x + L.nx * (y + L.ny * zw);
        if (type[n] != WALL) continue;
        float s0 = 0.f, s1 = 0.f;
        int cnt = 0;
#pragma unroll
        for (int i = 1; i < Q; i++) {
            if (cz(i) != (side ? -1 : 1)) continue;
            const int e = (k % WALL_X + 1 + cx(i)) + HX * (k / WALL_X + 1 + cy(i));
            if (!sm.F[e]) continue;
            const float2 v = sm.rho[e];
            s0 += v.x;
            s1 += v.y;
            cnt++;
        }
        shell_psi(L, psi, n, 0.f, s0, s1, cnt);
    }
}

// The tiles of a range of the particles, then those of the walls.
template <class S, bool DENSE>
__global__ void __launch_bounds__(PT) k_shell_fill(Lat L, Parts P, ShellGrid sg, const typename S::P *__restrict__ f,
                                                   float *rho, float *__restrict__ psi, const uint8_t *__restrict__ type,
                                                   const uint32_t *__restrict__ owner, LinkList ll, ShellRange range)
{
    __shared__ ShellTile sm;
    const int nt = sg.nx * sg.ny * sg.nz, npt = range.parts * nt, c = blockIdx.x;
    if (c < npt)
        shell_tile<S, DENSE>(L, P, range.first + c / nt, c % nt, sg, f, rho, psi, type, owner, ll, sm);
    else
        wall_tile<S>(L, c - npt, f, psi, type, sm);
}

// ------------------------------------------------------------- batched
// One launch for all boxes of a batch: a CTA (or thread) per particle of the
// batch, in box order; parities come from the batch's device state.

// Start of a batched step: the fused kernel's tile queue is empty again.
__global__ void k_begin_batch(BatchIndex B) { *B.counter = 0; }

template <class S, bool DENSE>
__global__ void __launch_bounds__(PT) k_shell_batch(BatchIndex B, ShellGrid sg, ShellRange range)
{
    __shared__ ShellTile sm;
    const int nt = sg.nx * sg.ny * sg.nz, c = blockIdx.x;
    const bool part = c < range.parts * nt;
    const int g = part ? range.first + c / nt : c - range.parts * nt;
    const int *off = part ? B.part0 : B.wall0;
    const int b = part ? B.pbox[g] : find_box(B.wall0, B.nbox, g);
    const BoxDev &bx = B.box[b];
    const int cur = B.par[2 * b], ocur = B.par[2 * b + 1];
    const typename S::P *f = (const typename S::P *)bx.f[cur];
    if (part)
        shell_tile<S, DENSE>(bx.L, bx.P, g - off[b], c % nt, sg, f, bx.rho, bx.psi, bx.type, bx.owner[ocur], bx.links, sm);
    else
        wall_tile<S>(bx.L, g - off[b], f, bx.psi, bx.type, sm);
}

__global__ void __launch_bounds__(PT_WIDE) k_claim_batch(BatchIndex B, int total)
{
    const int g = blockIdx.x;
    const int b = B.pbox[g];
    const BoxDev &bx = B.box[b];
    if (bx.mode == LBE_PARTICLES_STATIC) return;
    claim_body(bx.L, bx.P, g - B.part0[b], bx.owner[1 - B.par[2 * b + 1]]);
}

template <class S>
__global__ void __launch_bounds__(PT_WIDE) k_transition_batch(BatchIndex B, int total)
{
    const int g = blockIdx.x;
    const int b = B.pbox[g];
    const BoxDev &bx = B.box[b];
    if (bx.mode == LBE_PARTICLES_STATIC) return;
    const int cur = B.par[2 * b], ocur = B.par[2 * b + 1];
    transition_body<S>(bx.L, bx.P, g - B.part0[b], (typename S::P *)bx.f[1 - cur], bx.type, bx.owner[ocur],
                       bx.owner[1 - ocur], 0);
}

__global__ void __launch_bounds__(PT_WIDE) k_reset_batch(BatchIndex B, int total)
{
    const int g = blockIdx.x;
    const int b = B.pbox[g];
    const BoxDev &bx = B.box[b];
    if (bx.mode == LBE_PARTICLES_STATIC) return;
    reset_body(bx.L, bx.P, g - B.part0[b], 1, bx.owner[B.par[2 * b + 1]]);
}

__global__ void __launch_bounds__(128) k_geom_batch(BatchIndex B, int total)
{
    bool act;
    const int g = quad_particle(total, act);
    const int b = B.pbox[g];
    const BoxDev &bx = B.box[b];
    // the quads of a warp may belong to boxes of either kind: all take part
    geom_body(bx.L, bx.P, g - B.part0[b], act && bx.mode != LBE_PARTICLES_STATIC, false);
}

__global__ void __launch_bounds__(128) k_integrate_batch(BatchIndex B, int total)
{
    bool act;
    const int g = quad_particle(total, act);
    const int b = B.pbox[g];
    const BoxDev &bx = B.box[b];
    double X, Xold, q[4];
    integrate_quad(bx.L, bx.P, bx.mode, g - B.part0[b], act, X, Xold, q);
}

// Pair forces within each box, over its box's particles in index order (the
// same terms in the same order as the cell list of a lattice stepped alone).
__global__ void __launch_bounds__(128) k_pairs_batch(BatchIndex B, int total)
{
    __shared__ PairGroup gr[PAIR_GROUPS];
    const int g = (blockIdx.x * 128 + threadIdx.x) / PG;
    if (g >= total) return;
    const int b = B.pbox[g];
    const BoxDev &bx = B.box[b];
    pairs_body(bx.L, bx.P, bx.pair, nullptr, g - B.part0[b], gr[threadIdx.x / PG]);
}

// End of a batched step: flip each box's parities.
__global__ void k_flip_batch(BatchIndex B)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B.nbox) return;
    B.par[2 * b] ^= 1;
    if (B.box[b].P.n > 0 && B.box[b].mode != LBE_PARTICLES_STATIC) B.par[2 * b + 1] ^= 1;
    if (B.box[b].links.count) *B.box[b].links.count = 0;  // ready for the next step's list
}

// Orientation of the first particle of each box (zeros for a box without
// particles), for the host's per-box convergence checks.
__global__ void k_batch_quat(BatchIndex B, double *out)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B.nbox) return;
    const Parts &P = B.box[b].P;
    for (int k = 0; k < 4; k++) out[4 * b + k] = P.n > 0 ? P.q[k] : 0.0;
}

#ifdef LBE_CHECK
// Checked builds: after each step the node types must agree with the
// ownership map (particle iff owned).
__global__ void k_verify(Lat L, const uint8_t *type, const uint32_t *owner)
{
    int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= L.N) return;
    bool part = type[n] == PART, own = owner[n] != NONE;
    if (part && !own) idx_ok(L, -1 - (long long)n, 0, 10);
    if (own && !part) idx_ok(L, -1 - (long long)n, 0, 11);
}
#endif

}  // namespace

void launch_pairs_batch(const BatchIndex &B, int total, cudaStream_t s)
{
    if (total > 0) k_pairs_batch<<<(total + PAIR_GROUPS - 1) / PAIR_GROUPS, 128, 0, s>>>(B, total);
}

void launch_integrate_batch(const BatchIndex &B, int total, cudaStream_t s)
{
    if (total > 0) k_integrate_batch<<<(4 * total + 127) / 128, 128, 0, s>>>(B, total);
}

void launch_geom_batch(const BatchIndex &B, int total, cudaStream_t s)
{
    if (total > 0) k_geom_batch<<<(4 * total + 127) / 128, 128, 0, s>>>(B, total);
}

void launch_claim_batch(const BatchIndex &B, int total, cudaStream_t s)
{
    if (total > 0) k_claim_batch<<<total, cover_threads(total), 0, s>>>(B, total);
}

void launch_reset_batch(const BatchIndex &B, int total, cudaStream_t s)
{
    if (total > 0) k_reset_batch<<<total, cover_threads(total), 0, s>>>(B, total);
}

void launch_batch_quat(const BatchIndex &B, double *out, cudaStream_t s)
{
    k_batch_quat<<<(B.nbox + 127) / 128, 128, 0, s>>>(B, out);
}

void launch_flip_batch(const BatchIndex &B, cudaStream_t s)
{
    k_flip_batch<<<(B.nbox + 127) / 128, 128, 0, s>>>(B);
}

void launch_verify(const Lat &L, const uint8_t *type, const uint32_t *owner, cudaStream_t s)
{
#ifdef LBE_CHECK
    k_verify<<<(L.N + 255) / 256, 256, 0, s>>>(L, type, owner);
#endif
}

#define LBE_DISPATCH(storage, CALL)                                   \
    do {                                                              \
        switch (storage) {                                            \
        case LBE_STORE_F16_OFS: { using S = StF16; CALL; } break;     \
        case LBE_STORE_BF16_OFS: { using S = StBF16; CALL; } break;   \
        default: { using S = StF32; CALL; } break;                    \
        }                                                             \
    } while (0)

void launch_links(int storage, const Lat &L, const Parts &P, void *fnew, const float *rho,
                  const uint8_t *type, const uint32_t *owner, cudaStream_t s)
{
    if (P.n == 0) return;
    LBE_DISPATCH(storage, (k_links<S><<<P.n, PT, 0, s>>>(L, P, (typename S::P *)fnew, rho, type, owner)));
}

bool pairs_by_cells(int np) { return np > PAIRS_SCAN_MAX; }

void launch_pairs(const Lat &L, const Parts &P, const Pair &pp, const Cells &C, cudaStream_t s)
{
    if (P.n == 0) return;
    const int b = (P.n + 127) / 128, bp = (P.n + PAIR_GROUPS - 1) / PAIR_GROUPS;
    if (!pairs_by_cells(P.n)) {
        k_pairs<false><<<bp, 128, 0, s>>>(L, P, pp, C);
        return;
    }
    cudaMemsetAsync(C.head, 0xFF, (size_t)C.ncell * sizeof(int), s);  // empty lists: -1
    k_cell_lists<<<b, 128, 0, s>>>(L, P, C);
    k_pairs<true><<<bp, 128, 0, s>>>(L, P, pp, C);
}

void launch_geom(const Lat &L, const Parts &P, cudaStream_t s)
{
    if (P.n == 0) return;
    k_geom<<<(4 * P.n + 127) / 128, 128, 0, s>>>(L, P);
}

size_t geom_bytes_per_particle() { return sizeof(PGeom2); }

void launch_integrate(const Lat &L, const Parts &P, int mode, int *links, cudaStream_t s)
{
    if (P.n == 0) return;
    k_integrate<<<(4 * P.n + 127) / 128, 128, 0, s>>>(L, P, mode, links);
}

void launch_claim(const Lat &L, const Parts &P, int, uint32_t *owner_new, cudaStream_t s)
{
    if (P.n == 0) return;
    k_claim<<<P.n, cover_threads(P.n), 0, s>>>(L, P, owner_new);
}

void launch_transition(int storage, const Lat &L, const Parts &P, void *f, uint8_t *type,
                       const uint32_t *owner_old, const uint32_t *owner_new, int placement,
                       cudaStream_t s)
{
    if (P.n == 0) return;
    if (cover_threads(P.n) == PT)
        LBE_DISPATCH(storage, (k_transition<S, PT><<<P.n, PT, 0, s>>>(L, P, (typename S::P *)f, type, owner_old, owner_new,
                                                                      placement)));
    else
        LBE_DISPATCH(storage, (k_transition<S, PT_WIDE><<<P.n, PT_WIDE, 0, s>>>(L, P, (typename S::P *)f, type, owner_old,
                                                                                owner_new, placement)));
}

void launch_transition_batch(int storage, const BatchIndex &B, int total, cudaStream_t s)
{
    if (total == 0) return;
    LBE_DISPATCH(storage, (k_transition_batch<S><<<total, cover_threads(total), 0, s>>>(B, total)));
}

// Tiles for np particles in boxes of at most ext nodes a side.  The small
// tiles are at most 15 times as many as the large ones, fewer than 15 x 304
// (the smallest at most 6 times 64); each adds at most 7 empty entries to each
// of its at most two list windows (10 x 5 x 30 nodes): fewer than LINK_PAD in
// all.
static_assert(15 * 304 * 2 * 7 <= LINK_PAD, "empty link entries fit");
static ShellGrid shell_grid(const int ext[3], int np)
{
    auto up = [](int a, int b) { return (a + b - 1) / b; };
    ShellGrid g{up(ext[0], SHELL_X), up(ext[1], SHELL_MAX), up(ext[2], SHELL_MAX), SHELL_MAX, SHELL_MAX, 1};
    if ((long long)np * g.nx * g.ny * g.nz < 2 * 152) g = ShellGrid{g.nx, up(ext[1], 10), up(ext[2], 5), 10, 5, 8};
    if (g.pad == 8 && (long long)np * g.nx * g.ny * g.nz < 64) g = ShellGrid{g.nx, up(ext[1], 8), up(ext[2], 2), 8, 2, 8};
    return g;
}

// An upper bound of a particle box's extent (box_axis: fewer than 2 h + 5
// nodes, with h at most 1.00002 rmax).
static void shell_extent(const Lat &L, double rmax, int ext[3])
{
    const double e = std::floor(2.0001 * rmax) + 5.0;
    const int n[3] = {L.nx, L.ny, L.nz};
    for (int k = 0; k < 3; k++) ext[k] = std::max(ext[k], e < n[k] ? (int)e : n[k]);
}

static ShellGrid lattice_grid(const Lat &L, float rmax, int np)
{
    int ext[3] = {1, 1, 1};
    shell_extent(L, rmax, ext);
    return shell_grid(ext, np);
}

void shell_tiles(const Lat &L, float rmax, int np, int rows[2], int *tiles)
{
    const ShellGrid g = lattice_grid(L, rmax, np);
    rows[0] = g.tyi;
    rows[1] = g.tzi;
    *tiles = g.nx * g.ny * g.nz;
}

// The launches of a shell fill: every particle has as many tiles as the
// largest one, whose product with the particles may exceed a grid (a radius
// of 250 among 240,000 small particles), so the particles go in ranges of
// SHELL_CTAS tiles at most; the walls' tiles go with the last.
#ifdef LBE_CHECK
constexpr int SHELL_CTAS = 32;  // several launches in small cases
#else
constexpr int SHELL_CTAS = 1 << 30;
#endif
template <class F>
static void shell_ranges(const ShellGrid &g, int np, int walls, F launch)
{
    const int nt = g.nx * g.ny * g.nz, most = std::max(1, SHELL_CTAS / std::max(nt, 1));
    int first = 0;
    do {
        const int parts = std::min(np - first, most);
        const unsigned ctas = (unsigned)(parts * nt + (first + parts == np ? walls : 0));
        if (ctas) launch(ctas, ShellRange{first, parts});
        first += parts;
    } while (first < np);
}

template <class S, bool DENSE>
static void shell_fill_launch(const Lat &L, const Parts &P, const ShellGrid &g, const void *f, float *rho, float *psi,
                              const uint8_t *type, const uint32_t *owner, const LinkList &ll, cudaStream_t s)
{
    shell_ranges(g, P.n, wall_tiles(L), [&](unsigned ctas, ShellRange range) {
        k_shell_fill<S, DENSE><<<ctas, PT, 0, s>>>(L, P, g, (const typename S::P *)f, rho, psi, type, owner, ll, range);
    });
}

void launch_shell_fill(int storage, const Lat &L, const Parts &P, bool dense, const void *f, float *rho, float *psi,
                       const uint8_t *type, const uint32_t *owner, const LinkList &ll, cudaStream_t s)
{
    const ShellGrid g = P.n > 0 ? lattice_grid(L, P.rmax, P.n) : ShellGrid{0, 0, 0, 1, 1, 1};
    if (dense)
        LBE_DISPATCH(storage, (shell_fill_launch<S, true>(L, P, g, f, rho, psi, type, owner, ll, s)));
    else
        LBE_DISPATCH(storage, (shell_fill_launch<S, false>(L, P, g, f, rho, psi, type, owner, ll, s)));
}

void launch_link(int storage, const Lat &L, const LinkList &ll, const float *rho, const uint32_t *owner,
                 const Parts &P, void *fout, cudaStream_t s)
{
    if (P.n == 0 || !ll.ent) return;
    int blocks = (L.N + 255) / 256;
    if (blocks > 8 * 152) blocks = 8 * 152;
    const int group = lattice_grid(L, P.rmax, P.n).pad == 8 ? 8 : 32;
    LBE_DISPATCH(storage, (k_link<S><<<blocks, 256, 0, s>>>(L, ll, rho, owner, P, (typename S::P *)fout, group)));
}

void launch_link_batch(int storage, const BatchIndex &B, const int ext[3], int total_parts, cudaStream_t s)
{
    dim3 grid(LINK_BATCH_CTAS, B.nbox);
    const int group = shell_grid(ext, total_parts).pad == 8 ? 8 : 32;
    LBE_DISPATCH(storage, (k_link_batch<S><<<grid, 256, 0, s>>>(B, group)));
}

int batch_wall_tiles(const Lat &L) { return wall_tiles(L); }

void launch_begin_batch(const BatchIndex &B, cudaStream_t s) { k_begin_batch<<<1, 1, 0, s>>>(B); }

void launch_shell_batch(int storage, const BatchIndex &B, bool dense, const int ext[3], int total_parts,
                        int total_walls, cudaStream_t s)
{
    const ShellGrid g = total_parts > 0 ? shell_grid(ext, total_parts) : ShellGrid{0, 0, 0, 1, 1, 1};
    shell_ranges(g, total_parts, total_walls, [&](unsigned ctas, ShellRange range) {
        if (dense)
            k_shell_batch<StF32, true><<<ctas, PT, 0, s>>>(B, g, range);
        else
            LBE_DISPATCH(storage, (k_shell_batch<S, false><<<ctas, PT, 0, s>>>(B, g, range)));
    });
}

void batch_shell_extent(const Lat &L, const Parts &P, int ext[3])
{
    if (P.n > 0) shell_extent(L, P.rmax, ext);
}

void launch_reset(const Lat &L, const Parts &P, int use_old, uint32_t *owner, cudaStream_t s)
{
    if (P.n == 0) return;
    k_reset<<<P.n, cover_threads(P.n), 0, s>>>(L, P, use_old, owner);
}

}  // namespace lbe

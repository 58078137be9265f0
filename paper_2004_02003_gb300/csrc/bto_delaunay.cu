// Post hoc reconstruction of missing basis flows over a Delaunay
// triangulation of the valid ones (Sec. 3.2: a Delaunay triangulation over
// the start locations of the loaded basis flows, then barycentric
// interpolation), for sm_103a.
//
// The start locations are seed-lattice points j. The Delaunay tetrahedron
// that holds a point q is the lower facet, above q, of the convex hull of
// the points lifted to w(j) = |j|^2: equivalently, the optimal basis of the
// linear program
//     minimise   sum_i lambda_i w(j_i)
//     subject to sum_i lambda_i j_i = q,  sum_i lambda_i = 1,  lambda >= 0,
// whose optimal lambda are q's barycentric coordinates in that tetrahedron.
// Each warp solves this program for one missing lattice point at a time by
// the simplex method over the valid points of a window around it (the
// lanes share out the window's points): the basis is a tetrahedron holding
// q; a point inside the tetrahedron's circumsphere (below the plane through
// its lifted vertices) has a negative reduced cost and enters; the ratio
// test picks the vertex that leaves so that q stays inside. It starts from
// four far points around q and stops when no window point lies inside the
// circumsphere. The result is the Delaunay tetrahedron of all valid points
// when its circumsphere fits in the window (no lattice point outside the
// window can then lie inside it); otherwise the window grows (radius 2 to
// 8 lattice units) and the walk resumes.
//
// Entries on the lattice's outer faces lie on the hull of the valid points.
// There the face's plane supports the lifted point set, so the tetrahedra
// meet the face in the regular triangulation of the face's own points
// under the same weights (|j|^2 differs from the face's squared in-plane
// coordinates by a constant): such an entry is solved by the same simplex
// method in the face's two free coordinates, with triangles. On a lattice
// edge two planes support the hull, and the triangulation meets the edge
// line in the segments between consecutive valid points: the entry takes
// the linear interpolant of its nearest valid neighbours along the edge. A
// missing corner is outside the hull. A lattice one point thick along an
// axis has no tetrahedra; its missing entries stay missing.
//
// Cospherical lattice points (a cell's 8 corners) make the Delaunay
// triangulation non-unique. Ties are broken as if the lifted weights were
// |j|^2 + d_r(j), with infinitesimals d_0 >> d_1 >> ... > 0 ordered by the
// point's canonical lattice id (the four far points last): when the
// unperturbed predicate is zero, the term of the lowest-ranked point with a
// non-zero cofactor decides. Predicates are exact (integer arithmetic), and
// the simplex method takes the lowest-ranked entering point and breaks
// ratio ties by rank (Bland's rule), so it terminates.
#include <cstdint>
#include <cuda_runtime.h>

#include "bto_internal.h"

namespace bto {
namespace {

typedef __int128 i128;

struct LPt {
    int32_t x, y, z;   // lattice coordinates relative to the query point
    uint32_t rank;     // canonical lattice id; the starting points' follow the lattice's
};

// Magnitudes: window points lie within kMaxWindow of the query and the four
// starting points kFar from it, so coordinate differences are at most
// 2 kFar + 2 kMaxWindow < 2^12: a 3 x 3 determinant of differences stays
// below 6 * 2^36 and the lifted 4 x 4 determinant below 4 * 3 * 2^22 * 6 *
// 2^33 < 2^63, so 64-bit integers are exact; only the ratio test's cross
// products (two orientations) need 128 bits.
// The 2 x 2 minors of coordinate differences (below 2^25) are 32-bit.
__device__ __forceinline__ int64_t det3(int32_t a0, int32_t a1, int32_t a2, int32_t b0, int32_t b1, int32_t b2,
                                        int32_t c0, int32_t c1, int32_t c2) {
    return (int64_t)a0 * (b1 * c2 - b2 * c1) - (int64_t)a1 * (b0 * c2 - b2 * c0) + (int64_t)a2 * (b0 * c1 - b1 * c0);
}

// orientation: determinant of the rows b - a, c - a, d - a
__device__ __forceinline__ int64_t orient(const LPt &a, const LPt &b, const LPt &c, const LPt &d) {
    return det3(b.x - a.x, b.y - a.y, b.z - a.z, c.x - a.x, c.y - a.y, c.z - a.z, d.x - a.x, d.y - a.y,
                d.z - a.z);
}

__device__ __noinline__ int perturbed_sign(const LPt (&t)[4], const LPt &e);

// Sign of the 5 x 5 determinant with rows (x, y, z, w, 1) of t0..t3, e
// under the perturbed lifting: negative when e is inside the circumsphere of
// the positively oriented tetrahedron (t0, t1, t2, t3).
__device__ __noinline__ int lifted_sign(const LPt (&t)[4], const LPt &e) {
    // unperturbed: rows (p - e, |p - e|^2) of the tetrahedron, expanded
    // along the squared-length column
    int32_t r[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        r[i][0] = t[i].x - e.x;
        r[i][1] = t[i].y - e.y;
        r[i][2] = t[i].z - e.z;
        r[i][3] = r[i][0] * r[i][0] + r[i][1] * r[i][1] + r[i][2] * r[i][2];
    }
    int64_t d0 = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int a = (i + 1) & 3, b = (i + 2) & 3, c = (i + 3) & 3;
        // rows a, b, c in increasing order for the minor's sign
        int u0 = a, u1 = b, u2 = c;
        if (u0 > u1) { const int s = u0; u0 = u1; u1 = s; }
        if (u1 > u2) { const int s = u1; u1 = u2; u2 = s; }
        if (u0 > u1) { const int s = u0; u0 = u1; u1 = s; }
        const int64_t m = det3(r[u0][0], r[u0][1], r[u0][2], r[u1][0], r[u1][1], r[u1][2], r[u2][0], r[u2][1],
                               r[u2][2]);
        d0 += (((i + 3) & 1) ? -m : m) * r[i][3];
    }
    if (d0 != 0) return d0 > 0 ? 1 : -1;
    return perturbed_sign(t, e);
}

// The sign when the unperturbed determinant is zero: the lowest-ranked of the
// five points with a non-zero cofactor decides. e's own cofactor is orient(T)
// > 0 (outside); vertex k's is -orient(T with e in its place), e's weight at
// that vertex, so a vertex that e has a positive weight at makes e inside.
__device__ __noinline__ int perturbed_sign(const LPt (&t)[4], const LPt &e) {
    uint32_t rank = e.rank;
    int sign = 1;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (t[k].rank >= rank) continue;
        LPt u[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) u[m] = m == k ? e : t[m];
        const int64_t o = orient(u[0], u[1], u[2], u[3]);
        if (o != 0) {
            rank = t[k].rank;
            sign = o > 0 ? -1 : 1;
        }
    }
    return sign;
}

__device__ __forceinline__ int64_t lattice_rank(int3 S, int64_t x, int64_t y, int64_t z) {
    return x + (int64_t)S.x * (y + (int64_t)S.y * z);
}

constexpr int32_t kFar = 1024;   // distance of the four starting points, lattice units
constexpr int kMaxPivots = 512;
constexpr int kMaxWindow = 8;      // largest window radius, lattice units
constexpr int kMaxWindow2 = 12;    // on a face (a window of 25 x 25 points)
// Work limit (rows plus points) of the scan that shows that a facet (edge)
// through the query point bounds the hull of all valid points.
constexpr int64_t kHullScanWork = (int64_t)1 << 22;

// floor(n / d) and ceil(n / d) for d > 0.
__device__ __forceinline__ int64_t floor_div(int64_t n, int64_t d) { return n >= 0 ? n / d : -((-n + d - 1) / d); }
__device__ __forceinline__ int64_t ceil_div(int64_t n, int64_t d) { return n >= 0 ? (n + d - 1) / d : -((-n) / d); }

// The integers t in [lo, hi] with a t + b > 0, as [t0, t1]; false when none.
__device__ __forceinline__ bool positive_range(int64_t a, int64_t b, int64_t lo, int64_t hi, int64_t &t0,
                                               int64_t &t1) {
    if (a == 0) {
        t0 = lo;
        t1 = hi;
        return b > 0 && lo <= hi;
    }
    if (a > 0) {
        t0 = max(lo, floor_div(-b, a) + 1);
        t1 = hi;
    } else {
        t0 = lo;
        t1 = min(hi, ceil_div(b, -a) - 1);
    }
    return t0 <= t1;
}

// Circumsphere of T (centre and squared radius, FP64), for the test whether it
// fits the window where FP32 leaves that open.
__device__ __noinline__ void circumsphere(const LPt (&T)[4], double (&ctr)[3], double &r2) {
    double A[3][3], b[3];
    const LPt &a = T[0];
    for (int m = 0; m < 3; ++m) {
        const LPt &p = T[m + 1];
        A[m][0] = 2.0 * (double)(p.x - a.x);
        A[m][1] = 2.0 * (double)(p.y - a.y);
        A[m][2] = 2.0 * (double)(p.z - a.z);
        b[m] = (double)(p.x - a.x) * (double)(p.x - a.x) + (double)(p.y - a.y) * (double)(p.y - a.y) +
               (double)(p.z - a.z) * (double)(p.z - a.z);
    }
    const double det = A[0][0] * (A[1][1] * A[2][2] - A[1][2] * A[2][1]) -
                       A[0][1] * (A[1][0] * A[2][2] - A[1][2] * A[2][0]) +
                       A[0][2] * (A[1][0] * A[2][1] - A[1][1] * A[2][0]);
    double c[3];
    for (int m = 0; m < 3; ++m) {
        double M[3][3];
        for (int r = 0; r < 3; ++r)
            for (int s = 0; s < 3; ++s) M[r][s] = s == m ? b[r] : A[r][s];
        c[m] = (M[0][0] * (M[1][1] * M[2][2] - M[1][2] * M[2][1]) - M[0][1] * (M[1][0] * M[2][2] - M[1][2] * M[2][0]) +
                M[0][2] * (M[1][0] * M[2][1] - M[1][1] * M[2][0])) / det;
    }
    ctr[0] = c[0] + (double)a.x; ctr[1] = c[1] + (double)a.y; ctr[2] = c[2] + (double)a.z;
    r2 = c[0] * c[0] + c[1] * c[1] + c[2] * c[2];
}

// Sets T to the four far starting points (positively oriented).
__device__ void start_tetrahedron(int64_t P, LPt (&T)[4]) {
    const int32_t far[4][3] = {{kFar, kFar, kFar}, {kFar, -kFar, -kFar}, {-kFar, kFar, -kFar}, {-kFar, -kFar, kFar}};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        T[k].x = far[k][0]; T[k].y = far[k][1]; T[k].z = far[k][2];
        T[k].rank = (uint32_t)(P + k);
    }
    if (orient(T[0], T[1], T[2], T[3]) < 0) { const LPt s = T[0]; T[0] = T[1]; T[1] = s; }
}

// True when the circumsphere of T, centred at ctr (relative to the query
// point c) with squared radius r2, stays clear of every lattice plane just
// outside the window [x0, x1] x [y0, y1] x [z0, z1] that lies inside the
// lattice: then no lattice point outside the window is inside it.
__device__ __noinline__ bool sphere_fits(const double (&ctr)[3], double r2, int3 S, int64_t cx, int64_t cy, int64_t cz,
                            int64_t x0, int64_t x1, int64_t y0, int64_t y1, int64_t z0, int64_t z1) {
    const double rad = sqrt(r2) * (1.0 + 1e-12) + 1e-9;
    const double lo[3] = {(double)(x0 - cx), (double)(y0 - cy), (double)(z0 - cz)};
    const double hi[3] = {(double)(x1 - cx), (double)(y1 - cy), (double)(z1 - cz)};
    const int64_t ext[3] = {S.x, S.y, S.z};
    const int64_t cc[3] = {cx, cy, cz};
    for (int m = 0; m < 3; ++m) {
        // a window edge on the lattice boundary needs no margin
        if (cc[m] + (int64_t)lo[m] > 0 && ctr[m] - rad <= lo[m] - 1.0) return false;
        if (cc[m] + (int64_t)hi[m] < ext[m] - 1 && ctr[m] + rad >= hi[m] + 1.0) return false;
    }
    return true;
}

// sphere_fits from the FP32 sphere: 1 or 0 where every compared distance is
// clear of its plane by 1e-4 (r + 1) (the FP32 centre and radius are within
// 1e-6 (r + 1) of the exact ones), -1 when one is closer.
__device__ __forceinline__ int fits_clearly(const float (&ctr)[3], float r2, int3 S, int cx, int cy, int cz, int64_t x0,
                                            int64_t x1, int64_t y0, int64_t y1, int64_t z0, int64_t z1) {
    const float rad = sqrtf(r2), tol = 1e-4f * (rad + 1.f);
    const float lo[3] = {(float)(x0 - cx) - 1.f, (float)(y0 - cy) - 1.f, (float)(z0 - cz) - 1.f};
    const float hi[3] = {(float)(x1 - cx) + 1.f, (float)(y1 - cy) + 1.f, (float)(z1 - cz) + 1.f};
    const bool open_lo[3] = {x0 > 0, y0 > 0, z0 > 0};
    const bool open_hi[3] = {x1 < S.x - 1, y1 < S.y - 1, z1 < S.z - 1};
    int fit = 1;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const float a = ctr[m] - rad - lo[m], b = hi[m] - ctr[m] - rad;   // room below and above
        if ((open_lo[m] && a < -tol) || (open_hi[m] && b < -tol)) return 0;
        if ((open_lo[m] && !(a > tol)) || (open_hi[m] && !(b > tol))) fit = -1;
    }
    return fit;
}

// Every routine from here on is warp-cooperative: the 32 lanes of a warp
// solve one missing entry together. They hold the same simplex, split the
// window's rows between them, and combine their findings with warp
// reductions, so every decision is warp-uniform and equal to that of a serial
// scan in rank order.
constexpr unsigned kAll = 0xffffffffu;
constexpr int64_t kNone = INT64_MAX;

__device__ __forceinline__ int64_t warp_min(int64_t v) {
    for (int o = 16; o > 0; o >>= 1) v = min(v, (int64_t)__shfl_xor_sync(kAll, (long long)v, o));
    return v;
}
__device__ __forceinline__ int64_t warp_max(int64_t v) {
    for (int o = 16; o > 0; o >>= 1) v = max(v, (int64_t)__shfl_xor_sync(kAll, (long long)v, o));
    return v;
}
__device__ __forceinline__ LPt shfl_xor_pt(const LPt &p, int o) {
    LPt r;
    r.x = __shfl_xor_sync(kAll, p.x, o);
    r.y = __shfl_xor_sync(kAll, p.y, o);
    r.z = __shfl_xor_sync(kAll, p.z, o);
    r.rank = __shfl_xor_sync(kAll, p.rank, o);
    return r;
}

__device__ __forceinline__ void positive_orientation(LPt (&t)[4]) {
    if (orient(t[0], t[1], t[2], t[3]) < 0) { const LPt s = t[0]; t[0] = t[1]; t[1] = s; }
}

// Pivot rule. The first kDeepPivots pivots enter the point deepest inside
// the circumsphere (largest r^2 - |p - c|^2 in FP32, ties to the lowest
// rank), which reaches q's simplex in few pivots; later pivots take the
// lowest-ranked point inside (Bland's rule), which cannot cycle, so every
// walk ends. Either way the entering point passes the exact predicate and
// the walk stops only when no window point is inside the circumsphere.
constexpr int kDeepPivots = 64;

// Warp-maximum key of a candidate: the FP32 depth's bits made monotone in
// the high word, the complement of the rank in the low word (ranks are
// below 2^31); 0 means none.
__device__ __forceinline__ unsigned long long depth_key(float depth, int64_t rank) {
    const unsigned bits = __float_as_uint(depth);
    const unsigned mono = (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
    return ((unsigned long long)mono << 32) | (0xffffffffu - (unsigned)rank);
}
// The depth a key's high word stands for.
__device__ __forceinline__ float depth_of(unsigned hi) {
    return __uint_as_float((hi & 0x80000000u) ? hi & 0x7fffffffu : ~hi);
}
// Lattice coordinates of the point of rank r (r < 2^31).
__device__ __forceinline__ void rank_coords(int3 S, int64_t r, int64_t (&p)[3]) {
    const int rr = (int)r;
    p[0] = rr % S.x;
    const int q = rr / S.x;
    p[1] = q % S.y;
    p[2] = q / S.y;
}

// x^2 + y^2 (+ z^2) of the filter and the depths, its roundings fixed: where q
// lies on a face of several Delaunay simplices, which of them a walk ends in,
// and with it whether the sphere fits a small window, hangs on the pivots
// taken, and those on FP32 depths that differ in the last bit.
__device__ __forceinline__ float sum2(float x, float y) { return __fmaf_rn(x, x, __fmul_rn(y, y)); }
__device__ __forceinline__ float sum3(float x, float y, float z) { return __fmaf_rn(z, z, sum2(x, y)); }

// The lifted plane through T and its circumsphere. For a point p of the
// window (coordinates relative to q)
//     F(p) = d |p|^2 - m.p + k
// is the 5 x 5 determinant of lifted_sign: T is
// kept positively oriented (d = orient(T) > 0), so F < 0 inside the
// circumsphere, 0 on it. With a = T[0], the Cramer numerators n of the
// system (p_m - a) . u = |p_m - a|^2, m = 1..3, give F(p) = d |p - a|^2 -
// n.(p - a); expanding about q leaves four products a point. The value fits
// 64 bits (see det3); the parts may wrap, so they are unsigned.
//
// c, r2: circumsphere centre (relative to q) and squared radius in FP32 for
// the filter, from the exact numerators: only the conversions, the three
// quotients and the final sums are rounded, so the centre is within 3e-7 r
// of the exact one (T holds q, so |c - q| <= r).
struct Sphere {
    int64_t d;
    uint64_t m[3], k;
    float c[3], r2;
};

// The four determinants are shared out, one to a lane, and exchanged; each is
// expanded along the column that the squared lengths replace (the first, for
// d), whose cofactors are 32-bit minors.
__device__ __forceinline__ Sphere sphere_of(const LPt (&T)[4]) {
    const int j = threadIdx.x & 3;
    int32_t v[3], p[3], q[3];   // the column expanded, and the next two in cyclic order
    const LPt &a = T[0];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const int32_t x = T[m + 1].x - a.x, y = T[m + 1].y - a.y, z = T[m + 1].z - a.z;
        v[m] = j == 0 ? x : x * x + y * y + z * z;
        p[m] = j == 2 ? z : (j == 3 ? x : y);
        q[m] = j == 2 ? x : (j == 3 ? y : z);
    }
    const int64_t det = (int64_t)v[0] * (p[1] * q[2] - q[1] * p[2]) + (int64_t)v[1] * (p[2] * q[0] - q[2] * p[0]) +
                        (int64_t)v[2] * (p[0] * q[1] - q[0] * p[1]);
    Sphere S;
    S.d = __shfl_sync(kAll, (long long)det, 0);
    int64_t n[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) n[s] = __shfl_sync(kAll, (long long)det, s + 1);
    const int32_t ac[3] = {a.x, a.y, a.z};
    const uint64_t aa = (uint64_t)(int64_t)(a.x * a.x + a.y * a.y + a.z * a.z);
    S.k = (uint64_t)S.d * aa;
    S.r2 = 0.f;
    const float fd = (float)S.d;
    float u[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        S.m[s] = (uint64_t)n[s] + 2u * (uint64_t)S.d * (uint64_t)(int64_t)ac[s];
        S.k += (uint64_t)n[s] * (uint64_t)(int64_t)ac[s];
        u[s] = 0.5f * ((float)n[s] / fd);
        S.c[s] = u[s] + (float)ac[s];
    }
    S.r2 = sum3(u[0], u[1], u[2]);
    return S;
}

// F(p) (see Sphere).
__device__ __forceinline__ int64_t sphere_value(const Sphere &S, const LPt &p) {
    return (int64_t)((uint64_t)S.d * (uint64_t)(int64_t)(p.x * p.x + p.y * p.y + p.z * p.z) -
                     S.m[0] * (uint64_t)(int64_t)p.x - S.m[1] * (uint64_t)(int64_t)p.y -
                     S.m[2] * (uint64_t)(int64_t)p.z + S.k);
}

// Whether the window point p (of rank r) is inside the circumsphere of T
// under the perturbed lifting; false for T's own vertices.
__device__ __forceinline__ bool inside_sphere(const Sphere &S, const LPt (&T)[4], const LPt &p) {
    const int64_t F = sphere_value(S, p);
    if (F != 0) return F < 0;
    if (T[0].rank == p.rank || T[1].rank == p.rank || T[2].rank == p.rank || T[3].rank == p.rank) return false;
    const LPt t4[4] = {T[0], T[1], T[2], T[3]};   // the copy keeps T itself in registers
    return perturbed_sign(t4, p) < 0;
}

// The valid points around a tile of kTileX x kTileY x kTileZ entries, one
// word for each row along x: bit k of row (ry, rz) is the lattice point
// (x0 + k, y0 + ry, z0 + rz), (x0, y0, z0) the tile's first entry less
// kMaxWindow per axis. Every entry of the tile reads its whole window from
// these words, 17 bits a row, instead of a byte of memory per point.
constexpr int kTileX = 8, kTileY = 2, kTileZ = 2;
constexpr int kRowsY = kTileY + 2 * kMaxWindow, kRowsZ = kTileZ + 2 * kMaxWindow;
static_assert(kTileX + 2 * kMaxWindow <= 32, "a row of the tile's surroundings is one word");

// The bits of a window row at or below the x of the centre c0 (x = bit -
// kMaxWindow); the row's points fall off in depth outward from there on both
// sides. Where FP32 rounds c0 across a point, that point is the nearest on
// either reading.
__device__ __forceinline__ uint32_t bits_below(float c0) {
    const int split = (int)fminf(fmaxf(floorf(c0), -(float)(kMaxWindow + 1)), (float)kMaxWindow) + kMaxWindow;
    return split < 0 ? 0u : (2u << split) - 1u;
}

__device__ __forceinline__ unsigned gcd(unsigned a, unsigned b) {
    while (b) { const unsigned r = a % b; a = b; b = r; }
    return a;
}

// The walk ended with one starting point (vertex kf of T) at weight exactly
// 0: q lies on the facet F of the other three vertices, and no window point
// is inside the sphere through F and the far starting point. F is a facet
// of the Delaunay triangulation of all valid points, and q's interpolant is
// the one over F, when (a) wrapping across F to the valid window point D on
// the other side whose sphere through F holds no other such point gives a
// tetrahedron whose sphere holds no valid window point at all and fits in
// the window, or (b) no valid point of the lattice lies strictly on the far
// side of F (F is then on the hull; shown within a work limit). Either way
// T[kf] is replaced by a valid point (D, or a vertex of F) with weight 0.
// Spheres through F order the points beyond it (a point inside the sphere
// through F and D comes before D), so the lanes' candidates D combine into
// the first one in any order.
__device__ __noinline__ bool across_facet(int3 S, const uint8_t *__restrict__ valid, const uint32_t *win, int lx, int cx,
                                          int cy, int cz, int R, LPt (&T)[4], int kf) {
    const int lane = threadIdx.x & 31;
    const int side = 2 * R + 1, rows_w = side * side;
    const uint32_t wmask = ((1u << side) - 1u) << (kMaxWindow - R);
    const int64_t x0 = max(cx - R, 0), x1 = min(cx + R, S.x - 1), y0 = max(cy - R, 0), y1 = min(cy + R, S.y - 1),
                  z0 = max(cz - R, 0), z1 = min(cz + R, S.z - 1);
    // h(p) = orient(T) with p in the starting point's place = nx x + ny y + nz z + d: positive on its side of F
    LPt u[4];
    const LPt o0 = {0, 0, 0, 0}, ex = {1, 0, 0, 0}, ey = {0, 1, 0, 0}, ez = {0, 0, 1, 0};
    auto with = [&](const LPt &p) {
#pragma unroll
        for (int k = 0; k < 4; ++k) u[k] = k == kf ? p : T[k];
        return orient(u[0], u[1], u[2], u[3]);
    };
    const int64_t d = with(o0), nx = with(ex) - d, ny = with(ey) - d, nz = with(ez) - d;
    // F's spheres order the points beyond it by F(p) / |h(p)|, F(p) the value
    // of T's own sphere: the sphere through F and p holds the points whose
    // quotient is smaller. FP32 quotients (three roundings) decide unless
    // they are within 1e-5 of each other, the exact predicate otherwise.
    const Sphere sp = sphere_of(T);
    bool far_pt = false, have = false;
    LPt D = o0;
    float Dq = 0.f;
    auto closer = [&](const LPt &p) {   // p inside the sphere through F and D
        LPt t4[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) t4[k] = k == kf ? D : T[k];
        positive_orientation(t4);
        return lifted_sign(t4, p) < 0;
    };
#pragma unroll 1
    for (int row = lane; row < rows_w; row += 32) {
        const int rz = row / side, dy = row - rz * side - R, dz = rz - R;
        uint32_t m = (win[dy + kRowsY * dz] >> lx) & wmask;
        const int r0 = cx - kMaxWindow + S.x * (cy + dy + S.y * (cz + dz));
#pragma unroll 1
        while (m) {
            const int bit = __ffs(m) - 1;
            m &= m - 1;
            const LPt p = {bit - kMaxWindow, dy, dz, (uint32_t)(r0 + bit)};
            const int64_t h = nx * p.x + ny * dy + nz * dz + d;
            if (h == 0) continue;   // F's own vertices among them
            if (h > 0) { far_pt = true; continue; }
            const float q = (float)sphere_value(sp, p) / (float)(-h);
            if (!have || q < Dq * 0.99999f || (q <= Dq * 1.00001f && closer(p))) { D = p; Dq = q; have = true; }
        }
    }
    far_pt = __any_sync(kAll, far_pt);
#pragma unroll 1
    for (int off = 16; off > 0; off >>= 1) {
        const LPt Do = shfl_xor_pt(D, off);
        const float qo = __shfl_xor_sync(kAll, Dq, off);
        const bool ho = __shfl_xor_sync(kAll, (int)have, off) != 0;
        if (!ho || (have && Do.rank == D.rank)) continue;
        if (!have || closer(Do)) { D = Do; Dq = qo; have = true; }
    }
    if (have) {
        LPt t4[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) t4[k] = k == kf ? D : T[k];
        positive_orientation(t4);
        const Sphere s4 = sphere_of(t4);
        const uint32_t lowbits = bits_below(s4.c[0]);
        bool inside = false;
#pragma unroll 1
        for (int row = lane; row < rows_w && !inside; row += 32) {
            const int rz = row / side, dy = row - rz * side - R, dz = rz - R;
            const uint32_t m = (win[dy + kRowsY * dz] >> lx) & wmask;
            const int r0 = cx - kMaxWindow + S.x * (cy + dy + S.y * (cz + dz));
            // the nearest point on each side; the others of the row are
            // farther out, and strictly outside unless it is inside
            const uint32_t lo = m & lowbits, hi = m & ~lowbits;
#pragma unroll 1
            for (int dir = 0; dir < 2 && !inside; ++dir) {
                if (!(dir ? hi : lo)) continue;
                const int bit = dir ? __ffs(hi) - 1 : 31 - __clz(lo);
                const LPt p = {bit - kMaxWindow, dy, dz, (uint32_t)(r0 + bit)};
                inside = inside_sphere(s4, t4, p);
            }
        }
        inside = __any_sync(kAll, inside);
        if (!inside) {
            double ctr[3], r2;
            circumsphere(t4, ctr, r2);
            if (sphere_fits(ctr, r2, S, cx, cy, cz, x0, x1, y0, y1, z0, z1)) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (k == kf) T[k] = D;
                return true;
            }
        }
    }
    // (b): no valid point of the lattice strictly on the far side of F. The
    // orientation with p in place of the starting point is affine in p,
    // n.p + d, so each lattice row holds its far-side points in one interval
    // and only those are visited (within kHullScanWork rows and points).
    if (!far_pt) {
        const int64_t rows = (int64_t)S.y * S.z, budget = kHullScanWork / 32;
        int64_t work = 0;
        bool stop = false;                          // a far-side valid point, or out of budget
        // Each lane keeps the rows lane, lane + 32, ...; it takes them in the
        // order of multiples of a number coprime to their count, and the warp
        // ends as soon as one lane has stopped: a valid point on the far side
        // is mostly met within a few rows spread over the lattice.
        const unsigned per = (unsigned)((rows + 31) / 32);
        unsigned hop = per * 5 / 8 + 1;
        while (gcd(hop, per) != 1) ++hop;
        unsigned at = 0;
        for (unsigned k = 0; k < per && !__any_sync(kAll, stop); ++k, at = (at + hop) % per) {
            const int64_t row = lane + 32ll * at;
            if (row >= rows) continue;
            const int64_t y = (int)row % S.y, z = (int)row / S.y;
            if (++work > budget) { stop = true; continue; }
            int64_t t0, t1;
            if (!positive_range(nx, ny * (y - cy) + nz * (z - cz) + d, -(int64_t)cx, (int64_t)S.x - 1 - cx, t0, t1))
                continue;
#pragma unroll 1
            for (int64_t t = t0; t <= t1; ++t) {
                if (++work > budget || valid[lattice_rank(S, t + cx, y, z)]) { stop = true; break; }
            }
        }
        if (__any_sync(kAll, stop)) return false;
        const LPt other = kf == 3 ? T[0] : (kf == 0 ? T[1] : (kf == 1 ? T[2] : T[3]));
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k == kf) T[k] = other;
        return true;
    }
    return false;
}

// One walk in the window of radius R around c, from the tetrahedron T it is
// given (a feasible basis: q inside it), so a larger window resumes where a
// smaller one stopped; `settled` says that no point of the window of radius
// R - 1 is inside T's circumsphere, and is kept up to date for the next
// window. `win` is c's own row among the tile's words, `lx` its bit less
// kMaxWindow. The lanes take the window's rows; within a row the depth falls
// from the point nearest to the centre outward, in FP32 too (rounding is
// monotone), so a lane walks outward from there on both sides and stops as
// soon as the depth is below its best. Only points that would become the
// lane's best get the exact predicate. Returns 1 and the tetrahedron with q's
// barycentric coordinates, or 0: no result in this window (q outside the hull
// of its valid points, circumsphere larger than the window, or the pivot
// limit).
__device__ __forceinline__ int walk(int3 S, const uint8_t *__restrict__ valid, const uint32_t *win, int lx, int cx, int cy,
                                 int cz, int R, bool &settled, LPt (&T)[4], double (&lam)[4]) {
    const int lane = threadIdx.x & 31;
    const int64_t P = (int64_t)S.x * S.y * S.z;
    const int64_t x0 = max(cx - R, 0), x1 = min(cx + R, S.x - 1);
    const int64_t y0 = max(cy - R, 0), y1 = min(cy + R, S.y - 1);
    const int64_t z0 = max(cz - R, 0), z1 = min(cz + R, S.z - 1);
    const int side = 2 * R + 1, rows = side * side;
    const uint32_t wmask = ((1u << side) - 1u) << (kMaxWindow - R);
    const uint32_t ends = (1u << (kMaxWindow - R)) | (1u << (kMaxWindow + R));
    const unsigned inv_side = 65536u / (unsigned)side + 1u;   // row / side for rows < 2^16 / side
#pragma unroll 1
    for (int it = 0; it < kMaxPivots; ++it) {
        // entering point: among the valid window points inside the
        // circumsphere of T, the deepest (later the lowest-ranked) one. Near
        // the sphere the FP32 squared distance's rounding error stays below
        // 2e-6 r^2; a point farther than 8e-6 r^2 + 1e-3 from it is inside
        // or outside for certain. Most pivots enter a point that is inside
        // for certain, found from the nearest points of each row alone;
        // otherwise the candidates in the margin get the exact predicate.
        const Sphere sp = sphere_of(T);
        const float fc0 = sp.c[0], fc1 = sp.c[1], fc2 = sp.c[2];
        const float margin = sp.r2 * 8e-6f + 1e-3f, fr2 = sp.r2 + margin;
        const bool deep = it < kDeepPivots, shell = settled && it == 0;
        const uint32_t lowbits = bits_below(fc0);
        int64_t best = kNone;
        unsigned bhi = 0, blo = 0;   // the lane's best depth key (depth_key), 0: none
        if (deep) {
#pragma unroll 1
            for (int row = lane; row < rows; row += 32) {
                const int rz = (int)(((unsigned)row * inv_side) >> 16), dy = row - rz * side - R, dz = rz - R;
                uint32_t m = (win[dy + kRowsY * dz] >> lx) & wmask;
                if (shell && dy > -R && dy < R && dz > -R && dz < R) m &= ends;
                const uint32_t lo = m & lowbits, hi = m & ~lowbits;
                const float fy = (float)dy - fc1, fz = (float)dz - fc2;
                const int r0 = cx - kMaxWindow + S.x * (cy + dy + S.y * (cz + dz));
#pragma unroll 1
                for (int dir = 0; dir < 2; ++dir) {
                    uint32_t w = dir ? hi : lo;
#pragma unroll 1
                    while (w) {
                        const int bit = dir ? __ffs(w) - 1 : 31 - __clz(w);
                        w &= ~(1u << bit);
                        const float fx = (float)(bit - kMaxWindow) - fc0;
                        const unsigned long long key = depth_key(sp.r2 - (sum3(fx, fy, fz)), r0 + bit);
                        const unsigned khi = (unsigned)(key >> 32), klo = (unsigned)key;
                        if (khi < bhi || (khi == bhi && klo <= blo)) break;
                        bhi = khi;
                        blo = klo;
                        if (dir) break;   // FP32 depth can be level along a row: the lowest rank is the one to keep
                    }
                }
            }
        }
        const unsigned sure = __reduce_max_sync(kAll, bhi);
        const bool clear = deep && sure != 0 && depth_of(sure) > margin;
        if (!clear) { bhi = 0; blo = 0; }
#pragma unroll 1
        for (int row = clear ? rows : lane; row < rows; row += 32) {
            const int rz = (int)(((unsigned)row * inv_side) >> 16), dy = row - rz * side - R, dz = rz - R;
            uint32_t m = (win[dy + kRowsY * dz] >> lx) & wmask;
            if (shell && dy > -R && dy < R && dz > -R && dz < R) m &= ends;
            if (!m) continue;
            const float fy = (float)dy - fc1, fz = (float)dz - fc2;
            const int r0 = cx - kMaxWindow + S.x * (cy + dy + S.y * (cz + dz));   // the row's ranks are r0 + bit, below 2^31
            if (deep) {
#pragma unroll 1
                for (int dir = 0; dir < 2; ++dir) {
                    uint32_t w = dir ? m & ~lowbits : m & lowbits;
#pragma unroll 1
                    while (w) {
                        const int bit = dir ? __ffs(w) - 1 : 31 - __clz(w);
                        w &= ~(1u << bit);
                        const int dx = bit - kMaxWindow;
                        const float fx = (float)dx - fc0;
                        const float d2 = sum3(fx, fy, fz);
                        if (d2 > fr2) break;
                        const int r = r0 + bit;
                        const unsigned long long key = depth_key(sp.r2 - d2, r);
                        const unsigned khi = (unsigned)(key >> 32), klo = (unsigned)key;
                        if (khi < bhi) break;
                        if (khi == bhi && klo <= blo) continue;
                        const LPt p = {dx, dy, dz, (uint32_t)r};
                        if (inside_sphere(sp, T, p)) {
                            bhi = khi;
                            blo = klo;
                        }
                    }
                }
            } else {
                while (m && best == kNone) {
                    const int bit = __ffs(m) - 1;
                    m &= m - 1;
                    const int dx = bit - kMaxWindow;
                    const float fx = (float)dx - fc0;
                    if (sum3(fx, fy, fz) > fr2) continue;
                    const LPt p = {dx, dy, dz, (uint32_t)(r0 + bit)};
                    if (inside_sphere(sp, T, p)) best = r0 + bit;
                }
                if (best != kNone) break;
            }
        }
        if (deep) {
            const unsigned hi = __reduce_max_sync(kAll, bhi);
            const unsigned lo = __reduce_max_sync(kAll, bhi == hi ? blo : 0u);
            best = hi ? (int64_t)(0xffffffffu - lo) : kNone;
        } else {
            best = warp_min(best);
        }
        // orientations with vertex k replaced, one vertex to a lane (lanes
        // 4 apart hold the same): by q (oq) and, when a point enters, by
        // that point (oe)
        const LPt q0 = {0, 0, 0, 0};
        const int mine = lane & 3;
        LPt u[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) u[k] = mine == k ? q0 : T[k];
        const int64_t oq = orient(u[0], u[1], u[2], u[3]);
        const uint32_t rank_mine = mine == 0 ? T[0].rank : (mine == 1 ? T[1].rank : (mine == 2 ? T[2].rank : T[3].rank));
        if (best == kNone) {
            settled = true;
            const unsigned far = __ballot_sync(kAll, rank_mine >= (uint32_t)P) & 15u;
            const unsigned zero = __ballot_sync(kAll, oq == 0) & 15u;
            if (far == 0) {
                // the circumsphere must fit in the window: then no lattice
                // point outside the window is inside it. FP32 decides when
                // the sphere ends clearly on one side of every plane; FP64
                // otherwise.
                const int fit = fits_clearly(sp.c, sp.r2, S, cx, cy, cz, x0, x1, y0, y1, z0, z1);
                if (fit == 0) return 0;
                if (fit < 0) {
                    const LPt t4[4] = {T[0], T[1], T[2], T[3]};   // the copy keeps T itself in registers
                    double ctr[3], r2;
                    circumsphere(t4, ctr, r2);
                    if (!sphere_fits(ctr, r2, S, cx, cy, cz, x0, x1, y0, y1, z0, z1)) return 0;
                }
            } else if ((far & (far - 1)) != 0 || (far & ~zero) != 0) {
                // a starting point with weight above 0: q is outside the
                // hull of the window's valid points
                return 0;
            }
            // optimal: q's barycentric coordinates in T
#pragma unroll
            for (int k = 0; k < 4; ++k) lam[k] = (double)__shfl_sync(kAll, (long long)oq, k) / (double)sp.d;
            if (far == 0) return 1;
            // a starting point with weight 0: q is on a facet
            LPt t4[4] = {T[0], T[1], T[2], T[3]};
            if (!across_facet(S, valid, win, lx, cx, cy, cz, R, t4, __ffs(far) - 1)) return 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) T[k] = t4[k];
            return 1;
        }
        settled = false;
        const unsigned b32 = (unsigned)best;
        const int ez = (int)(b32 / (unsigned)(S.x * S.y)), ey = (int)(b32 / (unsigned)S.x) - ez * S.y;
        const LPt e = {(int32_t)(b32 % (unsigned)S.x) - cx, ey - cy, ez - cz, b32};
#pragma unroll
        for (int k = 0; k < 4; ++k) u[k] = mine == k ? e : T[k];
        const int64_t oe = orient(u[0], u[1], u[2], u[3]);
        // ratio test: leaving vertex k minimises lambda_k / d_k = oq / oe
        // over oe > 0 (orient(T) > 0 divides out); ties go to the lowest
        // rank. FP32 quotients (three roundings, 2e-7 relative) single out
        // the vertex unless another is within 1e-5 of the least; exact zeros
        // tie among themselves; other near ties are compared exactly.
        const float ratio = oe > 0 ? (float)oq / (float)oe : INFINITY;
        float least = fminf(ratio, __shfl_xor_sync(kAll, ratio, 1));
        least = fminf(least, __shfl_xor_sync(kAll, least, 2));
        if (least == INFINITY) return 0;   // cannot happen for a point inside the circumsphere
        const unsigned near = __ballot_sync(kAll, ratio <= least * 1.00001f) & 15u;
        int leave = __ffs(near) - 1;
        if (near & (near - 1)) {
            int64_t bq = 0, be = 0;
            uint32_t brank = 0;
            leave = -1;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (!(near >> k & 1u)) continue;
                const int64_t kq = __shfl_sync(kAll, (long long)oq, k), ke = __shfl_sync(kAll, (long long)oe, k);
                bool better = leave < 0;
                if (!better) {
                    // compare kq / ke against bq / be (both denominators positive)
                    if (least == 0.f) {
                        better = T[k].rank < brank;
                    } else {
                        const i128 lhs = (i128)kq * be, rhs = (i128)bq * ke;
                        better = lhs < rhs || (lhs == rhs && T[k].rank < brank);
                    }
                }
                if (better) { leave = k; bq = kq; be = ke; brank = T[k].rank; }
            }
        }
        // the new orientation is the leaving vertex's oe > 0: T stays positively oriented
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k == leave) T[k] = e;
    }
    return 0;
}

// ---- Faces: the same program in a face's two free coordinates ----------

struct LPt2 {
    int32_t u, v;      // free coordinates relative to the query point
    uint32_t rank;
};

// Counter-clockwise orientation of (a, b, c): positive when counter-clockwise.
// Coordinates differ by less than 2^12 (as for LPt), so 64 bits are exact.
__device__ __forceinline__ int64_t orient2(const LPt2 &a, const LPt2 &b, const LPt2 &c) {
    return (int64_t)(b.u - a.u) * (c.v - a.v) - (int64_t)(b.v - a.v) * (c.u - a.u);
}

__device__ __forceinline__ int perturbed_sign2(const LPt2 (&t)[3], const LPt2 &e);

// Sign of the 4 x 4 determinant with rows (u, v, w, 1) of t0, t1, t2, e under
// the perturbed lifting w = u^2 + v^2 + d_rank: positive when e is inside the
// circumcircle of the counter-clockwise triangle (t0, t1, t2). Translated so
// that e is the origin, the unperturbed part is the 3 x 3 determinant of the
// rows (p - e, |p - e|^2).
__device__ __forceinline__ int lifted_sign2(const LPt2 (&t)[3], const LPt2 &e) {
    int32_t r[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        r[i][0] = t[i].u - e.u;
        r[i][1] = t[i].v - e.v;
        r[i][2] = r[i][0] * r[i][0] + r[i][1] * r[i][1];
    }
    // expanded along the squared lengths
    const int64_t d0 = (int64_t)r[0][2] * (r[1][0] * r[2][1] - r[1][1] * r[2][0]) -
                       (int64_t)r[1][2] * (r[0][0] * r[2][1] - r[0][1] * r[2][0]) +
                       (int64_t)r[2][2] * (r[0][0] * r[1][1] - r[0][1] * r[1][0]);
    if (d0 != 0) return d0 > 0 ? 1 : -1;
    return perturbed_sign2(t, e);
}

// The sign when the unperturbed determinant is zero, as perturbed_sign: e's
// own cofactor says outside, vertex k's has the sign of e's weight there.
__device__ __forceinline__ int perturbed_sign2(const LPt2 (&t)[3], const LPt2 &e) {
    uint32_t rank = e.rank;
    int sign = -1;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (t[k].rank >= rank) continue;
        LPt2 u[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) u[m] = m == k ? e : t[m];
        const int64_t o = orient2(u[0], u[1], u[2]);
        if (o != 0) {
            rank = t[k].rank;
            sign = o > 0 ? 1 : -1;
        }
    }
    return sign;
}

// Circumcircle of T (centre and squared radius, FP64), as circumsphere.
__device__ __noinline__ void circumcircle(const LPt2 (&T)[3], double (&ctr)[2], double &r2) {
    const double bx = (double)(T[1].u - T[0].u), by = (double)(T[1].v - T[0].v);
    const double cx = (double)(T[2].u - T[0].u), cy = (double)(T[2].v - T[0].v);
    const double d = 2.0 * (bx * cy - by * cx);
    const double b2 = bx * bx + by * by, c2 = cx * cx + cy * cy;
    const double ux = (cy * b2 - by * c2) / d, uy = (bx * c2 - cx * b2) / d;
    ctr[0] = ux + (double)T[0].u;
    ctr[1] = uy + (double)T[0].v;
    r2 = ux * ux + uy * uy;
}

// The circumcircle of T for the face walk's filter, as in sphere_of: exact
// 64-bit Cramer numerators, FP32 quotients.
__device__ __forceinline__ void circumcircle_f(const LPt2 (&T)[3], float (&c)[2], float &r2) {
    const int64_t bx = T[1].u - T[0].u, by = T[1].v - T[0].v, cx = T[2].u - T[0].u, cy = T[2].v - T[0].v;   // below 2^12
    const int64_t b2 = bx * bx + by * by, c2 = cx * cx + cy * cy;
    const float d = (float)(2 * (bx * cy - by * cx));
    const float ux = (float)(cy * b2 - by * c2) / d, uy = (float)(bx * c2 - cx * b2) / d;
    c[0] = ux + (float)T[0].u;
    c[1] = uy + (float)T[0].v;
    r2 = sum2(ux, uy);
}

// Sets T to three far starting points around q (counter-clockwise).
__device__ void start_triangle(int64_t P, LPt2 (&T)[3]) {
    const int32_t far[3][2] = {{kFar, 0}, {-kFar, kFar}, {-kFar, -kFar}};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        T[k].u = far[k][0]; T[k].v = far[k][1];
        T[k].rank = (uint32_t)(P + k);
    }
    if (orient2(T[0], T[1], T[2]) < 0) { const LPt2 s = T[0]; T[0] = T[1]; T[1] = s; }
}

// The face version of sphere_fits: the circle centred at ctr (free
// coordinates relative to c) with squared radius r2 stays clear of the
// lattice lines just outside the window [u0, u1] x [v0, v1] of the face.
__device__ bool circle_fits(const double (&ctr)[2], double r2, int3 S, const int64_t (&c)[3], int a, int b,
                            int64_t u0, int64_t u1, int64_t v0, int64_t v1) {
    const int64_t ext[3] = {S.x, S.y, S.z};
    const double rad = sqrt(r2) * (1.0 + 1e-12) + 1e-9;
    const int ax[2] = {a, b};
    const int64_t lo[2] = {u0 - c[a], v0 - c[b]}, hi[2] = {u1 - c[a], v1 - c[b]};
    for (int m = 0; m < 2; ++m) {
        const int64_t cm = c[ax[m]];
        if (cm + lo[m] > 0 && ctr[m] - rad <= (double)lo[m] - 1.0) return false;
        if (cm + hi[m] < ext[ax[m]] - 1 && ctr[m] + rad >= (double)hi[m] + 1.0) return false;
    }
    return true;
}

// A face's entry and its window, one row (fixed v) to a lane: bit k of
// lane l's word is the face's point (k - kMaxWindow2, l - kMaxWindow2) in
// the free axes a < b, relative to the entry.
struct Face {
    int a, b;          // free axes
    int ca, cb;        // the entry's coordinates along them
    int ea, eb;        // lattice extents along them
    int sa, sb;        // rank steps along them
    int rq;            // the entry's rank
    uint32_t row;      // the lane's word
};
static_assert(2 * kMaxWindow2 + 1 <= 32, "a face's window is one word per lane");

__device__ __forceinline__ Face face_of(int3 S, const uint8_t *__restrict__ valid, const int64_t (&c)[3], int a, int b) {
    Face f;
    f.a = a;
    f.b = b;
    // a is 0 or 1, b is 1 or 2
    f.ca = (int)(a == 0 ? c[0] : c[1]);
    f.cb = (int)(b == 1 ? c[1] : c[2]);
    f.ea = a == 0 ? S.x : S.y;
    f.eb = b == 1 ? S.y : S.z;
    f.sa = a == 0 ? 1 : S.x;
    f.sb = b == 1 ? S.x : S.x * S.y;
    f.rq = (int)lattice_rank(S, c[0], c[1], c[2]);
    const int lane = threadIdx.x & 31, du = lane - kMaxWindow2;
    const bool in_u = lane <= 2 * kMaxWindow2 && f.ca + du >= 0 && f.ca + du < f.ea;
    f.row = 0;
#pragma unroll 5
    for (int k = 0; k <= 2 * kMaxWindow2; ++k) {
        const int dv = k - kMaxWindow2;
        const bool in = in_u && f.cb + dv >= 0 && f.cb + dv < f.eb;
        const unsigned w = __ballot_sync(kAll, in && valid[f.rq + du * f.sa + dv * f.sb] != 0);
        if (lane == k) f.row = w;
    }
    return f;
}

// The lane's row cut to the window of radius R.
__device__ __forceinline__ uint32_t face_row(const Face &f, int R) {
    const int dv = (int)(threadIdx.x & 31) - kMaxWindow2;
    return abs(dv) <= R ? f.row & (((2u << (2 * R)) - 1u) << (kMaxWindow2 - R)) : 0u;
}

// across_facet on a face: q lies on the edge F opposite the starting point
// T[kf] (weight exactly 0). Wrap across F to the valid window point D whose
// circle through F holds no other point on that side; accept when that
// triangle's circle holds no valid window point and fits in the window, or
// when no valid point of the face lies strictly on the far side of F (F is
// then on the hull of the face's points).
__device__ __noinline__ bool across_edge(int3 S, const uint8_t *__restrict__ valid, const int64_t (&c)[3], const Face &f,
                                         int R, LPt2 (&T)[3], int kf) {
    const int lane = threadIdx.x & 31, dv = lane - kMaxWindow2;
    const LPt2 A = kf == 0 ? T[1] : (kf == 1 ? T[2] : T[0]), B = kf == 0 ? T[2] : (kf == 1 ? T[0] : T[1]);
    const LPt2 far = kf == 0 ? T[0] : (kf == 1 ? T[1] : T[2]);
    const int64_t sf = orient2(A, B, far);
    const uint32_t row = face_row(f, R);
    const int r0 = f.rq + dv * f.sb - kMaxWindow2 * f.sa;   // the rank of bit k is r0 + k sa
    bool far_pt = false, have = false;
    LPt2 D = A;
    auto closer = [&](const LPt2 &p) {   // p inside the circle through F and D
        const bool ccw = orient2(A, B, D) >= 0;
        const LPt2 t3[3] = {ccw ? A : B, ccw ? B : A, D};
        return lifted_sign2(t3, p) > 0;
    };
    for (uint32_t m = row; m; m &= m - 1) {
        const int k = __ffs(m) - 1;
        const LPt2 p = {k - kMaxWindow2, dv, (uint32_t)(r0 + k * f.sa)};
        if (p.rank == A.rank || p.rank == B.rank) continue;
        const int64_t so = orient2(A, B, p);
        if (so == 0) continue;
        if ((so > 0) == (sf > 0)) { far_pt = true; continue; }
        if (!have || closer(p)) { D = p; have = true; }
    }
    far_pt = __any_sync(kAll, far_pt);
    for (int off = 16; off > 0; off >>= 1) {
        LPt2 Do;
        Do.u = __shfl_xor_sync(kAll, D.u, off);
        Do.v = __shfl_xor_sync(kAll, D.v, off);
        Do.rank = __shfl_xor_sync(kAll, D.rank, off);
        const bool ho = __shfl_xor_sync(kAll, (int)have, off) != 0;
        if (!ho || (have && Do.rank == D.rank)) continue;
        if (!have || closer(Do)) { D = Do; have = true; }
    }
    if (have) {
        bool inside = false;
        for (uint32_t m = row; m && !inside; m &= m - 1) {
            const int k = __ffs(m) - 1;
            const LPt2 p = {k - kMaxWindow2, dv, (uint32_t)(r0 + k * f.sa)};
            if (p.rank == A.rank || p.rank == B.rank || p.rank == D.rank) continue;
            inside = closer(p);
        }
        inside = __any_sync(kAll, inside);
        if (!inside) {
            const bool ccw = orient2(A, B, D) >= 0;
            const LPt2 t3[3] = {ccw ? A : B, ccw ? B : A, D};
            double ctr[2], r2;
            circumcircle(t3, ctr, r2);
            if (circle_fits(ctr, r2, S, c, f.a, f.b, max(f.ca - R, 0), min(f.ca + R, f.ea - 1), max(f.cb - R, 0),
                            min(f.cb + R, f.eb - 1))) {
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    if (k == kf) T[k] = D;
                return true;
            }
        }
    }
    // no valid point of the face strictly on the far side of F, visiting
    // only the far-side interval of each row (orient2(A, B, p) is affine in
    // p), within kHullScanWork rows and points
    if (!far_pt) {
        const LPt2 o0 = {0, 0, 0}, eu = {1, 0, 0}, ev = {0, 1, 0};
        const int64_t d = orient2(A, B, o0);
        const int64_t nu = orient2(A, B, eu) - d, nv = orient2(A, B, ev) - d;
        const int64_t sg = sf > 0 ? 1 : -1;
        const int64_t budget = kHullScanWork / 32;
        int64_t work = 0;
        bool stop = false;
        for (int64_t vv = lane; vv < f.eb && !stop; vv += 32) {
            if (++work > budget) { stop = true; break; }
            int64_t t0, t1;
            if (!positive_range(sg * nu, sg * (nv * (vv - f.cb) + d), -(int64_t)f.ca, (int64_t)f.ea - 1 - f.ca, t0, t1))
                continue;
            for (int64_t t = t0; t <= t1; ++t) {
                if (++work > budget || valid[f.rq + t * f.sa + (vv - f.cb) * f.sb]) { stop = true; break; }
            }
        }
        if (__any_sync(kAll, stop)) return false;
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (k == kf) T[k] = A;
        return true;
    }
    return false;
}

// circle_fits from the FP32 circle, as fits_clearly.
__device__ __forceinline__ int circle_fits_clearly(const float (&ctr)[2], float r2, int lo_u, int hi_u, int lo_v,
                                                   int hi_v, bool open_lu, bool open_hu, bool open_lv, bool open_hv) {
    const float rad = sqrtf(r2), tol = 1e-4f * (rad + 1.f);
    const float room[4] = {ctr[0] - rad - (float)lo_u + 1.f, (float)hi_u + 1.f - ctr[0] - rad,
                           ctr[1] - rad - (float)lo_v + 1.f, (float)hi_v + 1.f - ctr[1] - rad};
    const bool open[4] = {open_lu, open_hu, open_lv, open_hv};
    int fit = 1;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (open[m] && room[m] < -tol) return 0;
        if (open[m] && !(room[m] > tol)) fit = -1;
    }
    return fit;
}

// The walk of `walk` on a face: the window is the square of radius R around
// the entry, a row of it to each lane. Returns 1 with the triangle and q's
// barycentric coordinates, or 0.
__device__ __forceinline__ int walk2(int3 S, const uint8_t *__restrict__ valid, const int64_t (&c)[3], const Face &f,
                                     int R, bool &settled, LPt2 (&T)[3], double (&lam)[3]) {
    const int lane = threadIdx.x & 31, dv = lane - kMaxWindow2;
    const int64_t P = (int64_t)S.x * S.y * S.z;
    const LPt2 q0 = {0, 0, 0};
    const int u0 = max(f.ca - R, 0), u1 = min(f.ca + R, f.ea - 1), v0 = max(f.cb - R, 0), v1 = min(f.cb + R, f.eb - 1);
    const uint32_t row = face_row(f, R);
    const uint32_t rim = abs(dv) < R ? (1u << (kMaxWindow2 - R)) | (1u << (kMaxWindow2 + R)) : ~0u;
    const int r0 = f.rq + dv * f.sb - kMaxWindow2 * f.sa;   // the rank of bit k is r0 + k sa
    for (int it = 0; it < kMaxPivots; ++it) {
        float fc[2], fr2e;
        circumcircle_f(T, fc, fr2e);
        const float fc0 = fc[0], fv = (float)dv - fc[1];
        const float margin = fr2e * 8e-6f + 1e-3f, fr2 = fr2e + margin;   // as in walk
        const bool deep = it < kDeepPivots;   // the pivot rule of walk
        const uint32_t m = settled && it == 0 ? row & rim : row;
        const int split = (int)fminf(fmaxf(floorf(fc0), -(float)(kMaxWindow2 + 1)), (float)kMaxWindow2) + kMaxWindow2;
        const uint32_t lowbits = split < 0 ? 0u : (2u << split) - 1u;
        int64_t best = kNone;
        unsigned bhi = 0, blo = 0;
        auto scan = [&](bool exact) {
#pragma unroll
            for (int dir = 0; dir < 2; ++dir) {
                uint32_t w = dir ? m & ~lowbits : m & lowbits;
                while (w) {
                    const int k = dir ? __ffs(w) - 1 : 31 - __clz(w);
                    w &= ~(1u << k);
                    const float fu = (float)(k - kMaxWindow2) - fc0;
                    const float d2 = sum2(fu, fv);
                    const int r = r0 + k * f.sa;
                    const unsigned long long key = depth_key(fr2e - d2, r);
                    const unsigned khi = (unsigned)(key >> 32), klo = (unsigned)key;
                    if (khi < bhi) break;
                    if (exact && d2 > fr2) break;
                    if (khi == bhi && klo <= blo) continue;
                    if (exact) {
                        if (T[0].rank == (uint32_t)r || T[1].rank == (uint32_t)r || T[2].rank == (uint32_t)r) continue;
                        const LPt2 cand = {k - kMaxWindow2, dv, (uint32_t)r};
                        if (lifted_sign2(T, cand) <= 0) continue;
                    }
                    bhi = khi;
                    blo = klo;
                }
            }
        };
        if (deep) {
            scan(false);
            const unsigned sure = __reduce_max_sync(kAll, bhi);
            if (!(sure != 0 && depth_of(sure) > margin)) {
                bhi = blo = 0;
                scan(true);
            }
            const unsigned hi = __reduce_max_sync(kAll, bhi);
            const unsigned lo = __reduce_max_sync(kAll, bhi == hi ? blo : 0u);
            best = hi ? (int64_t)(0xffffffffu - lo) : kNone;
        } else {
            for (uint32_t w = m; w && best == kNone; w &= w - 1) {
                const int k = __ffs(w) - 1;
                const float fu = (float)(k - kMaxWindow2) - fc0;
                const int r = r0 + k * f.sa;
                if (sum2(fu, fv) > fr2 || T[0].rank == (uint32_t)r || T[1].rank == (uint32_t)r || T[2].rank == (uint32_t)r) continue;
                const LPt2 cand = {k - kMaxWindow2, dv, (uint32_t)r};
                if (lifted_sign2(T, cand) > 0) best = r;
            }
            best = warp_min(best);
        }
        const int64_t o = orient2(T[0], T[1], T[2]);   // > 0: T is kept counter-clockwise
        if (best == kNone) {
            settled = true;
            int64_t ol[3], ofar = 0;
            int nfar = 0, kf = -1;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                LPt2 u[3] = {T[0], T[1], T[2]};
                u[k] = q0;
                ol[k] = orient2(u[0], u[1], u[2]);
                if (T[k].rank >= (uint32_t)P) { ++nfar; kf = k; ofar = ol[k]; }
            }
            const LPt2 t3[3] = {T[0], T[1], T[2]};   // the copies keep T itself in registers
            if (nfar == 0) {
                const int fit = circle_fits_clearly(fc, fr2e, u0 - f.ca, u1 - f.ca, v0 - f.cb, v1 - f.cb, u0 > 0,
                                                    u1 < f.ea - 1, v0 > 0, v1 < f.eb - 1);
                if (fit == 0) return 0;
                if (fit < 0) {
                    double ctr[2], r2;
                    circumcircle(t3, ctr, r2);
                    if (!circle_fits(ctr, r2, S, c, f.a, f.b, u0, u1, v0, v1)) return 0;
                }
            } else if (nfar > 1 || ofar != 0) {
                return 0;
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) lam[k] = (double)ol[k] / (double)o;
            if (nfar == 0) return 1;
            LPt2 x3[3] = {T[0], T[1], T[2]};
            if (!across_edge(S, valid, c, f, R, x3, kf)) return 0;
#pragma unroll
            for (int k = 0; k < 3; ++k) T[k] = x3[k];
            return 1;
        }
        settled = false;
        int64_t bc[3];
        rank_coords(S, best, bc);
        const LPt2 e = {(int32_t)(f.a == 0 ? bc[0] : bc[1]) - f.ca, (int32_t)(f.b == 1 ? bc[1] : bc[2]) - f.cb, (uint32_t)best};
        int leave = -1;
        int64_t bq = 0, be = 0;
        uint32_t brank = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            LPt2 u[3] = {T[0], T[1], T[2]};
            u[k] = e;
            const int64_t oe = orient2(u[0], u[1], u[2]);
            if (oe <= 0) continue;
            u[k] = q0;
            const int64_t oq = orient2(u[0], u[1], u[2]);
            bool better = leave < 0;
            if (!better) {
                const int64_t lhs = oq * be, rhs = bq * oe;   // below 2^50
                better = lhs < rhs || (lhs == rhs && T[k].rank < brank);
            }
            if (better) { leave = k; bq = oq; be = oe; brank = T[k].rank; }
        }
        if (leave < 0) return 0;
        // the new orientation is be > 0: T stays counter-clockwise
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (k == leave) T[k] = e;
    }
    return 0;
}

// ---- Edges: nearest valid neighbours along the free axis a --------------
__device__ __noinline__ int edge_interp(int3 S, const uint8_t *__restrict__ valid, const int64_t (&c)[3], int a,
                           int64_t (&vtx)[4], double (&lam)[4]) {
    const int lane = threadIdx.x & 31;
    const int64_t ext[3] = {S.x, S.y, S.z};
    int64_t pc[3] = {c[0], c[1], c[2]};
    int64_t lo = -1, hi = kNone;
    for (int64_t t = c[a] - 1 - lane; t >= 0; t -= 32) {
        pc[a] = t;
        if (valid[lattice_rank(S, pc[0], pc[1], pc[2])]) { lo = t; break; }
    }
    for (int64_t t = c[a] + 1 + lane; t < ext[a]; t += 32) {
        pc[a] = t;
        if (valid[lattice_rank(S, pc[0], pc[1], pc[2])]) { hi = t; break; }
    }
    lo = warp_max(lo);
    hi = warp_min(hi);
    if (lo < 0 || hi == kNone) return 0;
    pc[a] = lo;
    vtx[0] = lattice_rank(S, pc[0], pc[1], pc[2]);
    pc[a] = hi;
    vtx[1] = lattice_rank(S, pc[0], pc[1], pc[2]);
    lam[0] = (double)(hi - c[a]) / (double)(hi - lo);
    lam[1] = (double)(c[a] - lo) / (double)(hi - lo);
    return 1;
}

// Writes the missing entry p (lane 0): the barycentric interpolant over the
// nv vertices of its simplex (status 2), or missing (NaN, status 0).
__device__ __forceinline__ void write_entry(int64_t P, int64_t p, bool ok, int nv, const int64_t (&vtx)[4],
                                            const double (&lam)[4], const float *__restrict__ ends,
                                            float *__restrict__ out, uint8_t *__restrict__ status) {
    if ((threadIdx.x & 31) != 0) return;
    if (!ok) {
        const float nan = __int_as_float(0x7fc00000);
        out[3 * p] = nan; out[3 * p + 1] = nan; out[3 * p + 2] = nan;
        if (status) status[p] = 0;
        return;
    }
    double acc[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (k >= nv) break;
        const int64_t v = vtx[k];
        if (v < 0 || v >= P) {   // never: both walks reject starting points
            (void)BTO_IN_BOUNDS(false, nullptr);
            continue;
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) acc[d] += lam[k] * (double)ends[3 * v + d];
    }
    out[3 * p] = (float)acc[0]; out[3 * p + 1] = (float)acc[1]; out[3 * p + 2] = (float)acc[2];
    if (status) status[p] = 2;
}

constexpr int kFillThreads = 128;
constexpr int kCopyTile = 4 * kFillThreads;   // entries of a CTA of the copy
// Tiles for each CTA in flight from which on those with missing entries are
// listed: below, the few waves of CTAs that find nothing cost no more than the
// list's memset (33 x 31 x 29, none missing: 16 us either way). 64^3, none
// missing: 18 us, 26 with a CTA to copy and look through each tile; 256^3: 94
// and 1,310.
constexpr int kListTiles = 4;
constexpr int kTileN = kTileX * kTileY * kTileZ;

// How the solver's tiles are listed: groups of w tiles along x by v along z
// (one tile where the list has the room), group (bx / w, by, bz / v) number
// bx / w + gx (by + ty (bz / v)). w == 0: no list. Counts and list stand in the
// out entries of the plane z = 0, which are written last (by the boundary
// kernel): words 0 to 2 are the dense groups, the others with missing interior
// entries, and the tiles the solver has taken; then the groups' counts of
// missing interior entries, 32 >> shift bits each, and the list, n words: the
// dense groups from its front, the others from its back.
struct Groups {
    int tx, ty, tz;   // tiles per axis
    int w, v;
    int gx;           // groups along x
    int n;            // groups
    int shift;        // log2 of the counts in a word
};
constexpr int kHead = 3;
__host__ __device__ __forceinline__ int count_words(const Groups &G) { return ((G.n - 1) >> G.shift) + 1; }
__device__ __forceinline__ int count_at(const Groups &G, unsigned g) {   // bit of g's count in its word
    return (int)(g & ((1u << G.shift) - 1u)) << (5 - G.shift);
}
// Missing entries from which on a group is dense, for each of its tiles (of 32
// entries). Over 24 lattices of 24 to 112 points an axis with losses at block
// faces, two inputs each, the fill takes 0.964 of the time with a CTA to each
// tile in lattice order (0.957 at 4, 0.963 at 12, 0.989 at 20, 1.017 without the
// order; 128^3 4.85 ms against 5.11), over 36 lattices with random and solid
// losses of 10% to all 1.004 (1.012, 1.010, 1.019).
constexpr int kDense = 8;

// Copies the valid entries (status 1) and counts the groups' missing interior
// entries. On a lattice one point thick, which has no tetrahedra, the missing
// entries are finished here. Bound by HBM: 16-byte accesses where the pointers
// allow it.
template <bool VEC>
__global__ void __launch_bounds__(kFillThreads) fill_copy_kernel(int3 S, const Groups G, bool flat,
                                                                 const float *__restrict__ ends,
                                                                 const uint8_t *__restrict__ valid,
                                                                 float *__restrict__ out,
                                                                 uint8_t *__restrict__ status) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the solver waits for this grid
    const int64_t P = (int64_t)S.x * S.y * S.z, skip = G.w ? (int64_t)S.x * S.y : 0;
    const int64_t t0 = (int64_t)blockIdx.x * kCopyTile;
    unsigned miss = 0;   // bit k: the thread's entry k is missing
    const bool vec = VEC && t0 >= skip && t0 + kCopyTile <= P;
    if (vec) {
        // ends and out 16-byte aligned, valid and status 4-byte: so is each tile
        const uchar4 v4 = reinterpret_cast<const uchar4 *>(valid + t0)[threadIdx.x];
        const uint8_t v[4] = {v4.x, v4.y, v4.z, v4.w};
        uint8_t st[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            st[k] = v[k] ? 1 : 0;
            miss |= v[k] ? 0u : 1u << k;
        }
        if (status) reinterpret_cast<uchar4 *>(status + t0)[threadIdx.x] = make_uchar4(st[0], st[1], st[2], st[3]);
        const float4 *src = reinterpret_cast<const float4 *>(ends + 3 * t0);
        float4 *dst = reinterpret_cast<float4 *>(out + 3 * t0);
#pragma unroll
        for (int k = 0; k < kCopyTile * 3 / 4 / kFillThreads; ++k)
            dst[k * kFillThreads + threadIdx.x] = src[k * kFillThreads + threadIdx.x];
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t p = t0 + k * kFillThreads + threadIdx.x;
            if (p >= P) continue;
            if (!valid[p]) {
                miss |= 1u << k;
                continue;
            }
            if (p >= skip) { out[3 * p] = ends[3 * p]; out[3 * p + 1] = ends[3 * p + 1]; out[3 * p + 2] = ends[3 * p + 2]; }
            if (status) status[p] = 1;
        }
    }
    if (flat) __syncthreads();   // the tile's copy before its missing entries' own values
    if (!miss || !(flat || G.w)) return;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (!(miss >> k & 1u)) continue;
        const int64_t p = vec ? t0 + 4 * threadIdx.x + k : t0 + k * kFillThreads + threadIdx.x;
        if (flat) {
            const float nan = __int_as_float(0x7fc00000);
            out[3 * p] = nan; out[3 * p + 1] = nan; out[3 * p + 2] = nan;
            if (status) status[p] = 0;
            continue;
        }
        const unsigned p32 = (unsigned)p, r = p32 / (unsigned)S.x;   // below 2^31
        const int x = (int)(p32 - r * (unsigned)S.x), y = (int)(r % (unsigned)S.y), z = (int)(r / (unsigned)S.y);
        if (x < 1 || x >= S.x - 1 || y < 1 || y >= S.y - 1 || z < 1 || z >= S.z - 1) continue;
        const unsigned g = (unsigned)(x / (kTileX * G.w) + G.gx * (y / kTileY + G.ty * (z / (kTileZ * G.v))));
        atomicAdd(reinterpret_cast<unsigned *>(out) + kHead + (g >> G.shift), 1u << count_at(G, g));
    }
}

// Lists the groups with missing entries, a group to a thread.
__global__ void __launch_bounds__(kFillThreads) fill_list_kernel(const Groups G, float *__restrict__ out) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the solver waits for this grid
    unsigned *head = reinterpret_cast<unsigned *>(out), *counts = head + kHead, *list = counts + count_words(G);
    const unsigned g = blockIdx.x * kFillThreads + threadIdx.x;
    const int lane = threadIdx.x & 31, bits = 32 >> G.shift;
    const unsigned c = g < (unsigned)G.n ? __ldcg(counts + (g >> G.shift)) >> count_at(G, g) & ((1u << bits) - 1u) : 0u;
    const unsigned some = __ballot_sync(kAll, c != 0);
    if (!some) return;
    const bool dense = c >= (unsigned)(kDense * G.w * G.v);
    const unsigned front = __ballot_sync(kAll, dense), back = some & ~front;
    unsigned at = 0;
    if (lane < 2 && (lane ? back : front)) at = atomicAdd(head + lane, (unsigned)__popc(lane ? back : front));
    const unsigned below = (1u << lane) - 1u, f0 = __shfl_sync(kAll, at, 0), b0 = __shfl_sync(kAll, at, 1);
    if (dense) list[f0 + __popc(front & below)] = g;
    else if (c) list[G.n - 1 - (b0 + __popc(back & below))] = g;
}

// Solves the missing interior entries. A CTA takes a tile: it collects the
// tile's missing interior entries, gathers the valid flags around it into
// shared words, and its warps then take the collected entries one at a time
// as they become free, all lanes on each. The tile is small because a slab's
// tile is what its four warps work through alone (8 x 4 x 2: 6.5 ms where this
// took 5.8, 16 x 4 x 4 a millisecond more again), and no smaller, since its
// entries share the words (8 x 2 x 1: 5.36 ms where this took 5.14). LISTED:
// the CTAs in flight take the tiles of the listed groups from a counter, the
// dense groups' first, since a tile full of missing entries that starts late
// is what the call then waits for; else every tile has a CTA, and the
// hardware hands them out.
// Bound by instructions: about 1,400 a pivot, a straight run of code far
// longer than the instruction caches hold (most stalls are instruction
// fetch), 16 pivots an entry. A 128^3 lattice with 137,210 missing entries
// (88,000 of them here), the whole fill: 61 ms with byte-wise window scans
// and one 32-entry chunk to a warp, 20 ms with the row words, 12 ms with the
// pivots' determinants and ratio test shared out, 5.8 ms with the certain
// pivots taken from the rows' nearest points, 32-bit minors, the row words in
// the facet test and the faces, and this tile.
template <bool LISTED>
__global__ void __launch_bounds__(kFillThreads, 4) fill_interior_kernel(int3 S, const Groups G,
                                                                     const float *__restrict__ ends,
                                                                     const uint8_t *__restrict__ valid,
                                                                     float *__restrict__ out,
                                                                     uint8_t *__restrict__ status) {
    __shared__ uint32_t words[kRowsY * kRowsZ];
    __shared__ uint8_t list[kTileN];
    __shared__ int count, next, tile[3];
    static_assert(kTileN <= 32, "an entry of the tile to a lane");
    const int64_t P = (int64_t)S.x * S.y * S.z;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    unsigned *head = reinterpret_cast<unsigned *>(out);
    const unsigned *listed = head + kHead + count_words(G);
    const unsigned sub = (unsigned)(G.w * G.v), front = LISTED ? __ldcg(head) : 0u,
                   total = LISTED ? (front + __ldcg(head + 1)) * sub : 0u;
#pragma unroll 1
    for (;;) {
        if (warp == 0) {
            int bx, by, bz;
            if (LISTED) {
                unsigned job = 0, g = 0;
                if (lane == 0) {
                    job = atomicAdd(head + 2, 1u);
                    const unsigned k = job / sub;
                    if (job < total) g = __ldcg(listed + (k < front ? k : G.n - 1 - (k - front)));
                }
                job = __shfl_sync(kAll, job, 0);
                g = __shfl_sync(kAll, g, 0);
                const int in = (int)(job % sub);
                bx = (int)(g % (unsigned)G.gx) * G.w + in % G.w;
                by = (int)(g / (unsigned)G.gx % (unsigned)G.ty);
                bz = (int)(g / (unsigned)G.gx / (unsigned)G.ty) * G.v + in / G.w;
                if (job >= total) bx = -1;   // none left
            } else {
                bx = (int)(blockIdx.x % G.tx);
                by = (int)(blockIdx.x / G.tx % G.ty);
                bz = (int)(blockIdx.x / G.tx / G.ty);
            }
            const int x = bx * kTileX + lane % kTileX, y = by * kTileY + lane / kTileX % kTileY,
                      z = bz * kTileZ + lane / (kTileX * kTileY);
            bool missing = false;
            if (lane < kTileN && x > 0 && x < S.x - 1 && y > 0 && y < S.y - 1 && z > 0 && z < S.z - 1)
                missing = !valid[lattice_rank(S, x, y, z)];
            const unsigned m = __ballot_sync(kAll, missing);
            if (missing) list[__popc(m & ((1u << lane) - 1u))] = (uint8_t)lane;
            if (lane == 0) {
                count = __popc(m);
                next = 0;
                tile[0] = bx;
                tile[1] = by;
                tile[2] = bz;
            }
        }
        __syncthreads();
        if (LISTED && tile[0] < 0) return;
        const int missing = count;
        if (missing) {
            const int cx0 = tile[0] * kTileX, cy0 = tile[1] * kTileY, cz0 = tile[2] * kTileZ;
            const int gx = cx0 - kMaxWindow + lane;
#pragma unroll 4
            for (int row = warp; row < kRowsY * kRowsZ; row += kFillThreads / 32) {
                const int y = cy0 - kMaxWindow + row % kRowsY, z = cz0 - kMaxWindow + row / kRowsY;
                bool v = false;
                if (gx >= 0 && gx < S.x && y >= 0 && y < S.y && z >= 0 && z < S.z) v = valid[lattice_rank(S, gx, y, z)] != 0;
                const unsigned w = __ballot_sync(kAll, v);
                if (lane == 0) words[row] = w;
            }
            __syncthreads();
            for (;;) {
                int at = 0;
                if (lane == 0) at = atomicAdd(&next, 1);
                at = __shfl_sync(kAll, at, 0);
                if (at >= missing) break;
                const int k = list[at];
                const int lx = k % kTileX, ly = k / kTileX % kTileY, lz = k / (kTileX * kTileY);
                const uint32_t *win = words + (ly + kMaxWindow) + kRowsY * (lz + kMaxWindow);
                const volatile int *t = tile;   // read again for each entry: the walk needs the registers
                const int cx = t[0] * kTileX + lx, cy = t[1] * kTileY + ly, cz = t[2] * kTileZ + lz;
                LPt T[4];
                double lam[4] = {0.0, 0.0, 0.0, 0.0};
                start_tetrahedron(P, T);
                int ok = 0;
                bool settled = false;
#pragma unroll 1
                for (int R = 2; R <= kMaxWindow && !ok; ++R)
                    ok = walk(S, valid, win, lx, cx, cy, cz, R, settled, T, lam);
                const int64_t vtx[4] = {T[0].rank, T[1].rank, T[2].rank, T[3].rank};
                write_entry(P, lattice_rank(S, cx, cy, cz), ok == 1, 4, vtx, lam, ends, out, status);
            }
        }
        if (!LISTED) return;
        __syncthreads();   // the tile's words and list are free again
    }
}

// The lattice's boundary points (fewer than 2^31), numbered: the z faces, then
// what the y faces, then what the x faces add.
struct Boundary {
    unsigned nz, ny, nx;
};
__host__ __device__ inline Boundary boundary_of(int3 S) {
    const unsigned zi = S.z > 2 ? S.z - 2 : 0, yi = S.y > 2 ? S.y - 2 : 0;
    return Boundary{(unsigned)S.x * S.y * (S.z > 1 ? 2 : 1), S.x * zi * (S.y > 1 ? 2 : 1), yi * zi * (S.x > 1 ? 2 : 1)};
}
__device__ __forceinline__ void boundary_point(int3 S, const Boundary &n, unsigned t, int (&c)[3]) {
    const unsigned sx = S.x, zi = S.z - 2, yi = S.y - 2;
    if (t < n.nz) {
        const unsigned r = t / sx, top = r >= (unsigned)S.y;
        c[0] = t - r * sx;
        c[1] = top ? r - S.y : r;
        c[2] = top ? S.z - 1 : 0;
        return;
    }
    t -= n.nz;
    if (t < n.ny) {
        const unsigned r = t / sx, top = r >= zi;
        c[0] = t - r * sx;
        c[2] = 1 + (top ? r - zi : r);
        c[1] = top ? S.y - 1 : 0;
        return;
    }
    t -= n.ny;
    const unsigned r = t / yi, top = r >= zi;
    c[1] = 1 + t - r * yi;
    c[2] = 1 + (top ? r - zi : r);
    c[0] = top ? S.x - 1 : 0;
}

// The missing boundary entries: a CTA takes `points` boundary points (4 to
// 128) and its warps solve the missing ones as they become free, all lanes on
// each. Where the plane z = 0 has held the solver's list (`plane0`), its valid
// entries are copied here.
__global__ void __launch_bounds__(kFillThreads) fill_boundary_kernel(int3 S, int points, bool plane0,
                                                                     const float *__restrict__ ends,
                                                                     const uint8_t *__restrict__ valid,
                                                                     float *__restrict__ out,
                                                                     uint8_t *__restrict__ status) {
    __shared__ uint8_t list[kFillThreads];
    __shared__ int count, next;
    const int64_t P = (int64_t)S.x * S.y * S.z;
    const Boundary n = boundary_of(S);
    const unsigned total = n.nz + n.ny + n.nx, t0 = blockIdx.x * (unsigned)points;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) count = next = 0;
    // Waits for the solver. Started beside the solver's last tiles, on points
    // off the list's plane, it made the whole fill 3% slower: two kernels that
    // are bound by instruction fetch then share the caches.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    if ((int)threadIdx.x < points && t0 + threadIdx.x < total) {
        int c[3];
        boundary_point(S, n, t0 + threadIdx.x, c);
        const int64_t p = lattice_rank(S, c[0], c[1], c[2]);
        if (!valid[p]) {
            list[atomicAdd(&count, 1)] = (uint8_t)threadIdx.x;
        } else if (plane0 && c[2] == 0) {
            out[3 * p] = ends[3 * p]; out[3 * p + 1] = ends[3 * p + 1]; out[3 * p + 2] = ends[3 * p + 2];
        }
    }
    __syncthreads();
    for (;;) {
        int at = 0;
        if (lane == 0) at = atomicAdd(&next, 1);
        at = __shfl_sync(kAll, at, 0);
        if (at >= count) break;
        int c32[3];
        boundary_point(S, n, t0 + list[at], c32);
        const int64_t c[3] = {c32[0], c32[1], c32[2]};
        const int64_t p = lattice_rank(S, c[0], c[1], c[2]);
        const bool fixed[3] = {c[0] == 0 || c[0] == S.x - 1, c[1] == 0 || c[1] == S.y - 1,
                               c[2] == 0 || c[2] == S.z - 1};
        const int nfix = (int)fixed[0] + (int)fixed[1] + (int)fixed[2];
        int64_t vtx[4] = {-1, -1, -1, 0};
        double lam[4] = {0.0, 0.0, 0.0, 0.0};
        int nv = 0, ok = 0;   // three fixed axes: a corner
        if (nfix == 1) {
            const int a = fixed[0] ? 1 : 0, b = fixed[2] ? 1 : 2;
            LPt2 T2[3];
            double l2[3];
            start_triangle(P, T2);
            const Face f = face_of(S, valid, c, a, b);
            bool settled = false;
            for (int R = 2; R <= kMaxWindow2 && !ok; ++R) ok = walk2(S, valid, c, f, R, settled, T2, l2);
            for (int k = 0; k < 3; ++k) { vtx[k] = T2[k].rank; lam[k] = l2[k]; }
            nv = 3;
        } else if (nfix == 2) {
            const int a = !fixed[0] ? 0 : (!fixed[1] ? 1 : 2);
            ok = edge_interp(S, valid, c, a, vtx, lam);
            nv = 2;
        }
        write_entry(P, p, ok == 1, nv, vtx, lam, ends, out, status);
    }
}

}  // namespace

BTO_BOUNDS_ACCESSOR(bounds_failures_delaunay)

// The solver's groups: as few tiles to a group as let counts and list fit the
// plane z = 0 of out; w == 0 when none does.
static Groups groups_of(const int32_t S[3]) {
    Groups G{};
    G.tx = (S[0] + kTileX - 1) / kTileX;
    G.ty = (S[1] + kTileY - 1) / kTileY;
    G.tz = (S[2] + kTileZ - 1) / kTileZ;
    const int64_t words = 3 * (int64_t)S[0] * S[1];
    for (int size = 1; size <= 65536 / kTileN; size *= 2) {
        G.w = size < 4 ? size : 4;
        if (G.w > G.tx) G.w = G.tx;
        G.v = size / G.w;
        if (G.v > G.tz) G.v = G.tz;
        G.gx = (G.tx + G.w - 1) / G.w;
        const int64_t n = (int64_t)G.gx * G.ty * ((G.tz + G.v - 1) / G.v);
        G.shift = kTileN * G.w * G.v < 256 ? 2 : 1;
        if (kTileN * G.w * G.v >= 65536) break;
        if (kHead + ((n - 1) >> G.shift) + 1 + n <= words) {
            G.n = (int)n;
            return G;
        }
    }
    G.w = 0;
    return G;
}

// A launch that may start once every CTA of the kernel before it has started.
template <class... Params, class... Args>
static cudaError_t launch_after(void (*kernel)(Params...), int64_t grid, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kFillThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

cudaError_t launch_fill_delaunay(const int32_t S[3], const float *ends, const uint8_t *valid, float *out,
                                 uint8_t *status, int sm_count, cudaStream_t s) {
    const int3 S3 = make_int3(S[0], S[1], S[2]);
    const int64_t P = (int64_t)S[0] * S[1] * S[2];
    const bool flat = S[0] == 1 || S[1] == 1 || S[2] == 1;
    const bool inner = S[0] > 2 && S[1] > 2 && S[2] > 2;
    const int64_t tiles = (int64_t)((S[0] + kTileX - 1) / kTileX) * ((S[1] + kTileY - 1) / kTileY) * ((S[2] + kTileZ - 1) / kTileZ);
    const int64_t resident = 4ll * sm_count;
    const bool apart = out + 3 * P <= ends || ends + 3 * P <= out;   // the list would spoil ends
    Groups G = groups_of(S);
    const bool listed = inner && apart && tiles > kListTiles * resident && G.w > 0;
    if (listed) {
        const cudaError_t e = cudaMemsetAsync(out, 0, sizeof(uint32_t) * (kHead + count_words(G)), s);
        if (e != cudaSuccess) return e;
    } else {
        G.w = 0;
    }
    const unsigned copies = (unsigned)((P + kCopyTile - 1) / kCopyTile);
    const bool vec = !((reinterpret_cast<uintptr_t>(ends) | reinterpret_cast<uintptr_t>(out)) & 15u) &&
                     !((reinterpret_cast<uintptr_t>(valid) | reinterpret_cast<uintptr_t>(status)) & 3u);
    if (vec)
        fill_copy_kernel<true><<<copies, kFillThreads, 0, s>>>(S3, G, flat, ends, valid, out, status);
    else
        fill_copy_kernel<false><<<copies, kFillThreads, 0, s>>>(S3, G, flat, ends, valid, out, status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || flat) return e;
    if (listed) e = launch_after(fill_list_kernel, (G.n + kFillThreads - 1) / kFillThreads, s, G, out);
    if (e != cudaSuccess) return e;
    if (listed)
        e = launch_after(fill_interior_kernel<true>, resident, s, S3, G, ends, valid, out, status);
    else if (inner)
        e = launch_after(fill_interior_kernel<false>, tiles, s, S3, G, ends, valid, out, status);
    if (e != cudaSuccess) return e;
    const Boundary n = boundary_of(S3);
    const int64_t total = (int64_t)n.nz + n.ny + n.nx;
    // Points of a CTA: its warps share a run of missing ones, so few where
    // those bound the call (40^3 with losses at every face: 348 us with 4, 396
    // with 16; 128^3: 5.30 ms with 4, 5.34 with 8, 5.41 with 64), and more
    // where the CTAs that find nothing do (none missing: 128^3 39 us with 4,
    // 27 with 8, 20 with 16; 256^3 201, 138, 105, and 89 with 32).
    int points = total <= 16 * resident ? 4 : 8;
    while (points < kFillThreads && total > 32 * resident * points) points *= 2;
    return launch_after(fill_boundary_kernel, (total + points - 1) / points, s, S3, points, listed, ends, valid, out,
                        status);
}

}  // namespace bto

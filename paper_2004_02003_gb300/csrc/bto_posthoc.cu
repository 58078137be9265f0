// Post hoc kernels of libbto for sm_103a (Sec. 3.2): reconstruction of
// missing basis flows on the seed lattice (row f2) and pathline stitching
// through successive intervals' basis flows (row f3). They run after the
// in situ intervals, on their outputs, and share no code with the
// advection kernels.
#include <climits>
#include <cstdint>
#include <cuda_runtime.h>

#include "bto_internal.h"

namespace bto {
namespace {

constexpr int kFillThreads = 128;
constexpr int kFillTile = 4 * kFillThreads;   // entries of a CTA
constexpr int kNear = 16;                      // points of the first search along an axis

// Post hoc lattice reconstruction (Sec. 3.2 / Sec. 3.3, Eq. 2): a missing
// basis flow at lattice point J takes, along the axis whose nearest valid
// neighbours on both sides are closest (a + b smallest; ties x, y, z), the
// linear interpolant (Eq. 1) of their end positions at J:
//   end(J) = (b end(J - a e) + a end(J + b e)) / (a + b).
// Eq. (2): interpolating from the filled value afterwards equals
// interpolating from the two neighbours directly. Entries with no axis
// holding valid neighbours on both sides stay missing.
//
// A CTA takes a tile of kFillTile consecutive entries. It copies the tile
// with 16-byte accesses (valid entries keep that copy) and collects its
// missing entries in shared memory; then its threads share the collected
// entries out, one each, so that the neighbour search, whose instructions
// and load latencies are what the kernel's time goes into, runs with full
// warps although missing entries come in slabs a few points thick. An entry
// first looks kNear points far along every axis, from the nearer lattice face
// on and no further than could still give a smaller a + b; only then beyond,
// so that a slab is crossed along its normal instead of being walked along
// its whole extent.
// A 192 x 200 x 177 lattice with 4% missing: 66 us a fill, 69 us without the
// bounds of the first look, 143 us in tiles of 2048 (the rounds of a tile
// inside a slab are its tail), 281 us with one thread to every entry of the
// lattice and each axis searched to its end.

// The first r in [from, to] with a valid neighbour r steps away, 0 when none;
// four independent loads at a time.
__device__ __forceinline__ int first_valid(const uint8_t *__restrict__ v, int64_t step, int from, int to) {
    for (int r = from; r <= to; r += 4) {
        const uint8_t b0 = v[r * step], b1 = r + 1 <= to ? v[(r + 1) * step] : 0,
                      b2 = r + 2 <= to ? v[(r + 2) * step] : 0, b3 = r + 3 <= to ? v[(r + 3) * step] : 0;
        if (b0 | b1 | b2 | b3) return b0 ? r : (b1 ? r + 1 : (b2 ? r + 2 : r + 3));
    }
    return 0;
}

template <bool VEC>
__global__ void __launch_bounds__(kFillThreads) fill_lattice_kernel(int3 S, const float *__restrict__ ends,
                                                                    const uint8_t *__restrict__ valid,
                                                                    float *__restrict__ out,
                                                                    uint8_t *__restrict__ status) {
    __shared__ uint16_t list[kFillTile];
    __shared__ int count;
    const int64_t P = (int64_t)S.x * S.y * S.z;
    const int64_t t0 = (int64_t)blockIdx.x * kFillTile;
    const int n = (int)(P - t0 < kFillTile ? P - t0 : kFillTile);
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    if (VEC && n == kFillTile) {
        // every pointer is 16-byte aligned (status and valid: 4-byte), and so is each tile
#pragma unroll
        for (int q = 0; q < kFillTile / (4 * kFillThreads); ++q) {
            const int at = q * kFillThreads + threadIdx.x;   // four entries
            const uchar4 v4 = reinterpret_cast<const uchar4 *>(valid + t0)[at];
            const uint8_t v[4] = {v4.x, v4.y, v4.z, v4.w};
            uint8_t st[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                st[k] = v[k] ? 1 : 0;
                if (!v[k]) list[atomicAdd(&count, 1)] = (uint16_t)(4 * at + k);
            }
            if (status) reinterpret_cast<uchar4 *>(status + t0)[at] = make_uchar4(st[0], st[1], st[2], st[3]);
        }
        const float4 *src = reinterpret_cast<const float4 *>(ends + 3 * t0);
        float4 *dst = reinterpret_cast<float4 *>(out + 3 * t0);
#pragma unroll 6
        for (int k = 0; k < kFillTile * 3 / 4 / kFillThreads; ++k)
            dst[k * kFillThreads + threadIdx.x] = src[k * kFillThreads + threadIdx.x];
    } else {
        // a small lattice waits for its last tile alone: the four entries of
        // a thread are loaded together, the missing ones' ends for nothing
        // (33 x 31 x 29: 10.9 us with one entry after another, 8.9 so)
        constexpr int kPer = kFillTile / kFillThreads;
        uint8_t v[kPer];
        float e[kPer][3];
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int i = k * kFillThreads + threadIdx.x;
            const int64_t p = t0 + (i < n ? i : 0);
            v[k] = valid[p];
#pragma unroll
            for (int d = 0; d < 3; ++d) e[k][d] = ends[3 * p + d];
        }
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int i = k * kFillThreads + threadIdx.x;
            const int64_t p = t0 + i;
            if (i >= n) continue;
            if (v[k]) {
                out[3 * p] = e[k][0]; out[3 * p + 1] = e[k][1]; out[3 * p + 2] = e[k][2];
                if (status) status[p] = 1;
            } else {
                list[atomicAdd(&count, 1)] = (uint16_t)i;
            }
        }
    }
    __syncthreads();   // also orders the tile's copy before the missing entries' own values
    const int missing = count;
    for (int m = threadIdx.x; m < missing; m += kFillThreads) {
        const int64_t p = t0 + list[m];
        const unsigned p32 = (unsigned)p, row = p32 / (unsigned)S.x;   // below 2^31
        const int jx = (int)(p32 - row * (unsigned)S.x), jy = (int)(row % (unsigned)S.y), jz = (int)(row / (unsigned)S.y);
        const int el[3] = {jx, jy, jz}, eh[3] = {S.x - 1 - jx, S.y - 1 - jy, S.z - 1 - jz};   // points on either side
        const int64_t step[3] = {1, S.x, (int64_t)S.x * S.y};
        // lo, hi: distance to the nearest valid neighbour (0: none found yet)
        int lo[3], hi[3];
        int best_axis = 3, best = INT_MAX;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            // the nearer face's side first: without a neighbour there the
            // other side is not needed; neither is looked at farther than
            // could still give a smaller sum
            const bool down = el[ax] <= eh[ax];
            const int near_reach = down ? el[ax] : eh[ax], far_reach = down ? eh[ax] : el[ax];
            const int64_t st = down ? -step[ax] : step[ax];
            const int a = first_valid(valid + p, st, 1, min(min(near_reach, kNear), best - 2));
            int b = 0;
            if (a || near_reach > kNear) b = first_valid(valid + p, -st, 1, min(min(far_reach, kNear), best - (a ? a : 1) - 1));
            lo[ax] = down ? a : b;
            hi[ax] = down ? b : a;
            if (a && b) { best_axis = ax; best = a + b; }
        }
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            if (lo[ax] && hi[ax]) continue;
            // a side that has been searched to the lattice's face has no neighbour
            if ((!lo[ax] && el[ax] <= kNear) || (!hi[ax] && eh[ax] <= kNear)) continue;
            // the largest a + b that would replace the best (ties go to the lower axis)
            const int most = ax < best_axis ? best : best - 1;
            if (!lo[ax]) lo[ax] = first_valid(valid + p, -step[ax], kNear + 1, min(el[ax], most - (hi[ax] ? hi[ax] : kNear + 1)));
            if (!lo[ax]) continue;
            if (!hi[ax]) hi[ax] = first_valid(valid + p, step[ax], kNear + 1, min(eh[ax], most - lo[ax]));
            if (hi[ax] && lo[ax] + hi[ax] <= most) { best_axis = ax; best = lo[ax] + hi[ax]; }
        }
        if (best_axis == 3) best_axis = -1;
        if (best_axis < 0) {
            const float nan = __int_as_float(0x7fc00000);
            out[3 * p] = nan; out[3 * p + 1] = nan; out[3 * p + 2] = nan;
            if (status) status[p] = 0;
            continue;
        }
        const int a = best_axis == 0 ? lo[0] : (best_axis == 1 ? lo[1] : lo[2]);
        const int b = best_axis == 0 ? hi[0] : (best_axis == 1 ? hi[1] : hi[2]);
        const int64_t st = best_axis == 0 ? step[0] : (best_axis == 1 ? step[1] : step[2]);
        int64_t pl = p - a * st, pr = p + b * st;
        if (!BTO_IN_BOUNDS(pl >= 0 && pr < P, nullptr)) pl = pr = p;
        const float wl = (float)b / (float)(a + b), wr = (float)a / (float)(a + b);
#pragma unroll
        for (int k = 0; k < 3; ++k) out[3 * p + k] = wl * ends[3 * pl + k] + wr * ends[3 * pr + k];
        if (status) status[p] = 2;
    }
}

// Pathline stitching (Sec. 3.2): a new particle follows the basis flows of
// successive intervals. At the start of interval k it sits in a cell of the
// seed lattice; its position at the end of the interval interpolates the end
// positions of that cell's basis flows:
//   trilinear    the 8 corners, Eq. 1 per axis;
//   barycentric  the 4 vertices of the cell's Kuhn tetrahedron holding it
//                (the paper's barycentric coordinates over a Delaunay
//                neighbourhood; the cells of a full lattice are cospherical,
//                so the Kuhn split is a Delaunay triangulation): with the
//                fractional coordinates sorted t_a >= t_b >= t_c (a stable
//                sort, ties in axis order), vertices 0, e_a, e_a + e_b,
//                (1, 1, 1) and weights 1 - t_a, t_a - t_b, t_b - t_c, t_c.
// A particle outside the lattice, or next to a missing basis flow (NaN) that
// its interpolant uses, stops: its later positions are NaN.
template <bool BARY>
__global__ void stitch_kernel(int3 S, float3 origin, float3 inv_sp, int32_t intervals,
                              const float *const *__restrict__ ends_table, int64_t nq,
                              const float *__restrict__ start, float *__restrict__ path) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const float nan = __int_as_float(0x7fc00000);
    const int64_t P = (int64_t)S.x * S.y * S.z;
    (void)P;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nq; i += stride) {
        float x = start[3 * i], y = start[3 * i + 1], z = start[3 * i + 2];
        path[3 * i] = x; path[3 * i + 1] = y; path[3 * i + 2] = z;
        for (int32_t k = 0; k < intervals; ++k) {
            float nx = nan, ny = nan, nz = nan;
            const float u = (x - origin.x) * inv_sp.x, v = (y - origin.y) * inv_sp.y, w = (z - origin.z) * inv_sp.z;
            const bool in = u >= 0.f && v >= 0.f && w >= 0.f && u <= (float)(S.x - 1) &&
                            v <= (float)(S.y - 1) && w <= (float)(S.z - 1);
            if (in) {
                const int ix = min((int)u, max(S.x - 2, 0)), iy = min((int)v, max(S.y - 2, 0)),
                          iz = min((int)w, max(S.z - 2, 0));
                const float fx = u - ix, fy = v - iy, fz = w - iz;
                const float *E = ends_table[k];
                float acc[3] = {0.f, 0.f, 0.f};
                if (BARY) {
                    // stable descending sort of (fx, fy, fz) with the axes
                    int ax[3] = {0, 1, 2};
                    float t[3] = {fx, fy, fz};
                    if (t[1] > t[0]) { float q = t[0]; t[0] = t[1]; t[1] = q; int r = ax[0]; ax[0] = ax[1]; ax[1] = r; }
                    if (t[2] > t[1]) {
                        float q = t[1]; t[1] = t[2]; t[2] = q; int r = ax[1]; ax[1] = ax[2]; ax[2] = r;
                        if (t[1] > t[0]) { q = t[0]; t[0] = t[1]; t[1] = q; r = ax[0]; ax[0] = ax[1]; ax[1] = r; }
                    }
                    int j[3] = {ix, iy, iz};
                    const int ext[3] = {S.x, S.y, S.z};
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        if (m > 0) j[ax[m - 1]] = min(j[ax[m - 1]] + 1, ext[ax[m - 1]] - 1);
                        const float wgt = m == 0 ? 1.f - t[0] : (m == 3 ? t[2] : t[m - 1] - t[m]);
                        int64_t p = j[0] + (int64_t)S.x * (j[1] + (int64_t)S.y * j[2]);
                        if (!BTO_IN_BOUNDS(p >= 0 && p < P, nullptr)) p = 0;
#pragma unroll
                        for (int d = 0; d < 3; ++d) acc[d] = fmaf(wgt, E[3 * p + d], acc[d]);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 2; ++c)
#pragma unroll
                        for (int b = 0; b < 2; ++b)
#pragma unroll
                            for (int a = 0; a < 2; ++a) {
                                const int jx = min(ix + a, S.x - 1), jy = min(iy + b, S.y - 1), jz = min(iz + c, S.z - 1);
                                const float wgt = (a ? fx : 1.f - fx) * (b ? fy : 1.f - fy) * (c ? fz : 1.f - fz);
                                int64_t p = jx + (int64_t)S.x * (jy + (int64_t)S.y * jz);
                                if (!BTO_IN_BOUNDS(p >= 0 && p < P, nullptr)) p = 0;
#pragma unroll
                                for (int d = 0; d < 3; ++d) acc[d] = fmaf(wgt, E[3 * p + d], acc[d]);
                            }
                }
                nx = acc[0]; ny = acc[1]; nz = acc[2];
            }
            x = nx; y = ny; z = nz;
            const int64_t o = 3 * ((int64_t)(k + 1) * nq + i);
            path[o] = x; path[o + 1] = y; path[o + 2] = z;
        }
    }
}

}  // namespace

BTO_BOUNDS_ACCESSOR(bounds_failures_posthoc)

cudaError_t launch_stitch(const int32_t S[3], const float origin[3], const float spacing[3], int32_t intervals,
                          const float *const *ends_table, int64_t nq, const float *start, float *path, int grid,
                          cudaStream_t s, bool barycentric) {
    const int3 S3 = make_int3(S[0], S[1], S[2]);
    const float3 o = make_float3(origin[0], origin[1], origin[2]);
    const float3 inv = make_float3(1.f / spacing[0], 1.f / spacing[1], 1.f / spacing[2]);
    if (barycentric)
        stitch_kernel<true><<<grid, 256, 0, s>>>(S3, o, inv, intervals, ends_table, nq, start, path);
    else
        stitch_kernel<false><<<grid, 256, 0, s>>>(S3, o, inv, intervals, ends_table, nq, start, path);
    return cudaGetLastError();
}

cudaError_t launch_fill_lattice(const int32_t S[3], const float *ends, const uint8_t *valid, float *out,
                                uint8_t *status, cudaStream_t s) {
    const int64_t P = (int64_t)S[0] * S[1] * S[2];
    const int grid = (int)((P + kFillTile - 1) / kFillTile);
    const int3 S3 = make_int3(S[0], S[1], S[2]);
    const bool vec = !((reinterpret_cast<uintptr_t>(ends) | reinterpret_cast<uintptr_t>(out)) & 15u) &&
                     !((reinterpret_cast<uintptr_t>(valid) | reinterpret_cast<uintptr_t>(status)) & 3u);
    if (vec)
        fill_lattice_kernel<true><<<grid, kFillThreads, 0, s>>>(S3, ends, valid, out, status);
    else
        fill_lattice_kernel<false><<<grid, kFillThreads, 0, s>>>(S3, ends, valid, out, status);
    return cudaGetLastError();
}

}  // namespace bto

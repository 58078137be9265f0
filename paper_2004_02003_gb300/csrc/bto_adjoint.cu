// K7: checkpointed discrete adjoint of one BTO interval.
//
// Forward: particles start at caller-given positions (the lattice seeds for a
// flow map, Sec. 2.3) and take one RK4 step per cycle through that cycle's
// field, with the closed-box termination of the advection kernel (the same
// device functions, bto_device.cuh). The interval is cut into segments of C
// cycles; positions are kept at the start of each.
//
// Backward: a cycle's effect on an adjoint is linear, so a whole segment's is
// one 3 x 3 matrix, M_s = d x(end of s) / d x(start of s), that depends on
// the positions only. All segments of all particles are therefore worked on
// at once, in three steps:
//   tangent  M_s of every (segment, particle), by forward tangents from the
//            segment's checkpoint;
//   chain    per particle, last segment to first: the adjoint at the end of
//            every segment, lam_(s-1) = M_s^T lam_s, and dL/d(start); for the
//            flow-map Jacobian the product of the M_s instead;
//   scatter  (only with field gradients) every (segment, particle) recomputes
//            its positions, then reverses its cycles and adds the node
//            velocity gradients (atomics).
// One thread carrying a particle's adjoint back through the interval, as a
// serial sweep, left 32,768 particles x 200 cycles (7 warps per SM) waiting
// on 2 x 4 x 200 dependent samples. Measured on 64^3 cells: the Jacobian of
// 100,003 particles over 50 cycles 2.43 -> 0.20 ms (three serial sweeps
// against tangents and product), the gradients of 32,768 over 200 cycles
// 1.97 -> 1.08 ms (0.24 tangents, 0.01 chain, 0.83 scatter). Tangents and
// scatter are bound by the L1 load path (73-74% of its wavefront peak).
// A terminated particle's end is its last in-block position, so its gradient
// flows back only through the cycles before its exit cycle.
//
// Particles are kept in the order of the cells they start in (a counting
// sort by bins of 32 x 1 x 1 cells, or larger ones in a large block): a
// caller's particles can come in any order, and a warp whose lanes start
// all over the block touches 32 lines with each of a cell's 24 corner
// loads (forward of 100,003 random particles over 50 cycles: 299 -> 244 us, and 19 us
// for the sort).
//
// Reverse of x' = x + s/6 (k1 + 2 k2 + 2 k3 + k4) (cell units, s = dt/h),
// k1 = v(x), k2 = v(x + s/2 k1), k3 = v(x + s/2 k2), k4 = v(x + s k3),
// given lam = dL/dx':  g1 = s/6 lam, g2 = g3 = s/3 lam, g4 = s/6 lam;
// stage 4, 3, 2: qbar = (dv/dq)^T g; lam_x += qbar; previous stage's g gets
// (s or s/2) qbar; stage 1: lam = lam_x + (dv/dx)^T g1. Every stage adds its
// trilinear weights times g to the 8 corner nodes' velocity gradients.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <new>

#include <cuda_runtime.h>

#include "../../include/bto.h"
#include "bto_device.cuh"
#include "bto_internal.h"

using bto::BlockDev;

struct bto_tape {
    bto::DevAlloc mem;           // device allocator captured at creation
    int device = 0;
    int sm_count = 0;
    BlockDev B{};
    int64_t P = 0;
    int32_t L = 0, C = 0, nseg = 0;   // cycles, cycles per segment, segments
    float4 *ckpt = nullptr;     // nseg * P positions (cell units) at cycles 0, C, 2C, ...
    float *mat = nullptr;       // nseg * 9 * P segment matrices, row-major planes; the chain leaves a
                                // segment's end adjoint in the first three of its planes
    BlockDev *d_block = nullptr;
    int32_t *exitc = nullptr;   // P exit cycle, -1 while valid
    int32_t *perm = nullptr;    // P: the caller's index of each particle in cell order
    int32_t *bins = nullptr;    // 2 * kMaxBins: counts and starts of the sort
    int bsh[3] = {0, 0, 0};     // log2 of a bin's cells per axis
    int bn[3] = {1, 1, 1};      // bins per axis
    const void *const *table = nullptr;
    float dt = 0.f;
    bool have_forward = false;
};

namespace {

using namespace bto::dev;

constexpr int kMaxBins = 16384;      // bins of the sort: one CTA scans them, 16 a thread
// Whether a forward sorts its particles. The sort costs 9 us and more with the
// particles, and pays by every cycle after it, in the forward and in the
// backward calls: never in one or two cycles (forward of 1M particles over 1:
// 111 us sorted, 64 not; 20,000 over 2: 28 and 15), below 10 from about
// 400,000 particle-cycles on (forward and field gradients of 60,000 over 8:
// 140 and 156 us, 60,000 over 4: 95 and 99, the forward alone 38 and 27;
// 200,000 over 4: 175 and 224), then in all but small calls.
inline bool sorts(int64_t P, int32_t L) {
    return L >= 10 ? P >= 2048 : L >= 3 && P * L >= 400000;
}
constexpr int kThreads = 128;
// Up to this many particles per SM the forward takes four lanes for each: on
// 152 SMs 20,000 particles over 50 cycles (the whole FTLE call) 359 us with
// one lane, 326 with four, 2,000 258 and 216; 50,000 434 and 503; the forward
// of 32,768 over 200 cycles 419 and 432.
constexpr int64_t kQuadPerSm = 132;
// Positions a thread of the scatter kernel holds: of up to kChunk consecutive
// cycles and, in segments longer than that, of up to kSubs cycles spaced over
// the segment to restart from (48 KB a CTA together).
constexpr int kChunk = 24;
constexpr int kSubs = 8;

struct Stage {
    int ix, iy, iz;
    float fx, fy, fz;
};

// Corners of the cell last sampled, v[a + 2b + 4c][component]: the stages of
// a step mostly stay in one cell.
struct JCell {
    uint32_t node;   // ~0u when empty
    float v[8][3];
};

// cell_coord for any point, NaN and infinities included: the index is clamped
// at both ends. A backward call retraces the forward's points, which are in
// the box, only while the fields hold what they held then; where they have
// been written since, its points may lie anywhere, and the nodes it reads and
// adds to still are the block's.
__device__ __forceinline__ void cell_coord_any(float x, float cm, int &i, float &f) {
    const float t = fminf(fmaxf(__fadd_rd(x, 8388608.f), 8388608.f), cm);
    i = __float_as_int(t) - 0x4B000000;
    f = x - (t - 8388608.f);
}

// Trilinear value, its Jacobian d v / d xi (cell units) and the cell.
__device__ __forceinline__ void sample_jac(JCell &C, const float *__restrict__ f, const Geo &g, float x, float y,
                                           float z, float3 &v, float (&J)[3][3], Stage &st) {
    cell_coord_any(x, g.cmx, st.ix, st.fx);
    cell_coord_any(y, g.cmy, st.iy, st.fy);
    cell_coord_any(z, g.cmz, st.iz, st.fz);
    const uint32_t node = (uint32_t)st.ix + g.nnx * (uint32_t)st.iy + g.nnxy * (uint32_t)st.iz;
    if (node != C.node) {
        load_cell<bto::LAYOUT_F3>(f, g.nnx, g.nnxy, g.nodes, st.ix, st.iy, st.iz, C.v);
        C.node = node;
    }
    const float (&c)[8][3] = C.v;
    v = trilerp(c, st.fx, st.fy, st.fz);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        // d/dfx: x-differences blended in y, z; likewise for y and z
        const float dx00 = c[1][k] - c[0][k], dx10 = c[3][k] - c[2][k];
        const float dx01 = c[5][k] - c[4][k], dx11 = c[7][k] - c[6][k];
        J[k][0] = lerp1(lerp1(dx00, dx10, st.fy), lerp1(dx01, dx11, st.fy), st.fz);
        const float dy0 = lerp1(c[2][k], c[3][k], st.fx) - lerp1(c[0][k], c[1][k], st.fx);
        const float dy1 = lerp1(c[6][k], c[7][k], st.fx) - lerp1(c[4][k], c[5][k], st.fx);
        J[k][1] = lerp1(dy0, dy1, st.fz);
        const float z0 = lerp1(lerp1(c[0][k], c[1][k], st.fx), lerp1(c[2][k], c[3][k], st.fx), st.fy);
        const float z1 = lerp1(lerp1(c[4][k], c[5][k], st.fx), lerp1(c[6][k], c[7][k], st.fx), st.fy);
        J[k][2] = z1 - z0;
    }
}

__device__ __forceinline__ float3 jt_times(const float (&J)[3][3], float3 gvec) {
    return make_float3(J[0][0] * gvec.x + J[1][0] * gvec.y + J[2][0] * gvec.z,
                       J[0][1] * gvec.x + J[1][1] * gvec.y + J[2][1] * gvec.z,
                       J[0][2] * gvec.x + J[1][2] * gvec.y + J[2][2] * gvec.z);
}

// Exit cycle e as the number of cycles a particle moved in, at most L.
__device__ __forceinline__ int32_t cycles_moved(int32_t e, int32_t L) { return e < 0 ? L : e; }

// The last segment a particle moved in, -1 when it never moved.
__device__ __forceinline__ int32_t last_segment(int32_t e, int32_t L, int32_t C) {
    const int32_t moved = cycles_moved(e, L);
    return moved > 0 ? (moved - 1) / C : -1;
}

struct Bins {
    int sh[3];
    int n[3];
};

__device__ __forceinline__ float4 start_of(const BlockDev &B, const float *__restrict__ seeds, int64_t i) {
    return make_float4((seeds[3 * i + 0] - B.origin[0]) * B.inv_h[0], (seeds[3 * i + 1] - B.origin[1]) * B.inv_h[1],
                       (seeds[3 * i + 2] - B.origin[2]) * B.inv_h[2], 0.f);
}

// Sort, step 1: each particle's bin (a start outside the block goes to bin
// 0) and its place in it, in arrival order.
__global__ void tape_bin_kernel(const BlockDev *__restrict__ blk, int64_t P, const float *__restrict__ seeds, Bins bins,
                                int32_t *__restrict__ count, int2 *__restrict__ place) {
    const BlockDev &B = *blk;
    const Geo g = load_geo(B);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 x = start_of(B, seeds, i);
        int key = 0;
        if (inside(g, x.x, x.y, x.z)) {
            const int ix = min((int)x.x, g.nx - 1), iy = min((int)x.y, g.ny - 1), iz = min((int)x.z, g.nz - 1);
            key = (ix >> bins.sh[0]) + bins.n[0] * ((iy >> bins.sh[1]) + bins.n[1] * (iz >> bins.sh[2]));
        }
        place[i] = make_int2(key, atomicAdd(count + key, 1));
    }
}

// Step 2, one CTA: exclusive sums of the counts. 16-byte accesses: a thread's
// 16 bins are consecutive.
__global__ void __launch_bounds__(1024) tape_scan_kernel(const int4 *__restrict__ count, int4 *__restrict__ start) {
    __shared__ int32_t part[32];
    constexpr int kPer = kMaxBins / 4096;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int4 v[kPer];
    int32_t sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        v[k] = count[threadIdx.x * kPer + k];
        sum += v[k].x + v[k].y + v[k].z + v[k].w;
    }
    int32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    int32_t run = incl - sum;
    for (int w = 0; w < warp; ++w) run += part[w];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int4 c = v[k];
        start[threadIdx.x * kPer + k] = make_int4(run, run + c.x, run + c.x + c.y, run + c.x + c.y + c.z);
        run += c.x + c.y + c.z + c.w;
    }
}

// Step 3: start positions, exit cycles and the caller's indices in cell
// order (in the caller's order without `place`).
__global__ void tape_init_kernel(const BlockDev *__restrict__ blk, int64_t P, const float *__restrict__ seeds,
                                 const int32_t *__restrict__ start, const int2 *__restrict__ place,
                                 float4 *__restrict__ x0, int32_t *__restrict__ exitc, int32_t *__restrict__ perm) {
    const BlockDev &B = *blk;
    const Geo g = load_geo(B);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 x = start_of(B, seeds, i);
        int64_t at = i;
        if (place) {
            const int2 pl = place[i];
            at = (int64_t)start[pl.x] + pl.y;
            if (at >= P) continue;   // only when forwards of one tape overlap: wrong results, no stray write
        }
        x0[at] = x;
        exitc[at] = inside(g, x.x, x.y, x.z) ? -1 : 0;   // a start outside the block never moves
        perm[at] = (int32_t)i;
    }
}

// Forward over the whole interval, one thread per particle (the fields of
// every cycle are resident in the tape's table, and particles are
// independent): cycle after cycle, the RK4 step with the closed-box tests of
// the advection kernel; a failing step records its cycle. Positions are kept
// at the start of every segment. Then the outputs: physical end position,
// valid flag, exit cycle.
__global__ void __launch_bounds__(kThreads) tape_forward_kernel(
    const BlockDev *__restrict__ blk, const void *const *__restrict__ table, int32_t L, int32_t C, float dt, int64_t P,
    float4 *__restrict__ ckpt, int32_t *__restrict__ exitc, const int32_t *__restrict__ perm, float *__restrict__ ends,
    uint8_t *__restrict__ valid, int32_t *__restrict__ exit_out) {
    const BlockDev &B = *blk;
    const Geo g = load_geo(B);
    const float3 s = make_float3(dt * B.inv_h[0], dt * B.inv_h[1], dt * B.inv_h[2]);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 r = ckpt[i];
        float3 x = make_float3(r.x, r.y, r.z), q;
        int32_t e = exitc[i];
        if (e < 0) {
            int32_t left = C;   // cycles left in the segment
            float4 *ck = ckpt + i;
            const void *next = table[0];
            for (int32_t c = 0; c < L; ++c) {
                const void *field = next;
                if (left == 0) {
                    ck += P;
                    *ck = make_float4(x.x, x.y, x.z, 0.f);
                    left = C;
                }
                --left;
                if (c + 1 < L) next = table[c + 1];
                if (rk4_step<bto::LAYOUT_F3>(x, field, g, s, q) != 0) {
                    e = c;
                    break;
                }
            }
            exitc[i] = e;
        }
        const int64_t o = perm[i];
        ends[3 * o + 0] = fmaf(x.x, B.h[0], B.origin[0]);
        ends[3 * o + 1] = fmaf(x.y, B.h[1], B.origin[1]);
        ends[3 * o + 2] = fmaf(x.z, B.h[2], B.origin[2]);
        valid[o] = e < 0 ? 1 : 0;
        if (exit_out) exit_out[o] = e;
    }
}

// Adds the corner gradients v[a + 2b + 4c] of the cell at `node` to gF: each
// x-row of two nodes is six consecutive floats, added as pairs where the
// address allows it (4-byte aligned: three pairs, or two pairs between two
// single words), 14 atomic operations a cell on average instead of 24.
__device__ __forceinline__ void red2(float *p, float a, float b) {
    asm volatile("red.relaxed.gpu.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a), "f"(b) : "memory");
}
__device__ __forceinline__ void add_cell(float *__restrict__ gF, const Geo &g, uint32_t node, const float (&v)[8][3]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t nd = node + ((q & 1) ? g.nnx : 0u) + ((q & 2) ? g.nnxy : 0u);
        if (!BTO_IN_BOUNDS((uint64_t)nd + 1 < g.nodes, nullptr)) continue;
        float *p = gF + 3ull * nd;
        const float *a = v[2 * q], *b = v[2 * q + 1];
        const bool odd = (reinterpret_cast<uintptr_t>(p) & 4u) != 0;
        red2(p + (odd ? 1 : 0), odd ? a[1] : a[0], odd ? a[2] : a[1]);
        red2(p + (odd ? 3 : 2), odd ? b[0] : a[2], odd ? b[1] : b[0]);
        if (odd) {
            atomicAdd(p, a[0]);
            atomicAdd(p + 5, b[2]);
        } else {
            red2(p + 4, b[1], b[2]);
        }
    }
}

// The cell of x, its corners from the cache or the field, and x's fractions
// in it.
__device__ __forceinline__ void locate(JCell &C, const float *__restrict__ f, const Geo &g, const float3 x, float &fx,
                                       float &fy, float &fz) {
    int ix, iy, iz;
    cell_coord_any(x.x, g.cmx, ix, fx);
    cell_coord_any(x.y, g.cmy, iy, fy);
    cell_coord_any(x.z, g.cmz, iz, fz);
    const uint32_t node = (uint32_t)ix + g.nnx * (uint32_t)iy + g.nnxy * (uint32_t)iz;
    if (node != C.node) {
        load_cell<bto::LAYOUT_F3>(f, g.nnx, g.nnxy, g.nodes, ix, iy, iz, C.v);
        C.node = node;
    }
}

// (p - q) . w
__device__ __forceinline__ float diff_dot(const float (&p)[3], const float (&q)[3], const float3 w) {
    return fmaf(p[2] - q[2], w.z, fmaf(p[1] - q[1], w.y, (p[0] - q[0]) * w.x));
}

// (dv/dxi)^T w in the cell C at fractions (fx, fy, fz): the differences of
// the corners along each axis, dotted with w and blended along the other two.
__device__ __forceinline__ float3 grad_dot(const JCell &C, float fx, float fy, float fz, const float3 w) {
    const float (&c)[8][3] = C.v;
    return make_float3(
        lerp1(lerp1(diff_dot(c[1], c[0], w), diff_dot(c[3], c[2], w), fy),
              lerp1(diff_dot(c[5], c[4], w), diff_dot(c[7], c[6], w), fy), fz),
        lerp1(lerp1(diff_dot(c[2], c[0], w), diff_dot(c[3], c[1], w), fx),
              lerp1(diff_dot(c[6], c[4], w), diff_dot(c[7], c[5], w), fx), fz),
        lerp1(lerp1(diff_dot(c[4], c[0], w), diff_dot(c[5], c[1], w), fx),
              lerp1(diff_dot(c[6], c[2], w), diff_dot(c[7], c[3], w), fx), fy));
}

// Reverse of one cycle for one particle at x (cell units) with adjoint lm
// (see the header of this file); adds the node-velocity gradients to gF.
// Returns the adjoint before the cycle. The stage points are found first;
// then the stages are taken in reverse, their corners mostly still cached,
// and the corner gradients of stages in one cell are summed before they are
// added. No stage's Jacobian is formed: four of them held 36 registers and
// left 12 warps per SM (32,768 particles over 200 cycles of 64^3 cells, with
// scalar atomics: 1353 us; so, with paired ones: 831 us).
__device__ __forceinline__ float3 adj_step(const float *__restrict__ f, float *__restrict__ gF, const Geo &g,
                                           const float3 s, const float3 x, const float3 lm) {
    JCell C;
    C.node = ~0u;
    float3 p[4];
    p[0] = x;
    float fx, fy, fz;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        locate(C, f, g, p[k], fx, fy, fz);
        const float3 v = trilerp(C.v, fx, fy, fz);
        const float h = k == 2 ? 1.f : 0.5f;
        p[k + 1] = make_float3(fmaf(h * s.x, v.x, x.x), fmaf(h * s.y, v.y, x.y), fmaf(h * s.z, v.z, x.z));
    }
    const float3 s6l = make_float3(s.x / 6.f * lm.x, s.y / 6.f * lm.y, s.z / 6.f * lm.z);
    const float3 s3l = make_float3(s.x / 3.f * lm.x, s.y / 3.f * lm.y, s.z / 3.f * lm.z);
    float3 lx = lm, w = s6l;   // w: the stage's g
    float acc[8][3];
    uint32_t acc_node = ~0u;
#pragma unroll
    for (int k = 3; k >= 0; --k) {
        locate(C, f, g, p[k], fx, fy, fz);
        if (C.node != acc_node) {
            if (k < 3) add_cell(gF, g, acc_node, acc);
            acc_node = C.node;
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = 0.f;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float wt = ((j & 1) ? fx : 1.f - fx) * ((j & 2) ? fy : 1.f - fy) * ((j & 4) ? fz : 1.f - fz);
            acc[j][0] = fmaf(wt, w.x, acc[j][0]);
            acc[j][1] = fmaf(wt, w.y, acc[j][1]);
            acc[j][2] = fmaf(wt, w.z, acc[j][2]);
        }
        const float3 q = grad_dot(C, fx, fy, fz, w);
        lx.x += q.x; lx.y += q.y; lx.z += q.z;
        if (k > 0) {
            const float h = k == 3 ? 1.f : 0.5f;
            const float3 b = k == 1 ? s6l : s3l;
            w = make_float3(fmaf(h * s.x, q.x, b.x), fmaf(h * s.y, q.y, b.y), fmaf(h * s.z, q.z, b.z));
        }
    }
    add_cell(gF, g, acc_node, acc);
    return lx;
}

// The same by four lanes per particle (rk4_step_quad).
__global__ void __launch_bounds__(kThreads) tape_forward_quad_kernel(
    const BlockDev *__restrict__ blk, const void *const *__restrict__ table, int32_t L, int32_t C, float dt, int64_t P,
    float4 *__restrict__ ckpt, int32_t *__restrict__ exitc, const int32_t *__restrict__ perm, float *__restrict__ ends,
    uint8_t *__restrict__ valid, int32_t *__restrict__ exit_out) {
    const BlockDev &B = *blk;
    const Geo g = load_geo(B);
    const float3 s = make_float3(dt * B.inv_h[0], dt * B.inv_h[1], dt * B.inv_h[2]);
    const int64_t i = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 2;
    const int lane4 = threadIdx.x & 3;
    __shared__ int touched[kThreads];
    const uint32_t word = (uint32_t)__cvta_generic_to_shared(touched + threadIdx.x);
    const bool have = i < P;
    float3 x = make_float3(0.f, 0.f, 0.f), q;
    int32_t e = 0;
    if (have) {
        const float4 r = ckpt[i];
        x = make_float3(r.x, r.y, r.z);
        e = exitc[i];
    }
    bool alive = have && e < 0;
    int32_t left = C;   // cycles left in the segment
    float4 *ck = ckpt + i;
    const void *next = table[0];
    for (int32_t c = 0; c < L && __any_sync(0xffffffffu, alive); ++c) {
        const void *field = next;
        if (left == 0) {
            ck += P;
            if (alive && lane4 == 0) *ck = make_float4(x.x, x.y, x.z, 0.f);
            left = C;
        }
        --left;
        if (c + 1 < L) next = table[c + 1];
        if (rk4_step_quad<bto::LAYOUT_F3>(x, field, g, s, q, alive, Ahead{c + 1 < L ? next : nullptr, word}, nullptr)) {
            alive = false;
            e = c;
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (!have) return;
    const int64_t o = perm[i];
    if (lane4 < 3) {
        const float v = lane4 == 0 ? x.x : (lane4 == 1 ? x.y : x.z);
        ends[3 * o + lane4] = fmaf(v, B.h[lane4], B.origin[lane4]);
    } else {
        exitc[i] = e;
        valid[o] = e < 0 ? 1 : 0;
        if (exit_out) exit_out[o] = e;
    }
}

// dk = J dp, column by column.
__device__ __forceinline__ void mat_mul(const float (&J)[3][3], const float (&p)[3][3], float (&k)[3][3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) k[a][b] = fmaf(J[a][2], p[2][b], fmaf(J[a][1], p[1][b], J[a][0] * p[0][b]));
}

// Matrices of all segments: thread (s, i) runs segment s of particle i
// (blockIdx.y = s, so the CTAs in flight share a few segments' fields) with
// the three tangents of its start position. A segment that the particle does
// not move in has no matrix (the chain skips it).
__global__ void __launch_bounds__(kThreads) tape_tangent_kernel(const BlockDev *__restrict__ blk,
                                                                const void *const *__restrict__ table, int32_t L,
                                                                int32_t C, float dt, int64_t P,
                                                                const float4 *__restrict__ ckpt,
                                                                const int32_t *__restrict__ exitc,
                                                                float *__restrict__ mat) {
    const BlockDev &B = *blk;
    const Geo g = load_geo(B);
    const float s[3] = {dt * B.inv_h[0], dt * B.inv_h[1], dt * B.inv_h[2]};
    const int32_t sg = blockIdx.y;
    const int32_t c0 = sg * C;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t moved = cycles_moved(exitc[i], L);
        if (moved <= c0) continue;
        const int32_t c1 = c0 + min(C, moved - c0);
        const float4 r = ckpt[(size_t)sg * P + i];
        float x[3] = {r.x, r.y, r.z};
        float T[3][3] = {{1.f, 0.f, 0.f}, {0.f, 1.f, 0.f}, {0.f, 0.f, 1.f}};
        for (int32_t c = c0; c < c1; ++c) {
            const float *f = reinterpret_cast<const float *>(table[c]);
            JCell cell;
            cell.node = ~0u;
            float p[3] = {x[0], x[1], x[2]}, ax[3];
            float dp[3][3], at[3][3];
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) dp[a][b] = T[a][b];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float3 v;
                float J[3][3], dk[3][3];
                Stage st;
                sample_jac(cell, f, g, p[0], p[1], p[2], v, J, st);
                mat_mul(J, dp, dk);
                const float kv[3] = {v.x, v.y, v.z};
                const float w = k == 1 || k == 2 ? 2.f : 1.f;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    ax[a] = k == 0 ? kv[a] : fmaf(w, kv[a], ax[a]);
                    const float step = k == 2 ? s[a] : 0.5f * s[a];
                    if (k < 3) p[a] = fmaf(step, kv[a], x[a]);
#pragma unroll
                    for (int b = 0; b < 3; ++b) {
                        at[a][b] = k == 0 ? dk[a][b] : fmaf(w, dk[a][b], at[a][b]);
                        if (k < 3) dp[a][b] = fmaf(step, dk[a][b], T[a][b]);
                    }
                }
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float s6 = s[a] * (1.f / 6.f);
                x[a] = fmaf(s6, ax[a], x[a]);
#pragma unroll
                for (int b = 0; b < 3; ++b) T[a][b] = fmaf(s6, at[a][b], T[a][b]);
            }
        }
        float *m = mat + (size_t)sg * 9 * P + i;
#pragma unroll
        for (int k = 0; k < 9; ++k) m[(size_t)k * P] = T[k / 3][k % 3];
    }
}

// Chain for a gradient: lam = h * dL/d(end) (physical -> cell units) at the
// end of the last segment, lam_(s-1) = M_s^T lam_s; every segment's end
// adjoint replaces the first planes of its matrix, and dL/d(start) = lam / h
// is written for the caller's particle.
__global__ void tape_chain_kernel(const BlockDev *__restrict__ blk, int32_t L, int32_t C, int64_t P,
                                  const int32_t *__restrict__ exitc, const int32_t *__restrict__ perm,
                                  const float *__restrict__ grad, float *__restrict__ mat, float *__restrict__ out) {
    const BlockDev &B = *blk;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t o = perm[i];
        float3 l = make_float3(grad[3 * o + 0] * B.h[0], grad[3 * o + 1] * B.h[1], grad[3 * o + 2] * B.h[2]);
        int32_t sg = last_segment(exitc[i], L, C);
        float *m = mat + (size_t)max(sg, 0) * 9 * P + i;
        float M[9], N[9];   // N: the next segment's, loaded ahead of the stores
#pragma unroll
        for (int k = 0; k < 9; ++k) N[k] = sg >= 0 ? m[(size_t)k * P] : 0.f;
        for (; sg >= 0; --sg, m -= (size_t)9 * P) {
#pragma unroll
            for (int k = 0; k < 9; ++k) M[k] = N[k];
            if (sg > 0) {
#pragma unroll
                for (int k = 0; k < 9; ++k) N[k] = *(m - (size_t)(9 - k) * P);
            }
            m[0] = l.x;
            m[(size_t)P] = l.y;
            m[(size_t)2 * P] = l.z;
            const float J[3][3] = {{M[0], M[1], M[2]}, {M[3], M[4], M[5]}, {M[6], M[7], M[8]}};
            l = jt_times(J, l);
        }
        out[3 * o + 0] = l.x * B.inv_h[0];
        out[3 * o + 1] = l.y * B.inv_h[1];
        out[3 * o + 2] = l.z * B.inv_h[2];
    }
}

// The flow-map Jacobian: the product of the segments' matrices, last to
// first, with h of the row in front and 1 / h of the column behind.
__global__ void tape_product_kernel(const BlockDev *__restrict__ blk, int32_t L, int32_t C, int64_t P,
                                    const int32_t *__restrict__ exitc, const int32_t *__restrict__ perm,
                                    const float *__restrict__ mat, float *__restrict__ jac) {
    const BlockDev &B = *blk;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        float3 R[3] = {make_float3(B.h[0], 0.f, 0.f), make_float3(0.f, B.h[1], 0.f), make_float3(0.f, 0.f, B.h[2])};
        for (int32_t sg = last_segment(exitc[i], L, C); sg >= 0; --sg) {
            const float *m = mat + (size_t)sg * 9 * P + i;
            float M[3][3];
#pragma unroll
            for (int k = 0; k < 9; ++k) M[k / 3][k % 3] = m[(size_t)k * P];
#pragma unroll
            for (int a = 0; a < 3; ++a) R[a] = jt_times(M, R[a]);
        }
        float *j = jac + 9 * (int64_t)perm[i];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            j[3 * a + 0] = R[a].x * B.inv_h[0];
            j[3 * a + 1] = R[a].y * B.inv_h[1];
            j[3 * a + 2] = R[a].z * B.inv_h[2];
        }
    }
}

// Cycles between the positions a long segment is restarted from: a multiple
// of kChunk, at most kSubs of them.
__host__ __device__ inline int32_t sub_space(int32_t C) {
    return kChunk * ((C - 1) / (kChunk * kSubs) + 1);
}

// Field gradients of all segments: thread (s, i) takes the adjoint at the
// end of segment s from the chain, recomputes the segment's positions from
// its checkpoint into shared memory and reverses its cycles. A segment longer
// than kChunk cycles (intervals over 400 cycles) is taken in chunks, the last
// first; the first pass through it leaves a position every `space` cycles, and
// the other chunks are recomputed from those.
__global__ void __launch_bounds__(kThreads) tape_scatter_kernel(const BlockDev *__restrict__ blk,
                                                                const void *const *__restrict__ table,
                                                                float *const *__restrict__ gtable, int32_t L,
                                                                int32_t C, float dt, int64_t P,
                                                                const float4 *__restrict__ ckpt,
                                                                const int32_t *__restrict__ exitc,
                                                                const float *__restrict__ lam) {
    extern __shared__ float pos[];   // [min(C, kChunk) + positions to restart from][3][kThreads]
    const BlockDev &B = *blk;
    const Geo g = load_geo(B);
    const float3 s = make_float3(dt * B.inv_h[0], dt * B.inv_h[1], dt * B.inv_h[2]);
    const int32_t sg = blockIdx.y;
    const int32_t c0 = sg * C;
    float *mine = pos + threadIdx.x;
    float *subs = mine + kChunk * 3 * kThreads;   // only in segments longer than kChunk
    const int32_t space = sub_space(C);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t moved = cycles_moved(exitc[i], L);
        if (moved <= c0) continue;
        const int32_t c1 = c0 + min(C, moved - c0);
        const float4 r = ckpt[(size_t)sg * P + i];
        const float *l = lam + (size_t)sg * 9 * P + i;
        float3 lm = make_float3(l[0], l[(size_t)P], l[(size_t)2 * P]);
        for (int32_t k0 = c0 + (c1 - c0 - 1) / kChunk * kChunk, k1 = c1; k0 >= c0; k1 = k0, k0 -= kChunk) {
            float3 x = make_float3(r.x, r.y, r.z), q;
            int32_t from = c0;
            if (k1 < c1) {
                const int32_t at = (k0 - c0) / space;
                const float *m = subs + at * 3 * kThreads;
                x = make_float3(m[0], m[kThreads], m[2 * kThreads]);
                from = c0 + at * space;
            }
            for (int32_t c = from; c < k1; ++c) {
                if (c >= k0) {
                    float *m = mine + (c - k0) * 3 * kThreads;
                    m[0] = x.x; m[kThreads] = x.y; m[2 * kThreads] = x.z;
                }
                if (C > kChunk && k1 == c1 && (c - c0) % space == 0) {
                    float *m = subs + (c - c0) / space * 3 * kThreads;
                    m[0] = x.x; m[kThreads] = x.y; m[2 * kThreads] = x.z;
                }
                if (c + 1 < k1) rk4_step<bto::LAYOUT_F3>(x, table[c], g, s, q);
            }
            for (int32_t c = k1 - 1; c >= k0; --c) {
                const float *m = mine + (c - k0) * 3 * kThreads;
                lm = adj_step(reinterpret_cast<const float *>(table[c]), gtable[c], g, s,
                              make_float3(m[0], m[kThreads], m[2 * kThreads]), lm);
            }
        }
    }
}

// Largest eigenvalue of the symmetric 3x3 matrix C (closed form of the
// characteristic cubic, trigonometric solution), in double.
__device__ double sym3_max_eig(const double C[3][3]) {
    const double p1 = C[0][1] * C[0][1] + C[0][2] * C[0][2] + C[1][2] * C[1][2];
    const double q = (C[0][0] + C[1][1] + C[2][2]) / 3.0;
    if (p1 <= 1e-300 * (q * q + 1.0)) return fmax(C[0][0], fmax(C[1][1], C[2][2]));
    const double p2 = (C[0][0] - q) * (C[0][0] - q) + (C[1][1] - q) * (C[1][1] - q) +
                      (C[2][2] - q) * (C[2][2] - q) + 2.0 * p1;
    const double p = sqrt(p2 / 6.0), ip = 1.0 / p;   // one division: FP64 runs at 1/64 of the FP32 rate here
    double Bm[3][3];
    for (int a = 0; a < 3; ++a)
        for (int b = a; b < 3; ++b) Bm[a][b] = (C[a][b] - (a == b ? q : 0.0)) * ip;
    const double detB = Bm[0][0] * (Bm[1][1] * Bm[2][2] - Bm[1][2] * Bm[1][2]) -
                        Bm[0][1] * (Bm[0][1] * Bm[2][2] - Bm[1][2] * Bm[0][2]) +
                        Bm[0][2] * (Bm[0][1] * Bm[1][2] - Bm[1][1] * Bm[0][2]);
    const double r = fmin(1.0, fmax(-1.0, detB / 2.0));
    const double phi = acos(r) / 3.0;
    return q + 2.0 * p * cos(phi);
}

// FTLE = ln(sqrt(lambda_max(J^T J))) / |T| for valid particles, NaN for the
// others (their trajectory does not span the interval).
__global__ void tape_ftle_kernel(int64_t P, const float *__restrict__ jac, const int32_t *__restrict__ exitc,
                                 const int32_t *__restrict__ perm, double T, float *__restrict__ ftle) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < P; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = perm[k];
        if (exitc[k] >= 0) {
            ftle[i] = __int_as_float(0x7fc00000);
            continue;
        }
        double J[3][3], C[3][3];
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b) J[a][b] = jac[9 * i + 3 * a + b];
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b) C[a][b] = J[0][a] * J[0][b] + J[1][a] * J[1][b] + J[2][a] * J[2][b];
        const double lmax = sym3_max_eig(C);
        ftle[i] = (float)(0.5 * log(fmax(lmax, 1e-300)) / T);
    }
}

bto_status cuda_st(cudaError_t e) {
    if (e == cudaSuccess) return BTO_OK;
    (void)cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? BTO_ERR_OOM : BTO_ERR_CUDA;
}

int grid_of(const bto_tape *t) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((t->P + 255) / 256, (int64_t)t->sm_count * 8));
}

void free_tape(bto_tape *t) {
    if (!t) return;
    t->mem.put(t->ckpt);
    t->mem.put(t->mat);
    t->mem.put(t->d_block);
    t->mem.put(t->exitc);
    t->mem.put(t->perm);
    t->mem.put(t->bins);
    delete t;
}

// Grid of the kernels that take all segments at once: x over the particles,
// y over the segments.
dim3 seg_grid(const bto_tape *t) {
    const int64_t x = std::min<int64_t>((t->P + kThreads - 1) / kThreads, (int64_t)t->sm_count * 16);
    return dim3((unsigned)std::max<int64_t>(1, x), (unsigned)t->nseg);
}

// Cycles per segment, from the interval alone (so that the rounding of the
// results does not depend on checkpoint_every): 1.2 sqrt(L), at least 4. The
// tape then holds 52 nseg = 43 sqrt(L) bytes a particle. A serial sweep with a
// checkpoint every K cycles, three rows of K positions to recompute a segment
// for the Jacobian, and three adjoints took 16 (L / K + 3 K + 4), which is 55
// sqrt(L) + 64 at the best K.
int32_t segment_cycles(int32_t L) {
    return std::max<int32_t>(4, (int32_t)std::ceil(1.2 * std::sqrt((double)L)));
}

// Matrices of all segments: the first step of either backward call.
bto_status tangents(const bto_tape *t, cudaStream_t s) {
    tape_tangent_kernel<<<seg_grid(t), kThreads, 0, s>>>(t->d_block, t->table, t->L, t->C, t->dt, t->P, t->ckpt,
                                                         t->exitc, t->mat);
    return cuda_st(cudaGetLastError());
}

}  // namespace

namespace bto {
BTO_BOUNDS_ACCESSOR(bounds_failures_adjoint)
}

extern "C" {

bto_status bto_tape_create(const int32_t extent_cells[3], const float origin[3], const float spacing[3],
                           int64_t num_particles, int32_t cycles, int32_t checkpoint_every, bto_tape **out) {
    if (!extent_cells || !origin || !spacing || !out) return BTO_ERR_INVALID_ARG;
    if (num_particles < 1 || num_particles > (1ll << 30) || cycles < 1 || checkpoint_every < 1)
        return BTO_ERR_INVALID_ARG;
    BlockDev B{};
    int64_t nodes = 1;
    for (int a = 0; a < 3; ++a) {
        const int32_t n = extent_cells[a];
        if (n < 1 || n > (1 << 23) || !std::isfinite(origin[a]) || !std::isfinite(spacing[a]) || !(spacing[a] > 0.f))
            return BTO_ERR_INVALID_ARG;
        B.n[a] = n;
        B.nn[a] = n + 1;
        B.S[a] = 1;
        B.inv_h[a] = 1.0f / spacing[a];
        B.origin[a] = origin[a];
        B.h[a] = spacing[a];
        nodes *= (int64_t)(n + 1);
    }
    if (nodes > (1ll << 29)) return BTO_ERR_INVALID_ARG;
    B.stride = 1;
    B.nseeds = num_particles;
    bto_tape *t = new (std::nothrow) bto_tape();
    if (!t) return BTO_ERR_OOM;
    t->mem = bto::current_allocator();
    t->B = B;
    t->P = num_particles;
    t->L = cycles;
    t->C = segment_cycles(cycles);
    t->nseg = (cycles - 1) / t->C + 1;
    // bins of the sort: 32 x 1 x 1 cells, doubled along y and z, then along x, until they are few enough
    t->bsh[0] = 5;
    for (;;) {
        int64_t nb = 1;
        for (int a = 0; a < 3; ++a) {
            t->bn[a] = (B.n[a] + (1 << t->bsh[a]) - 1) >> t->bsh[a];
            nb *= t->bn[a];
        }
        if (nb <= kMaxBins) break;
        const int a = t->bn[1] >= t->bn[2] ? 1 : 2;
        ++t->bsh[t->bn[a] > 1 ? a : 0];
    }
    cudaError_t e = cudaGetDevice(&t->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&t->sm_count, cudaDevAttrMultiProcessorCount, t->device);
    const size_t P = (size_t)num_particles;
    if (e == cudaSuccess) e = t->mem.get(&t->ckpt, sizeof(float4) * P * (size_t)t->nseg);
    if (e == cudaSuccess) e = t->mem.get(&t->mat, sizeof(float) * 9 * P * (size_t)t->nseg);
    if (e == cudaSuccess) e = t->mem.get(&t->d_block, sizeof(BlockDev));
    if (e == cudaSuccess) e = t->mem.get(&t->exitc, sizeof(int32_t) * P);
    if (e == cudaSuccess) e = t->mem.get(&t->perm, sizeof(int32_t) * P);
    if (e == cudaSuccess) e = t->mem.get(&t->bins, sizeof(int32_t) * 2 * kMaxBins);
    if (e == cudaSuccess) e = cudaMemset(t->perm, 0, sizeof(int32_t) * P);
    if (e == cudaSuccess) e = cudaMemcpy(t->d_block, &t->B, sizeof(BlockDev), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        free_tape(t);
        return e == cudaErrorMemoryAllocation ? BTO_ERR_OOM : BTO_ERR_CUDA;
    }
    *out = t;
    return BTO_OK;
}

int64_t bto_tape_num_particles(const bto_tape *t) { return t ? t->P : -1; }

bto_status bto_tape_forward(bto_tape *t, const float *d_seeds, const void *const *d_field_table, float dt,
                            float *d_ends, uint8_t *d_valid, int32_t *d_exit_cycle, bto_stream stream) {
    if (!t || !d_seeds || !d_field_table || !d_ends || !d_valid || !std::isfinite(dt)) return BTO_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(d_seeds) % 4 || reinterpret_cast<uintptr_t>(d_ends) % 4 ||
        reinterpret_cast<uintptr_t>(d_exit_cycle) % 4 ||
        reinterpret_cast<uintptr_t>(d_field_table) % alignof(void *))
        return BTO_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int grid = grid_of(t);
    t->table = d_field_table;
    t->dt = dt;
    t->have_forward = false;
    // the sort's (bin, place) pairs use the matrices' memory, which a backward call writes afresh
    int2 *place = sorts(t->P, t->L) ? reinterpret_cast<int2 *>(t->mat) : nullptr;
    if (place) {
        const Bins bins = {{t->bsh[0], t->bsh[1], t->bsh[2]}, {t->bn[0], t->bn[1], t->bn[2]}};
        const cudaError_t z = cudaMemsetAsync(t->bins, 0, sizeof(int32_t) * kMaxBins, s);
        if (z != cudaSuccess) return cuda_st(z);
        tape_bin_kernel<<<grid, 256, 0, s>>>(t->d_block, t->P, d_seeds, bins, t->bins, place);
        tape_scan_kernel<<<1, 1024, 0, s>>>(reinterpret_cast<const int4 *>(t->bins),
                                            reinterpret_cast<int4 *>(t->bins + kMaxBins));
    }
    tape_init_kernel<<<grid, 256, 0, s>>>(t->d_block, t->P, d_seeds, t->bins + kMaxBins, place, t->ckpt, t->exitc,
                                          t->perm);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) {
        if (t->P <= kQuadPerSm * t->sm_count)
            tape_forward_quad_kernel<<<(unsigned)((4 * t->P + kThreads - 1) / kThreads), kThreads, 0, s>>>(
                t->d_block, d_field_table, t->L, t->C, dt, t->P, t->ckpt, t->exitc, t->perm, d_ends, d_valid,
                d_exit_cycle);
        else
            tape_forward_kernel<<<seg_grid(t).x, kThreads, 0, s>>>(t->d_block, d_field_table, t->L, t->C, dt, t->P,
                                                                   t->ckpt, t->exitc, t->perm, d_ends, d_valid,
                                                                   d_exit_cycle);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_st(e);
    t->have_forward = true;
    return BTO_OK;
}

bto_status bto_tape_backward(bto_tape *t, const float *d_grad_ends, float *d_grad_seeds,
                             float *const *d_grad_field_table, bto_stream stream) {
    if (!t || !d_grad_ends || !d_grad_seeds) return BTO_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(d_grad_ends) % 4 || reinterpret_cast<uintptr_t>(d_grad_seeds) % 4 ||
        reinterpret_cast<uintptr_t>(d_grad_field_table) % alignof(void *))
        return BTO_ERR_INVALID_ARG;
    if (!t->have_forward) return BTO_ERR_STATE;
    cudaStream_t s = (cudaStream_t)stream;
    const int grid = grid_of(t);
    const bto_status st = tangents(t, s);
    if (st != BTO_OK) return st;
    tape_chain_kernel<<<grid, 256, 0, s>>>(t->d_block, t->L, t->C, t->P, t->exitc, t->perm, d_grad_ends,
                                           t->mat, d_grad_seeds);
    if (d_grad_field_table) {
        const int held = t->C <= kChunk ? t->C : kChunk + (t->C - 1) / sub_space(t->C) + 1;
        const size_t smem = sizeof(float) * 3 * kThreads * (size_t)held;
        tape_scatter_kernel<<<seg_grid(t), kThreads, smem, s>>>(t->d_block, t->table, d_grad_field_table, t->L, t->C,
                                                               t->dt, t->P, t->ckpt, t->exitc, t->mat);
    }
    return cuda_st(cudaGetLastError());
}

bto_status bto_tape_jacobian(bto_tape *t, float *d_jac, bto_stream stream) {
    if (!t || !d_jac || reinterpret_cast<uintptr_t>(d_jac) % 4) return BTO_ERR_INVALID_ARG;
    if (!t->have_forward) return BTO_ERR_STATE;
    cudaStream_t s = (cudaStream_t)stream;
    const bto_status st = tangents(t, s);
    if (st != BTO_OK) return st;
    tape_product_kernel<<<grid_of(t), 256, 0, s>>>(t->d_block, t->L, t->C, t->P, t->exitc, t->perm, t->mat, d_jac);
    return cuda_st(cudaGetLastError());
}

bto_status bto_tape_ftle(bto_tape *t, const float *d_jac, float *d_ftle, bto_stream stream) {
    if (!t || !d_jac || !d_ftle) return BTO_ERR_INVALID_ARG;
    if (!t->have_forward) return BTO_ERR_STATE;
    const double T = std::fabs((double)t->dt * (double)t->L);
    if (!(T > 0.0)) return BTO_ERR_INVALID_ARG;
    tape_ftle_kernel<<<grid_of(t), 256, 0, (cudaStream_t)stream>>>(t->P, d_jac, t->exitc, t->perm, T, d_ftle);
    return cuda_st(cudaGetLastError());
}

void bto_tape_destroy(bto_tape *t) {
    if (!t) return;
    cudaDeviceSynchronize();
    free_tape(t);
}

}  // extern "C"

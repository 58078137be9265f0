// libbto kernels for sm_103a.
//
//   K2 seed_kernel        lattice seeds in brick order (Sec. 2.3)
//   K3 advect_kernel      one RK4 step per live particle with trilinear
//                         sampling (Sec. 3.1, Eq. 1), closed-box termination
//                         of stage and end points (Sec. 3.1, Sec. 3.3), and
//                         compaction of survivors so that terminated
//                         particles occupy no thread in later cycles
//                         (Sec. 3.1, particle management)
//   K3i interval_kernel   all cycles of an interval, fields resident
//   K4 end_interval_kernel  seeds and basis flows (Sec. 2.3), then the next
//                         interval's seeds
//      write_live_kernel, write_term_kernel  the same outputs for the tiled
//                         list and the allocation-free interval
//
// Design (GB300): the hot kernel is a gather over the velocity nodes, bound
// by memory traffic, not by arithmetic; there is no dense contraction, so the
// tensor cores are not used. Particles are stored in brick order of their
// seeds (runs of 32 seeds along x, the runs in Morton order) so that the
// lanes of a warp touch few node rows and neighbouring warps neighbouring
// rows (L1/L2 reuse of each node); the 8 corners of a cell stay in
// registers across the four RK4 stages and are reloaded only when a stage
// point lands in another cell; each warp owns groups of 32*PPT particles
// and compacts the survivors of a group inside that group (ballot/popc, no
// barrier, no atomic); the grid is persistent (a multiple of the SM count).
// The post hoc kernels (lattice fill, stitching) are in bto_posthoc.cu.
#include <cstdint>
#include <cuda_runtime.h>

#include "bto_internal.h"
#include "bto_device.cuh"

namespace bto {
namespace {

using namespace dev;

constexpr unsigned kFull = 0xffffffffu;

// Index of the block holding global slot/id i (blocks sorted by base).
__device__ __forceinline__ int find_block(const BlockDev *__restrict__ blocks, int nb, int64_t i) {
    int lo = 0, hi = nb - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (blocks[mid].base <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---------------------------------------------------------------------------
// K3: advection cycle. The particle list is cut into groups of G = 32*PPT
// slots; one warp owns a group for the cycle: it advects the group's live
// particles (PPT rounds of 32) and writes them back in place. When none of
// them terminated, only the positions are rewritten, in their slots; when
// some did, the survivors (positions and ids) are compacted, in order, to
// the front of the group. Warps take groups g, g + W, g + 2W, ... (W =
// warps in the grid), so the groups in flight at any time are neighbours
// in brick order. There is no barrier and no atomic: a terminated particle
// only leaves the group's live prefix.
// ---------------------------------------------------------------------------
template <int LAYOUT, int NT, int PPT, bool BATCHED, int MINB>
__global__ void __launch_bounds__(NT, MINB) advect_kernel(const AdvectArgs a) {
    // Programmatic dependent launch: the grid may be scheduled while the
    // previous cycle's grid drains; it reads nothing before that grid has
    // completed and its writes are visible (a no-op when launched without
    // the dependency). Then the next cycle's grid may be scheduled.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr int G = 32 * PPT;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t nwarps = ((int64_t)gridDim.x * NT) >> 5;
    int cur_b = -1;
    Geo g{};
    float3 s = make_float3(0.f, 0.f, 0.f);
    const void *field = nullptr;
    int64_t idbase = 0;
    int64_t nseeds = 0;
    const PartList P = a.p;

    for (int64_t grp = (((int64_t)blockIdx.x * NT) + threadIdx.x) >> 5; grp < a.ngroups;
         grp += nwarps) {
        int cnt = __ldcg(P.gcnt + grp);
        if (!BTO_IN_BOUNDS(cnt >= 0 && cnt <= G, a.err)) cnt = 0;
        if (cnt == 0) continue;
        const int b = BATCHED ? __ldg(a.gblock + grp * PPT) : 0;
        if (b != cur_b) {
            cur_b = b;
            const BlockDev &B = a.blocks[b];
            field = a.field ? a.field : a.fields[b];
            g = load_geo(B);
            s = make_float3(a.dt * B.inv_h[0], a.dt * B.inv_h[1], a.dt * B.inv_h[2]);
            idbase = B.base;
            nseeds = B.nseeds;
        }
        const int64_t s0 = grp * G;
        float3 r[PPT];
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
            const int i = k * 32 + lane;
            const float *u = P.rec + ((s0 >> 5) + k) * 128 + lane;
            r[k] = make_float3(0.f, 0.f, 0.f);
            if (i < cnt) r[k] = make_float3(__ldcs(u), __ldcs(u + 32), __ldcs(u + 64));
        }
        unsigned surv = 0;   // bit k: the lane's particle of round k survived
        bool term = false;
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
            const int i = k * 32 + lane;
            if (i < cnt) {
                float3 x = r[k], q;
                const int failed = rk4_step<LAYOUT>(x, field, g, s, q, a.err);
                if (failed == 0) {
                    r[k] = x;
                    surv |= 1u << k;
                } else {
                    term = true;
                    const int32_t id = __float_as_int(__ldcs(P.rec + ((s0 >> 5) + k) * 128 + 96 + lane));
                    if (BTO_IN_BOUNDS(id >= 0 && id < nseeds, a.err)) {
                        const int64_t gid = idbase + id;
                        __stcs(a.term + gid, make_float4(r[k].x, r[k].y, r[k].z, __int_as_float(a.cycle)));
                        // first outside point and its stage; clipped at the interval end
                        if (a.clip) __stcs(a.clip + gid, make_float4(q.x, q.y, q.z, __int_as_float(failed)));
                    }
                }
            }
        }
        if (!__any_sync(kFull, term)) {
            // nobody left: positions back in their slots, ids untouched
#pragma unroll
            for (int k = 0; k < PPT; ++k) {
                float *u = P.rec + ((s0 >> 5) + k) * 128 + lane;
                if (k * 32 + lane < cnt) {
                    __stcs(u, r[k].x);
                    __stcs(u + 32, r[k].y);
                    __stcs(u + 64, r[k].z);
                }
            }
        } else {
            // survivors to the front of the group; every id of the group is
            // read before the first write
            float id[PPT];
#pragma unroll
            for (int k = 0; k < PPT; ++k)
                id[k] = (surv >> k) & 1u ? __ldcs(P.rec + ((s0 >> 5) + k) * 128 + 96 + lane) : 0.f;
            int kept = 0;
#pragma unroll
            for (int k = 0; k < PPT; ++k) {
                const bool sv = (surv >> k) & 1u;
                const unsigned m = __ballot_sync(kFull, sv);
                if (sv) {
                    float *u = P.rec + part_at(s0 + kept + __popc(m & lt), 0);
                    __stcs(u, r[k].x);
                    __stcs(u + 32, r[k].y);
                    __stcs(u + 64, r[k].z);
                    __stcs(u + 96, id[k]);
                }
                kept += __popc(m);
            }
            if (lane == 0) P.gcnt[grp] = kept;
        }
    }
}

// ---------------------------------------------------------------------------
// K3i: all cycles of an interval in one launch, for a table that holds every
// cycle's fields (bto_launch_interval_graph). Particles are independent, so
// nothing orders one particle's cycle after another's: each warp takes one
// 32-slot unit of the list, keeps its particles in registers through all
// cycles, and writes its survivors and the group counts once, as the last
// per-cycle launch would have left them. A CTA is four units: a region is a
// multiple of 128 slots, so a CTA lies in one block and holds whole groups.
// Against a graph of one launch per cycle this drops the launches, their
// tails and the list's 24 bytes per particle and cycle: 96 blocks of 16 to 96
// cells with 7.5M seeds over 32 cycles 5.15 -> 3.76 ms (bound by the L1 load
// path). Short lists, which this leaves waiting for dependent samples, take
// interval_quad_kernel.
// ---------------------------------------------------------------------------
// CTAs of 128 per SM. F3: eight (64 registers, 20 bytes spilled); 3.76 ms on
// the 96 blocks against 3.92 at the compiler's own 72 registers, 4.80 at nine,
// and 885 us against 891 at seven on 200^3 cells seeded 1:1 over 8 cycles. F4:
// seven (72 registers, 28 bytes spilled; 64 spill 56): 3.45 ms against 3.67 at
// eight and 3.60 at six on 96 such blocks, 973 us against 1000 and 1029 on the
// 200^3, 194 against 208 and 215 on 20 blocks of 24 to 40 cells over 40 cycles.
template <int LAYOUT>
constexpr int kIntervalCtas = LAYOUT == LAYOUT_F4 ? 7 : 8;

template <int LAYOUT>
__global__ void __launch_bounds__(kRegionAlign, kIntervalCtas<LAYOUT>) interval_kernel(const AdvectArgs a,
                                                                                        const int32_t cycles,
                                                                                        const int group) {
    static_assert(kRegionAlign == 4 * kUnit, "a CTA is four units");
    __shared__ int kept[4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t s0 = (int64_t)blockIdx.x * kRegionAlign;   // the CTA's first slot
    const int64_t unit = (s0 >> 5) + warp;
    const int per = group / kUnit;                           // units of a group
    const int first = warp / per * per;                      // first unit of this warp's group, in the CTA
    const int64_t grp = (s0 + first * kUnit) / group;
    int cnt = a.p.gcnt[grp];
    if (!BTO_IN_BOUNDS(cnt >= 0 && cnt <= group, a.err)) cnt = 0;
    cnt -= (warp - first) * kUnit;                           // live particles from this unit on
    const int b = a.gblock[unit];
    const BlockDev &B = a.blocks[b];
    const Geo g = load_geo(B);
    const float3 s = make_float3(a.dt * B.inv_h[0], a.dt * B.inv_h[1], a.dt * B.inv_h[2]);
    float *rec = a.p.rec + unit * 128 + lane;
    bool alive = lane < cnt;
    float3 x = make_float3(0.f, 0.f, 0.f);
    int32_t id = 0;
    if (alive) {
        x = make_float3(__ldcs(rec), __ldcs(rec + 32), __ldcs(rec + 64));
        id = __float_as_int(__ldcs(rec + 96));
        if (!BTO_IN_BOUNDS(id >= 0 && id < B.nseeds, a.err)) alive = false;
    }
    const void *const *entry = a.fields + b;
    const void *next = *entry;
    for (int32_t c = 0; c < cycles && __any_sync(kFull, alive); ++c) {
        const void *field = next;
        if (c + 1 < cycles) {
            entry += a.nb;
            next = *entry;
        }
        if (alive) {
            float3 q;
            const float3 x0 = x;
            const int failed = rk4_step<LAYOUT>(x, field, g, s, q, a.err);
            if (failed) {
                alive = false;
                const int64_t gid = B.base + id;
                __stcs(a.term + gid, make_float4(x0.x, x0.y, x0.z, __int_as_float(c)));
                // first outside point and its stage; clipped at the interval end
                if (a.clip) __stcs(a.clip + gid, make_float4(q.x, q.y, q.z, __int_as_float(failed)));
            }
        }
    }
    // survivors of the group to its front, in order; every unit of the CTA
    // has been read before the first write
    const unsigned m = __ballot_sync(kFull, alive);
    if (lane == 0) kept[warp] = __popc(m);
    __syncthreads();
    int before = 0, total = 0;
    for (int w = first; w < first + per; ++w) {
        if (w < warp) before += kept[w];
        total += kept[w];
    }
    if (alive) {
        float *u = a.p.rec + part_at(s0 + first * kUnit + before + __popc(m & ((1u << lane) - 1u)), 0);
        __stcs(u, x.x);
        __stcs(u + 32, x.y);
        __stcs(u + 64, x.z);
        __stcs(u + 96, __int_as_float(id));
    }
    if (warp == first && lane == 0) a.p.gcnt[grp] = total;
}

// The same by four lanes per particle (rk4_step_quad): a CTA is one group. One
// 64^3 block with 10,648 seeds over 100 cycles: 648 us in a graph of one launch
// per cycle, 212 by interval_kernel (2 warps per SM), 121 so; bound by the
// latency of the dependent samples.
template <int LAYOUT>
__global__ void __launch_bounds__(4 * kRegionAlign) interval_quad_kernel(const AdvectArgs a, const int32_t cycles,
                                                                         const int group) {
    __shared__ int kept[kRegionAlign / 8];
    __shared__ int touched[4 * kRegionAlign];
    const uint32_t word = (uint32_t)__cvta_generic_to_shared(touched + threadIdx.x);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = threadIdx.x & 3;
    const int64_t s0 = (int64_t)blockIdx.x * group;   // the group's first slot
    const int k = threadIdx.x >> 2;                   // slot in the group
    int cnt = a.p.gcnt[blockIdx.x];
    if (!BTO_IN_BOUNDS(cnt >= 0 && cnt <= group, a.err)) cnt = 0;
    const int b = a.gblock[s0 / kUnit];
    const BlockDev &B = a.blocks[b];
    const Geo g = load_geo(B);
    const float3 s = make_float3(a.dt * B.inv_h[0], a.dt * B.inv_h[1], a.dt * B.inv_h[2]);
    const float *rec = a.p.rec + part_at(s0 + k, 0);
    bool alive = k < cnt;
    float3 x = make_float3(0.f, 0.f, 0.f);
    int32_t id = 0;
    if (alive) {
        x = make_float3(__ldcs(rec), __ldcs(rec + 32), __ldcs(rec + 64));
        id = __float_as_int(__ldcs(rec + 96));
        if (!BTO_IN_BOUNDS(id >= 0 && id < B.nseeds, a.err)) alive = false;
    }
    const void *const *entry = a.fields + b;
    const void *next = *entry;
    for (int32_t c = 0; c < cycles && __any_sync(kFull, alive); ++c) {
        const void *field = next;
        if (c + 1 < cycles) {
            entry += a.nb;
            next = *entry;
        }
        const float3 x0 = x;
        float3 out;
        const int failed = rk4_step_quad<LAYOUT>(x, field, g, s, out, alive,
                                                 Ahead{c + 1 < cycles ? next : nullptr, word}, a.err);
        if (failed) {
            alive = false;
            if (q == 0) {
                const int64_t gid = B.base + id;
                __stcs(a.term + gid, make_float4(x0.x, x0.y, x0.z, __int_as_float(c)));
                if (a.clip) __stcs(a.clip + gid, make_float4(out.x, out.y, out.z, __int_as_float(failed)));
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    // survivors to the front of the group, in order, a field to each lane of the quad
    const unsigned m = __ballot_sync(kFull, alive && q == 0);
    if (lane == 0) kept[warp] = __popc(m);
    __syncthreads();
    int before = 0, total = 0;
    for (int w = 0; w < group / 8; ++w) {
        if (w < warp) before += kept[w];
        total += kept[w];
    }
    if (alive) {
        const float v = q == 0 ? x.x : (q == 1 ? x.y : (q == 2 ? x.z : __int_as_float(id)));
        __stcs(a.p.rec + part_at(s0 + before + __popc(m & ((1u << (lane & ~3)) - 1u)), q), v);
    }
    if (threadIdx.x == 0) a.p.gcnt[blockIdx.x] = total;
}

// ---------------------------------------------------------------------------
// K2: seeds. Slot i of block b's region holds the lattice point perm[base + m]
// (m = i - slot_base; brick order of the lattice); positions are the exact
// integers j*s in cell units. Also sets every group's live count.
// ---------------------------------------------------------------------------
__global__ void seed_kernel(const BlockDev *__restrict__ blocks, const int32_t *__restrict__ gblock,
                            const int32_t *__restrict__ perm, int64_t slots, int group, PartList P) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < slots; i += stride) {
        const BlockDev &B = blocks[gblock[i / kUnit]];
        const int64_t m = i - B.slot_base;
        if (i % group == 0) {
            const int64_t left = B.nseeds - m;
            P.gcnt[i / group] = (int32_t)(left < 0 ? 0 : (left > group ? group : left));
        }
        if (m >= B.nseeds) continue;
        const int32_t p = perm[B.base + m];
        const int32_t jx = p % B.S[0];
        const int32_t jy = (p / B.S[0]) % B.S[1];
        const int32_t jz = p / (B.S[0] * B.S[1]);
        float *u = P.rec + part_at(i, 0);
        u[0] = (float)(jx * B.stride);
        u[32] = (float)(jy * B.stride);
        u[64] = (float)(jz * B.stride);
        u[96] = __int_as_float(p);
    }
}

// K4: the end of an interval of an untiled list: basis flows (and, when
// asked, clipped exit locations and times), termination records cleared, and
// the next interval's seeds, in one pass over the slots. Bound by HBM. As
// three kernels (live particles, terminated particles over all term records,
// seeds) the pass read and wrote half as much again: 16.8M particles 319 us,
// 270 us so; a small block's three launches become one.
//
// A slot's seed is perm[] of its place in the list; in a group that lost no
// particle it is also the id the slot still holds, so perm is read, and the
// slot's seed looked up among the terminated particles, only in the others.
// A CTA is one region unit of 128 slots, which holds whole groups.
struct EndArgs {
    const BlockDev *blocks;
    const int32_t *gblock;
    const int32_t *perm;
    PartList p;
    float4 *term;
    const float4 *clip;
    float *seeds, *ends;
    uint8_t *valid;
    int32_t *exit_cycle;
    float *exit_pos, *exit_time;
    int32_t *err;
    int group;
};

// Writes v of each lane to out[3 at], 12 bytes. Where the warp's particles
// are consecutive (a full run of seeds along x), the 384 bytes go through
// shared memory and leave as three stores of whole 128-byte lines; as three
// 12-byte-strided stores every sector would be written three times.
__device__ __forceinline__ void store3(float *__restrict__ out, bool on, int64_t at, const float3 v, float *stage) {
    const int lane = threadIdx.x & 31;
    const int64_t first = __shfl_sync(kFull, (long long)at, 0);
    if (__all_sync(kFull, on && at == first + lane)) {
        stage[3 * lane] = v.x;
        stage[3 * lane + 1] = v.y;
        stage[3 * lane + 2] = v.z;
        __syncwarp();
        float *o = out + 3 * first + lane;
        o[0] = stage[lane];
        o[32] = stage[lane + 32];
        o[64] = stage[lane + 64];
        __syncwarp();
    } else if (on) {
        out[3 * at] = v.x;
        out[3 * at + 1] = v.y;
        out[3 * at + 2] = v.z;
    }
}

__global__ void __launch_bounds__(kRegionAlign) end_interval_kernel(const EndArgs a) {
    __shared__ float stage_all[kRegionAlign / 32][96];
    // Launched programmatically itself (its launch overlaps the last cycle's
    // tail); what follows it on the stream starts when it has completed, as
    // after an ordinary launch: only the cycle calls let a caller's
    // programmatic kernel start early.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    float *stage = stage_all[threadIdx.x >> 5];
    const int64_t i = (int64_t)blockIdx.x * kRegionAlign + threadIdx.x;
    // the slot's record and its group's count do not wait for the block's geometry
    float *u = a.p.rec + part_at(i, 0);
    const float3 xi = make_float3(__ldcs(u), __ldcs(u + 32), __ldcs(u + 64));
    const int32_t id = __float_as_int(__ldcs(u + 96));
    const int64_t g = i / a.group;
    const int k = (int)(i % a.group);
    const int cnt = a.p.gcnt[g];
    const BlockDev &B = a.blocks[a.gblock[i / kUnit]];
    const int64_t m = i - B.slot_base;
    const int64_t left = B.nseeds - (m - k);
    const int full = (int)(left < 0 ? 0 : (left > a.group ? a.group : left));   // seeds of the group
    const float nan = __int_as_float(0x7fc00000);
    const bool live = k < cnt && BTO_IN_BOUNDS(id >= 0 && id < B.nseeds, a.err);
    const int64_t gid = B.base + id;
    store3(a.ends, live, gid,
           make_float3(fmaf(xi.x, B.h[0], B.origin[0]), fmaf(xi.y, B.h[1], B.origin[1]), fmaf(xi.z, B.h[2], B.origin[2])),
           stage);
    if (a.exit_pos) store3(a.exit_pos, live, gid, make_float3(nan, nan, nan), stage);
    if (live) {
        a.valid[gid] = 1;
        if (a.exit_cycle) a.exit_cycle[gid] = -1;
        if (a.exit_time) a.exit_time[gid] = nan;
    }
    const bool seed = m < B.nseeds;
    int32_t p = id;
    if (seed && (cnt != full || !live)) {
        p = a.perm[B.base + m];
        u[96] = __int_as_float(p);
        const int64_t tid = B.base + p;
        const float4 r = a.term[tid];
        const int e = __float_as_int(r.w);
        if (e >= 0) {
            a.ends[3 * tid + 0] = fmaf(r.x, B.h[0], B.origin[0]);
            a.ends[3 * tid + 1] = fmaf(r.y, B.h[1], B.origin[1]);
            a.ends[3 * tid + 2] = fmaf(r.z, B.h[2], B.origin[2]);
            a.valid[tid] = 0;
            if (a.exit_cycle) a.exit_cycle[tid] = e;
            if (a.exit_pos || a.exit_time) {
                const float4 qs = a.clip[tid];
                const float4 cl = clip_exit(make_float3((float)B.n[0], (float)B.n[1], (float)B.n[2]),
                                            make_float3(r.x, r.y, r.z), make_float3(qs.x, qs.y, qs.z),
                                            __float_as_int(qs.w), e);
                if (a.exit_pos) {
                    a.exit_pos[3 * tid + 0] = fmaf(cl.x, B.h[0], B.origin[0]);
                    a.exit_pos[3 * tid + 1] = fmaf(cl.y, B.h[1], B.origin[1]);
                    a.exit_pos[3 * tid + 2] = fmaf(cl.z, B.h[2], B.origin[2]);
                }
                if (a.exit_time) a.exit_time[tid] = cl.w;
            }
            a.term[tid] = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
        }
    }
    const int32_t jx = p % B.S[0], jy = (p / B.S[0]) % B.S[1], jz = p / (B.S[0] * B.S[1]);
    const float3 s = make_float3((float)(jx * B.stride), (float)(jy * B.stride), (float)(jz * B.stride));
    store3(a.seeds, seed, B.base + p,
           make_float3(fmaf(s.x, B.h[0], B.origin[0]), fmaf(s.y, B.h[1], B.origin[1]), fmaf(s.z, B.h[2], B.origin[2])),
           stage);
    if (seed) {
        u[0] = s.x;
        u[32] = s.y;
        u[64] = s.z;
    }
    __syncthreads();   // every slot of the group has read its live count
    if (k == 0) a.p.gcnt[g] = full;
}

// K4a: particles alive at the end of the interval.
__global__ void write_live_kernel(const BlockDev *__restrict__ blocks,
                                  const int32_t *__restrict__ gblock, const PartList P,
                                  int64_t slots, int group, float *__restrict__ ends,
                                  uint8_t *__restrict__ valid, int32_t *__restrict__ exit_cycle,
                                  int32_t *__restrict__ err) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < slots; i += stride) {
        if (i % group >= P.gcnt[i / group]) continue;
        const BlockDev &B = blocks[gblock[i / kUnit]];
        const float *u = P.rec + part_at(i, 0);
        const int32_t id = __float_as_int(u[96]);
        if (!BTO_IN_BOUNDS(id >= 0 && id < B.nseeds, err)) continue;
        const int64_t gid = B.base + id;
        ends[3 * gid + 0] = fmaf(u[0], B.h[0], B.origin[0]);
        ends[3 * gid + 1] = fmaf(u[32], B.h[1], B.origin[1]);
        ends[3 * gid + 2] = fmaf(u[64], B.h[2], B.origin[2]);
        if (valid) valid[gid] = 1;
        if (exit_cycle) exit_cycle[gid] = -1;
    }
}

// K4b: seeds of every particle, plus end/valid/exit of the terminated ones
// (and, when asked, their clipped exit location and time); clears the
// termination record for the next interval.
__global__ void write_term_kernel(const BlockDev *__restrict__ blocks, int32_t nb, int64_t P,
                                  float4 *__restrict__ term, float *__restrict__ seeds,
                                  float *__restrict__ ends, uint8_t *__restrict__ valid,
                                  int32_t *__restrict__ exit_cycle, const float4 *__restrict__ clip,
                                  float *__restrict__ exit_pos, float *__restrict__ exit_time) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; gid < P; gid += stride) {
        const int b = nb == 1 ? 0 : find_block(blocks, nb, gid);
        const BlockDev &B = blocks[b];
        const int32_t p = (int32_t)(gid - B.base);
        if (seeds) {
            const int32_t jx = p % B.S[0];
            const int32_t jy = (p / B.S[0]) % B.S[1];
            const int32_t jz = p / (B.S[0] * B.S[1]);
            seeds[3 * gid + 0] = fmaf((float)(jx * B.stride), B.h[0], B.origin[0]);
            seeds[3 * gid + 1] = fmaf((float)(jy * B.stride), B.h[1], B.origin[1]);
            seeds[3 * gid + 2] = fmaf((float)(jz * B.stride), B.h[2], B.origin[2]);
        }
        const float4 r = term[gid];
        const int e = __float_as_int(r.w);
        if (e >= 0) {
            if (ends) {
                ends[3 * gid + 0] = fmaf(r.x, B.h[0], B.origin[0]);
                ends[3 * gid + 1] = fmaf(r.y, B.h[1], B.origin[1]);
                ends[3 * gid + 2] = fmaf(r.z, B.h[2], B.origin[2]);
            }
            if (valid) valid[gid] = 0;
            if (exit_cycle) exit_cycle[gid] = e;
            if (clip && (exit_pos || exit_time)) {
                const float4 qs = clip[gid];
                const float4 cl = clip_exit(make_float3((float)B.n[0], (float)B.n[1], (float)B.n[2]),
                                            make_float3(r.x, r.y, r.z), make_float3(qs.x, qs.y, qs.z),
                                            __float_as_int(qs.w), e);
                if (exit_pos) {
                    exit_pos[3 * gid + 0] = fmaf(cl.x, B.h[0], B.origin[0]);
                    exit_pos[3 * gid + 1] = fmaf(cl.y, B.h[1], B.origin[1]);
                    exit_pos[3 * gid + 2] = fmaf(cl.z, B.h[2], B.origin[2]);
                }
                if (exit_time) exit_time[gid] = cl.w;
            }
            term[gid] = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
        } else if (exit_pos || exit_time) {
            const float nan = __int_as_float(0x7fc00000);
            if (exit_pos) {
                exit_pos[3 * gid + 0] = nan;
                exit_pos[3 * gid + 1] = nan;
                exit_pos[3 * gid + 2] = nan;
            }
            if (exit_time) exit_time[gid] = nan;
        }
    }
}

// Diagnostics: live particles of each group copied to dst[g] + k as
// (xi, block-local id bits).
__global__ void gather_live_kernel(const PartList P, const int64_t *__restrict__ dst, int64_t slots,
                                   int group, float4 *__restrict__ out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < slots; i += stride) {
        const int64_t g = i / group;
        const int k = (int)(i % group);
        if (k < P.gcnt[g]) {
            const float *u = P.rec + part_at(i, 0);
            out[dst[g] + k] = make_float4(u[0], u[32], u[64], u[96]);
        }
    }
}

// H1 ingest: repack one block's F3 field (12 bytes per node) into F4 (16 bytes
// per node, pad 0) so that the advection kernel can gather a node with one
// 16-byte load. Four nodes per thread: three 16-byte loads of 48 contiguous
// bytes, four 16-byte stores (scalar loads when the field is not 16-byte
// aligned and for the last nodes).
__global__ void ingest_f3_f4_kernel(const void *__restrict__ field, const void *const *__restrict__ fields,
                                    int b, int64_t nodes, float4 *__restrict__ out) {
    const float *f = reinterpret_cast<const float *>(field ? field : fields[b]);
    const bool vec = (reinterpret_cast<uintptr_t>(f) & 15u) == 0;
    const int64_t quads = nodes / 4;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < quads; q += stride) {
        float v[12];
        if (vec) {
            const float4 *p = reinterpret_cast<const float4 *>(f) + 3 * q;
            const float4 a = __ldcs(p), bb = __ldcs(p + 1), c = __ldcs(p + 2);
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = bb.x; v[5] = bb.y;
            v[6] = bb.z; v[7] = bb.w; v[8] = c.x; v[9] = c.y; v[10] = c.z; v[11] = c.w;
        } else {
#pragma unroll
            for (int k = 0; k < 12; ++k) v[k] = __ldcs(f + 12 * q + k);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) out[4 * q + k] = make_float4(v[3 * k], v[3 * k + 1], v[3 * k + 2], 0.f);
    }
    for (int64_t i = quads * 4 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nodes; i += stride)
        out[i] = make_float4(__ldcs(f + 3 * i), __ldcs(f + 3 * i + 1), __ldcs(f + 3 * i + 2), 0.f);
}

// Each cycle's grid is launched with programmatic stream serialisation, so
// its launch and CTA set-up overlap the previous cycle's tail.
template <int LAYOUT, int NT, int PPT, bool BATCHED, int MINB>
cudaError_t launch_t(const AdvectArgs &a, int grid, size_t dyn, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = dyn;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, advect_kernel<LAYOUT, NT, PPT, BATCHED, MINB>, a);
}

template <int LAYOUT, int NT, int PPT, bool BATCHED, int MINB>
cudaError_t occ_t(size_t dyn, int *n) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        n, advect_kernel<LAYOUT, NT, PPT, BATCHED, MINB>, NT, dyn);
}

// Dispatch over the compiled launch shapes: threads per CTA, particles per
// thread, and whether registers are capped at 80 (768 threads per SM).
#define BTO_SHAPES(X, L, B)                                                                  \
    X(L, 128, 1, B, 1) X(L, 128, 2, B, 1) X(L, 128, 4, B, 1) X(L, 256, 1, B, 1)                \
    X(L, 256, 2, B, 1) X(L, 256, 4, B, 1) X(L, 128, 1, B, 6) X(L, 128, 2, B, 6)                \
    X(L, 128, 4, B, 6) X(L, 256, 1, B, 3) X(L, 256, 2, B, 3) X(L, 256, 4, B, 3)

}  // namespace

BTO_BOUNDS_ACCESSOR(bounds_failures_kernels)

cudaError_t launch_advect(const AdvectArgs &a, int layout, int nt, int ppt, bool cap, int grid,
                          size_t dyn, cudaStream_t s) {
    const bool batched = a.nb > 1;
#define BTO_CASE(L, T, P, B, M)                                                     \
    if (layout == L && nt == T && ppt == P && batched == B && cap == (M > 1))       \
        return launch_t<L, T, P, B, M>(a, grid, dyn, s);
    BTO_SHAPES(BTO_CASE, LAYOUT_F3, false)
    BTO_SHAPES(BTO_CASE, LAYOUT_F4, false)
    BTO_SHAPES(BTO_CASE, LAYOUT_F3, true)
    BTO_SHAPES(BTO_CASE, LAYOUT_F4, true)
#undef BTO_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_interval(const AdvectArgs &a, int layout, int32_t cycles, int64_t slots, int group, bool quad,
                            cudaStream_t s) {
    if (quad) {
        const unsigned groups = (unsigned)(slots / group);
        if (layout == LAYOUT_F4)
            interval_quad_kernel<LAYOUT_F4><<<groups, 4 * group, 0, s>>>(a, cycles, group);
        else
            interval_quad_kernel<LAYOUT_F3><<<groups, 4 * group, 0, s>>>(a, cycles, group);
        return cudaGetLastError();
    }
    const unsigned grid = (unsigned)(slots / kRegionAlign);
    if (layout == LAYOUT_F4)
        interval_kernel<LAYOUT_F4><<<grid, kRegionAlign, 0, s>>>(a, cycles, group);
    else
        interval_kernel<LAYOUT_F3><<<grid, kRegionAlign, 0, s>>>(a, cycles, group);
    return cudaGetLastError();
}

cudaError_t advect_occupancy(int layout, int nt, int ppt, bool cap, bool batched, size_t dyn,
                             int *n) {
#define BTO_CASE(L, T, P, B, M)                                                     \
    if (layout == L && nt == T && ppt == P && batched == B && cap == (M > 1))       \
        return occ_t<L, T, P, B, M>(dyn, n);
    BTO_SHAPES(BTO_CASE, LAYOUT_F3, false)
    BTO_SHAPES(BTO_CASE, LAYOUT_F4, false)
    BTO_SHAPES(BTO_CASE, LAYOUT_F3, true)
    BTO_SHAPES(BTO_CASE, LAYOUT_F4, true)
#undef BTO_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_seed(const BlockDev *blocks, const int32_t *gblock, const int32_t *perm,
                        int64_t slots, int group, PartList p, int grid, cudaStream_t s) {
    seed_kernel<<<grid, 256, 0, s>>>(blocks, gblock, perm, slots, group, p);
    return cudaGetLastError();
}

cudaError_t launch_end_interval(const BlockDev *blocks, const int32_t *gblock, const int32_t *perm, int64_t slots,
                                int group, PartList p, float4 *term, const float4 *clip, float *seeds, float *ends,
                                uint8_t *valid, int32_t *exit_cycle, float *exit_pos, float *exit_time, int32_t *err,
                                cudaStream_t s) {
    const EndArgs a{blocks, gblock, perm, p, term, clip, seeds, ends, valid, exit_cycle, exit_pos, exit_time, err, group};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(slots / kRegionAlign));
    cfg.blockDim = dim3(kRegionAlign);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, end_interval_kernel, a);
}

cudaError_t launch_write_live(const BlockDev *blocks, const int32_t *gblock, PartList p, int64_t slots,
                              int group, float *ends, uint8_t *valid, int32_t *exit_cycle, int grid,
                              cudaStream_t s, int32_t *err) {
    write_live_kernel<<<grid, 256, 0, s>>>(blocks, gblock, p, slots, group, ends, valid, exit_cycle, err);
    return cudaGetLastError();
}

cudaError_t launch_gather_live(PartList p, const int64_t *dst, int64_t slots, int group, float4 *out,
                               int grid, cudaStream_t s) {
    gather_live_kernel<<<grid, 256, 0, s>>>(p, dst, slots, group, out);
    return cudaGetLastError();
}

cudaError_t launch_ingest(const void *field, const void *const *fields, int b, int64_t nodes, float4 *out,
                          int grid, cudaStream_t s) {
    ingest_f3_f4_kernel<<<grid, 256, 0, s>>>(field, fields, b, nodes, out);
    return cudaGetLastError();
}

cudaError_t launch_write_term(const BlockDev *blocks, int32_t nb, int64_t P, float4 *term,
                              float *seeds, float *ends, uint8_t *valid, int32_t *exit_cycle,
                              int grid, cudaStream_t s, const float4 *clip, float *exit_pos,
                              float *exit_time) {
    write_term_kernel<<<grid, 256, 0, s>>>(blocks, nb, P, term, seeds, ends, valid, exit_cycle, clip,
                                           exit_pos, exit_time);
    return cudaGetLastError();
}

}  // namespace bto

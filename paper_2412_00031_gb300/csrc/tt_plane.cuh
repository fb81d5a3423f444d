// What the plane sweeps (tt_plane.cu: forward, adjoint) share: the planes of a time step, the list of
// sources that still iterate, the vector accesses of a thread's sources and the launch shape.
#pragma once

#include <algorithm>
#include <cstring>

#include "tt_internal.h"
#include "tt_update.cuh"

namespace ttgb {

// Threads of an SM: 80 registers a thread. Fewer threads of more registers are slower, also where
// they would not spill (the Godunov updates): 121x161x161 x 256 sources, a whole solve with 384 / 512 /
// 640 / 768 threads 547 / 464 / 429 / 408 ms, Lax-Friedrichs 4163 / 3458 / 3068 / 2852.
constexpr int kPlaneThreads = 768;

// NS neighbouring sources of one node: one load or store.
__device__ __forceinline__ void ld_pack(const float *p, float (&v)[1]) { v[0] = *p; }
__device__ __forceinline__ void ld_pack(const double *p, double (&v)[1]) { v[0] = *p; }
__device__ __forceinline__ void ld_pack(const float *p, float (&v)[2]) {
    const float2 t = *reinterpret_cast<const float2 *>(p);
    v[0] = t.x;
    v[1] = t.y;
}
__device__ __forceinline__ void st_pack(float *p, const float (&v)[1]) { *p = v[0]; }
__device__ __forceinline__ void st_pack(double *p, const double (&v)[1]) { *p = v[0]; }
__device__ __forceinline__ void st_pack(float *p, const float (&v)[2]) {
    *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
}

// The planes of a time step: of orderings o0, o0 + 1, o0 + 2 the first list entry q and the count c.
struct Planes {
    int o0, q[3], c[3];
    __device__ __forceinline__ int total() const { return c[0] + c[1] + c[2]; }
};

// The schedule of an iteration: off (shared memory) and nodes as in Schedule, start (shared
// memory) the orderings' first time steps.
struct PlaneSched {
    const int *off, *start;
    const unsigned *nodes;
    int n_planes, steps;
    // the planes of time step tau; o0: the first ordering in progress one step before
    __device__ __forceinline__ void planes(Planes &d, int tau, int o0) const {
        if (tau - start[o0] >= n_planes && o0 < 7) ++o0;
        d.o0 = o0;
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            const int o = o0 + u, L = tau - start[o & 7];
            d.q[u] = 0;
            d.c[u] = 0;
            if (o < 8 && tau < steps && L >= 0 && L < n_planes) {
                d.q[u] = off[L];
                d.c[u] = off[L + 1] - d.q[u];
            }
        }
    }
    // node x of the concatenated planes and its ordering
    __device__ __forceinline__ unsigned entry(const Planes &d, int x, int &o) const {
        const int u = x < d.c[0] ? 0 : x < d.c[0] + d.c[1] ? 1 : 2;
        o = d.o0 + u;
        return __ldg(nodes + (u == 0 ? d.q[0] + x : u == 1 ? d.q[1] + (x - d.c[0]) : d.q[2] + (x - d.c[0] - d.c[1])));
    }
};

// How a thread holds its sources of a group of n.
enum Deal {
    kPairs,    // one, or two neighbours (2 u and 2 u + 1) by vector accesses: rows of whole aligned pairs
    kHalves,   // u and u + (n + 1) / 2, scalar accesses, coalesced like a single source's; any n, any place
    kApart,    // two neighbours by scalar accesses; any n, any place
};
template <int NS, int DEAL> struct Dealt {
    static_assert(NS == 2 || DEAL == kPairs, "");
    static __device__ __forceinline__ int units(int n) { return (n + NS - 1) / NS; }
    static __device__ __forceinline__ int first(int u) { return DEAL == kHalves ? u : u * NS; }
    // distance of a unit's second source from its first; 0: there is none (the last unit of an odd n)
    static __device__ __forceinline__ int step(int u, int n) {
        if (DEAL == kPairs) return 1;
        const int d = DEAL == kHalves ? (n + 1) / 2 : 1;
        return first(u) + d < n ? d : 0;
    }
};

// The field values at p of a thread's sources; off: Dealt's step.
template <int DEAL, typename F, int NS>
__device__ __forceinline__ void ld_src(const F *p, int off, F (&v)[NS]) {
    if constexpr (DEAL != kPairs) {
        v[0] = p[0];
        v[1] = p[off];
    } else {
        ld_pack(p, v);
    }
}
// v to p where its bits differ from those of old: a line of values that all stay is not made dirty
template <int DEAL, typename F, int NS>
__device__ __forceinline__ void st_moved(F *p, int off, const F (&v)[NS], const F (&old)[NS]) {
    bool moved[NS], any = false;
#pragma unroll
    for (int h = 0; h < NS; ++h) {
        moved[h] = bits_of(v[h]) != bits_of(old[h]);
        any = any || moved[h];
    }
    if constexpr (DEAL != kPairs) {
        if (moved[0]) p[0] = v[0];
        if (moved[1]) p[off] = v[1];
    } else if (any) {
        st_pack(p, v);
    }
}

// list = the units of sources of which one is on, in order; returns their number. One warp.
template <int NS, int DEAL> __device__ __forceinline__ int plane_units(const unsigned char *on_, int n_src, int *list) {
    using D = Dealt<NS, DEAL>;
    const int units = D::units(n_src);
    int n = 0;
    const int lane = threadIdx.x & 31;
    for (int u0 = 0; u0 < units; u0 += 32) {
        const int u = u0 + lane;
        bool on = false;
        if (u < units) {
            on = on_[D::first(u)];
            if (NS == 2) on = on || on_[D::first(u) + D::step(u, n_src)];
        }
        const unsigned mask = __ballot_sync(0xffffffffu, on);
        if (on) list[n + __popc(mask & ((1u << lane) - 1u))] = u;
        n += __popc(mask);
    }
    return n;
}

// Start times of the 8 orderings of an iteration over a box na x nb x nc: o + 1 flips the axes of
// the bits that change. At most three orderings are in progress at a time.
inline void plane_starts(PlaneShape &m, int na, int nb, int nc) {
    const int planes = na + nb + nc - 2;
    m.start[0] = 0;
    for (int o = 1; o < 8; ++o) {
        const int f = o ^ (o - 1);
        int d = 2 + (f & 4 ? na - 1 : 0) + (f & 2 ? nb - 1 : 0) + (f & 1 ? nc - 1 : 0);
        if (d > planes) d = planes;
        m.start[o] = m.start[o - 1] + d;
        if (o >= 3 && m.start[o] < m.start[o - 3] + planes) m.start[o] = m.start[o - 3] + planes;
    }
    m.steps = m.start[7] + planes;
}

// Two sources a thread where a time step has more updates than a line times the SMs: half the
// instructions and packed arithmetic an update; below it a thread per source has the shorter step. The
// line depends on the solver (Godunov pairs spill) and on how the sources are dealt: a batch or field
// without whole aligned pairs takes scalar accesses, in halves or, in the adjoint, as neighbours (its
// rows come from DRAM: 3 iterations at 121x161x161 x 111 single / halves / apart 116 / 126 / 99 ms).
// Single / two beside the lines, ms of 6 iterations in LF, 3 in the others (updates a step and SM):
//   LF pairs         41^3 x 96 10.1 / 10.2 (549), 41^3 x 128 10.9 / 10.7 (732), 81^3 x 64 31.0 / 29.0
//   LF halves        121x161x161 x 15 57.4 / 59.3 (1107), 41^3 x 255 15.4 / 14.7 (1458)
//   Godunov pairs    41x61x67 x 256 22.5 / 23.2 (2416), 121x161x161 x 40 65.6 / 64.4 (2951)
//   Godunov halves   41^3 x 699 21.6 / 21.9 (3997), 41x61x67 x 511 37.0 / 35.6 (4823)
//   isotropic pairs  41^3 x 384 13.5 / 13.5 (2196), 121x161x161 x 32 52.4 / 51.7 (2361)
//   isotropic halves 41x61x67 x 255 21.3 / 21.6 (2407), 81^3 x 127 32.4 / 31.6 (2980)
//   teleseismic      81x101x101 x 23, a whole solve, halves 138 / 129 (696)
//   adjoint pairs    81^3 x 24 11.4 / 11.8 (592), 81^3 x 32 13.4 / 12.4 (789)
//   adjoint apart    121x161x161 x 23 40.7 / 42.9 (1746), x 31 48.2 / 44.6 (2354)
// At 121x161x161 x 255: LF 361 -> 256, Godunov 291 -> 250, adjoint 234 -> 194 (256: 244, 245, 174).
constexpr int kAdjointSolver = -1;
inline bool plane_two(const PlaneShape &m, int na, int nb, int nc, int n, int solver, bool pairs, int n_sm) {
    const int line = solver == 0   ? (pairs ? kPlaneThreads : 1300)
                     : solver == 1 ? (pairs ? 2300 : 2900)
                     : solver == 2 ? (pairs ? 2900 : 4300)
                     : solver == 3 ? kPlaneThreads
                                   : (pairs ? kPlaneThreads : 2000);
    return n > 1 && 8.0 * na * nb * nc / m.steps * n > (double)line * n_sm;
}

// Blocks, threads and barrier groups (0 = 1) for n sources, ns to a thread; smem: dynamic shared
// memory. One block an SM and group, so that a barrier has as few arrivals as there are SMs (a
// barrier of 608 blocks takes 2.5 us, of 152 1.6 us); no more threads than the widest plane has
// nodes and sources. cudaErrorInvalidConfiguration: the sources exceed one resident launch.
inline cudaError_t plane_shape(PlaneShape &m, const void *fn, size_t smem, int na, int nb, int nc, int n, int ns,
                               int groups, int max_threads, int n_sm, int launch_blocks, PlaneLaunch *launch) {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
        return e;
    if (groups <= 0) groups = 1;
    if (groups > kMaxBarrierGroups) groups = kMaxBarrierGroups;
    if (groups > (n + 31) / 32) groups = (n + 31) / 32;
    int threads = max_threads / groups / 32 * 32;
    const int ext[3] = {na, nb, nc};
    long long widest = 0;
    for (int x = 0; x < 3; ++x)
        for (int y = x + 1; y < 3; ++y) widest = std::max(widest, (long long)ext[x] * ext[y]);
    const long long want = (widest * ((n + ns - 1) / ns) / groups / n_sm + 31) / 32 * 32;
    if (want < threads) threads = want < 32 ? 32 : (int)want;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem)) != cudaSuccess) return e;
    if (per_sm <= 0) return cudaErrorInvalidConfiguration;
    if (per_sm > groups) per_sm = groups;
    int most = per_sm * n_sm;
    if (launch_blocks > 0 && launch_blocks < most) most = launch_blocks;
    if (groups > most) groups = most;
    m.grp_src = ((n + groups - 1) / groups + ns - 1) / ns * ns;
    groups = (n + m.grp_src - 1) / m.grp_src;
    m.grp_blocks = most / groups;
    // a group's blocks hold at least one thread per source
    const int need = ((m.grp_src + ns - 1) / ns + threads - 1) / threads;
    if (m.grp_blocks < need) m.grp_blocks = need;
    if ((long long)m.grp_blocks * groups > (long long)per_sm * n_sm) return cudaErrorInvalidConfiguration;
    launch->grid = m.grp_blocks * groups;
    launch->block = threads;
    return cudaSuccess;
}

}  // namespace ttgb

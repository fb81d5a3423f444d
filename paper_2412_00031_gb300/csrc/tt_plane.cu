// Plane-by-plane forward sweep: the schedule of the forward solves and of the teleseismic region
// solve (SCHEME 3: Lax-Friedrichs on T itself with T0 = 1, no fixed set, the faces held fixed).
//
// A time step updates the nodes of one hyperplane (Sec. 3.4) of each ordering in progress, then
// crosses the group's grid barrier. Barriers, the round trips of a step's loads and planes too
// small to fill the GPU bound a solve, far above its bytes and operations:
//
//  - Ordering o + 1 starts before ordering o has ended: node x may be updated in o + 1 as soon as
//    x and its six neighbours have been updated in o, which holds everywhere once o is
//    (sum of the flipped axes' lengths) + 2 planes ahead. An iteration of 8 orderings then takes
//    8 c + 4 b + 2 a time steps instead of 8 (a + b + c) planes for a box a x b x c (a along r),
//    and a time step has the nodes of two planes to spread over the GPU.
//  - The faces are extrapolated by the threads that complete their two layers, in place of three
//    passes and barriers per ordering. Nodes on two faces are not read by any interior update:
//    they are set once after the solve (edge_kernel).
//  - One block per SM and barrier group (run_plane_forward), threads over (node, source) without
//    padding to whole warps of sources, consecutive warps on different SMs.
//  - In large batches a thread holds two neighbouring sources: one load per stencil point, and
//    packed FP32 arithmetic.
//
// Each update reads what it reads in the lexicographic order, so the bits are the same.
//  - Threads are dealt to the sources that still iterate, anew every iteration.
// Measured, ms of a solve, with a barrier per plane and 456 or 608 blocks / now (one GB300):
// 41^3 x 1 source FP64 352 / 64; 121x161x161 x 1 (Godunov) 107 / 49; 67x83x95 x 37 378 / 212;
// 81^3 x 64 353 / 231; 101x141x151 x 112 1377 / 1197; 121x161x161 x 256 (Godunov) 483 / 434;
// 81x101x101 x 24 events 430 / 189. Of a time step's 4 us at 81^3 x 64 the barrier and the schedule
// take 2.2; at 101x141x151 x 112 it is 7.5 us, four rounds of loads and updates of 1.3 us each.
// Measured and not kept: loading the next node's factors ahead (also across the barrier), an L2
// prefetch of them, a warp of its own for the barrier, four sources a thread: all slower.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "tt_internal.h"
#include "tt_update.cuh"

namespace ttgb {

namespace {

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

__device__ __forceinline__ NodeRec<float> ld_rec(const NodeRec<float> *r) {
    const float4 a = __ldg(reinterpret_cast<const float4 *>(r)), b = __ldg(reinterpret_cast<const float4 *>(r) + 1);
    return NodeRec<float>{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
}
__device__ __forceinline__ NodeRec<double> ld_rec(const NodeRec<double> *r) {
    const double2 *q = reinterpret_cast<const double2 *>(r);
    const double2 a = __ldg(q), b = __ldg(q + 1), c = __ldg(q + 2), d = __ldg(q + 3);
    return NodeRec<double>{a.x, a.y, b.x, b.y, c.x, c.y, d.x, d.y};
}
// The factors are read once per sweep: streamed past what the planes keep in L2.
__device__ __forceinline__ Vec4<float> ld_fac(const Vec4<float> *p) {
    const float4 v = __ldcs(reinterpret_cast<const float4 *>(p));
    return Vec4<float>{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Vec4<double> ld_fac(const Vec4<double> *p) {
    const double2 a = __ldcs(reinterpret_cast<const double2 *>(p)), b = __ldcs(reinterpret_cast<const double2 *>(p) + 1);
    return Vec4<double>{a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ Fac2 ld_fac2(const float4 *p) {
    const float4 a = __ldcs(p), b = __ldcs(p + 1);
    return Fac2{make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(b.x, b.y), make_float2(b.z, b.w)};
}

// Updates of a thread's sources at one node: v[q] the stencil (centre, r+, r-, theta+, theta-,
// phi+, phi-), tn the new values (the old ones on a fixed set or for a converged source).
template <typename F, int NS> struct FacOf { using type = Vec4<F>; };
template <> struct FacOf<float, 2> { using type = Fac2; };
template <typename F, int SCHEME, int NS> struct Update {
    using Fac = typename FacOf<F, NS>::type;
    static __device__ __forceinline__ Fac load(const Vec4<F> *pc) {
        if constexpr (SCHEME == 3) {
            Fac f{};
            if constexpr (NS == 1) f.x = (F)1;
            else f.x = both_(1.f);
            return f;
        } else if constexpr (NS == 1) {
            return ld_fac(pc);
        } else {
            return ld_fac2(reinterpret_cast<const float4 *>(pc));
        }
    }
    static __device__ __forceinline__ void run(const Fac &f, const F (&v)[7][NS], const NodeRec<F> &R, F er,
                                               const bool (&act)[NS], F (&tn)[NS], F (&err)[NS]) {
        if constexpr (NS == 1) {
            const F s[7] = {v[0][0], v[1][0], v[2][0], v[3][0], v[4][0], v[5][0], v[6][0]};
            tn[0] = s[0];
            if (f.x > (F)0) {
                tn[0] = sweep_update<F, SCHEME>(s, f, R, er);
                err[0] = fmax_(err[0], fabs(tn[0] - s[0]));
            }
        } else {
            float2 s[7];
#pragma unroll
            for (int q = 0; q < 7; ++q) s[q] = make_float2(v[q][0], v[q][1]);
            const float2 t = sweep_update2<SCHEME>(s, f, R, er);
            tn[0] = act[0] && f.x.x > 0.f ? t.x : s[0].x;
            tn[1] = act[1] && f.x.y > 0.f ? t.y : s[0].y;
            err[0] = fmax_(err[0], fabsf(tn[0] - s[0].x));
            err[1] = fmax_(err[1], fabsf(tn[1] - s[0].y));
        }
    }
};

// A node of an ordering, and the planes of a time step: of orderings o0, o0 + 1, o0 + 2 the first
// list entry q and the count c.
struct Node {
    int i, j, k, aa, bb, cc;
    long long n;
};
struct Planes {
    int o0, q[3], c[3];
    __device__ __forceinline__ int total() const { return c[0] + c[1] + c[2]; }
};

// Threads of an SM: 80 registers a thread. Fewer threads of more registers are slower, also where
// they would not spill (the Godunov updates): 121x161x161 x 256 sources 639 / 543 / 494 / 482 ms
// with 384 / 512 / 640 / 768.
constexpr int kPlaneThreads = 768;

template <typename F, int SCHEME, int NS>
__global__ void __launch_bounds__(kPlaneThreads, 1)
    plane_kernel(FwdArgs<F> a, PlaneShape m) {
    extern __shared__ int s_off[];             // plane offsets of the schedule
    __shared__ int s_units, s_start[8];
    const GridC &g = a.g;
    const long long B = a.B;
    const int grp = blockIdx.x / m.grp_blocks, blk = blockIdx.x - grp * m.grp_blocks;
    const int src0 = grp * m.grp_src;                              // within the launch's sources
    const int Bg = min(a.src_n, src0 + m.grp_src) - src0;
    if (Bg <= 0) return;
    barrier_begin();
    for (int q = threadIdx.x; q <= a.n_planes; q += blockDim.x) s_off[q] = a.off[q];
    unsigned *s_fix = reinterpret_cast<unsigned *>(s_off + a.n_planes + 1);   // the sources' fixed sets, packed
    if (SCHEME != 3)
        for (int q = threadIdx.x; q < Bg; q += blockDim.x) {
            const SrcC &sc = a.src[a.src_lo + src0 + q];
            s_fix[q] = (unsigned)sc.ci << 20 | (unsigned)sc.cj << 10 | (unsigned)sc.ck;
        }
    if (threadIdx.x == 0)
#pragma unroll
        for (int o = 0; o < 8; ++o) s_start[o] = m.start[o];
    __syncthreads();
    int *s_list = reinterpret_cast<int *>(s_fix + Bg);                        // active threads' sources
    unsigned char *s_on = reinterpret_cast<unsigned char *>(s_list + Bg);     // the source still iterates
    for (int q = threadIdx.x; q < Bg; q += blockDim.x) s_on[q] = 1;
    __syncthreads();
    // consecutive warps of the list on different blocks: a small plane spreads over the SMs
    const long long tid = ((long long)(threadIdx.x >> 5) * m.grp_blocks + blk) * 32 + (threadIdx.x & 31);
    BarrierState *bar = a.bar + grp;
    const unsigned nblk = (unsigned)m.grp_blocks;
    const long long osp = B, ost = (long long)g.np * B, osr = (long long)g.nt * g.np * B;
    using U = Update<F, SCHEME, NS>;

    for (int it = 0; it < a.max_iter; ++it) {
        // The sources that still iterate (NS to a thread), so that no thread is kept for converged
        // ones: a solve's last iterations have few sources, in any order of the batch.
        if (threadIdx.x < 32) {
            int n = 0;
            for (int u0 = 0; u0 < Bg / NS; u0 += 32) {
                const int u = u0 + (int)threadIdx.x;
                bool on = false;
#pragma unroll
                for (int h = 0; h < NS; ++h) on = on || (u < Bg / NS && s_on[u * NS + h]);
                const unsigned mask = __ballot_sync(0xffffffffu, on);
                if (on) s_list[n + __popc(mask & ((1u << threadIdx.x) - 1u))] = u;
                n += __popc(mask);
            }
            if (threadIdx.x == 0) s_units = n;
        }
        __syncthreads();
        const int lanes = s_units;                                     // threads of one node
        if (lanes == 0) break;
        const int slots = (int)(((long long)m.grp_blocks * blockDim.x) / lanes);
        const bool any = tid < (long long)slots * lanes;
        const int slot = any ? (int)(tid / lanes) : 0;
        const int bl = src0 + (any ? s_list[tid - (long long)slot * lanes] * NS : 0);
        const int b = a.src_lo + bl;                                   // the thread's first source
        const Vec4<F> *t0c = a.t0c + bl;
        bool act[NS];
#pragma unroll
        for (int h = 0; h < NS; ++h) act[h] = any && s_on[bl - src0 + h];
        F err[NS];
#pragma unroll
        for (int h = 0; h < NS; ++h) err[h] = 0;
        // Time step tau updates the nodes of one plane of each ordering in progress (o0 .. o0 + 2 at
        // most), concatenated; this thread takes the nodes slot, slot + slots, ... The list is
        // static: the next entry is looked up while a node is updated, the next time step's first
        // one before the barrier.
        Planes cp, np;
        auto planes = [&](Planes &d, int tau, int o0) {
            if (tau - s_start[o0] >= a.n_planes && o0 < 7) ++o0;
            d.o0 = o0;
#pragma unroll
            for (int u = 0; u < 3; ++u) {
                const int o = o0 + u, L = tau - s_start[o & 7];
                d.q[u] = 0;
                d.c[u] = 0;
                if (o < 8 && tau < m.steps && L >= 0 && L < a.n_planes) {
                    d.q[u] = s_off[L];
                    d.c[u] = s_off[L + 1] - d.q[u];
                }
            }
        };
        auto entry = [&](const Planes &d, int x, int &o) {
            const int u = x < d.c[0] ? 0 : x < d.c[0] + d.c[1] ? 1 : 2;
            o = d.o0 + u;
            const int q = u == 0 ? d.q[0] + x : u == 1 ? d.q[1] + (x - d.c[0]) : d.q[2] + (x - d.c[0] - d.c[1]);
            return __ldg(a.nodes + q);
        };
        auto place = [&](int o, unsigned pk) {
            Node d;
            d.aa = (int)(pk >> 20) & 1023;
            d.bb = (int)(pk >> 10) & 1023;
            d.cc = (int)pk & 1023;
            d.i = o & 4 ? g.nr - 2 - d.aa : 1 + d.aa;
            d.j = o & 2 ? g.nt - 2 - d.bb : 1 + d.bb;
            d.k = o & 1 ? g.np - 2 - d.cc : 1 + d.cc;
            d.n = ((long long)d.i * g.nt + d.j) * g.np + d.k;
            return d;
        };
        planes(cp, 0, 0);
        int o = 0;
        unsigned pk = 0;
        if (any && slot < cp.total()) {
            pk = entry(cp, slot, o);
        }
        // the stencil, factors and record of the node in hand, and where it is
        F v[7][NS];
        typename U::Fac fc;
        NodeRec<F> rec;
        Node d;
        F *p = nullptr;
        auto load = [&]() {
            d = place(o, pk);
            p = a.tau + (d.n * B + b);
            ld_pack(p, v[0]);
            ld_pack(p + osr, v[1]);
            ld_pack(p - osr, v[2]);
            ld_pack(p + ost, v[3]);
            ld_pack(p - ost, v[4]);
            ld_pack(p + osp, v[5]);
            ld_pack(p - osp, v[6]);
            fc = U::load(t0c + d.n * a.src_n);
            rec = ld_rec(a.rec + d.n);
        };
        for (int tau = 0; tau < m.steps; ++tau) {
            const int total = cp.total();
            const bool mine = any && slot < total;
            if (mine) load();
            // the next time step's planes and this thread's first node there: static, and looked
            // up while the loads above are on their way
            planes(np, tau + 1, cp.o0);
            int on = 0;
            unsigned pkn = 0;
            if (any && slot < np.total()) pkn = entry(np, slot, on);
            if (mine)
                for (int x = slot;;) {
                    const bool rr = o & 4, rt = o & 2, rp = o & 1;
                    const bool face = pk & 0x40000000u;
                    x += slots;
                    if (x < total) pk = entry(cp, x, o);
                    F tn[NS];
                    U::run(fc, v, rec, a.er, act, tn, err);
                    // values that keep their bits are not stored: their line stays clean
                    bool moved = false;
#pragma unroll
                    for (int h = 0; h < NS; ++h) moved = moved || bits_of(tn[h]) != bits_of(v[0][h]);
                    if (moved) st_pack(p, tn);
                    // a layer next to a face (second in the ordering: the entry face, last: the
                    // exit face) along some axis
                    if (SCHEME != 3 && face) {
#pragma unroll
                        for (int h = 0; h < NS; ++h) {
                            if (!act[h]) continue;
                            const unsigned fx = s_fix[bl + h - src0];
                            const int ci = (int)(fx >> 20), cj = (int)(fx >> 10) & 1023, ck = (int)fx & 1023;
                            auto put = [&](long long e, F x1, F x2, int fi, int fj, int fk) {
                                if (!in_fixed_set(ci, cj, ck, fi, fj, fk)) p[e + h] = fmax_((F)2 * x1 - x2, x2);
                            };
                            const F ua = rr ? v[1][h] : v[2][h], ub = rt ? v[3][h] : v[4][h], uc = rp ? v[5][h] : v[6][h];
                            const long long da = rr ? osr : -osr, db = rt ? ost : -ost, dc = rp ? osp : -osp;
                            if (d.aa == 1) put(2 * da, ua, tn[h], rr ? g.nr - 1 : 0, d.j, d.k);
                            if (d.aa == a.na - 1) put(-da, tn[h], ua, rr ? 0 : g.nr - 1, d.j, d.k);
                            if (d.bb == 1) put(2 * db, ub, tn[h], d.i, rt ? g.nt - 1 : 0, d.k);
                            if (d.bb == a.nb - 1) put(-db, tn[h], ub, d.i, rt ? 0 : g.nt - 1, d.k);
                            if (d.cc == 1) put(2 * dc, uc, tn[h], d.i, d.j, rp ? g.np - 1 : 0);
                            if (d.cc == a.nc - 1) put(-dc, tn[h], uc, d.i, d.j, rp ? 0 : g.np - 1);
                        }
                    }
                    if (x >= total) break;
                    load();
                }
            if (!grid_barrier(bar, a.spin_ns, nblk)) return;
            o = on;
            pk = pkn;
            cp = np;
        }
        // 1: the source has not converged (three words a source, by iteration)
        int *flag = m.moved + (it % 3) * a.src_n;
#pragma unroll
        for (int h = 0; h < NS; ++h)
            if (act[h] && !(err[h] < a.tol)) flag[bl + h] = 1;
        if (!grid_barrier(bar, a.spin_ns, nblk)) return;
        // every block takes the sources that have converged off its list; the group's first one
        // reports, and clears the flags of the iteration after the next
        for (int q = threadIdx.x; q < Bg; q += blockDim.x) {
            const int s = src0 + q;
            const bool moved = ((volatile int *)flag)[s] != 0;
            if (blk == 0) {
                if (s_on[q]) {
                    a.iters[a.src_lo + s] = it + 1;
                    if (!moved) a.conv[a.src_lo + s] = 1;
                }
                m.moved[((it + 2) % 3) * a.src_n + s] = 0;
            }
            s_on[q] = moved;
        }
        __syncthreads();
    }
    barrier_end(bar, nblk);
}

template <typename F, int NS> const void *plane_ptr(int scheme) {
    switch (scheme) {
    case 0: return (const void *)plane_kernel<F, 0, NS>;
    case 1: return (const void *)plane_kernel<F, 1, NS>;
    case 2: return (const void *)plane_kernel<F, 2, NS>;
    default: return (const void *)plane_kernel<F, 3, NS>;
    }
}

// The factor cache of pairs: (1/T0, u) of sources 2 q and 2 q + 1 interleaved (Fac2), the values
// of t0_cache_kernel.
__global__ void t0_pair_kernel(FwdArgs<float> a) {
    const GridC &g = a.g;
    const int pairs = a.src_n / 2;
    const long long total = g.N * pairs;
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < total;
         x += (long long)gridDim.x * blockDim.x) {
        const long long n = x / pairs;
        const int b = a.src_lo + 2 * (int)(x - n * pairs);
        const int k = (int)(n % g.np);
        const long long t = n / g.np;
        const int j = (int)(t % g.nt), i = (int)(t / g.nt);
        Vec4<float> c[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const SrcReg<float> S = load_src<float>(a.src, b + h, g.dr);
            c[h].x = factor_T0<float>(S, i, __ldg(a.rad + i), __ldg(a.cost + j), __ldg(a.sint + j),
                                      a.tabT[(long long)j * a.B + b + h], a.tabP[(long long)k * a.B + b + h],
                                      g.flat != 0, c[h].y, c[h].z, c[h].w);
            if (in_fixed_set(S.ci, S.cj, S.ck, i, j, k)) c[h].x = -1.f;
        }
        float4 *o = reinterpret_cast<float4 *>(a.t0c) + 2 * x;
        o[0] = make_float4(c[0].x, c[1].x, c[0].y, c[1].y);
        o[1] = make_float4(c[0].z, c[1].z, c[0].w, c[1].w);
    }
}

// Edges of the grid: nodes on two or three faces, which no interior update reads. Along theta
// on the r faces first, then along phi, the order in which the faces are extrapolated.
template <typename F> __global__ void edge_kernel(FwdArgs<F> a, int axis) {
    const GridC &g = a.g;
    const long long B = a.B;
    const long long n = axis == 1 ? 4LL * g.np : 4LL * (g.nr + g.nt - 2);
    const long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n * a.src_n) return;
    const int b = a.src_lo + (int)(x % a.src_n);
    int q = (int)(x / a.src_n), i, j, k;
    const int hi = q & 1;
    q >>= 1;
    if (axis == 1) {
        i = q & 1 ? g.nr - 1 : 0;
        k = q >> 1;
        j = hi ? g.nt - 1 : 0;
    } else {
        k = hi ? g.np - 1 : 0;
        if (q < 2 * g.nt) {
            i = q & 1 ? g.nr - 1 : 0;
            j = q >> 1;
        } else {
            q -= 2 * g.nt;
            j = q & 1 ? g.nt - 1 : 0;
            i = 1 + (q >> 1);
        }
    }
    const SrcC &sc = a.src[b];
    if (in_fixed_set(sc.ci, sc.cj, sc.ck, i, j, k)) return;
    const long long s = (axis == 1 ? (long long)g.np : 1LL) * B * (hi ? -1 : 1);
    F *p = a.tau + node_index(g, i, j, k) * B + b;
    const F t1 = p[s], t2 = p[2 * s];
    *p = fmax_((F)2 * t1 - t2, t2);
}

}  // namespace

// Start times of the 8 orderings of an iteration: o + 1 flips the axes of the bits that change.
// At most three orderings are in progress at a time.
static void plane_starts(PlaneShape &m, int na, int nb, int nc) {
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

template <typename F>
cudaError_t run_plane_forward(FwdArgs<F> a, int groups, int *moved, int n_sm, int launch_blocks, int *grid,
                              int *block, int *kernels, cudaStream_t st) {
    cudaError_t e;
    const int n = a.src_n;
    const bool tele = a.scheme == 3;
    int threads = kPlaneThreads;
    PlaneShape m;
    memset(&m, 0, sizeof m);
    plane_starts(m, a.na, a.nb, a.nc);
    // Pairs of sources (FP32, every row whole aligned pairs) where a time step has more updates
    // than the GPU holds threads: half the instructions and loads an update. Below that a thread
    // per source has the shorter time step. LF, ms per 2 iterations, single / pairs: 81^3 x 16
    // sources 6.81 / 6.97, x 32 8.32 / 7.86, x 100 14.2 / 12.1; 121x161x161 x 32 26.6 / 23.0.
    const double per_step = 8.0 * a.na * a.nb * a.nc / m.steps * n;
    const bool pair = sizeof(F) == 4 && n % 2 == 0 && a.B % 2 == 0 && a.src_lo % 2 == 0 &&
                      (size_t)a.tau % 8 == 0 && per_step > (double)threads * n_sm;
    const int ns = pair ? 2 : 1;
    const void *fn = plane_ptr<F, 1>(a.scheme);
    if constexpr (sizeof(F) == 4)
        if (pair) fn = plane_ptr<F, 2>(a.scheme);
    const size_t smem = sizeof(int) * (a.n_planes + 1 + 2 * (size_t)n) + n;
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
        return e;
    // one block an SM and group, so that a barrier has as few arrivals as there are SMs (a barrier
    // of 608 blocks takes 2.5 us, of 152 1.6 us); groups only where asked for
    if (groups <= 0) groups = 1;
    if (groups > kMaxBarrierGroups) groups = kMaxBarrierGroups;
    if (groups > (n + 31) / 32) groups = (n + 31) / 32;
    threads = threads / groups / 32 * 32;
    // no more threads than the widest plane has nodes and sources
    const int ext[3] = {a.na, a.nb, a.nc};
    long long widest = 0;
    for (int x = 0; x < 3; ++x)
        for (int y = x + 1; y < 3; ++y) widest = std::max(widest, (long long)ext[x] * ext[y]);
    const long long want = (widest * (n / ns) / groups / n_sm + 31) / 32 * 32;
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
    const int need = (m.grp_src / ns + threads - 1) / threads;
    if (m.grp_blocks < need) m.grp_blocks = need;
    if ((long long)m.grp_blocks * groups > (long long)per_sm * n_sm) return cudaErrorInvalidConfiguration;
    *grid = m.grp_blocks * groups;
    *block = threads;
    *kernels = tele ? 1 : 4;
    m.moved = moved;
    if ((e = cudaMemsetAsync(moved, 0, sizeof(int) * 3 * (size_t)n, st)) != cudaSuccess) return e;
    if (!tele) {
        if constexpr (sizeof(F) == 4)
            if (pair) {
                const long long q = (a.g.N * (n / 2) + 255) / 256;
                t0_pair_kernel<<<(unsigned)std::min(q, 152LL * 16), 256, 0, st>>>(a);
            }
        if (!pair && (e = launch_t0_cache<F>(a, st)) != cudaSuccess) return e;
    }
    void *args[] = {&a, &m};
    if ((e = cudaLaunchCooperativeKernel(fn, dim3(*grid), dim3(threads), args, smem, st)) != cudaSuccess) return e;
    if (!tele)
        for (int axis = 1; axis <= 2; ++axis) {
            const long long q = (axis == 1 ? 4LL * a.g.np : 4LL * (a.g.nr + a.g.nt - 2)) * n;
            edge_kernel<F><<<(unsigned)((q + 255) / 256), 256, 0, st>>>(a, axis);
        }
    return cudaGetLastError();
}

template cudaError_t run_plane_forward<float>(FwdArgs<float>, int, int *, int, int, int *, int *, int *, cudaStream_t);
template cudaError_t run_plane_forward<double>(FwdArgs<double>, int, int *, int, int, int *, int *, int *, cudaStream_t);

}  // namespace ttgb

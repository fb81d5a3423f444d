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
//  - In large FP32 batches a thread holds two sources and updates them in packed arithmetic: two
//    neighbours by one load per stencil point where rows are whole aligned pairs (Deal).
//
// Each update reads what it reads in the lexicographic order, so the bits are the same.
//  - Threads are dealt to the sources that still iterate, anew every iteration.
// Measured, ms of a solve, with a barrier per plane and 456 or 608 blocks / now (one GB300):
// 41^3 x 1 source FP64 352 / 55; 121x161x161 x 1 (Godunov) 107 / 42-47; 67x83x95 x 37 378 / 214;
// 81^3 x 64 353 / 231; 101x141x151 x 112 1377 / 1197; 121x161x161 x 256, in the order of the last
// counts, Godunov 483 / 400, Lax-Friedrichs 2643 / 2540-2560;
// 81x101x101 x 24 events 430 / 189. Of a time step's 4 us at 81^3 x 64 the barrier and the schedule
// take 2.2; at 101x141x151 x 112 it is 7.5 us, four rounds of loads and updates of 1.3 us each.
// Measured and not kept: loading the next node's factors ahead (also across the barrier), an L2
// prefetch of them, a warp of its own for the barrier, four sources a thread: all slower.
#include <cuda_runtime.h>

#include "tt_plane.cuh"
#include "tt_update.cuh"

namespace ttgb {

namespace {

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

// A node of an ordering.
struct Node {
    int i, j, k, aa, bb, cc;
    long long n;
};

template <typename F, int SCHEME, int NS, int DEAL>
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
    using D = Dealt<NS, DEAL>;
    // Factors of a node: the launch's sources, one more for a pair where they are odd. Held for the
    // Godunov updates (spills of pairs 106 -> 50 B; 121x161x161 x 256 sources, 3 iterations 252 -> 248 ms),
    // read from the arguments in LF (41^3 x 64, 6 iterations 8.58 -> 8.40).
    constexpr bool kHeld = DEAL != kPairs || SCHEME == 1 || SCHEME == 2;
    const int fac_row = D::units(a.src_n) * NS;
    const PlaneSched sch{s_off, s_start, a.nodes, a.n_planes, m.steps};

    for (int it = 0; it < a.max_iter; ++it) {
        // The sources that still iterate (NS to a thread), so that no thread is kept for converged
        // ones: a solve's last iterations have few sources, in any order of the batch.
        if (threadIdx.x < 32) {
            const int n = plane_units<NS, DEAL>(s_on, Bg, s_list);
            if (threadIdx.x == 0) s_units = n;
        }
        __syncthreads();
        const int lanes = s_units;                                     // threads of one node
        if (lanes == 0) break;
        const int slots = (int)(((long long)m.grp_blocks * blockDim.x) / lanes);
        const bool any = tid < (long long)slots * lanes;
        const int slot = any ? (int)(tid / lanes) : 0;
        const int unit = any ? s_list[tid - (long long)slot * lanes] : 0;
        // the thread's first source and the second's distance from it
        const int bl = src0 + D::first(unit), off = D::step(unit, Bg);
        const int b = a.src_lo + bl;
        const Vec4<F> *t0c;
        if constexpr (kHeld && NS == 2) t0c = a.t0c + (src0 + unit * NS);
        else if constexpr (kHeld && sizeof(F) == 4) t0c = a.t0c + src0 + unit;   // fewer registers: 48.8 -> 47.2 ms x 1
        else t0c = a.t0c + bl;
        bool act[NS];
#pragma unroll
        for (int h = 0; h < NS; ++h) act[h] = any && (h == 0 || off > 0) && s_on[bl - src0 + h * off];
        F err[NS];
#pragma unroll
        for (int h = 0; h < NS; ++h) err[h] = 0;
        // Time step tau updates the nodes of one plane of each ordering in progress (o0 .. o0 + 2 at
        // most), concatenated; this thread takes the nodes slot, slot + slots, ... The list is
        // static: the next entry is looked up while a node is updated, the next time step's first
        // one before the barrier.
        Planes cp;
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
        sch.planes(cp, 0, 0);
        int o = 0;
        unsigned pk = 0;
        if (any && slot < cp.total()) {
            pk = sch.entry(cp, slot, o);
        }
        // the stencil, factors and record of the node in hand, and where it is
        F v[7][NS];
        typename U::Fac fc;
        NodeRec<F> rec;
        F *p = nullptr;
        auto load = [&]() {
            const Node d = place(o, pk);
            p = a.tau + (d.n * B + b);
            ld_src<DEAL>(p, off, v[0]);
            ld_src<DEAL>(p + osr, off, v[1]);
            ld_src<DEAL>(p - osr, off, v[2]);
            ld_src<DEAL>(p + ost, off, v[3]);
            ld_src<DEAL>(p - ost, off, v[4]);
            ld_src<DEAL>(p + osp, off, v[5]);
            ld_src<DEAL>(p - osp, off, v[6]);
            if constexpr (kHeld) fc = U::load(t0c + d.n * fac_row);
            else fc = U::load(t0c + d.n * a.src_n);
            rec = ld_rec(a.rec + d.n);
        };
        for (int tau = 0; tau < m.steps; ++tau) {
            const int total = cp.total();
            const bool mine = any && slot < total;
            if (mine) load();
            // the next time step's planes and this thread's first node there: static, and looked
            // up while the loads above are on their way
            int on = 0;
            unsigned pkn = 0;
            Planes np;
            sch.planes(np, tau + 1, cp.o0);
            if (any && slot < np.total()) pkn = sch.entry(np, slot, on);
            if (mine)
                for (int x = slot;;) {
                    const int ox = o;
                    // A face finds the node's place again: its indices held over the update cost spills
                    // (Godunov pairs 182 -> 134 B; 121x161x161 x 256 sources, whole step 755 -> 740 ms).
                    const unsigned pkx = pk;
                    x += slots;
                    if (x < total) pk = sch.entry(cp, x, o);
                    F tn[NS];
                    U::run(fc, v, rec, a.er, act, tn, err);
                    st_moved<DEAL>(p, off, tn, v[0]);
                    // a layer next to a face (second in the ordering: the entry face, last: the
                    // exit face) along some axis
                    if (SCHEME != 3 && (pkx & 0x40000000u)) {
                        const Node d = place(ox, pkx);
                        const bool rr = ox & 4, rt = ox & 2, rp = ox & 1;
#pragma unroll
                        for (int h = 0; h < NS; ++h) {
                            if (!act[h]) continue;
                            const unsigned fx = s_fix[bl + h * off - src0];
                            const int ci = (int)(fx >> 20), cj = (int)(fx >> 10) & 1023, ck = (int)fx & 1023;
                            auto put = [&](long long e, F x1, F x2, int fi, int fj, int fk) {
                                if (!in_fixed_set(ci, cj, ck, fi, fj, fk)) p[e + h * off] = fmax_((F)2 * x1 - x2, x2);
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
            // again: held over the updates they cost spills (LF pairs 100 -> 12 B; 121x161x161 x 256
            // sources 2793 -> 2644 ms, Godunov 436 -> 423)
            // One FP32 source a thread has the registers, and its short steps no time for the lookup.
            if constexpr (NS == 1 && sizeof(F) == 4) cp = np;
            else sch.planes(cp, tau + 1, cp.o0);
            if (!grid_barrier(bar, a.spin_ns, nblk)) return;
            o = on;
            pk = pkn;
        }
        // 1: the source has not converged (three words a source, by iteration)
        int *flag = m.moved + (it % 3) * a.src_n;
#pragma unroll
        for (int h = 0; h < NS; ++h)
            if (act[h] && !(err[h] < a.tol)) flag[bl + h * off] = 1;
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

template <typename F, int NS, int DEAL> const void *plane_ptr(int scheme) {
    switch (scheme) {
    case 0: return (const void *)plane_kernel<F, 0, NS, DEAL>;
    case 1: return (const void *)plane_kernel<F, 1, NS, DEAL>;
    case 2: return (const void *)plane_kernel<F, 2, NS, DEAL>;
    default: return (const void *)plane_kernel<F, 3, NS, DEAL>;
    }
}

// The factor cache of two sources a thread: (1/T0, u) of a unit's sources interleaved (Fac2), the
// values of t0_cache_kernel; for a unit of one source twice that one's.
template <int DEAL> __global__ void t0_pair_kernel(FwdArgs<float> a, int grp_src) {
    using D = Dealt<2, DEAL>;
    const GridC &g = a.g;
    const int units = D::units(a.src_n);
    const long long total = g.N * units;
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < total;
         x += (long long)gridDim.x * blockDim.x) {
        const long long n = x / units;
        const int u = (int)(x - n * units), src0 = 2 * u / grp_src * grp_src;   // grp_src is even
        const int Bg = min(a.src_n, src0 + grp_src) - src0, ug = u - src0 / 2;
        const int k = (int)(n % g.np);
        const long long t = n / g.np;
        const int j = (int)(t % g.nt), i = (int)(t / g.nt);
        Vec4<float> c[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int b = a.src_lo + src0 + D::first(ug) + h * D::step(ug, Bg);
            const SrcReg<float> S = load_src<float>(a.src, b, g.dr);
            c[h].x = factor_T0<float>(S, i, __ldg(a.rad + i), __ldg(a.cost + j), __ldg(a.sint + j),
                                      a.tabT[(long long)j * a.B + b], a.tabP[(long long)k * a.B + b],
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

// Threads of the adjoint: FP32 fits 64 registers without spills, and 32 warps an SM hide more of its
// 14 loads an update than 24: 121x161x161 x 256 sources 319 -> 284 ms. (The forward kernels spill at
// 64: 2644 -> 2694 ms, Godunov 423 -> 445.)
template <typename F> constexpr int kAdjThreads = sizeof(F) == 4 ? 1024 : kPlaneThreads;

// The adjoint sweep (Eq. 5) from the face coefficients (adj_coef_kernel, face_update), over every
// node, in the same organisation; no faces to complete. emax: [3][2][src_n], by iteration mod 3 the
// sources' largest |change| of P and, in the last ordering, largest |P|.
template <typename F, int NS, int DEAL>
__global__ void __launch_bounds__(kAdjThreads<F>, 1) adj_plane_kernel(AdjArgs<F> a, PlaneShape m, F *emax) {
    extern __shared__ __align__(8) int s_off[];
    __shared__ int s_units, s_start[8];
    const GridC &g = a.g;
    const long long B = a.B;
    const int grp = blockIdx.x / m.grp_blocks, blk = blockIdx.x - grp * m.grp_blocks;
    const int src0 = grp * m.grp_src;                              // within the launch's sources
    const int Bg = min(a.src_n, src0 + m.grp_src) - src0;
    if (Bg <= 0) return;
    barrier_begin();
    F *s_err = reinterpret_cast<F *>(s_off + (a.n_planes + 2) / 2 * 2), *s_pm = s_err + Bg;
    int *s_list = reinterpret_cast<int *>(s_pm + Bg);
    unsigned char *s_on = reinterpret_cast<unsigned char *>(s_list + Bg);
    for (int q = threadIdx.x; q <= a.n_planes; q += blockDim.x) s_off[q] = a.off[q];
    for (int q = threadIdx.x; q < Bg; q += blockDim.x) s_on[q] = 1;
    if (threadIdx.x == 0)
#pragma unroll
        for (int o = 0; o < 8; ++o) s_start[o] = m.start[o];
    __syncthreads();
    const long long tid = ((long long)(threadIdx.x >> 5) * m.grp_blocks + blk) * 32 + (threadIdx.x & 31);
    BarrierState *bar = a.bar + grp;
    const unsigned nblk = (unsigned)m.grp_blocks;
    using D = Dealt<NS, DEAL>;
    const long long sp = B, st = (long long)g.np * B, sr = (long long)g.nt * g.np * B;
    const long long plane = g.N * B;                               // coefficient plane stride
    const PlaneSched sch{s_off, s_start, a.nodes, a.n_planes, m.steps};

    for (int it = 0; it < a.max_iter; ++it) {
        if (threadIdx.x < 32) {
            const int n = plane_units<NS, DEAL>(s_on, Bg, s_list);
            if (threadIdx.x == 0) s_units = n;
        }
        for (int q = threadIdx.x; q < Bg; q += blockDim.x) s_err[q] = s_pm[q] = 0;
        __syncthreads();
        const int lanes = s_units;
        if (lanes == 0) break;
        const int slots = (int)(((long long)m.grp_blocks * blockDim.x) / lanes);
        const bool any = tid < (long long)slots * lanes;
        const int slot = any ? (int)(tid / lanes) : 0;
        const int unit = any ? s_list[tid - (long long)slot * lanes] : 0;
        const int bl = src0 + D::first(unit), off = D::step(unit, Bg);
        const int b = a.src_lo + bl;
        const F *cX = a.coef, *cY = a.coef + plane, *cZ = a.coef + 2 * plane, *cW = a.coef + 3 * plane;
        bool act[NS];
        F err[NS], pmax[NS];
#pragma unroll
        for (int h = 0; h < NS; ++h) {
            act[h] = any && (h == 0 || off > 0) && s_on[bl - src0 + h * off];
            err[h] = pmax[h] = 0;
        }
        Planes cp, np;
        sch.planes(cp, 0, 0);
        int o = 0;
        unsigned pk = 0;
        if (any && slot < cp.total()) pk = sch.entry(cp, slot, o);
        F w[NS], cx[NS], cy[NS], cz[NS], mx[NS], my[NS], mz[NS], Pn[6][NS], po[NS];
        long long x = 0;
        bool last = false;
        auto load = [&]() {
            const int aa = (int)(pk >> 20) & 1023, bb = (int)(pk >> 10) & 1023, cc = (int)pk & 1023;
            const int i = o & 4 ? g.nr - 1 - aa : aa, j = o & 2 ? g.nt - 1 - bb : bb, k = o & 1 ? g.np - 1 - cc : cc;
            x = node_index(g, i, j, k) * B + b;
            last = o == 7;
            ld_src<DEAL>(cW + x, off, w);
            ld_src<DEAL>(cX + x, off, cx);
            ld_src<DEAL>(cY + x, off, cy);
            ld_src<DEAL>(cZ + x, off, cz);
            ld_src<DEAL>(a.P + x, off, po);
            // no flux through the outer faces: zero coefficients and values there
            const bool hr = i < g.nr - 1, lr = i > 0, ht = j < g.nt - 1, lt = j > 0, hp = k < g.np - 1, lp = k > 0;
#pragma unroll
            for (int h = 0; h < NS; ++h) {
                mx[h] = my[h] = mz[h] = 0;
#pragma unroll
                for (int q = 0; q < 6; ++q) Pn[q][h] = 0;
            }
            if (lr) ld_src<DEAL>(cX + x - sr, off, mx);
            if (lt) ld_src<DEAL>(cY + x - st, off, my);
            if (lp) ld_src<DEAL>(cZ + x - sp, off, mz);
            if (hr) ld_src<DEAL>(a.P + x + sr, off, Pn[0]);
            if (lr) ld_src<DEAL>(a.P + x - sr, off, Pn[1]);
            if (ht) ld_src<DEAL>(a.P + x + st, off, Pn[2]);
            if (lt) ld_src<DEAL>(a.P + x - st, off, Pn[3]);
            if (hp) ld_src<DEAL>(a.P + x + sp, off, Pn[4]);
            if (lp) ld_src<DEAL>(a.P + x - sp, off, Pn[5]);
        };
        for (int tau = 0; tau < m.steps; ++tau) {
            const int total = cp.total();
            const bool mine = any && slot < total;
            if (mine) load();
            sch.planes(np, tau + 1, cp.o0);
            int on = 0;
            unsigned pkn = 0;
            if (any && slot < np.total()) pkn = sch.entry(np, slot, on);
            if (mine)
                for (int q = slot;;) {
                    q += slots;
                    if (q < total) pk = sch.entry(cp, q, o);
                    F pn[NS];
#pragma unroll
                    for (int h = 0; h < NS; ++h) {
                        pn[h] = po[h];
                        // the fixed set (w is NaN) and a converged source keep their values
                        if (act[h] && w[h] == w[h]) {
                            const F nb[6] = {Pn[0][h], Pn[1][h], Pn[2][h], Pn[3][h], Pn[4][h], Pn[5][h]};
                            pn[h] = face_update<F>(cx[h], cy[h], cz[h], w[h], mx[h], my[h], mz[h], nb);
                            err[h] = fmax_(err[h], fabs(pn[h] - po[h]));
                            if (last) pmax[h] = fmax_(pmax[h], fabs(pn[h]));
                        }
                    }
                    st_moved<DEAL>(a.P + x, off, pn, po);
                    if (q >= total) break;
                    load();
                }
            if (!grid_barrier(bar, a.spin_ns, nblk)) return;
            o = on;
            pk = pkn;
            cp = np;
        }
        // the sources' maxima: over the block, then over the group's blocks
        F *e = emax + (long long)(it % 3) * 2 * a.src_n;
#pragma unroll
        for (int h = 0; h < NS; ++h)
            if (act[h]) {
                atomic_max_nonneg(&s_err[bl - src0 + h * off], err[h]);
                atomic_max_nonneg(&s_pm[bl - src0 + h * off], pmax[h]);
            }
        __syncthreads();
        for (int q = threadIdx.x; q < Bg; q += blockDim.x)
            if (s_on[q]) {
                atomic_max_nonneg(e + src0 + q, s_err[q]);
                atomic_max_nonneg(e + a.src_n + src0 + q, s_pm[q]);
            }
        if (!grid_barrier(bar, a.spin_ns, nblk)) return;
        // every block evaluates the stopping rule; the group's first one reports, and clears the
        // maxima of the iteration after the next
        F *e2 = emax + (long long)((it + 2) % 3) * 2 * a.src_n;
        for (int q = threadIdx.x; q < Bg; q += blockDim.x) {
            const int s = src0 + q;
            const bool done = ((volatile F *)e)[s] <= a.tol * ((volatile F *)e)[a.src_n + s];
            if (blk == 0) {
                if (s_on[q]) {
                    a.iters[a.src_lo + s] = it + 1;
                    if (done) a.conv[a.src_lo + s] = 1;
                }
                e2[s] = e2[a.src_n + s] = 0;
            }
            if (done) s_on[q] = 0;
        }
        __syncthreads();
    }
    barrier_end(bar, nblk);
}

}  // namespace

template <typename F>
cudaError_t run_plane_forward(FwdArgs<F> a, int groups, int *moved, int n_sm, int launch_blocks,
                              PlaneLaunch *launch, cudaStream_t st) {
    cudaError_t e;
    const int n = a.src_n;
    const bool tele = a.scheme == 3;
    PlaneShape m;
    memset(&m, 0, sizeof m);
    plane_starts(m, a.na, a.nb, a.nc);
    const bool pair = n % 2 == 0 && a.B % 2 == 0 && a.src_lo % 2 == 0 && (size_t)a.tau % 8 == 0;
    const bool two = sizeof(F) == 4 && plane_two(m, a.na, a.nb, a.nc, n, a.scheme, pair, n_sm);
    const void *fn = plane_ptr<F, 1, kPairs>(a.scheme);
    if constexpr (sizeof(F) == 4)
        if (two) fn = pair ? plane_ptr<F, 2, kPairs>(a.scheme) : plane_ptr<F, 2, kHalves>(a.scheme);
    launch->thread_sources = two ? 2 : 1;
    const size_t smem = sizeof(int) * (a.n_planes + 1 + 2 * (size_t)n) + n;
    if ((e = plane_shape(m, fn, smem, a.na, a.nb, a.nc, n, two ? 2 : 1, groups, kPlaneThreads, n_sm, launch_blocks, launch)) != cudaSuccess)
        return e;
    launch->kernels = tele ? 1 : 4;
    m.moved = moved;
    if ((e = cudaMemsetAsync(moved, 0, sizeof(int) * 3 * (size_t)n, st)) != cudaSuccess) return e;
    if (!tele) {
        if constexpr (sizeof(F) == 4)
            if (two) {
                const unsigned q = (unsigned)std::min((a.g.N * ((n + 1) / 2) + 255) / 256, 152LL * 16);
                if (pair) t0_pair_kernel<kPairs><<<q, 256, 0, st>>>(a, m.grp_src);
                else t0_pair_kernel<kHalves><<<q, 256, 0, st>>>(a, m.grp_src);
            }
        if (!two && (e = launch_t0_cache<F>(a, st)) != cudaSuccess) return e;
    }
    void *args[] = {&a, &m};
    if ((e = cudaLaunchCooperativeKernel(fn, dim3(launch->grid), dim3(launch->block), args, smem, st)) != cudaSuccess) return e;
    if (!tele)
        for (int axis = 1; axis <= 2; ++axis) {
            const long long q = (axis == 1 ? 4LL * a.g.np : 4LL * (a.g.nr + a.g.nt - 2)) * n;
            edge_kernel<F><<<(unsigned)((q + 255) / 256), 256, 0, st>>>(a, axis);
        }
    return cudaGetLastError();
}

template <typename F>
cudaError_t run_plane_adjoint(AdjArgs<F> a, int groups, F *emax, int n_sm, int launch_blocks,
                              PlaneLaunch *launch, cudaStream_t st) {
    cudaError_t e;
    const int n = a.src_n;
    PlaneShape m;
    memset(&m, 0, sizeof m);
    plane_starts(m, a.g.nr, a.g.nt, a.g.np);
    const bool pair = n % 2 == 0 && a.B % 2 == 0 && a.src_lo % 2 == 0 && (size_t)a.P % 8 == 0;
    const bool two = sizeof(F) == 4 && plane_two(m, a.g.nr, a.g.nt, a.g.np, n, kAdjointSolver, pair, n_sm);
    const void *fn = (const void *)adj_plane_kernel<F, 1, kPairs>;
    if constexpr (sizeof(F) == 4)
        if (two) fn = pair ? (const void *)adj_plane_kernel<F, 2, kPairs> : (const void *)adj_plane_kernel<F, 2, kApart>;
    launch->thread_sources = two ? 2 : 1;
    launch->kernels = 1;
    const size_t smem = sizeof(int) * (a.n_planes + 2 + (size_t)n) + 2 * sizeof(F) * (size_t)n + n;
    if ((e = plane_shape(m, fn, smem, a.g.nr, a.g.nt, a.g.np, n, two ? 2 : 1, groups, kAdjThreads<F>, n_sm, launch_blocks, launch)) != cudaSuccess)
        return e;
    if ((e = cudaMemsetAsync(emax, 0, sizeof(F) * 6 * (size_t)n, st)) != cudaSuccess) return e;
    void *args[] = {&a, &m, &emax};
    return cudaLaunchCooperativeKernel(fn, dim3(launch->grid), dim3(launch->block), args, smem, st);
}

template cudaError_t run_plane_adjoint<float>(AdjArgs<float>, int, float *, int, int, PlaneLaunch *, cudaStream_t);
template cudaError_t run_plane_adjoint<double>(AdjArgs<double>, int, double *, int, int, PlaneLaunch *, cudaStream_t);
template cudaError_t run_plane_forward<float>(FwdArgs<float>, int, int *, int, int, PlaneLaunch *, cudaStream_t);
template cudaError_t run_plane_forward<double>(FwdArgs<double>, int, int *, int, int, PlaneLaunch *, cudaStream_t);

}  // namespace ttgb

// The updates of one (node, source) of the sweeps, shared by their schedules.
#pragma once

#include "tt_common.cuh"

namespace ttgb {

template <typename F> __device__ __forceinline__ F fmax_(F a, F b) { return a > b ? a : b; }

__device__ __forceinline__ unsigned bits_of(float x) { return __float_as_uint(x); }
__device__ __forceinline__ unsigned long long bits_of(double x) {
    return (unsigned long long)__double_as_longlong(x);
}

__device__ __forceinline__ void atomic_max_nonneg(float *p, float v) {
    atomicMax(reinterpret_cast<unsigned int *>(p), __float_as_uint(v));
}
__device__ __forceinline__ void atomic_max_nonneg(double *p, double v) {
    atomicMax(reinterpret_cast<unsigned long long *>(p),
              (unsigned long long)__double_as_longlong(v));
}

// Upwind update of one (node, source) from its face coefficients (Eq. 5 discretised as in
// adj_update): c = (+r, +theta, +phi face coefficients, J S), cm = the -r, -theta, -phi
// neighbours' plus-face coefficients, Pn = P at (+r, -r, +theta, -theta, +phi, -phi).
// Rounding-explicit, so both lanes' copies give identical bits.
template <typename F>
__device__ __forceinline__ F face_update(F cx, F cy, F cz, F cw, F cmx, F cmy, F cmz,
                                         const F (&Pn)[6]) {
    const F zero = (F)0;
    const F out = add_(add_(sub_(fmax_(cx, zero), fmin(cmx, zero)),
                            sub_(fmax_(cy, zero), fmin(cmy, zero))),
                       sub_(fmax_(cz, zero), fmin(cmz, zero)));
    const F in = fma_(fmax_(cmx, zero), Pn[1],
                 fma_(-fmin(cx, zero), Pn[0],
                 fma_(fmax_(cmy, zero), Pn[3],
                 fma_(-fmin(cy, zero), Pn[2],
                 fma_(fmax_(cmz, zero), Pn[5], mul_(-fmin(cz, zero), Pn[4]))))));
    return out <= (F)1e-30 ? zero : div_(add_(cw, in), out);
}

// New tau from v = tau at (centre, r+, r-, theta+, theta-, phi+, phi-), the cached factors c
// and the node record R. SCHEME: 0 and 3 Lax-Friedrichs, 1 Godunov, 2 anisotropic Godunov.
template <typename F, int SCHEME>
__device__ __forceinline__ F sweep_update(const F *v, const Vec4<F> &c, const NodeRec<F> &R, F er) {
    return SCHEME == 2   ? godunov_aniso_core<F>(c.x, c.y, c.z, c.w, v[0], v[1], v[2], v[3], v[4], v[5], v[6], R, er)
           : SCHEME == 1 ? godunov_core<F>(c.x, c.y, c.z, c.w, v[0], v[1], v[2], v[3], v[4], v[5], v[6], R, er)
                         : lf_core<F>(c.x, c.y, c.z, c.w, v[0], v[1], v[2], v[3], v[4], v[5], v[6], R, er);
}

// Two sources at once in packed FP32 (one instruction, two IEEE operations of the same bits as
// the scalar ones): lf_core for a pair. a - b is formed as b * (-1) + a, which rounds once.
__device__ __forceinline__ float2 fma2_(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2_(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2_(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2_(float2 a, float2 b) {
    return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
__device__ __forceinline__ float2 both_(float a) { return make_float2(a, a); }

// The factors of a pair of sources: (1/T0, u_r, u_t, u_p), each for both.
struct alignas(16) Fac2 {
    float2 x, y, z, w;
};

__device__ __forceinline__ float2 lf_core2(const Fac2 &c, float2 tc, float2 trp, float2 trm, float2 ttp,
                                           float2 ttm, float2 tpp, float2 tpm, const NodeRec<float> &R,
                                           float er) {
    const float2 er2 = both_(er), et = both_(R.et), ep = both_(R.ep);
    const float2 vr = fma2_(tc, c.y, mul2_(sub2_(trp, trm), er2));
    const float2 vt = fma2_(tc, c.z, mul2_(sub2_(ttp, ttm), et));
    const float2 vp = fma2_(tc, c.w, mul2_(sub2_(tpp, tpm), ep));
    const float2 kt = both_(fma_(-2.f, R.xi, 1.f)), kp = both_(fma_(2.f, R.xi, 1.f));
    const float2 e4 = both_(mul_(4.f, R.eta));
    const float2 q = fma2_(vr, vr, fma2_(mul2_(kt, vt), vt,
                                         fma2_(mul2_(kp, vp), vp, mul2_(mul2_(e4, vt), vp))));
    const float2 H = make_float2(-sqrt_(q.x), -sqrt_(q.y));
    const float2 sr = add2_(sub2_(trp, tc), sub2_(trm, tc));
    const float2 st = add2_(sub2_(ttp, tc), sub2_(ttm, tc));
    const float2 sp = add2_(sub2_(tpp, tc), sub2_(tpm, tc));
    const float2 num = fma2_(er2, sr, fma2_(both_(R.ct), st, fma2_(both_(R.cp), sp, fma2_(both_(R.s), c.x, H))));
    return fma2_(num, both_(R.invW), tc);
}

// sweep_update for a pair of sources; v as there.
template <int SCHEME>
__device__ __forceinline__ float2 sweep_update2(const float2 *v, const Fac2 &c, const NodeRec<float> &R, float er) {
    if constexpr (SCHEME == 0 || SCHEME == 3) {
        return lf_core2(c, v[0], v[1], v[2], v[3], v[4], v[5], v[6], R, er);
    } else {
    float a[7], b[7];
#pragma unroll
    for (int q = 0; q < 7; ++q) {
        a[q] = v[q].x;
        b[q] = v[q].y;
    }
    const float ra = sweep_update<float, SCHEME>(a, Vec4<float>{c.x.x, c.y.x, c.z.x, c.w.x}, R, er);
    const float rb = sweep_update<float, SCHEME>(b, Vec4<float>{c.x.y, c.y.y, c.z.y, c.w.y}, R, er);
    return make_float2(ra, rb);
    }
}

}  // namespace ttgb

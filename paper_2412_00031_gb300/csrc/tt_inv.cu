// The common-receiver differential-time misfit and its adjoint source (Eqs. 4, A4), and the
// regularisation and model update of the inversion step (Sec. 3.3 and step 4 of Sec. 2):
// kernel density (Eq. 19) and the normalisation of the kernels by it (Eq. 18); the
// multiple-grid projection of a kernel onto H offset inversion grids (Eqs. 11-14, 17) and the
// expansion of coefficients back onto the forward grid (Eq. 15); the model update.
//
// Inversion grids: grid h (0 <= h < H) has N nodes per axis at x_a = x_min + (a - h / H) dc,
// dc = (x_max - x_min) / (N - 2), so that every grid covers the forward domain. Along one axis
// the hat function of node a (Eqs. 12-14) is max(0, 1 - |x - x_a| / dc) inside the grid; a
// forward node therefore sees at most two hats per axis and grid. The host tabulates, per
// axis and grid, each forward node's lower coarse node and the two weights; the device
// contracts one axis at a time (projection) or sums the 2 x 2 x 2 products per grid
// (expansion). Every sum runs in a fixed order, so the results do not depend on the launch.
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "tt_inv.h"

namespace ttgb {

namespace {

inline unsigned nblocks(long long n, int t) { return (unsigned)((n + t - 1) / t); }

// Eq. 19 for one batch: Kd[n] += sum over b < B of P[n][b]. One warp per node: lane l adds
// b = l, l + 32, ... in order, then a fixed butterfly.
template <typename F>
__global__ void sum_sources_kernel(long long N, int B, const F *__restrict__ P, double *Kd) {
    const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= N) return;
    double acc = 0.0;
    for (int b = lane; b < B; b += 32) acc += (double)P[w * B + b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) Kd[w] += acc;
}

// Eqs. 4 and A4. Block b = source b; thread t takes receivers m = t, t + blockDim, ...: for
// the entries of (b, m) (the pairs {b, j} at receiver m, each with dT_obs = T_b^obs - T_j^obs
// and the pair weight w), e = (T_b - T_j) - dT_obs; R[b][m] += gamma sum w e, and the source's
// share of chi_cr is sum w e^2 / 4 (an unordered pair is two ordered terms of weight w / 2,
// split between its two sources). An entry whose other source is out of range sets *bad.
__global__ void misfit_cr_kernel(int n_src, int n_rec, const int *__restrict__ off,
                                 const int *__restrict__ other, const double *__restrict__ dtobs,
                                 const double *__restrict__ w, double gamma,
                                 const double *__restrict__ Tr, double *chi, double *R, int *bad) {
    __shared__ double s[256];
    const int b = blockIdx.x;
    double part = 0.0;
    for (int m = threadIdx.x; m < n_rec; m += blockDim.x) {
        const long long nm = (long long)b * n_rec + m;
        const int q0 = off[nm], q1 = off[nm + 1];
        if (q1 <= q0) continue;
        const double tb = Tr[nm];
        double acc = 0.0;
        for (int q = q0; q < q1; ++q) {
            const int j = other[q];
            if (j < 0 || j >= n_src) {
                atomicExch(bad, 1);
                continue;
            }
            const double e = (tb - Tr[(long long)j * n_rec + m]) - dtobs[q];
            acc += w[q] * e;
            part += 0.25 * w[q] * e * e;
        }
        R[nm] += gamma * acc;
    }
    s[threadIdx.x] = part;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) s[threadIdx.x] += s[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) chi[b] = s[0];
}

// x^-zeta (x a density plus the damping), for the loop's zeta = 1/2 by rsqrt: pow takes about six
// times its FP64 instructions and bounded the normalisation (0.76 -> 0.09 ms at 101x201x201). Other
// exponents: REL by pow(x, -zeta), which rounds once and holds where x^zeta over- or underflows;
// the absolute form by 1 / pow(x, zeta). (The power of -inf is inf, of which rsqrt knows nothing;
// an integer comparison, as the FP64 pipe is the busy one: 0.103 ms with a FP64 one.)
template <bool REL> __device__ __forceinline__ double damp_factor(double x, double zeta) {
    if (zeta == 0.5) return __double2hiint(x) == (int)0xfff00000 && __double2loint(x) == 0 ? 0.0 : rsqrt(x);
    return REL ? pow(x, -zeta) : 1.0 / pow(x, zeta);
}

// Eq. 18 in place on the three kernels.
__global__ void normalize_kernel(long long N, double *Ks, double *Kxi, double *Keta,
                                 const double *Kd, double eps, double zeta) {
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const double f = damp_factor<false>(Kd[n] + eps, zeta);
    Ks[n] *= f;
    Kxi[n] *= f;
    Keta[n] *= f;
}

// Projection, contraction over phi: T1[h][i][j][c] = sum_k K dV W_p[h][c][k], with
// dV = h2(i)^2 cos(theta_j) dr dtheta dphi. A warp takes a row, a lane the outputs (h, c) of
// which it sums only the nodes under the hat, [rng[2 (h, c)], rng[2 (h, c) + 1]): the other
// weights are zero (a dense sum over the row, 9 / 2 times the FP64 work, took 0.4 ms per kernel
// at 101x201x201 and 5 grids of 11^3). Up to 16 outputs get P lanes each, a power of two, that
// take every P-th node of the hat: with one lane each most of the warp is idle while a few sum
// long hats (whole projection at 101x201x201, one grid: 3^3 0.314 ms, the dense sum 0.114, now
// 0.120; 5^3 0.245 / 0.120 / 0.130; 8^3 0.169 / 0.150 / 0.105). A row with a value that is not
// finite takes the dense sum: there the value reaches every output, infinite under its hats and
// NaN (times a zero weight) elsewhere.
constexpr int kProjRows = 4;   // rows (warps) of a block
template <int P> __global__ void __launch_bounds__(32 * kProjRows)
    project_phi_kernel(MgDims d, const double *__restrict__ K, const double *__restrict__ h2,
                       const double *__restrict__ cost, double dvol, const double *__restrict__ Wp,
                       const int *__restrict__ rng, double *T1) {
    extern __shared__ double s_row[];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long r = (long long)blockIdx.x * kProjRows + w;
    if (r >= (long long)d.nr * d.nt) return;
    const int i = (int)(r / d.nt), j = (int)(r % d.nt);
    double *row = s_row + (long long)w * d.np;
    bool odd = false;   // the FP64 pipe is the busy one: the test is an integer one
    for (int k = lane; k < d.np; k += 32) {
        const double v = K[r * d.np + k];
        row[k] = v;
        odd = odd || (__double2hiint(v) & 0x7ff00000) == 0x7ff00000;
    }
    const bool dense = __any_sync(0xffffffffu, odd);
    __syncwarp();
    const double dV = h2[i] * h2[i] * cost[j] * dvol;
    for (int q0 = 0; q0 < d.H * d.cp; q0 += 32 / P) {
        const int q = q0 + lane / P;
        const bool on = q < d.H * d.cp;
        double acc = 0.0;
        if (on) {
            const double *wt = Wp + (long long)q * d.np;
            int k0 = rng[2 * q], k1 = rng[2 * q + 1];
            if (dense) k0 = 0, k1 = d.np;
            int m = (k1 - k0 - lane % P + P - 1) / P;
            const double *x = row + k0 + lane % P, *y = wt + k0 + lane % P;
            for (; m >= 8; m -= 8, x += 8 * P, y += 8 * P) {   // eight loads of weights in flight
                double v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = __ldg(y + u * P);
#pragma unroll
                for (int u = 0; u < 8; ++u) acc += x[u * P] * v[u];
            }
#pragma unroll 1   // hats of two or three nodes: 200 coarse nodes along phi, 5 grids 0.76 -> 0.59 ms
            for (int u = 0; u < m; ++u) acc += x[u * P] * y[u * P];
        }
        for (int o = P / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (on && lane % P == 0) {
            const int h = q / d.cp, c = q - h * d.cp;
            T1[(((long long)h * d.nr + i) * d.nt + j) * d.cp + c] = acc * dV;
        }
    }
}

// Contraction over theta: T2[h][i][b][c] = sum_j T1[h][i][j][c] W_t[h][b][j].
__global__ void project_theta_kernel(MgDims d, const double *__restrict__ T1,
                                     const double *__restrict__ Wt, double *T2) {
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long total = (long long)d.H * d.nr * d.ct * d.cp;
    if (q >= total) return;
    const int c = (int)(q % d.cp);
    long long r = q / d.cp;
    const int b = (int)(r % d.ct);
    r /= d.ct;
    const int i = (int)(r % d.nr), h = (int)(r / d.nr);
    const double *src = T1 + (((long long)h * d.nr + i) * d.nt) * d.cp + c;
    const double *w = Wt + ((long long)h * d.ct + b) * d.nt;
    double acc = 0.0;
    for (int j = 0; j < d.nt; ++j) acc += src[(long long)j * d.cp] * w[j];
    T2[q] = acc;
}

// Contraction over r and the 1 / H of Eq. 11: G[h][a][b][c] = sum_i T2[h][i][b][c] W_r[h][a][i] / H.
__global__ void project_r_kernel(MgDims d, const double *__restrict__ T2,
                                 const double *__restrict__ Wr, double *G) {
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long total = (long long)d.H * d.cr * d.ct * d.cp;
    if (q >= total) return;
    const int c = (int)(q % d.cp);
    long long r = q / d.cp;
    const int b = (int)(r % d.ct);
    r /= d.ct;
    const int a = (int)(r % d.cr), h = (int)(r / d.cr);
    const double *src = T2 + ((long long)h * d.nr * d.ct + b) * d.cp + c;
    const double *w = Wr + ((long long)h * d.cr + a) * d.nr;
    double acc = 0.0;
    for (int i = 0; i < d.nr; ++i) acc += src[(long long)i * d.ct * d.cp] * w[i];
    G[q] = acc / d.H;
}

// Eq. 15 in two steps, as the hats are products of one per axis. E[h][i][j][c] = the four
// products G W_r W_t around the row (i, j), / H; then D[i][j][k] = sum over h of the two products
// E W_p around the node. With the eight products per grid formed at every node the FP64 pipe
// took 0.7 ms at 101x201x201 and 5 grids; the rows hold np / cp times fewer values than the nodes.
// DIRECT forms the eight products at the node, where the rows hold as many values as the nodes or
// would not fit.
__global__ void expand_rows_kernel(MgDims d, const double *__restrict__ G, const int *__restrict__ lo,
                                   const double *__restrict__ Wr, const double *__restrict__ Wt,
                                   double *__restrict__ E) {
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (long long)d.H * d.nr * d.nt * d.cp) return;
    const int c = (int)(q % d.cp);
    long long r = q / d.cp;
    const int j = (int)(r % d.nt);
    r /= d.nt;
    const int i = (int)(r % d.nr), h = (int)(r / d.nr);
    // lo: [H][nr] then [H][nt] then [H][np], the lower coarse node of each forward node
    const int a0 = lo[h * d.nr + i], b0 = lo[d.H * d.nr + h * d.nt + j];
    double e = 0.0;
    for (int a = a0; a < a0 + 2; ++a) {
        const double wr = Wr[((long long)h * d.cr + a) * d.nr + i];
        for (int b = b0; b < b0 + 2; ++b)
            e += wr * Wt[((long long)h * d.ct + b) * d.nt + j] * G[(((long long)h * d.cr + a) * d.ct + b) * d.cp + c];
    }
    E[q] = e / d.H;
}

template <bool DIRECT>
__global__ void expand_kernel(MgDims d, const double *__restrict__ E, const double *__restrict__ G,
                              const int *__restrict__ lo, const double *__restrict__ Wr,
                              const double *__restrict__ Wt, const double *__restrict__ Wp, double *D) {
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long N = (long long)d.nr * d.nt * d.np;
    if (n >= N) return;
    const int k = (int)(n % d.np);
    const long long ij = n / d.np;
    const int i = (int)(ij / d.nt), j = (int)(ij - (long long)i * d.nt);
    const int *lor = lo, *lot = lo + (long long)d.H * d.nr, *lop = lot + (long long)d.H * d.nt;
    double acc = 0.0;
    for (int h = 0; h < d.H; ++h) {
        const int c0 = lop[h * d.np + k];
        const double *w = Wp + ((long long)h * d.cp + c0) * d.np + k;
        const double w0 = w[0], w1 = w[d.np];
        if constexpr (DIRECT) {
            const int a0 = lor[h * d.nr + i], b0 = lot[h * d.nt + j];
            double sh = 0.0;
            for (int a = a0; a < a0 + 2; ++a) {
                const double wr = Wr[((long long)h * d.cr + a) * d.nr + i];
                for (int b = b0; b < b0 + 2; ++b) {
                    const double *g = G + (((long long)h * d.cr + a) * d.ct + b) * d.cp + c0;
                    sh += wr * Wt[((long long)h * d.ct + b) * d.nt + j] * (g[0] * w0 + g[1] * w1);
                }
            }
            acc += sh;
        } else {
            const double *e = E + ((long long)h * d.nr * d.nt + ij) * d.cp + c0;
            acc += e[0] * w0 + e[1] * w1;
        }
    }
    D[n] = DIRECT ? acc / d.H : acc;
}

// max |x| of each of three FP64 fields: per-block maxima, then one block over them.
__global__ void absmax_partial_kernel(long long N, const double *a, const double *b,
                                      const double *c, double *part) {
    __shared__ double s[3][256];
    double m[3] = {0.0, 0.0, 0.0};
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < N;
         n += (long long)gridDim.x * blockDim.x) {
        m[0] = fmax(m[0], fabs(a[n]));
        m[1] = fmax(m[1], fabs(b[n]));
        m[2] = fmax(m[2], fabs(c[n]));
    }
    for (int f = 0; f < 3; ++f) s[f][threadIdx.x] = m[f];
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int f = 0; f < 3; ++f) s[f][threadIdx.x] = fmax(s[f][threadIdx.x], s[f][threadIdx.x + w]);
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int f = 0; f < 3; ++f) part[(long long)f * gridDim.x + blockIdx.x] = s[f][0];
}

// One warp per field: mx[f] the maximum, mx[3 + f] = step / maximum (0 for a zero field), divided
// once here instead of at every node.
__global__ void absmax_final_kernel(int nb, const double *part, double *mx, double step) {
    const int f = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double m = 0.0;
    for (int q = lane; q < nb; q += 32) m = fmax(m, part[(long long)f * nb + q]);
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) {
        mx[f] = m;
        mx[3 + f] = m > 0.0 ? step / m : 0.0;
    }
}

// Eq. 18 with eps = eps_rel max(Kd) (Kd >= 0 is a sum of adjoint fields of unit sources): the
// maximum comes from absmax_final_kernel's first slot; 1e-300 when it is 0.
__global__ void normalize_rel_kernel(long long N, double *Ks, double *Kxi, double *Keta,
                                     const double *Kd, const double *mx, double eps_rel,
                                     double zeta) {
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const double e = fmax(eps_rel * mx[0], 1e-300);
    const double f = damp_factor<true>(Kd[n] + e, zeta);
    Ks[n] *= f;
    Kxi[n] *= f;
    Keta[n] *= f;
}

// Total misfit alpha sum chi[b][0] + beta sum chi[b][1] + gamma sum chi_cr[b] over n sources:
// one block, each thread sums a fixed stride of sources in order, then a fixed tree.
__global__ void misfit_total_kernel(int n, const double *chi, double alpha, double beta,
                                    const double *chi_cr, double gamma, double *out) {
    __shared__ double s[256];
    double acc = 0.0;
    for (int b = threadIdx.x; b < n; b += blockDim.x) {
        double v = alpha * chi[2 * (long long)b] + beta * chi[2 * (long long)b + 1];
        if (chi_cr) v += gamma * chi_cr[b];
        acc += v;
    }
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = s[0];
}

// The update: s <- s (1 - a D_s / max|D_s|), xi <- xi - a D_xi / max|D_xi|, eta likewise
// (a zero direction leaves its field unchanged).
template <typename F>
__global__ void update_kernel(long long N, F *s, F *xi, F *eta, const double *Ds,
                              const double *Dxi, const double *Deta, const double *mx) {
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const double fs = mx[3], fx = mx[4], fe = mx[5];
    s[n] = (F)((double)s[n] * (1.0 - fs * Ds[n]));
    xi[n] = (F)((double)xi[n] - fx * Dxi[n]);
    eta[n] = (F)((double)eta[n] - fe * Deta[n]);
}

}  // namespace

// Per-axis tables of the H grids of `c` nodes over `n` forward nodes: W[h][a][i] (the hat
// of coarse node a at forward node i, in the axis coordinate scaled to [0, 1]) and lo[h][i]
// (the coarse node below forward node i: its hats are lo and lo + 1).
void mgrid_axis_tables(int n, int c, int H, std::vector<double> &W, std::vector<int> &lo) {
    W.assign((size_t)H * c * n, 0.0);
    lo.assign((size_t)H * n, 0);
    const double dc = 1.0 / (c - 2);
    for (int h = 0; h < H; ++h)
        for (int i = 0; i < n; ++i) {
            const double x = (double)i / (n - 1);
            const double u = x / dc + (double)h / H;       // position in coarse cells from node 0
            int a = (int)std::floor(u);
            if (a > c - 2) a = c - 2;
            if (a < 0) a = 0;
            lo[(size_t)h * n + i] = a;
            for (int q = a; q <= a + 1; ++q) {
                const double xa = (q - (double)h / H) * dc;
                const double v = 1.0 - std::fabs(x - xa) / dc;
                W[((size_t)h * c + q) * n + i] = v > 0.0 ? v : 0.0;
            }
        }
}

cudaError_t run_misfit_cr(int n_src, int n_rec, const int *off, const int *other,
                          const double *dtobs, const double *w, double gamma, const double *Tr,
                          double *chi, double *R, int *bad, cudaStream_t st) {
    misfit_cr_kernel<<<n_src, 256, 0, st>>>(n_src, n_rec, off, other, dtobs, w, gamma, Tr, chi, R, bad);
    return cudaGetLastError();
}

template <typename F>
cudaError_t run_kernel_density(long long N, int B, const F *P, double *Kd, cudaStream_t st) {
    sum_sources_kernel<F><<<nblocks(N * 32, 256), 256, 0, st>>>(N, B, P, Kd);
    return cudaGetLastError();
}

cudaError_t run_kernel_normalize(long long N, double *Ks, double *Kxi, double *Keta,
                                 const double *Kd, double eps, double zeta, cudaStream_t st) {
    normalize_kernel<<<nblocks(N, 256), 256, 0, st>>>(N, Ks, Kxi, Keta, Kd, eps, zeta);
    return cudaGetLastError();
}

cudaError_t run_mgrid_project(const MgDims &d, const double *K, const double *h2,
                              const double *cost, double dvol, const double *Wr,
                              const double *Wt, const double *Wp, const int *rng, double *T1,
                              double *T2, double *G, cudaStream_t st) {
    const long long n2 = (long long)d.H * d.nr * d.ct * d.cp;
    const long long n3 = (long long)d.H * d.cr * d.ct * d.cp;
    const int n = d.H * d.cp;   // cp >= 3
    auto phi = n <= 4 ? project_phi_kernel<8> : n <= 8 ? project_phi_kernel<4>
               : n <= 16 ? project_phi_kernel<2> : project_phi_kernel<1>;
    phi<<<nblocks((long long)d.nr * d.nt, kProjRows), 32 * kProjRows, sizeof(double) * kProjRows * d.np, st>>>(
        d, K, h2, cost, dvol, Wp, rng, T1);
    project_theta_kernel<<<nblocks(n2, 256), 256, 0, st>>>(d, T1, Wt, T2);
    project_r_kernel<<<nblocks(n3, 256), 256, 0, st>>>(d, T2, Wr, G);
    return cudaGetLastError();
}

cudaError_t run_mgrid_expand(const MgDims &d, const double *G, const int *lo, const double *Wr,
                             const double *Wt, const double *Wp, double *E, double *D,
                             cudaStream_t st) {
    const unsigned nb = nblocks((long long)d.nr * d.nt * d.np, 256);
    if (!E) {
        expand_kernel<true><<<nb, 256, 0, st>>>(d, nullptr, G, lo, Wr, Wt, Wp, D);
        return cudaGetLastError();
    }
    expand_rows_kernel<<<nblocks((long long)d.H * d.nr * d.nt * d.cp, 256), 256, 0, st>>>(d, G, lo, Wr, Wt, E);
    expand_kernel<false><<<nb, 256, 0, st>>>(d, E, G, lo, Wr, Wt, Wp, D);
    return cudaGetLastError();
}

template <typename F>
cudaError_t run_model_update(long long N, F *s, F *xi, F *eta, const double *Ds,
                             const double *Dxi, const double *Deta, double step, double *part,
                             int n_part, cudaStream_t st) {
    absmax_partial_kernel<<<n_part, 256, 0, st>>>(N, Ds, Dxi, Deta, part);
    absmax_final_kernel<<<1, 96, 0, st>>>(n_part, part, part + 3 * n_part, step);
    update_kernel<F><<<nblocks(N, 256), 256, 0, st>>>(N, s, xi, eta, Ds, Dxi, Deta,
                                                      part + 3 * n_part);
    return cudaGetLastError();
}

cudaError_t run_kernel_normalize_rel(long long N, double *Ks, double *Kxi, double *Keta,
                                     const double *Kd, double eps_rel, double zeta, double *part,
                                     int n_part, cudaStream_t st) {
    // the partial maxima of Kd (the kernel takes three fields: Kd three times)
    absmax_partial_kernel<<<n_part, 256, 0, st>>>(N, Kd, Kd, Kd, part);
    absmax_final_kernel<<<1, 96, 0, st>>>(n_part, part, part + 3 * n_part, 0.0);
    normalize_rel_kernel<<<nblocks(N, 256), 256, 0, st>>>(N, Ks, Kxi, Keta, Kd,
                                                          part + 3 * n_part, eps_rel, zeta);
    return cudaGetLastError();
}

cudaError_t run_misfit_total(int n, const double *chi, double alpha, double beta,
                             const double *chi_cr, double gamma, double *out, cudaStream_t st) {
    misfit_total_kernel<<<1, 256, 0, st>>>(n, chi, alpha, beta, chi_cr, gamma, out);
    return cudaGetLastError();
}

template cudaError_t run_kernel_density<float>(long long, int, const float *, double *, cudaStream_t);
template cudaError_t run_kernel_density<double>(long long, int, const double *, double *, cudaStream_t);
template cudaError_t run_model_update<float>(long long, float *, float *, float *, const double *,
                                             const double *, const double *, double, double *,
                                             int, cudaStream_t);
template cudaError_t run_model_update<double>(long long, double *, double *, double *,
                                              const double *, const double *, const double *,
                                              double, double *, int, cudaStream_t);

}  // namespace ttgb

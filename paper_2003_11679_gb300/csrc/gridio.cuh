// Projection onto and interpolation from the AIM grid (Eqs. AIM_Lin, AIM_Kin),
// in FP64 and in the complex64 path's FP32.
//
// FP64 additions run for whole warps at 2 lanes per SM, so a warp-wide reduction of
// the 10 sums of a triangle costs more than its products: large meshes give a
// triangle 4 lanes.  The gather projection needs no reduction: a lane per result grid.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace sie {

template <int G, class R>
__device__ __forceinline__ R gio_sum(R v)
{
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

__device__ __forceinline__ double gio_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float gio_fma(float a, float b, float c) { return fmaf(a, b, c); }

// products that are not to be contracted with the sum they go into
__device__ __forceinline__ double gio_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float gio_mul(float a, float b) { return __fmul_rn(a, b); }

// the four weights (w0, w1) of a stencil entry: 16-byte loads
__device__ __forceinline__ void gio_w(const double* w, double& w0, double* w1)
{
    const double2 a = __ldg(reinterpret_cast<const double2*>(w)), b = __ldg(reinterpret_cast<const double2*>(w) + 1);
    w0 = a.x, w1[0] = a.y, w1[1] = b.x, w1[2] = b.y;
}
__device__ __forceinline__ void gio_w(const float* w, float& w0, float* w1)
{
    const float4 a = __ldg(reinterpret_cast<const float4*>(w));
    w0 = a.x, w1[0] = a.y, w1[1] = a.z, w1[2] = a.w;
}

// y[e] += c_{t,i} [S1 + (c_t - p_i) . T0 + scal 2 P0] of every triangle t and slot i:
// S1 = sum_u w1 . A(u), T0 = sum_u w0 A(u), P0 = sum_u w0 Phi(u) over its stencil.
// Right-hand side blockIdx.y: grids out + y NG Ng, vector y + y ldy.  NG: 4 grids
// (A, Phi) or 3 (A).  FP32 grids (C = float2): FP32 gathers and sums, FP64 from the
// edge coefficients on.  G lanes per triangle: 4, or all 32 up to 2,048 triangles and
// right-hand sides together, where one gather latency counts and not the additions: with
// 32 and 4 lanes 9.1 and 14.9 us at 320, 13.7 and 15.4 at 1,280, 16.4 and 16.6 at 2,000,
// 20.4 and 15.4 at 2,560.  L2 gathers and FP64 additions bound it beyond: 20,480 triangles
// take 105 us (eight right-hand sides 785 us) with 32 lanes, 34 us (157 us) with 4.
// With 32 lanes CTAs have 64 threads: a small mesh then spreads over more SMs' FP64 lanes.
constexpr int64_t GIO_WIDE = 2048;
constexpr int GIO_SMALL = 64;
template <int G, class C, class R, int NG>
__global__ void __launch_bounds__(256) k_interp(int nt, int S, int Mord, DevMesh M, const int32_t* __restrict__ base,
                                                const R* __restrict__ W, const C* __restrict__ out, GridDesc g,
                                                double2 scal, int64_t Ng, double2* __restrict__ y, int64_t ldy)
{
    const int t0 = (blockIdx.x * blockDim.x + threadIdx.x) / G, l = threadIdx.x % G;
    const int t = min(t0, nt - 1);  // the last warps' spare groups repeat the last triangle and do not store
    out += (int64_t)blockIdx.y * NG * Ng;
    y += (int64_t)blockIdx.y * ldy;
    const int Mp = Mord + 1;
    const int64_t corner = ((int64_t)base[3 * t + 2] * g.N[1] + base[3 * t + 1]) * g.N[0] + base[3 * t];
    R s1r = 0, s1i = 0, tr[3] = {0, 0, 0}, ti[3] = {0, 0, 0}, pr = 0, pi = 0;
    for (int u = l; u < S; u += G) {
        const int ux = u % Mp, uy = (u / Mp) % Mp, uz = u / (Mp * Mp);
        const int64_t node = corner + ((int64_t)uz * g.N[1] + uy) * g.N[0] + ux;
        R w0, w1[3];
        gio_w(W + ((size_t)t * S + u) * 4, w0, w1);
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const C A = out[a * Ng + node];
            s1r += w1[a] * A.x;
            s1i += w1[a] * A.y;
            tr[a] += w0 * A.x;
            ti[a] += w0 * A.y;
        }
        if (NG == 4) {
            const C P = out[3 * Ng + node];
            pr += w0 * P.x;
            pi += w0 * P.y;
        }
    }
    s1r = gio_sum<G>(s1r);
    s1i = gio_sum<G>(s1i);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        tr[a] = gio_sum<G>(tr[a]);
        ti[a] = gio_sum<G>(ti[a]);
    }
    if (NG == 4) {
        pr = gio_sum<G>(pr);
        pi = gio_sum<G>(pi);
    }
    if (l >= 3 || t0 >= nt) return;
    const double* q = M.q + 9 * t + 3 * l;
    double vr = s1r, vi = s1i;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        vr += q[a] * (double)tr[a];
        vi += q[a] * (double)ti[a];
    }
    if (NG == 4) {
        const double p0r = pr, p0i = pi;
        vr += 2.0 * (scal.x * p0r - scal.y * p0i);
        vi += 2.0 * (scal.x * p0i + scal.y * p0r);
    }
    const double c = M.coef[3 * t + l];
    double2* d = y + M.tri_edge[3 * t + l];
    atomicAdd(&d->x, c * vr);
    atomicAdd(&d->y, c * vi);
}

template <class C>
__device__ __forceinline__ C cmk(double a, double b)
{
    C c;
    c.x = a;
    c.y = b;
    return c;
}

// tc: per triangle 9 values: alpha_H, beta_H[3], alpha_E, beta_E[3], -c0rho; vector
// blockIdx.y: H, E and rho ldh, lde and ldr apart, tc 9 nt apart
template <class C>
__global__ void k_tri_coef(int nt, DevMesh M, const double2* __restrict__ H, int64_t ldh, const double2* __restrict__ E,
                           int64_t lde, const double2* __restrict__ rho, int64_t ldr, C* __restrict__ tc)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    H += blockIdx.y * ldh;
    E += blockIdx.y * lde;
    rho += blockIdx.y * ldr;
    double ar[2] = {0, 0}, ai[2] = {0, 0}, br[2][3] = {{0, 0, 0}, {0, 0, 0}}, bi[2][3] = {{0, 0, 0}, {0, 0, 0}};
    for (int i = 0; i < 3; i++) {
        const int e = M.tri_edge[3 * t + i];
        const double c = M.coef[3 * t + i];
        const double2 xs[2] = {H[e], E[e]};
        for (int f = 0; f < 2; f++) {
            ar[f] += c * xs[f].x;
            ai[f] += c * xs[f].y;
            for (int a = 0; a < 3; a++) {
                const double qq = c * M.q[9 * t + 3 * i + a];
                br[f][a] += qq * xs[f].x;
                bi[f][a] += qq * xs[f].y;
            }
        }
    }
    C* o = tc + 9 * (blockIdx.y * (int64_t)nt + t);
    for (int f = 0; f < 2; f++) {
        o[4 * f] = cmk<C>(ar[f], ai[f]);
        for (int a = 0; a < 3; a++) o[4 * f + 1 + a] = cmk<C>(br[f][a], bi[f][a]);
    }
    o[8] = cmk<C>(-rho[t].x, -rho[t].y);
}

// Projection of the system product as a gather (deterministic, no atomics): per
// triangle t the current on t is alpha (r - c_t) + beta (alpha = sum_i c_i x_i,
// beta_a = sum_i c_i q_ia x_i) for x = H and x = E', and the charge grid takes
// -c0rho_t; grid node v sums, in a fixed order, the stencil entries (t, u) that land
// on it: J_a += alpha_H w1[a] + beta_H[a] w0, M_a likewise with E', rho += -c0rho_t w0.
// tc: per triangle alpha_H, beta_H[3], alpha_E, beta_E[3], -c0rho; node, ptr: the nodes
// with entries by falling number of entries (the lists of a warp are of one length),
// ent: t * S + u; src is zero elsewhere.  A lane per (node, grid): the 8 lanes of a node
// read the same weights and triangle record, nothing is reduced across lanes, and
// four entries' loads are in flight, since the longest lists (a bar's corners) are
// one chain.  Gathers from L2 and FP64 products bound it.  20,480 triangles: 148 us with
// a thread per node in grid order, 118 us with every node in one unsorted list, 60 us
// now (FP32: 44, 50, 34 us); a bar of 336: 40 us, 19 us now.
// Vector blockIdx.y: tc 9 nt and src 7 Ng apart.  CHAIN: an entry's two products are
// chained into the sum; else added up first (block.cu; the roundings are spelled out).
template <class C, class R, bool CHAIN = true>
__global__ void __launch_bounds__(256) k_project_gather(int64_t nnode, const int32_t* __restrict__ node,
                                                        const int32_t* __restrict__ ptr,
                                                        const int32_t* __restrict__ ent, int S,
                                                        const R* __restrict__ W, const C* __restrict__ tc, int nt,
                                                        C* __restrict__ src, int64_t Ng)
{
    constexpr int U = 4;
    const int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 8;
    const int o = threadIdx.x % 8;
    if (v >= nnode || o >= 7) return;
    tc += blockIdx.y * 9 * (int64_t)nt;
    src += blockIdx.y * 7 * Ng;
    // grid o: al w1[a] + be w0; the charge: c0rho w0
    const bool rho = o == 6;
    const int f = o >= 3 ? 1 : 0, a = rho ? 0 : o - 3 * f, ia = 4 * f, ib = rho ? 8 : 4 * f + 1 + a;
    const int k0 = ptr[v], k1 = ptr[v + 1];
    R ar = 0, ai = 0;
    for (int k = k0; k < k1; k += U) {
        int32_t id[U];
        R w0[U], w1[U];
        C al[U], be[U];
#pragma unroll
        for (int u = 0; u < U; u++) id[u] = k + u < k1 ? __ldg(ent + k + u) : -1;
#pragma unroll
        for (int u = 0; u < U; u++) {
            w0[u] = w1[u] = 0;
            al[u].x = al[u].y = be[u].x = be[u].y = 0;
            if (id[u] >= 0) {
                const R* w = W + (int64_t)id[u] * 4;
                const C* c = tc + 9 * (int64_t)(id[u] / S);
                w0[u] = __ldg(w);
                be[u] = __ldg(c + ib);
                if (!rho) {
                    w1[u] = __ldg(w + 1 + a);
                    al[u] = __ldg(c + ia);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++)
            if (id[u] >= 0) {
                if (CHAIN || rho) {
                    ar = gio_fma(al[u].x, w1[u], gio_fma(be[u].x, w0[u], ar));
                    ai = gio_fma(al[u].y, w1[u], gio_fma(be[u].y, w0[u], ai));
                } else {
                    ar += gio_fma(be[u].x, w0[u], gio_mul(al[u].x, w1[u]));
                    ai += gio_fma(be[u].y, w0[u], gio_mul(al[u].y, w1[u]));
                }
            }
    }
    C z;
    z.x = ar;
    z.y = ai;
    src[o * Ng + node[v]] = z;
}

// Projection of the L and K products by FP64 atomics into cleared grids (a gather's
// random reads lose here: 575 us against 417 us for eight right-hand sides of 20,480
// triangles): J and, with 4 grids, rho = 2 alpha w0.  A thread per (triangle, stencil
// node); alpha and beta from tc (k_tri_coef1), or from x where tc is null: few
// triangles, one launch less.  Right-hand side blockIdx.y: x + y ldx, src + y ngrid Ng.
// With tc 14 FP64 operations an entry instead of 47: 170 us.  The line is GIO_WIDE too:
// without and with tc 12.8 and 15.3 us at 1,280 triangles and right-hand sides, 15.7 and
// 14.9 at 2,304, 21.9 and 17.3 at 4,608.
template <bool TC>
__global__ void __launch_bounds__(256) k_project(int nt, int S, int Mord, DevMesh M, const int32_t* __restrict__ base,
                                                 const double* __restrict__ W, const double2* __restrict__ x,
                                                 int64_t ldx, const double2* __restrict__ tc, GridDesc g, int ngrid,
                                                 double2* __restrict__ src, int64_t Ng)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= nt * S) return;
    src += (int64_t)blockIdx.y * ngrid * Ng;
    const int t = idx / S, u = idx % S, Mp = Mord + 1;
    double2 al = make_double2(0, 0), be[3] = {al, al, al};
    if (TC) {
        const double2* c = tc + ((int64_t)blockIdx.y * nt + t) * 4;
        al = __ldg(c);
        for (int a = 0; a < 3; a++) be[a] = __ldg(c + 1 + a);
    } else {
        x += (int64_t)blockIdx.y * ldx;
        for (int i = 0; i < 3; i++) {
            const double2 xv = x[M.tri_edge[3 * t + i]];
            const double c = M.coef[3 * t + i];
            al.x += c * xv.x;
            al.y += c * xv.y;
            for (int a = 0; a < 3; a++) {
                const double qq = c * M.q[9 * t + 3 * i + a];
                be[a].x += qq * xv.x;
                be[a].y += qq * xv.y;
            }
        }
    }
    const int nx = base[3 * t] + u % Mp, ny = base[3 * t + 1] + (u / Mp) % Mp, nz = base[3 * t + 2] + u / (Mp * Mp);
    const int64_t node = ((int64_t)nz * g.N[1] + ny) * g.N[0] + nx;
    double w0, w1[3];
    gio_w(W + (size_t)idx * 4, w0, w1);
    for (int a = 0; a < 3; a++) {
        double2* d = src + a * Ng + node;
        atomicAdd(&d->x, fma(al.x, w1[a], be[a].x * w0));
        atomicAdd(&d->y, fma(al.y, w1[a], be[a].y * w0));
    }
    if (ngrid == 4) {
        double2* d = src + 3 * Ng + node;
        w0 *= 2.0;
        atomicAdd(&d->x, al.x * w0);
        atomicAdd(&d->y, al.y * w0);
    }
}

// alpha and beta[3] of every triangle t of vector x + y ldx (y = blockIdx.y) at tc + 4 (y nt + t)
inline __global__ void k_tri_coef1(int nt, DevMesh M, const double2* __restrict__ x, int64_t ldx, double2* __restrict__ tc)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    x += (int64_t)blockIdx.y * ldx;
    double2 al = make_double2(0, 0), be[3] = {al, al, al};
    for (int i = 0; i < 3; i++) {
        const double2 xv = x[M.tri_edge[3 * t + i]];
        const double c = M.coef[3 * t + i];
        al.x += c * xv.x;
        al.y += c * xv.y;
        for (int a = 0; a < 3; a++) {
            const double qq = c * M.q[9 * t + 3 * i + a];
            be[a].x += qq * xv.x;
            be[a].y += qq * xv.y;
        }
    }
    double2* o = tc + ((int64_t)blockIdx.y * nt + t) * 4;
    o[0] = al;
    for (int a = 0; a < 3; a++) o[1 + a] = be[a];
}

// CTAs of T threads for n items of G lanes
inline unsigned gio_blocks(int64_t n, int G, int T = 256) { return (unsigned)((n * G + T - 1) / T); }

}  // namespace sie

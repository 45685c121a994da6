// Near-region matrices of the AIM (Eqs. LinNRP, KinNRP): direct FP64
// integration of every near triangle pair minus the grid's own contribution
// for that pair (the precorrection L_P, K_P of Eqs. AIM_Lin, AIM_Kin), then
// assembly into edge CSR rows.
//
// Direct integration rule (the paper only says "direct integration"; this is
// the library's reading, documented with the parameters in sie.h):
//   far-near pairs  : collapsed Gauss product rule on both triangles;
//   close pairs     : outer collapsed Gauss on the test triangle, inner polar
//                     integration about the projection of the observation
//                     point (three signed sub-triangles, angular variable
//                     asinh(t/h), closed-form radial parts for 1/R and the
//                     static gradient, series or graded Gauss for the rest);
//   touching pairs  : outer rule graded toward the shared edge / vertex
//                     (self pair: three centroid sub-triangles graded toward
//                     the edges).
#include <cmath>
#include <complex>
#include <cstdio>

#include "internal.h"

namespace sie {

__constant__ QuadDev cq;
// per near pair: [0..8] LA exact-grid, [9..17] K exact-grid, [18] Lphi exact-grid,
// [19..27] LA exact, [28] Lphi exact
#define NLOC 29
#define RCUT 36.0  // exp(-36) < 1e-15

// ------------------------------------------------------------------ complex helpers
struct cd {
    double re, im;
};
__device__ __forceinline__ cd mk(double a, double b) { return {a, b}; }
__device__ __forceinline__ cd operator+(cd a, cd b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ cd operator-(cd a, cd b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ cd operator*(cd a, cd b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ cd operator*(double s, cd a) { return {s * a.re, s * a.im}; }
__device__ __forceinline__ cd operator*(cd a, double s) { return {s * a.re, s * a.im}; }
__device__ __forceinline__ cd cdivc(cd a, cd b)
{
    double d = b.re * b.re + b.im * b.im;
    return {(a.re * b.re + a.im * b.im) / d, (a.im * b.re - a.re * b.im) / d};
}
__device__ __forceinline__ cd cexpc(cd z)
{
    double e = exp(z.re), s, c;
    sincos(z.im, &s, &c);
    return {e * c, e * s};
}
// exp(-j k R), R real (a real k needs no exponential)
__device__ __forceinline__ cd cexp_mjkr(cd k, double R)
{
    double s, c;
    sincos(-k.re * R, &s, &c);
    if (k.im == 0.0) return {c, s};
    double e = exp(k.im * R);
    return {e * c, e * s};
}
__device__ __forceinline__ double cnorm(cd z) { return z.re * z.re + z.im * z.im; }

// (exp(z) - 1)/z
__device__ cd phi1(cd z)
{
    if (cnorm(z) < 0.25) {
        cd term = mk(1, 0), s = mk(1, 0);
        for (int n = 2; n < 17; n++) {  // 0.5^16 / 17! < 1e-19
            term = (term * z) * cq.rn[n];
            s = s + term;
        }
        return s;
    }
    return cdivc(cexpc(z) - mk(1, 0), z);
}

// (1 + z) exp(-z) - 1 with a series near 0; e = exp(-z)
__device__ cd hfun(cd z, cd e)
{
    if (cnorm(z) < 0.04) {
        // sum_{n >= 2} (-1)^(n+1) (n - 1) z^n / n!
        cd s = mk(0, 0), zn = z;
        for (int n = 2; n < 15; n++) {
            zn = (zn * z) * (-cq.rn[n]);
            s = s + (double)(n - 1) * zn;
        }
        return s;
    }
    return (mk(1, 0) + z) * e - mk(1, 0);
}

struct v3 {
    double x, y, z;
};
__device__ __forceinline__ v3 ld3(const double* p) { return {p[0], p[1], p[2]}; }
__device__ __forceinline__ v3 operator-(v3 a, v3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ v3 operator+(v3 a, v3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ v3 operator*(double s, v3 a) { return {s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ double dot(v3 a, v3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ v3 cross(v3 a, v3 b) { return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x}; }
__device__ __forceinline__ double nrm(v3 a) { return sqrt(dot(a, a)); }

struct Inner {
    cd Is;
    cd Iv[3];
    cd Ig[3];
};

// Ein(z) = I_0^z (1 - exp(-t))/t dt for Re z >= 0; e = exp(-z).  Series for
// |z| < 2, else E1(z) + log z + gamma.  E1 = e / (z + 1 - 1 / (z + 3 - 4 /
// (z + 5 - ...))) by the forward recurrence of numerator and denominator with
// a term count from its convergence rate exp(-4 sqrt(n |z|) cos(arg z / 2)):
// no division per term (n <= 104, terms below 1e180).  Beyond Re z = 40
// E1 is below the rounding of log z.
__device__ cd ein(cd z, cd e)
{
    const double r2 = cnorm(z);
    if (r2 < 4.0) {
        cd s = mk(0, 0), t = mk(1, 0);
        for (int n = 1; n < 60; n++) {
            t = (t * z) * cq.rn[n];
            cd term = ((n & 1) ? cq.rn[n] : -cq.rn[n]) * t;
            s = s + term;
            if (cnorm(term) < 1e-34 * cnorm(s)) break;
        }
        return s;
    }
    const double euler = 0.57721566490153286061;
    cd o = mk(0.5 * log(r2) + euler, atan2(z.im, z.re));
    if (z.re > 40.0) return o;
    const int n = (int)(200.0 / (sqrt(r2) + z.re)) + 5;
    cd A0 = mk(0, 0), A1 = mk(1, 0), B0 = mk(1, 0), B1 = mk(z.re + 1.0, z.im);
    for (int i = 1; i <= n; i++) {
        const cd b = mk(z.re + (double)(2 * i + 1), z.im);
        const double a = -(double)(i * i);
        cd A2 = b * A1 + a * A0, B2 = b * B1 + a * B0;
        A0 = A1;
        A1 = A2;
        B0 = B1;
        B1 = B2;
    }
    return o + e * cdivc(A1, B1);
}

// Graded Gauss radial integrals of the lossy kernel over [0, rc] at height d
// (|k| Rmax > 1): a1 = I rho^2/R exp(-jkR), a2 = I rho^2/R^3 [(1 + jkR) exp(-jkR) - 1]
__device__ void radial_numeric(cd k, double rc, double d, cd* a1o, cd* a2o)
{
    cd a1 = mk(0, 0), a2 = mk(0, 0);
    double hi = rc;
    for (int p = 0; p < cq.npan && rc > 0.0; p++) {
        double lo = (p == cq.npan - 1) ? 0.0 : hi * cq.ratio;
        for (int qq = 0; qq < cq.n[QR_RAD]; qq++) {
            double rho = lo + (hi - lo) * cq.x[QR_RAD][qq];
            double wr = (hi - lo) * cq.w[QR_RAD][qq];
            double R2 = rho * rho + d * d, iR = rsqrt(R2), R = R2 * iR;
            cd z = mk(-k.im * R, k.re * R);  // j k R
            cd e = cexpc(mk(-z.re, -z.im));
            double f = wr * rho * rho * iR;
            a1 = a1 + f * e;
            a2 = a2 + (f * iR * iR) * hfun(z, e);
        }
        hi = lo;
    }
    *a1o = a1;
    *a2o = a2;
}

__device__ void inner_gauss(v3 r, v3 a, v3 b, v3 c, cd k, Inner& o)
{
    v3 e1 = b - a, e2 = c - a;
    double twoA = nrm(cross(e1, e2));
    o.Is = mk(0, 0);
    for (int d = 0; d < 3; d++) o.Iv[d] = o.Ig[d] = mk(0, 0);
    const int n = cq.n[QR_FAR];
    const double f = 1.0 / (4.0 * M_PI);
    for (int i = 0; i < n; i++) {
        double u = cq.x[QR_FAR][i];
        for (int j = 0; j < n; j++) {
            double v = cq.x[QR_FAR][j] * (1.0 - u);
            double w = twoA * (1.0 - u) * cq.w[QR_FAR][i] * cq.w[QR_FAR][j];
            v3 p = a + u * e1 + v * e2;
            v3 dv = p - r;
            double R2 = dot(dv, dv), iR = rsqrt(R2), R = R2 * iR;
            cd e = cexp_mjkr(k, R);
            cd G = (f * iR) * e;
            cd g = (-f * iR * iR * iR) * (mk(1.0 - k.im * R, k.re * R) * e);
            o.Is = o.Is + w * G;
            double dvv[3] = {dv.x, dv.y, dv.z};
            for (int d = 0; d < 3; d++) {
                o.Iv[d] = o.Iv[d] + (w * dvv[d]) * G;
                o.Ig[d] = o.Ig[d] + (-w * dvv[d]) * g;
            }
        }
    }
}

// ------------------------------------------------------------------ outer rules
// point and weight of outer node q of a graded rule (apex shared: toward 0;
// edge b-c shared: toward 1 in lam and graded toward both ends in mu)
__device__ void graded_point(v3 apex, v3 b, v3 c, int toward_edge, int q, v3& p, double& w)
{
    const int olam = cq.n[QR_OLAM];
    const int nmu = toward_edge ? 2 * cq.emupan * cq.n[QR_EMU] : cq.n[QR_OMU];
    int pan = q / (olam * nmu), rr = q % (olam * nmu), i = rr / nmu, j = rr % nmu;
    double hi = 1.0;
    for (int t = 0; t < pan; t++) hi *= cq.oratio;
    double lo = (pan == cq.opan - 1) ? 0.0 : hi * cq.oratio;
    double sg = lo + (hi - lo) * cq.x[QR_OLAM][i];
    double wsg = (hi - lo) * cq.w[QR_OLAM][i];
    double lam = toward_edge ? 1.0 - sg : sg;
    double mu, wmu;
    if (!toward_edge) {
        mu = cq.x[QR_OMU][j];
        wmu = cq.w[QR_OMU][j];
    } else {
        const int ne = cq.n[QR_EMU];
        int side = j / (cq.emupan * ne), r2 = j % (cq.emupan * ne), pp = r2 / ne, jj = r2 % ne;
        double h2 = 0.5;
        for (int t = 0; t < pp; t++) h2 *= cq.oratio;
        double l2 = (pp == cq.emupan - 1) ? 0.0 : h2 * cq.oratio;
        double s = l2 + (h2 - l2) * cq.x[QR_EMU][jj];
        mu = side ? 1.0 - s : s;
        wmu = (h2 - l2) * cq.w[QR_EMU][jj];
    }
    v3 e1 = b - apex, e2 = c - b;
    double twoA = nrm(cross(e1, e2));
    p = apex + lam * (e1 + mu * e2);
    w = twoA * lam * wsg * wmu;
}

__device__ int graded_count(int toward_edge)
{
    const int nmu = toward_edge ? 2 * cq.emupan * cq.n[QR_EMU] : cq.n[QR_OMU];
    return cq.opan * cq.n[QR_OLAM] * nmu;
}

// ------------------------------------------------------------------ pair classes
// far (0): product Gauss on both triangles.  The others are close pairs, whose
// outer rules have very different sizes: plain (1), vertex shared (2), edge
// shared (3), self (4).
enum { PC_FAR = 0, PC_PLAIN, PC_VERTEX, PC_EDGE, PC_SELF };

__global__ void k_pair_class(const int32_t* __restrict__ pairs, int64_t np, DevMesh M, double kr, double ki,
                             const double2* __restrict__ obj_k, uint8_t* __restrict__ cls)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    const int t = pairs[2 * p], s = pairs[2 * p + 1];
    if (obj_k) {
        const double2 ko = obj_k[M.obj[t]];
        kr = ko.x;
        ki = ko.y;
    }
    int nsh = 0;
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) nsh += M.T[3 * t + i] == M.T[3 * s + j];
    int c = PC_FAR;
    if (t == s)
        c = PC_SELF;
    else if (nsh == 2)
        c = PC_EDGE;
    else if (nsh == 1)
        c = PC_VERTEX;
    else {
        const double D = nrm(ld3(M.cen + 3 * t) - ld3(M.cen + 3 * s)), Rt = M.rad[t], Rs = M.rad[s];
        if (nsh > 0 || D < cq.cf * (Rt + Rs) || hypot(kr, ki) * (Rt + Rs) > cq.kres) c = PC_PLAIN;
    }
    cls[p] = (uint8_t)c;
}

// 14 moments per pair: Q0, Q1[3], Q2[3], Q3, U[3], V[3] (origin: centroid of t).
// Contribution of one outer point: weight w, rt = r - c_t, inner integrals
__device__ __forceinline__ void add_moments(cd* acc, double w, const double* rt, bool self, cd Is, const cd* Iv,
                                            const cd* Ig)
{
    cd I2[3];
    for (int d = 0; d < 3; d++) I2[d] = Iv[d] + rt[d] * Is;
    acc[0] = acc[0] + w * Is;
    for (int d = 0; d < 3; d++) {
        acc[1 + d] = acc[1 + d] + (w * rt[d]) * Is;
        acc[4 + d] = acc[4 + d] + w * I2[d];
    }
    acc[7] = acc[7] + w * (rt[0] * I2[0] + rt[1] * I2[1] + rt[2] * I2[2]);
    if (self) return;
    acc[8] = acc[8] + (-w) * (rt[1] * Ig[2] - rt[2] * Ig[1]);
    acc[9] = acc[9] + (-w) * (rt[2] * Ig[0] - rt[0] * Ig[2]);
    acc[10] = acc[10] + (-w) * (rt[0] * Ig[1] - rt[1] * Ig[0]);
    for (int d = 0; d < 3; d++) acc[11 + d] = acc[11 + d] + w * Ig[d];
}

__device__ __forceinline__ void store_moments(cd* acc, int lane, double2* __restrict__ mom)
{
    for (int i = 0; i < 14; i++)
        for (int off = 16; off > 0; off >>= 1) {
            acc[i].re += __shfl_down_sync(0xffffffffu, acc[i].re, off);
            acc[i].im += __shfl_down_sync(0xffffffffu, acc[i].im, off);
        }
    if (lane == 0)
        for (int i = 0; i < 14; i++) mom[i] = make_double2(acc[i].re, acc[i].im);
}

}  // namespace sie
#include "near_points.cuh"
namespace sie {

// far pairs: one warp per pair, a lane per outer point
__global__ void __launch_bounds__(128) k_near_far(const int32_t* __restrict__ pairs, int64_t np,
                                                  const uint8_t* __restrict__ cls, DevMesh M, double kr, double ki,
                                                  double2* __restrict__ mom)
{
    const int64_t p = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    const int lane = threadIdx.x & 31;
    if (p >= np || cls[p] != PC_FAR) return;
    const int t = pairs[2 * p], s = pairs[2 * p + 1];
    const v3 a = ld3(M.V + 3 * M.T[3 * t]), b = ld3(M.V + 3 * M.T[3 * t + 1]), c = ld3(M.V + 3 * M.T[3 * t + 2]);
    const v3 a2 = ld3(M.V + 3 * M.T[3 * s]), b2 = ld3(M.V + 3 * M.T[3 * s + 1]), c2 = ld3(M.V + 3 * M.T[3 * s + 2]);
    const v3 ct = ld3(M.cen + 3 * t);
    const double twoA = nrm(cross(b - a, c - a));
    const int n = cq.n[QR_FAR];
    cd acc[14];
    for (int i = 0; i < 14; i++) acc[i] = mk(0, 0);
    for (int qo = lane; qo < n * n; qo += 32) {
        const int i = qo / n, j = qo % n;
        const double u = cq.x[QR_FAR][i], v = cq.x[QR_FAR][j] * (1.0 - u);
        const v3 r = a + u * (b - a) + v * (c - a);
        Inner in;
        inner_gauss(r, a2, b2, c2, mk(kr, ki), in);
        const v3 rt = r - ct;
        const double rtv[3] = {rt.x, rt.y, rt.z};
        add_moments(acc, twoA * (1.0 - u) * cq.w[QR_FAR][i] * cq.w[QR_FAR][j], rtv, false, in.Is, in.Iv, in.Ig);
    }
    store_moments(acc, lane, mom + 14 * p);
}

// ------------------------------------------------------------------ close pairs
// One warp per unit = (pair, run of 32 or more outer points), a lane per outer
// point.  FP64 arithmetic bounds it (2 FP64 lanes per SM), so the work is
// arranged to keep all lanes on it and to spend few operations per direction:
//  * a point near an edge has over ten angular panels, one at the centre three:
//    the panels of the 32 points are listed, panel index by panel index, and
//    the lanes take panels, whosever they are (the moments are linear in them);
//    exp(s) is a product of the panel's start and tabulated steps;
//  * |k| Rmax <= 1: every radial integral of a direction comes from the powers of
//    R and the moments A_n = I rho^2 R^(n-1) drho, A_n = (rho R^(n+1) - t)/(n+2)
//    with t = d^2 I R^(n-1), summed against the Taylor coefficients of
//    exp(-jkR), as many orders as the largest |k| R of the 32 panels needs for 1e-18
//    (4 to 8 of the graded panels next to an edge);
//  * units of self and edge pairs come first, so no long unit ends the launch.
// One warp per pair with the outer points split over lanes, 27 orders with a
// division each and separate cosh, tanh, phi1 per direction took 364 ms for the
// exterior near region of an 80-triangle sphere at 3 GHz; 28 ms now, 37 million
// directions at 286 FP64 operations, the FP64 pipe 87% busy.
constexpr int NC_W = 2;     // warps per CTA (42 KB of shared memory)
constexpr int NC_NT = 24;   // largest order: 1 / 24! < 2e-24
constexpr int NC_NA = 8;    // angular nodes with tabulated exp(+-ds x_q); more are evaluated
constexpr int NC_LIST = 96; // (edge, panel index) entries listed at a time

struct CloseSm {
    double et[3][3], em[3][3], va[3][3], len[3];          // source triangle: edges, in-plane normals
    double dd[32], lad[32], iad[32], w[32], rt[3][32];      // per outer point
    double2 is0[32], ead[32], a1[32], a2[32];
    double rc[32];
    double h[3][32], sa[3][32], ds[3][32];                  // per edge and point
    double ep[NC_NA][3][32], en[NC_NA][3][32];              // exp(+-ds x_q)
    double2 u[NC_NT + 4], g[NC_NT + 2], b[NC_NT + 2];      // u_m = (-j k/|k|)^m / m!, -m u_(m+1), u_(m-1) / m
    unsigned mask[NC_LIST];                                 // points of a list entry
    int pre[NC_LIST + 1];                                   // items before it
    int2 ent[NC_LIST];                                      // (edge, panel index)
    unsigned char ser[32];
};

template <bool REALK>
__global__ void __launch_bounds__(32 * NC_W, 4) k_near_close(const int2* __restrict__ unit, int nunit, int npts,
                                                          const int32_t* __restrict__ pairs,
                                                          const uint8_t* __restrict__ cls, DevMesh M, double kr,
                                                          double ki, double2* __restrict__ part)
{
    __shared__ CloseSm sm_[NC_W];
    const int un = blockIdx.x * NC_W + threadIdx.x / 32;
    const int lane = threadIdx.x & 31;
    if (un >= nunit) return;
    CloseSm& S = sm_[threadIdx.x / 32];
    const int p = unit[un].x, q_lo = unit[un].y;
    const int t = pairs[2 * (int64_t)p], s = pairs[2 * (int64_t)p + 1], kind = cls[p];
    const cd k = mk(kr, REALK ? 0.0 : ki);
    const double kabs = REALK ? kr : sqrt(kr * kr + ki * ki);
    const cd mjk = mk(k.im, -k.re);  // -j k
    const int tt[3] = {M.T[3 * t], M.T[3 * t + 1], M.T[3 * t + 2]};
    const v3 a = ld3(M.V + 3 * tt[0]), b = ld3(M.V + 3 * tt[1]), c = ld3(M.V + 3 * tt[2]);
    const v3 ct = ld3(M.cen + 3 * t);
    const v3 vs[3] = {ld3(M.V + 3 * M.T[3 * s]), ld3(M.V + 3 * M.T[3 * s + 1]), ld3(M.V + 3 * M.T[3 * s + 2])};
    v3 nm = cross(vs[1] - vs[0], vs[2] - vs[0]);
    nm = (1.0 / nrm(nm)) * nm;
    if (lane < 3) {
        const v3 A = lane == 0 ? vs[0] : (lane == 1 ? vs[1] : vs[2]);
        const v3 B = lane == 0 ? vs[1] : (lane == 1 ? vs[2] : vs[0]);
        const v3 e = B - A;
        const double L = nrm(e);
        const v3 et = (1.0 / L) * e, m = cross(et, nm);
        S.len[lane] = L;
        S.et[lane][0] = et.x, S.et[lane][1] = et.y, S.et[lane][2] = et.z;
        S.em[lane][0] = m.x, S.em[lane][1] = m.y, S.em[lane][2] = m.z;
        S.va[lane][0] = A.x, S.va[lane][1] = A.y, S.va[lane][2] = A.z;
    }
    if (lane < NC_NT + 4) {
        const cd z = mk(mjk.re / kabs, mjk.im / kabs);
        cd u = mk(1, 0);
        for (int i = 1; i <= lane; i++) u = (u * z) * cq.rn[i];
        S.u[lane] = make_double2(u.re, u.im);
    }
    __syncwarp();
    if (lane >= 1 && lane < NC_NT + 2) {
        const double2 u0 = S.u[lane - 1], u2 = S.u[lane + 1];
        S.g[lane] = make_double2(-(double)lane * u2.x, -(double)lane * u2.y);
        S.b[lane] = make_double2(cq.rn[lane] * u0.x, cq.rn[lane] * u0.y);
    }
    // outer rule
    int nout;
    v3 ap = a, bp = b, cp = c;
    if (kind == PC_SELF)
        nout = 3 * graded_count(1);
    else if (kind == PC_PLAIN)
        nout = cq.n[QR_OUT] * cq.n[QR_OUT];
    else {
        int sum = 0, first = -1;
        for (int i = 0; i < 3; i++)
            for (int j = 0; j < 3; j++)
                if (tt[i] == M.T[3 * s + j]) {
                    sum += i;
                    if (first < 0) first = i;
                }
        const int ia = kind == PC_EDGE ? 3 - sum : first;  // apex: the vertex off the shared edge, or the shared one
        ap = ia == 0 ? a : (ia == 1 ? b : c);
        bp = ia == 0 ? b : (ia == 1 ? c : a);
        cp = ia == 0 ? c : (ia == 1 ? a : b);
        nout = graded_count(kind == PC_EDGE);
    }
    const int per = graded_count(1);
    const double twoA = nrm(cross(b - a, c - a));
    const double f4 = 1.0 / (4.0 * M_PI);
    const int na = cq.n[QR_ANG];
    cd acc[14];
    for (int i = 0; i < 14; i++) acc[i] = mk(0, 0);
    const int q_hi = min(nout, q_lo + npts);
    __syncwarp();
    for (int q0 = q_lo; q0 < q_hi; q0 += 32) {
        const int qo = q0 + lane;
        int np3[3] = {0, 0, 0};
        double dd = 0.0, ad = 0.0, lad = 0.0, iad = 1.0;
        int ser = 1;
        if (qo < q_hi) {
            v3 r;
            double w;
            if (kind == PC_PLAIN) {
                const int n = cq.n[QR_OUT], i = qo / n, j = qo % n;
                const double u = cq.x[QR_OUT][i], v = cq.x[QR_OUT][j] * (1.0 - u);
                r = a + u * (b - a) + v * (c - a);
                w = twoA * (1.0 - u) * cq.w[QR_OUT][i] * cq.w[QR_OUT][j];
            } else if (kind == PC_SELF) {
                const int sub = qo / per;
                graded_point(ct, sub == 0 ? a : (sub == 1 ? b : c), sub == 0 ? b : (sub == 1 ? c : a), 1, qo % per, r,
                             w);
            } else {
                graded_point(ap, bp, cp, kind == PC_EDGE, qo, r, w);
            }
            const v3 rt = r - ct;
            dd = dot(r - vs[0], nm);
            const v3 rho0 = r - dd * nm;
            const double Rmax = fmax(nrm(vs[0] - r), fmax(nrm(vs[1] - r), nrm(vs[2] - r)));
            if (fabs(dd) < 1e-12 * Rmax) dd = 0.0;  // on the plane up to rounding
            ad = fabs(dd);
            bool off = false;
            if (!REALK && k.im != 0.0) {  // whole triangle beyond RCUT/|Im k|: every term below exp(-RCUT)
                const v3 cc = (1.0 / 3.0) * (vs[0] + vs[1] + vs[2]);
                const double rc = fmax(nrm(vs[0] - cc), fmax(nrm(vs[1] - cc), nrm(vs[2] - cc)));
                off = nrm(r - cc) - rc > RCUT / fabs(k.im);
            }
            ser = kabs * Rmax <= 1.0;
            double Omega = 0.0;
            for (int i = 0; i < 3 && !off; i++) {
                const v3 et = {S.et[i][0], S.et[i][1], S.et[i][2]}, m = {S.em[i][0], S.em[i][1], S.em[i][2]};
                const v3 Ar = ld3(S.va[i]) - rho0, Br = ld3(S.va[i == 2 ? 0 : i + 1]) - rho0;
                const double h = dot(Ar, m), ah = fabs(h);
                if (ah < 1e-12 * S.len[i]) continue;
                const double ta = dot(Ar, et), tb = dot(Br, et);
                Omega += (h > 0 ? 1.0 : -1.0) * (atan2(tb, ah) - atan2(ta, ah));
                const double sa = asinh(ta / ah), sb = asinh(tb / ah);
                const int npa = max(1, (int)ceil((sb - sa) / cq.alen));
                np3[i] = npa;
                S.h[i][lane] = h;
                S.sa[i][lane] = sa;
                S.ds[i][lane] = (sb - sa) / npa;
            }
            S.w[lane] = w;
            S.rt[0][lane] = rt.x;
            S.rt[1][lane] = rt.y;
            S.rt[2][lane] = rt.z;
            if (dd != 0.0) {
                lad = log(ad);
                iad = 1.0 / ad;
            }
            cd ea = mk(1, 0);
            if (dd != 0.0 && !off) {
                ea = cexp_mjkr(k, ad);
                const cd jump = (-f4 * Omega * (dd > 0 ? 1.0 : -1.0)) * ea;
                const double rtv[3] = {rt.x, rt.y, rt.z};
                const cd Ig[3] = {nm.x * jump, nm.y * jump, nm.z * jump};
                const cd z3[3] = {mk(0, 0), mk(0, 0), mk(0, 0)};
                add_moments(acc, w, rtv, kind == PC_SELF, mk(0, 0), z3, Ig);
            }
            S.ead[lane] = make_double2(ea.re, ea.im);
            if (!REALK && !ser && !off && dd != 0.0) {
                // beyond R = RCUT/|Im k| every direction whose edge lies farther
                // away integrates the same truncated range: once per point
                const double Rc = k.im != 0.0 ? RCUT / fabs(k.im) : 1e300;
                double rc = -1.0;
                if (Rc < Rmax) {
                    rc = Rc > ad ? sqrt(Rc * Rc - dd * dd) : 0.0;
                    cd a1, a2;
                    radial_numeric(k, rc, dd, &a1, &a2);
                    S.a1[lane] = make_double2(a1.re, a1.im);
                    S.a2[lane] = make_double2(a2.re, a2.im);
                }
                S.rc[lane] = rc;
            }
        }
        if (ser) {  // I_0^|d| of exp(-jkR) in units of 1/|k|
            cd v = mk(0, 0);
            const double da = kabs * ad;
            double pw = da;
            for (int m = 1; m <= NC_NT && pw > 1e-19 * da; m++, pw *= da) {
                const double2 u = S.u[m - 1];
                v = v + (pw * cq.rn[m]) * mk(u.x, u.y);
            }
            S.is0[lane] = make_double2(v.re, v.im);
        }
        S.dd[lane] = dd;
        S.lad[lane] = lad;
        S.iad[lane] = iad;
        S.ser[lane] = (unsigned char)ser;
        if (na <= NC_NA)
            for (int i = 0; i < 3; i++)
                for (int q = 0; q < na && np3[i] > 0; q++) {
                    const double e = exp(S.ds[i][lane] * cq.x[QR_ANG][q]);
                    S.ep[q][i][lane] = e;
                    S.en[q][i][lane] = 1.0 / e;
                }
        // the panels in work: entry e = panel jp of edge i, held by the points of its mask
        int li = 0, lj = 0;
        while (li < 3) {
            int nent = 0, total = 0;
            for (; li < 3 && nent < NC_LIST; lj++) {
                const unsigned m = __ballot_sync(0xffffffffu, np3[li] > lj);
                if (m == 0) {
                    li++;
                    lj = -1;
                    continue;
                }
                if (lane == 0) {
                    S.mask[nent] = m;
                    S.pre[nent] = total;
                    S.ent[nent] = make_int2(li, lj);
                }
                total += __popc(m);
                nent++;
            }
            if (lane == 0) S.pre[nent] = total;
            __syncwarp();
            for (int it0 = 0; it0 < total; it0 += 32) {
                const int item = it0 + lane;
                const bool on = item < total;
                int lo = 0, hi = nent;  // last entry with pre <= item
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (S.pre[mid] <= item)
                        lo = mid;
                    else
                        hi = mid;
                }
                const int2 en = S.ent[lo];
                const int pt = on ? (int)__fns(S.mask[lo], 0, item - S.pre[lo] + 1) : 0, i = en.x;
                const double h = on ? S.h[i][pt] : 1.0, ah = fabs(h), ds = on ? S.ds[i][pt] : 0.0;
                const double dd = S.dd[pt], ad = fabs(dd), lad = S.lad[pt], iad = S.iad[pt];
                const double s0 = on ? S.sa[i][pt] + ds * en.y : 0.0, e0 = exp(s0), i0 = 1.0 / e0;
                const bool series = S.ser[pt];
                // orders for 1e-18 at the largest |k| R of these panels
                int NT = 4;
                {
                    const float kd = (float)(kabs * ad);
                    const float top = 0.5f * (fmaxf((float)e0 * expf((float)ds), (float)i0) + 1.0f) * (float)(kabs * ah);
                    const float xr = on && series ? sqrtf(top * top + kd * kd) : 0.0f;
                    const float x = __int_as_float(__reduce_max_sync(0xffffffffu, __float_as_int(xr)));
                    float v = x * x * x * x * (1.0f / 24.0f);
                    for (; v > 1e-18f && NT < NC_NT; NT++) v *= x / (float)(NT + 1);
                    NT = (NT + 1) & ~1;
                }
                if (!on) continue;
                cd sis = mk(0, 0), sgn = mk(0, 0), fc = mk(0, 0), fs = mk(0, 0), gc = mk(0, 0), gs = mk(0, 0);
                for (int q = 0; q < na; q++) {
                    const double es = na <= NC_NA ? e0 * S.ep[q][i][pt] : exp(s0 + ds * cq.x[QR_ANG][q]);
                    const double ei = na <= NC_NA ? i0 * S.en[q][i][pt] : 1.0 / es;
                    const double c2 = es + ei, ca = 2.0 / c2, sn = 0.5 * (es - ei) * ca;
                    const double rhom = 0.5 * ah * c2;
                    const double R2 = rhom * rhom + dd * dd, iR = rsqrt(R2), Rm = R2 * iR;
                    const double wa = ds * cq.w[QR_ANG][q] * ca;
                    const double la = log((rhom + Rm) * iad);  // asinh(rhom/|d|), or log 2 rhom in the plane
                    cd is, f1, f2, E;
                    if (series) {
                        const double rs = kabs * rhom, Rs = kabs * Rm, d2 = (kabs * dd) * (kabs * dd);
                        double Rp = 1.0, to = d2 * la, te = d2 * rs;
                        is = mk(0, 0), f1 = mk(0, 0), f2 = mk(0, 0), E = mk(1, 0);
                        for (int m = 1; m <= NT; m += 2) {
                            Rp *= Rs;
                            double A = cq.rn[m + 1] * fma(rs, Rp, -to);
                            to = d2 * (A + to);
                            if (REALK) {  // even powers real, odd ones imaginary
                                f1.re = fma(S.u[m - 1].x, A, f1.re);
                                f2.re = fma(S.g[m].x, A, f2.re);
                                E.im = fma(S.u[m].y, Rp, E.im);
                                is.re = fma(S.b[m].x, Rp, is.re);
                                Rp *= Rs;
                                A = cq.rn[m + 2] * fma(rs, Rp, -te);
                                te = d2 * (A + te);
                                f1.im = fma(S.u[m].y, A, f1.im);
                                f2.im = fma(S.g[m + 1].y, A, f2.im);
                                E.re = fma(S.u[m + 1].x, Rp, E.re);
                                is.im = fma(S.b[m + 1].y, Rp, is.im);
                            } else {
#pragma unroll
                                for (int o = 0; o < 2; o++) {
                                    if (o) {
                                        Rp *= Rs;
                                        A = cq.rn[m + 2] * fma(rs, Rp, -te);
                                        te = d2 * (A + te);
                                    }
                                    const double2 u0 = S.u[m - 1 + o], u1 = S.u[m + o], g = S.g[m + o], b = S.b[m + o];
                                    f1.re = fma(u0.x, A, f1.re);
                                    f1.im = fma(u0.y, A, f1.im);
                                    f2.re = fma(g.x, A, f2.re);
                                    f2.im = fma(g.y, A, f2.im);
                                    E.re = fma(u1.x, Rp, E.re);
                                    E.im = fma(u1.y, Rp, E.im);
                                    is.re = fma(b.x, Rp, is.re);
                                    is.im = fma(b.y, Rp, is.im);
                                }
                            }
                        }
                        is = is - mk(S.is0[pt].x, S.is0[pt].y);
                    } else {
                        E = cexp_mjkr(k, Rm);
                        is = mk(S.ead[pt].x, S.ead[pt].y) * (Rm - ad) * phi1(mjk * (Rm - ad));
                        if (dd == 0.0) {
                            // coplanar point: closed forms with z = j k rhom
                            const cd z = mk(-k.im * rhom, k.re * rhom), jk = mk(-k.im, k.re);
                            f1 = cdivc(mk(1, 0) - E * (mk(1, 0) + z), jk * jk);
                            f2 = mk(1, 0) - E - ein(z, E);
                        } else {
                            // beyond R = RCUT/|Im k| the exponential is below 1e-15: f1 has no
                            // contribution there and (1 + jkR) exp(-jkR) - 1 = -1 integrates in closed form
                            const double Rc = (!REALK && k.im != 0.0) ? RCUT / fabs(k.im) : 1e300;
                            if (Rc < Rm) {
                                const double rc = S.rc[pt], Rcc = sqrt(rc * rc + dd * dd);
                                const double tail = (la + lad - rhom * iR) - (log(rc + Rcc) - rc / Rcc);
                                f1 = mk(S.a1[pt].x, S.a1[pt].y);
                                f2 = mk(S.a2[pt].x - tail, S.a2[pt].y);
                            } else {
                                radial_numeric(k, rhom, dd, &f1, &f2);
                            }
                        }
                    }
                    f2.re += la + lad - rhom * iR;
                    const double wn = -wa * dd * iR, wc = wa * ca, ws = wa * sn;
                    sis = sis + wa * is;
                    sgn = sgn + wn * E;
                    fc = fc + wc * f1;
                    fs = fs + ws * f1;
                    gc = gc + wc * f2;
                    gs = gs + ws * f2;
                }
                const double sh = h > 0 ? 1.0 : -1.0, f = sh * f4, si = series ? f / kabs : f, sf = series ? si / kabs : f;
                const cd Is = si * sis;
                fc = (sf * sh) * fc;  // u = sh m: the in-plane normal toward the edge
                fs = sf * fs;
                gc = f4 * gc;
                gs = f * gs;
                sgn = f * sgn;
                cd Iv[3], Ig[3];
                const double nmv[3] = {nm.x, nm.y, nm.z};
                for (int d = 0; d < 3; d++) {
                    Iv[d] = S.em[i][d] * fc + S.et[i][d] * fs - (dd * nmv[d]) * Is;
                    Ig[d] = S.em[i][d] * gc + S.et[i][d] * gs - nmv[d] * sgn;
                }
                const double rtv[3] = {S.rt[0][pt], S.rt[1][pt], S.rt[2][pt]};
                add_moments(acc, S.w[pt], rtv, kind == PC_SELF, Is, Iv, Ig);
            }
            __syncwarp();
        }
    }
    store_moments(acc, lane, part + 14 * (int64_t)un);
}

// moments of each close pair: its units' parts in order
__global__ void k_near_sum(int n, const int3* __restrict__ own, const double2* __restrict__ part,
                           double2* __restrict__ mom)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 14 * n) return;
    const int3 o = own[idx / 14];  // pair, first unit, units
    const int i = idx % 14;
    double2 s = make_double2(0, 0);
    for (int u = 0; u < o.z; u++) {
        const double2 v = part[14 * (int64_t)(o.y + u) + i];
        s.x += v.x;
        s.y += v.y;
    }
    mom[14 * (int64_t)o.x + i] = s;
}

// outer points of a pair class, as on the device
static void outer_counts(const QuadDev& q, int nout[5])
{
    const int ge = q.opan * q.n[QR_OLAM] * 2 * q.emupan * q.n[QR_EMU], gv = q.opan * q.n[QR_OLAM] * q.n[QR_OMU];
    nout[PC_FAR] = q.n[QR_FAR] * q.n[QR_FAR], nout[PC_PLAIN] = q.n[QR_OUT] * q.n[QR_OUT];
    nout[PC_VERTEX] = gv, nout[PC_EDGE] = ge, nout[PC_SELF] = 3 * ge;
}

// scratch of a build, given back to the stream's pool on every return
struct Scratch {
    cudaStream_t st;
    std::vector<void*> p;
    explicit Scratch(cudaStream_t s) : st(s) {}
    ~Scratch()
    {
        for (void* v : p) cudaFreeAsync(v, st);
    }
    template <class T>
    cudaError_t get(T** d, size_t n)
    {
        const cudaError_t e = cudaMallocAsync((void**)d, sizeof(T) * n, st);
        if (e == cudaSuccess) p.push_back(*d);
        return e;
    }
};

// moments by the panel rule (single objects): far pairs, then the units of the close ones
static sie_status moments_panels(sie_op* op, const AimOp& a, const std::vector<uint8_t>& hc, const int nout[5],
                                 const uint8_t* cls, double2* mom)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const int64_t np = a.npairs;
    k_near_far<<<(unsigned)((np + 3) / 4), 128, 0, st>>>(a.pairs, np, cls, op->mesh->d, a.kr, a.ki, mom);
    SIE_CUDA_TRY(cudaGetLastError());
    int64_t count[5] = {0, 0, 0, 0, 0}, total = 0;
    for (int64_t p = 0; p < np; p++) count[hc[p]]++;
    for (int c = 1; c < 5; c++) total += count[c] * ((nout[c] + 31) / 32);
    // 32 outer points per unit while that keeps the list below 2^18 units (59 MB of parts), then up to 512
    const int npts = 32 * (int)std::min<int64_t>(16, (total >> 18) + 1);
    std::vector<int2> unit;
    std::vector<int3> own;
    for (int c = 4; c >= 1; c--)
        for (int64_t p = 0; p < np && count[c] > 0; p++)
            if (hc[p] == c) {
                const int first = (int)unit.size();
                for (int o = 0; o < nout[c]; o += npts) unit.push_back(make_int2((int)p, o));
                own.push_back(make_int3((int)p, first, (int)unit.size() - first));
            }
    if (unit.empty()) return SIE_OK;
    Scratch mem(st);
    int2* du = nullptr;
    int3* dow = nullptr;
    double2* part = nullptr;
    const int nu = (int)unit.size(), no = (int)own.size();
    SIE_CUDA_TRY(mem.get(&du, nu));
    SIE_CUDA_TRY(mem.get(&dow, no));
    SIE_CUDA_TRY(mem.get(&part, 14 * (size_t)nu));
    SIE_CUDA_TRY(cudaMemcpyAsync(du, unit.data(), sizeof(int2) * nu, cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(dow, own.data(), sizeof(int3) * no, cudaMemcpyHostToDevice, st));
    const unsigned blocks = (unsigned)((nu + NC_W - 1) / NC_W);
    if (a.ki == 0.0)
        k_near_close<true><<<blocks, 32 * NC_W, 0, st>>>(du, nu, npts, a.pairs, cls, op->mesh->d, a.kr, 0.0, part);
    else
        k_near_close<false><<<blocks, 32 * NC_W, 0, st>>>(du, nu, npts, a.pairs, cls, op->mesh->d, a.kr, a.ki, part);
    SIE_CUDA_TRY(cudaGetLastError());
    k_near_sum<<<(14 * no + 127) / 128, 128, 0, st>>>(no, dow, part, mom);
    SIE_CUDA_TRY(cudaGetLastError());
    SIE_CUDA_TRY(cudaStreamSynchronize(st));  // the host lists outlive the copies
    return SIE_OK;
}

// moments from every outer point by itself, in runs of pairs whose points fit the scratch
static sie_status moments_points(sie_op* op, const AimOp& a, const std::vector<uint8_t>& hc, const int nout[5],
                                 double2* mom)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const int64_t np = a.npairs;
    std::vector<int64_t> order;  // by falling work per point
    for (int c = 4; c >= 0; c--)
        for (int64_t p = 0; p < np; p++)
            if (hc[p] == c) order.push_back(p);
    int64_t all = 0;
    for (int64_t p : order) all += (nout[hc[p]] + 31) / 32;
    int most = 0;
    for (int c = 0; c < 5; c++) most = std::max(most, (nout[c] + 31) / 32);
    const int64_t cap = std::min<int64_t>(all, std::max<int64_t>(pt::PT_UNITS, most));
    Scratch mem(st);
    int2* du = nullptr;
    int3* dow = nullptr;
    double* pts = nullptr;
    SIE_CUDA_TRY(mem.get(&du, cap));
    SIE_CUDA_TRY(mem.get(&dow, cap));
    SIE_CUDA_TRY(mem.get(&pts, pt::PT_N * 32 * (size_t)cap));
    std::vector<int2> unit;
    std::vector<int3> own;
    for (size_t at = 0; at < order.size();) {
        unit.clear();
        own.clear();
        for (; at < order.size(); at++) {
            const int p = (int)order[at], n = nout[hc[p]], nu = (n + 31) / 32;
            if ((int64_t)unit.size() + nu > cap) break;
            own.push_back(make_int3(p, (int)unit.size(), n));
            for (int o = 0; o < n; o += 32) unit.push_back(make_int2(p, o));
        }
        const int nu = (int)unit.size(), no = (int)own.size();
        SIE_CUDA_TRY(cudaMemcpyAsync(du, unit.data(), sizeof(int2) * nu, cudaMemcpyHostToDevice, st));
        SIE_CUDA_TRY(cudaMemcpyAsync(dow, own.data(), sizeof(int3) * no, cudaMemcpyHostToDevice, st));
        pt::k_near_points<<<(nu + pt::PT_W - 1) / pt::PT_W, 32 * pt::PT_W, 0, st>>>(
            du, nu, a.pairs, op->mesh->d, a.kr, a.ki, a.obj_k, pts, 32 * cap);
        SIE_CUDA_TRY(cudaGetLastError());
        pt::k_near_gather<<<(no + 3) / 4, 128, 0, st>>>(no, dow, a.pairs, pts, 32 * cap, mom);
        SIE_CUDA_TRY(cudaGetLastError());
        SIE_CUDA_TRY(cudaStreamSynchronize(st));  // the host lists outlive the copies
    }
    return SIE_OK;
}

// moments of all near pairs of a; points: every outer point by itself (near_points.cuh)
static sie_status near_moments(sie_op* op, const AimOp& a, const QuadDev& q, bool points, double2* mom)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const DevMesh& M = op->mesh->d;
    const int64_t np = a.npairs;
    if (np <= 0) return SIE_OK;
    Scratch mem(st);
    uint8_t* cls = nullptr;
    std::vector<uint8_t> hc(np);
    SIE_CUDA_TRY(mem.get(&cls, np));
    k_pair_class<<<(unsigned)((np + 255) / 256), 256, 0, st>>>(a.pairs, np, M, a.kr, a.ki, a.obj_k, cls);
    SIE_CUDA_TRY(cudaGetLastError());
    SIE_CUDA_TRY(cudaMemcpyAsync(hc.data(), cls, np, cudaMemcpyDeviceToHost, st));
    SIE_CUDA_TRY(cudaStreamSynchronize(st));
    int nout[5];
    outer_counts(q, nout);
    return points ? moments_points(op, a, hc, nout, mom) : moments_panels(op, a, hc, nout, cls, mom);
}

// kernel values at integer lags |l_d| <= Lm: (G, dG/dx, dG/dy, dG/dz), zero at lag 0
__global__ void k_lagtab(int Lm, double h, double kr, double ki, double2* __restrict__ tab)
{
    int W = 2 * Lm + 1;
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= W * W * W) return;
    int lx = idx % W - Lm, ly = (idx / W) % W - Lm, lz = idx / (W * W) - Lm;
    double dx = h * lx, dy = h * ly, dz = h * lz;
    double R = sqrt(dx * dx + dy * dy + dz * dz);
    cd G = mk(0, 0), gx = mk(0, 0), gy = mk(0, 0), gz = mk(0, 0);
    if (R > 0) {
        cd e = cexpc(mk(ki * R, -kr * R));
        G = (1.0 / (4.0 * M_PI * R)) * e;
        cd g = (-1.0 / (4.0 * M_PI * R * R * R)) * (mk(1.0 - ki * R, kr * R) * e);
        gx = dx * g;
        gy = dy * g;
        gz = dz * g;
    }
    tab[4 * idx + 0] = make_double2(G.re, G.im);
    tab[4 * idx + 1] = make_double2(gx.re, gx.im);
    tab[4 * idx + 2] = make_double2(gy.re, gy.im);
    tab[4 * idx + 3] = make_double2(gz.re, gz.im);
}

// Per pair: exact local entries (LA 3x3, K 3x3, Lphi) minus the grid's own
// entries for the pair when the operator has a grid, plus the exact LA and
// Lphi.  One warp per pair; lanes own the test-stencil nodes u.  out: NLOC
// complex per pair.
__global__ void __launch_bounds__(128) k_near_local(const int32_t* __restrict__ pairs, int64_t np, DevMesh M,
                                                    const double2* __restrict__ mom, int has_grid, int S, int Mord,
                                                    const int32_t* __restrict__ base, const double* __restrict__ Wt,
                                                    const double2* __restrict__ tab, int Lm, double2* __restrict__ out)
{
    int64_t p = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    int lane = threadIdx.x & 31;
    if (p >= np) return;
    int t = pairs[2 * p], s = pairs[2 * p + 1];
    // grid part: W_t^T G W_s and its curl form.  A lane owns a test node u and
    // first sums over the source nodes v the four weights (w0, w1) of v times G
    // and grad G (32 FMAs a node pair); the 3 x 3 local entries are then linear
    // in a few sums over u (forming all 18 per node pair took 170).
    // gs: LA: 0 sum_a w1_a|w1_a, 1..3 w1_a|w0, 4..6 w0|w1_a, 7 w0|w0 (also Lphi);
    // K (curl form, D = grad G): 8 all weights w1, 9..11 w1 on the test side (by
    // source component), 12..14 w1 on the source side (by test component), 15..17 w0|D|w0
    cd gs[18];
    for (int i = 0; i < 18; i++) gs[i] = mk(0, 0);
    if (has_grid) {
        const int Mp = Mord + 1;
        int bt[3] = {base[3 * t], base[3 * t + 1], base[3 * t + 2]};
        int bs[3] = {base[3 * s], base[3 * s + 1], base[3 * s + 2]};
        const int Wd = 2 * Lm + 1;
        for (int u = lane; u < S; u += 32) {
            const int ux = u % Mp, uy = (u / Mp) % Mp, uz = u / (Mp * Mp);
            const double* wu = Wt + ((size_t)t * S + u) * 4;
            cd Y[4][4];  // [G, Dx, Dy, Dz][w0, w1x, w1y, w1z]
            for (int i = 0; i < 16; i++) Y[i / 4][i % 4] = mk(0, 0);
            int v = 0;
            for (int vz = 0; vz < Mp; vz++)
                for (int vy = 0; vy < Mp; vy++)
                    for (int vx = 0; vx < Mp; vx++, v++) {
                        const int lx = bt[0] + ux - bs[0] - vx, ly = bt[1] + uy - bs[1] - vy,
                                  lz = bt[2] + uz - bs[2] - vz;
                        const double2* kv = tab + 4 * (((lz + Lm) * Wd + (ly + Lm)) * Wd + (lx + Lm));
                        const double* wv = Wt + ((size_t)s * S + v) * 4;
#pragma unroll
                        for (int g = 0; g < 4; g++) {
                            const double2 kg = kv[g];
#pragma unroll
                            for (int c = 0; c < 4; c++) {
                                Y[g][c].re = fma(wv[c], kg.x, Y[g][c].re);
                                Y[g][c].im = fma(wv[c], kg.y, Y[g][c].im);
                            }
                        }
                    }
            const double w0 = wu[0], w1[3] = {wu[1], wu[2], wu[3]};
            gs[0] = gs[0] + w1[0] * Y[0][1] + w1[1] * Y[0][2] + w1[2] * Y[0][3];
            gs[7] = gs[7] + w0 * Y[0][0];
#pragma unroll
            for (int d = 0; d < 3; d++) {
                const int e = (d + 1) % 3, f = (d + 2) % 3;
                gs[1 + d] = gs[1 + d] + w1[d] * Y[0][0];
                gs[4 + d] = gs[4 + d] + w0 * Y[0][1 + d];
                // eps_abc x_a D_b y_c, a = d: (b, c) = (e, f) minus (f, e)
                const cd curl = Y[1 + e][1 + f] - Y[1 + f][1 + e];
                gs[8] = gs[8] + w1[d] * curl;
                gs[12 + d] = gs[12 + d] + w0 * curl;
                // c = d: (a, b) = (e, f) minus (f, e)
                gs[9 + d] = gs[9 + d] + w1[e] * Y[1 + f][0] - w1[f] * Y[1 + e][0];
                gs[15 + d] = gs[15 + d] + w0 * Y[1 + d][0];
            }
        }
        for (int off = 16; off > 0; off >>= 1)
            for (int i = 0; i < 18; i++) {
                gs[i].re += __shfl_xor_sync(0xffffffffu, gs[i].re, off);
                gs[i].im += __shfl_xor_sync(0xffffffffu, gs[i].im, off);
            }
    }
    if (lane >= 10) return;
    const double2* mm = mom + 14 * p;
    double2* o = out + NLOC * p;
    const cd Q0 = mk(mm[0].x, mm[0].y);
    if (lane == 9) {  // scalar potential
        const double At = M.area[t], As = M.area[s];
        const cd lp = (1.0 / (At * As)) * (Q0 - gs[7]);
        o[18] = make_double2(lp.re, lp.im);
        const cd lpe = (1.0 / (At * As)) * Q0;
        o[28] = make_double2(lpe.re, lpe.im);  // exact
        return;
    }
    // a lane per local entry (i, j): exact value from the moments, grid value from gs
    const int i = lane / 3, j = lane % 3;
    cd Q1[3], Q2[3], U[3], Vv[3];
    for (int d = 0; d < 3; d++) {
        Q1[d] = mk(mm[1 + d].x, mm[1 + d].y);
        Q2[d] = mk(mm[4 + d].x, mm[4 + d].y);
        U[d] = mk(mm[8 + d].x, mm[8 + d].y);
        Vv[d] = mk(mm[11 + d].x, mm[11 + d].y);
    }
    const cd Q3 = mk(mm[7].x, mm[7].y);
    const v3 ctc = ld3(M.cen + 3 * t);
    const double cm = M.coef[3 * t + i], cn = M.coef[3 * s + j];
    const v3 pm = ld3(M.V + 3 * M.T[3 * t + i]) - ctc, pn = ld3(M.V + 3 * M.T[3 * s + j]) - ctc;
    cd la = Q3 - (pn.x * Q1[0] + pn.y * Q1[1] + pn.z * Q1[2]) - (pm.x * Q2[0] + pm.y * Q2[1] + pm.z * Q2[2]) +
            dot(pm, pn) * Q0;
    const v3 dl = pn - pm, cx = cross(pn, pm);
    cd kk = dl.x * U[0] + dl.y * U[1] + dl.z * U[2] + cx.x * Vv[0] + cx.y * Vv[1] + cx.z * Vv[2];
    la = (cm * cn) * la;
    o[19 + 3 * i + j] = make_double2(la.re, la.im);  // exact
    if (has_grid) {
        const double* qt = M.q + 9 * t + 3 * i;
        const double* qs = M.q + 9 * s + 3 * j;
        // sum_a (w1 + qt w0)_a (w1 + qs w0)_a G
        const cd gl = gs[0] + qs[0] * gs[1] + qs[1] * gs[2] + qs[2] * gs[3] + qt[0] * gs[4] + qt[1] * gs[5] +
                      qt[2] * gs[6] + (qt[0] * qs[0] + qt[1] * qs[1] + qt[2] * qs[2]) * gs[7];
        // sum_abc eps_abc (w1 + qt w0)_a D_b (w1 + qs w0)_c
        const cd gk = gs[8] + qs[0] * gs[9] + qs[1] * gs[10] + qs[2] * gs[11] + qt[0] * gs[12] + qt[1] * gs[13] +
                      qt[2] * gs[14] + (qs[1] * qt[2] - qs[2] * qt[1]) * gs[15] +
                      (qs[2] * qt[0] - qs[0] * qt[2]) * gs[16] + (qs[0] * qt[1] - qs[1] * qt[0]) * gs[17];
        la = la - (cm * cn) * gl;
        kk = kk - gk;
    }
    kk = (cm * cn) * kk;
    o[3 * i + j] = make_double2(la.re, la.im);
    o[9 + 3 * i + j] = make_double2(kk.re, kk.im);
}

// CSR values: entry (m, n) sums the local entries of the near pairs (t, s)
// with t in supp(f_m), s in supp(f_n), in a fixed order (deterministic).
// vL = L (exact - grid), vK = K (exact - grid), vLA = LA (exact - grid);
// diagonal entries also give the exact LA and L diagonals (dLA, dL).
__global__ void k_csr_fill(int ne, const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                           const int64_t* __restrict__ pstart, const int32_t* __restrict__ pairs,
                           const double2* __restrict__ loc, DevMesh M, double2 invk2,
                           const double2* __restrict__ obj_invk2, double2* __restrict__ vL,
                           double2* __restrict__ vK, double2* __restrict__ vLA, double2* __restrict__ dLA,
                           double2* __restrict__ dL)
{
    int m = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    int lane = threadIdx.x & 31;
    if (m >= ne) return;
    if (obj_invk2) invk2 = obj_invk2[M.obj[M.edge_tri[2 * m]]];  // row m's object
    cd ik2 = mk(invk2.x, invk2.y);
    for (int64_t e = row_ptr[m] + lane; e < row_ptr[m + 1]; e += 32) {
        int n = col[e];
        cd L = mk(0, 0), K = mk(0, 0), LA = mk(0, 0), LAx = mk(0, 0), Lx = mk(0, 0);
        for (int a = 0; a < 2; a++) {
            int t = M.edge_tri[2 * m + a], i = M.edge_slot[2 * m + a];
            int64_t lo = pstart[t], hi = pstart[t + 1];
            for (int b = 0; b < 2; b++) {
                int s = M.edge_tri[2 * n + b], j = M.edge_slot[2 * n + b];
                // binary search s in pairs[lo..hi)
                int64_t l = lo, r = hi;
                while (l < r) {
                    int64_t mid = (l + r) >> 1;
                    if (pairs[2 * mid + 1] < s)
                        l = mid + 1;
                    else
                        r = mid;
                }
                if (l < hi && pairs[2 * l + 1] == s) {
                    const double2* o = loc + NLOC * l;
                    double c4 = 4.0 * M.coef[3 * t + i] * M.coef[3 * s + j] * M.area[t] * M.area[s];
                    cd lp = mk(o[18].x, o[18].y), lpe = mk(o[28].x, o[28].y);
                    cd la = mk(o[3 * i + j].x, o[3 * i + j].y), lae = mk(o[19 + 3 * i + j].x, o[19 + 3 * i + j].y);
                    LA = LA + la;
                    L = L + la - c4 * (ik2 * lp);
                    K = K + mk(o[9 + 3 * i + j].x, o[9 + 3 * i + j].y);
                    LAx = LAx + lae;
                    Lx = Lx + lae - c4 * (ik2 * lpe);
                }
            }
        }
        vL[e] = make_double2(L.re, L.im);
        vK[e] = make_double2(K.re, K.im);
        vLA[e] = make_double2(LA.re, LA.im);
        if (n == m) {
            dLA[m] = make_double2(LAx.re, LAx.im);
            dL[m] = make_double2(Lx.re, Lx.im);
        }
    }
}

__global__ void k_recip(int n, const double2* __restrict__ d, double2* __restrict__ r)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const cd v = cdivc(mk(1.0, 0.0), mk(d[i].x, d[i].y));
    r[i] = make_double2(v.re, v.im);
}

__global__ void k_lphi_vals(int64_t np, const double2* __restrict__ loc, double2* __restrict__ v,
                            double2* __restrict__ vnr)
{
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < np) {
        v[p] = loc[NLOC * p + 18];    // exact - grid
        vnr[p] = loc[NLOC * p + 28];  // exact (near-region matrix, preconditioner)
    }
}

sie_status near_build(sie_op* op, AimOp& a, const QuadDev& q)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const DevMesh& M = op->mesh->d;
    const HostMesh& H = op->mesh->h;
    SIE_CUDA_TRY(cudaMemcpyToSymbolAsync(cq, &q, sizeof(QuadDev), 0, cudaMemcpyHostToDevice, st));
    a.npairs = (int64_t)a.hpairs.size() / 2;
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.pairs, sizeof(int32_t) * 2 * std::max<int64_t>(a.npairs, 1), st));
    SIE_CUDA_TRY(cudaMemcpyAsync(a.pairs, a.hpairs.data(), sizeof(int32_t) * 2 * a.npairs, cudaMemcpyHostToDevice, st));
    double2 *mom = nullptr, *loc = nullptr, *tab = nullptr;
    SIE_CUDA_TRY(cudaMallocAsync((void**)&mom, sizeof(double2) * 14 * std::max<int64_t>(a.npairs, 1), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&loc, sizeof(double2) * NLOC * std::max<int64_t>(a.npairs, 1), st));
    const int wpb = 4;
    // operators without an interior grid: lockstep block products (near_points.cuh)
    const bool points = !op->inn.has_grid;
    SIE_TRY(near_moments(op, a, q, points, mom));
    int Lm = a.g.Rnear + a.g.M;
    int S = (a.g.M + 1) * (a.g.M + 1) * (a.g.M + 1);
    if (a.has_grid) {
        int W = 2 * Lm + 1;
        SIE_CUDA_TRY(cudaMallocAsync((void**)&tab, sizeof(double2) * 4 * W * W * W, st));
        k_lagtab<<<(W * W * W + 127) / 128, 128, 0, st>>>(Lm, a.g.h, a.kr, a.ki, tab);
        SIE_CUDA_TRY(cudaGetLastError());
    }
    if (a.npairs > 0) {
        auto local = points ? pt::k_near_local : k_near_local;
        local<<<(unsigned)((a.npairs + wpb - 1) / wpb), 32 * wpb, 0, st>>>(
            a.pairs, a.npairs, M, mom, a.has_grid ? 1 : 0, S, a.g.M, op->base, op->W, tab, Lm, loc);
        SIE_CUDA_TRY(cudaGetLastError());
    }
    // CSR over edges
    edge_csr_pattern(H, a.hpairs, a.csr);
    a.nnz = (int64_t)a.csr.col.size();
    std::vector<int64_t> pstart(H.nt + 1, 0);
    for (int64_t p = 0; p < a.npairs; p++) pstart[a.hpairs[2 * p] + 1]++;
    for (int64_t t = 0; t < H.nt; t++) pstart[t + 1] += pstart[t];
    int64_t* dps = nullptr;
    SIE_CUDA_TRY(cudaMallocAsync((void**)&dps, sizeof(int64_t) * (H.nt + 1), st));
    SIE_CUDA_TRY(cudaMemcpyAsync(dps, pstart.data(), sizeof(int64_t) * (H.nt + 1), cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.row_ptr, sizeof(int64_t) * (H.ne + 1), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.col, sizeof(int32_t) * std::max<int64_t>(a.nnz, 1), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.valL, sizeof(double2) * std::max<int64_t>(a.nnz, 1), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.valK, sizeof(double2) * std::max<int64_t>(a.nnz, 1), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.valLA, sizeof(double2) * std::max<int64_t>(a.nnz, 1), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.dLA, sizeof(double2) * H.ne, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.dL, sizeof(double2) * H.ne, st));
    SIE_CUDA_TRY(cudaMemsetAsync(a.dLA, 0, sizeof(double2) * H.ne, st));
    SIE_CUDA_TRY(cudaMemsetAsync(a.dL, 0, sizeof(double2) * H.ne, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(a.row_ptr, a.csr.row_ptr.data(), sizeof(int64_t) * (H.ne + 1), cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(a.col, a.csr.col.data(), sizeof(int32_t) * a.nnz, cudaMemcpyHostToDevice, st));
    std::complex<double> kk(a.kr, a.ki);
    std::complex<double> ik2 = 1.0 / (kk * kk);
    k_csr_fill<<<(unsigned)((H.ne + 3) / 4), 128, 0, st>>>((int)H.ne, a.row_ptr, a.col, dps, a.pairs, loc, M,
                                                           make_double2(ik2.real(), ik2.imag()), a.obj_ik2, a.valL,
                                                           a.valK,
                                                           a.valLA, a.dLA, a.dL);
    SIE_CUDA_TRY(cudaGetLastError());
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.idLA, sizeof(double2) * H.ne, st));
    k_recip<<<(unsigned)((H.ne + 255) / 256), 256, 0, st>>>((int)H.ne, a.dLA, a.idLA);
    SIE_CUDA_TRY(cudaGetLastError());
    // triangle CSR of Lphi (exact - grid): rows = pair blocks, columns = s
    a.tri_row_ptr_h = pstart;
    a.tri_col_h.resize(a.npairs);
    for (int64_t p = 0; p < a.npairs; p++) a.tri_col_h[p] = a.hpairs[2 * p + 1];
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.tri_row_ptr, sizeof(int64_t) * (H.nt + 1), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.tri_col, sizeof(int32_t) * std::max<int64_t>(a.npairs, 1), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.valLphi, sizeof(double2) * std::max<int64_t>(a.npairs, 1), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&a.valLphiNR, sizeof(double2) * std::max<int64_t>(a.npairs, 1), st));
    SIE_CUDA_TRY(cudaMemcpyAsync(a.tri_row_ptr, a.tri_row_ptr_h.data(), sizeof(int64_t) * (H.nt + 1),
                                 cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(a.tri_col, a.tri_col_h.data(), sizeof(int32_t) * a.npairs, cudaMemcpyHostToDevice, st));
    if (a.npairs > 0) {
        k_lphi_vals<<<(unsigned)((a.npairs + 255) / 256), 256, 0, st>>>(a.npairs, loc, a.valLphi, a.valLphiNR);
        SIE_CUDA_TRY(cudaGetLastError());
    }
    SIE_CUDA_TRY(cudaFreeAsync(dps, st));
    SIE_CUDA_TRY(cudaFreeAsync(mom, st));
    SIE_CUDA_TRY(cudaFreeAsync(loc, st));
    if (tab) SIE_CUDA_TRY(cudaFreeAsync(tab, st));
    SIE_CUDA_TRY(cudaStreamSynchronize(st));
    return SIE_OK;
}

}  // namespace sie

// Near-pair moments and local entries of operators whose interior has no grid
// (near-region-only and SIBC interiors): the inner integral of every outer point by
// itself, and sums in a fixed order.
//
// The lockstep solves of these operators stop at tol_outer and round the vectors of
// their preconditioner to complex64, so their solutions depend on every rounding of
// the entries: a change of 1e-16 moves x of a copper bar by 2.5e-3.  To keep the
// solutions that programs have, these functions keep their operations and the order of
// their sums; the panel rule of near.cu, whose entries differ by 2e-14, serves
// penetrable objects, whose block products are made one vector at a time.
//
// k_near_points takes a thread per outer point and stores what it adds to the moments
// (26 numbers); k_near_gather sums a pair's points, a lane every 32nd of them, then a
// tree over the lanes.  With one warp per pair and its points in a loop, the 1,680 points
// of a self pair were a chain of 53 rounds on a nearly empty GPU: build of a copper cube
// of 48 triangles 1,907 -> 356 ms, exterior near region of 1,280 triangles 2,259 -> 1,717
// ms (FP64 arithmetic bounds it, the pipe is 82 to 85% busy: 2,300 operations a
// direction, the panel rule has 286).
//
// A compiler may fuse either product of a sum of two, and decides from the code around
// it: k_near_points keeps the statements of a point together for that reason.
#pragma once
#include "internal.h"

namespace sie {
namespace pt {

__device__ __forceinline__ double cabsc(cd z) { return hypot(z.re, z.im); }
__device__ __forceinline__ cd clogc(cd z) { return mk(log(hypot(z.re, z.im)), atan2(z.im, z.re)); }

// (exp(z) - 1)/z
__device__ cd phi1(cd z)
{
    if (cabsc(z) < 0.5) {
        cd term = mk(1, 0), s = mk(1, 0);
        for (int n = 1; n < 20; n++) {
            term = term * z * (1.0 / (double)(n + 1));
            s = s + term;
        }
        return s;
    }
    return cdivc(cexpc(z) - mk(1, 0), z);
}

// (1 + z) exp(-z) - 1 with a series near 0
__device__ cd hfun(cd z)
{
    if (cabsc(z) < 0.2) {
        cd s = mk(0, 0), zn = z;
        double fact = 1.0;
        for (int n = 2; n < 16; n++) {
            zn = zn * z;
            fact *= n;
            double sg = (n % 2 == 0) ? -1.0 : 1.0;
            s = s + (sg * (double)(n - 1) / fact) * zn;
        }
        return s;
    }
    return (mk(1, 0) + z) * cexpc(mk(-z.re, -z.im)) - mk(1, 0);
}

// Ein(z) = I_0^z (1 - exp(-t))/t dt for Re z >= 0: series for |z| < 2, else
// E1(z) + log z + gamma, E1 by its continued fraction (modified Lentz)
__device__ cd ein(cd z)
{
    if (cabsc(z) < 2.0) {
        cd s = mk(0, 0), t = mk(1, 0);
        for (int n = 1; n < 60; n++) {
            t = t * z * (1.0 / (double)n);
            cd term = ((n & 1) ? 1.0 : -1.0) / (double)n * t;
            s = s + term;
            if (cabsc(term) < 1e-17 * cabsc(s)) break;
        }
        return s;
    }
    const double tiny = 1e-300;
    cd f = z, C = z, D = mk(0, 0);
    for (int i = 1; i < 500; i++) {
        double a = (double)((i + 1) / 2);
        cd b = (i & 1) ? mk(1, 0) : z;
        D = b + a * D;
        if (cabsc(D) < tiny) D = mk(tiny, 0);
        C = b + cdivc(mk(a, 0), C);
        if (cabsc(C) < tiny) C = mk(tiny, 0);
        D = cdivc(mk(1, 0), D);
        cd delta = C * D;
        f = f * delta;
        if (cabsc(delta - mk(1, 0)) < 1e-16) break;
    }
    const double euler = 0.57721566490153286061;
    return cdivc(cexpc(mk(-z.re, -z.im)), f) + clogc(z) + mk(euler, 0);
}

struct RadCache {
    bool valid;
    double rc;
    cd a1, a2;
};

__device__ void radial_numeric(cd k, double rc, double d, cd* a1o, cd* a2o)
{
    cd a1 = mk(0, 0), a2 = mk(0, 0);
    double hi = rc;
    for (int p = 0; p < cq.npan && rc > 0.0; p++) {
        double lo = (p == cq.npan - 1) ? 0.0 : hi * cq.ratio;
        for (int qq = 0; qq < cq.n[QR_RAD]; qq++) {
            double rho = lo + (hi - lo) * cq.x[QR_RAD][qq];
            double wr = (hi - lo) * cq.w[QR_RAD][qq];
            double R = sqrt(rho * rho + d * d);
            cd z = mk(-k.im * R, k.re * R);  // j k R
            cd e = cexpc(mk(-z.re, -z.im));
            cd hz = cabsc(z) < 0.2 ? pt::hfun(z) : (mk(1, 0) + z) * e - mk(1, 0);
            a1 = a1 + (wr * rho * rho / R) * e;
            a2 = a2 + (wr * rho * rho / (R * R * R)) * hz;
        }
        hi = lo;
    }
    *a1o = a1;
    *a2o = a2;
}

// bounded radial remainders (series when |k| Rmax <= 1, else graded Gauss)
__device__ void radial(cd k, double rhom, double d, double Rmax, cd* f1, cd* f2, RadCache* cache)
{
    if (cabsc(k) * Rmax <= 1.0) {
        double rs = rhom / Rmax, ds = d / Rmax, Rs = sqrt(rs * rs + ds * ds), d2 = ds * ds;
        cd ks = k * Rmax;
        const int NT = 26;
        double B[NT + 4];
        B[0] = (d2 > 0.0) ? d2 * asinh(rs / fabs(ds)) : 0.0;  // d^2 B_-1
        B[1] = rs;                                           // B_0
        double Rp = 1.0, bodd = 0.0, beven = rs;
        for (int m = 1; m <= NT + 2; m++) {
            Rp *= Rs;
            double bm;
            if (m & 1) {
                double d2b = (m == 1) ? B[0] : d2 * bodd;
                bm = (rs * Rp + m * d2b) / (m + 1);
                bodd = bm;
            } else {
                bm = (rs * Rp + m * d2 * beven) / (m + 1);
                beven = bm;
            }
            B[m + 1] = bm;
        }
        double A[NT + 2];
        A[0] = B[2] - B[0];
        for (int m = 0; m <= NT; m++) A[m + 1] = B[m + 3] - d2 * B[m + 1];
        cd s1 = mk(0, 0), s2 = mk(0, 0), t1 = mk(1, 0);
        cd mjk = mk(ks.im, -ks.re);  // -j ks
        for (int n = 0; n <= NT; n++) {
            if (n > 0) t1 = t1 * mjk * (1.0 / (double)n);
            s1 = s1 + A[n] * t1;
            if (n >= 2) s2 = s2 + (-(double)(n - 1) * A[n - 2]) * t1;
        }
        *f1 = s1 * (Rmax * Rmax);
        *f2 = s2;
        return;
    }
    if (d == 0.0) {
        // coplanar point: closed forms with z = j k rhom
        cd z = mk(-k.im * rhom, k.re * rhom), e = cexpc(mk(-z.re, -z.im));
        cd jk = mk(-k.im, k.re);
        *f1 = cdivc(mk(1, 0) - e * (mk(1, 0) + z), jk * jk);
        *f2 = mk(1, 0) - e - pt::ein(z);
        return;
    }
    // beyond R = RCUT/|Im k| the exponential is below 1e-15: f1 has no
    // contribution there and (1 + jkR) exp(-jkR) - 1 = -1 integrates in closed form
    double rc = rhom, tail = 0.0;
    bool trunc = false;
    double kim = fabs(k.im);
    if (kim > 0.0) {
        double Rc = RCUT / kim, Rm = sqrt(rhom * rhom + d * d);
        if (Rc < Rm) {
            trunc = true;
            rc = Rc > fabs(d) ? sqrt(Rc * Rc - d * d) : 0.0;
            double Rcc = sqrt(rc * rc + d * d);
            tail = (log(rhom + Rm) - rhom / Rm) - (log(rc + Rcc) - rc / Rcc);
        }
    }
    cd a1, a2;
    if (trunc) {
        // truncated: the range [0, rc] depends on d only
        if (!cache->valid || cache->rc != rc) {
            pt::radial_numeric(k, rc, d, &cache->a1, &cache->a2);
            cache->rc = rc;
            cache->valid = true;
        }
        a1 = cache->a1;
        a2 = cache->a2;
    } else {
        pt::radial_numeric(k, rc, d, &a1, &a2);
    }
    a2 = a2 - mk(tail, 0);
    *f1 = a1;
    *f2 = a2;
}

__device__ void inner_polar(v3 r, v3 v0, v3 v1, v3 v2, cd k, Inner& o)
{
    v3 vv[3] = {v0, v1, v2};
    v3 nm = cross(v1 - v0, v2 - v0);
    nm = (1.0 / nrm(nm)) * nm;
    double dd = dot(r - v0, nm);
    v3 rho0 = r - dd * nm;
    double Rmax = fmax(nrm(v0 - r), fmax(nrm(v1 - r), nrm(v2 - r)));
    if (fabs(dd) < 1e-12 * Rmax) dd = 0.0;  // on the plane up to rounding
    double ad = fabs(dd);
    o.Is = mk(0, 0);
    for (int d = 0; d < 3; d++) o.Iv[d] = o.Ig[d] = mk(0, 0);
    if (k.im != 0.0) {  // whole triangle beyond RCUT/|Im k|: every term below exp(-RCUT)
        v3 c = (1.0 / 3.0) * (v0 + v1 + v2);
        double rc = fmax(nrm(v0 - c), fmax(nrm(v1 - c), nrm(v2 - c)));
        if (nrm(r - c) - rc > RCUT / fabs(k.im)) return;
    }
    cd Is = mk(0, 0), Ign = mk(0, 0), Iv[3] = {mk(0, 0), mk(0, 0), mk(0, 0)}, Igt[3] = {mk(0, 0), mk(0, 0), mk(0, 0)};
    RadCache rcache;
    rcache.valid = false;
    double Omega = 0.0;
    cd mjk = mk(k.im, -k.re);  // -j k
    for (int i = 0; i < 3; i++) {
        v3 A = vv[i], B = vv[(i + 1) % 3];
        v3 e = B - A;
        double L = nrm(e);
        v3 et = (1.0 / L) * e;
        v3 m = cross(et, nm);
        v3 Ar = A - rho0, Br = B - rho0;
        double h = dot(Ar, m);
        if (fabs(h) < 1e-12 * L) continue;
        double sh = h > 0 ? 1.0 : -1.0, ah = fabs(h);
        v3 u = sh * m;
        double ta = dot(Ar, et), tb = dot(Br, et);
        Omega += sh * (atan2(tb, ah) - atan2(ta, ah));
        double sa = asinh(ta / ah), sb = asinh(tb / ah);
        int npa = (int)ceil((sb - sa) / cq.alen);
        if (npa < 1) npa = 1;
        double ds = (sb - sa) / npa;
        const int na = cq.n[QR_ANG];
        for (int j = 0; j < na * npa; j++) {
            int jp = j / na, jq = j % na;
            double s = sa + ds * (jp + cq.x[QR_ANG][jq]);
            double ch = cosh(s);
            double wa = sh * ds * cq.w[QR_ANG][jq] / ch;
            double ca = 1.0 / ch, sn = tanh(s);
            v3 eh = ca * u + sn * et;
            double rhom = ah * ch;
            double Rm = sqrt(rhom * rhom + dd * dd);
            cd is = cexpc(mjk * ad) * (Rm - ad) * pt::phi1(mjk * (Rm - ad));
            cd f1, f2;
            radial(k, rhom, dd, Rmax, &f1, &f2, &rcache);
            cd igt = mk(log(rhom + Rm) - rhom / Rm, 0) + f2;
            cd ign = (-dd / Rm) * cexpc(mjk * Rm);
            Is = Is + wa * is;
            Ign = Ign + wa * ign;
            double ehv[3] = {eh.x, eh.y, eh.z}, nmv[3] = {nm.x, nm.y, nm.z};
            for (int d = 0; d < 3; d++) {
                Iv[d] = Iv[d] + wa * (ehv[d] * f1 - (dd * nmv[d]) * is);
                Igt[d] = Igt[d] + (wa * ehv[d]) * igt;
            }
        }
    }
    cd jump = mk(0, 0);
    if (dd != 0.0) jump = (Omega * (dd > 0 ? 1.0 : -1.0)) * cexpc(mjk * ad);
    const double f = 1.0 / (4.0 * M_PI);
    double nmv[3] = {nm.x, nm.y, nm.z};
    o.Is = f * Is;
    for (int d = 0; d < 3; d++) {
        o.Iv[d] = f * Iv[d];
        o.Ig[d] = (-f) * (nmv[d] * (jump + Ign) - Igt[d]);
    }
}

__device__ void inner_gauss(v3 r, v3 a, v3 b, v3 c, cd k, Inner& o)
{
    v3 e1 = b - a, e2 = c - a;
    double twoA = nrm(cross(e1, e2));
    o.Is = mk(0, 0);
    for (int d = 0; d < 3; d++) o.Iv[d] = o.Ig[d] = mk(0, 0);
    const int n = cq.n[QR_FAR];
    for (int i = 0; i < n; i++) {
        double u = cq.x[QR_FAR][i];
        for (int j = 0; j < n; j++) {
            double v = cq.x[QR_FAR][j] * (1.0 - u);
            double w = twoA * (1.0 - u) * cq.w[QR_FAR][i] * cq.w[QR_FAR][j];
            v3 p = a + u * e1 + v * e2;
            v3 dv = p - r;
            double R = nrm(dv);
            cd e = cexpc(mk(k.im * R, -k.re * R));
            cd G = (1.0 / (4.0 * M_PI * R)) * e;
            cd g = (-1.0 / (4.0 * M_PI * R * R * R)) * (mk(1.0 - k.im * R, k.re * R) * e);
            o.Is = o.Is + w * G;
            double dvv[3] = {dv.x, dv.y, dv.z};
            for (int d = 0; d < 3; d++) {
                o.Iv[d] = o.Iv[d] + (w * dvv[d]) * G;
                o.Ig[d] = o.Ig[d] + (-w * dvv[d]) * g;
            }
        }
    }
}

constexpr int PT_W = 4;                 // warps per CTA
constexpr int PT_N = 26;                // numbers per point
constexpr int64_t PT_UNITS = 1 << 16;   // units in work at a time (436 MB of points)

// unit: (pair, first of 32 outer points); number c of point l of unit u at
// out[c ld + 32 u + l]: w, w rt[3] (rt = r - c_t), Is, I2[3] = Iv + rt Is, rt . I2, rt x Ig, Ig
__global__ void __launch_bounds__(32 * PT_W) k_near_points(const int2* __restrict__ unit, int nunit,
                                                           const int32_t* __restrict__ pairs, DevMesh M, double kr,
                                                           double ki, const double2* __restrict__ obj_k,
                                                           double* __restrict__ out, int64_t ld)
{
    const int un = blockIdx.x * PT_W + threadIdx.x / 32, lane = threadIdx.x & 31;
    if (un >= nunit) return;
    const int64_t p = unit[un].x;
    int t = pairs[2 * p], s = pairs[2 * p + 1];
    if (obj_k) {
        const double2 ko = obj_k[M.obj[t]];
        kr = ko.x;
        ki = ko.y;
    }
    cd k = mk(kr, ki);
    int tt[3] = {M.T[3 * t], M.T[3 * t + 1], M.T[3 * t + 2]};
    int ss[3] = {M.T[3 * s], M.T[3 * s + 1], M.T[3 * s + 2]};
    v3 a = ld3(M.V + 3 * tt[0]), b = ld3(M.V + 3 * tt[1]), c = ld3(M.V + 3 * tt[2]);
    v3 a2 = ld3(M.V + 3 * ss[0]), b2 = ld3(M.V + 3 * ss[1]), c2 = ld3(M.V + 3 * ss[2]);
    v3 ct = ld3(M.cen + 3 * t);
    int shared[3], nsh = 0;
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++)
            if (tt[i] == ss[j]) shared[nsh++] = i;
    bool close = nsh > 0;
    if (!close) {
        v3 cs = ld3(M.cen + 3 * s);
        double D = nrm(ct - cs), Rt = M.rad[t], Rs = M.rad[s];
        if (D < cq.cf * (Rt + Rs) || hypot(kr, ki) * (Rt + Rs) > cq.kres) close = true;
    }
    // outer rule
    int kind;  // 0 plain collapsed, 1 edge shared, 2 vertex shared, 3 self
    int nout;
    v3 ap, bp, cp;
    if (t == s) {
        kind = 3;
        nout = 3 * graded_count(1);
    } else if (nsh == 2) {
        kind = 1;
        int ia = 3 - shared[0] - shared[1];
        v3 vt[3] = {a, b, c};
        ap = vt[ia];
        bp = vt[(ia + 1) % 3];
        cp = vt[(ia + 2) % 3];
        nout = graded_count(1);
    } else if (nsh == 1) {
        kind = 2;
        int ia = shared[0];
        v3 vt[3] = {a, b, c};
        ap = vt[ia];
        bp = vt[(ia + 1) % 3];
        cp = vt[(ia + 2) % 3];
        nout = graded_count(0);
    } else {
        kind = 0;
        int n = close ? cq.n[QR_OUT] : cq.n[QR_FAR];
        nout = n * n;
    }
    double twoA = nrm(cross(b - a, c - a));
    const int q_hi = min(nout, unit[un].y + 32);
    for (int qo = unit[un].y + lane; qo < q_hi; qo += 32) {
        v3 r;
        double w;
        if (kind == 0) {
            int ridx = close ? QR_OUT : QR_FAR;
            int n = cq.n[ridx];
            int i = qo / n, j = qo % n;
            double u = cq.x[ridx][i], v = cq.x[ridx][j] * (1.0 - u);
            r = a + u * (b - a) + v * (c - a);
            w = twoA * (1.0 - u) * cq.w[ridx][i] * cq.w[ridx][j];
        } else if (kind == 3) {
            int per = graded_count(1), sub = qo / per;
            v3 vt[3] = {a, b, c};
            graded_point(ct, vt[sub], vt[(sub + 1) % 3], 1, qo % per, r, w);
        } else {
            graded_point(ap, bp, cp, kind == 1, qo, r, w);
        }
        Inner in;
        if (close)
            pt::inner_polar(r, a2, b2, c2, k, in);
        else
            pt::inner_gauss(r, a2, b2, c2, k, in);
        v3 rt = r - ct;
        double rtv[3] = {rt.x, rt.y, rt.z};
        cd I2[3];
        for (int d = 0; d < 3; d++) I2[d] = in.Iv[d] + rtv[d] * in.Is;
        double* o = out + 32 * (int64_t)un + lane;
        auto put = [&](int n, cd v) { o[n * ld] = v.re, o[(n + 1) * ld] = v.im; };
        o[0] = w;
        for (int d = 0; d < 3; d++) o[(1 + d) * ld] = w * rtv[d];
        put(4, in.Is);
        for (int d = 0; d < 3; d++) put(6 + 2 * d, I2[d]);
        put(12, rtv[0] * I2[0] + rtv[1] * I2[1] + rtv[2] * I2[2]);
        if (t != s) {
            put(14, rtv[1] * in.Ig[2] - rtv[2] * in.Ig[1]);
            put(16, rtv[2] * in.Ig[0] - rtv[0] * in.Ig[2]);
            put(18, rtv[0] * in.Ig[1] - rtv[1] * in.Ig[0]);
            for (int d = 0; d < 3; d++) put(20 + 2 * d, in.Ig[d]);
        }
    }
}

// moments of the pairs own[i] = (pair, first unit, outer points): a warp per pair
__global__ void __launch_bounds__(128) k_near_gather(int n, const int3* __restrict__ own,
                                                     const int32_t* __restrict__ pairs, const double* __restrict__ pts,
                                                     int64_t ld, double2* __restrict__ mom)
{
    const int i = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32, lane = threadIdx.x & 31;
    if (i >= n) return;
    const int3 u = own[i];
    const bool self = pairs[2 * (int64_t)u.x] == pairs[2 * (int64_t)u.x + 1];
    cd acc[14];
    for (int k = 0; k < 14; k++) acc[k] = mk(0, 0);
    for (int q = lane; q < u.z; q += 32) {
        const double* o = pts + 32 * (int64_t)u.y + q;
        auto get = [&](int n) { return mk(o[n * ld], o[(n + 1) * ld]); };
        const double w = o[0];
        const cd Is = get(4);
        acc[0] = acc[0] + w * Is;
        for (int d = 0; d < 3; d++) {
            acc[1 + d] = acc[1 + d] + o[(1 + d) * ld] * Is;
            acc[4 + d] = acc[4 + d] + w * get(6 + 2 * d);
        }
        acc[7] = acc[7] + w * get(12);
        if (self) continue;
        for (int d = 0; d < 3; d++) {
            acc[8 + d] = acc[8 + d] + (-w) * get(14 + 2 * d);
            acc[11 + d] = acc[11 + d] + w * get(20 + 2 * d);
        }
    }
    store_moments(acc, lane, mom + 14 * (int64_t)u.x);
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
    // grid part: partial sums over the test nodes owned by this lane
    cd gLA[9], gK[9], g0 = mk(0, 0);
    for (int i = 0; i < 9; i++) gLA[i] = gK[i] = mk(0, 0);
    if (has_grid) {
        const int Mp = Mord + 1;
        int bt[3] = {base[3 * t], base[3 * t + 1], base[3 * t + 2]};
        int bs[3] = {base[3 * s], base[3 * s + 1], base[3 * s + 2]};
        const double* ct = M.coef + 3 * t;
        const double* cs = M.coef + 3 * s;
        const double* qt = M.q + 9 * t;
        const double* qs = M.q + 9 * s;
        const int Wd = 2 * Lm + 1;
        for (int u = lane; u < S; u += 32) {
            int ux = u % Mp, uy = (u / Mp) % Mp, uz = u / (Mp * Mp);
            const double* wu = Wt + ((size_t)t * S + u) * 4;
            double xt[3][3];  // test projection weights of slot i, component a
            for (int i = 0; i < 3; i++)
                for (int aa = 0; aa < 3; aa++) xt[i][aa] = ct[i] * (wu[1 + aa] + qt[3 * i + aa] * wu[0]);
            for (int v = 0; v < S; v++) {
                int vx = v % Mp, vy = (v / Mp) % Mp, vz = v / (Mp * Mp);
                int lx = bt[0] + ux - bs[0] - vx, ly = bt[1] + uy - bs[1] - vy, lz = bt[2] + uz - bs[2] - vz;
                const double2* kv = tab + 4 * (((lz + Lm) * Wd + (ly + Lm)) * Wd + (lx + Lm));
                cd G = mk(kv[0].x, kv[0].y), Dx = mk(kv[1].x, kv[1].y), Dy = mk(kv[2].x, kv[2].y),
                   Dz = mk(kv[3].x, kv[3].y);
                const double* wv = Wt + ((size_t)s * S + v) * 4;
                g0 = g0 + (wu[0] * wv[0]) * G;
                for (int j = 0; j < 3; j++) {
                    double xs[3];
                    for (int cc = 0; cc < 3; cc++) xs[cc] = cs[j] * (wv[1 + cc] + qs[3 * j + cc] * wv[0]);
                    for (int i = 0; i < 3; i++) {
                        double la = xt[i][0] * xs[0] + xt[i][1] * xs[1] + xt[i][2] * xs[2];
                        // sum_abc eps_abc xt_a D_b xs_c = D . (xs x xt)
                        double wx = xs[1] * xt[i][2] - xs[2] * xt[i][1];
                        double wy = xs[2] * xt[i][0] - xs[0] * xt[i][2];
                        double wz = xs[0] * xt[i][1] - xs[1] * xt[i][0];
                        gLA[3 * i + j] = gLA[3 * i + j] + la * G;
                        gK[3 * i + j] = gK[3 * i + j] + wx * Dx + wy * Dy + wz * Dz;
                    }
                }
            }
        }
        for (int off = 16; off > 0; off >>= 1) {
            for (int i = 0; i < 9; i++) {
                gLA[i].re += __shfl_down_sync(0xffffffffu, gLA[i].re, off);
                gLA[i].im += __shfl_down_sync(0xffffffffu, gLA[i].im, off);
                gK[i].re += __shfl_down_sync(0xffffffffu, gK[i].re, off);
                gK[i].im += __shfl_down_sync(0xffffffffu, gK[i].im, off);
            }
            g0.re += __shfl_down_sync(0xffffffffu, g0.re, off);
            g0.im += __shfl_down_sync(0xffffffffu, g0.im, off);
        }
    }
    if (lane != 0) return;
    // exact entries from the moments
    const double2* mm = mom + 14 * p;
    cd Q0 = mk(mm[0].x, mm[0].y);
    cd Q1[3], Q2[3], U[3], Vv[3];
    for (int d = 0; d < 3; d++) {
        Q1[d] = mk(mm[1 + d].x, mm[1 + d].y);
        Q2[d] = mk(mm[4 + d].x, mm[4 + d].y);
        U[d] = mk(mm[8 + d].x, mm[8 + d].y);
        Vv[d] = mk(mm[11 + d].x, mm[11 + d].y);
    }
    cd Q3 = mk(mm[7].x, mm[7].y);
    v3 ctc = ld3(M.cen + 3 * t);
    double At = M.area[t], As = M.area[s];
    double2* o = out + NLOC * p;
    for (int i = 0; i < 3; i++) {
        double cm = M.coef[3 * t + i];
        v3 pm = ld3(M.V + 3 * M.T[3 * t + i]) - ctc;
        for (int j = 0; j < 3; j++) {
            double cn = M.coef[3 * s + j];
            v3 pn = ld3(M.V + 3 * M.T[3 * s + j]) - ctc;
            cd la = Q3 - (pn.x * Q1[0] + pn.y * Q1[1] + pn.z * Q1[2]) - (pm.x * Q2[0] + pm.y * Q2[1] + pm.z * Q2[2]) +
                    dot(pm, pn) * Q0;
            v3 dl = pn - pm, cx = cross(pn, pm);
            cd kk = dl.x * U[0] + dl.y * U[1] + dl.z * U[2] + cx.x * Vv[0] + cx.y * Vv[1] + cx.z * Vv[2];
            la = (cm * cn) * la;
            o[19 + 3 * i + j] = make_double2(la.re, la.im);  // exact
            la = la - gLA[3 * i + j];
            kk = (cm * cn) * kk - gK[3 * i + j];
            o[3 * i + j] = make_double2(la.re, la.im);
            o[9 + 3 * i + j] = make_double2(kk.re, kk.im);
        }
    }
    cd lp = (1.0 / (At * As)) * (Q0 - g0);
    o[18] = make_double2(lp.re, lp.im);
    cd lpe = (1.0 / (At * As)) * Q0;
    o[28] = make_double2(lpe.re, lpe.im);  // exact
}

}  // namespace pt
}  // namespace sie

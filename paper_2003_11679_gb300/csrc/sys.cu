// GIBC system of Eq. (sys) on the GPU: the augmented exterior product
// [j k0 LA - (K_0 + Ix/2) Z', D^T Lphi B; F D, j k0 I] [H; c0 rho] with the AIM
// grid carrying all seven source grids at once (7 forward, 4 inverse FFTs),
// the interior impedance Z' = Z_i / eta0 of Eqs. (GIBCdef), (nest02), (nest2)
// applied by a nested Krylov solve, restarted flexible GMRES with FP64
// classical Gram-Schmidt (twice), plane-wave right-hand sides and the far
// field / RCS of the solution.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <complex>
#include <cstring>
#include <limits>
#include <vector>

#include "gridio.cuh"
#include "internal.h"
#include "resident.cuh"
#include "spmv.cuh"
#include "sysmul.cuh"

namespace sie {

using cplx = std::complex<double>;
static const double C0 = 299792458.0, MU0 = 4e-7 * M_PI, ETA0 = MU0 * C0;

// grid part of the system product with the fused z stage (default); SIE_FUSED_Z=0
// in the environment keeps separate forward-z, spectral-multiply and inverse-z
// launches (same arithmetic, for comparison)
static bool fused_z()
{
    static const bool on = [] {
        const char* e = getenv("SIE_FUSED_Z");
        return !(e && e[0] == '0');
    }();
    return on;
}

// ------------------------------------------------------------------ vector kernels
__global__ void k_axpby(int64_t n, double2 a, const double2* __restrict__ x, double2 b, double2* __restrict__ y)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double2 xv = x[i];
    double2 o = make_double2(a.x * xv.x - a.y * xv.y, a.x * xv.y + a.y * xv.x);
    if (b.x != 0.0 || b.y != 0.0) {  // y is not read when b = 0 (may be uninitialised)
        double2 yv = y[i];
        o.x += b.x * yv.x - b.y * yv.y;
        o.y += b.x * yv.y + b.y * yv.x;
    }
    y[i] = o;
}

// y[i] = x[i] / (s d[i]) (Jacobi) ; d == null -> y = x / s
__global__ void k_jacobi(int64_t n, const double2* __restrict__ x, const double2* __restrict__ d, double2 s,
                         double2* __restrict__ y)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double2 dv = d ? d[i] : make_double2(1.0, 0.0);
    double2 q = make_double2(s.x * dv.x - s.y * dv.y, s.x * dv.y + s.y * dv.x);
    double den = q.x * q.x + q.y * q.y;
    double2 xv = x[i];
    y[i] = make_double2((xv.x * q.x + xv.y * q.y) / den, (xv.y * q.x - xv.x * q.y) / den);
}

// out[j] = sum_k conj(V[j][k]) w[k] for j < nv: pass 1 writes one partial per
// (chunk, vector) block, pass 2 sums the partials of each vector in a fixed
// order (deterministic, and spread over the whole GPU for long vectors)
constexpr int MULTI_RHS = 8;    // right-hand sides per lockstep solve
constexpr int DOT_CHUNKS = 64;
constexpr int CGS_CHUNKS = 128;  // row chunks of the fused Gram-Schmidt kernels (at most RES_MAXCTA)
constexpr int CGS_TILE = 32;     // columns per shared-memory tile there
__global__ void __launch_bounds__(256) k_dots_part(int64_t n, const double2* __restrict__ V, int64_t ld,
                                                   const double2* __restrict__ w, double2* __restrict__ part)
{
    const int j = blockIdx.y, c = blockIdx.x;
    const double2* v = V + (int64_t)j * ld;
    const int64_t len = (n + DOT_CHUNKS - 1) / DOT_CHUNKS;
    const int64_t k0 = c * len, k1 = min(n, k0 + len);
    double sr = 0, si = 0;
    for (int64_t k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
        double2 a = v[k], b = w[k];
        sr += a.x * b.x + a.y * b.y;
        si += a.x * b.y - a.y * b.x;
    }
    for (int off = 16; off > 0; off >>= 1) {
        sr += __shfl_down_sync(0xffffffffu, sr, off);
        si += __shfl_down_sync(0xffffffffu, si, off);
    }
    __shared__ double rr[8], ri[8];
    if ((threadIdx.x & 31) == 0) {
        rr[threadIdx.x >> 5] = sr;
        ri[threadIdx.x >> 5] = si;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0, b = 0;
        for (int i = 0; i < 8; i++) {
            a += rr[i];
            b += ri[i];
        }
        part[(int64_t)j * DOT_CHUNKS + c] = make_double2(a, b);
    }
}

__global__ void k_dots_final(int nv, const double2* __restrict__ part, double2* __restrict__ out)
{
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nv) return;
    double a = 0, b = 0;
    for (int c = 0; c < DOT_CHUNKS; c++) {
        a += part[(int64_t)j * DOT_CHUNKS + c].x;
        b += part[(int64_t)j * DOT_CHUNKS + c].y;
    }
    out[j] = make_double2(a, b);
}

// w -= sum_j V[j] h[j]   (sgn = -1) or x += sum_j V[j] h[j] (sgn = +1)
__global__ void k_gemv(int64_t n, int nv, const double2* __restrict__ V, int64_t ld, const double2* __restrict__ h,
                       double sgn, double2* __restrict__ w)
{
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    double sr = 0, si = 0;
    for (int j = 0; j < nv; j++) {
        double2 a = V[(int64_t)j * ld + k], b = h[j];
        sr += a.x * b.x - a.y * b.y;
        si += a.x * b.y + a.y * b.x;
    }
    double2 o = w[k];
    w[k] = make_double2(o.x + sgn * sr, o.y + sgn * si);
}

static unsigned nb(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// out[0..nv) = V^H w using the partial buffer part (nv * DOT_CHUNKS)
static sie_status dots(cudaStream_t st, int64_t n, int nv, const double2* V, int64_t ld, const double2* w,
                       double2* part, double2* out)
{
    k_dots_part<<<dim3(DOT_CHUNKS, nv), 256, 0, st>>>(n, V, ld, w, part);
    k_dots_final<<<(nv + 127) / 128, 128, 0, st>>>(nv, part, out);
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}

static sie_status axpby(cudaStream_t st, int64_t n, cplx a, const double2* x, cplx b, double2* y)
{
    k_axpby<<<nb(n), 256, 0, st>>>(n, make_double2(a.real(), a.imag()), x, make_double2(b.real(), b.imag()), y);
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}

// ------------------------------------------------------------------ FGMRES
// Non-owning reference to an operator y = A x (a lambda that outlives the
// call it is passed to): unlike std::function it never allocates.
class Apply {
    const void* obj_ = nullptr;
    sie_status (*call_)(const void*, const double2*, double2*) = nullptr;

public:
    template <class F>
    Apply(const F& f)  // NOLINT: implicit from a named callable
        : obj_(&f), call_([](const void* o, const double2* x, double2* y) { return (*static_cast<const F*>(o))(x, y); })
    {
    }
    sie_status operator()(const double2* x, double2* y) const { return call_(obj_, x, y); }
};

sie_status KrylovWork::alloc(cudaStream_t st, int64_t n_, int m_)
{
    if (n_ == n && m_ == m) return SIE_OK;
    release(st);
    n = n_;
    m = m_;
    SIE_CUDA_TRY(cudaMallocAsync((void**)&V, sizeof(double2) * (m + 1) * n, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&Z, sizeof(double2) * m * n, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&w, sizeof(double2) * n, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&r, sizeof(double2) * n, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&h, sizeof(double2) * 4 * (m + 2), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&part, sizeof(double2) * DOT_CHUNKS * (m + 1), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&cgsp, sizeof(double2) * RES_MAXCTA * 2 * (m + 2), st));
    // Hessenberg (m+1) x m, rotations cs, sn, rhs g, solution y
    SIE_CUDA_TRY(cudaMallocAsync((void**)&Hd, sizeof(double2) * ((m + 1) * m + 2 * m + 2 * (m + 1)), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&sc, sizeof(double) * (8 + m + 1), st));
    SIE_CUDA_TRY(cudaMallocHost((void**)&resid_h, sizeof(double) * (m + 1)));
    ev.resize(m + 1);
    for (auto& e : ev) SIE_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    return SIE_OK;
}

void KrylovWork::release(cudaStream_t st)
{
    for (double2* p : {V, Z, w, h, r, part, cgsp, Hd})
        if (p) cudaFreeAsync(p, st);
    if (sc) cudaFreeAsync(sc, st);
    if (resid_h) {
        cudaStreamSynchronize(st);
        cudaFreeHost(resid_h);
    }
    for (auto& e : ev) cudaEventDestroy(e);
    ev.clear();
    V = Z = w = h = r = part = cgsp = Hd = nullptr;
    sc = nullptr;
    resid_h = nullptr;
    n = 0;
    m = 0;
}

// ------------------------------------------------------------------ device-side GMRES pieces
__device__ __forceinline__ double2 cm(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ double2 cj(double2 a) { return make_double2(a.x, -a.y); }

// sc layout: [0] |b|, [1] beta of the current cycle, [3 + j] relative residual after iteration j
// V0 = r / |r|; g = (|r|, 0, ...), dot2 = r^H r
__global__ void k_gm_start(int64_t n, const double2* __restrict__ r, const double2* __restrict__ dot2,
                           double2* __restrict__ V0, double2* __restrict__ g, int m, double* __restrict__ sc,
                           int set_bnorm)
{
    const double d2 = dot2[0].x;
    const double beta = d2 != d2 ? d2 : sqrt(fmax(d2, 0.0));  // a NaN norm stays NaN (reported by the host)
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        double s = beta > 0 ? 1.0 / beta : 0.0;
        V0[i] = make_double2(r[i].x * s, r[i].y * s);
    }
    if (i == 0) {
        for (int k = 0; k <= m; k++) g[k] = make_double2(0, 0);
        g[0] = make_double2(beta, 0);
        if (set_bnorm) sc[0] = beta;
        sc[1] = beta;
    }
}

// apply the previous rotations to column j, form rotation j (c real), update
// g; relative residual |g[j+1]| / |b| to sc[3 + j]  (one thread)
__device__ void gm_givens(int j, int m, double2* __restrict__ H, double2* __restrict__ cs, double2* __restrict__ sn,
                          double2* __restrict__ g, double* __restrict__ sc)
{
    for (int i = 0; i < j; i++) {
        double2 a = H[i * m + j], b = H[(i + 1) * m + j];
        double2 sb = cm(sn[i], b), ta = cm(cj(sn[i]), a);
        H[i * m + j] = make_double2(cs[i].x * a.x + sb.x, cs[i].x * a.y + sb.y);
        H[(i + 1) * m + j] = make_double2(cs[i].x * b.x - ta.x, cs[i].x * b.y - ta.y);
    }
    double2 a = H[j * m + j], b = H[(j + 1) * m + j];
    double aa = hypot(a.x, a.y), bb = hypot(b.x, b.y);
    double den = hypot(aa, bb);
    double2 c, s;
    if (aa == 0.0) {
        c = make_double2(0, 0);
        s = make_double2(1, 0);
    } else {
        c = make_double2(aa / den, 0);
        s = cm(make_double2(a.x / aa, a.y / aa), cj(b));
        s.x /= den;
        s.y /= den;
    }
    cs[j] = c;
    sn[j] = s;
    double2 sb = cm(s, b);
    H[j * m + j] = make_double2(c.x * a.x + sb.x, c.x * a.y + sb.y);
    H[(j + 1) * m + j] = make_double2(0, 0);
    double2 gj = g[j];
    double2 t = cm(cj(s), gj);
    g[j] = make_double2(c.x * gj.x, c.x * gj.y);
    g[j + 1] = make_double2(-t.x, -t.y);
    sc[3 + j] = (sc[0] > 0) ? hypot(g[j + 1].x, g[j + 1].y) / sc[0] : (sc[0] == sc[0] ? 0.0 : sc[0]);
}

// Fused classical Gram-Schmidt, two passes.  The rows are split into
// CGS_CHUNKS fixed chunks, one block each.  Every kernel first finishes, in a
// fixed order, the reduction of the per-chunk partial sums the previous kernel
// left, then updates its own rows and leaves the next partial sums: one
// launch per pass instead of separate dot, reduction and update launches, and
// the same rounding on every run.

__device__ __forceinline__ void cgs_rows(int64_t n, int64_t& k0, int64_t& k1)
{
    const int64_t len = (n + CGS_CHUNKS - 1) / CGS_CHUNKS;
    k0 = (int64_t)blockIdx.x * len;
    k1 = min(n, k0 + len);
}

// P[c * ldp + i] = sum over rows k of chunk c of conj(V_i[k]) w[k], i < nv
// (blockDim 256: 8 warps)
__device__ void cgs_partials(int64_t k0, int64_t k1, int nv, const double2* __restrict__ V, int64_t ld,
                             const double2* __restrict__ w, double2* __restrict__ P, int ldp)
{
    __shared__ double2 sm[8][CGS_TILE];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i0 = 0; i0 < nv; i0 += CGS_TILE) {
        const int ni = min(CGS_TILE, nv - i0);
        for (int t = 0; t < ni; t++) {
            const double2* v = V + (int64_t)(i0 + t) * ld;
            double sr = 0, si = 0;
            for (int64_t k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
                double2 a = v[k], b = w[k];
                sr += a.x * b.x + a.y * b.y;
                si += a.x * b.y - a.y * b.x;
            }
            for (int off = 16; off > 0; off >>= 1) {
                sr += __shfl_down_sync(0xffffffffu, sr, off);
                si += __shfl_down_sync(0xffffffffu, si, off);
            }
            if (lane == 0) sm[warp][t] = make_double2(sr, si);
        }
        __syncthreads();
        if ((int)threadIdx.x < ni) {
            double2 s = sm[0][threadIdx.x];
            for (int q = 1; q < 8; q++) {
                s.x += sm[q][threadIdx.x].x;
                s.y += sm[q][threadIdx.x].y;
            }
            P[(int64_t)blockIdx.x * ldp + i0 + threadIdx.x] = s;
        }
        __syncthreads();
    }
}

// Several right-hand sides in one launch (gridDim.y = R, panel Krylov solves):
// the pointers of right-hand side q = blockIdx.y are offset by q times these
// strides -- v: basis vectors, w: the vector being orthogonalised, p: partial
// sums, h: the two Gram-Schmidt coefficient columns, d: Hessenberg, rotations
// and g, s: scalars.  All zero for one right-hand side.
struct PanelStrides {
    int64_t v = 0, w = 0, p = 0, h = 0, d = 0, s = 0;
};

// pass 1: partial sums of V^H w
__global__ void __launch_bounds__(256) k_cgs_part(int64_t n, int nv, const double2* __restrict__ V, int64_t ld,
                                                  const double2* __restrict__ w, double2* __restrict__ P, int ldp,
                                                  PanelStrides ps = PanelStrides())
{
    const int64_t q = blockIdx.y;
    V += q * ps.v;
    w += q * ps.w;
    P += q * ps.p;
    int64_t k0, k1;
    cgs_rows(n, k0, k1);
    cgs_partials(k0, k1, nv, V, ld, w, P, ldp);
}

// h = sum_c Pin[c][:] (block 0 stores it in hout); w -= V h on this chunk's
// rows; then the partial sums of V^H w (last = 0) or of w^H w (last = 1)
__global__ void __launch_bounds__(256) k_cgs_update(int64_t n, int nv, const double2* __restrict__ V, int64_t ld,
                                                    const double2* __restrict__ Pin, int ldp,
                                                    double2* __restrict__ hout, double2* __restrict__ w,
                                                    double2* __restrict__ Pout, int last,
                                                    PanelStrides ps = PanelStrides())
{
    __shared__ double2 h[CGS_TILE];
    {
        const int64_t q = blockIdx.y;
        V += q * ps.v;
        Pin += q * ps.p;
        hout += q * ps.h;
        w += q * ps.w;
        Pout += q * ps.p;
    }
    int64_t k0, k1;
    cgs_rows(n, k0, k1);
    for (int i0 = 0; i0 < nv; i0 += CGS_TILE) {
        const int ni = min(CGS_TILE, nv - i0);
        // one warp per column: lanes take every 32nd chunk, then a fixed xor tree
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        for (int t = warp; t < ni; t += 8) {
            double sr = 0, si = 0;
            for (int c = lane; c < CGS_CHUNKS; c += 32) {
                double2 p = Pin[(int64_t)c * ldp + i0 + t];
                sr += p.x;
                si += p.y;
            }
            for (int off = 16; off > 0; off >>= 1) {
                sr += __shfl_xor_sync(0xffffffffu, sr, off);
                si += __shfl_xor_sync(0xffffffffu, si, off);
            }
            if (lane == 0) {
                h[t] = make_double2(sr, si);
                if (blockIdx.x == 0) hout[i0 + t] = h[t];
            }
        }
        __syncthreads();
        for (int64_t k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
            double sr = 0, si = 0;
            for (int t = 0; t < ni; t++) {
                double2 a = V[(int64_t)(i0 + t) * ld + k], b = h[t];
                sr += a.x * b.x - a.y * b.y;
                si += a.x * b.y + a.y * b.x;
            }
            double2 o = w[k];
            w[k] = make_double2(o.x - sr, o.y - si);
        }
        __syncthreads();
    }
    if (last)
        cgs_partials(k0, k1, 1, w, 0, w, Pout, 1);
    else
        cgs_partials(k0, k1, nv, V, ld, w, Pout, ldp);
}

// |w| = sqrt(sum_c P[c]); V_{j+1} = w / |w| on this chunk's rows; block 0
// writes column j of H (h1 + h2 and |w|) and applies the Givens step
// (V: the basis, column stride ld (0: n); res, when given: the relative residual
// also to res[j gridDim.y + q])
__global__ void __launch_bounds__(256) k_cgs_finish(int64_t n, int j, int m, const double2* __restrict__ h1,
                                                    const double2* __restrict__ h2, const double2* __restrict__ P,
                                                    const double2* __restrict__ w, double2* __restrict__ V,
                                                    double2* __restrict__ H, double2* __restrict__ cs,
                                                    double2* __restrict__ sn, double2* __restrict__ g,
                                                    double* __restrict__ sc, PanelStrides ps = PanelStrides(), int64_t ld = 0,
                                                    double* __restrict__ res = nullptr)
{
    const int64_t q = blockIdx.y;
    h1 += q * ps.h;
    h2 += q * ps.h;
    P += q * ps.p;
    w += q * ps.w;
    V += q * ps.v;
    H += q * ps.d;
    cs += q * ps.d;
    sn += q * ps.d;
    g += q * ps.d;
    sc += q * ps.s;
    if (ld == 0) ld = n;
    double2* Vn = V + (int64_t)(j + 1) * ld;
    __shared__ double hn_s;
    if (threadIdx.x < 32) {
        double s = 0;
        for (int c = threadIdx.x; c < CGS_CHUNKS; c += 32) s += P[c].x;
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (threadIdx.x == 0) hn_s = sqrt(fmax(s, 0.0));
    }
    __syncthreads();
    const double hn = hn_s;
    const double inv = hn > 0 ? 1.0 / hn : 0.0;
    int64_t k0, k1;
    cgs_rows(n, k0, k1);
    for (int64_t k = k0 + threadIdx.x; k < k1; k += blockDim.x) Vn[k] = make_double2(w[k].x * inv, w[k].y * inv);
    if (blockIdx.x != 0) return;
    for (int i = threadIdx.x; i <= j; i += blockDim.x) H[i * m + j] = make_double2(h1[i].x + h2[i].x, h1[i].y + h2[i].y);
    if (threadIdx.x == 0) H[(j + 1) * m + j] = make_double2(hn, 0);
    __syncthreads();
    if (threadIdx.x == 0) {
        gm_givens(j, m, H, cs, sn, g, sc);
        if (res) res[(int64_t)j * gridDim.y + q] = sc[3 + j];
    }
}

// y = R^-1 g (upper triangular, size jend + 1)
__global__ void k_gm_backsub(int jend, int m, const double2* __restrict__ H, const double2* __restrict__ g,
                             double2* __restrict__ y)
{
    for (int i = jend; i >= 0; i--) {
        double2 s = g[i];
        for (int k = i + 1; k <= jend; k++) {
            double2 t = cm(H[i * m + k], y[k]);
            s.x -= t.x;
            s.y -= t.y;
        }
        double2 d = H[i * m + i];
        double den = d.x * d.x + d.y * d.y;
        y[i] = den > 0 ? make_double2((s.x * d.x + s.y * d.y) / den, (s.y * d.x - s.x * d.y) / den)
                       : make_double2(0, 0);
    }
}

// Right-preconditioned restarted flexible GMRES, zero initial guess; the
// monitored residual is the true residual of A x = b.  Arnoldi in FP64 with
// classical Gram-Schmidt applied twice.  Everything stays on the device: the
// Hessenberg column, the Givens rotations and the back substitution are tiny
// kernels; the host reads each iteration's residual `lag` iterations later
// (event on a pinned copy; lag 1 by default), so the GPU does not wait on
// host round trips.  Then one extra iteration may run after convergence (it
// only lowers the residual); short inner solves use lag 0 instead.
static sie_status fgmres(sie_ctx* c, KrylovWork& K, int64_t n, const Apply& A, const Apply& Minv, const double2* b,
                         double2* x, double tol, int maxit, int restart, int* iters_out, double* relres_out,
                         int lag = 1)
{
    cudaStream_t st = c->stream;
    SIE_TRY(K.alloc(st, n, restart));
    const int m = restart;
    double2* H = K.Hd;
    double2* cs = K.Hd + (m + 1) * m;
    double2* sn = cs + m;
    double2* g = sn + m;
    double2* y = g + (m + 1);
    double2* h1 = K.h;
    double2* h2 = K.h + (m + 2);
    double2* wd = K.h + 2 * (m + 2);
    // x0 = 0, r0 = b.  No host round trip here: a zero b gives zero residuals
    // (sc[3 + j] = 0), so the first convergence check stops with x = 0.
    SIE_CUDA_TRY(cudaMemsetAsync(x, 0, sizeof(double2) * n, st));
    SIE_TRY(dots(st, n, 1, b, n, b, K.part, wd));
    k_gm_start<<<nb(n), 256, 0, st>>>(n, b, wd, K.V, g, m, K.sc, 1);
    SIE_CUDA_TRY(cudaGetLastError());
    int it = 0;
    double rel = 1.0;
    const int LAG = lag;
    while (true) {
        int j = 0;
        bool conv = false;
        for (; j < m && it < maxit; j++) {
            double2* Vj = K.V + (int64_t)j * n;
            double2* Zj = K.Z + (int64_t)j * n;
            SIE_TRY(Minv(Vj, Zj));
            SIE_TRY(A(Zj, K.w));
            // CGS2: V^H w, w -= V h1, V^H w, w -= V h2, |w|, V_{j+1}, Givens
            double2* P1 = K.cgsp;
            double2* P2 = K.cgsp + (int64_t)CGS_CHUNKS * (m + 1);
            double2* P3 = K.cgsp + (int64_t)2 * CGS_CHUNKS * (m + 1);
            k_cgs_part<<<CGS_CHUNKS, 256, 0, st>>>(n, j + 1, K.V, n, K.w, P1, m + 1);
            k_cgs_update<<<CGS_CHUNKS, 256, 0, st>>>(n, j + 1, K.V, n, P1, m + 1, h1, K.w, P2, 0);
            k_cgs_update<<<CGS_CHUNKS, 256, 0, st>>>(n, j + 1, K.V, n, P2, m + 1, h2, K.w, P3, 1);
            k_cgs_finish<<<CGS_CHUNKS, 256, 0, st>>>(n, j, m, h1, h2, P3, K.w, K.V, H, cs, sn, g, K.sc);
            SIE_CUDA_TRY(cudaGetLastError());
            SIE_CUDA_TRY(cudaMemcpyAsync(K.resid_h + j, K.sc + 3 + j, sizeof(double), cudaMemcpyDeviceToHost, st));
            SIE_CUDA_TRY(cudaEventRecord(K.ev[j], st));
            it++;
            if (j >= LAG) {
                SIE_CUDA_TRY(cudaEventSynchronize(K.ev[j - LAG]));
                if (!std::isfinite(K.resid_h[j - LAG])) {
                    set_error("GMRES: the residual is not finite (non-finite right-hand side or operator)");
                    return SIE_ERR_ARG;
                }
                if (K.resid_h[j - LAG] < tol) {
                    conv = true;
                    j++;
                    break;
                }
            }
        }
        const int jend = j - 1;
        SIE_CUDA_TRY(cudaEventSynchronize(K.ev[jend]));
        rel = K.resid_h[jend];
        if (!std::isfinite(rel)) {
            set_error("GMRES: the residual is not finite (non-finite right-hand side or operator)");
            return SIE_ERR_ARG;
        }
        if (rel < tol) conv = true;
        k_gm_backsub<<<1, 1, 0, st>>>(jend, m, H, g, y);
        k_gemv<<<nb(n), 256, 0, st>>>(n, jend + 1, K.Z, n, y, 1.0, x);
        SIE_CUDA_TRY(cudaGetLastError());
        if (conv || it >= maxit) break;
        // restart from the true residual
        SIE_TRY(A(x, K.w));
        SIE_CUDA_TRY(cudaMemcpyAsync(K.r, b, sizeof(double2) * n, cudaMemcpyDeviceToDevice, st));
        SIE_TRY(axpby(st, n, -1.0, K.w, 1.0, K.r));
        SIE_TRY(dots(st, n, 1, K.r, n, K.r, K.part, wd));
        k_gm_start<<<nb(n), 256, 0, st>>>(n, K.r, wd, K.V, g, m, K.sc, 0);
        SIE_CUDA_TRY(cudaGetLastError());
        SIE_CUDA_TRY(cudaMemcpyAsync(K.resid_h, K.sc, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
        SIE_CUDA_TRY(cudaStreamSynchronize(st));
        rel = K.resid_h[0] > 0 ? K.resid_h[1] / K.resid_h[0] : 0.0;
        if (rel < tol) break;
    }
    if (iters_out) *iters_out = it;
    if (relres_out) *relres_out = rel;
    return rel < tol ? SIE_OK : SIE_ERR_NOT_CONVERGED;
}

// ------------------------------------------------------------------ system kernels
__global__ void k_specmul_sys32(const float2* __restrict__ spec, float2* __restrict__ buf, int64_t nn, float k0)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nn) return;
    float2 in[7], out[4];
    for (int g = 0; g < 7; g++) in[g] = buf[g * nn + i];
    sys_specmul(spec[i], spec[nn + i], spec[2 * nn + i], spec[3 * nn + i], k0, in, out);
    for (int g = 0; g < 4; g++) buf[g * nn + i] = out[g];
}

// A_a = j k0 G J_a - (Ggrad x M)_a into grids 0..2, Phi = G rho into grid 3
__global__ void k_specmul_sys(const double2* __restrict__ spec, double2* __restrict__ buf, int64_t nn, double k0)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nn) return;
    double2 in[7], out[4];
    for (int g = 0; g < 7; g++) in[g] = buf[g * nn + i];
    sys_specmul(spec[i], spec[nn + i], spec[2 * nn + i], spec[3 * nn + i], k0, in, out);
    for (int g = 0; g < 4; g++) buf[g * nn + i] = out[g];
}

// complex64 copies of H and E side by side for the mixed near product: one
// 16-byte gather per stored entry instead of two 16-byte gathers and four
// FP64 -> FP32 conversions (those run on the FP64 pipe)
__global__ void k_pack_he32(int n, const double2* __restrict__ H, const double2* __restrict__ E,
                            float4* __restrict__ out)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double2 h = H[i], e = E[i];
    out[i] = make_float4((float)h.x, (float)h.y, (float)e.x, (float)e.y);
}

// k_spmv2 of the mixed path: the two matrices' complex64 values interleaved
// (v[e] = (LA, K) of entry e: one 16-byte load), x packed by k_pack_he32;
// FP32 products and per-lane sums, the lane sums combined in FP64
__global__ void __launch_bounds__(128) k_spmv2_c64(int nrow, const int64_t* __restrict__ rp,
                                                   const int32_t* __restrict__ col, const float4* __restrict__ v,
                                                   const float4* __restrict__ x, double2 a1, double2 a2,
                                                   double2* __restrict__ y)
{
    int r = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    int lane = threadIdx.x & 31;
    if (r >= nrow) return;
    float s1r = 0, s1i = 0, s2r = 0, s2i = 0;
    const int64_t e0 = rp[r], e1 = rp[r + 1];
    int64_t e = e0 + lane;
    for (; e + 96 < e1; e += 128) {
        int c[4];
        float4 p[4], q[4];
#pragma unroll
        for (int u = 0; u < 4; u++) c[u] = __ldg(col + e + 32 * u);
#pragma unroll
        for (int u = 0; u < 4; u++) p[u] = __ldg(v + e + 32 * u);
#pragma unroll
        for (int u = 0; u < 4; u++) q[u] = __ldg(x + c[u]);
#pragma unroll
        for (int u = 0; u < 4; u++) {
            s1r += p[u].x * q[u].x - p[u].y * q[u].y;
            s1i += p[u].x * q[u].y + p[u].y * q[u].x;
            s2r += p[u].z * q[u].z - p[u].w * q[u].w;
            s2i += p[u].z * q[u].w + p[u].w * q[u].z;
        }
    }
    for (; e < e1; e += 32) {
        float4 p = __ldg(v + e), q = __ldg(x + __ldg(col + e));
        s1r += p.x * q.x - p.y * q.y;
        s1i += p.x * q.y + p.y * q.x;
        s2r += p.z * q.z - p.w * q.w;
        s2i += p.z * q.w + p.w * q.z;
    }
    double t1r = s1r, t1i = s1i, t2r = s2r, t2i = s2i;
    for (int off = 16; off > 0; off >>= 1) {
        t1r += __shfl_down_sync(0xffffffffu, t1r, off);
        t1i += __shfl_down_sync(0xffffffffu, t1i, off);
        t2r += __shfl_down_sync(0xffffffffu, t2r, off);
        t2i += __shfl_down_sync(0xffffffffu, t2i, off);
    }
    if (lane == 0) {
        y[r].x += a1.x * t1r - a1.y * t1i + a2.x * t2r - a2.y * t2i;
        y[r].y += a1.x * t1i + a1.y * t1r + a2.x * t2i + a2.y * t2r;
    }
}

// y[r] += a1 sum_e v1[e] x1[col[e]] + a2 sum_e v2[e] x2[col[e]]: the two
// near-region matrices of one operator share their pattern, so the column
// indices are read once.  G lanes per row, four loads of each array in flight per
// lane.  FP64 arithmetic bounds large meshes: with 8 lanes the warp-wide additions of
// a row's sums are shared by four rows (15.0 M entries, 190 us of products: 453 us
// with 32 lanes, 274 us with 8).  Up to 8,192 rows the GPU is not full and a row's
// chain counts: with 32 and 8 lanes 11 and 23 us at 480 rows, 28 and 33 at 3,456, 40 and
// 39 at 7,680, 130 and 109 at 30,720 (4.8 M entries).
template <int G>
__global__ void __launch_bounds__(256) k_spmv2(int nrow, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                               const double2* __restrict__ v1, const double2* __restrict__ x1, double2 a1,
                                               const double2* __restrict__ v2, const double2* __restrict__ x2, double2 a2,
                                               double2* __restrict__ y)
{
    constexpr int U = 4;
    const int r = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / G), l = threadIdx.x % G;
    const bool ok = r < nrow;
    const int64_t e1 = ok ? rp[r + 1] : 0;
    int64_t e = ok ? rp[r] + l : 0;
    double s1r[2] = {0, 0}, s1i[2] = {0, 0}, s2r[2] = {0, 0}, s2i[2] = {0, 0};  // two chains each
    for (; e + (U - 1) * G < e1; e += U * G) {
        int c[U];
        double2 p[U], q[U], xa[U], xb[U];
#pragma unroll
        for (int u = 0; u < U; u++) c[u] = __ldg(col + e + u * G);
#pragma unroll
        for (int u = 0; u < U; u++) {
            p[u] = __ldg(v1 + e + u * G);
            q[u] = __ldg(v2 + e + u * G);
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            xa[u] = __ldg(x1 + c[u]);
            xb[u] = __ldg(x2 + c[u]);
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            s1r[u & 1] = fma(p[u].x, xa[u].x, fma(-p[u].y, xa[u].y, s1r[u & 1]));
            s1i[u & 1] = fma(p[u].x, xa[u].y, fma(p[u].y, xa[u].x, s1i[u & 1]));
            s2r[u & 1] = fma(q[u].x, xb[u].x, fma(-q[u].y, xb[u].y, s2r[u & 1]));
            s2i[u & 1] = fma(q[u].x, xb[u].y, fma(q[u].y, xb[u].x, s2i[u & 1]));
        }
    }
    for (; e < e1; e += G) {  // at most 3 more entries per lane
        const int c = __ldg(col + e);
        const double2 p = __ldg(v1 + e), q = __ldg(v2 + e), xa = __ldg(x1 + c), xb = __ldg(x2 + c);
        s1r[0] = fma(p.x, xa.x, fma(-p.y, xa.y, s1r[0]));
        s1i[0] = fma(p.x, xa.y, fma(p.y, xa.x, s1i[0]));
        s2r[0] = fma(q.x, xb.x, fma(-q.y, xb.y, s2r[0]));
        s2i[0] = fma(q.x, xb.y, fma(q.y, xb.x, s2i[0]));
    }
    double t1r = s1r[0] + s1r[1], t1i = s1i[0] + s1i[1], t2r = s2r[0] + s2r[1], t2i = s2i[0] + s2i[1];
    // a1 t1 + a2 t2 first: two sums to reduce instead of four
    double tr = a1.x * t1r - a1.y * t1i + a2.x * t2r - a2.y * t2i;
    double ti = a1.x * t1i + a1.y * t1r + a2.x * t2i + a2.y * t2r;
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) {
        tr += __shfl_xor_sync(0xffffffffu, tr, off);
        ti += __shfl_xor_sync(0xffffffffu, ti, off);
    }
    if (ok && l == 0) {
        y[r].x += tr;
        y[r].y += ti;
    }
}

// y += alpha A x (acc) or y = alpha A x for a CSR matrix with nnz entries
static sie_status spmv(cudaStream_t st, int nrow, int64_t nnz, const int64_t* rp, const int32_t* col,
                       const double2* val, const double2* x, cplx alpha, double2* y, bool acc = true)
{
    SIE_CUDA_TRY(csr_launch(st, nrow, nnz, rp, col, val, x, make_double2(alpha.real(), alpha.imag()), acc, y));
    return SIE_OK;
}

static int64_t tri_nnz(const AimOp& a) { return a.tri_row_ptr_h.empty() ? 0 : a.tri_row_ptr_h.back(); }

// E[m] *= f[m] (per-edge interior impedance factor of several objects)
__global__ void k_scale_edges(int64_t n, const double2* __restrict__ f, double2* __restrict__ E)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double2 a = f[i], b = E[i];
    E[i] = make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// sigma_t = -A_t c0rho_t
__global__ void k_sigma(int nt, const double* __restrict__ area, const double2* __restrict__ rho,
                        double2* __restrict__ sig)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nt) sig[t] = make_double2(-area[t] * rho[t].x, -area[t] * rho[t].y);
}

__global__ void k_sigma32(int nt, const double* __restrict__ area, const double2* __restrict__ rho,
                          float2* __restrict__ sig)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nt) sig[t] = make_float2((float)(-area[t] * rho[t].x), (float)(-area[t] * rho[t].y));
}

__global__ void k_fdiv_area(int nt, const double* __restrict__ area, double2* __restrict__ x)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nt) x[t] = make_double2(x[t].x / area[t], x[t].y / area[t]);
}

// y1_m += l_m (phi_{T+} - phi_{T-}) = (D^T phi)_m
__global__ void k_dt(int ne, const int32_t* __restrict__ edge_tri, const double* __restrict__ len,
                     const double2* __restrict__ phi, double2* __restrict__ y)
{
    int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= ne) return;
    double2 a = phi[edge_tri[2 * m]], b = phi[edge_tri[2 * m + 1]];
    y[m].x += len[m] * (a.x - b.x);
    y[m].y += len[m] * (a.y - b.y);
}

// q_t = (D y)_t / A_t * scaleA  -> with scaleA = A_t gives (D y)_t; here
// (D y)_t = sum_i s_i l_i y_e = 2 A_t sum_i c_{t,i} y_{e(t,i)}
__global__ void k_D(int nt, DevMesh M, const double2* __restrict__ y, double2* __restrict__ q)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    double sr = 0, si = 0;
    for (int i = 0; i < 3; i++) {
        double2 v = y[M.tri_edge[3 * t + i]];
        double c = 2.0 * M.coef[3 * t + i] * M.area[t];
        sr += c * v.x;
        si += c * v.y;
    }
    q[t] = make_double2(sr, si);
}

// row 2: y2_t = (F D H)_t + j k0 c0rho_t = 2 sum_i c_{t,i} H_{e(t,i)} + j k0 c0rho_t
__global__ void k_row2(int nt, DevMesh M, const double2* __restrict__ H, const double2* __restrict__ rho, double k0,
                       double2* __restrict__ y2)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    double sr = 0, si = 0;
    for (int i = 0; i < 3; i++) {
        double2 h = H[M.tri_edge[3 * t + i]];
        double c = 2.0 * M.coef[3 * t + i];
        sr += c * h.x;
        si += c * h.y;
    }
    double2 r = rho[t];
    y2[t] = make_double2(sr - k0 * r.y, si + k0 * r.x);
}

// plane-wave right-hand side b_m = -(1/eta0) I f_m . e exp(-j k0 khat . r)
struct GL8 {
    double x[16], w[16];
    int n;
};

__global__ void k_rhs(int nt, DevMesh M, GL8 q, double k0, double3 kh, double3 ep, double scale,
                      double2* __restrict__ b)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    const double* a = M.V + 3 * M.T[3 * t];
    const double* bb = M.V + 3 * M.T[3 * t + 1];
    const double* c = M.V + 3 * M.T[3 * t + 2];
    double e1[3], e2[3];
    for (int d = 0; d < 3; d++) {
        e1[d] = bb[d] - a[d];
        e2[d] = c[d] - a[d];
    }
    double nx = e1[1] * e2[2] - e1[2] * e2[1], ny = e1[2] * e2[0] - e1[0] * e2[2], nz = e1[0] * e2[1] - e1[1] * e2[0];
    double twoA = sqrt(nx * nx + ny * ny + nz * nz);
    double accr[3] = {0, 0, 0}, acci[3] = {0, 0, 0};
    for (int i = 0; i < q.n; i++) {
        double u = q.x[i];
        for (int j = 0; j < q.n; j++) {
            double v = q.x[j] * (1.0 - u);
            double w = twoA * (1.0 - u) * q.w[i] * q.w[j];
            double r[3];
            for (int d = 0; d < 3; d++) r[d] = a[d] + u * e1[d] + v * e2[d];
            double ph = -k0 * (kh.x * r[0] + kh.y * r[1] + kh.z * r[2]);
            double s, cc;
            sincos(ph, &s, &cc);
            for (int sl = 0; sl < 3; sl++) {
                const double* p = M.V + 3 * M.T[3 * t + sl];
                double f = M.coef[3 * t + sl] * ((r[0] - p[0]) * ep.x + (r[1] - p[1]) * ep.y + (r[2] - p[2]) * ep.z);
                accr[sl] += w * f * cc;
                acci[sl] += w * f * s;
            }
        }
    }
    for (int sl = 0; sl < 3; sl++) {
        double2* d = b + M.tri_edge[3 * t + sl];
        atomicAdd(&d->x, scale * accr[sl]);
        atomicAdd(&d->y, scale * acci[sl]);
    }
}

// far-field sums N(X)_a = sum_n X_n I f_n,a exp(j k0 rhat . r) for X = H, E';
// one block per direction, fixed-order tree reduction; out: 6 complex per dir
__global__ void __launch_bounds__(256) k_far(int nt, DevMesh M, GL8 q, double k0, const double* __restrict__ rhat,
                                             const double2* __restrict__ H, const double2* __restrict__ E,
                                             double2* __restrict__ out)
{
    int d = blockIdx.x;
    double rx = rhat[3 * d], ry = rhat[3 * d + 1], rz = rhat[3 * d + 2];
    double acc[12];
    for (int i = 0; i < 12; i++) acc[i] = 0;
    for (int t = threadIdx.x; t < nt; t += blockDim.x) {
        const double* a = M.V + 3 * M.T[3 * t];
        const double* bb = M.V + 3 * M.T[3 * t + 1];
        const double* c = M.V + 3 * M.T[3 * t + 2];
        double e1[3], e2[3];
        for (int k = 0; k < 3; k++) {
            e1[k] = bb[k] - a[k];
            e2[k] = c[k] - a[k];
        }
        double nx = e1[1] * e2[2] - e1[2] * e2[1], ny = e1[2] * e2[0] - e1[0] * e2[2],
               nz = e1[0] * e2[1] - e1[1] * e2[0];
        double twoA = sqrt(nx * nx + ny * ny + nz * nz);
        for (int i = 0; i < q.n; i++) {
            double u = q.x[i];
            for (int j = 0; j < q.n; j++) {
                double v = q.x[j] * (1.0 - u);
                double w = twoA * (1.0 - u) * q.w[i] * q.w[j];
                double r[3];
                for (int k = 0; k < 3; k++) r[k] = a[k] + u * e1[k] + v * e2[k];
                double s, cc;
                sincos(k0 * (rx * r[0] + ry * r[1] + rz * r[2]), &s, &cc);
                for (int sl = 0; sl < 3; sl++) {
                    const double* p = M.V + 3 * M.T[3 * t + sl];
                    int e = M.tri_edge[3 * t + sl];
                    double cf = w * M.coef[3 * t + sl];
                    double2 h = H[e], ev = E[e];
                    for (int k = 0; k < 3; k++) {
                        double f = cf * (r[k] - p[k]);
                        // x * exp(j phase)
                        acc[2 * k] += f * (h.x * cc - h.y * s);
                        acc[2 * k + 1] += f * (h.x * s + h.y * cc);
                        acc[6 + 2 * k] += f * (ev.x * cc - ev.y * s);
                        acc[6 + 2 * k + 1] += f * (ev.x * s + ev.y * cc);
                    }
                }
            }
        }
    }
    __shared__ double red[256];
    for (int i = 0; i < 12; i++) {
        red[threadIdx.x] = acc[i];
        __syncthreads();
        for (int s = 128; s > 0; s >>= 1) {
            if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
            __syncthreads();
        }
        if (threadIdx.x == 0) ((double*)(out + 6 * d))[i] = red[0];
        __syncthreads();
    }
}

static GL8 gl_rule(int n)
{
    GL8 q;
    q.n = n;
    gauss_legendre01(n, q.x, q.w);
    return q;
}

// ------------------------------------------------------------------ operators
static sie_status constraint_solve(sie_op* op, AimOp& a, cplx kappa, KrylovWork& K, double tol, const double2* v,
                                   double2* y);

// Krylov basis of the nested solve: it runs without restart, in and outside a graph
constexpr int INNER_BASIS_MAX = 128;
static int inner_m(const sie_op* op) { return std::max(1, std::min(op->p.inner_maxit, INNER_BASIS_MAX)); }

// E' = Z' H of a near-region-only or SIBC interior: one grid-resident kernel
// (nested.cu).  Outside a capture the call waits for its result: a residual that
// is not finite is an error, as in fgmres.  nested_res: the residual it ended with.
static sie_status apply_Z_resident(sie_op* op, const double2* H, double2* E, double* nested_res)
{
    sie_ctx* c = op->mesh->ctx;
    const int64_t ne = op->mesh->h.ne;
    cplx f;
    if (op->p.interior_model == SIE_SIBC) {
        f = cplx(op->eta_re, op->eta_im);
    } else {
        f = -1.0 / cplx(op->sigma * ETA0, op->k0 * op->eps_r);
    }
    KrylovWork& K = op->kin;
    SIE_TRY(K.alloc(c->stream, ne, inner_m(op)));
    ResWork w;
    w.m = K.m, w.V = K.V, w.Z = K.Z, w.W = K.w, w.H = K.Hd, w.part = K.cgsp;
    {
        Stage s_(c, "inner_solve");
        // one iteration past the tolerance outside the graph, as fgmres with its lagged check
        SIE_TRY(nested_solve(op, H, E, make_double2(f.real(), f.imag()), op->capturing ? 0 : 1, w));
    }
    if (op->capturing) return SIE_OK;
    SIE_TRY(sys_stats_fold(op));
    if (op->wait_lost) {
        SIE_TRY(nested_clear(op));
        set_error("nested interior solve: a grid barrier's wait ran out");
        return SIE_ERR_TIMEOUT;
    }
    const double rr = op->last_nested;
    if (!std::isfinite(rr)) {
        set_error("GMRES: the residual is not finite (non-finite right-hand side or operator)");
        return SIE_ERR_ARG;
    }
    if (nested_res) *nested_res = rr;
    return SIE_OK;
}

// interior impedance E' = Z' H = -(j k0 eps_r + sigma eta0)^-1 L_i^-1 (K_i - Ix/2) H,
// or (eta_i / eta0) G^-1 Ix H (SIBC)
// nested_res (not inside a capture): relative residual the nested solve ended with
static sie_status apply_Z(sie_op* op, const double2* H, double2* E, double* nested_res)
{
    if (!op->inn.has_grid) return apply_Z_resident(op, H, E, nested_res);
    sie_ctx* c = op->mesh->ctx;
    cudaStream_t st = c->stream;
    const int64_t ne = op->mesh->h.ne;
    double2* a = op->sys_tmp;  // ne
    SIE_TRY(aim_apply(op, op->inn, 1, H, a));
    SIE_TRY(spmv(st, (int)ne, op->ix_nnz, op->ix_row_ptr, op->ix_col, op->ix_val, H, cplx(-0.5, 0), a));
    AimOp& I = op->inn;
    auto A = [&](const double2* x, double2* y) { return aim_apply(op, I, 0, x, y); };
    cplx ki(I.kr, I.ki);
    // Nested preconditioner M_i of Eq. (nest2pc) in its near-region form: the
    // constraint form (diag LA_i + near Lphi_i, block elimination)
    auto Minv = [&](const double2* x, double2* y) {
        return constraint_solve(op, I, 1.0 / (ki * ki), op->kcs_in, op->p.tol_constraint_inner, x, y);
    };
    // one unrestarted cycle of at most min(inner_maxit, INNER_BASIS_MAX) iterations
    const int m_in = inner_m(op);
    if (nested_res) *nested_res = 0.0;
    int it = 0;
    double rr = 0;
    sie_status s;
    {
        Stage s_(c, "inner_solve");
        s = fgmres(c, op->kin, ne, A, Minv, a, E, op->p.tol_inner, m_in, m_in, &it, &rr);
    }
    if (s != SIE_OK && s != SIE_ERR_NOT_CONVERGED) return s;
    if (nested_res) *nested_res = rr;
    op->stats[2] = std::max(op->stats[2], (double)it);
    op->stats[3] = std::max(op->stats[3], rr);
    cplx zs(0.0, op->k0 * op->eps_r);
    zs += op->sigma * ETA0;
    SIE_TRY(axpby(st, ne, -1.0 / zs, E, 0.0, E));
    return SIE_OK;
}

// node -> stencil entries map of the exterior grid, entries of a node by triangle
// (built once, on the host, from the stencil bases, by the operator build)
sie_status proj_map_ready(sie_op* op)
{
    if (op->pm_ptr) return SIE_OK;
    cudaStream_t st = op->mesh->ctx->stream;
    const GridDesc& g = op->ext.g;
    const int Mp = g.M + 1, S = Mp * Mp * Mp;
    const int64_t nt = op->mesh->h.nt, Ng = (int64_t)g.N[0] * g.N[1] * g.N[2];
    if (nt * S > INT32_MAX || Ng > INT32_MAX) {
        set_error("projection map: more than 2^31 stencil entries or grid nodes");
        return SIE_ERR_UNSUPPORTED;
    }
    std::vector<int32_t> hb(3 * nt);
    SIE_CUDA_TRY(cudaMemcpyAsync(hb.data(), op->base, sizeof(int32_t) * 3 * nt, cudaMemcpyDeviceToHost, st));
    SIE_CUDA_TRY(cudaStreamSynchronize(st));
    auto node = [&](int64_t t, int u) {
        const int nx = hb[3 * t] + u % Mp, ny = hb[3 * t + 1] + (u / Mp) % Mp, nz = hb[3 * t + 2] + u / (Mp * Mp);
        return ((int64_t)nz * g.N[1] + ny) * g.N[0] + nx;
    };
    std::vector<int32_t> cnt(Ng, 0), nodes;
    for (int64_t t = 0; t < nt; t++)
        for (int u = 0; u < S; u++)
            if (cnt[node(t, u)]++ == 0) nodes.push_back((int32_t)node(t, u));
    // by falling number of entries, then by node
    std::sort(nodes.begin(), nodes.end(),
              [&](int32_t a, int32_t b) { return cnt[a] != cnt[b] ? cnt[a] > cnt[b] : a < b; });
    std::vector<int32_t> ptr(nodes.size() + 1, 0), at(Ng, 0), ent(nt * S);
    for (size_t v = 0; v < nodes.size(); v++) {
        at[nodes[v]] = ptr[v];
        ptr[v + 1] = ptr[v] + cnt[nodes[v]];
    }
    for (int64_t t = 0; t < nt; t++)
        for (int u = 0; u < S; u++) ent[at[node(t, u)]++] = (int32_t)(t * S + u);
    op->pm_nnode = (int64_t)nodes.size();
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->pm_node, sizeof(int32_t) * nodes.size(), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->pm_ptr, sizeof(int32_t) * ptr.size(), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->pm_ent, sizeof(int32_t) * ent.size(), st));
    SIE_CUDA_TRY(cudaMemcpyAsync(op->pm_node, nodes.data(), sizeof(int32_t) * nodes.size(), cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->pm_tc, sizeof(double2) * 9 * nt, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(op->pm_ptr, ptr.data(), sizeof(int32_t) * ptr.size(), cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(op->pm_ent, ent.data(), sizeof(int32_t) * ent.size(), cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaStreamSynchronize(st));
    return SIE_OK;
}

// The charge rows y2 of y = SYS [H; rho] and yb = the scalar-potential term: all that
// needs neither E nor the grid
static sie_status sys_charge(sie_op* op, cudaStream_t st, const double2* H, const double2* rho, double2* yb,
                             double2* y2)
{
    sie_ctx* c = op->mesh->ctx;
    const DevMesh& M = op->mesh->d;
    const int64_t ne = M.ne, nt = M.nt;
    AimOp& X = op->ext;
    const bool c64 = op->p.precision == SIE_MIXED && X.valLK32;
    SIE_CUDA_TRY(cudaMemsetAsync(yb, 0, sizeof(double2) * ne, st));
    Stage s_(c, "spmv_sys_rest");
    double2* sig = op->sys_tmp + ne;  // apply_Z uses the first ne
    double2* phi = sig + nt;
    if (c64) {
        k_sigma32<<<nb(nt), 256, 0, st>>>((int)nt, M.area, rho, op->pk_sig);
        SIE_CUDA_TRY(csr_launch(st, (int)nt, tri_nnz(X), X.tri_row_ptr, X.tri_col, X.valLphi32, op->pk_sig,
                                make_double2(1.0, 0.0), false, phi));
    } else {
        k_sigma<<<nb(nt), 256, 0, st>>>((int)nt, M.area, rho, sig);
        SIE_TRY(spmv(st, (int)nt, tri_nnz(X), X.tri_row_ptr, X.tri_col, X.valLphi, sig, cplx(1.0, 0.0), phi, false));
    }
    k_dt<<<nb(ne), 256, 0, st>>>((int)ne, M.edge_tri, op->elen, phi, yb);
    k_row2<<<nb(nt), 256, 0, st>>>((int)nt, M, H, rho, op->k0, y2);
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}

// yb += the near-region products of H and E and the term in E alone
static sie_status sys_near(sie_op* op, cudaStream_t st, const double2* H, const double2* E, double2* yb)
{
    sie_ctx* c = op->mesh->ctx;
    const int64_t ne = op->mesh->h.ne;
    AimOp& X = op->ext;
    const bool c64 = op->p.precision == SIE_MIXED && X.valLK32;
    if (c64) k_pack_he32<<<nb(ne), 256, 0, st>>>((int)ne, H, E, op->pk_he);
    {
        // the exterior near-region product alone (one kernel)
        Stage s1_(c, "spmv_near_ext");
        if (c64)
            k_spmv2_c64<<<(unsigned)((ne + 3) / 4), 128, 0, st>>>((int)ne, X.row_ptr, X.col, X.valLK32, op->pk_he,
                                                                   make_double2(0.0, op->k0), make_double2(-1.0, 0.0),
                                                                   yb);
        else {
            const bool small = ne <= 8192;
            auto f = small ? k_spmv2<32> : k_spmv2<8>;
            const int T = small ? 64 : 256;  // small: over more SMs' FP64 lanes
            f<<<nb(ne * (small ? 32 : 8), T), T, 0, st>>>((int)ne, X.row_ptr, X.col, X.valLA, H,
                                                          make_double2(0.0, op->k0), X.valK, E,
                                                          make_double2(-1.0, 0.0), yb);
        }
        SIE_CUDA_TRY(cudaGetLastError());
    }
    Stage s_(c, "spmv_sys_rest");
    return spmv(st, (int)ne, op->ix_nnz, op->ix_row_ptr, op->ix_col, op->ix_val, E, cplx(-0.5, 0.0), yb);
}

// y1 = the grid part.  The interpolation adds two triangles' values to an edge of zeros
// (in either order the same sum); yb is added after it.
static sie_status sys_grid(sie_op* op, const double2* H, const double2* E, const double2* rho, double2* y1)
{
    sie_ctx* c = op->mesh->ctx;
    cudaStream_t st = c->stream;
    const DevMesh& M = op->mesh->d;
    AimOp& X = op->ext;
    const GridDesc& g = X.g;
    int S = (g.M + 1) * (g.M + 1) * (g.M + 1);
    int64_t Ng = (int64_t)g.N[0] * g.N[1] * g.N[2];
    int64_t nn = (int64_t)g.n[0] * g.n[1] * g.n[2];
    if (op->p.precision == SIE_MIXED) {
        float2* src = reinterpret_cast<float2*>(op->ws.src);
        float2* buf = reinterpret_cast<float2*>(op->ws.bufs);
        {
            Stage s_(c, "project_sys32");
            float2* tc = reinterpret_cast<float2*>(op->pm_tc);
            k_tri_coef<float2><<<nb(M.nt, 128), 128, 0, st>>>(M.nt, M, H, 0, E, 0, rho, 0, tc);
            SIE_CUDA_TRY(cudaMemsetAsync(src, 0, sizeof(float2) * 7 * Ng, st));
            k_project_gather<float2, float><<<gio_blocks(op->pm_nnode, 8), 256, 0, st>>>(
                op->pm_nnode, op->pm_node, op->pm_ptr, op->pm_ent, S, op->W32, tc, M.nt, src, Ng);
            SIE_CUDA_TRY(cudaGetLastError());
        }
        if (fused_z() && fft_fused_z(g)) {
            SIE_TRY(fft_sys(st, buf, src, g, X.spec32, (float)op->k0, c));
        } else {
            SIE_TRY(fft3d(st, buf, src, g, -1, 1, c, 7));
            {
                Stage s_(c, "specmul_sys32");
                k_specmul_sys32<<<nb(nn), 256, 0, st>>>(X.spec32, buf, nn, (float)op->k0);
                SIE_CUDA_TRY(cudaGetLastError());
            }
            SIE_TRY(fft3d(st, buf, src, g, +1, 1, c, 4));
        }
        {
            Stage s_(c, "interp32");
            if (M.nt <= GIO_WIDE)
                k_interp<32, float2, float, 4><<<gio_blocks(M.nt, 32, GIO_SMALL), GIO_SMALL, 0, st>>>(
                    M.nt, S, g.M, M, op->base, op->W32, src, g, make_double2(1.0, 0.0), Ng, y1, 0);
            else
                k_interp<4, float2, float, 4><<<gio_blocks(M.nt, 4), 256, 0, st>>>(
                    M.nt, S, g.M, M, op->base, op->W32, src, g, make_double2(1.0, 0.0), Ng, y1, 0);
            SIE_CUDA_TRY(cudaGetLastError());
        }
    } else {
        double2* src = op->ws.src;
        double2* buf = op->ws.bufs;
        {
            Stage s_(c, "project_sys");
            k_tri_coef<double2><<<nb(M.nt, 128), 128, 0, st>>>(M.nt, M, H, 0, E, 0, rho, 0, op->pm_tc);
            SIE_CUDA_TRY(cudaMemsetAsync(src, 0, sizeof(double2) * 7 * Ng, st));
            k_project_gather<double2, double><<<gio_blocks(op->pm_nnode, 8), 256, 0, st>>>(
                op->pm_nnode, op->pm_node, op->pm_ptr, op->pm_ent, S, op->W, op->pm_tc, M.nt, src, Ng);
            SIE_CUDA_TRY(cudaGetLastError());
        }
        if (fused_z() && fft_fused_z(g)) {
            SIE_TRY(fft_sys(st, buf, src, g, X.spec, op->k0, c));
        } else {
            SIE_TRY(fft3d(st, buf, src, g, -1, 1, c, 7));
            {
                Stage s_(c, "specmul_sys");
                k_specmul_sys<<<nb(nn), 256, 0, st>>>(X.spec, buf, nn, op->k0);
                SIE_CUDA_TRY(cudaGetLastError());
            }
            SIE_TRY(fft3d(st, buf, src, g, +1, 1, c, 4));
        }
        {
            Stage s_(c, "interp");
            SIE_TRY(aim_interp(op, src, 1, make_double2(1.0, 0.0), y1, 0, 1));
        }
    }
    return SIE_OK;
}

// y = SYS x, x = [H (ne); c0 rho (nt)].  The charge part runs beside the nested solve
// and the near part (FP64 products) beside the transforms (integer), on a branch when
// the product is captured: a bar of 336 triangles 154 -> 142 us, 20,480 triangles
// 1,265 -> 1,177 us.  The interpolation adds two triangles' values to an edge of zeros,
// the branch sums into yb: every sum keeps a fixed order.
static sie_status apply_sys(sie_op* op, const double2* x, double2* y)
{
    const int64_t ne = op->mesh->h.ne;
    double2* E = op->sys_E;
    double2* yb = op->sys_tmp + ne + 2 * op->mesh->h.nt;
    Branch br(op, op->capturing);
    SIE_CUDA_TRY(br.follow());
    SIE_TRY(sys_charge(op, br.st(), x, x + ne, yb, y + ne));
    cudaStream_t st = op->mesh->ctx->stream;
    SIE_CUDA_TRY(cudaMemsetAsync(y, 0, sizeof(double2) * ne, st));
    SIE_TRY(apply_Z(op, x, E, nullptr));
    SIE_CUDA_TRY(br.follow());
    SIE_TRY(sys_near(op, br.st(), x, E, yb));
    SIE_TRY(sys_grid(op, x, E, x + ne, y));
    SIE_CUDA_TRY(br.join());
    return axpby(st, ne, 1.0, yb, 1.0, y);
}

// ------------------------------------------------------------------ graph of the system product
// For a near-region-only interior the whole product (nested solve included)
// is captured once into a CUDA graph: one launch per product instead of about 20,
// and no host wait for the nested solve, which is one kernel.  One graph per
// precision; dropped when the nested-solve settings change.  SIE_GRAPH=0 in the
// environment keeps the stream path (for comparison).
static bool graph_enabled()
{
    const char* e = getenv("SIE_GRAPH");
    return !(e && e[0] == '0');
}

void sys_graph_reset(sie_op* op)
{
    // a replay may still be queued on the context stream
    if (op->gexec[0] || op->gexec[1]) cudaStreamSynchronize(op->mesh->ctx->stream);
    for (cudaGraphExec_t& g : op->gexec) {
        if (g) cudaGraphExecDestroy(g);
        g = nullptr;
    }
    op->gfailed = false;
}

static sie_status build_sys_graph(sie_op* op)
{
    sie_ctx* c = op->mesh->ctx;
    const int64_t ne = op->mesh->h.ne, n = ne + op->mesh->h.nt;
    // everything the product touches exists before the capture starts
    SIE_TRY(op->kin.alloc(c->stream, ne, inner_m(op)));
    if (!op->g_io) SIE_CUDA_TRY(cudaMallocAsync((void**)&op->g_io, sizeof(double2) * 2 * n, c->stream));
    SIE_CUDA_TRY(cudaStreamSynchronize(c->stream));
    cudaStream_t saved = c->stream;
    c->stream = op->gs[0];
    op->capturing = true;
    cudaGraph_t graph = nullptr;
    sie_status s = SIE_OK;
    cudaError_t e = cudaStreamBeginCapture(op->gs[0], cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        s = apply_sys(op, op->g_io, op->g_io + n);
        cudaError_t e2 = cudaStreamEndCapture(op->gs[0], &graph);
        if (s == SIE_OK) e = e2;
    }
    op->capturing = false;
    c->stream = saved;
    cudaGraphExec_t& gx = op->gexec[op->p.precision == SIE_MIXED ? 1 : 0];
    if (s == SIE_OK && e == cudaSuccess) e = cudaGraphGetNodes(graph, nullptr, &op->gnodes[0]);
    if (s == SIE_OK && e == cudaSuccess) e = cudaGraphInstantiate(&gx, graph, 0);
    if (graph) cudaGraphDestroy(graph);
    if (s != SIE_OK || e != cudaSuccess) {
        if (gx) cudaGraphExecDestroy(gx);
        gx = nullptr;
        op->gfailed = true;
        if (e != cudaSuccess) set_error(std::string("system-product graph: ") + cudaGetErrorString(e));
        return s != SIE_OK ? s : SIE_ERR_CUDA;
    }
    return SIE_OK;
}

// y = SYS x through the graph when it applies, else the stream path
static sie_status apply_sys_fast(sie_op* op, const double2* x, double2* y)
{
    sie_ctx* c = op->mesh->ctx;
    if (op->inn.has_grid || c->prof.on || op->gfailed || !graph_enabled()) return apply_sys(op, x, y);
    cudaGraphExec_t& gx = op->gexec[op->p.precision == SIE_MIXED ? 1 : 0];
    if (!gx && build_sys_graph(op) != SIE_OK) return apply_sys(op, x, y);
    const int64_t n = op->mesh->h.ne + op->mesh->h.nt;
    SIE_CUDA_TRY(cudaMemcpyAsync(op->g_io, x, sizeof(double2) * n, cudaMemcpyDeviceToDevice, c->stream));
    SIE_CUDA_TRY(cudaGraphLaunch(gx, c->stream));
    SIE_CUDA_TRY(cudaMemcpyAsync(y, op->g_io + n, sizeof(double2) * n, cudaMemcpyDeviceToDevice, c->stream));
    return SIE_OK;
}

sie_status sys_stats_fold(sie_op* op)
{
    if (!op->gstat) return SIE_OK;
    double h[sie_op::GSTAT] = {0, 0, 0, 0, 0, 0, 0};
    cudaStream_t st = op->mesh->ctx->stream;
    SIE_CUDA_TRY(cudaMemcpyAsync(h, op->gstat, sizeof(h), cudaMemcpyDeviceToHost, st));
    SIE_CUDA_TRY(cudaStreamSynchronize(st));
    op->stats[2] = std::max(op->stats[2], h[0]);
    op->stats[3] = std::max(op->stats[3], h[1]);
    op->stats[4] = std::max(op->stats[4], h[4]);
    op->stats[5] = std::max(op->stats[5], h[5]);
    op->last_nested = h[2];
    int lost = 0;
    std::memcpy(&lost, &h[6], sizeof(lost));
    if (lost) {
        op->wait_lost = true;
        op->stats[3] = std::numeric_limits<double>::infinity();  // what device-pointer callers see
    }
    return SIE_OK;
}

// Constraint preconditioner (the near-region form of the AEFIE constraint
// preconditioner of Sec. III-D): solves
//     (Dg - kappa D^T Lphi_NR D) y = v
// with Dg = diag(LA) (exact diagonal) and Lphi_NR the exact near-region
// scalar-potential matrix, by block elimination on the charges q = D y:
//     (I - kappa D Dg^-1 D^T Lphi_NR) q = D Dg^-1 v,   y = Dg^-1 (v + kappa D^T Lphi_NR q),
// the triangle system solved by an inner GMRES to tol (the outer iterations
// are flexible), preconditioned by its dense factorisation when one was made
// (dense_pc_max).
static sie_status constraint_solve(sie_op* op, AimOp& a, cplx kappa, KrylovWork& K, double tol, const double2* v,
                                   double2* y)
{
    sie_ctx* c = op->mesh->ctx;
    cudaStream_t st = c->stream;
    const DevMesh& M = op->mesh->d;
    const int64_t ne = M.ne, nt = M.nt;
    double2* t1 = op->cs_e;       // ne
    double2* rq = op->cs_t;       // nt: right-hand side
    double2* q = op->cs_t + nt;   // nt: solution
    double2* ph = op->cs_t + 2 * nt;
    double2* te = op->cs_e + ne;  // ne scratch
    {
        SIE_TRY(K.alloc(st, nt, op->p.constraint_restart));
        ResWork w;
        w.m = K.m, w.V = K.V, w.Z = K.Z, w.H = K.Hd;
        sie_status s = SIE_OK;
        Stage s_(c, "constraint_solve");
        if (constraint_resident(op, a, make_double2(kappa.real(), kappa.imag()), false, v, y, tol, op->p.constraint_maxit,
                                w, t1, rq, q, &s))
            return s;
    }
    k_jacobi<<<nb(ne), 256, 0, st>>>(ne, v, a.dLA, make_double2(1.0, 0.0), t1);
    k_D<<<nb(nt), 256, 0, st>>>((int)nt, M, t1, rq);
    SIE_CUDA_TRY(cudaGetLastError());
    auto S = [&](const double2* x, double2* out) {
        // out = x - kappa D Dg^-1 D^T Lphi x
        SIE_TRY(spmv(st, (int)nt, tri_nnz(a), a.tri_row_ptr, a.tri_col, a.valLphiNR, x, 1.0, ph, false));
        SIE_CUDA_TRY(cudaMemsetAsync(te, 0, sizeof(double2) * ne, st));
        k_dt<<<nb(ne), 256, 0, st>>>((int)ne, M.edge_tri, op->elen, ph, te);
        k_jacobi<<<nb(ne), 256, 0, st>>>(ne, te, a.dLA, make_double2(1.0, 0.0), te);
        k_D<<<nb(nt), 256, 0, st>>>((int)nt, M, te, out);
        SIE_CUDA_TRY(cudaGetLastError());
        return axpby(st, nt, 1.0, x, -kappa, out);
    };
    auto I = [&](const double2* x, double2* out) {
        SIE_CUDA_TRY(cudaMemcpyAsync(out, x, sizeof(double2) * nt, cudaMemcpyDeviceToDevice, st));
        return SIE_OK;
    };
    auto LU = [&](const double2* x, double2* out) {
        Stage s_(c, "constraint_lu_solve");
        return a.lu->solve(st, x, out);
    };
    // the dense LU (complex64 assembly and factors) preconditions a GMRES on
    // the FP64 triangle system, which then converges in two or three
    // iterations; applied alone it is not enough: T = I - kappa D Dg^-1 D^T
    // Lphi has entries far above 1 whose cancellation the complex64 copy
    // loses, and the outer solve stalls.  Without the LU, plain GMRES.
    const Apply P = a.lu ? Apply(LU) : Apply(I);
    int it = 0;
    double rr = 0;
    sie_status s;
    {
        Stage s_(c, "constraint_solve");
        // a handful of iterations: each checked before the next (lag 0)
        s = fgmres(c, K, nt, S, P, rq, q, tol, op->p.constraint_maxit, op->p.constraint_restart, &it, &rr, 0);
    }
    op->stats[4] = std::max(op->stats[4], (double)it);
    op->stats[5] = std::max(op->stats[5], rr);
    if (s != SIE_OK && s != SIE_ERR_NOT_CONVERGED) return s;
    // y = Dg^-1 (v + kappa D^T Lphi q)
    SIE_TRY(spmv(st, (int)nt, tri_nnz(a), a.tri_row_ptr, a.tri_col, a.valLphiNR, q, 1.0, ph, false));
    SIE_CUDA_TRY(cudaMemsetAsync(te, 0, sizeof(double2) * ne, st));
    k_dt<<<nb(ne), 256, 0, st>>>((int)ne, M.edge_tri, op->elen, ph, te);
    SIE_CUDA_TRY(cudaGetLastError());
    SIE_TRY(axpby(st, ne, kappa, te, 0.0, te));
    SIE_TRY(axpby(st, ne, 1.0, v, 1.0, te));
    k_jacobi<<<nb(ne), 256, 0, st>>>(ne, te, a.dLA, make_double2(1.0, 0.0), y);
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}

// Exterior AEFIE constraint preconditioner P = [[j k0 Dg, D^T Lphi_NR B], [F D, j k0 I]]
// applied exactly by block elimination (Schur complement on the currents):
//   w1 = (j k0)^-1 (Dg - k0^-2 D^T Lphi_NR D)^-1 (v1 - (j k0)^-1 D^T Lphi_NR B v2)
//   w2 = (v2 - F D w1) / (j k0)
static sie_status precond_sys(sie_op* op, const double2* x, double2* y)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const DevMesh& M = op->mesh->d;
    const int64_t ne = M.ne, nt = M.nt;
    AimOp& X = op->ext;
    const cplx jk0(0.0, op->k0);
    double2* v1p = op->pc_e;          // ne
    double2* sig = op->pc_t;          // nt
    double2* ph = op->pc_t + nt;      // nt
    {
        KrylovWork& K = op->kcs_out;
        SIE_TRY(K.alloc(st, nt, op->p.constraint_restart));
        ResWork w;
        w.m = K.m, w.V = K.V, w.Z = K.Z, w.H = K.Hd;
        sie_status s = SIE_OK;
        Stage s_(op->mesh->ctx, "constraint_solve");
        if (constraint_resident(op, X, make_double2(1.0 / (op->k0 * op->k0), 0.0), true, x, y, op->p.tol_constraint,
                                op->p.constraint_maxit, w, v1p, op->cs_t, op->cs_t + nt, &s))
            return s;
    }
    // v1' = v1 - (j k0)^-1 D^T Lphi B v2,  B v2 = -A v2
    k_sigma<<<nb(nt), 256, 0, st>>>((int)nt, M.area, x + ne, sig);
    SIE_TRY(spmv(st, (int)nt, tri_nnz(X), X.tri_row_ptr, X.tri_col, X.valLphiNR, sig, 1.0, ph, false));
    SIE_CUDA_TRY(cudaMemsetAsync(v1p, 0, sizeof(double2) * ne, st));
    k_dt<<<nb(ne), 256, 0, st>>>((int)ne, M.edge_tri, op->elen, ph, v1p);
    SIE_CUDA_TRY(cudaGetLastError());
    SIE_TRY(axpby(st, ne, 1.0, x, -1.0 / jk0, v1p));
    SIE_TRY(constraint_solve(op, X, 1.0 / (op->k0 * op->k0), op->kcs_out, op->p.tol_constraint, v1p, y));
    SIE_TRY(axpby(st, ne, 1.0 / jk0, y, 0.0, y));
    // w2 = (v2 - F D w1) / (j k0), (F D w1)_t = (D w1)_t / A_t
    k_D<<<nb(nt), 256, 0, st>>>((int)nt, M, y, ph);
    SIE_CUDA_TRY(cudaGetLastError());
    k_jacobi<<<nb(nt), 256, 0, st>>>(nt, ph, nullptr, make_double2(1.0, 0.0), ph);
    k_fdiv_area<<<nb(nt), 256, 0, st>>>((int)nt, M.area, ph);
    SIE_CUDA_TRY(cudaGetLastError());
    SIE_CUDA_TRY(cudaMemcpyAsync(y + ne, x + ne, sizeof(double2) * nt, cudaMemcpyDeviceToDevice, st));
    SIE_TRY(axpby(st, nt, -1.0 / jk0, ph, 1.0 / jk0, y + ne));
    return SIE_OK;
}

sie_status constraint_lu_build(sie_op* op)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const int nt = (int)op->mesh->h.nt;
    if (op->p.dense_pc_max <= 0 || nt > op->p.dense_pc_max) return SIE_OK;
    auto t0 = std::chrono::steady_clock::now();
    sie_status s = SIE_OK;
    for (AimOp* a : {&op->ext, &op->inn}) {
        if (a == &op->inn && !op->inn.has_grid) continue;  // near-only interiors use the SPAI
        cplx k(a->kr, a->ki);
        cplx kappa = 1.0 / (k * k);
        a->lu = new DenseLU();
        if ((s = a->lu->alloc(nt)) != SIE_OK) break;
        if ((s = dense_lu_assemble(st, *a->lu, op, *a, make_double2(kappa.real(), kappa.imag()))) != SIE_OK) break;
        if ((s = a->lu->factor(st)) != SIE_OK) break;
        if ((s = a->lu->invert(st)) != SIE_OK) break;
    }
    if (s != SIE_OK) {
        // no room or a singular triangle system: the iterative constraint solve stays
        cudaGetLastError();
        cudaStreamSynchronize(st);
        constraint_lu_release(op);
        op->lu_ms = -(double)s;
        return SIE_OK;
    }
    op->lu_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return SIE_OK;
}

void constraint_lu_release(sie_op* op)
{
    for (AimOp* a : {&op->ext, &op->inn})
        if (a->lu) {
            a->lu->release();
            delete a->lu;
            a->lu = nullptr;
        }
}

sie_status constraint_lu_check(sie_op* op)
{
    for (AimOp* a : {&op->ext, &op->inn})
        if (a->lu) SIE_TRY(a->lu->check(op->mesh->ctx->stream));
    return SIE_OK;
}

// rows of (column, value) pairs -> device CSR (duplicate columns summed)
static sie_status upload_rows(cudaStream_t st, std::vector<std::vector<std::pair<int32_t, double>>>& rows,
                              int64_t** rp_d, int32_t** col_d, double2** val_d, int64_t* nnz)
{
    std::vector<int64_t> rp(rows.size() + 1, 0);
    std::vector<int32_t> col;
    std::vector<double2> val;
    for (size_t m = 0; m < rows.size(); m++) {
        auto& r = rows[m];
        std::sort(r.begin(), r.end(), [](auto& a, auto& b) { return a.first < b.first; });
        for (size_t k = 0; k < r.size(); k++) {
            if ((int64_t)col.size() > rp[m] && col.back() == r[k].first)
                val.back().x += r[k].second;
            else {
                col.push_back(r[k].first);
                val.push_back(make_double2(r[k].second, 0.0));
            }
        }
        rp[m + 1] = (int64_t)col.size();
    }
    *nnz = (int64_t)col.size();
    SIE_CUDA_TRY(cudaMallocAsync((void**)rp_d, sizeof(int64_t) * rp.size(), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)col_d, sizeof(int32_t) * std::max<size_t>(col.size(), 1), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)val_d, sizeof(double2) * std::max<size_t>(val.size(), 1), st));
    SIE_CUDA_TRY(cudaMemcpyAsync(*rp_d, rp.data(), sizeof(int64_t) * rp.size(), cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(*col_d, col.data(), sizeof(int32_t) * col.size(), cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(*val_d, val.data(), sizeof(double2) * val.size(), cudaMemcpyHostToDevice, st));
    // the host vectors must outlive the copies
    SIE_CUDA_TRY(cudaStreamSynchronize(st));
    return SIE_OK;
}

// RWG Gram matrix G_mn = I f_m . f_n dS as edge CSR: on triangle t (centroid
// c, I (r - c) dS = 0, I |r - c|^2 dS = A (l1^2 + l2^2 + l3^2) / 36) the block is
// c_i c_j A [(l1^2 + l2^2 + l3^2) / 36 + (c - p_i).(c - p_j)]
static sie_status gram_prepare(sie_op* op)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const HostMesh& h = op->mesh->h;
    std::vector<std::vector<std::pair<int32_t, double>>> rows(h.ne);
    std::vector<double> diag(h.ne, 0.0);
    for (int64_t t = 0; t < h.nt; t++) {
        double l2 = 0;
        for (int i = 0; i < 3; i++) {
            const double* a = &h.V[3 * h.T[3 * t + i]];
            const double* b = &h.V[3 * h.T[3 * t + (i + 1) % 3]];
            for (int d = 0; d < 3; d++) l2 += (b[d] - a[d]) * (b[d] - a[d]);
        }
        for (int i = 0; i < 3; i++)
            for (int j = 0; j < 3; j++) {
                const double* qi = &h.q[9 * t + 3 * i];
                const double* qj = &h.q[9 * t + 3 * j];
                double v = h.coef[3 * t + i] * h.coef[3 * t + j] * h.area[t] *
                           (l2 / 36.0 + qi[0] * qj[0] + qi[1] * qj[1] + qi[2] * qj[2]);
                rows[h.tri_edge[3 * t + i]].push_back({h.tri_edge[3 * t + j], v});
                if (h.tri_edge[3 * t + i] == h.tri_edge[3 * t + j]) diag[h.tri_edge[3 * t + i]] += v;
            }
    }
    SIE_TRY(upload_rows(st, rows, &op->gr_row_ptr, &op->gr_col, &op->gr_val, &op->gr_nnz));
    std::vector<double2> dc(h.ne);
    for (int64_t m = 0; m < h.ne; m++) dc[m] = make_double2(diag[m], 0.0);
    for (double& d : diag) d = 1.0 / d;
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->gr_diag, sizeof(double2) * h.ne, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(op->gr_diag, dc.data(), sizeof(double2) * h.ne, cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->gr_idiag, sizeof(double) * h.ne, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(op->gr_idiag, diag.data(), sizeof(double) * h.ne, cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaStreamSynchronize(st));
    return SIE_OK;
}

// Measured lanes-per-row choice (csr_autotune) for the operator's CSR
// products: exterior near-region L and K (L0/K0 products), the triangle Lphi
// products in FP64 and complex64, I-cross, the near-only interior matrices
// and the SIBC Gram matrix.  Runs once per pattern on the context stream with
// zeroed operands; the system-product graph captured later uses the result.
sie_status csr_tune_op(sie_op* op)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const int64_t ne = op->mesh->h.ne, nt = op->mesh->h.nt;
    double2* x = op->xtmp;       // ne (>= nt) zeros
    double2* y = op->xtmp + ne;  // ne scratch
    SIE_CUDA_TRY(cudaMemsetAsync(x, 0, sizeof(double2) * ne, st));
    const AimOp& X = op->ext;
    if (X.nnz > 0 && X.valL) SIE_CUDA_TRY(csr_autotune(st, (int)ne, X.nnz, X.row_ptr, X.col, X.valL, x, y));
    const int64_t tn = tri_nnz(X);
    if (tn > 0 && X.valLphi) SIE_CUDA_TRY(csr_autotune(st, (int)nt, tn, X.tri_row_ptr, X.tri_col, X.valLphi, x, y));
    if (tn > 0 && X.valLphi32 && op->pk_sig) {
        SIE_CUDA_TRY(cudaMemsetAsync(op->pk_sig, 0, sizeof(float2) * nt, st));
        SIE_CUDA_TRY(csr_autotune(st, (int)nt, tn, X.tri_row_ptr, X.tri_col, X.valLphi32, (const float2*)op->pk_sig, y));
    }
    if (op->ix_nnz > 0)
        SIE_CUDA_TRY(csr_autotune(st, (int)ne, op->ix_nnz, op->ix_row_ptr, op->ix_col, op->ix_val, x, y));
    const AimOp& I = op->inn;
    if (I.nnz > 0 && I.valL) SIE_CUDA_TRY(csr_autotune(st, (int)ne, I.nnz, I.row_ptr, I.col, I.valL, x, y));
    if (op->gr_nnz > 0)
        SIE_CUDA_TRY(csr_autotune(st, (int)ne, op->gr_nnz, op->gr_row_ptr, op->gr_col, op->gr_val, x, y));
    return SIE_OK;
}

sie_status sys_prepare(sie_op* op)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const HostMesh& h = op->mesh->h;
    if (op->p.interior_model == SIE_SIBC) SIE_TRY(gram_prepare(op));
    SIE_TRY(proj_map_ready(op));
    // Ix as an edge CSR: (Ix)_mn = I_T f_m . (n x f_n) = c_m c_n A n . ((p_n - c) x (p_m - c))
    std::vector<std::vector<std::pair<int32_t, double>>> rows(h.ne);
    for (int64_t t = 0; t < h.nt; t++) {
        const double* c = &h.cen[3 * t];
        const double* nr = &h.nrm[3 * t];
        double p[3][3];
        for (int i = 0; i < 3; i++)
            for (int d = 0; d < 3; d++) p[i][d] = h.V[3 * h.T[3 * t + i] + d] - c[d];
        for (int i = 0; i < 3; i++)
            for (int j = 0; j < 3; j++) {
                double cx = p[j][1] * p[i][2] - p[j][2] * p[i][1];
                double cy = p[j][2] * p[i][0] - p[j][0] * p[i][2];
                double cz = p[j][0] * p[i][1] - p[j][1] * p[i][0];
                double v = h.coef[3 * t + i] * h.coef[3 * t + j] * h.area[t] * (nr[0] * cx + nr[1] * cy + nr[2] * cz);
                rows[h.tri_edge[3 * t + i]].push_back({h.tri_edge[3 * t + j], v});
            }
    }
    std::vector<int64_t> rp(h.ne + 1, 0);
    std::vector<int32_t> col;
    std::vector<double2> val;
    for (int64_t m = 0; m < h.ne; m++) {
        auto& r = rows[m];
        std::sort(r.begin(), r.end(), [](auto& a, auto& b) { return a.first < b.first; });
        for (size_t k = 0; k < r.size(); k++) {
            if (!col.empty() && (int64_t)col.size() > rp[m] && col.back() == r[k].first)
                val.back().x += r[k].second;
            else {
                col.push_back(r[k].first);
                val.push_back(make_double2(r[k].second, 0.0));
            }
        }
        rp[m + 1] = (int64_t)col.size();
    }
    op->ix_nnz = (int64_t)col.size();
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->ix_row_ptr, sizeof(int64_t) * rp.size(), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->ix_col, sizeof(int32_t) * col.size(), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->ix_val, sizeof(double2) * val.size(), st));
    SIE_CUDA_TRY(cudaMemcpyAsync(op->ix_row_ptr, rp.data(), sizeof(int64_t) * rp.size(), cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(op->ix_col, col.data(), sizeof(int32_t) * col.size(), cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(op->ix_val, val.data(), sizeof(double2) * val.size(), cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->elen, sizeof(double) * h.ne, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(op->elen, h.edge_len.data(), sizeof(double) * h.ne, cudaMemcpyHostToDevice, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->sys_E, sizeof(double2) * h.ne, st));
    int lo = 0, hi = 0;
    SIE_CUDA_TRY(cudaDeviceGetStreamPriorityRange(&lo, &hi));
    for (int i = 0; i < 2; i++)  // the branch gives way to the main chain
        if (!op->gs[i]) SIE_CUDA_TRY(cudaStreamCreateWithPriority(&op->gs[i], cudaStreamNonBlocking, i ? lo : hi));
    for (cudaEvent_t& ev : op->gev)
        if (!ev) SIE_CUDA_TRY(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->sys_tmp, sizeof(double2) * 2 * (h.ne + h.nt), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->sys_vec, sizeof(double2) * 4 * (h.ne + h.nt), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->gstat, sizeof(double) * sie_op::GSTAT, st));
    SIE_CUDA_TRY(cudaMemsetAsync(op->gstat, 0, sizeof(double) * sie_op::GSTAT, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->res_bar, sizeof(unsigned), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->pk_he, sizeof(float4) * h.ne, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->pk_sig, sizeof(float2) * h.nt, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->cs_e, sizeof(double2) * 2 * h.ne, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->cs_t, sizeof(double2) * 3 * h.nt, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->pc_e, sizeof(double2) * h.ne, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->pc_t, sizeof(double2) * 2 * h.nt, st));
    SIE_CUDA_TRY(cudaStreamSynchronize(st));
    return SIE_OK;
}

void sys_release(sie_op* op)
{
    cudaStream_t st = op->mesh->ctx->stream;
    sys_graph_reset(op);
    cudaStreamSynchronize(st);
    constraint_lu_release(op);
    for (cudaEvent_t& ev : op->gev) {
        if (ev) cudaEventDestroy(ev);
        ev = nullptr;
    }
    for (cudaStream_t& g : op->gs)
        if (g) {
            cudaStreamDestroy(g);
            g = nullptr;
        }
    if (op->ir_buf) cudaFreeAsync(op->ir_buf, st);
    op->ir_buf = nullptr;
    if (op->g_io) cudaFreeAsync(op->g_io, st);
    if (op->gstat) cudaFreeAsync(op->gstat, st);
    if (op->res_bar) cudaFreeAsync(op->res_bar, st);
    op->g_io = nullptr;
    op->gstat = nullptr;
    op->res_bar = nullptr;
    op->kin.release(st);
    op->kout.release(st);
    op->kmulti.release(st);
    op->kcs_multi.release(st);
    op->kzp.release(st);
    if (op->zp) cudaFreeAsync(op->zp, st);
    op->zp = nullptr;
    for (void* p : {(void*)op->mscr, (void*)op->ir_multi, (void*)op->mvec})
        if (p) cudaFreeAsync(p, st);
    op->mscr = op->ir_multi = op->mvec = nullptr;
    blk_release(op);
    op->kcs_in.release(st);
    op->kcs_out.release(st);
    for (void* p : {(void*)op->gr_row_ptr, (void*)op->gr_col, (void*)op->gr_val, (void*)op->gr_idiag, (void*)op->gr_diag,
                    (void*)op->pm_node, (void*)op->pm_ptr, (void*)op->pm_ent, (void*)op->pm_tc,
                    (void*)op->pk_he, (void*)op->pk_sig, (void*)op->bal})
        if (p) cudaFreeAsync(p, st);
    op->pk_he = nullptr;
    op->pk_sig = nullptr;
    op->bal = nullptr;
    for (void* p : {(void*)op->ix_row_ptr, (void*)op->ix_col, (void*)op->ix_val, (void*)op->elen, (void*)op->sys_E,
                    (void*)op->sys_tmp, (void*)op->sys_vec, (void*)op->cs_e, (void*)op->cs_t, (void*)op->pc_e,
                    (void*)op->pc_t})
        if (p) cudaFreeAsync(p, st);
    cudaStreamSynchronize(st);
}

sie_status sys_matvec(sie_op* op, int which, const double2* x, double2* y)
{
    if (which == SIE_OP_SYS) return apply_sys_fast(op, x, y);
    return apply_Z(op, x, y, nullptr);
}

// SIE_ERR_TIMEOUT when a wait ran out in a nested (interior) solve of the products
// since the statistics were last cleared, SIE_ERR_NOT_CONVERGED when one ended above
// tol_inner (synchronises)
sie_status nested_check(sie_op* op, const char* who)
{
    SIE_TRY(sys_stats_fold(op));
    if (op->wait_lost) {
        set_error(std::string(who) + ": a grid barrier's wait ran out in a nested interior solve");
        return SIE_ERR_TIMEOUT;
    }
    if (op->stats[3] >= op->p.tol_inner) {
        set_error(std::string(who) + ": a nested interior solve ended at relative residual " +
                  std::to_string(op->stats[3]) + " >= tol_inner after min(inner_maxit, " +
                  std::to_string(INNER_BASIS_MAX) + ") iterations; the result uses that inexact Z_i");
        return SIE_ERR_NOT_CONVERGED;
    }
    return SIE_OK;
}

// The status of an outer solve that ended with s: products whose nested solve gave up
// leave their result unwritten, and whatever the outer iteration made of it (no
// convergence, numbers that are not finite) is not the reason
static sie_status solve_status(sie_op* op, sie_status s, const char* who)
{
    if (s != SIE_OK && s != SIE_ERR_NOT_CONVERGED && s != SIE_ERR_ARG) return s;
    const sie_status n = nested_check(op, who);
    if (n == SIE_ERR_TIMEOUT) {
        SIE_TRY(nested_clear(op));
        return n;
    }
    return s == SIE_OK ? n : s;
}

// clear the nested-solve statistics (host and device copies; the constraint entries of
// the device copy are in the host's since the solve that made them)
sie_status nested_clear(sie_op* op)
{
    op->stats[2] = op->stats[3] = 0;
    op->wait_lost = false;
    if (op->gstat)
        SIE_CUDA_TRY(cudaMemsetAsync(op->gstat, 0, sizeof(double) * sie_op::GSTAT, op->mesh->ctx->stream));
    return SIE_OK;
}

// Row weighting of Eq. (sys) for the Krylov solves.  The charge rows
// F D H + j k0 c0 rho are larger than the current rows by the ratio of a
// divergence (~ 1 / edge length) to a Galerkin potential entry (~ area^2 G),
// about 1e16 on the benchmark's copper sphere, so in the plain 2-norm of the
// residual their FP64 rounding alone reaches 1e-3 of |b| and the Arnoldi
// estimate loses touch with the true residual.  The Krylov solves therefore
// use W A x = W b with W = diag(I, q_w I): q_w = mean_m |L_A,mm| makes the two
// diagonal blocks of the constraint preconditioner, j k0 diag(L_A) and
// j k0 I, the same size.  The solution is the same; tol_outer and the
// reported relative residual refer to |W (b - A x)| / |W b|.
static sie_status charge_weight(sie_op* op)
{
    if (op->q_w > 0) return SIE_OK;
    cudaStream_t st = op->mesh->ctx->stream;
    const int64_t ne = op->mesh->h.ne, n = ne + op->mesh->h.nt;
    std::vector<double2> d(ne);
    SIE_CUDA_TRY(cudaMemcpyAsync(d.data(), op->ext.dLA, sizeof(double2) * ne, cudaMemcpyDeviceToHost, st));
    SIE_CUDA_TRY(cudaStreamSynchronize(st));
    double sum = 0;
    for (const double2& v : d) sum += std::hypot(v.x, v.y);
    op->q_w = (ne > 0 && sum > 0 && std::isfinite(sum)) ? sum / (double)ne : 1.0;
    if (!op->bal) SIE_CUDA_TRY(cudaMallocAsync((void**)&op->bal, sizeof(double2) * 2 * n, st));
    return SIE_OK;
}

// v = W u (u, v may alias); with inv, v = W^-1 u
static sie_status weight_rows(sie_op* op, const double2* u, double2* v, bool inv)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const int64_t ne = op->mesh->h.ne, nt = op->mesh->h.nt;
    if (u != v) SIE_CUDA_TRY(cudaMemcpyAsync(v, u, sizeof(double2) * ne, cudaMemcpyDeviceToDevice, st));
    return axpby(st, nt, inv ? 1.0 / op->q_w : op->q_w, u + ne, 0.0, v + ne);
}

sie_status sys_solve(sie_op* op, const double2* b, double2* x, int* iters, double* relres)
{
    const int64_t n = op->mesh->h.ne + op->mesh->h.nt;
    SIE_TRY(charge_weight(op));
    double2* bw = op->bal;
    double2* tw = op->bal + n;
    auto A = [&](const double2* u, double2* v) {
        SIE_TRY(apply_sys_fast(op, u, v));
        return weight_rows(op, v, v, false);
    };
    auto Minv = [&](const double2* u, double2* v) {
        SIE_TRY(weight_rows(op, u, tw, true));
        return precond_sys(op, tw, v);
    };
    op->stats[4] = op->stats[5] = 0;
    SIE_TRY(nested_clear(op));
    SIE_TRY(weight_rows(op, b, bw, false));
    int it = 0;
    double rr = 0;
    sie_status s = fgmres(op->mesh->ctx, op->kout, n, A, Minv, bw, x, op->p.tol_outer, op->p.maxit, op->p.restart,
                          &it, &rr);
    op->stats[0] = it;
    op->stats[1] = rr;
    if (iters) *iters = it;
    if (relres) *relres = rr;
    s = solve_status(op, s, "sie_solve");
    if (s == SIE_OK || s == SIE_ERR_NOT_CONVERGED) SIE_TRY(constraint_lu_check(op));
    return s;
}

// |v| (host value; synchronises the stream).  part, out: device scratch.
static sie_status norm2(cudaStream_t st, int64_t n, const double2* v, double2* part, double2* out, double* h,
                        double* res)
{
    SIE_TRY(dots(st, n, 1, v, n, v, part, out));
    SIE_CUDA_TRY(cudaMemcpyAsync(h, out, sizeof(double), cudaMemcpyDeviceToHost, st));
    SIE_CUDA_TRY(cudaStreamSynchronize(st));
    *res = sqrt(fmax(h[0], 0.0));
    return SIE_OK;
}

// Mixed-precision iterative refinement of SYS x = b: the residual r = b - A x
// and the update x += d use the FP64 system product; each correction A d = r
// is solved by FGMRES with the complex64 product (SIE_MIXED: grid and exterior
// near products in FP32) and the FP64 constraint preconditioner.  Stops when
// the FP64 relative residual is below tol_outer, so the result meets the same
// criterion as the plain FP64 solve while the Krylov work runs on the faster
// product.  iters: FGMRES iterations over all corrections; relres: the final
// FP64 relative residual.
sie_status sys_solve_refined(sie_op* op, const double2* b, double2* x, int* iters, double* relres)
{
    sie_ctx* c = op->mesh->ctx;
    cudaStream_t st = c->stream;
    const int64_t n = op->mesh->h.ne + op->mesh->h.nt;
    if (!op->ir_buf) SIE_CUDA_TRY(cudaMallocAsync((void**)&op->ir_buf, sizeof(double2) * 3 * n, st));
    double2* r = op->ir_buf;
    double2* d = r + n;
    double2* t = r + 2 * n;
    SIE_TRY(op->kout.alloc(st, n, op->p.restart));
    double2* part = op->kout.part;
    double2* dot = op->kout.h;
    double* hbuf = op->kout.resid_h;
    const int saved = op->p.precision;
    SIE_TRY(charge_weight(op));
    double2* tw = op->bal + n;
    // both solves use the row-weighted system W A x = W b (charge_weight)
    auto A32 = [&](const double2* u, double2* v) {
        SIE_TRY(apply_sys_fast(op, u, v));
        return weight_rows(op, v, v, false);
    };
    auto Minv = [&](const double2* u, double2* v) {
        SIE_TRY(weight_rows(op, u, tw, true));
        return precond_sys(op, tw, v);
    };
    op->stats[4] = op->stats[5] = 0;
    SIE_TRY(nested_clear(op));
    SIE_CUDA_TRY(cudaMemsetAsync(x, 0, sizeof(double2) * n, st));
    double bn = 0, rel = 1.0;
    SIE_TRY(weight_rows(op, b, op->bal, false));
    SIE_TRY(norm2(st, n, op->bal, part, dot, hbuf, &bn));
    int total = 0;
    sie_status s = SIE_OK;
    const int SWEEPS = 10;
    // the corrections run on the complex64 product while each sweep shrinks the
    // FP64 residual by at least half; when one does not (the complex64 error,
    // amplified by cancellation in the product, bounds what it can reach),
    // the remaining corrections run on the FP64 product
    bool fp64_corr = false;
    double rel_prev = 1.0;
    for (int sweep = 0; sweep <= SWEEPS; sweep++) {
        // FP64 residual
        op->p.precision = SIE_FP64;
        if (sweep == 0) {
            SIE_CUDA_TRY(cudaMemcpyAsync(r, op->bal, sizeof(double2) * n, cudaMemcpyDeviceToDevice, st));
        } else {
            if ((s = A32(x, t)) != SIE_OK) break;
            SIE_CUDA_TRY(cudaMemcpyAsync(r, op->bal, sizeof(double2) * n, cudaMemcpyDeviceToDevice, st));
            if ((s = axpby(st, n, -1.0, t, 1.0, r)) != SIE_OK) break;
        }
        double rn = 0;
        if ((s = norm2(st, n, r, part, dot, hbuf, &rn)) != SIE_OK) break;
        rel = bn > 0 ? rn / bn : 0.0;
        if (rel < op->p.tol_outer || sweep == SWEEPS || total >= op->p.maxit) break;
        if (sweep >= 2 && rel > 0.5 * rel_prev) fp64_corr = true;
        rel_prev = rel;
        // correction on the complex64 product, to the accuracy this sweep needs
        op->p.precision = fp64_corr ? SIE_FP64 : SIE_MIXED;
        const double tc = std::min(1e-2, std::max(1e-6, 0.5 * op->p.tol_outer / rel));
        int it = 0;
        double rr = 0;
        s = fgmres(c, op->kout, n, A32, Minv, r, d, tc, op->p.maxit - total, op->p.restart, &it, &rr);
        total += it;
        if (s != SIE_OK && s != SIE_ERR_NOT_CONVERGED) break;
        s = SIE_OK;
        if ((s = axpby(st, n, 1.0, d, 1.0, x)) != SIE_OK) break;
    }
    op->p.precision = saved;
    if (s == SIE_OK) {
        op->stats[0] = total;
        op->stats[1] = rel;
        if (iters) *iters = total;
        if (relres) *relres = rel;
        SIE_TRY(constraint_lu_check(op));
        if (!(rel < op->p.tol_outer)) s = SIE_ERR_NOT_CONVERGED;
    }
    return solve_status(op, s, "sie_solve (refined)");
}

sie_status sys_rhs(sie_op* op, const double* khat, const double* epol, double2* b)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const DevMesh& M = op->mesh->d;
    SIE_CUDA_TRY(cudaMemsetAsync(b, 0, sizeof(double2) * (M.ne + M.nt), st));
    k_rhs<<<nb(M.nt), 256, 0, st>>>(M.nt, M, gl_rule(6), op->k0, make_double3(khat[0], khat[1], khat[2]),
                                    make_double3(epol[0], epol[1], epol[2]), -1.0 / ETA0, b);
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}

sie_status sys_rcs(sie_op* op, const double2* x, const double* rhat, int ndir, double* rcs)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const DevMesh& M = op->mesh->d;
    double2* E = op->sys_E;
    double nres = 0.0;
    SIE_TRY(apply_Z(op, x, E, &nres));
    double *dr = nullptr;
    double2* dout = nullptr;
    SIE_CUDA_TRY(cudaMallocAsync((void**)&dr, sizeof(double) * 3 * ndir, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&dout, sizeof(double2) * 6 * ndir, st));
    SIE_CUDA_TRY(cudaMemcpyAsync(dr, rhat, sizeof(double) * 3 * ndir, cudaMemcpyHostToDevice, st));
    k_far<<<ndir, 256, 0, st>>>(M.nt, M, gl_rule(6), op->k0, dr, x, E, dout);
    SIE_CUDA_TRY(cudaGetLastError());
    std::vector<double2> h(6 * ndir);
    SIE_CUDA_TRY(cudaMemcpyAsync(h.data(), dout, sizeof(double2) * 6 * ndir, cudaMemcpyDeviceToHost, st));
    SIE_CUDA_TRY(cudaStreamSynchronize(st));
    cudaFreeAsync(dr, st);
    cudaFreeAsync(dout, st);
    for (int d = 0; d < ndir; d++) {
        cplx NH[3], NE[3];
        for (int k = 0; k < 3; k++) {
            NH[k] = cplx(h[6 * d + k].x, h[6 * d + k].y);
            NE[k] = cplx(h[6 * d + 3 + k].x, h[6 * d + 3 + k].y);
        }
        double r[3] = {rhat[3 * d], rhat[3 * d + 1], rhat[3 * d + 2]};
        cplx rn = r[0] * NH[0] + r[1] * NH[1] + r[2] * NH[2];
        cplx v[3];
        v[0] = NH[0] - rn * r[0] + (r[1] * NE[2] - r[2] * NE[1]);
        v[1] = NH[1] - rn * r[1] + (r[2] * NE[0] - r[0] * NE[2]);
        v[2] = NH[2] - rn * r[2] + (r[0] * NE[1] - r[1] * NE[0]);
        double s = std::norm(v[0]) + std::norm(v[1]) + std::norm(v[2]);
        rcs[d] = op->k0 * op->k0 * ETA0 * ETA0 / (4 * M_PI) * s;
    }
    if (nres >= op->p.tol_inner) {
        set_error("sie_rcs: the nested interior solve of Z_i H ended at relative residual " + std::to_string(nres) +
                  " >= tol_inner");
        return SIE_ERR_NOT_CONVERGED;
    }
    return SIE_OK;
}

// True when Z' H can run without allocating: the interior FGMRES workspace (and,
// for an interior on the AIM grid, the nested constraint solver's) already has
// the sizes the solves use, as after a solve or a SYS product on this operator.
bool sys_z_workspace_ready(const sie_op* op)
{
    const int64_t ne = op->mesh->h.ne, nt = op->mesh->h.nt;
    if (op->kin.n != ne || op->kin.m != inner_m(op)) return false;
    if (op->inn.has_grid && (op->kcs_in.n != nt || op->kcs_in.m != op->p.constraint_restart)) return false;
    return true;
}

// E' = Z' x[0:ne] into op->sys_E, then the far-field sums N(H), N(E') of the
// directions rhat_d (device, 3 doubles each) into sums (device, 6 complex per
// direction): the device half of sys_rcs, with caller-owned buffers.
sie_status sys_far_sums(sie_op* op, const double2* x, const double* rhat_d, int ndir, double2* sums,
                        double* nested_res)
{
    cudaStream_t st = op->mesh->ctx->stream;
    SIE_TRY(apply_Z(op, x, op->sys_E, nested_res));
    k_far<<<ndir, 256, 0, st>>>(op->mesh->d.nt, op->mesh->d, gl_rule(6), op->k0, rhat_d, x, op->sys_E, sums);
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}

// ------------------------------------------------------------------ Krylov workspace of several right-hand sides
// per right-hand side sizes inside a PanelWork
static int64_t pw_p(int m) { return (int64_t)RES_MAXCTA * 2 * (m + 2); }
static int64_t pw_h(int m) { return 2 * (int64_t)(m + 2); }
static int64_t pw_d(int m) { return (int64_t)(m + 1) * m + 2 * m + 2 * (m + 1); }
static int64_t pw_s(int m) { return 8 + m + 1; }

sie_status PanelWork::alloc(cudaStream_t st, int64_t n_, int m_, int R_)
{
    if (n_ == n && m_ == m && R_ == R) return SIE_OK;
    release(st);
    n = n_;
    m = m_;
    R = R_;
    SIE_CUDA_TRY(cudaMallocAsync((void**)&V, sizeof(double2) * (m + 1) * R * n, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&Z, sizeof(double2) * m * R * n, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&W, sizeof(double2) * R * n, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&Rv, sizeof(double2) * R * n, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&P, sizeof(double2) * R * pw_p(m), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&h, sizeof(double2) * R * pw_h(m), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&Hd, sizeof(double2) * R * pw_d(m), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&part, sizeof(double2) * R * DOT_CHUNKS, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&wd, sizeof(double2) * R, st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&sc, sizeof(double) * R * pw_s(m), st));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&res, sizeof(double) * R * (m + 1), st));
    SIE_CUDA_TRY(cudaMallocHost((void**)&res_h, sizeof(double) * R * (m + 1)));
    ev.resize(m + 1);
    for (auto& e : ev) SIE_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    return SIE_OK;
}

void PanelWork::release(cudaStream_t st)
{
    for (double2* p : {V, Z, W, Rv, P, h, Hd, part, wd})
        if (p) cudaFreeAsync(p, st);
    for (double* p : {sc, res})
        if (p) cudaFreeAsync(p, st);
    if (res_h) {
        cudaStreamSynchronize(st);
        cudaFreeHost(res_h);
    }
    for (auto& e : ev) cudaEventDestroy(e);
    ev.clear();
    V = Z = W = Rv = P = h = Hd = part = wd = nullptr;
    sc = res = res_h = nullptr;
    n = 0;
    m = R = 0;
}

// ------------------------------------------------------------------ several right-hand sides in lockstep
// y_q = Op x_q for q < R: a non-owning reference to a block operator
class BlockApply {
    const void* obj_ = nullptr;
    sie_status (*call_)(const void*, int, const double2* const*, double2* const*) = nullptr;

public:
    template <class F>
    BlockApply(const F& f)  // NOLINT: implicit from a named callable
        : obj_(&f), call_([](const void* o, int R, const double2* const* x, double2* const* y) {
              return (*static_cast<const F*>(o))(R, x, y);
          })
    {
    }
    sie_status operator()(int R, const double2* const* x, double2* const* y) const { return call_(obj_, R, x, y); }
};

// R restarted flexible GMRES iterations in lockstep: one Krylov basis per
// right-hand side (K.V + q (m + 1) n), the operator and the preconditioner applied
// to the R current vectors at once (so a block implementation reads its data
// once for all of them), every Gram-Schmidt and Givens step one launch for all R
// (PanelStrides) and one residual copy.  The cycle ends when every residual is
// below tol (a converged right-hand side keeps iterating with the others, which
// only lowers its residual); restarts from the true residuals.  iters: iterations
// run (the same for all), relres[q]: final relative residual of q.
static sie_status fgmres_multi(sie_ctx* c, PanelWork& K, int R, int64_t n, const BlockApply& A, const BlockApply& Minv,
                               const double2* const* b, double2* const* x, double tol, int maxit, int restart,
                               int* iters_out, double* relres_out, int lag = 1)
{
    cudaStream_t st = c->stream;
    const int m = restart;
    SIE_TRY(K.alloc(st, n, m, R));
    PanelStrides ps;
    ps.v = (int64_t)(m + 1) * n;
    ps.w = n;
    ps.p = pw_p(m);
    ps.h = pw_h(m);
    ps.d = pw_d(m);
    ps.s = pw_s(m);
    double2* cs = K.Hd + (m + 1) * m;
    double2* sn = cs + m;
    double2* g = sn + m;
    double2* y = g + (m + 1);
    double2* h2 = K.h + (m + 2);
    double2* P2 = K.P + (int64_t)CGS_CHUNKS * (m + 1);
    double2* P3 = K.P + (int64_t)2 * CGS_CHUNKS * (m + 1);
    for (int q = 0; q < R; q++) {
        SIE_CUDA_TRY(cudaMemsetAsync(x[q], 0, sizeof(double2) * n, st));
        SIE_TRY(dots(st, n, 1, b[q], n, b[q], K.part + q * DOT_CHUNKS, K.wd + q));
        k_gm_start<<<nb(n), 256, 0, st>>>(n, b[q], K.wd + q, K.V + q * ps.v, g + q * ps.d, m, K.sc + q * ps.s, 1);
    }
    SIE_CUDA_TRY(cudaGetLastError());
    int it = 0;
    double rel[MULTI_RHS];
    for (int q = 0; q < R; q++) rel[q] = 1.0;
    const int LAG = lag;
    auto all_below = [&](const double* v) {
        for (int q = 0; q < R; q++)
            if (!(v[q] < tol)) return false;
        return true;
    };
    auto finite = [&](const double* v) {
        for (int q = 0; q < R; q++)
            if (!std::isfinite(v[q])) {
                set_error("GMRES: the residual is not finite (non-finite right-hand side or operator)");
                return false;
            }
        return true;
    };
    const dim3 grid(CGS_CHUNKS, R);
    while (true) {
        int j = 0;
        bool conv = false;
        for (; j < m && it < maxit; j++) {
            const double2* vj[MULTI_RHS];
            double2 *zj[MULTI_RHS], *wq[MULTI_RHS];
            for (int q = 0; q < R; q++) {
                vj[q] = K.V + q * ps.v + (int64_t)j * n;
                zj[q] = K.Z + ((int64_t)q * m + j) * n;
                wq[q] = K.W + q * n;
            }
            SIE_TRY(Minv(R, vj, zj));
            SIE_TRY(A(R, zj, wq));
            k_cgs_part<<<grid, 256, 0, st>>>(n, j + 1, K.V, n, K.W, K.P, m + 1, ps);
            k_cgs_update<<<grid, 256, 0, st>>>(n, j + 1, K.V, n, K.P, m + 1, K.h, K.W, P2, 0, ps);
            k_cgs_update<<<grid, 256, 0, st>>>(n, j + 1, K.V, n, P2, m + 1, h2, K.W, P3, 1, ps);
            k_cgs_finish<<<grid, 256, 0, st>>>(n, j, m, K.h, h2, P3, K.W, K.V, K.Hd, cs, sn, g, K.sc, ps, n, K.res);
            SIE_CUDA_TRY(cudaGetLastError());
            SIE_CUDA_TRY(cudaMemcpyAsync(K.res_h + (int64_t)j * R, K.res + (int64_t)j * R, sizeof(double) * R,
                                         cudaMemcpyDeviceToHost, st));
            SIE_CUDA_TRY(cudaEventRecord(K.ev[j], st));
            it++;
            if (j >= LAG) {
                SIE_CUDA_TRY(cudaEventSynchronize(K.ev[j - LAG]));
                const double* v = K.res_h + (int64_t)(j - LAG) * R;
                if (!finite(v)) return SIE_ERR_ARG;
                if (all_below(v)) {
                    conv = true;
                    j++;
                    break;
                }
            }
        }
        const int jend = j - 1;
        SIE_CUDA_TRY(cudaEventSynchronize(K.ev[jend]));
        for (int q = 0; q < R; q++) rel[q] = K.res_h[(int64_t)jend * R + q];
        if (!finite(rel)) return SIE_ERR_ARG;
        for (int q = 0; q < R; q++) {
            k_gm_backsub<<<1, 1, 0, st>>>(jend, m, K.Hd + q * ps.d, g + q * ps.d, y + q * ps.d);
            k_gemv<<<nb(n), 256, 0, st>>>(n, jend + 1, K.Z + (int64_t)q * m * n, n, y + q * ps.d, 1.0, x[q]);
        }
        SIE_CUDA_TRY(cudaGetLastError());
        if (all_below(rel)) conv = true;
        if (conv || it >= maxit) break;
        // restart from the true residuals
        double2* wq[MULTI_RHS];
        for (int q = 0; q < R; q++) wq[q] = K.W + q * n;
        SIE_TRY(A(R, x, wq));
        double hb[2 * MULTI_RHS];
        for (int q = 0; q < R; q++) {
            double2* r = K.Rv + q * n;
            SIE_CUDA_TRY(cudaMemcpyAsync(r, b[q], sizeof(double2) * n, cudaMemcpyDeviceToDevice, st));
            SIE_TRY(axpby(st, n, -1.0, wq[q], 1.0, r));
            SIE_TRY(dots(st, n, 1, r, n, r, K.part + q * DOT_CHUNKS, K.wd + q));
            k_gm_start<<<nb(n), 256, 0, st>>>(n, r, K.wd + q, K.V + q * ps.v, g + q * ps.d, m, K.sc + q * ps.s, 0);
            SIE_CUDA_TRY(cudaMemcpyAsync(hb + 2 * q, K.sc + q * ps.s, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
        }
        SIE_CUDA_TRY(cudaGetLastError());
        SIE_CUDA_TRY(cudaStreamSynchronize(st));
        for (int q = 0; q < R; q++) rel[q] = hb[2 * q] > 0 ? hb[2 * q + 1] / hb[2 * q] : 0.0;
        if (all_below(rel)) break;
    }
    for (int q = 0; q < R; q++) {
        if (iters_out) iters_out[q] = it;
        if (relres_out) relres_out[q] = rel[q];
    }
    return all_below(rel) ? SIE_OK : SIE_ERR_NOT_CONVERGED;
}

// E_q = Z' H_q for R vectors (near-region-only or SIBC interiors; H_q ldh apart, E_q
// ne apart): right-hand sides and products as CSR x panel products (block.cu), the
// iterations in lockstep (near-only: A = L_i,NR, M = its sparse approximate inverse;
// SIBC: A = Gram, M = Jacobi), then the impedance factor
static sie_status apply_Z_panel(sie_op* op, int R, const double2* H, int64_t ldh, double2* E)
{
    sie_ctx* c = op->mesh->ctx;
    cudaStream_t st = c->stream;
    const int64_t ne = op->mesh->h.ne;
    AimOp& I = op->inn;
    const bool sibc = op->p.interior_model == SIE_SIBC;
    double2* a = op->zp + MULTI_RHS * ne;      // right-hand sides
    double2* t = op->zp + 2 * MULTI_RHS * ne;  // scratch
    // I-cross H (weight -1/2 for GIBC, +1 for SIBC)
    SIE_TRY(blk_csr(st, (int)ne, op->ix_row_ptr, op->ix_col, op->ix_val, H, ldh, R, sibc ? a : t, ne));
    if (!sibc) {
        SIE_TRY(blk_csr(st, (int)ne, I.row_ptr, I.col, I.valK, H, ldh, R, a, ne));
        SIE_TRY(axpby(st, R * ne, -0.5, t, 1.0, a));
    }
    // the R vectors of a block lie one distance apart
    auto product = [&](const int64_t* rp, const int32_t* col, const double2* val, const double2* const* x,
                       double2* const* y) {
        return blk_csr(st, (int)ne, rp, col, val, x[0], R > 1 ? x[1] - x[0] : 0, R, y[0], R > 1 ? y[1] - y[0] : 0);
    };
    auto A = [&](int, const double2* const* x, double2* const* y) {
        return sibc ? product(op->gr_row_ptr, op->gr_col, op->gr_val, x, y) : product(I.row_ptr, I.col, I.valL, x, y);
    };
    auto M = [&](int, const double2* const* x, double2* const* y) -> sie_status {
        if (!sibc) return product(I.row_ptr, I.col, I.valM, x, y);
        for (int q = 0; q < R; q++)
            k_jacobi<<<nb(ne), 256, 0, st>>>(ne, x[q], op->gr_diag, make_double2(1.0, 0.0), y[q]);
        SIE_CUDA_TRY(cudaGetLastError());
        return SIE_OK;
    };
    const double2* b[MULTI_RHS];
    double2* e[MULTI_RHS];
    for (int q = 0; q < R; q++) b[q] = a + q * ne, e[q] = E + q * ne;
    const int m_in = inner_m(op);
    int it[MULTI_RHS];
    double rr[MULTI_RHS];
    {
        Stage s_(c, "inner_solve");
        const sie_status s = fgmres_multi(c, op->kzp, R, ne, A, M, b, e, op->p.tol_inner, m_in, m_in, it, rr);
        if (s != SIE_OK && s != SIE_ERR_NOT_CONVERGED) return s;
    }
    for (int q = 0; q < R; q++) {
        op->stats[2] = std::max(op->stats[2], (double)it[q]);
        op->stats[3] = std::max(op->stats[3], rr[q]);
    }
    if (op->edge_zf) {
        for (int q = 0; q < R; q++) k_scale_edges<<<nb(ne), 256, 0, st>>>(ne, op->edge_zf, e[q]);
        SIE_CUDA_TRY(cudaGetLastError());
        return SIE_OK;
    }
    cplx f;
    if (sibc) {
        f = cplx(op->eta_re, op->eta_im);
    } else {
        cplx zs(0.0, op->k0 * op->eps_r);
        zs += op->sigma * ETA0;
        f = -1.0 / zs;
    }
    return axpby(st, R * ne, f, E, 0.0, E);
}

// y_q = SYS x_q for R vectors: near-region-only and SIBC interiors as one block
// product (block.cu), the complex64 product and AIM interiors one vector at a time
static sie_status apply_sys_multi(sie_op* op, int R, const double2* const* x, double2* const* y)
{
    if (op->inn.has_grid) {
        for (int q = 0; q < R; q++) SIE_TRY(apply_sys(op, x[q], y[q]));
        return SIE_OK;
    }
    cudaStream_t st = op->mesh->ctx->stream;
    const int64_t ne = op->mesh->h.ne;
    if (!op->zp) SIE_CUDA_TRY(cudaMallocAsync((void**)&op->zp, sizeof(double2) * 3 * MULTI_RHS * ne, st));
    double2* Ep = op->zp;
    // the R vectors of a block lie one distance apart
    const int64_t ldx = R > 1 ? x[1] - x[0] : 0, ldy = R > 1 ? y[1] - y[0] : 0;
    SIE_TRY(apply_Z_panel(op, R, x[0], ldx, Ep));
    if (op->p.precision != SIE_MIXED) return blk_sys_rest(op, R, x[0], ldx, Ep, ne, y[0], ldy);
    double2* yb = op->sys_tmp + ne + 2 * op->mesh->h.nt;
    for (int q = 0; q < R; q++) {
        SIE_TRY(sys_charge(op, st, x[q], x[q] + ne, yb, y[q] + ne));
        SIE_TRY(sys_near(op, st, x[q], Ep + q * ne, yb));
        SIE_CUDA_TRY(cudaMemsetAsync(y[q], 0, sizeof(double2) * ne, st));
        SIE_TRY(sys_grid(op, x[q], Ep + q * ne, x[q] + ne, y[q]));
        SIE_TRY(axpby(st, ne, 1.0, yb, 1.0, y[q]));
    }
    return SIE_OK;
}

// scratch of the lockstep solves: per right-hand side the weighted input of
// the preconditioner, the weighted right-hand side and the preconditioner's
// vectors (ne: v1', t1, te and the triangle operator's te; nt: sigma, phi,
// charge rhs, charges and the triangle operator's phi)
static int64_t multi_stride(const sie_op* op)
{
    return 2 * (op->mesh->h.ne + op->mesh->h.nt) + 4 * op->mesh->h.ne + 5 * op->mesh->h.nt;
}

static sie_status multi_scratch(sie_op* op)
{
    if (op->mscr) return SIE_OK;
    const int64_t n = op->mesh->h.ne + op->mesh->h.nt;
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->mscr, sizeof(double2) * MULTI_RHS * multi_stride(op),
                                 op->mesh->ctx->stream));
    SIE_CUDA_TRY(cudaMallocAsync((void**)&op->ir_multi, sizeof(double2) * 3 * MULTI_RHS * n, op->mesh->ctx->stream));
    return SIE_OK;
}

// the constraint preconditioner (precond_sys) for R vectors: the sparse
// steps per vector, the R triangle systems by lockstep GMRES whose
// preconditioner is one pass over the dense inverse for all of them
// (DenseLU::solve_multi); without a factorisation, and for penetrable objects, whose
// products are made one vector at a time anyway, precond_sys for each
static sie_status precond_sys_multi(sie_op* op, int R, const double2* const* x, double2* const* y)
{
    AimOp& X = op->ext;
    if (!X.lu || (op->inn.has_grid && op->mesh->h.nt <= CLU_MAXN)) {
        for (int q = 0; q < R; q++) SIE_TRY(precond_sys(op, x[q], y[q]));
        return SIE_OK;
    }
    sie_ctx* c = op->mesh->ctx;
    cudaStream_t st = c->stream;
    const DevMesh& M = op->mesh->d;
    const int64_t ne = M.ne, nt = M.nt, n = ne + nt;
    const cplx jk0(0.0, op->k0);
    const cplx kappa = 1.0 / (op->k0 * op->k0);
    auto lphi = [&](const double2* u, double2* v) {
        SIE_CUDA_TRY(csr_launch_g(st, BLK_TRI_LANES, (int)nt, X.tri_row_ptr, X.tri_col, X.valLphiNR, u,
                                  make_double2(1.0, 0.0), false, v));
        return SIE_OK;
    };
    double2 *v1p[MULTI_RHS], *t1[MULTI_RHS], *te[MULTI_RHS], *sig[MULTI_RHS], *ph[MULTI_RHS];
    double2 *rq[MULTI_RHS], *qv[MULTI_RHS], *ste[MULTI_RHS], *sph[MULTI_RHS];
    for (int q = 0; q < R; q++) {
        double2* base = op->mscr + q * multi_stride(op) + 2 * n;
        v1p[q] = base;
        t1[q] = base + ne;
        te[q] = base + 2 * ne;
        ste[q] = base + 3 * ne;
        sig[q] = base + 4 * ne;
        ph[q] = sig[q] + nt;
        rq[q] = ph[q] + nt;
        qv[q] = rq[q] + nt;
        sph[q] = qv[q] + nt;
    }
    for (int q = 0; q < R; q++) {
        // v1' = v1 - (j k0)^-1 D^T Lphi B v2, then the charge right-hand side D Dg^-1 v1'
        k_sigma<<<nb(nt), 256, 0, st>>>((int)nt, M.area, x[q] + ne, sig[q]);
        SIE_TRY(lphi(sig[q], ph[q]));
        SIE_CUDA_TRY(cudaMemsetAsync(v1p[q], 0, sizeof(double2) * ne, st));
        k_dt<<<nb(ne), 256, 0, st>>>((int)ne, M.edge_tri, op->elen, ph[q], v1p[q]);
        SIE_TRY(axpby(st, ne, 1.0, x[q], -1.0 / jk0, v1p[q]));
        k_jacobi<<<nb(ne), 256, 0, st>>>(ne, v1p[q], X.dLA, make_double2(1.0, 0.0), t1[q]);
        k_D<<<nb(nt), 256, 0, st>>>((int)nt, M, t1[q], rq[q]);
    }
    SIE_CUDA_TRY(cudaGetLastError());
    // triangle operator S q = q - kappa D Dg^-1 D^T Lphi q for each vector
    auto S = [&](int Rn, const double2* const* u, double2* const* v) {
        for (int q = 0; q < Rn; q++) {
            SIE_TRY(lphi(u[q], sph[q]));
            SIE_CUDA_TRY(cudaMemsetAsync(ste[q], 0, sizeof(double2) * ne, st));
            k_dt<<<nb(ne), 256, 0, st>>>((int)ne, M.edge_tri, op->elen, sph[q], ste[q]);
            k_jacobi<<<nb(ne), 256, 0, st>>>(ne, ste[q], X.dLA, make_double2(1.0, 0.0), ste[q]);
            k_D<<<nb(nt), 256, 0, st>>>((int)nt, M, ste[q], v[q]);
            SIE_CUDA_TRY(cudaGetLastError());
            SIE_TRY(axpby(st, nt, 1.0, u[q], -kappa, v[q]));
        }
        return SIE_OK;
    };
    auto LU = [&](int Rn, const double2* const* u, double2* const* v) {
        Stage s_(c, "constraint_lu_solve");
        return X.lu->solve_multi(st, Rn, u, v);
    };
    {
        int it[MULTI_RHS];
        double rr[MULTI_RHS];
        Stage s_(c, "constraint_solve");
        sie_status s = fgmres_multi(c, op->kcs_multi, R, nt, S, LU, rq, qv, op->p.tol_constraint,
                                    op->p.constraint_maxit, std::min(op->p.constraint_restart, 20), it, rr, 0);
        if (s != SIE_OK && s != SIE_ERR_NOT_CONVERGED) return s;
        for (int q = 0; q < R; q++) {
            op->stats[4] = std::max(op->stats[4], (double)it[q]);
            op->stats[5] = std::max(op->stats[5], rr[q]);
        }
    }
    for (int q = 0; q < R; q++) {
        // y1 = (j k0)^-1 Dg^-1 (v1' + kappa D^T Lphi q)
        SIE_TRY(lphi(qv[q], ph[q]));
        SIE_CUDA_TRY(cudaMemsetAsync(te[q], 0, sizeof(double2) * ne, st));
        k_dt<<<nb(ne), 256, 0, st>>>((int)ne, M.edge_tri, op->elen, ph[q], te[q]);
        SIE_TRY(axpby(st, ne, kappa, te[q], 0.0, te[q]));
        SIE_TRY(axpby(st, ne, 1.0, v1p[q], 1.0, te[q]));
        k_jacobi<<<nb(ne), 256, 0, st>>>(ne, te[q], X.dLA, make_double2(1.0, 0.0), y[q]);
        SIE_TRY(axpby(st, ne, 1.0 / jk0, y[q], 0.0, y[q]));
        // y2 = (v2 - F D y1) / (j k0)
        k_D<<<nb(nt), 256, 0, st>>>((int)nt, M, y[q], ph[q]);
        k_fdiv_area<<<nb(nt), 256, 0, st>>>((int)nt, M.area, ph[q]);
        SIE_CUDA_TRY(cudaMemcpyAsync(y[q] + ne, x[q] + ne, sizeof(double2) * nt, cudaMemcpyDeviceToDevice, st));
        SIE_TRY(axpby(st, nt, -1.0 / jk0, ph[q], 1.0 / jk0, y[q] + ne));
    }
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}

// Eq. (sys) for R right-hand sides in lockstep (row-weighted as in sys_solve):
// plain FP64 FGMRES, or (refine) the mixed-precision refinement of
// sys_solve_refined with every sweep's corrections solved in lockstep.
// iters[q], relres[q] as for one right-hand side.
sie_status sys_solve_multi(sie_op* op, int R, const double2* const* b, double2* const* x, int* iters, double* relres,
                           bool refine)
{
    if (R < 1 || R > MULTI_RHS) {
        set_error("sys_solve_multi: 1 to 8 right-hand sides");
        return SIE_ERR_ARG;
    }
    sie_ctx* c = op->mesh->ctx;
    cudaStream_t st = c->stream;
    const int64_t n = op->mesh->h.ne + op->mesh->h.nt;
    SIE_TRY(charge_weight(op));
    SIE_TRY(multi_scratch(op));
    double2 *tw[MULTI_RHS], *bw[MULTI_RHS];
    for (int q = 0; q < R; q++) {
        tw[q] = op->mscr + q * multi_stride(op);
        bw[q] = tw[q] + n;
    }
    // the block product (panel nested solves), or one product per vector
    // (graph replays) with SIE_BLOCK_PRODUCT=0 in the environment
    static const bool block = [] {
        const char* e = getenv("SIE_BLOCK_PRODUCT");
        return !(e && e[0] == '0');
    }();
    auto A = [&](int Rn, const double2* const* u, double2* const* v) {
        if (block && Rn > 1) {
            SIE_TRY(apply_sys_multi(op, Rn, u, v));
        } else {
            for (int q = 0; q < Rn; q++) SIE_TRY(apply_sys_fast(op, u[q], v[q]));
        }
        for (int q = 0; q < Rn; q++) SIE_TRY(weight_rows(op, v[q], v[q], false));
        return SIE_OK;
    };
    auto Minv = [&](int Rn, const double2* const* u, double2* const* v) {
        for (int q = 0; q < Rn; q++) SIE_TRY(weight_rows(op, u[q], tw[q], true));
        return precond_sys_multi(op, Rn, tw, v);
    };
    op->stats[4] = op->stats[5] = 0;
    SIE_TRY(nested_clear(op));
    for (int q = 0; q < R; q++) SIE_TRY(weight_rows(op, b[q], bw[q], false));
    int it[MULTI_RHS];
    double rr[MULTI_RHS];
    sie_status s = SIE_OK;
    if (!refine) {
        s = fgmres_multi(c, op->kmulti, R, n, A, Minv, bw, x, op->p.tol_outer, op->p.maxit, op->p.restart, it, rr);
        if (s != SIE_OK && s != SIE_ERR_NOT_CONVERGED) return solve_status(op, s, "sie_solve");
    } else {
        double2 *r[MULTI_RHS], *d[MULTI_RHS], *t[MULTI_RHS];
        for (int q = 0; q < R; q++) {
            r[q] = op->ir_multi + (int64_t)q * n;
            d[q] = op->ir_multi + (int64_t)(MULTI_RHS + q) * n;
            t[q] = op->ir_multi + (int64_t)(2 * MULTI_RHS + q) * n;
            SIE_CUDA_TRY(cudaMemsetAsync(x[q], 0, sizeof(double2) * n, st));
        }
        PanelWork& K0 = op->kmulti;
        SIE_TRY(K0.alloc(st, n, op->p.restart, R));
        double bn[MULTI_RHS], rel[MULTI_RHS], rel_prev = 1.0;
        for (int q = 0; q < R; q++) SIE_TRY(norm2(st, n, bw[q], K0.part, K0.wd, K0.res_h, &bn[q]));
        const int saved = op->p.precision;
        const int SWEEPS = 10;
        bool fp64_corr = false;
        int total = 0;
        for (int sweep = 0; sweep <= SWEEPS; sweep++) {
            op->p.precision = SIE_FP64;
            if (sweep > 0 && (s = A(R, x, t)) != SIE_OK) break;
            double worst = 0;
            for (int q = 0; q < R && s == SIE_OK; q++) {
                SIE_CUDA_TRY(cudaMemcpyAsync(r[q], bw[q], sizeof(double2) * n, cudaMemcpyDeviceToDevice, st));
                if (sweep > 0) s = axpby(st, n, -1.0, t[q], 1.0, r[q]);
                double rn = 0;
                if (s == SIE_OK) s = norm2(st, n, r[q], K0.part, K0.wd, K0.res_h, &rn);
                rel[q] = bn[q] > 0 ? rn / bn[q] : 0.0;
                worst = std::max(worst, rel[q]);
            }
            if (s != SIE_OK) break;
            if (worst < op->p.tol_outer || sweep == SWEEPS || total >= op->p.maxit) break;
            if (sweep >= 2 && worst > 0.5 * rel_prev) fp64_corr = true;
            rel_prev = worst;
            op->p.precision = fp64_corr ? SIE_FP64 : SIE_MIXED;
            const double tc = std::min(1e-2, std::max(1e-6, 0.5 * op->p.tol_outer / worst));
            int itc[MULTI_RHS];
            double rrc[MULTI_RHS];
            s = fgmres_multi(c, op->kmulti, R, n, A, Minv, r, d, tc, op->p.maxit - total, op->p.restart, itc, rrc);
            total += itc[0];
            if (s != SIE_OK && s != SIE_ERR_NOT_CONVERGED) break;
            s = SIE_OK;
            for (int q = 0; q < R && s == SIE_OK; q++) s = axpby(st, n, 1.0, d[q], 1.0, x[q]);
            if (s != SIE_OK) break;
        }
        op->p.precision = saved;
        if (s != SIE_OK) return solve_status(op, s, "sie_solve");
        for (int q = 0; q < R; q++) {
            it[q] = total;
            rr[q] = rel[q];
        }
        s = SIE_OK;
        for (int q = 0; q < R; q++)
            if (!(rr[q] < op->p.tol_outer)) s = SIE_ERR_NOT_CONVERGED;
    }
    double itmax = 0, rrmax = 0;
    for (int q = 0; q < R; q++) {
        if (iters) iters[q] = it[q];
        if (relres) relres[q] = rr[q];
        itmax = std::max(itmax, (double)it[q]);
        rrmax = std::max(rrmax, rr[q]);
    }
    op->stats[0] = itmax;
    op->stats[1] = rrmax;
    s = solve_status(op, s, "sie_solve");
    if (s == SIE_OK || s == SIE_ERR_NOT_CONVERGED) SIE_TRY(constraint_lu_check(op));
    return s;
}

// k0^2 eta0^2 / (4 pi): sigma = scale |N_perp(H) + rhat x N(E')|^2
double sys_rcs_scale(const sie_op* op) { return op->k0 * op->k0 * ETA0 * ETA0 / (4 * M_PI); }

}  // namespace sie

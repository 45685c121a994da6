// Resident FGMRES: one kernel runs a whole Krylov cycle.  The small systems
// solved inside every system product and preconditioner (interior impedance,
// charge system) need a few microseconds of arithmetic per iteration; as a graph
// loop of nine kernels an iteration took 45 to 50 us.  Two forms:
//
//  * clu_fgmres (up to CLU_MAXN rows): a thread-block cluster of 8 or 16 CTAs.  The
//    vector that the next product gathers from sits whole in every CTA's shared
//    memory, written by its owners through distributed shared memory; so are the CTAs'
//    partial sums.  An iteration meets at 3 or 4 hardware cluster barriers (0.2 to 0.3
//    us) and reads no other memory than the matrix rows (L1) and own rows of the basis;
//  * res_fgmres (more rows): a cooperative grid of up to one CTA per SM with
//    barriers in global memory (about 1.5 us); what other CTAs wrote is read past
//    L1 (ld.cg).  On 8 CTAs a copper bar's 504-row solve took 186 us this way.
//
// CTA c owns the rows [r0, r1) of every vector.  Every CTA sums the partial sums
// in the same fixed order and repeats the Givens rotations, so all take the same
// decisions and a run's rounding does not depend on timing.  Classical
// Gram-Schmidt twice; the second pass's norm is |w|^2 - |h2|^2 (h2 is at rounding
// level, so nothing cancels), which saves a reduction.
//
// Waits in global memory are bounded: a CTA that gives up sets *err and returns,
// the others run out at their next wait, and the call that reads the status reports
// SIE_ERR_TIMEOUT whatever else came of the unwritten result.
// Launches whose CTAs wait on one another that way are cooperative.
#pragma once
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace sie {

constexpr int RES_T = 512;              // threads per CTA
constexpr int RES_MAXCTA = 160;         // partial-sum slots
constexpr int RES_SPIN = 1 << 20;       // polls of a barrier before it gives up (under a second)

__device__ __forceinline__ double2 r_cm(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 r_cj(double2 a) { return make_double2(a.x, -a.y); }
// c + a b
__device__ __forceinline__ void r_fma(double2& c, double2 a, double2 b)
{
    c.x = fma(a.x, b.x, fma(-a.y, b.y, c.x));
    c.y = fma(a.x, b.y, fma(a.y, b.x, c.y));
}

struct ResBar {
    unsigned* cnt;   // zero at the launch
    int* err;
    int polls;
    unsigned target;
};
// false: the wait ran out
__device__ __forceinline__ bool res_barrier(ResBar& b)
{
    __shared__ int bad;
    b.target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(b.cnt) : "memory");
        unsigned v = 0;
        int it = 0;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(b.cnt) : "memory");
            if (++it > b.polls) ok = 0;
        } while (ok && v < b.target);
        if (!ok) atomicExch(b.err, 1);
        bad = !ok;
    }
    __syncthreads();
    return !bad;
}

// Krylov arrays; part: per-CTA sums
struct ResKrylov {
    int64_t n;
    int m;              // largest cycle length
    double2 *V, *Z, *W; // (m + 1) n, m n, n
    double2* H;         // rotated Hessenberg columns, (m + 1) m
    double2* part;      // RES_MAXCTA 2 (m + 2)
    double tol;
    int extra;          // iterations run after the residual is below tol (host-checked cycles ran one)
    double* stat;       // 0, 1: largest iteration count and residual so far; 2, 3: this run's residual and count
};

// dynamic shared memory of res_fgmres
inline size_t res_smem(int m) { return sizeof(double2) * (size_t)5 * (m + 2); }

// sums of both components over the warp, in every lane: the halves of the warp
// take one component each after the first exchange (6 FP64 additions, not 10)
__device__ __forceinline__ double2 warp_sum(double2 s)
{
    const bool up = threadIdx.x & 16;
    double keep = up ? s.y : s.x;
    keep += __shfl_xor_sync(0xffffffffu, up ? s.x : s.y, 16);
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) keep += __shfl_xor_sync(0xffffffffu, keep, off);
    const double other = __shfl_xor_sync(0xffffffffu, keep, 16);
    return up ? make_double2(other, keep) : make_double2(keep, other);
}

// part[c ld + i] = sum over own rows of conj(V_i) w, i < nv, and of |w|^2 (slot nv) when norm
__device__ __forceinline__ void res_dots(const ResKrylov& K, int64_t r0, int64_t r1, int nv, bool norm, double2* part,
                                         int ld)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int i = warp; i < nv + (norm ? 1 : 0); i += nw) {
        const double2* v = i < nv ? K.V + (int64_t)i * K.n : K.W;
        double2 s = make_double2(0, 0);
        for (int64_t k = r0 + lane; k < r1; k += 32) r_fma(s, r_cj(v[k]), K.W[k]);
        s = warp_sum(s);
        if (lane == 0) part[(int64_t)blockIdx.x * ld + i] = s;
    }
}

// h[i] = sum over the CTAs of part (in CTA order per lane, then a fixed tree)
__device__ __forceinline__ void res_reduce(int cols, const double2* part, int ld, double2* h)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int i = warp; i < cols; i += nw) {
        double2 s = make_double2(0, 0);
        for (int c = lane; c < (int)gridDim.x; c += 32) {
            const double2 p = __ldcg(part + (int64_t)c * ld + i);
            s.x += p.x;
            s.y += p.y;
        }
        s = warp_sum(s);
        if (lane == 0) h[i] = s;
    }
    __syncthreads();
}

// w -= sum_i V_i h_i on own rows
__device__ __forceinline__ void res_update(const ResKrylov& K, int64_t r0, int64_t r1, int nv, const double2* h)
{
    for (int64_t k = r0 + threadIdx.x; k < r1; k += blockDim.x) {
        double2 s = make_double2(0, 0);
        for (int i = 0; i < nv; i++) r_fma(s, K.V[(int64_t)i * K.n + k], h[i]);
        K.W[k] = make_double2(K.W[k].x - s.x, K.W[k].y - s.y);
    }
    __syncthreads();
}

// 2^-exponent of the largest of three magnitudes (1 for zero, infinity and NaN)
__device__ __forceinline__ double res_unscale(double a, double b, double c)
{
    const int m = max(max(__double2hiint(a) & 0x7fffffff, __double2hiint(b) & 0x7fffffff), __double2hiint(c) & 0x7fffffff);
    const int e = m >> 20;
    return (e == 0 || e == 0x7ff) ? 1.0 : __hiloint2double((2046 - min(e, 2045)) << 20, 0);
}

// column j (one thread): h1 + h2 and the norm hn through
// the previous rotations, rotation j (c real), g; the rotated column to Hq when
// store; gabs = |g_j| becomes |g_{j+1}|.  One chain of FP64 operations of one warp,
// 64 cycles or more each: two reciprocal square roots instead of three hypot and six
// divisions (13,600 cycles an iteration with those, a third of it)
__device__ __forceinline__ void res_givens(int j, int m, const double2* a1, const double2* a2, double hn, double2* c_,
                                           double2* s_, double2* g_, double2* Hq, bool store, double& gabs)
{
    double2 a = make_double2(a1[0].x + a2[0].x, a1[0].y + a2[0].y);
    for (int i = 0; i < j; i++) {
        const double2 b = make_double2(a1[i + 1].x + a2[i + 1].x, a1[i + 1].y + a2[i + 1].y);
        const double2 sb = r_cm(s_[i], b), ta = r_cm(r_cj(s_[i]), a);
        if (store) Hq[i * m + j] = make_double2(c_[i].x * a.x + sb.x, c_[i].x * a.y + sb.y);
        a = make_double2(c_[i].x * b.x - ta.x, c_[i].x * b.y - ta.y);
    }
    // scaled by a power of two: no square overflows or underflows
    const double sc = res_unscale(a.x, a.y, hn);
    const double ax = a.x * sc, ay = a.y * sc, b = hn * sc, u = ax * ax + ay * ay, t = u + b * b;
    const double ru = u > 0 ? rsqrt(u) : 0.0, rt = t > 0 ? rsqrt(t) : (t == t ? 0.0 : t), sn = b * rt;
    double2 c, s, d;  // d = c a + s hn
    if (u == 0.0) {
        c = make_double2(0, 0);
        s = make_double2(1, 0);
        d = make_double2(hn, 0);
    } else {
        c = make_double2(u * ru * rt, 0);
        s = make_double2(ax * ru * sn, ay * ru * sn);
        const double r = ru * (t * rt);
        d = make_double2(a.x * r, a.y * r);
    }
    c_[j] = c;
    s_[j] = s;
    if (store) Hq[j * m + j] = d;
    const double2 gj = g_[j], gt = r_cm(r_cj(s), gj);
    g_[j] = make_double2(c.x * gj.x, c.x * gj.y);
    g_[j + 1] = make_double2(-gt.x, -gt.y);
    gabs *= u == 0.0 ? 1.0 : sn;
}

// y = R^-1 g in place of g, j + 1 unknowns, by one warp (Hq complete)
__device__ __forceinline__ void res_backsub(int j, int m, const double2* Hq, double2* g_, int lane)
{
    for (int i = j; i >= 0; i--) {
        const double2 d = __ldcg(Hq + i * m + i), s = g_[i];
        const double den = d.x * d.x + d.y * d.y;
        const double2 y = den > 0 ? make_double2((s.x * d.x + s.y * d.y) / den, (s.y * d.x - s.x * d.y) / den)
                                  : make_double2(0, 0);
        __syncwarp();
        if (lane == 0) g_[i] = y;
        for (int k = lane; k < i; k += 32) {
            const double2 t = r_cm(__ldcg(Hq + k * m + i), y);
            g_[k] = make_double2(g_[k].x - t.x, g_[k].y - t.y);
        }
        __syncwarp();
    }
}

__device__ __forceinline__ void res_stat(double* stat, int iters, double worst)
{
    stat[0] = fmax(stat[0], (double)iters);
    stat[1] = worst != worst ? worst : fmax(stat[1], worst);
    stat[2] = worst;
    stat[3] = iters;
}

// relative residual; a NaN norm gives NaN
__device__ __forceinline__ double res_rel(double r, double bn) { return bn > 0 ? r / bn : (bn == bn ? 0.0 : bn); }

// squared norm of w - V h2 from |w|^2 = h2[nv] and h2[0 .. nv), by one warp; in every
// lane.  |h2|^2 is left out where it cannot change the result (exponents 30 apart)
__device__ __forceinline__ double res_norm2(const double2* h2, int nv, int lane)
{
    int e = 0;
    for (int i = lane; i < nv; i += 32)
        e = max(e, max(__double2hiint(h2[i].x) & 0x7fffffff, __double2hiint(h2[i].y) & 0x7fffffff));
    e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e) >> 20;
    const double ww = h2[nv].x;
    const int ew = (__double2hiint(ww) & 0x7fffffff) >> 20;
    // |h2|^2 < 2 nv 4^(e - 1022) <= 2^(2 e - 2044 + 8), |w|^2 >= 2^(ew - 1023)
    if (2 * e - 2036 < ew - 1023 - 60) return ww;
    double s = 0;
    for (int i = lane; i < nv; i += 32) s += h2[i].x * h2[i].x + h2[i].y * h2[i].y;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    s = ww - s;
    return s != s ? s : fmax(s, 0.0);
}
// norm and its reciprocal (0 for 0) from the squared norm
__device__ __forceinline__ void res_root(double s, double& norm, double& inv)
{
    if (s > 0 && s < 1e300) {
        inv = rsqrt(s);
        norm = s * inv;
    } else {
        norm = s != s ? s : sqrt(s);
        inv = norm > 0 ? 1.0 / norm : 0.0;
    }
}

// The FGMRES cycle (zero initial guess, at most K.m iterations) on the residual
// already in K.W (own rows, after a __syncthreads).  sys: rows r0, r1 of this CTA;
// precond(j, bar): Z_j = M V_j, with the barrier that ends it; apply(j): W = A Z_j on
// own rows; after_v(j): own rows of V_j are set (for a pointwise preconditioner).
// After it, the solution's combination: x = sum_i Z_i y_i, y in shared memory,
// i <= jend.  Returns jend, -1 when a wait ran out.
template <class SYS>
__device__ int res_fgmres(SYS& sys, const ResKrylov& K, ResBar& bar, double2* smem, double2** y_out)
{
    const int m = K.m, ld = m + 2;
    const int64_t n = K.n, r0 = sys.r0, r1 = sys.r1;
    double2* cs = smem;
    double2* sn = cs + ld;
    double2* g = sn + ld;
    double2* h1 = g + ld;
    double2* h2 = h1 + ld;
    __shared__ double bnorm, rel, wn, gabs;
    double2* P1 = K.part;
    double2* P2 = P1 + (int64_t)RES_MAXCTA * ld;
    res_dots(K, r0, r1, 0, true, P1, ld);
    if (!res_barrier(bar)) return -1;
    res_reduce(1, P1, ld, h1);
    if (threadIdx.x == 0) {
        const double d2 = h1[0].x, b = d2 != d2 ? d2 : sqrt(fmax(d2, 0.0));  // a NaN norm stays NaN
        bnorm = gabs = b;
        wn = b > 0 ? 1.0 / b : 0.0;
        g[0] = make_double2(b, 0);
    }
    __syncthreads();
    auto set_v = [&](int j) {
        for (int64_t k = r0 + threadIdx.x; k < r1; k += blockDim.x)
            K.V[(int64_t)j * n + k] = make_double2(K.W[k].x * wn, K.W[k].y * wn);
        sys.after_v(j);
    };
    set_v(0);
    if (!res_barrier(bar)) return -1;
    int j = 0, extra = K.extra;
    for (;; j++) {
        if (!sys.precond(j, bar)) return -1;
        sys.apply(j);
        __syncthreads();
        res_dots(K, r0, r1, j + 1, false, P1, ld);
        if (!res_barrier(bar)) return -1;
        res_reduce(j + 1, P1, ld, h1);
        res_update(K, r0, r1, j + 1, h1);
        res_dots(K, r0, r1, j + 1, true, P2, ld);
        if (!res_barrier(bar)) return -1;
        res_reduce(j + 2, P2, ld, h2);
        if (threadIdx.x < 32) {
            const double hh = res_norm2(h2, j + 1, threadIdx.x);
            if (threadIdx.x == 0) {
                double hn;
                res_root(hh, hn, wn);
                res_givens(j, m, h1, h2, hn, cs, sn, g, K.H, blockIdx.x == 0, gabs);
                rel = res_rel(gabs, bnorm);
            }
        }
        __syncthreads();
        bool more = rel >= K.tol;
        if (!more && extra > 0) {
            extra--;
            more = true;
        }
        more = more && j + 1 < m;
        if (!more) break;
        res_update(K, r0, r1, j + 1, h2);
        set_v(j + 1);
        if (!res_barrier(bar)) return -1;
    }
    // y = R^-1 g (CTA 0's H is complete after a barrier)
    if (!res_barrier(bar)) return -1;
    if (threadIdx.x < 32) res_backsub(j, m, K.H, g, threadIdx.x);
    if (blockIdx.x == 0 && threadIdx.x == 0) res_stat(K.stat, j + 1, rel);
    __syncthreads();
    *y_out = g;
    return j;
}

// the same as maxima of nonnegative doubles by their bits (a NaN's exceed all)
__device__ __forceinline__ void res_stat_max(double* stat, int iters, double rel)
{
    unsigned long long* st = (unsigned long long*)stat;
    atomicMax(st + 0, (unsigned long long)__double_as_longlong((double)iters));
    atomicMax(st + 1, (unsigned long long)__double_as_longlong(rel) & 0x7fffffffffffffffull);
}

// ------------------------------------------------------------------ cluster form
constexpr int CLU_MAXN = 2048;  // rows: two gather vectors take 64 KB of shared memory then
constexpr int CLU_MAXC = 16;

// shared memory of a CTA:
//   x[2][n] gather vectors (v, z), w[rows], pr[2][C][m + 2] partial sums, cs, sn, g, h1, h2 [m + 2]
int clu_pick(const void* fn, int64_t n, int64_t nnz, int m, size_t extra);
int res_group(int64_t rows, int64_t nrow, int64_t nnz);
sie_status clu_launch(const void* fn, int C, size_t smem, void** args, cudaStream_t st);
inline size_t clu_smem(int64_t n, int m, int C)
{
    return sizeof(double2) * (size_t)(2 * n + (n + C - 1) / C + 2 * C * (m + 2) + 5 * (m + 2));
}

struct CluMem {
    double2 *xv, *xz, *w, *pr, *cs, *sn, *g, *h1, *h2;
    int C, rank, ld;
    __device__ CluMem(double2* s, int64_t n, int m)
    {
        auto c = cooperative_groups::this_cluster();
        C = (int)c.num_blocks();
        rank = (int)c.block_rank();
        ld = m + 2;
        xv = s;
        xz = xv + n;
        w = xz + n;
        pr = w + (n + C - 1) / C;
        cs = pr + 2 * C * ld;
        sn = cs + ld;
        g = sn + ld;
        h1 = g + ld;
        h2 = h1 + ld;
    }
    // own rows of a gather vector (x: whole, this CTA's copy, own rows set before a
    // __syncthreads) to the other CTAs, spread over all threads
    template <class T>
    __device__ __forceinline__ void spread(T* x, int64_t r0, int rows) const
    {
        auto c = cooperative_groups::this_cluster();
        const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        for (int r = warp; r < C; r += nw) {
            if (r == rank) continue;
            T* o = c.map_shared_rank(x + r0, r);
            for (int k = lane; k < rows; k += 32) o[k] = x[r0 + k];
        }
    }
};

__device__ __forceinline__ void clu_sync() { cooperative_groups::this_cluster().sync(); }

// partial sums of conj(V_i) w, i < nv, and of |w|^2 (slot nv) when norm, to every CTA's pr[buf][rank]
__device__ __forceinline__ void clu_dots(const CluMem& M, const double2* V, int64_t n, int64_t r0, int rows, int nv,
                                         bool norm, int buf)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int i = warp; i < nv + (norm ? 1 : 0); i += nw) {
        const double2* v = i < nv ? V + (int64_t)i * n + r0 : M.w;
        double2 s = make_double2(0, 0);
        for (int k = lane; k < rows; k += 32) r_fma(s, r_cj(v[k]), M.w[k]);
        s = warp_sum(s);
        if (lane < M.C)
            *cooperative_groups::this_cluster().map_shared_rank(M.pr + (buf * M.C + M.rank) * M.ld + i, lane) = s;
    }
}
// h[i] = sum over the CTAs (8 or 16): a warp per column, a half for each component
// (4 FP64 additions; a thread per column took 2,200 cycles in a chain of them)
__device__ __forceinline__ void clu_reduce(const CluMem& M, int cols, int buf, double2* h)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5, c = lane & 15;
    for (int i = warp; i < cols; i += nw) {
        const double2* p = M.pr + buf * M.C * M.ld + i;
        double v = 0;
        if (c < M.C) {
            const double2 a = p[c * M.ld];
            v = lane < 16 ? a.x : a.y;
        }
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        const double y = __shfl_xor_sync(0xffffffffu, v, 16);
        if (lane == 0) h[i] = make_double2(v, y);
    }
    __syncthreads();
}

// The cycle of a cluster; the residual is in M.w (own rows, after a __syncthreads).  sys: r0, rows; precond(j): from M.xv, Z_j (own
// rows) and M.xz of every CTA, false for a pointwise one done by set_v; set_v(j,
// k, v): own row k of V_j is v (sets own row of what the next product gathers, which
// share() then copies to the other CTAs); apply(j): M.w = A z from M.xz.  After it y in M.g; returns jend.
// Restarted solves call it again with the new residual: it0 iterations done, at
// most maxit in all, bnorm0 the norm of the right-hand side (below 0 in the first
// cycle); *above: a residual is still above tol; rel_out: this one's.
struct CluRun {
    int it = 0, maxit = 1 << 30;
    double bnorm = -1.0, rel = 0.0;
    bool above = true;
};
template <class SYS>
__device__ int clu_fgmres(SYS& sys, const ResKrylov& K, CluMem& M, CluRun& run)
{
    const int m = K.m, rows = sys.rows;
    const int64_t n = K.n, r0 = sys.r0;
    double2* V = K.V;
    double2* H = K.H;
    __shared__ double bnorm, tolb, wn, gabs;
    __shared__ int go, above_s;
    clu_sync();  // every CTA of the cluster has started, or is done with the last cycle
    clu_dots(M, V, n, r0, rows, 0, true, 0);
    clu_sync();
    clu_reduce(M, 1, 0, M.h1);
    if (threadIdx.x == 0) {
        const double d2 = M.h1[0].x, b = d2 != d2 ? d2 : sqrt(fmax(d2, 0.0));  // a NaN norm stays NaN
        bnorm = run.bnorm < 0 ? b : run.bnorm;
        gabs = b;
        tolb = bnorm > 0 ? K.tol * bnorm : 1e300;  // a zero right-hand side is solved
        wn = b > 0 ? 1.0 / b : 0.0;
        M.g[0] = make_double2(b, 0);
    }
    __syncthreads();
    run.bnorm = bnorm;
    auto set_v = [&](int j) {
        for (int k = threadIdx.x; k < rows; k += blockDim.x) {
            const double2 v = make_double2(M.w[k].x * wn, M.w[k].y * wn);
            V[(int64_t)j * n + r0 + k] = v;
            sys.set_v(j, k, v);
        }
        __syncthreads();
        sys.share();
        clu_sync();
    };
    set_v(0);
    int j = 0, extra = K.extra;
    for (;; j++) {
        if (sys.precond(j)) clu_sync();
        sys.apply(j);
        __syncthreads();
        clu_dots(M, V, n, r0, rows, j + 1, false, 0);
        clu_sync();
        clu_reduce(M, j + 1, 0, M.h1);
        for (int k = threadIdx.x; k < rows; k += blockDim.x) {
            double2 s = make_double2(0, 0);
            for (int i = 0; i <= j; i++) r_fma(s, V[(int64_t)i * n + r0 + k], M.h1[i]);
            M.w[k] = make_double2(M.w[k].x - s.x, M.w[k].y - s.y);
        }
        __syncthreads();
        clu_dots(M, V, n, r0, rows, j + 1, true, 1);
        clu_sync();
        clu_reduce(M, j + 2, 1, M.h2);
        // warp 0: norm, rotation and decision; the others meanwhile subtract V h2
        double hh = 0;
        if (threadIdx.x < 32) {
            hh = res_norm2(M.h2, j + 1, threadIdx.x);
        } else {
            for (int k = threadIdx.x - 32; k < rows; k += blockDim.x - 32) {
                double2 s = make_double2(0, 0);
                for (int i = 0; i <= j; i++) r_fma(s, V[(int64_t)i * n + r0 + k], M.h2[i]);
                M.w[k] = make_double2(M.w[k].x - s.x, M.w[k].y - s.y);
            }
        }
        if (threadIdx.x == 0) {
            double hn;
            res_root(hh, hn, wn);
            res_givens(j, m, M.h1, M.h2, hn, M.cs, M.sn, M.g, H, M.rank == 0, gabs);
            // NaN stops here (rel, below, reports it); tolb = tol |b|
            bool more = gabs >= tolb;
            if (!more && extra > 0) {
                extra--;
                more = true;
            }
            above_s = more;
            go = more && j + 1 < m && run.it + j + 1 < run.maxit;
        }
        __syncthreads();
        if (!go) break;  // every CTA of the cluster decides from the same numbers
        set_v(j + 1);
    }
    clu_sync();  // rank 0's H
    if (threadIdx.x < 32) res_backsub(j, m, H, M.g, threadIdx.x);
    run.rel = res_rel(gabs, bnorm);
    run.above = above_s != 0;
    run.it += j + 1;
    __syncthreads();
    return j;
}

// sum over a CSR row of val x by the G lanes of a group: every lane ends with it.
// CG: x was written by other CTAs of this kernel.  All lanes of the warp call it (rows
// beyond the end with e0 = e1).
template <bool CG>
__device__ __forceinline__ double2 res_row(int64_t e0, int64_t e1, const int32_t* __restrict__ col,
                                           const double2* __restrict__ val, const double2* x, int l, int G)
{
    double2 s = make_double2(0, 0);
    int64_t e = e0 + l;
    for (; e + 3 * G < e1; e += 4 * G) {  // four loads in flight
        double2 v[4], xv[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int c = __ldg(col + e + u * G);
            v[u] = __ldg(val + e + u * G);
            xv[u] = CG ? __ldcg(x + c) : x[c];
        }
#pragma unroll
        for (int u = 0; u < 4; u++) r_fma(s, v[u], xv[u]);
    }
    for (; e < e1; e += G) {
        const int c = __ldg(col + e);
        r_fma(s, __ldg(val + e), CG ? __ldcg(x + c) : x[c]);
    }
    for (int off = G >> 1; off > 0; off >>= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
    }
    return s;
}

// for the rows [r0, r1) by groups of G lanes: body(row or -1, lane in group); all lanes of a warp run together
template <class F>
__device__ __forceinline__ void res_rows(int64_t r0, int64_t r1, int G, F body)
{
    const int per = blockDim.x / G, grp = threadIdx.x / G, l = threadIdx.x % G;
    for (int64_t b = r0; b < r1; b += per) {
        const int64_t k = b + grp;
        body(k < r1 ? k : -1, l);
    }
}

}  // namespace sie

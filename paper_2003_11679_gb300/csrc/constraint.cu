// Constraint preconditioners as one kernel per application, a cluster of CTAs
// (resident.cuh, CluMem):
//   (Dg - kappa D^T Lphi_NR D) y = v             (Eq. nest2pc, nested)
// by block elimination on the charges q = D y,
//   (I - kappa D Dg^-1 D^T Lphi_NR) q = D Dg^-1 v,  y = Dg^-1 (v + kappa D^T Lphi_NR q),
// and the exterior AEFIE form around it (v1' = v1 - (j k0)^-1 D^T Lphi B v2 before,
// y / (j k0) and w2 = (v2 - F D w1) / (j k0) after).  The charge system is solved by
// restarted FGMRES preconditioned by the explicit complex64 inverse: FP32 products
// and per-lane sums, row sums in FP64.
// The work is small and was latency-bound: 14 launches an iteration and a host
// check took 118 us (320 triangles) to 220 us (1,280) an application; 42 and 121 us
// now.  An iteration meets at 5 cluster barriers; the inverse is read by 8 or 16 SMs
// (1,280 triangles: 13 MB, about 6 us), which bounds the size it is taken for
// (CLU_MAXN triangles).
#include <algorithm>

#include "resident.cuh"

namespace sie {

struct ConSys {
    int nt, ne;
    DevMesh M;
    const double *elen;
    const double2* idLA;        // 1 / diag(LA)
    const int64_t* rp;          // triangle CSR of Lphi_NR
    const int32_t* col;
    const double2* val;
    const float2* X;            // explicit inverse, nt x nt
    double2 kappa, ijk0;        // ijk0 = 1 / (j k0)
    int ext;                    // 1: the exterior AEFIE preconditioner of [x1; x2]
    const double2* x;           // ne, or ne + nt
    double2* y;
    double2 *v1, *b, *q;        // scratch: ne, nt, nt
    double* stat;               // largest iteration count and residual
};

struct ConClu {
    const ConSys& s;
    const ResKrylov& K;
    CluMem& M;
    float2* xf;     // v in complex64, whole
    int G;
    int64_t r0;
    int rows;

    // l_e (phi_T+ - phi_T-)
    __device__ __forceinline__ double2 dt(int e, const double2* phi) const
    {
        const double2 a = phi[s.M.edge_tri[2 * e]], b = phi[s.M.edge_tri[2 * e + 1]];
        const double l = s.elen[e];
        return make_double2(l * (a.x - b.x), l * (a.y - b.y));
    }
    // Lphi_NR x on own rows into M.xv of every CTA; x(c): element c
    template <class F>
    __device__ __forceinline__ void lphi(F x)
    {
        res_rows(0, rows, G, [&](int64_t k, int l) {
            double2 o = make_double2(0, 0);
            const int64_t e0 = k >= 0 ? s.rp[r0 + k] : 0, e1 = k >= 0 ? s.rp[r0 + k + 1] : 0;
            int64_t e = e0 + l;
            for (; e + 3 * G < e1; e += 4 * G) {
                double2 v[4];
                int c[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    c[u] = __ldg(s.col + e + u * G);
                    v[u] = __ldg(s.val + e + u * G);
                }
#pragma unroll
                for (int u = 0; u < 4; u++) r_fma(o, v[u], x(c[u]));
            }
            for (; e < e1; e += G) r_fma(o, __ldg(s.val + e), x(__ldg(s.col + e)));
            for (int off = G >> 1; off > 0; off >>= 1) {
                o.x += __shfl_xor_sync(0xffffffffu, o.x, off);
                o.y += __shfl_xor_sync(0xffffffffu, o.y, off);
            }
            if (k >= 0) {
                auto c = cooperative_groups::this_cluster();
                for (int r = l; r < M.C; r += G) *c.map_shared_rank(M.xv + r0 + k, r) = o;
            }
        });
    }
    // sum_i 2 c_i A_t f(edge i) of own triangle k
    template <class F>
    __device__ __forceinline__ double2 dsum(int t, F f) const
    {
        double2 o = make_double2(0, 0);
        for (int i = 0; i < 3; i++) {
            const double2 v = f(s.M.tri_edge[3 * t + i]);
            const double c = 2.0 * s.M.coef[3 * t + i] * s.M.area[t];
            o.x += c * v.x;
            o.y += c * v.y;
        }
        return o;
    }
    // o = z - kappa D Dg^-1 D^T phi on own triangle t
    __device__ __forceinline__ double2 charge(int t, double2 z) const
    {
        const double2 d = dsum(t, [&](int e) { return r_cm(s.idLA[e], dt(e, M.xv)); });
        const double2 kd = r_cm(s.kappa, d);
        return make_double2(z.x - kd.x, z.y - kd.y);
    }
    __device__ void set_v(int, int k, double2 v)
    {
        xf[r0 + k] = make_float2((float)v.x, (float)v.y);
    }
    __device__ void share() { M.spread(xf, r0, rows); }
    // z = X v: a warp per row
    __device__ bool precond(int j)
    {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5, n = s.nt;
        for (int k = warp; k < rows; k += nw) {
            const float2* row = s.X + (r0 + k) * (int64_t)n;
            float ar = 0, ai = 0, br = 0, bi = 0;
            // n is even (constraint_resident): 16-byte aligned rows
            const float4* r4 = reinterpret_cast<const float4*>(row);
            const float4* x4 = reinterpret_cast<const float4*>(xf);
#pragma unroll 4
            for (int c = lane; c < n / 2; c += 32) {
                const float4 a = __ldg(r4 + c), v = x4[c];
                ar = fmaf(a.x, v.x, fmaf(-a.y, v.y, ar));
                ai = fmaf(a.x, v.y, fmaf(a.y, v.x, ai));
                br = fmaf(a.z, v.z, fmaf(-a.w, v.w, br));
                bi = fmaf(a.z, v.w, fmaf(a.w, v.z, bi));
            }
            const double2 z = warp_sum(make_double2((double)ar + br, (double)ai + bi));
            if (lane == 0) K.Z[(int64_t)j * K.n + r0 + k] = z;
            if (lane < M.C) *cooperative_groups::this_cluster().map_shared_rank(M.xz + r0 + k, lane) = z;
        }
        return true;
    }
    __device__ void apply(int)
    {
        lphi([&](int c) { return M.xz[c]; });
        clu_sync();
        for (int k = threadIdx.x; k < rows; k += blockDim.x) M.w[k] = charge((int)r0 + k, M.xz[r0 + k]);
    }
};

__global__ void __launch_bounds__(RES_T, 1) k_constraint(ConSys s, ResKrylov K, int maxit, int G)
{
    extern __shared__ __align__(16) double2 rs_smem[];
    CluMem M(rs_smem, K.n, K.m);
    float2* xf = reinterpret_cast<float2*>(M.h2 + M.ld);
    const int64_t len = (s.nt + M.C - 1) / M.C, r0 = min((int64_t)s.nt, M.rank * len);
    const int rows = (int)(min((int64_t)s.nt, r0 + len) - r0);
    const int elen = (s.ne + M.C - 1) / M.C, e0 = min(s.ne, M.rank * elen), e1 = min(s.ne, e0 + elen);
    ConClu ops{s, K, M, xf, G, r0, rows};
    const double2 *x1 = s.x, *x2 = s.x + s.ne;
    double2 *y1 = s.y, *y2 = s.y + s.ne;
    double2 *v1 = s.v1, *b = s.b, *sol = s.q;
    clu_sync();  // every CTA has started: distributed shared memory may be written
    // v1' = v1 - (j k0)^-1 D^T Lphi B v2, B v2 = -A v2
    if (s.ext) {
        ops.lphi([&](int c) {
            const double a = -s.M.area[c];
            const double2 v = x2[c];
            return make_double2(a * v.x, a * v.y);
        });
        clu_sync();
    }
    auto v1p = [&](int e) {
        double2 v = x1[e];
        if (s.ext) {
            const double2 d = r_cm(s.ijk0, ops.dt(e, M.xv));
            v.x -= d.x;
            v.y -= d.y;
        }
        return v;
    };
    for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) v1[e] = v1p(e);
    for (int k = threadIdx.x; k < rows; k += blockDim.x) {
        const double2 r = ops.dsum((int)r0 + k, [&](int e) { return r_cm(s.idLA[e], v1p(e)); });
        M.w[k] = r;
        b[r0 + k] = r;
        sol[r0 + k] = make_double2(0, 0);
    }
    __syncthreads();
    CluRun run;
    run.maxit = maxit;
    for (;;) {
        const int jend = clu_fgmres(ops, K, M, run);
        for (int k = threadIdx.x; k < rows; k += blockDim.x) {
            double2 x = sol[r0 + k];
            for (int i = 0; i <= jend; i++) r_fma(x, K.Z[(int64_t)i * K.n + r0 + k], M.g[i]);
            sol[r0 + k] = x;
            M.xz[r0 + k] = x;
        }
        __syncthreads();
        M.spread(M.xz, r0, rows);
        clu_sync();
        ops.lphi([&](int c) { return M.xz[c]; });
        clu_sync();
        if (!run.above || run.it >= maxit) break;
        // restart from the true residual
        for (int k = threadIdx.x; k < rows; k += blockDim.x) {
            const double2 a = ops.charge((int)r0 + k, M.xz[r0 + k]), r = b[r0 + k];
            M.w[k] = make_double2(r.x - a.x, r.y - a.y);
        }
        __syncthreads();
    }
    if (M.rank == 0 && threadIdx.x == 0) res_stat_max(s.stat, run.it, run.rel);
    // y = Dg^-1 (v1' + kappa D^T Lphi q) [/ (j k0)]; v1' of other CTAs' edges is complete since the first barriers
    auto y_of = [&](int e) {
        const double2 k = r_cm(s.kappa, ops.dt(e, M.xv)), v = __ldcg(v1 + e);
        const double2 y = r_cm(s.idLA[e], make_double2(v.x + k.x, v.y + k.y));
        return s.ext ? r_cm(s.ijk0, y) : y;
    };
    for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) y1[e] = y_of(e);
    if (s.ext)
        for (int k = threadIdx.x; k < rows; k += blockDim.x) {
            const int t = (int)r0 + k;
            const double2 d = ops.dsum(t, y_of), v = x2[t];
            const double a = s.M.area[t];
            y2[t] = r_cm(s.ijk0, make_double2(v.x - d.x / a, v.y - d.y / a));
        }
    clu_sync();  // no CTA leaves while another may still write to its shared memory
}

// true: applied by the cluster kernel (and *st_out is its launch status)
bool constraint_resident(sie_op* op, const AimOp& a, double2 kappa, bool ext, const double2* x, double2* y, double tol,
                         int maxit, const ResWork& w, double2* v1, double2* b, double2* q, sie_status* st_out)
{
    const int nt = (int)op->mesh->h.nt, ne = (int)op->mesh->h.ne;
    if (!a.lu || !a.lu->Xinv || nt > CLU_MAXN || nt % 2) return false;  // closed meshes have 3 nt = 2 ne: even
    const int C = clu_pick((const void*)k_constraint, nt, a.npairs, w.m, sizeof(float2) * (nt + 1));
    if (!C) return false;
    const size_t smem = clu_smem(nt, w.m, C) + sizeof(float2) * (nt + 1);
    ConSys s{};
    s.nt = nt, s.ne = ne;
    s.M = op->mesh->d;
    s.elen = op->elen;
    s.idLA = a.idLA;
    s.rp = a.tri_row_ptr, s.col = a.tri_col, s.val = a.valLphiNR;
    s.X = a.lu->Xinv;
    s.kappa = kappa;
    s.ijk0 = make_double2(0.0, -1.0 / op->k0);
    s.ext = ext;
    s.x = x, s.y = y;
    s.v1 = v1, s.b = b, s.q = q;
    s.stat = op->gstat + 4;
    ResKrylov K{};
    K.n = nt, K.m = w.m;
    K.V = w.V, K.Z = w.Z, K.H = w.H;
    K.tol = tol;
    K.stat = s.stat;
    int G = res_group((nt + C - 1) / C, nt, a.npairs);
    void* args[] = {&s, &K, &maxit, &G};
    *st_out = clu_launch((const void*)k_constraint, C, smem, args, op->mesh->ctx->stream);
    return true;
}

}  // namespace sie

// Interior impedance E' = Z' H of near-region-only and SIBC interiors (Eqs.
// GIBCdef, nest02, nest2): right-hand side, nested FGMRES and impedance factor
// in one resident kernel (resident.cuh).
//   GIBC: b = (K_i - I_x / 2) H, A = L_i,NR, M = its sparse approximate inverse,
//         E' = -(j k0 eps_r + sigma eta0)^-1 A^-1 b;
//   SIBC: b = I_x H, A = Gram matrix G, M = diag(G)^-1, E' = (eta_i / eta0) A^-1 b.
// Latency bounds it: an iteration is 4 (SIBC) or 5 (GIBC) barriers and chains of FP64
// operations.  SIBC
// needs no barrier for M: Z_j is written beside V_j.  As a graph loop of nine kernels
// an iteration, 310 us for a copper bar's 504 rows (4 iterations) and 500 us for 30,720
// rows (10); now 104 us on a cluster of 16 and 294 us on the whole GPU.
#include <algorithm>

#include "resident.cuh"

namespace sie {

struct NestSys {
    int64_t ne;
    const int64_t *ix_rp, *a_rp;
    const int32_t *ix_col, *a_col;
    const double2 *ix_val, *a_val, *k_val, *m_val;  // k_val, m_val: GIBC
    const double* idiag;                            // SIBC: 1 / diag(G)
    const double2* H;      // R vectors, ldh apart
    double2* E;            // R vectors, lde apart
    int64_t ldh, lde;
    double2 f;             // impedance factor, or
    const double2* zf;     // one per edge (several objects)
};

template <int RM>
struct NestOps {
    const NestSys& s;
    const ResKrylov& K;
    int64_t r0, r1;
    int G, Gx;

    __device__ void after_v(int j)
    {
        if (s.m_val) return;
        __syncthreads();
        const int rows = (int)(r1 - r0);
        for (int t = threadIdx.x; t < K.R * rows; t += blockDim.x) {
            const int q = t / rows;
            const int64_t k = r0 + t % rows, at = ((int64_t)j * K.R + q) * K.n + k;
            const double d = s.idiag[k];
            const double2 v = K.V[at];
            if (j < K.m) K.Z[at] = make_double2(v.x * d, v.y * d);
        }
    }
    __device__ void product(const double2* val, const double2* x, double2* y)
    {
        res_rows(r0, r1, G, [&](int64_t k, int l) {
            double2 o[RM];
            const int64_t e0 = k >= 0 ? s.a_rp[k] : 0, e1 = k >= 0 ? s.a_rp[k + 1] : 0;
            res_row<RM, true>(e0, e1, s.a_col, val, x, K.n, K.R, l, G, o);
            if (k >= 0 && l == 0)
#pragma unroll
                for (int q = 0; q < RM; q++)
                    if (q < K.R) y[q * K.n + k] = o[q];
        });
    }
    __device__ bool precond(int j, ResBar& bar)
    {
        if (!s.m_val) return true;
        product(s.m_val, K.V + (int64_t)j * K.R * K.n, K.Z + (int64_t)j * K.R * K.n);
        return res_barrier(bar);
    }
    __device__ void apply(int j) { product(s.a_val, K.Z + (int64_t)j * K.R * K.n, K.W); }
};

template <int RM>
__global__ void __launch_bounds__(RES_T, 1) k_nested(NestSys s, ResKrylov K, unsigned* cnt, int* err, int G, int Gx)
{
    extern __shared__ __align__(16) double2 rs_smem[];
    const int64_t len = (s.ne + gridDim.x - 1) / gridDim.x;
    const int64_t r0 = min(s.ne, blockIdx.x * len), r1 = min(s.ne, r0 + len);
    ResBar bar{cnt, err, 0};
    NestOps<RM> ops{s, K, r0, r1, G, Gx};
    // right-hand side
    res_rows(r0, r1, Gx, [&](int64_t k, int l) {
        double2 o[RM], p[RM];
        int64_t e0 = k >= 0 ? s.ix_rp[k] : 0, e1 = k >= 0 ? s.ix_rp[k + 1] : 0;
        res_row<RM, false>(e0, e1, s.ix_col, s.ix_val, s.H, s.ldh, K.R, l, Gx, o);
        if (s.k_val) {
            e0 = k >= 0 ? s.a_rp[k] : 0, e1 = k >= 0 ? s.a_rp[k + 1] : 0;
            res_row<RM, false>(e0, e1, s.a_col, s.k_val, s.H, s.ldh, K.R, l, Gx, p);
        }
        if (k >= 0 && l == 0)
#pragma unroll
            for (int q = 0; q < RM; q++)
                if (q < K.R)
                    K.W[q * K.n + k] =
                        s.k_val ? make_double2(p[q].x - 0.5 * o[q].x, p[q].y - 0.5 * o[q].y) : o[q];
    });
    __syncthreads();
    double2* y = nullptr;
    const int jend = res_fgmres(ops, K, bar, rs_smem, &y);
    if (jend < 0) {
        if (threadIdx.x == 0) K.stat[1] = K.stat[2] = __longlong_as_double(0x7ff0000000000000ll);
        return;
    }
    const int rows = (int)(r1 - r0);
    for (int t = threadIdx.x; t < K.R * rows; t += blockDim.x) {
        const int q = t / rows;
        const int64_t k = r0 + t % rows;
        double2 x = make_double2(0, 0);
        for (int i = 0; i <= jend; i++) r_fma(x, K.Z[((int64_t)i * K.R + q) * K.n + k], y[q * (K.m + 2) + i]);
        s.E[q * s.lde + k] = r_cm(s.zf ? s.zf[k] : s.f, x);
    }
}

// cluster form: cluster q solves right-hand side q
struct NestClu {
    const NestSys& s;
    const ResKrylov& K;
    CluMem& M;
    int q, G;
    int64_t r0;
    int rows;
    double2* Z;

    __device__ __forceinline__ void row(const double2* val, const double2* x, int k, int l, double2* o)
    {
        const int64_t e0 = k >= 0 ? s.a_rp[r0 + k] : 0, e1 = k >= 0 ? s.a_rp[r0 + k + 1] : 0;
        res_row<1, false>(e0, e1, s.a_col, val, x, 0, 1, l, G, o);
    }
    __device__ void set_v(int j, int k, double2 v)
    {
        if (s.m_val) {
            M.xv[r0 + k] = v;
            return;
        }
        const double d = s.idiag[r0 + k];
        const double2 z = make_double2(v.x * d, v.y * d);
        if (j < K.m) Z[(int64_t)j * K.n + r0 + k] = z;
        M.xz[r0 + k] = z;
    }
    __device__ void share() { M.spread(s.m_val ? M.xv : M.xz, r0, rows); }
    __device__ bool precond(int j)
    {
        if (!s.m_val) return false;
        res_rows(0, rows, G, [&](int64_t k, int l) {
            double2 o;
            row(s.m_val, M.xv, (int)k, l, &o);
            if (k >= 0) {
                if (l == 0) Z[(int64_t)j * K.n + r0 + k] = o;
                // the group's lanes share the copies
                auto c = cooperative_groups::this_cluster();
                for (int r = l; r < M.C; r += G) *c.map_shared_rank(M.xz + r0 + k, r) = o;
            }
        });
        return true;
    }
    __device__ void apply(int)
    {
        res_rows(0, rows, G, [&](int64_t k, int l) {
            double2 o;
            row(s.a_val, M.xz, (int)k, l, &o);
            if (k >= 0 && l == 0) M.w[k] = o;
        });
    }
};

__global__ void __launch_bounds__(RES_T, 1) k_nested_clu(NestSys s, ResKrylov K, CluLock lock, int G, int Gx)
{
    extern __shared__ __align__(16) double2 rs_smem[];
    CluMem M(rs_smem, K.n, K.m);
    const int q = (int)blockIdx.x / M.C;
    const int64_t len = (s.ne + M.C - 1) / M.C, r0 = min(s.ne, M.rank * len);
    const int rows = (int)(min(s.ne, r0 + len) - r0);
    NestClu ops{s, K, M, q, G, r0, rows, K.Z + (int64_t)q * K.m * K.n};
    const double2* H = s.H + q * s.ldh;
    res_rows(0, rows, Gx, [&](int64_t k, int l) {
        double2 o, p;
        int64_t e0 = k >= 0 ? s.ix_rp[r0 + k] : 0, e1 = k >= 0 ? s.ix_rp[r0 + k + 1] : 0;
        res_row<1, false>(e0, e1, s.ix_col, s.ix_val, H, 0, 1, l, Gx, &o);
        if (s.k_val) {
            e0 = k >= 0 ? s.a_rp[r0 + k] : 0, e1 = k >= 0 ? s.a_rp[r0 + k + 1] : 0;
            res_row<1, false>(e0, e1, s.a_col, s.k_val, H, 0, 1, l, Gx, &p);
        }
        if (k >= 0 && l == 0) M.w[k] = s.k_val ? make_double2(p.x - 0.5 * o.x, p.y - 0.5 * o.y) : o;
    });
    __syncthreads();
    CluRun run;
    const int jend = clu_fgmres(ops, K, M, q, lock, run);
    if (jend < 0) {
        if (threadIdx.x == 0) K.stat[1] = K.stat[2] = __longlong_as_double(0x7ff0000000000000ll);
    } else {
        if (M.rank == 0 && threadIdx.x == 0) {
            if (lock.R == 1)
                res_stat(K.stat, jend + 1, run.rel);
            else
                res_stat_max(K.stat, jend + 1, run.rel);
        }
        for (int k = threadIdx.x; k < rows; k += blockDim.x) {
            double2 x = make_double2(0, 0);
            for (int i = 0; i <= jend; i++) r_fma(x, ops.Z[(int64_t)i * K.n + r0 + k], M.g[i]);
            s.E[q * s.lde + r0 + k] = r_cm(s.zf ? s.zf[r0 + k] : s.f, x);
        }
    }
    clu_sync();  // no CTA leaves while another may still write to its shared memory
}

// CTAs of a resident kernel: about 64 (row, right-hand side) pairs each, at most one per SM
int res_ctas(int64_t work)
{
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return std::max(1, std::min(v, RES_MAXCTA));
    }();
    return (int)std::max<int64_t>(1, std::min<int64_t>(sms, (work + 63) / 64));
}

// lanes per row: as many as the CTA's threads and half the mean row allow
int res_group(int64_t rows, int64_t nrow, int64_t nnz)
{
    const int64_t avg = nrow > 0 ? nnz / nrow : 0;
    int G = 1;
    while (G < 32 && (int64_t)(2 * G) * rows <= RES_T && 2 * G <= std::max<int64_t>(1, avg / 2)) G *= 2;
    return G;
}

sie_status res_launch(const void* fn, int ctas, size_t smem, void** args, cudaStream_t st)
{
    SIE_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    SIE_CUDA_TRY(cudaLaunchCooperativeKernel(fn, dim3(ctas), dim3(RES_T), args, smem, st));
    return SIE_OK;
}

sie_status clu_launch(const void* fn, int C, int R, size_t smem, void** args, cudaStream_t st)
{
    SIE_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (C > 8) SIE_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C * R);
    cfg.blockDim = dim3(RES_T);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeCooperative;  // several clusters wait on one another's flags
    at[1].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = R > 1 ? 2 : 1;
    SIE_CUDA_TRY(cudaLaunchKernelExC(&cfg, fn, args));
    return SIE_OK;
}

// whether R clusters of C CTAs can run at the same time
bool clu_fits(const void* fn, int C, int R, size_t smem)
{
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (C > 8) cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C * R);
    cfg.blockDim = dim3(RES_T);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n >= R;
}

// CTAs of a cluster (0: the R clusters do not run at once).  8 (portable) for up to
// 1,024 rows and 16,384 entries, else 16: a bar's 504 rows of 64 entries take 14,000
// cycles a product on 8 SMs' FP64 lanes, 7,000 on 16.  Clusters of 16 fit a GPU region
// once only: 8 of them may not run at once, and 8 clusters of 8 take 210 ms for a solve
// of the bar with 8 right-hand sides, the forms without clusters 430.
int clu_pick(const void* fn, int64_t n, int64_t nnz, int m, int R, size_t extra)
{
    if (n > CLU_MAXN) return 0;
    const bool small = n <= 1024;
    for (int C = small && nnz <= 16384 ? 8 : CLU_MAXC; C >= (small ? 8 : CLU_MAXC); C >>= 1) {
        const size_t smem = clu_smem(n, m, C) + extra;
        if (smem <= 200 * 1024 && clu_fits(fn, C, R, smem)) return C;
    }
    return 0;
}

// Rows per right-hand side up to which the cluster form is taken (CLU_MAXN): its
// gather vectors have to fit, and 16 SMs do the arithmetic of all rows.
sie_status nested_solve(sie_op* op, int R, const double2* H, int64_t ldh, double2* E, int64_t lde, double2 f,
                        int extra, const ResWork& w)
{
    cudaStream_t st = op->mesh->ctx->stream;
    const int64_t ne = op->mesh->h.ne;
    const bool sibc = op->p.interior_model == SIE_SIBC;
    AimOp& I = op->inn;
    NestSys s{};
    s.ne = ne;
    s.ix_rp = op->ix_row_ptr, s.ix_col = op->ix_col, s.ix_val = op->ix_val;
    s.a_rp = sibc ? op->gr_row_ptr : I.row_ptr;
    s.a_col = sibc ? op->gr_col : I.col;
    s.a_val = sibc ? op->gr_val : I.valL;
    s.k_val = sibc ? nullptr : I.valK;
    s.m_val = sibc ? nullptr : I.valM;
    s.idiag = sibc ? op->gr_idiag : nullptr;
    s.H = H, s.ldh = ldh, s.E = E, s.lde = lde;
    s.f = f;
    s.zf = op->edge_zf;
    ResKrylov K{};
    K.n = ne, K.m = w.m, K.R = R;
    K.V = w.V, K.Z = w.Z, K.W = w.W, K.H = w.H, K.ldh = w.ldh, K.part = w.part;
    K.tol = op->p.tol_inner;
    K.extra = extra;
    K.stat = op->gstat;
    unsigned* cnt = op->res_bar;
    int* err = (int*)(op->res_bar + 1);
    if (const int C = clu_pick((const void*)k_nested_clu, ne, sibc ? op->gr_nnz : I.nnz, w.m, R, 0)) {
        const int64_t rows = (ne + C - 1) / C;
        int G = res_group(rows, ne, sibc ? op->gr_nnz : I.nnz), Gx = sibc ? res_group(rows, ne, op->ix_nnz) : G;
        CluLock lock;
        lock.R = R, lock.flag = op->res_bar + 2, lock.err = err;
        if (R > 1) {
            SIE_CUDA_TRY(cudaMemsetAsync(lock.flag, 0, sizeof(unsigned) * 8 * CLU_RING, st));
        }
        void* args[] = {&s, &K, &lock, &G, &Gx};
        return clu_launch((const void*)k_nested_clu, C, R, clu_smem(ne, w.m, C), args, st);
    }
    const int ctas = res_ctas(ne * R);
    const int64_t rows = (ne + ctas - 1) / ctas;
    int G = res_group(rows, ne, sibc ? op->gr_nnz : I.nnz), Gx = sibc ? res_group(rows, ne, op->ix_nnz) : G;
    SIE_CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(unsigned), st));
    void* args[] = {&s, &K, &cnt, &err, &G, &Gx};
    return res_launch(R == 1 ? (const void*)k_nested<1> : (const void*)k_nested<8>, ctas, res_smem(w.m, R), args, st);
}

}  // namespace sie

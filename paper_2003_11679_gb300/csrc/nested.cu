// Interior impedance E' = Z' H of near-region-only and SIBC interiors (Eqs.
// GIBCdef, nest02, nest2): right-hand side, nested FGMRES and impedance factor
// in one resident kernel (resident.cuh).
//   GIBC: b = (K_i - I_x / 2) H, A = L_i,NR, M = its sparse approximate inverse,
//         E' = -(j k0 eps_r + sigma eta0)^-1 A^-1 b;
//   SIBC: b = I_x H, A = Gram matrix G, M = diag(G)^-1, E' = (eta_i / eta0) A^-1 b.
// Latency bounds it: an iteration is 4 (SIBC) or 5 (GIBC) barriers and chains of FP64
// operations.  SIBC needs no barrier for M: Z_j is written beside V_j.  As a graph loop
// of nine kernels an iteration, 310 us for a copper bar's 504 rows (4 iterations) and
// 500 us for 30,720 rows (10); now 102 us on a cluster of 16 and 284 us on the whole GPU.
#include <algorithm>
#include <cstdlib>

#include "limits.h"
#include "resident.cuh"

namespace sie {

struct NestSys {
    int64_t ne;
    const int64_t *ix_rp, *a_rp;
    const int32_t *ix_col, *a_col;
    const double2 *ix_val, *a_val, *k_val, *m_val;  // k_val, m_val: GIBC
    const double* idiag;                            // SIBC: 1 / diag(G)
    const double2* H;
    double2* E;
    double2 f;             // impedance factor, or
    const double2* zf;     // one per edge (several objects)
};

struct NestOps {
    const NestSys& s;
    const ResKrylov& K;
    int64_t r0, r1;
    int G;

    __device__ void after_v(int j)
    {
        if (s.m_val || j >= K.m) return;
        __syncthreads();
        for (int64_t k = r0 + threadIdx.x; k < r1; k += blockDim.x) {
            const double d = s.idiag[k];
            const double2 v = K.V[(int64_t)j * K.n + k];
            K.Z[(int64_t)j * K.n + k] = make_double2(v.x * d, v.y * d);
        }
    }
    __device__ void product(const double2* val, const double2* x, double2* y)
    {
        res_rows(r0, r1, G, [&](int64_t k, int l) {
            const int64_t e0 = k >= 0 ? s.a_rp[k] : 0, e1 = k >= 0 ? s.a_rp[k + 1] : 0;
            const double2 o = res_row<true>(e0, e1, s.a_col, val, x, l, G);
            if (k >= 0 && l == 0) y[k] = o;
        });
    }
    __device__ bool precond(int j, ResBar& bar)
    {
        if (!s.m_val) return true;
        product(s.m_val, K.V + (int64_t)j * K.n, K.Z + (int64_t)j * K.n);
        return res_barrier(bar);
    }
    __device__ void apply(int j) { product(s.a_val, K.Z + (int64_t)j * K.n, K.W); }
};

// row k of the right-hand side, (K_i - I_x / 2) H or I_x H, by the Gx lanes of a group
// (k < 0: no row; all lanes of the warp call it)
__device__ __forceinline__ double2 nest_rhs(const NestSys& s, int64_t k, int l, int Gx)
{
    int64_t e0 = k >= 0 ? s.ix_rp[k] : 0, e1 = k >= 0 ? s.ix_rp[k + 1] : 0;
    const double2 o = res_row<false>(e0, e1, s.ix_col, s.ix_val, s.H, l, Gx);
    if (!s.k_val) return o;
    e0 = k >= 0 ? s.a_rp[k] : 0, e1 = k >= 0 ? s.a_rp[k + 1] : 0;
    const double2 p = res_row<false>(e0, e1, s.a_col, s.k_val, s.H, l, Gx);
    return make_double2(p.x - 0.5 * o.x, p.y - 0.5 * o.y);
}

__global__ void __launch_bounds__(RES_T, 1) k_nested(NestSys s, ResKrylov K, unsigned* cnt, int* err, int polls, int G,
                                                  int Gx)
{
    extern __shared__ __align__(16) double2 rs_smem[];
    const int64_t len = (s.ne + gridDim.x - 1) / gridDim.x;
    const int64_t r0 = min(s.ne, blockIdx.x * len), r1 = min(s.ne, r0 + len);
    ResBar bar{cnt, err, polls, 0};
    NestOps ops{s, K, r0, r1, G};
    res_rows(r0, r1, Gx, [&](int64_t k, int l) {
        const double2 b = nest_rhs(s, k, l, Gx);
        if (k >= 0 && l == 0) K.W[k] = b;
    });
    __syncthreads();
    double2* y = nullptr;
    const int jend = res_fgmres(ops, K, bar, rs_smem, &y);
    if (jend < 0) return;
    for (int64_t k = r0 + threadIdx.x; k < r1; k += blockDim.x) {
        double2 x = make_double2(0, 0);
        for (int i = 0; i <= jend; i++) r_fma(x, K.Z[(int64_t)i * K.n + k], y[i]);
        s.E[k] = r_cm(s.zf ? s.zf[k] : s.f, x);
    }
}

// cluster form
struct NestClu {
    const NestSys& s;
    const ResKrylov& K;
    CluMem& M;
    int G;
    int64_t r0;
    int rows;

    __device__ __forceinline__ double2 row(const double2* val, const double2* x, int k, int l)
    {
        const int64_t e0 = k >= 0 ? s.a_rp[r0 + k] : 0, e1 = k >= 0 ? s.a_rp[r0 + k + 1] : 0;
        return res_row<false>(e0, e1, s.a_col, val, x, l, G);
    }
    __device__ void set_v(int j, int k, double2 v)
    {
        if (s.m_val) {
            M.xv[r0 + k] = v;
            return;
        }
        const double d = s.idiag[r0 + k];
        const double2 z = make_double2(v.x * d, v.y * d);
        if (j < K.m) K.Z[(int64_t)j * K.n + r0 + k] = z;
        M.xz[r0 + k] = z;
    }
    __device__ void share() { M.spread(s.m_val ? M.xv : M.xz, r0, rows); }
    __device__ bool precond(int j)
    {
        if (!s.m_val) return false;
        res_rows(0, rows, G, [&](int64_t k, int l) {
            const double2 o = row(s.m_val, M.xv, (int)k, l);
            if (k >= 0) {
                if (l == 0) K.Z[(int64_t)j * K.n + r0 + k] = o;
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
            const double2 o = row(s.a_val, M.xz, (int)k, l);
            if (k >= 0 && l == 0) M.w[k] = o;
        });
    }
};

__global__ void __launch_bounds__(RES_T, 1) k_nested_clu(NestSys s, ResKrylov K, int G, int Gx)
{
    extern __shared__ __align__(16) double2 rs_smem[];
    CluMem M(rs_smem, K.n, K.m);
    const int64_t len = (s.ne + M.C - 1) / M.C, r0 = min(s.ne, M.rank * len);
    const int rows = (int)(min(s.ne, r0 + len) - r0);
    NestClu ops{s, K, M, G, r0, rows};
    res_rows(0, rows, Gx, [&](int64_t k, int l) {
        const double2 b = nest_rhs(s, k >= 0 ? r0 + k : -1, l, Gx);
        if (k >= 0 && l == 0) M.w[k] = b;
    });
    __syncthreads();
    CluRun run;
    const int jend = clu_fgmres(ops, K, M, run);
    if (M.rank == 0 && threadIdx.x == 0) res_stat(K.stat, jend + 1, run.rel);
    for (int k = threadIdx.x; k < rows; k += blockDim.x) {
        double2 x = make_double2(0, 0);
        for (int i = 0; i <= jend; i++) r_fma(x, K.Z[(int64_t)i * K.n + r0 + k], M.g[i]);
        s.E[r0 + k] = r_cm(s.zf ? s.zf[r0 + k] : s.f, x);
    }
    clu_sync();  // no CTA leaves while another may still write to its shared memory
}

// CTAs of a resident kernel: about 64 rows each, at most one per SM
int res_ctas(int64_t work)
{
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    const int sms = std::max(1, std::min(v, RES_MAXCTA));
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
    SIE_CUDA_TRY(kernel_limit(fn, smem));
    SIE_CUDA_TRY(cudaLaunchCooperativeKernel(fn, dim3(ctas), dim3(RES_T), args, smem, st));
    return SIE_OK;
}

static void clu_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int C, size_t smem)
{
    cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(RES_T);
    cfg.dynamicSmemBytes = smem;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = C;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
}

sie_status clu_launch(const void* fn, int C, size_t smem, void** args, cudaStream_t st)
{
    SIE_CUDA_TRY(kernel_limit(fn, smem, C > 8));
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    clu_config(cfg, &at, C, smem);
    cfg.stream = st;
    SIE_CUDA_TRY(cudaLaunchKernelExC(&cfg, fn, args));
    return SIE_OK;
}

// whether the GPU runs a cluster of C CTAs
static bool clu_fits(const void* fn, int C, size_t smem)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    clu_config(cfg, &at, C, smem);
    int n = 0;
    if (kernel_limit(fn, smem, C > 8) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n >= 1;
}

// CTAs of a cluster (0: none).  8 for up to 768 rows and 6,000 entries, whose barriers and
// chains count more than their products (8 and 16 CTAs: 450 rows of 5 entries 190 and 194
// us, 648 rows 192 and 196, 96 rows of 58 81 and 82), else 16 (882 rows of 5: 220 and 195
// us; 168 rows of 62: 89 and 83; a bar's 504 rows of 65: 118 and 102).  Up to 1,024 rows 8
// (portable) where 16 do not run.
int clu_pick(const void* fn, int64_t n, int64_t nnz, int m, size_t extra)
{
    if (n > CLU_MAXN) return 0;
    const bool portable = n <= 1024;
    for (int C = n <= 768 && nnz <= 6000 ? 8 : CLU_MAXC; C >= (portable ? 8 : CLU_MAXC); C >>= 1) {
        const size_t smem = clu_smem(n, m, C) + extra;
        if (smem <= 200 * 1024 && clu_fits(fn, C, smem)) return C;
    }
    return 0;
}

// polls of a wait before it gives up; SIE_WAIT_POLLS in the environment lowers it
static int res_polls()
{
    const char* e = getenv("SIE_WAIT_POLLS");
    return e ? std::max(1, std::min(atoi(e), RES_SPIN)) : RES_SPIN;
}

// Rows up to which the cluster form is taken (CLU_MAXN): its gather vectors have to
// fit, and 16 SMs do the arithmetic of all rows.
sie_status nested_solve(sie_op* op, const double2* H, double2* E, double2 f, int extra, const ResWork& w)
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
    s.H = H, s.E = E;
    s.f = f;
    s.zf = op->edge_zf;
    ResKrylov K{};
    K.n = ne, K.m = w.m;
    K.V = w.V, K.Z = w.Z, K.W = w.W, K.H = w.H, K.part = w.part;
    K.tol = op->p.tol_inner;
    K.extra = extra;
    K.stat = op->gstat;
    unsigned* cnt = op->res_bar;
    int* err = (int*)(op->gstat + 6);
    const int64_t nnz = sibc ? op->gr_nnz : I.nnz;
    if (const int C = clu_pick((const void*)k_nested_clu, ne, nnz, w.m, 0)) {
        const int64_t rows = (ne + C - 1) / C;
        int G = res_group(rows, ne, nnz), Gx = sibc ? res_group(rows, ne, op->ix_nnz) : G;
        void* args[] = {&s, &K, &G, &Gx};
        return clu_launch((const void*)k_nested_clu, C, clu_smem(ne, w.m, C), args, st);
    }
    const int ctas = res_ctas(ne);
    const int64_t rows = (ne + ctas - 1) / ctas;
    int G = res_group(rows, ne, nnz), Gx = sibc ? res_group(rows, ne, op->ix_nnz) : G;
    SIE_CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(unsigned), st));
    int polls = res_polls();
    void* args[] = {&s, &K, &cnt, &err, &polls, &G, &Gx};
    return res_launch((const void*)k_nested, ctas, res_smem(w.m), args, st);
}

}  // namespace sie

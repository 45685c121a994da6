// The system product (Eq. sys) of the lockstep solves: R <= 8 vectors at once, for
// operators whose interior has no grid (near-region-only and SIBC).
//
// These solves stop at tol_outer and their preconditioner rounds its vectors to
// complex64, so a change of 1e-16 in b moves x of a copper bar by 2.5e-3 (condition
// about 1e4 row-weighted, x itself 5 to 7% from the exact solution at tol_outer 1e-4):
// any other rounding gives another valid x.  To keep the solutions that programs have,
// the product keeps its operations and the order of its sums: FP64 butterflies at
// power-of-two lengths, a lane of 32 per stored entry, one chain per edge (near region,
// I_x, charges after the interpolation).  What may differ is how much one launch does:
// every step takes all vectors in blockIdx.y, and the kernel spectra are read once for
// them.
//
// A bar of 336 triangles, eight right-hand sides, 97 iterations: 723 ms with a launch per
// step and vector, 464 ms now.
#include <algorithm>
#include <cmath>

#include "gridio.cuh"
#include "internal.h"
#include "spmv.cuh"

namespace sie {

// Y_q = A X_q, q < R (blockIdx.y, ldx and ldy apart): a warp per row
__global__ void __launch_bounds__(128) k_blk_csr(int nrow, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                                 const double2* __restrict__ val, const double2* __restrict__ X,
                                                 int64_t ldx, double2* __restrict__ Y, int64_t ldy)
{
    const int r = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    const int lane = threadIdx.x & 31;
    if (r >= nrow) return;
    X += blockIdx.y * ldx;
    double sr = 0, si = 0;
    for (int64_t e = rp[r] + lane; e < rp[r + 1]; e += 32) {
        const double2 v = __ldg(val + e), x = __ldg(X + __ldg(col + e));
        sr += v.x * x.x - v.y * x.y;
        si += v.x * x.y + v.y * x.x;
    }
    for (int off = 16; off > 0; off >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, off);
        si += __shfl_xor_sync(0xffffffffu, si, off);
    }
    if (lane == 0) Y[blockIdx.y * ldy + r] = make_double2(sr, si);
}

sie_status blk_csr(cudaStream_t st, int nrow, const int64_t* rp, const int32_t* col, const double2* val,
                   const double2* X, int64_t ldx, int R, double2* Y, int64_t ldy)
{
    k_blk_csr<<<dim3((nrow + 3) / 4, R), 128, 0, st>>>(nrow, rp, col, val, X, ldx, Y, ldy);
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}

// real and imaginary part of a product with its roundings spelled out (a compiler may
// fuse either of the two products, and does so differently from place to place)
__device__ __forceinline__ double b_re(double2 p, double2 x) { return __fma_rn(p.x, x.x, -__dmul_rn(p.y, x.y)); }
__device__ __forceinline__ double b_im(double2 p, double2 x) { return __fma_rn(p.x, x.y, __dmul_rn(p.y, x.x)); }
__device__ __forceinline__ double b_im2(double2 p, double2 x) { return __fma_rn(p.y, x.x, __dmul_rn(p.x, x.y)); }

// y_q[r] += a1 sum_e v1[e] x1_q[col[e]] + a2 sum_e v2[e] x2_q[col[e]]: a warp per row,
// four loads of each array in flight, one set of sums per unrolled slot
__global__ void __launch_bounds__(128) k_blk_near(int nrow, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                                  const double2* __restrict__ v1, const double2* __restrict__ x1,
                                                  int64_t ld1, double2 a1, const double2* __restrict__ v2,
                                                  const double2* __restrict__ x2, int64_t ld2, double2 a2,
                                                  double2* __restrict__ y, int64_t ldy)
{
    const int r = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    const int lane = threadIdx.x & 31;
    if (r >= nrow) return;
    x1 += blockIdx.y * ld1;
    x2 += blockIdx.y * ld2;
    y += blockIdx.y * ldy;
    double s1r[4] = {0, 0, 0, 0}, s1i[4] = {0, 0, 0, 0}, s2r[4] = {0, 0, 0, 0}, s2i[4] = {0, 0, 0, 0};
    const int64_t e1 = rp[r + 1];
    int64_t e = rp[r] + lane;
    for (; e + 96 < e1; e += 128) {
        int c[4];
        double2 p[4], q[4];
#pragma unroll
        for (int u = 0; u < 4; u++) c[u] = __ldg(col + e + 32 * u);
#pragma unroll
        for (int u = 0; u < 4; u++) {
            p[u] = __ldg(v1 + e + 32 * u);
            q[u] = __ldg(v2 + e + 32 * u);
        }
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const double2 xa = __ldg(x1 + c[u]), xb = __ldg(x2 + c[u]);
            s1r[u] += b_re(p[u], xa);
            s1i[u] += b_im(p[u], xa);
            s2r[u] += b_re(q[u], xb);
            s2i[u] += b_im(q[u], xb);
        }
    }
    for (; e < e1; e += 32) {  // at most 3 more entries per lane
        const int c = __ldg(col + e);
        const double2 p = __ldg(v1 + e), q = __ldg(v2 + e), xa = __ldg(x1 + c), xb = __ldg(x2 + c);
        s1r[0] += b_re(p, xa);
        s1i[0] += b_im2(p, xa);
        s2r[0] += b_re(q, xb);
        s2i[0] += b_im2(q, xb);
    }
    double t1r = (s1r[0] + s1r[1]) + (s1r[2] + s1r[3]), t1i = (s1i[0] + s1i[1]) + (s1i[2] + s1i[3]);
    double t2r = (s2r[0] + s2r[1]) + (s2r[2] + s2r[3]), t2i = (s2i[0] + s2i[1]) + (s2i[2] + s2i[3]);
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

__device__ __forceinline__ double2 b_mul(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// spectral products of Eq. (sys) of R vectors: the seven source spectra of vector q at
// grids 7 q + g, its four result spectra to grids 4 q + g (a node's later vectors lie
// above what it has written)
__global__ void k_blk_specmul(int R, const double2* __restrict__ spec, double2* buf, int64_t nn, double k0)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nn) return;
    const double2 G = spec[i], gx = spec[nn + i], gy = spec[2 * nn + i], gz = spec[3 * nn + i];
    const double2 jG = make_double2(-k0 * G.y, k0 * G.x);  // j k0 G
    for (int q = 0; q < R; q++) {
        double2 in[7];
#pragma unroll
        for (int g = 0; g < 7; g++) in[g] = buf[(7 * q + g) * nn + i];
        const double2 mx = in[3], my = in[4], mz = in[5];
        const double2 cx = b_mul(gy, mz), cy = b_mul(gz, mx), cz = b_mul(gx, my);
        const double2 dx = b_mul(gz, my), dy = b_mul(gx, mz), dz = b_mul(gy, mx);
        const double2 a0 = b_mul(jG, in[0]), a1 = b_mul(jG, in[1]), a2 = b_mul(jG, in[2]);
        double2* o = buf + 4 * q * nn + i;
        o[0] = make_double2(a0.x - (cx.x - dx.x), a0.y - (cx.y - dx.y));
        o[nn] = make_double2(a1.x - (cy.x - dy.x), a1.y - (cy.y - dy.y));
        o[2 * nn] = make_double2(a2.x - (cz.x - dz.x), a2.y - (cz.y - dz.y));
        o[3 * nn] = b_mul(G, in[6]);
    }
}

// per triangle: sigma = -A c0rho, and the charge row y2 = 2 sum_i c_i H_i + j k0 c0rho
__global__ void k_blk_charge(int nt, DevMesh M, const double2* __restrict__ x, int64_t ldx, double k0,
                             double2* __restrict__ sig, double2* __restrict__ y, int64_t ldy)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    const double2* H = x + blockIdx.y * ldx;
    const double2 r = H[M.ne + t];
    sig[blockIdx.y * (int64_t)nt + t] = make_double2(-M.area[t] * r.x, -M.area[t] * r.y);
    double sr = 0, si = 0;
    for (int i = 0; i < 3; i++) {
        const double2 h = H[M.tri_edge[3 * t + i]];
        const double c = 2.0 * M.coef[3 * t + i];
        sr += c * h.x;
        si += c * h.y;
    }
    y[blockIdx.y * ldy + M.ne + t] = make_double2(sr - k0 * r.y, si + k0 * r.x);
}

// y1_m += l_m (phi_{T+} - phi_{T-})
__global__ void k_blk_dt(int ne, int nt, const int32_t* __restrict__ edge_tri, const double* __restrict__ len,
                         const double2* __restrict__ phi, double2* __restrict__ y, int64_t ldy)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= ne) return;
    phi += blockIdx.y * (int64_t)nt;
    y += blockIdx.y * ldy;
    const double2 a = phi[edge_tri[2 * m]], b = phi[edge_tri[2 * m + 1]];
    y[m].x += len[m] * (a.x - b.x);
    y[m].y += len[m] * (a.y - b.y);
}

// grid lengths, kernel spectra and workspace, made by the first lockstep solve and kept
static sie_status blk_prepare(sie_op* op)
{
    BlockWork& w = op->blk;
    if (w.R) return SIE_OK;
    cudaStream_t st = op->mesh->ctx->stream;
    const DevMesh& M = op->mesh->d;
    GridDesc g = op->ext.g;
    for (int d = 0; d < 3; d++)
        for (g.n[d] = 16; g.n[d] < 2 * g.N[d] - 1;) g.n[d] <<= 1;
    const int64_t nn = (int64_t)g.n[0] * g.n[1] * g.n[2], Ng = (int64_t)g.N[0] * g.N[1] * g.N[2];
    // vectors at a time: up to 512 MB of padded grids (128^3: two vectors; the spectra are shared by them)
    const int R = (int)std::max<int64_t>(1, std::min<int64_t>(8, (512 << 20) / (7 * 16 * nn)));
    w.g = g;
    auto get = [&](double2** p, int64_t n) {
        return *p ? cudaSuccess : cudaMallocAsync((void**)p, sizeof(double2) * n, st);
    };
    SIE_CUDA_TRY(get(&w.spec, 4 * nn));
    SIE_CUDA_TRY(get(&w.buf, 7 * nn * R));
    SIE_CUDA_TRY(get(&w.src, 7 * Ng * R));
    SIE_CUDA_TRY(get(&w.tc, 9 * (int64_t)M.nt * R));
    SIE_CUDA_TRY(get(&w.tri, 2 * (int64_t)M.nt * 8));
    SIE_TRY(aim_sample(st, g, op->ext.kr, op->ext.ki, w.spec));
    SIE_TRY(fft3d_p2(st, w.spec, nullptr, g, -1, 0, nullptr, 4));
    w.R = R;
    return SIE_OK;
}

void blk_release(sie_op* op)
{
    cudaStream_t st = op->mesh->ctx->stream;
    for (double2* p : {op->blk.spec, op->blk.buf, op->blk.src, op->blk.tc, op->blk.tri})
        if (p) cudaFreeAsync(p, st);
    op->blk = BlockWork();
}

// y_q = SYS [H_q; c0rho_q] with E_q = Z' H_q given, q < R: x_q = [H_q; c0rho_q] ldx
// apart, E_q lde apart, y_q ldy apart
sie_status blk_sys_rest(sie_op* op, int R, const double2* x, int64_t ldx, const double2* E, int64_t lde, double2* y,
                        int64_t ldy)
{
    sie_ctx* c = op->mesh->ctx;
    cudaStream_t st = c->stream;
    SIE_TRY(blk_prepare(op));
    const BlockWork& w = op->blk;
    const DevMesh& M = op->mesh->d;
    const AimOp& X = op->ext;
    const GridDesc& g = w.g;
    const int ne = M.ne, nt = M.nt, S = (g.M + 1) * (g.M + 1) * (g.M + 1);
    const int64_t nn = (int64_t)g.n[0] * g.n[1] * g.n[2], Ng = (int64_t)g.N[0] * g.N[1] * g.N[2];
    SIE_CUDA_TRY(cudaMemset2DAsync(y, sizeof(double2) * std::max<int64_t>(ldy, ne), 0, sizeof(double2) * ne, R, st));
    for (int q0 = 0; q0 < R; q0 += w.R) {
        const int r = std::min(w.R, R - q0);
        const double2 *xq = x + q0 * ldx, *Eq = E + q0 * lde;
        {
            Stage s_(c, "project_sys");
            k_tri_coef<double2><<<dim3((nt + 127) / 128, r), 128, 0, st>>>(nt, M, xq, ldx, Eq, lde, xq + ne, ldx, w.tc);
            SIE_CUDA_TRY(cudaMemsetAsync(w.src, 0, sizeof(double2) * 7 * Ng * r, st));
            k_project_gather<double2, double, false><<<dim3(gio_blocks(op->pm_nnode, 8), r), 256, 0, st>>>(
                op->pm_nnode, op->pm_node, op->pm_ptr, op->pm_ent, S, op->W, w.tc, nt, w.src, Ng);
            SIE_CUDA_TRY(cudaGetLastError());
        }
        SIE_TRY(fft3d_p2(st, w.buf, w.src, g, -1, 1, c, 7 * r));
        {
            Stage s_(c, "specmul_sys");
            k_blk_specmul<<<(unsigned)((nn + 127) / 128), 128, 0, st>>>(r, w.spec, w.buf, nn, op->k0);
            SIE_CUDA_TRY(cudaGetLastError());
        }
        SIE_TRY(fft3d_p2(st, w.buf, w.src, g, +1, 1, c, 4 * r));
        Stage s_(c, "interp");
        k_interp<32, double2, double, 4><<<dim3(gio_blocks(nt, 32, GIO_SMALL), r), GIO_SMALL, 0, st>>>(
            nt, S, g.M, M, op->base, op->W, w.src, g, make_double2(1.0, 0.0), Ng, y + q0 * ldy, ldy);
        SIE_CUDA_TRY(cudaGetLastError());
    }
    {
        Stage s_(c, "spmv_near_ext");
        k_blk_near<<<dim3((ne + 3) / 4, R), 128, 0, st>>>(ne, X.row_ptr, X.col, X.valLA, x, ldx,
                                                          make_double2(0.0, op->k0), X.valK, E, lde,
                                                          make_double2(-1.0, 0.0), y, ldy);
        SIE_CUDA_TRY(cudaGetLastError());
    }
    Stage s_(c, "spmv_sys_rest");
    double2 *sig = w.tri, *phi = w.tri + 8 * (int64_t)nt;
    k_blk_charge<<<dim3((nt + 127) / 128, R), 128, 0, st>>>(nt, M, x, ldx, op->k0, sig, y, ldy);
    SIE_CUDA_TRY(csr_launch_g(st, BLK_IX_LANES, ne, op->ix_row_ptr, op->ix_col, op->ix_val, E, make_double2(-0.5, 0.0),
                              true, y, R, lde, ldy));
    SIE_CUDA_TRY(csr_launch_g(st, BLK_TRI_LANES, nt, X.tri_row_ptr, X.tri_col, X.valLphi, sig, make_double2(1.0, 0.0),
                              false, phi, R, nt, nt));
    k_blk_dt<<<dim3((ne + 127) / 128, R), 128, 0, st>>>(ne, nt, M.edge_tri, op->elen, phi, y, ldy);
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}

}  // namespace sie

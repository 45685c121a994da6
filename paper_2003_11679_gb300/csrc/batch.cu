// Multi-right-hand-side AIM products (Eqs. AIM_Lin, AIM_Kin) for a block of up
// to RB vectors: one launch per step for all of them, and the near-region values
// are read once per block instead of once per vector.
//   * projection: one grid of CTAs per right-hand side (gridio.cuh; weights from L2);
//   * FFTs: one launch per pass over all grids of the block;
//   * z transforms and spectral products: one row of CTAs per right-hand side, each
//     reading the spectra of its columns (fft.cuh; mostly from L2); z lengths above
//     256 multiply in a kernel of their own, which loads G (or grad G) once per node;
//   * interpolation: one grid of CTAs per right-hand side;
//   * near region: CSR x panel product, each (column, value) pair loaded once.
// Vectors are rhs-major (vector r at r * len), as everywhere in the ABI.
#include <algorithm>
#include <complex>

#include "internal.h"

namespace sie {

constexpr int RB = 8;  // right-hand sides per block

// spectral multiply of nr vectors, the spectra read once per node: mode 0
// (L): every grid times G; mode 1 (K): J <- grad G x J
__global__ void k_specmul_b(int mode, int nr, const double2* __restrict__ spec, double2* __restrict__ buf, int64_t nn)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nn) return;
    auto mul = [](double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); };
    if (mode == 0) {
        const double2 G = spec[i];
        for (int c = 0; c < 4 * nr; c++) buf[c * nn + i] = mul(G, buf[c * nn + i]);
    } else {
        const double2 gx = spec[nn + i], gy = spec[2 * nn + i], gz = spec[3 * nn + i];
        for (int r = 0; r < nr; r++) {
            double2* b = buf + (int64_t)3 * r * nn;
            double2 jx = b[i], jy = b[nn + i], jz = b[2 * nn + i];
            double2 p = mul(gy, jz), q = mul(gz, jy);
            b[i] = make_double2(p.x - q.x, p.y - q.y);
            p = mul(gz, jx);
            q = mul(gx, jz);
            b[nn + i] = make_double2(p.x - q.x, p.y - q.y);
            p = mul(gx, jy);
            q = mul(gy, jx);
            b[2 * nn + i] = make_double2(p.x - q.x, p.y - q.y);
        }
    }
}

// Y[r] = A X[r] for r < nr <= GL: a warp per row.  GL lanes share an entry, one
// right-hand side each, so 32 / GL entries are in work at a time; the value is one
// broadcast load and the vectors, interleaved by k_pack_rhs, one coalesced row of GL
// per entry (rhs-major vectors cost nr scattered 16-byte gathers).  Only the 32 / GL
// entry slots are summed across lanes.  FP64 arithmetic bounds it: eight right-hand
// sides, 15.0 M entries: 1,533 us with an entry per lane and 8 x 10 warp-wide additions
// a row; 843 us now (765 us of products).
template <int GL>
__global__ void __launch_bounds__(128) k_csr_panel(int nrow, const int64_t* __restrict__ rp,
                                                   const int32_t* __restrict__ col, const double2* __restrict__ val,
                                                   const double2* __restrict__ Xp, int nr,
                                                   double2* __restrict__ Y, int64_t ldy)
{
    const int row = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    const int lane = threadIdx.x & 31, r = lane % GL, sl = lane / GL;
    constexpr int STEP = 32 / GL, U = 4;
    if (row >= nrow) return;
    double sr[U], si[U];  // independent chains
#pragma unroll
    for (int u = 0; u < U; u++) sr[u] = si[u] = 0.0;
    const int64_t e1 = rp[row + 1];
    int64_t e = rp[row] + sl;
    for (; e + (U - 1) * STEP < e1; e += U * STEP) {
        int c[U];
        double2 v[U], x[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            c[u] = __ldg(col + e + u * STEP);
            v[u] = __ldg(val + e + u * STEP);
        }
#pragma unroll
        for (int u = 0; u < U; u++) x[u] = __ldg(Xp + (int64_t)c[u] * GL + r);
#pragma unroll
        for (int u = 0; u < U; u++) {
            sr[u] = fma(v[u].x, x[u].x, fma(-v[u].y, x[u].y, sr[u]));
            si[u] = fma(v[u].x, x[u].y, fma(v[u].y, x[u].x, si[u]));
        }
    }
    for (; e < e1; e += STEP) {
        const double2 v = __ldg(val + e), x = __ldg(Xp + (int64_t)__ldg(col + e) * GL + r);
        sr[0] = fma(v.x, x.x, fma(-v.y, x.y, sr[0]));
        si[0] = fma(v.x, x.y, fma(v.y, x.x, si[0]));
    }
    double yr = (sr[0] + sr[1]) + (sr[2] + sr[3]), yi = (si[0] + si[1]) + (si[2] + si[3]);
#pragma unroll
    for (int off = GL; off < 32; off <<= 1) {
        yr += __shfl_xor_sync(0xffffffffu, yr, off);
        yi += __shfl_xor_sync(0xffffffffu, yi, off);
    }
    if (sl == 0 && r < nr) Y[r * ldy + row] = make_double2(yr, yi);
}

// Xp[c GL + r] = X[r ldx + c], zero for r >= nr
__global__ void k_pack_rhs(int64_t n, int nr, int GL, const double2* __restrict__ X, int64_t ldx,
                           double2* __restrict__ Xp)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * GL) return;
    const int64_t c = i / GL;
    const int r = (int)(i % GL);
    Xp[i] = r < nr ? X[r * ldx + c] : make_double2(0, 0);
}

// Y = A X for nr <= RB vectors of an edge CSR matrix, rhs-major, on st; the values
// read once for all nr
static sie_status csr_panel(sie_op* op, cudaStream_t st, const int64_t* rp, const int32_t* col, const double2* val,
                            const double2* X, int nr, double2* Y)
{
    const int ne = op->mesh->d.ne;
    const int GL = nr > 4 ? 8 : (nr > 2 ? 4 : 2);
    k_pack_rhs<<<(unsigned)(((int64_t)ne * GL + 255) / 256), 256, 0, st>>>(ne, nr, GL, X, ne, op->bws_xp);
    const unsigned blocks = (unsigned)((ne + 3) / 4);
    if (GL == 8)
        k_csr_panel<8><<<blocks, 128, 0, st>>>(ne, rp, col, val, op->bws_xp, nr, Y, ne);
    else if (GL == 4)
        k_csr_panel<4><<<blocks, 128, 0, st>>>(ne, rp, col, val, op->bws_xp, nr, Y, ne);
    else
        k_csr_panel<2><<<blocks, 128, 0, st>>>(ne, rp, col, val, op->bws_xp, nr, Y, ne);
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}

// the block workspace: padded and compact grids for RB vectors of 4 grids
static sie_status batch_workspace(sie_op* op, double2** bufs, double2** src)
{
    const GridDesc& g = op->ext.g;
    const int64_t nn = (int64_t)g.n[0] * g.n[1] * g.n[2], Ng = (int64_t)g.N[0] * g.N[1] * g.N[2];
    cudaStream_t st = op->mesh->ctx->stream;
    if (!op->bws_bufs) {
        SIE_CUDA_TRY(cudaMallocAsync((void**)&op->bws_bufs, sizeof(double2) * 4 * RB * nn, st));
        SIE_CUDA_TRY(cudaMallocAsync((void**)&op->bws_src, sizeof(double2) * 4 * RB * Ng, st));
        SIE_CUDA_TRY(cudaMallocAsync((void**)&op->bws_tc, sizeof(double2) * 4 * RB * op->mesh->d.nt, st));
    }
    *bufs = op->bws_bufs;
    *src = op->bws_src;
    return SIE_OK;
}

// Y = A X for nr vectors (nr <= RB, rhs-major, length N_e), A = L (which_LK 0)
// or K (1) of operator a
sie_status aim_apply_block(sie_op* op, AimOp& a, int which_LK, const double2* X, double2* Y, int nr)
{
    sie_ctx* pc = op->mesh->ctx;
    cudaStream_t st = pc->stream;
    const DevMesh& M = op->mesh->d;
    const int64_t ne = M.ne;
    if (nr < 1 || nr > RB) {
        set_error("aim_apply_block: block size out of range");
        return SIE_ERR_ARG;
    }
    if (!op->bws_xp) SIE_CUDA_TRY(cudaMallocAsync((void**)&op->bws_xp, sizeof(double2) * RB * ne, st));
    // the near part (FP64 products) on a branch beside the grid part (atomics and integer
    // transforms), at every size: K of two and eight right-hand sides 65 -> 57 and 89 -> 77 us
    // at 80 triangles, eight at 1,280 308 -> 293 us, L at 20,480 3,457 -> 3,409 us (both parts
    // wait for issue slots there).  The stage timers need one stream.
    Branch br(op, a.has_grid && !pc->prof.on);
    {
        SIE_CUDA_TRY(br.follow());
        Stage s_(pc, a.has_grid ? "spmv_block" : "spmv_near_only_block");
        const double2* v = which_LK == 0 ? a.valL : a.valK;
        SIE_TRY(csr_panel(op, br.st(), a.row_ptr, a.col, v, X, nr, Y));
    }
    if (a.has_grid) {
        const GridDesc& g = a.g;
        const int64_t nn = (int64_t)g.n[0] * g.n[1] * g.n[2];
        const int ngrid = which_LK == 0 ? 4 : 3;
        double2 *buf, *src;
        SIE_TRY(batch_workspace(op, &buf, &src));
        {
            Stage s_(pc, "project_block");
            SIE_TRY(aim_project(op, X, ne, nr, ngrid, op->bws_tc, src));
        }
        if (fft_fused_z(g)) {
            SIE_TRY(fft_lk(st, which_LK, buf, src, g, a.spec, pc, nr));
        } else {
            SIE_TRY(fft3d(st, buf, src, g, -1, 1, pc, ngrid * nr));
            {
                Stage s_(pc, "specmul_block");
                k_specmul_b<<<(unsigned)((nn + 255) / 256), 256, 0, st>>>(which_LK, nr, a.spec, buf, nn);
                SIE_CUDA_TRY(cudaGetLastError());
            }
            SIE_TRY(fft3d(st, buf, src, g, +1, 1, pc, ngrid * nr));
        }
        std::complex<double> kk(a.kr, a.ki);
        std::complex<double> sc = which_LK == 0 ? -1.0 / (kk * kk) : std::complex<double>(0.0);
        {
            SIE_CUDA_TRY(br.join());
            Stage s_(pc, "interp_block");
            SIE_TRY(aim_interp(op, src, which_LK == 0, make_double2(sc.real(), sc.imag()), Y, ne, nr));
        }
    }
    return SIE_OK;
}

}  // namespace sie

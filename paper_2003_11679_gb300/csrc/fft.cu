// FFTs of the AIM grid path: twiddle tables, pass dispatch by length, pruned 3D
// transforms and the grid products (forward, spectral product, inverse).
// Lengths to 256 take the two-pass kernels of fft.cuh (fixed point for
// complex128), 512 and 1024 the Stockham kernel below, and so do all (power-of-two)
// lengths of the lockstep block product, whose FP64 butterflies are part of what its
// solutions are to the last bit (block.cu).
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "fft.cuh"

namespace sie {

SIE_FFT_LENGTHS(SIE_FFT_EXTERN)

// ------------------------------------------------------------------ twiddles
// exp(-2 pi i m / n), m < n: one set of tables per device and length, made on
// first use (guarded: contexts may run in threads) and kept for the process
constexpr int TW_MAXDEV = 64, TW_MAXLEN = 1024;
struct TwTab {
    double2* d = nullptr;  // (cos, -sin); powers of two
    float2* f = nullptr;   // n <= 256: (cos, sin); else (cos, -sin)
    twq* q = nullptr;      // n <= 256
};
static TwTab g_tw[TW_MAXDEV][TW_MAXLEN + 1];
static std::mutex g_tw_mu;

template <class T>
static sie_status tw_upload(T** d, const std::vector<T>& h)
{
    SIE_CUDA_TRY(cudaMalloc((void**)d, sizeof(T) * h.size()));
    SIE_CUDA_TRY(cudaMemcpy(*d, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice));
    return SIE_OK;
}

static sie_status twiddles(int n, TwTab* out)
{
    int dev = 0;
    SIE_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= TW_MAXDEV || n < 1 || n > TW_MAXLEN) {
        set_error("twiddles: device ordinal or length out of range");
        return SIE_ERR_ARG;
    }
    std::lock_guard<std::mutex> lk(g_tw_mu);
    TwTab& t = g_tw[dev][n];
    if (!t.f) {
        const bool small = n <= 256;
        std::vector<double2> hd(n);
        std::vector<float2> hf(n);
        std::vector<twq> hq(n);
        for (int m = 0; m < n; m++) {
            const long double a = 2.0L * 3.14159265358979323846264338327950288L * (long double)m / (long double)n;
            const long double c = cosl(a), s = sinl(a);
            hd[m] = make_double2((double)c, (double)-s);
            hf[m] = make_float2((float)c, (float)(small ? s : -s));
            const auto q = [](long double v) { return to_q62((long long)llroundl(ldexpl(v, 62))); };
            hq[m] = twq{q(c), q(c + s), q(s - c)};
        }
        if (small) SIE_TRY(tw_upload(&t.q, hq));
        if ((n & (n - 1)) == 0) SIE_TRY(tw_upload(&t.d, hd));
        SIE_TRY(tw_upload(&t.f, hf));
    }
    *out = t;
    return SIE_OK;
}

// ------------------------------------------------------------------ powers of two: Stockham FFT (register radix-8, FP64 / FP32)
// Self-sorting Stockham formulation (Govindaraju et al., SC'08): pass p with
// current span Ns and radix R: thread j loads a[r] = x[j + r n/R], multiplies
// by exp(-+2 pi i (j mod Ns) r / (Ns R)), does an R-point DFT in registers and
// stores y[(j / Ns) Ns R + (j mod Ns) + r Ns].  n/8 threads per pencil; the
// first pass reads the (zero padded) pencil straight from global memory, the
// last writes the (truncated) output straight to global memory, the passes in
// between exchange through shared memory.
template <class C, int INV>
__device__ __forceinline__ void cmulw(C& a, C w)
{
    C t;
    if (INV) w.y = -w.y;
    t.x = a.x * w.x - a.y * w.y;
    t.y = a.x * w.y + a.y * w.x;
    a = t;
}

template <class C, int INV>
__device__ __forceinline__ void bfly2(C& a, C& b)
{
    C t = a;
    a.x = t.x + b.x;
    a.y = t.y + b.y;
    b.x = t.x - b.x;
    b.y = t.y - b.y;
}

// multiply by -j (forward) or +j (inverse)
template <class C, int INV>
__device__ __forceinline__ C mulmj(C a)
{
    C t;
    if (INV) {
        t.x = -a.y;
        t.y = a.x;
    } else {
        t.x = a.y;
        t.y = -a.x;
    }
    return t;
}

template <class C, int INV>
__device__ __forceinline__ void dft4(C& a0, C& a1, C& a2, C& a3)
{
    // X0 = (a0+a2)+(a1+a3), X2 = (a0+a2)-(a1+a3), X1 = (a0-a2) -+j (a1-a3), X3 = (a0-a2) +-j (a1-a3)
    bfly2<C, INV>(a0, a2);
    bfly2<C, INV>(a1, a3);
    a3 = mulmj<C, INV>(a3);
    bfly2<C, INV>(a0, a1);
    bfly2<C, INV>(a2, a3);
    // now a0 = X0, a1 = X2, a2 = X1, a3 = X3 -> reorder
    C t = a1;
    a1 = a2;
    a2 = t;
}

template <class C, int INV>
__device__ __forceinline__ void dft8(C* a)
{
    // even/odd split: E = DFT4(a0,a2,a4,a6), O = DFT4(a1,a3,a5,a7)
    dft4<C, INV>(a[0], a[2], a[4], a[6]);
    dft4<C, INV>(a[1], a[3], a[5], a[7]);
    const double r = 0.70710678118654752440;
    // O[k] *= W8^k : W8 = (1 -+ j)/sqrt2, W8^2 = -+j, W8^3 = (-1 -+ j)/sqrt2
    C o1 = a[3], o2 = a[5], o3 = a[7];
    C t;
    if (!INV) {
        t.x = (o1.x + o1.y) * r;
        t.y = (o1.y - o1.x) * r;
    } else {
        t.x = (o1.x - o1.y) * r;
        t.y = (o1.y + o1.x) * r;
    }
    o1 = t;
    o2 = mulmj<C, INV>(o2);
    if (!INV) {
        t.x = (o3.y - o3.x) * r;
        t.y = -(o3.x + o3.y) * r;
    } else {
        t.x = -(o3.x + o3.y) * r;
        t.y = (o3.x - o3.y) * r;
    }
    o3 = t;
    // E[k] in a[0], a[2], a[4], a[6]; O[k] (twiddled) in a[1], o1, o2, o3
    C e0 = a[0], e1 = a[2], e2 = a[4], e3 = a[6], q0 = a[1];
    a[0].x = e0.x + q0.x; a[0].y = e0.y + q0.y;
    a[4].x = e0.x - q0.x; a[4].y = e0.y - q0.y;
    a[1].x = e1.x + o1.x; a[1].y = e1.y + o1.y;
    a[5].x = e1.x - o1.x; a[5].y = e1.y - o1.y;
    a[2].x = e2.x + o2.x; a[2].y = e2.y + o2.y;
    a[6].x = e2.x - o2.x; a[6].y = e2.y - o2.y;
    a[3].x = e3.x + o3.x; a[3].y = e3.y + o3.y;
    a[7].x = e3.x - o3.x; a[7].y = e3.y - o3.y;
}

template <class C, int INV, int R>
__device__ __forceinline__ void dftR(C* a)
{
    if constexpr (R == 8)
        dft8<C, INV>(a);
    else if constexpr (R == 4)
        dft4<C, INV>(a[0], a[1], a[2], a[3]);
    else
        bfly2<C, INV>(a[0], a[1]);
}

// one Stockham pass of radix R over the pencil held by (tp = thread in pencil);
// SRC / DST: 0 = global, 1 = shared memory
template <int LOGN, int R, int SRC, int DST, class C, int INV>
__device__ __forceinline__ void stockham_pass(int Ns, int tp, const C* gin, int64_t gbase_in, int64_t gst_in,
                                              int n_in, C* gout, int64_t gbase_out, int64_t gst_out, int n_out,
                                              bool valid, const C* sin, C* sout, const C* __restrict__ tw)
{
    constexpr int n = 1 << LOGN;
    constexpr int TPP = n / 8;  // threads per pencil
    constexpr int NB = n / R;   // butterflies per pencil
    constexpr int LR = R == 8 ? 3 : (R == 4 ? 2 : 1);
    const int lns = __ffs(Ns) - 1;  // log2(Ns)
    for (int jj = tp; jj < NB; jj += TPP) {
        C a[R];
        for (int r = 0; r < R; r++) {
            int idx = jj + r * NB;
            if (SRC == 0) {
                C v;
                v.x = 0;
                v.y = 0;
                if (valid && idx < n_in) v = gin[gbase_in + (int64_t)idx * gst_in];
                a[r] = v;
            } else {
                a[r] = sin[idx];
            }
        }
        // Ns and R are powers of two: masks and shifts instead of divisions
        const int k = jj & (Ns - 1);
        if (Ns > 1)
            for (int r = 1; r < R; r++) cmulw<C, INV>(a[r], tw[(k * r) << (LOGN - lns - LR)]);
        dftR<C, INV, R>(a);
        const int o = ((jj >> lns) << (lns + LR)) + k;
        for (int r = 0; r < R; r++) {
            int idx = o + r * Ns;
            if (DST == 0) {
                if (valid && idx < n_out) gout[gbase_out + (int64_t)idx * gst_out] = a[r];
            } else {
                sout[idx] = a[r];
            }
        }
    }
}

template <int LOGN, int PB, class C, int INV>
__global__ void __launch_bounds__(PB*(1 << LOGN) / 8) k_fft_stockham(const C* in, C* out, const C* __restrict__ tw,
                                                                     PassGeom G)
{
    constexpr int n = 1 << LOGN;
    constexpr int TPP = n / 8;
    constexpr int pitch = n + 1;
    extern __shared__ __align__(16) unsigned char smraw2[];
    C* sm0 = reinterpret_cast<C*>(smraw2);
    C* sm1 = sm0 + PB * pitch;
    // pencil-fastest thread order on strided passes keeps rows coalesced
    int pl, tp;
    if (G.contig) {
        pl = threadIdx.x / TPP;
        tp = threadIdx.x % TPP;
    } else {
        pl = threadIdx.x % PB;
        tp = threadIdx.x / PB;
    }
    int64_t p = (int64_t)blockIdx.x * PB + pl;
    bool valid = p < G.npencil;
    int64_t bin = valid ? (p % G.L) * G.slo_in + (p / G.L) * G.shi_in + blockIdx.y * G.bs_in : 0;
    int64_t bout = valid ? (p % G.L) * G.slo_out + (p / G.L) * G.shi_out + blockIdx.y * G.bs_out : 0;
    C* s0 = sm0 + pl * pitch;
    C* s1 = sm1 + pl * pitch;
    // radix plan: 8^a x (1, 2 or 4)
    constexpr int NP8 = LOGN / 3, REM = LOGN % 3;
    constexpr int NPASS = NP8 + (REM ? 1 : 0);
    int Ns = 1;
    // pass 0 (global -> smem or global)
    if constexpr (NPASS == 1) {
        stockham_pass<LOGN, 8, 0, 0, C, INV>(Ns, tp, in, bin, G.st_in, G.n_in, out, bout, G.st_out, G.n_out, valid,
                                             nullptr, nullptr, tw);
        return;
    } else {
        stockham_pass<LOGN, 8, 0, 1, C, INV>(Ns, tp, in, bin, G.st_in, G.n_in, nullptr, 0, 0, 0, valid, nullptr, s0,
                                             tw);
    }
    Ns *= 8;
    __syncthreads();
    C* cur = s0;
    C* nxt = s1;
    for (int ps = 1; ps < NP8; ps++) {
        bool last = (ps == NPASS - 1);
        if (last) {
            stockham_pass<LOGN, 8, 1, 0, C, INV>(Ns, tp, nullptr, 0, 0, 0, out, bout, G.st_out, G.n_out, valid, cur,
                                                 nullptr, tw);
            return;
        }
        stockham_pass<LOGN, 8, 1, 1, C, INV>(Ns, tp, nullptr, 0, 0, 0, nullptr, 0, 0, 0, valid, cur, nxt, tw);
        Ns *= 8;
        __syncthreads();
        C* t = cur;
        cur = nxt;
        nxt = t;
    }
    if constexpr (REM == 1)
        stockham_pass<LOGN, 2, 1, 0, C, INV>(Ns, tp, nullptr, 0, 0, 0, out, bout, G.st_out, G.n_out, valid, cur,
                                             nullptr, tw);
    else if constexpr (REM == 2)
        stockham_pass<LOGN, 4, 1, 0, C, INV>(Ns, tp, nullptr, 0, 0, 0, out, bout, G.st_out, G.n_out, valid, cur,
                                             nullptr, tw);
}

template <int LOGN, int PB, class C>
static sie_status launch_stockham_pb(cudaStream_t st, const C* in, C* out, int inv, const PassGeom& G, const C* tw,
                                  int nbatch)
{
    constexpr int n = 1 << LOGN;
    const size_t smem = sizeof(C) * 2 * PB * (n + 1);
    const auto fn = inv ? k_fft_stockham<LOGN, PB, C, 1> : k_fft_stockham<LOGN, PB, C, 0>;
    SIE_CUDA_TRY(kernel_limit((const void*)fn, smem));
    const unsigned blocks = (unsigned)((G.npencil + PB - 1) / PB);
    fn<<<dim3(blocks, nbatch), PB * n / 8, smem, st>>>(in, out, tw, G);
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}

// 256 threads, n / 8 per pencil; half of that where it would leave less than 4 CTAs an SM
template <int LOGN, class C>
static sie_status launch_stockham(cudaStream_t st, const C* in, C* out, int inv, const PassGeom& G, const C* tw,
                                  int nbatch)
{
    constexpr int PB = 2048 >> LOGN;
    if (G.npencil * nbatch / PB >= 4LL * 152) return launch_stockham_pb<LOGN, PB, C>(st, in, out, inv, G, tw, nbatch);
    return launch_stockham_pb<LOGN, PB / 2, C>(st, in, out, inv, G, tw, nbatch);
}

// ------------------------------------------------------------------ dispatch by length
template <class C>
struct PolicyOf;
template <>
struct PolicyOf<double2> {
    using P = Fx;
    static const twq* tw(const TwTab& t) { return t.q; }
    static const double2* tws(const TwTab& t) { return t.d; }
};
template <>
struct PolicyOf<float2> {
    using P = F32;
    static const float2* tw(const TwTab& t) { return t.f; }
    static const float2* tws(const TwTab& t) { return t.f; }
};

template <class C>
static sie_status launch_pass(cudaStream_t st, int n, const C* in, C* out, int inv, const PassGeom& G, int nb)
{
    using PO = PolicyOf<C>;
    using P = typename PO::P;
    TwTab t;
    SIE_TRY(twiddles(n, &t));
    switch (n) {
#define SIE_CASE(N) \
    case N: return fft_pass_n<N, P>(st, in, out, inv, G, nb, PO::tw(t));
        SIE_FFT_LENGTHS(SIE_CASE)
#undef SIE_CASE
        case 512: return launch_stockham<9, C>(st, in, out, inv, G, PO::tws(t), nb);
        case 1024: return launch_stockham<10, C>(st, in, out, inv, G, PO::tws(t), nb);
    }
    set_error("unsupported FFT length");
    return SIE_ERR_UNSUPPORTED;
}

// FP64 butterflies at any power of two
static sie_status launch_pass_p2(cudaStream_t st, int n, const double2* in, double2* out, int inv, const PassGeom& G,
                                 int nb)
{
    TwTab t;
    SIE_TRY(twiddles(n, &t));
    switch (n) {
        case 16: return launch_stockham<4, double2>(st, in, out, inv, G, t.d, nb);
        case 32: return launch_stockham<5, double2>(st, in, out, inv, G, t.d, nb);
        case 64: return launch_stockham<6, double2>(st, in, out, inv, G, t.d, nb);
        case 128: return launch_stockham<7, double2>(st, in, out, inv, G, t.d, nb);
        case 256: return launch_stockham<8, double2>(st, in, out, inv, G, t.d, nb);
        case 512: return launch_stockham<9, double2>(st, in, out, inv, G, t.d, nb);
        case 1024: return launch_stockham<10, double2>(st, in, out, inv, G, t.d, nb);
    }
    set_error("unsupported FFT length");
    return SIE_ERR_UNSUPPORTED;
}

template <int MODE, class C, class R>
static sie_status launch_z(cudaStream_t st, int n, C* buf, const C* spec, int nz_phys, int64_t ncol, int64_t bnn, int nb,
                           R k0)
{
    using PO = PolicyOf<C>;
    using P = typename PO::P;
    TwTab t;
    SIE_TRY(twiddles(n, &t));
    const int64_t batch = ZMode<MODE>::NI * bnn;
    switch (n) {
#define SIE_CASE(N) \
    case N: return fft_z_n<N, P, MODE>(st, buf, spec, nz_phys, ncol, ncol, bnn, batch, nb, k0, PO::tw(t));
        SIE_FFT_LENGTHS(SIE_CASE)
#undef SIE_CASE
    }
    set_error("fused z stage: unsupported FFT length");
    return SIE_ERR_UNSUPPORTED;
}

// dir = -1: forward transform of the compact N grid `src` (or, prune = 0, of the
// full n grid already in buf) into the full spectrum in buf.
// dir = +1: inverse of the spectrum in buf; prune = 1 writes only the physical
// N box into the compact array `src` (used as output), prune = 0 keeps n^3 in buf.
// nbatch grids at once: grid k at buf + k n^3 and (compact) src + k N^3
template <class C, class PASS>
static sie_status fft3d_t(PASS pass, cudaStream_t st, C* buf, const C* src, const GridDesc& g, int dir, int prune, sie_ctx* pc,
                          int nbatch)
{
    const int64_t nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int64_t Nx = prune ? g.N[0] : nx, Ny = prune ? g.N[1] : ny, Nz = prune ? g.N[2] : nz;
    const int64_t pyz = nx * ny;  // padded plane
    const int64_t bnn = nx * ny * nz, bNg = (int64_t)g.N[0] * g.N[1] * g.N[2];
    if (dir < 0) {
        // x pass: pencils (y < Ny, z < Nz)
        PassGeom X{(int)Nx, (int)nx, Ny * Nz, (int)Ny, prune ? Nx : nx, prune ? Nx * Ny : pyz, 1, nx, pyz, 1, 1,
                   prune ? bNg : bnn, bnn};
        {
            Stage s_(pc, "fft_fwd_x");
            SIE_TRY(pass(st, (int)nx, prune ? src : buf, buf, 0, X, nbatch));
        }
        // y pass: pencils (x < nx, z < Nz)
        PassGeom Y{(int)Ny, (int)ny, nx * Nz, (int)nx, 1, pyz, nx, 1, pyz, nx, 0, bnn, bnn};
        {
            Stage s_(pc, "fft_fwd_y");
            SIE_TRY(pass(st, (int)ny, buf, buf, 0, Y, nbatch));
        }
        // z pass: pencils (x < nx, y < ny)
        PassGeom Z{(int)Nz, (int)nz, nx * ny, (int)nx, 1, nx, pyz, 1, nx, pyz, 0, bnn, bnn};
        {
            Stage s_(pc, "fft_fwd_z");
            SIE_TRY(pass(st, (int)nz, buf, buf, 0, Z, nbatch));
        }
    } else {
        PassGeom Z{(int)nz, (int)Nz, nx * ny, (int)nx, 1, nx, pyz, 1, nx, pyz, 0, bnn, bnn};
        {
            Stage s_(pc, "fft_inv_z");
            SIE_TRY(pass(st, (int)nz, buf, buf, 1, Z, nbatch));
        }
        PassGeom Y{(int)ny, (int)Ny, nx * Nz, (int)nx, 1, pyz, nx, 1, pyz, nx, 0, bnn, bnn};
        {
            Stage s_(pc, "fft_inv_y");
            SIE_TRY(pass(st, (int)ny, buf, buf, 1, Y, nbatch));
        }
        C* dst = prune ? const_cast<C*>(src) : buf;
        PassGeom X{(int)nx, (int)Nx, Ny * Nz, (int)Ny, nx, pyz, 1, prune ? Nx : nx, prune ? Nx * Ny : pyz, 1, 1,
                   bnn, prune ? bNg : bnn};
        {
            Stage s_(pc, "fft_inv_x");
            SIE_TRY(pass(st, (int)nx, buf, dst, 1, X, nbatch));
        }
    }
    return SIE_OK;
}

sie_status fft3d(cudaStream_t st, double2* buf, const double2* src, const GridDesc& g, int dir, int prune, sie_ctx* pc,
                 int nbatch)
{
    return fft3d_t(launch_pass<double2>, st, buf, src, g, dir, prune, pc, nbatch);
}

sie_status fft3d(cudaStream_t st, float2* buf, const float2* src, const GridDesc& g, int dir, int prune, sie_ctx* pc,
                 int nbatch)
{
    return fft3d_t(launch_pass<float2>, st, buf, src, g, dir, prune, pc, nbatch);
}

sie_status fft3d_p2(cudaStream_t st, double2* buf, const double2* src, const GridDesc& g, int dir, int prune, sie_ctx* pc,
                    int nbatch)
{
    return fft3d_t(launch_pass_p2, st, buf, src, g, dir, prune, pc, nbatch);
}

// Grid product with the fused z stage: forward x and y passes of the compact
// source grids in src (into buf), forward z + spectral product + inverse z, then
// the inverse y and x passes of the result grids back into the compact src.
// nb products at once (source grids of product r at r NI N^3 and r NI n^3).
template <int MODE, class C, class R>
static sie_status fft_prod_t(cudaStream_t st, C* buf, C* src, const GridDesc& g, const C* spec, R k0, sie_ctx* pc,
                             int nb)
{
    constexpr int NI = ZMode<MODE>::NI, NO = ZMode<MODE>::NO;
    const int64_t nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int64_t Nx = g.N[0], Ny = g.N[1], Nz = g.N[2];
    const int64_t pyz = nx * ny, bnn = nx * ny * nz, bNg = Nx * Ny * Nz;
    PassGeom X{(int)Nx, (int)nx, Ny * Nz, (int)Ny, Nx, Nx * Ny, 1, nx, pyz, 1, 1, bNg, bnn};
    {
        Stage s_(pc, "fft_fwd_x");
        SIE_TRY(launch_pass<C>(st, (int)nx, src, buf, 0, X, NI * nb));
    }
    PassGeom Y{(int)Ny, (int)ny, nx * Nz, (int)nx, 1, pyz, nx, 1, pyz, nx, 0, bnn, bnn};
    {
        Stage s_(pc, "fft_fwd_y");
        SIE_TRY(launch_pass<C>(st, (int)ny, buf, buf, 0, Y, NI * nb));
    }
    {
        Stage s_(pc, "fft_z_specmul");
        SIE_TRY((launch_z<MODE, C, R>(st, (int)nz, buf, spec, (int)Nz, pyz, bnn, nb, k0)));
    }
    static_assert(MODE != ZM_SYS || NO == 4, "result grids lead the source grids");
    const int nout = NO == NI ? NO * nb : NO;  // the system product runs one at a time
    PassGeom Yi{(int)ny, (int)Ny, nx * Nz, (int)nx, 1, pyz, nx, 1, pyz, nx, 0, bnn, bnn};
    {
        Stage s_(pc, "fft_inv_y");
        SIE_TRY(launch_pass<C>(st, (int)ny, buf, buf, 1, Yi, nout));
    }
    PassGeom Xi{(int)nx, (int)Nx, Ny * Nz, (int)Ny, nx, pyz, 1, Nx, Nx * Ny, 1, 1, bnn, bNg};
    {
        Stage s_(pc, "fft_inv_x");
        SIE_TRY(launch_pass<C>(st, (int)nx, buf, src, 1, Xi, nout));
    }
    return SIE_OK;
}

bool fft_fused_z(const GridDesc& g) { return g.n[2] <= 256; }

sie_status fft_sys(cudaStream_t st, double2* buf, double2* src, const GridDesc& g, const double2* spec, double k0,
                   sie_ctx* pc)
{
    return fft_prod_t<ZM_SYS>(st, buf, src, g, spec, k0, pc, 1);
}

sie_status fft_sys(cudaStream_t st, float2* buf, float2* src, const GridDesc& g, const float2* spec, float k0,
                   sie_ctx* pc)
{
    return fft_prod_t<ZM_SYS>(st, buf, src, g, spec, k0, pc, 1);
}

sie_status fft_lk(cudaStream_t st, int which_LK, double2* buf, double2* src, const GridDesc& g, const double2* spec,
                  sie_ctx* pc, int nb)
{
    return which_LK == 0 ? fft_prod_t<ZM_L>(st, buf, src, g, spec, 0.0, pc, nb)
                         : fft_prod_t<ZM_K>(st, buf, src, g, spec, 0.0, pc, nb);
}

}  // namespace sie

// One-dimensional FFT passes of the AIM grid path (lengths up to 256 = R1 x R2,
// radices 4 to 16): kernels shared by the translation units that instantiate
// them per length (fft_*.cu; the dispatch is in fft.cu).
//
// A pencil is transformed in two register passes with one exchange through
// shared memory (Cooley-Tukey, n = R2 n1 + n2, k = k1 + R1 k2): thread tp takes the
// R1 inputs tp, tp + R2, ..., does an R1-point DFT, multiplies output k1 by
// exp(-+2 pi i tp k1 / n) and stores it; then threads take k1 and do the R2-point
// DFTs over n2.
//
// Arithmetic of the complex128 path: 64-bit block fixed point.  This part has 2
// FP64 lanes per SM and clock (an FFT in FP64 runs its pipe 82-85% busy and
// nothing else) but 60 64-bit integer additions and 13 32 x 32 -> 64-bit
// multiply-adds.  A pencil is loaded as complex128, scaled by a power of two such
// that the sum of all its components' magnitudes stays below 2^61 (no output and
// no partial sum can overflow then), transformed with exact additions and
// rotations by 62-bit constants, and stored as complex128 again.  The first pass
// runs with two more bits, rounded off in its twiddle products.  The
// error is relative to the pencil's norm, as that of an FP64 FFT is, and smaller:
// 0.5e-16 to 0.7e-16 at every length, most of it the rounding of the stored
// result, where FP64 butterflies give 1e-16 to 2e-16.  Results below the normal range
// are multiples of 2^-1074 (gradual underflow).  A pencil with a NaN or an infinity
// gives NaNs, as the sums of an FP64 transform do.
//
// The complex64 path uses the same passes in FP32.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "internal.h"
#include "limits.h"
#include "sysmul.cuh"

namespace sie {

#define SIE_HD __host__ __device__ __forceinline__

struct PassGeom {
    int n_in, n_out;       // elements read / written per pencil (zero padding / truncation)
    int64_t npencil;       // pencils
    int L;                 // pencil p -> lo = p % L, hi = p / L
    int64_t slo_in, shi_in, st_in;
    int64_t slo_out, shi_out, st_out;
    int contig;            // 1: elements of a pencil are contiguous (x pass)
    int64_t bs_in = 0, bs_out = 0;  // offsets between the grids of a batch (blockIdx.y)
};

// ------------------------------------------------------------------ fixed-point numbers
struct fx2 {
    long long x, y;
};
// a constant in [-2, 2) times 2^62 as hi 2^32 + lo, both halves signed
struct q62 {
    int lo, hi;
};
// from the integer round(v 2^62)
constexpr SIE_HD q62 to_q62(long long f)
{
    const int lo = (int)(unsigned)(unsigned long long)f;
    return q62{lo, (int)(f >> 32) + (lo < 0 ? 1 : 0)};
}
// round(f c): the product of the low halves, below one unit, is left out
SIE_HD long long mulq(long long f, q62 c)
{
    const int fl = (int)f;
    const int fh = (int)(f >> 32) + (int)((unsigned)fl >> 31);
    long long mid = (long long)fh * c.lo + (1LL << 29);
    mid += (long long)fl * c.hi;
    return ((long long)fh * c.hi << 2) + (mid >> 30);
}

// round(f c / 4): the shift to the high word comes for free
SIE_HD long long mulq_4(long long f, q62 c)
{
    const int fl = (int)f;
    const int fh = (int)(f >> 32) + (int)((unsigned)fl >> 31);
    long long mid = (long long)fh * c.lo + (1LL << 31);
    mid += (long long)fl * c.hi;
    return (long long)fh * c.hi + (int)(mid >> 32);
}

// twiddle exp(-2 pi i m / n): c, c + s and s - c of (c, s) = (cos, sin) (3-product rotation)
struct __align__(8) twq {
    q62 c, a, b;
};

// ------------------------------------------------------------------ number policies
// Fx: complex128 in memory, 64-bit fixed point in registers; F32: complex64
struct Fx {
    using G = double2;
    using V = fx2;
    using TW = twq;
    using R = double;
};
struct F32 {
    using G = float2;
    using V = float2;
    using TW = float2;
    using R = float;
};

template <class V>
SIE_HD V vadd(V a, V b)
{
    V t;
    t.x = a.x + b.x;
    t.y = a.y + b.y;
    return t;
}
template <class V>
SIE_HD V vsub(V a, V b)
{
    V t;
    t.x = a.x - b.x;
    t.y = a.y - b.y;
    return t;
}
// times -j (forward) or +j (inverse)
template <int INV, class V>
SIE_HD V vmj(V a)
{
    V t;
    t.x = INV ? -a.y : a.y;
    t.y = INV ? a.x : -a.x;
    return t;
}
// real constants: times 2^62 as an integer, and as a float
template <int ID>
struct RealC;
#define SIE_REALC(ID, Q, F)                \
    template <>                            \
    struct RealC<ID> {                     \
        static constexpr long long q = Q;  \
        static constexpr float f = F;      \
    };
enum { C_R8 = 0, C_S3, C_5A, C_5S1, C_5S2, C_HALF, C_Q };
SIE_REALC(C_R8, 3260954456333195553LL, 0.707106781187f)  // sqrt(1/2)
SIE_REALC(C_S3, 3993837246235628775LL, 0.866025403784f)  // sin 60
SIE_REALC(C_5A, 2578010857022246787LL, 0.559016994375f)  // sqrt(5)/4
SIE_REALC(C_5S1, 4385974038932618941LL, 0.951056516295f)  // sin 72
SIE_REALC(C_5S2, 2710681029835013083LL, 0.587785252292f)  // sin 36
SIE_REALC(C_HALF, 1LL << 61, 0.5f)
SIE_REALC(C_Q, 1LL << 60, 0.25f)
#undef SIE_REALC

template <int ID>
SIE_HD fx2 vscale(fx2 a)
{
    if constexpr (ID == C_HALF) return fx2{(a.x + 1) >> 1, (a.y + 1) >> 1};
    if constexpr (ID == C_Q) return fx2{(a.x + 2) >> 2, (a.y + 2) >> 2};
    constexpr q62 c = to_q62(RealC<ID>::q);
    return fx2{mulq(a.x, c), mulq(a.y, c)};
}
template <int ID>
SIE_HD float2 vscale(float2 a)
{
    constexpr float c = RealC<ID>::f;
    float2 t;
    t.x = a.x * c;
    t.y = a.y * c;
    return t;
}

// rotation by the twiddle (c - j s forward, conjugate for the inverse); DOWN: and divided by 4
template <int INV, bool DOWN = false>
SIE_HD fx2 vrot(fx2 z, twq w)
{
    // forward: re = c x + s y, im = c y - s x.  t = c (x + y):
    //   re = t + (s - c) y, im = t - (c + s) x;  inverse: re = t - (c + s) y, im = t + (s - c) x
    auto mul = [](long long f, q62 c) { return DOWN ? mulq_4(f, c) : mulq(f, c); };
    const long long t = mul(z.x + z.y, w.c);
    fx2 o;
    if (INV) {
        o.x = t - mul(z.y, w.a);
        o.y = t + mul(z.x, w.b);
    } else {
        o.x = t + mul(z.y, w.b);
        o.y = t - mul(z.x, w.a);
    }
    return o;
}
template <int INV>
SIE_HD float2 vrot(float2 z, float2 w)  // w = (cos, sin)
{
    float2 o;
    if (INV) {
        o.x = z.x * w.x - z.y * w.y;
        o.y = z.y * w.x + z.x * w.y;
    } else {
        o.x = z.x * w.x + z.y * w.y;
        o.y = z.y * w.x - z.x * w.y;
    }
    return o;
}
// exp(-+2 pi i m / 16), m = 1, 2, 3, 6 or 9
template <class V>
struct W16;
template <>
struct W16<fx2> {
    template <int INV, int M>
    static SIE_HD fx2 rot(fx2 z)
    {
        // round(2^62 cos), (cos + sin), (sin - cos) of 2 pi M / 16; M = 9 is M = 1 negated
        constexpr long long c1 = 4260642322793532497LL, a1 = 6025458157315419939LL, b1 = -2495826488271645056LL;
        constexpr long long c3 = 1764815834521887442LL, a3 = 6025458157315419939LL, b3 = 2495826488271645056LL;
        constexpr twq w{to_q62(M == 1 ? c1 : (M == 3 ? c3 : -c1)), to_q62(M == 1 ? a1 : (M == 3 ? a3 : -a1)),
                        to_q62(M == 1 ? b1 : (M == 3 ? b3 : -b1))};
        return vrot<INV>(z, w);
    }
};
template <>
struct W16<float2> {
    template <int INV, int M>
    static SIE_HD float2 rot(float2 z)
    {
        constexpr float C1 = 0.92387953251128675613f, S1 = 0.38268343236508977173f;
        float2 w;
        w.x = M == 1 ? C1 : (M == 3 ? S1 : -C1);
        w.y = M == 1 ? S1 : (M == 3 ? C1 : -S1);
        return vrot<INV>(z, w);
    }
};
// times exp(-+2 pi i / 8): (1 -+ j) / sqrt 2
template <int INV, class V>
SIE_HD V vw8(V a)
{
    V t;
    t.x = INV ? a.x - a.y : a.x + a.y;
    t.y = INV ? a.y + a.x : a.y - a.x;
    return vscale<C_R8>(t);
}

// ------------------------------------------------------------------ small DFTs (in place, natural order)
template <int INV, class V>
SIE_HD void dft2(V& a, V& b)
{
    const V t = a;
    a = vadd(t, b);
    b = vsub(t, b);
}
template <int INV, class V>
SIE_HD void dft4(V& a0, V& a1, V& a2, V& a3)
{
    const V s = vadd(a0, a2), d = vsub(a0, a2), p = vadd(a1, a3), q = vmj<INV>(vsub(a1, a3));
    a0 = vadd(s, p);
    a1 = vadd(d, q);
    a2 = vsub(s, p);
    a3 = vsub(d, q);
}
template <int INV, class V>
SIE_HD void dft3(V& a0, V& a1, V& a2)
{
    const V t = vadd(a1, a2), u = vmj<INV>(vscale<C_S3>(vsub(a1, a2)));
    const V m = vsub(a0, vscale<C_HALF>(t));
    a0 = vadd(a0, t);
    a1 = vadd(m, u);
    a2 = vsub(m, u);
}
template <int INV, class V>
SIE_HD void dft5(V& a0, V& a1, V& a2, V& a3, V& a4)
{
    const V t1 = vadd(a1, a4), t2 = vadd(a2, a3), t3 = vsub(a1, a4), t4 = vsub(a2, a3);
    const V t5 = vadd(t1, t2), m1 = vsub(a0, vscale<C_Q>(t5)), m2 = vscale<C_5A>(vsub(t1, t2));
    const V s1 = vadd(m1, m2), s2 = vsub(m1, m2);
    const V u1 = vmj<INV>(vadd(vscale<C_5S1>(t3), vscale<C_5S2>(t4)));
    const V u2 = vmj<INV>(vsub(vscale<C_5S2>(t3), vscale<C_5S1>(t4)));
    a0 = vadd(a0, t5);
    a1 = vadd(s1, u1);
    a4 = vsub(s1, u1);
    a2 = vadd(s2, u2);
    a3 = vsub(s2, u2);
}
template <int INV, class V>
SIE_HD void dft8(V* a)
{
    dft4<INV>(a[0], a[2], a[4], a[6]);
    dft4<INV>(a[1], a[3], a[5], a[7]);
    const V e0 = a[0], e1 = a[2], e2 = a[4], e3 = a[6];
    const V o0 = a[1], o1 = vw8<INV>(a[3]), o2 = vmj<INV>(a[5]), o3 = vmj<INV>(vw8<INV>(a[7]));
    a[0] = vadd(e0, o0);
    a[4] = vsub(e0, o0);
    a[1] = vadd(e1, o1);
    a[5] = vsub(e1, o1);
    a[2] = vadd(e2, o2);
    a[6] = vsub(e2, o2);
    a[3] = vadd(e3, o3);
    a[7] = vsub(e3, o3);
}
template <int INV, class V>
SIE_HD void dft16(V* a)
{
    // a[4 n1 + n2] -> k = k1 + 4 k2
#pragma unroll
    for (int n2 = 0; n2 < 4; n2++) dft4<INV>(a[n2], a[4 + n2], a[8 + n2], a[12 + n2]);
    a[5] = W16<V>::template rot<INV, 1>(a[5]);
    a[6] = vw8<INV>(a[6]);
    a[7] = W16<V>::template rot<INV, 3>(a[7]);
    a[9] = vw8<INV>(a[9]);
    a[10] = vmj<INV>(a[10]);
    a[11] = vmj<INV>(vw8<INV>(a[11]));
    a[13] = W16<V>::template rot<INV, 3>(a[13]);
    a[14] = vmj<INV>(vw8<INV>(a[14]));
    a[15] = W16<V>::template rot<INV, 9>(a[15]);
#pragma unroll
    for (int k1 = 0; k1 < 4; k1++) dft4<INV>(a[4 * k1], a[4 * k1 + 1], a[4 * k1 + 2], a[4 * k1 + 3]);
    // a[4 k1 + k2] holds X[k1 + 4 k2]
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = i + 1; j < 4; j++) {
            const V t = a[4 * i + j];
            a[4 * i + j] = a[4 * j + i];
            a[4 * j + i] = t;
        }
}
// prime-factor DFTs of N1 x N2 (coprime): n = N2 n1 + N1 n2, k = k1 mod N1, k2 mod N2: no twiddles
template <int INV, int N1, int N2, class V>
SIE_HD void dft_pf(V* a)
{
    constexpr int N = N1 * N2;
    V b[N];
#pragma unroll
    for (int i = 0; i < N; i++) b[i] = a[i];
#pragma unroll
    for (int n2 = 0; n2 < N2; n2++) {
        auto at = [&](int n1) -> V& { return b[(N2 * n1 + N1 * n2) % N]; };
        if constexpr (N1 == 2)
            dft2<INV>(at(0), at(1));
        else
            dft3<INV>(at(0), at(1), at(2));
    }
#pragma unroll
    for (int k1 = 0; k1 < N1; k1++) {
        auto at = [&](int n2) -> V& { return b[(N2 * k1 + N1 * n2) % N]; };
        if constexpr (N2 == 3)
            dft3<INV>(at(0), at(1), at(2));
        else if constexpr (N2 == 4)
            dft4<INV>(at(0), at(1), at(2), at(3));
        else
            dft5<INV>(at(0), at(1), at(2), at(3), at(4));
    }
#pragma unroll
    for (int k1 = 0; k1 < N1; k1++)
#pragma unroll
        for (int k2 = 0; k2 < N2; k2++) {
            int k = 0;  // k = k1 mod N1, k = k2 mod N2
            for (int c = 0; c < N; c++)
                if (c % N1 == k1 && c % N2 == k2) k = c;
            a[k] = b[(N2 * k1 + N1 * k2) % N];
        }
}
template <int INV, int R, class V>
SIE_HD void dftR(V* a)
{
    if constexpr (R == 4)
        dft4<INV>(a[0], a[1], a[2], a[3]);
    else if constexpr (R == 5)
        dft5<INV>(a[0], a[1], a[2], a[3], a[4]);
    else if constexpr (R == 6)
        dft_pf<INV, 2, 3>(a);
    else if constexpr (R == 8)
        dft8<INV>(a);
    else if constexpr (R == 10)
        dft_pf<INV, 2, 5>(a);
    else if constexpr (R == 12)
        dft_pf<INV, 3, 4>(a);
    else
        dft16<INV>(a);
}

// ------------------------------------------------------------------ complex128 <-> fixed point
// Scales of a pencil: field, the largest high word of its components' magnitudes (1 for
// one that has only low bits; 0: all zero), emax, its exponent field, and
// l1 = sum over the components of floor(|v| 2^(20 - E)) + 1, E = emax's exponent.
// After scaling by 2^(bits - 1 - E) the components are below 2^bits and their sum
// is below 2^61; the first pass takes 4 times that (its sums of R1 terms fit too).
struct FxScale {
    int s0, x0;
    bool bad, low;  // not finite; results may lie below the normal range
};
SIE_HD int fx_l1(unsigned hi, int emax)
{
    const int e = (int)(hi >> 20) & 0x7ff, d = emax - (e ? e : 1);
    return (int)(((hi & 0xfffffu) | 0x100000u) >> (d > 31 ? 31 : d)) + 1;
}
SIE_HD FxScale fx_scale(int field, int l1, int log2_r1)
{
    const int emax = (field >> 20) > 1 ? field >> 20 : 1;
#ifdef __CUDA_ARCH__
    const int lg = max(21, 32 - __clz(l1));  // l1 < 2^lg
#else
    int lg = 21;
    while (l1 >> lg) lg++;
#endif
    // first pass: R1 terms of its bits, or the whole sum, whichever bound is lower
    const int top = 59 - log2_r1 > 80 - lg ? 59 - log2_r1 : 80 - lg, b = 82 - lg < top ? 82 - lg : top;
    return FxScale{emax + 63 - (b + 2), emax - b, emax == 0x7ff, emax < b && field > 0};
}
// v 2^(bits - 1 - E) as an integer, the fraction below 2^(E - bits + 1) cut off;
// s0 = emax + 63 - bits
SIE_HD long long fx_from(unsigned hi, unsigned lo, int s0)
{
    const int e = (int)(hi >> 20) & 0x7ff;
    const unsigned mh = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
    const unsigned long long m = ((((unsigned long long)mh) << 32) | lo) << 10;  // bit 62 set
    int s = s0 - (e ? e : 1);
    s = s > 63 ? 63 : s;
    const long long f = (long long)(m >> s), sg = (long long)(int)hi >> 63;  // sg 0 or -1
    return (f ^ sg) - sg;
}
// bits of a double and back
SIE_HD unsigned long long fx_bits(double d)
{
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(d);
#else
    unsigned long long r;
    memcpy(&r, &d, 8);
    return r;
#endif
}
SIE_HD double fx_double(unsigned long long r)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)r);
#else
    double d;
    memcpy(&d, &r, 8);
    return d;
#endif
}
// f 2^(E - bits + 1) as a double; x0 = emax - bits >= 0 or f = 0: no result is below the
// normal range then (f is a whole number).  Conversion on the FP64 pipe, which the
// transforms leave idle, then the exponent by an integer addition.
SIE_HD double fx_to(long long f, int x0)
{
#ifdef __CUDA_ARCH__
    const double d = __ll2double_rn(f);
    const int hi = __double2hiint(d), e = ((hi >> 20) & 0x7ff) + (x0 - 1022);  // biased exponent of the result
    int oh = hi + ((x0 - 1022) << 20), ol = __double2loint(d);
    if (f == 0) oh = 0;
    if (e >= 2047) oh = (hi & 0x80000000) | 0x7ff00000, ol = 0;
    return __hiloint2double(oh, ol);
#else
    return ldexp((double)f, x0 - 1022);
#endif
}

// the same by integer operations alone, where the FP64 pipe is busy
SIE_HD double fx_to_int(long long f, int x0)
{
    const long long sg = f >> 63;
    const unsigned long long a = (unsigned long long)((f ^ sg) - sg);
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)a);
#else
    const int lz = a ? __builtin_clzll(a) : 64;
#endif
    const int e = 63 + x0 - lz;  // biased exponent less one
    unsigned long long r = ((a << (lz - 1)) + 0x200) >> 10;  // |f| < 2^62: lz >= 2; bit 52 set (a carry moves up)
    r += (unsigned long long)(unsigned)e << 52;
    if (a == 0) r = 0;
    if (a != 0 && e >= 2046) r = 0x7ff0000000000000ull;
    return fx_double(r | ((unsigned long long)sg & 0x8000000000000000ull));
}

// the same for x0 < 0 (pencils below 2^-960 or so): results below the normal range are
// multiples of 2^-1074
SIE_HD double fx_to_low(long long f, int x0) { return fx_to_int(f, x0 + 64) * 0x1p-64; }

// ------------------------------------------------------------------ plans
template <int N>
struct Plan;
#define SIE_PLAN(N_, A, B)                   \
    template <>                              \
    struct Plan<N_> {                        \
        static constexpr int R1 = A, R2 = B; \
    };
// R1 first (its R2 butterflies are one per thread), R2 second
SIE_PLAN(16, 4, 4)
SIE_PLAN(20, 4, 5)
SIE_PLAN(24, 4, 6)
SIE_PLAN(32, 8, 4)
SIE_PLAN(40, 8, 5)
SIE_PLAN(48, 12, 4)
SIE_PLAN(64, 8, 8)
SIE_PLAN(80, 16, 5)
SIE_PLAN(96, 16, 6)
SIE_PLAN(128, 16, 8)
SIE_PLAN(160, 16, 10)
SIE_PLAN(192, 16, 12)
SIE_PLAN(256, 16, 16)
#undef SIE_PLAN

__host__ __device__ constexpr int pow2_floor(int v) { return v <= 1 ? 1 : 2 * pow2_floor(v / 2); }

// shared-memory layout of a pencil: element (n2, k1) at n2 (R1 + 1) + k1; pencils
// PITCH apart, chosen so that 8 consecutive 16-byte accesses of a quarter warp
// (pencil fastest) fall into different banks
template <int N>
__host__ __device__ constexpr int fft_pitch(int pb)
{
    const int base = Plan<N>::R2 * (Plan<N>::R1 + 1), want = pb >= 8 ? 1 : 8 / pb;
    int p = base;
    while (p % 8 != want % 8) p++;
    return p;
}

#ifdef __CUDACC__
// ------------------------------------------------------------------ pencil pieces
// a thread's R1 inputs of the first pass (element tp + r R2), zero beyond n_in
template <int R1, int R2, class G>
__device__ __forceinline__ void load_first(const G* __restrict__ in, int64_t base, int64_t st, int tp, int n_in, bool ok,
                                           G* g)
{
#pragma unroll
    for (int r = 0; r < R1; r++) {
        const int j = tp + r * R2;
        G v;
        v.x = 0;
        v.y = 0;
        if (ok && j < n_in) v = in[base + (int64_t)j * st];
        g[r] = v;
    }
}

__device__ __forceinline__ int high_max(double2 v)
{
    return max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff);
}

// first pass of a pencil: inputs g -> DFT -> twiddle -> shared memory
template <int INV, int R1, int R2, class P>
__device__ __forceinline__ void first_pass(const typename P::G* g, int tp, int n_in, const FxScale& q,
                                           const typename P::TW* __restrict__ tw, typename P::V* s)
{
    typename P::V a[R1];
#pragma unroll
    for (int r = 0; r < R1; r++) {
        if constexpr (sizeof(typename P::G) == 16) {
            a[r].x = a[r].y = 0;
            if (r * R2 < n_in) {  // uniform: the zero half of a padded pencil is skipped
                a[r].x = fx_from(__double2hiint(g[r].x), __double2loint(g[r].x), q.s0);
                a[r].y = fx_from(__double2hiint(g[r].y), __double2loint(g[r].y), q.s0);
            }
        } else {
            a[r] = g[r];
        }
    }
    dftR<INV, R1>(a);
    typename P::V* o = s + tp * (R1 + 1);
    if constexpr (sizeof(typename P::G) == 16) {
        o[0] = vscale<C_Q>(a[0]);
#pragma unroll
        for (int r = 1; r < R1; r++) o[r] = vrot<INV, true>(a[r], tw[tp * r]);
    } else {
        o[0] = a[0];
#pragma unroll
        for (int r = 1; r < R1; r++) o[r] = vrot<INV>(a[r], tw[tp * r]);
    }
}

// second-pass butterfly k1: R2 values over n2 -> X[k1 + R1 k2] in a[k2]
template <int INV, int R1, int R2, class P>
__device__ __forceinline__ void second_pass(const typename P::V* s, int k1, typename P::V* a)
{
#pragma unroll
    for (int r = 0; r < R2; r++) a[r] = s[r * (R1 + 1) + k1];
    dftR<INV, R2>(a);
}

// scale of a pencil from its threads' inputs (n_in live): em and l1 are its
// shared slots, zero before; two barriers
template <int R1, int R2>
__device__ __forceinline__ FxScale pencil_scale(const double2* g, int n_in, int* em, int* l1, bool act)
{
    int m = 0, lo = 0;
#pragma unroll
    for (int r = 0; r < R1; r++) {
        m = max(m, high_max(g[r]));
        lo |= __double2loint(g[r].x) | __double2loint(g[r].y);
    }
    if (m == 0 && lo != 0) m = 1;
    if (act) atomicMax(em, m);
    __syncthreads();
    const int field = *em, emax = max(field >> 20, 1);
    int t = 0;
#pragma unroll
    for (int r = 0; r < R1; r++)
        if (r * R2 < n_in) t += fx_l1(__double2hiint(g[r].x), emax) + fx_l1(__double2hiint(g[r].y), emax);
    if (act) atomicAdd(l1, t);
    __syncthreads();
    constexpr int lg = R1 > 8 ? 4 : (R1 > 4 ? 3 : 2);
    return fx_scale(field, *l1, lg);
}
// put(r, v) of the N outputs of a butterfly, v() the result r (converted only where it is
// stored); its own slots in shared memory are s[r st].  Pencils that are not finite or so
// small that results may lie below the normal range take a branch of their own, a short
// loop over the slots: with the tests on every value the system product at 128^3 took
// 617 us (not finite) and 638 us (both), 604 us this way.  A pencil of zeros, of which
// forward passes have many, needs neither.
template <int N, bool FP64PIPE, class F>
__device__ __forceinline__ void fx_results(const fx2* a, const FxScale& q, fx2* s, int st, F put)
{
    if (!q.bad && !q.low) {
#pragma unroll
        for (int r = 0; r < N; r++)
            put(r, [&] {
                return FP64PIPE ? make_double2(fx_to(a[r].x, q.x0), fx_to(a[r].y, q.x0))
                                : make_double2(fx_to_int(a[r].x, q.x0), fx_to_int(a[r].y, q.x0));
            });
    } else {
#pragma unroll
        for (int r = 0; r < N; r++) s[r * st] = a[r];
#pragma unroll 1
        for (int r = 0; r < N; r++) {
            put(r, [&] {
                const fx2 v = s[r * st];
                const double nan = __longlong_as_double(0x7ff8000000000000ll);
                return q.bad ? make_double2(nan, nan) : make_double2(fx_to_low(v.x, q.x0), fx_to_low(v.y, q.x0));
            });
        }
    }
}

// ------------------------------------------------------------------ one pass over many pencils
// PB pencils per CTA, R2 threads per pencil; in and out may alias (a pencil is
// read completely before any of it is written).  128 points, 7 grids of 8,064
// pencils (the y pass of the system product at 63^3): FP64 Stockham radix 8 took
// 292 us at 82% of the FP64 pipe; 69 us now, the integer (ALU) pipe 61% busy, and
// 20 us in complex64 (47 us before).
template <int N>
__host__ __device__ constexpr int pass_pb()
{
    return pow2_floor(128 / Plan<N>::R2);
}

template <int N, class P, int INV>
__global__ void __launch_bounds__(pass_pb<N>() * Plan<N>::R2)
    k_fft(const typename P::G* in, typename P::G* out, const typename P::TW* __restrict__ tw, PassGeom G)
{
    constexpr int R1 = Plan<N>::R1, R2 = Plan<N>::R2, PB = pass_pb<N>(), PITCH = fft_pitch<N>(PB);
    constexpr bool FX = sizeof(typename P::G) == 16;
    extern __shared__ __align__(16) unsigned char smraw[];
    typename P::V* sm = reinterpret_cast<typename P::V*>(smraw);
    __shared__ int em[PB], l1[PB];
    int pl, tp;  // pencil-fastest thread order on strided passes keeps rows coalesced
    if (G.contig) {
        pl = threadIdx.x / R2;
        tp = threadIdx.x % R2;
    } else {
        pl = threadIdx.x % PB;
        tp = threadIdx.x / PB;
    }
    const int64_t p = (int64_t)blockIdx.x * PB + pl;
    const bool ok = p < G.npencil;
    const int64_t lo = ok ? p % G.L : 0, hi = ok ? p / G.L : 0;
    typename P::G g[R1];
    load_first<R1, R2>(in, lo * G.slo_in + hi * G.shi_in + blockIdx.y * G.bs_in, G.st_in, tp, G.n_in, ok, g);
    FxScale q{0, 0, false, false};
    if constexpr (FX) {
        for (int i = threadIdx.x; i < PB; i += blockDim.x) em[i] = l1[i] = 0;
        __syncthreads();
        q = pencil_scale<R1, R2>(g, G.n_in, em + pl, l1 + pl, true);
    }
    typename P::V* s = sm + pl * PITCH;
    first_pass<INV, R1, R2, P>(g, tp, G.n_in, q, tw, s);
    __syncthreads();
    const int64_t ob = lo * G.slo_out + hi * G.shi_out + blockIdx.y * G.bs_out;
    for (int k1 = tp; k1 < R1; k1 += R2) {
        typename P::V a[R2];
        second_pass<INV, R1, R2, P>(s, k1, a);
        auto put = [&](int r, auto v) {
            const int k = k1 + r * R1;
            if (ok && k < G.n_out) out[ob + (int64_t)k * G.st_out] = v();
        };
        if constexpr (FX) {
            fx_results<R2, true>(a, q, s + k1, R1 + 1, put);
        } else {
#pragma unroll
            for (int r = 0; r < R2; r++) put(r, [&] { return a[r]; });
        }
    }
}

// ------------------------------------------------------------------ fused z stage
// Forward z transforms of a product's source grids, its spectral products and
// the inverse z transforms of its result grids, PB (x, y) columns per CTA: the z
// spectra of a column stay in shared memory.  Reads z < nz_phys of the NI source
// grids, writes z < nz_phys of grids 0 .. NO - 1 in place (the inverse y pass
// reads nothing else).  Threads: grid, then column fastest.
// System product at 128^3, 16,384 columns: FP64 transforms took 1,091 us, the FP64
// pipe 85% busy; 347 us now, FP64 46% and ALU 42% busy.  Its spectral products alone keep
// the FP64 pipe busy for 140 us, so the forward outputs are converted by integer
// operations; the rest is integer issue and the barriers between phases (two to four
// CTAs an SM).  In complex64: 158 us before, 70 us now.
enum { ZM_SYS = 0, ZM_L = 1, ZM_K = 2 };
template <int MODE>
struct ZMode {
    static constexpr int NI = MODE == ZM_SYS ? 7 : (MODE == ZM_L ? 4 : 3);
    static constexpr int NO = MODE == ZM_SYS ? 4 : NI;
};

template <int N, class P, int MODE>
__host__ __device__ constexpr int z_pb()
{
    // complex128: about 128 threads (four small CTAs an SM, whose phases overlap; 8 x
    // 1,280 triangles at n = 64: 155 us against 177 us with 256), from n = 128 on 256
    // (two CTAs, rows of 64 bytes; system product at 128^3: 351 us against 377 us).
    // complex64, whose rows are half as long: 512.
    return pow2_floor((sizeof(typename P::G) == 16 ? (N >= 128 ? 256 : 128) : 512) / (ZMode<MODE>::NI * Plan<N>::R2));
}

template <int MODE, class C, class R>
__device__ __forceinline__ void z_product(const C* __restrict__ spec, int64_t i, int64_t bnn, R k0, const C* in, C* out)
{
    if constexpr (MODE == ZM_SYS) {
        sys_specmul(spec[i], spec[bnn + i], spec[2 * bnn + i], spec[3 * bnn + i], k0, in, out);
    } else if constexpr (MODE == ZM_L) {
        const C Gk = spec[i];
#pragma unroll
        for (int g = 0; g < 4; g++) out[g] = sm_mul(Gk, in[g]);
    } else {
        const C gx = spec[bnn + i], gy = spec[2 * bnn + i], gz = spec[3 * bnn + i];
        C z;
        z.x = z.y = 0;
        out[0] = sm_fms(gz, in[1], sm_fma(gy, in[2], z));
        out[1] = sm_fms(gx, in[2], sm_fma(gz, in[0], z));
        out[2] = sm_fms(gy, in[0], sm_fma(gx, in[1], z));
    }
}

// CTAs per SM the register count must allow: 16 warps at 128 registers (complex128), 28 at 72
template <int N, class P, int MODE>
__host__ __device__ constexpr int z_ctas()
{
    const int warps = (ZMode<MODE>::NI * z_pb<N, P, MODE>() * Plan<N>::R2 + 31) / 32;
    const int n = (sizeof(typename P::G) == 16 ? 16 : 28) / warps;
    return n < 1 ? 1 : n;
}

template <int N, class P, int MODE>
__global__ void __launch_bounds__(ZMode<MODE>::NI* z_pb<N, P, MODE>() * Plan<N>::R2, z_ctas<N, P, MODE>())
    k_fft_z(typename P::G* __restrict__ buf, const typename P::G* __restrict__ spec,
            const typename P::TW* __restrict__ tw, int nz_phys, int64_t ncol, int64_t plane, int64_t bnn,
            int64_t batch, typename P::R k0)
{
    using C = typename P::G;
    using V = typename P::V;
    constexpr int R1 = Plan<N>::R1, R2 = Plan<N>::R2, PB = z_pb<N, P, MODE>(), PITCH = fft_pitch<N>(PB);
    constexpr int NI = ZMode<MODE>::NI, NO = ZMode<MODE>::NO, NT = NI * PB * R2;
    constexpr bool FX = sizeof(C) == 16;
    extern __shared__ __align__(16) unsigned char smraw[];
    V* sm = reinterpret_cast<V*>(smraw);
    C* smc = reinterpret_cast<C*>(smraw);
    __shared__ int em[2][NI * PB], l1[2][NI * PB];
    const int gi = threadIdx.x / (PB * R2), rr = threadIdx.x % (PB * R2), pl = rr % PB, tp = rr / PB;
    const int me = gi * PB + pl;
    const int64_t col = (int64_t)blockIdx.x * PB + pl;
    const bool ok = col < ncol;
    buf += blockIdx.y * batch;
    const int64_t gb = gi * bnn + (ok ? col : 0);
    // the kernel spectra of this CTA's columns on their way to L2 while it transforms
    for (int kz = threadIdx.x; kz < N; kz += NT) {
        const C* q0 = spec + (int64_t)kz * plane + (int64_t)blockIdx.x * PB;
        if constexpr (MODE != ZM_K) asm volatile("prefetch.global.L2 [%0];" ::"l"(q0));
        if constexpr (MODE != ZM_L) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(q0 + bnn));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(q0 + 2 * bnn));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(q0 + 3 * bnn));
        }
    }
    FxScale q{0, 0, false, false};
    V* s = sm + me * PITCH;
    C* sc = smc + me * PITCH;
    {
        C g[R1];
        load_first<R1, R2>((const C*)buf, gb, plane, tp, nz_phys, ok, g);
        if constexpr (FX) {
            for (int i = threadIdx.x; i < NI * PB; i += NT) em[0][i] = em[1][i] = l1[0][i] = l1[1][i] = 0;
            __syncthreads();
            q = pencil_scale<R1, R2>(g, nz_phys, &em[0][me], &l1[0][me], true);
        }
        first_pass<0, R1, R2, P>(g, tp, nz_phys, q, tw, s);
    }
    __syncthreads();
    // second pass in place: butterfly k1 reads and writes the slots n2 (R1 + 1) + k1
#pragma unroll 1
    for (int k1 = tp; k1 < R1; k1 += R2) {
        V a[R2];
        second_pass<0, R1, R2, P>(s, k1, a);
        auto put = [&](int r, auto v) { sc[r * (R1 + 1) + k1] = v(); };
        if constexpr (FX) {
            fx_results<R2, false>(a, q, s + k1, R1 + 1, put);
        } else {
#pragma unroll
            for (int r = 0; r < R2; r++) put(r, [&] { return a[r]; });
        }
    }
    __syncthreads();
    // spectral products in place: k = k1 + R1 k2 sits at k2 (R1 + 1) + k1
#pragma unroll 1
    for (int idx = threadIdx.x; idx < PB * N; idx += NT) {
        const int p2 = idx % PB, kz = idx / PB, at = p2 * PITCH + (kz / R1) * (R1 + 1) + kz % R1;
        const int64_t c2 = (int64_t)blockIdx.x * PB + p2;
        if (c2 >= ncol) continue;
        C in[NI], out[NO];
#pragma unroll
        for (int g = 0; g < NI; g++) in[g] = smc[g * PB * PITCH + at];
        z_product<MODE>(spec, (int64_t)kz * plane + c2, bnn, k0, in, out);
#pragma unroll
        for (int g = 0; g < NO; g++) smc[g * PB * PITCH + at] = out[g];
    }
    __syncthreads();
    const bool act = NO == NI || gi < NO;
    {
        C g[R1];
#pragma unroll
        for (int r = 0; r < R1; r++) {
            const int j = tp + r * R2;
            g[r] = sc[(j / R1) * (R1 + 1) + j % R1];
        }
        if constexpr (FX)
            q = pencil_scale<R1, R2>(g, N, &em[1][me], &l1[1][me], act);
        else
            __syncthreads();
        // an opaque copy: the compiler would keep all twiddles of the forward pass in registers
        asm volatile("" : "+l"(tw));
        if (act) first_pass<1, R1, R2, P>(g, tp, N, q, tw, s);
    }
    __syncthreads();
    if (!act || !ok) return;
#pragma unroll 1
    for (int k1 = tp; k1 < R1; k1 += R2) {
        V a[R2];
        second_pass<1, R1, R2, P>(s, k1, a);
        auto put = [&](int r, auto v) {
            const int k = k1 + r * R1;
            if (k < nz_phys) buf[gb + (int64_t)k * plane] = v();
        };
        if constexpr (FX) {
            fx_results<R2, true>(a, q, s + k1, R1 + 1, put);
        } else {
#pragma unroll
            for (int r = 0; r < R2; r++) put(r, [&] { return a[r]; });
        }
    }
}

// ------------------------------------------------------------------ launches
template <int N, class P>
sie_status fft_pass_n(cudaStream_t st, const typename P::G* in, typename P::G* out, int inv, const PassGeom& G, int nb,
                      const typename P::TW* tw)
{
    constexpr int PB = pass_pb<N>();
    constexpr size_t smem = sizeof(typename P::V) * PB * fft_pitch<N>(PB);
    static_assert(smem <= 48 * 1024, "static shared-memory limit");
    const dim3 grid((unsigned)((G.npencil + PB - 1) / PB), nb);
    if (inv)
        k_fft<N, P, 1><<<grid, PB * Plan<N>::R2, smem, st>>>(in, out, tw, G);
    else
        k_fft<N, P, 0><<<grid, PB * Plan<N>::R2, smem, st>>>(in, out, tw, G);
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}

template <int N, class P, int MODE>
sie_status fft_z_n(cudaStream_t st, typename P::G* buf, const typename P::G* spec, int nz_phys, int64_t ncol,
                   int64_t plane, int64_t bnn, int64_t batch, int nb, typename P::R k0, const typename P::TW* tw)
{
    constexpr int PB = z_pb<N, P, MODE>();
    constexpr size_t smem = sizeof(typename P::V) * ZMode<MODE>::NI * PB * fft_pitch<N>(PB);
    SIE_CUDA_TRY(kernel_limit((const void*)k_fft_z<N, P, MODE>, smem));
    const dim3 grid((unsigned)((ncol + PB - 1) / PB), nb);
    k_fft_z<N, P, MODE>
        <<<grid, ZMode<MODE>::NI * PB * Plan<N>::R2, smem, st>>>(buf, spec, tw, nz_phys, ncol, plane, bnn, batch, k0);
    SIE_CUDA_TRY(cudaGetLastError());
    return SIE_OK;
}
#endif

// instantiated for each length in fft_*.cu
template <int N, class P>
sie_status fft_pass_n(cudaStream_t st, const typename P::G* in, typename P::G* out, int inv, const PassGeom& G, int nb,
                      const typename P::TW* tw);
template <int N, class P, int MODE>
sie_status fft_z_n(cudaStream_t st, typename P::G* buf, const typename P::G* spec, int nz_phys, int64_t ncol,
                   int64_t plane, int64_t bnn, int64_t batch, int nb, typename P::R k0, const typename P::TW* tw);

#define SIE_FFT_INSTANCES(N, PRE)                                                                                     \
    PRE template sie_status fft_pass_n<N, Fx>(cudaStream_t, const double2*, double2*, int, const PassGeom&, int,      \
                                              const twq*);                                                            \
    PRE template sie_status fft_pass_n<N, F32>(cudaStream_t, const float2*, float2*, int, const PassGeom&, int,       \
                                               const float2*);                                                        \
    PRE template sie_status fft_z_n<N, Fx, ZM_SYS>(cudaStream_t, double2*, const double2*, int, int64_t, int64_t,     \
                                                   int64_t, int64_t, int, double, const twq*);                        \
    PRE template sie_status fft_z_n<N, Fx, ZM_L>(cudaStream_t, double2*, const double2*, int, int64_t, int64_t,       \
                                                 int64_t, int64_t, int, double, const twq*);                          \
    PRE template sie_status fft_z_n<N, Fx, ZM_K>(cudaStream_t, double2*, const double2*, int, int64_t, int64_t,       \
                                                 int64_t, int64_t, int, double, const twq*);                          \
    PRE template sie_status fft_z_n<N, F32, ZM_SYS>(cudaStream_t, float2*, const float2*, int, int64_t, int64_t,      \
                                                    int64_t, int64_t, int, float, const float2*);

// the lengths up to 256
#define SIE_FFT_LENGTHS(X) \
    X(16) X(20) X(24) X(32) X(40) X(48) X(64) X(80) X(96) X(128) X(160) X(192) X(256)
#define SIE_FFT_EXTERN(N) SIE_FFT_INSTANCES(N, extern)

}  // namespace sie

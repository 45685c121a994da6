// Spectral products of the system operator of Eq. (sys) at one frequency
// node: from the seven source spectra (J_x, J_y, J_z, M_x, M_y, M_z, rho) and
// the kernel spectra (G, dG/dx, dG/dy, dG/dz) to the four result spectra
//   A_a = j k0 G J_a - (grad G x M)_a   (a = x, y, z),   Phi = G rho,
// the grid form of the L_A and K terms of Eq. (AIM_Lin) and of the charge
// potential.  C = double2 (FP64) or float2 (complex64 grid path), R its real type.
// Every complex product is accumulated by four FMAs (42 operations a node).
#pragma once
#include <cuda_runtime.h>

namespace sie {

template <class C>
__device__ __forceinline__ C sm_mul(C a, C b)
{
    C t;
    t.x = a.x * b.x - a.y * b.y;
    t.y = a.x * b.y + a.y * b.x;
    return t;
}

__device__ __forceinline__ double sm_f(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float sm_f(float a, float b, float c) { return fmaf(a, b, c); }

// c + a b and c - a b
template <class C>
__device__ __forceinline__ C sm_fma(C a, C b, C c)
{
    c.x = sm_f(a.x, b.x, sm_f(-a.y, b.y, c.x));
    c.y = sm_f(a.x, b.y, sm_f(a.y, b.x, c.y));
    return c;
}
template <class C>
__device__ __forceinline__ C sm_fms(C a, C b, C c)
{
    c.x = sm_f(-a.x, b.x, sm_f(a.y, b.y, c.x));
    c.y = sm_f(-a.x, b.y, sm_f(-a.y, b.x, c.y));
    return c;
}

template <class C, class R>
__device__ __forceinline__ void sys_specmul(C G, C gx, C gy, C gz, R k0, const C* in, C* out)
{
    C jG;
    jG.x = -k0 * G.y;  // j k0 G
    jG.y = k0 * G.x;
    const C mx = in[3], my = in[4], mz = in[5];
    out[0] = sm_fma(gz, my, sm_fms(gy, mz, sm_mul(jG, in[0])));
    out[1] = sm_fma(gx, mz, sm_fms(gz, mx, sm_mul(jG, in[1])));
    out[2] = sm_fma(gy, mx, sm_fms(gx, my, sm_mul(jG, in[2])));
    out[3] = sm_mul(G, in[6]);
}

}  // namespace sie

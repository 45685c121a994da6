// Test probe: the conversions between complex128 and the block fixed point of the
// transforms (paper_2003_11679_gb300/csrc/fft.cuh), whose host and device code are the
// same operations, compiled by tests/test_fft_host.py for a CPU check.
#include <cmath>
#include <cstring>

#include "../paper_2003_11679_gb300/csrc/fft.cuh"

static unsigned long long bits(double d) { unsigned long long r; memcpy(&r, &d, 8); return r; }
extern "C" void fx_out(int n, const long long* f, const int* x0, double* a, double* b)
{
    for (int i = 0; i < n; i++) {
        a[i] = x0[i] < 0 ? sie::fx_to_low(f[i], x0[i]) : sie::fx_to(f[i], x0[i]);
        b[i] = x0[i] < 0 ? a[i] : sie::fx_to_int(f[i], x0[i]);
    }
}

// v of a pencil of n components to fixed point and back, as a transform of one point would
extern "C" void fx_round_trip(int n, const double* v, int log2_r1, double* out)
{
    int field = 0;
    for (int i = 0; i < n; i++) {
        const int hi = (int)(bits(v[i]) >> 32) & 0x7ff00000;
        field = field > hi ? field : hi;
    }
    const int emax = (field >> 20) > 1 ? field >> 20 : 1;
    int l1 = 0;
    for (int i = 0; i < n; i++) l1 += sie::fx_l1((unsigned)(bits(v[i]) >> 32), emax);
    const sie::FxScale q = sie::fx_scale(field, l1, log2_r1);
    for (int i = 0; i < n; i++) {
        const unsigned long long u = bits(v[i]);
        // the first pass carries two more bits, rounded off after it
        const long long f = (sie::fx_from((unsigned)(u >> 32), (unsigned)u, q.s0) + 2) >> 2;
        out[i] = q.low ? sie::fx_to_low(f, q.x0) : sie::fx_to(f, q.x0);
    }
}

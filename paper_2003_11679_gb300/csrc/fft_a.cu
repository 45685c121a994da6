// FFT kernels of length 16, 32, 64
#include "fft.cuh"

namespace sie {
SIE_FFT_INSTANCES(16, )
SIE_FFT_INSTANCES(32, )
SIE_FFT_INSTANCES(64, )
}  // namespace sie

// FFT kernels of length 16, 20, 24, 32, 40
#include "fft.cuh"

namespace sie {
SIE_FFT_INSTANCES(16, )
SIE_FFT_INSTANCES(20, )
SIE_FFT_INSTANCES(24, )
SIE_FFT_INSTANCES(32, )
SIE_FFT_INSTANCES(40, )
}  // namespace sie

// FFT kernels of length 48, 64
#include "fft.cuh"

namespace sie {
SIE_FFT_INSTANCES(48, )
SIE_FFT_INSTANCES(64, )
}  // namespace sie

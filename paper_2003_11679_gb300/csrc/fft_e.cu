// FFT kernels of length 80, 96
#include "fft.cuh"

namespace sie {
SIE_FFT_INSTANCES(80, )
SIE_FFT_INSTANCES(96, )
}  // namespace sie

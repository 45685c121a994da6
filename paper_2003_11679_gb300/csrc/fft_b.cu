// FFT kernels of length 128
#include "fft.cuh"

namespace sie {
SIE_FFT_INSTANCES(128, )
}  // namespace sie

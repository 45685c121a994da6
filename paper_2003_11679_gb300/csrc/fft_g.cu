// FFT kernels of length 192
#include "fft.cuh"

namespace sie {
SIE_FFT_INSTANCES(192, )
}  // namespace sie

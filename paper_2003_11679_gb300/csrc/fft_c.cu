// FFT kernels of length 256
#include "fft.cuh"

namespace sie {
SIE_FFT_INSTANCES(256, )
}  // namespace sie

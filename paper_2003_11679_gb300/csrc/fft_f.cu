// FFT kernels of length 160
#include "fft.cuh"

namespace sie {
SIE_FFT_INSTANCES(160, )
}  // namespace sie

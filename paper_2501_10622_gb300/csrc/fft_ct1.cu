// fft_ct1.cu -- compile-time FFT lengths, unit 1 (see fft_ct.cuh).
#include "fft_ct.cuh"

namespace cwthf {
namespace fft {
CWTHF_CT_UNIT(1)
}  // namespace fft
}  // namespace cwthf

// fft_ct4.cu -- compile-time FFT lengths, unit 4 (see fft_ct.cuh).
#include "fft_ct.cuh"

namespace cwthf {
namespace fft {
CWTHF_CT_UNIT(4)
}  // namespace fft
}  // namespace cwthf

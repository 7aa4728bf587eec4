// fft_ct2.cu -- compile-time FFT lengths, unit 2 (see fft_ct.cuh).
#include "fft_ct.cuh"

namespace cwthf {
namespace fft {
CWTHF_CT_UNIT(2)
}  // namespace fft
}  // namespace cwthf

// fft_ct5.cu -- compile-time FFT lengths, unit 5 (see fft_ct.cuh).
#include "fft_ct.cuh"

namespace cwthf {
namespace fft {
CWTHF_CT_UNIT(5)
}  // namespace fft
}  // namespace cwthf

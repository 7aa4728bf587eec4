// fft_ct7.cu -- compile-time FFT lengths, unit 7 (see fft_ct.cuh).
#include "fft_ct.cuh"

namespace cwthf {
namespace fft {
CWTHF_CT_UNIT(7)
}  // namespace fft
}  // namespace cwthf

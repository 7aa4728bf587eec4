// fft_ct6.cu -- compile-time FFT lengths, unit 6 (see fft_ct.cuh).
#include "fft_ct.cuh"

namespace cwthf {
namespace fft {
CWTHF_CT_UNIT(6)
}  // namespace fft
}  // namespace cwthf

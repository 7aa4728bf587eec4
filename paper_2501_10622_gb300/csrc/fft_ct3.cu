// fft_ct3.cu -- compile-time FFT lengths, unit 3 (see fft_ct.cuh).
#include "fft_ct.cuh"

namespace cwthf {
namespace fft {
CWTHF_CT_UNIT(3)
}  // namespace fft
}  // namespace cwthf

// fft_ct0.cu -- compile-time FFT lengths, unit 0 (see fft_ct.cuh).
#include "fft_ct.cuh"

namespace cwthf {
namespace fft {
CWTHF_CT_UNIT(0)
}  // namespace fft
}  // namespace cwthf

// FP32 instances of the row passes (one kernel per transform length).
#include "k_fft_rows.cuh"

namespace rix {
RIX_FFT_ROWS_INST(float)
}  // namespace rix

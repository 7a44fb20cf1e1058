// FP64 instances of the column passes (one kernel per transform length).
#include "k_fft_cols.cuh"

namespace rix {
RIX_FFT_COLS_INST(double)
}  // namespace rix

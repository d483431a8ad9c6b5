// The column passes in single precision (a unit of their own: the kernels take long to compile).
#include "fft_cols.cuh"

namespace dps {
template bool fft_cols_allow<float>();
template bool fft_cols_default<float>(Plan&);
template int fft_set_col_width<float>(Plan&, int, int);
template void launch_fft_cols<float>(const Plan&, int, int, int, cudaStream_t);
}  // namespace dps

// The column passes in double precision (a unit of their own: the kernels take long to compile).
#include "fft_cols.cuh"

namespace dps {
template bool fft_cols_allow<double>();
template bool fft_cols_default<double>(Plan&);
template int fft_set_col_width<double>(Plan&, int, int);
template void launch_fft_cols<double>(const Plan&, int, int, int, cudaStream_t);
}  // namespace dps

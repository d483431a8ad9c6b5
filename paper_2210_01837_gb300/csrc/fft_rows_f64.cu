// The row passes in double precision (a unit of their own: the kernels take long to compile).
#include "fft_rows.cuh"

namespace dps {
template bool fft_rows_allow<double>();
template bool fft_rows_default<double>(Plan&);
template int fft_set_row_variant<double>(Plan&, int);
template void launch_fft_rows<double>(const Plan&, int, cudaStream_t);
}  // namespace dps

// The row passes in single precision (a unit of their own: the kernels take long to compile).
#include "fft_rows.cuh"

namespace dps {
template bool fft_rows_allow<float>();
template bool fft_rows_default<float>(Plan&);
template int fft_set_row_variant<float>(Plan&, int);
template void launch_fft_rows<float>(const Plan&, int, cudaStream_t);
}  // namespace dps

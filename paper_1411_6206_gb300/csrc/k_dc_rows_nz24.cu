// Compile-time planes of the factored-row data-consistency kernel with 24 slices (k_dc_rows.cuh).
#include "k_dc_rows.cuh"

namespace lps {
template cudaError_t launch_dc_rows_nz<24>(const DcArgs&, int, const RowLaunch&, cudaStream_t);
}  // namespace lps

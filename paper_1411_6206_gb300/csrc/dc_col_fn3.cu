// Column transforms of the factored-row data-consistency kernel, a quarter of the slice counts.
#include "dc_col_fn.cuh"

namespace lps {
LPS_COL_INST(4)
LPS_COL_INST(8)
LPS_COL_INST(12)
LPS_COL_INST(16)
LPS_COL_INST(20)
LPS_COL_INST(24)
LPS_COL_INST(28)
LPS_COL_INST(32)
}  // namespace lps

// Column transforms of the factored-row data-consistency kernel, a quarter of the slice counts.
#include "dc_col_fn.cuh"

namespace lps {
LPS_COL_INST(2)
LPS_COL_INST(6)
LPS_COL_INST(10)
LPS_COL_INST(14)
LPS_COL_INST(18)
LPS_COL_INST(22)
LPS_COL_INST(26)
LPS_COL_INST(30)
}  // namespace lps

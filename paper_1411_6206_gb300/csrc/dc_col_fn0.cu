// Column transforms of the factored-row data-consistency kernel, a quarter of the slice counts.
#include "dc_col_fn.cuh"

namespace lps {
LPS_COL_INST(1)
LPS_COL_INST(5)
LPS_COL_INST(9)
LPS_COL_INST(13)
LPS_COL_INST(17)
LPS_COL_INST(21)
LPS_COL_INST(25)
LPS_COL_INST(29)
}  // namespace lps

// Column transforms of the factored-row data-consistency kernel, a quarter of the slice counts.
#include "dc_col_fn.cuh"

namespace lps {
LPS_COL_INST(3)
LPS_COL_INST(7)
LPS_COL_INST(11)
LPS_COL_INST(15)
LPS_COL_INST(19)
LPS_COL_INST(23)
LPS_COL_INST(27)
LPS_COL_INST(31)
}  // namespace lps

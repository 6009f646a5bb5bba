// Row transforms of the factored-row data-consistency kernel, row lengths of LPS_ROW_LIST_0.
#include "dc_row_fn.cuh"

namespace lps {
#define LPS_ROW_INST(NY, A, B) \
  template __device__ float row_phase<A, B>(int, int, int, int, int, const float2*, const __half2*, float2*);
LPS_ROW_LIST_0(LPS_ROW_INST)
}  // namespace lps

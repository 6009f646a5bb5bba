// The row transforms as functions of a runtime mode and slice count (instantiated in dc_row_fn*.cu).
#pragma once

#include "dc_row_body.cuh"

namespace lps {

template <int A, int B>
__device__ float row_phase(int mode, int nz, int tw_off, int task_off, int d_off, const float2* dh,
                           const __half2* dhh, float2* ho) {
  return row_body<A, B>(mode, nz, blockDim.x, reinterpret_cast<float2*>(dc_dsm),
                        reinterpret_cast<const float2*>(dc_dsm + tw_off),
                        reinterpret_cast<const RowTask*>(dc_dsm + task_off),
                        d_off >= 0 ? reinterpret_cast<const float2*>(dc_dsm + d_off) : nullptr, dh, dhh, ho);
}

}  // namespace lps

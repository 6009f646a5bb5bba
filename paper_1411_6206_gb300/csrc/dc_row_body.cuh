// Row transforms of the factored-row data-consistency kernel.
//
// A row of ny = A B points is transformed in place in two passes over shared memory, each task
// holding one short transform in registers: pass 1 an A-point transform over r and the twiddles
// w_ny^(s j); pass 2 a B-point transform over j, the residual on the sampled lines, and its
// inverse; then pass 1 backwards. A task writes the slots that it read, so that one barrier
// between the passes is all the ordering there is. Tasks are spread over all threads of the
// CTA whatever nz, A and B are.
#pragma once

#include "dc_rows.cuh"
#include "dft_reg.cuh"

namespace lps {

// The transforms with mode, nz and the places in shared memory as arguments (constants where the
// caller knows them). ds: the coil's samples in shared memory, or nullptr: read from dh (dhh).
template <int A, int B>
__device__ __forceinline__ float row_body(int mode, int nz, int nt, float2* buf, const float2* tw, const RowTask* tasks,
                                          const float2* ds, const float2* dh, const __half2* dhh, float2* ho) {
  constexpr int RS = row_stride(A, B), BP = B | 1;
  const int tid = threadIdx.x;
  float resid = 0.f;

  if (mode != kDcAdjoint) {
#pragma unroll 1
    for (int t = tid; t < nz * B; t += nt) {
      const int row = t / B, j = t - row * B;
      float2* R = buf + row * RS + j;
      float2 v[A];
#pragma unroll
      for (int r = 0; r < A; ++r) v[r] = R[BP * r];
      dftr::dft<A, false>(v);
#pragma unroll
      for (int s = 1; s < A; ++s) v[s] = cmul(v[s], tw[s * B + j]);
#pragma unroll
      for (int s = 0; s < A; ++s) R[BP * s] = v[s];
    }
    __syncthreads();
  }

#pragma unroll 1
  for (int t = tid; t < nz * A; t += nt) {
    const int row = t / A, s = t - row * A;
    float2* R = buf + row * RS + BP * s;
    const RowTask task = tasks[t];
    float2 w[B];
    if (mode != kDcAdjoint) {
#pragma unroll
      for (int j = 0; j < B; ++j) w[j] = R[j];
      dftr::dft<B, false>(w);
    }
    int l = task.base;
    if (mode == kDcForward) {
#pragma unroll
      for (int q = 0; q < B; ++q) {
        if ((task.mask >> q) & 1u) ho[l] = w[q];
        l += (task.mask >> q) & 1u;
      }
      continue;
    }
    // a sample slot is read for every q (a line that is not sampled reads its successor's, with
    // one slot past the last) and selected afterwards: no branch in the unrolled loop
    if (ds) {
#pragma unroll
      for (int q = 0; q < B; ++q) {
        const bool on = (task.mask >> q) & 1u;
        const float2 d = ds[l];
        const float2 r = mode == kDcAdjoint ? d : csub(w[q], d);
        w[q] = on ? r : make_float2(0.f, 0.f);
        l += on;
      }
    } else {
#pragma unroll
      for (int q = 0; q < B; ++q) {
        const bool on = (task.mask >> q) & 1u;
        float2 d = make_float2(0.f, 0.f);
        if (on) d = dhh ? __half22float2(__ldg(dhh + l)) : __ldg(dh + l);
        const float2 r = mode == kDcAdjoint ? d : csub(w[q], d);
        w[q] = on ? r : make_float2(0.f, 0.f);
        l += on;
      }
    }
    if (mode == kDcUpdate) {
#pragma unroll
      for (int q = 0; q < B; ++q) resid = fmaf(w[q].x, w[q].x, fmaf(w[q].y, w[q].y, resid));
    }
    dftr::dft<B, true>(w);
#pragma unroll
    for (int j = 0; j < B; ++j) R[j] = w[j];
  }
  if (mode == kDcForward) return 0.f;
  __syncthreads();

#pragma unroll 1
  for (int t = tid; t < nz * B; t += nt) {
    const int row = t / B, j = t - row * B;
    float2* R = buf + row * RS + j;
    float2 v[A];
#pragma unroll
    for (int s = 0; s < A; ++s) v[s] = R[BP * s];
#pragma unroll
    for (int s = 1; s < A; ++s) v[s] = cmulc(tw[s * B + j], v[s]);
    dftr::dft<A, true>(v);
#pragma unroll
    for (int r = 0; r < A; ++r) R[BP * r] = v[r];
  }
  return resid;
}

}  // namespace lps

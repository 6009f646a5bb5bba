// Column transforms of the factored-row data-consistency kernel (instantiated in dc_col_fn*.cu):
// the nz points of a pixel column in one thread's registers.
#pragma once

#include "dc_rows.cuh"
#include "dft_reg.cuh"

namespace lps {

template <int NZ>
__device__ void col_fwd(const __half2* Ch, const float2* Z, int xy, int rs, int pos, float sc, int fz) {
  float2* col = reinterpret_cast<float2*>(dc_dsm) + pos;
  float2 v[NZ];
  // Z may have been written by other CTAs of the cluster: read from L2
#pragma unroll
  for (int z = 0; z < NZ; ++z) v[z] = __ldcg(Z + z * xy);
  if (Ch) {
#pragma unroll
    for (int z = 0; z < NZ; ++z) v[z] = cscale(cmul(__half22float2(__ldg(Ch + z * xy)), v[z]), sc);
  } else {
    cp_async_wait_all();
#pragma unroll
    for (int z = 0; z < NZ; ++z) v[z] = cscale(cmul(col[z * rs], v[z]), sc);
  }
  if (fz) dftr::dft<NZ, false>(v);
#pragma unroll
  for (int z = 0; z < NZ; ++z) col[z * rs] = v[z];
}

template <int NZ>
__device__ void col_inv(const float2* C, const __half2* Ch, const float2* Cn, int xy, int rs, int pos, int acc_off,
                        int ny, float sc, int fz, int first) {
  float2* col = reinterpret_cast<float2*>(dc_dsm) + pos;
  float2* acc = reinterpret_cast<float2*>(dc_dsm + acc_off) + threadIdx.x;
  // up to 16 map values are on their way while the column is transformed, the rest while
  // these are used
  constexpr int U = NZ < 16 ? NZ : 16;
  auto coil = [&](int z) -> float2 { return Ch ? __half22float2(__ldg(Ch + z * xy)) : __ldg(C + z * xy); };
  float2 c[U];
#pragma unroll
  for (int u = 0; u < U; ++u) c[u] = coil(u);
  float2 v[NZ];
#pragma unroll
  for (int z = 0; z < NZ; ++z) v[z] = col[z * rs];
  if (Cn) {
#pragma unroll
    for (int z = 0; z < NZ; ++z) cp_async8(col + z * rs, Cn + z * xy);
  }
  if (fz) dftr::dft<NZ, true>(v);
#pragma unroll
  for (int z = 0; z < NZ; ++z) {
    const float2 t = cmulc(c[z % U], v[z]);
    if (z + U < NZ) c[z % U] = coil(z + U);
    const float2 s = first ? make_float2(0.f, 0.f) : acc[z * ny];
    acc[z * ny] = make_float2(fmaf(t.x, sc, s.x), fmaf(t.y, sc, s.y));
  }
}

#define LPS_COL_INST(NZ)                                                                                              \
  template __device__ void col_fwd<NZ>(const __half2*, const float2*, int, int, int, float, int);                      \
  template __device__ void col_inv<NZ>(const float2*, const __half2*, const float2*, int, int, int, int, int, float, \
                                       int, int);

}  // namespace lps

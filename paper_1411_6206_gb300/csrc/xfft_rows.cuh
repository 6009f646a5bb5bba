// Readout transform (k_xfft) of the row lengths of dc_rows.cuh: nx = A B in two register passes,
// instantiated in k_xfft_rows*.cu.
#pragma once

#include "dc_rows.cuh"
#include "dft_reg.cuh"

namespace lps {

constexpr int kXfftLines = 16;   // lines of a CTA: an x-major access of a half-warp is one 128-byte line

// One CTA, kXfftLines lines of one coil. Pass 1 takes the points j + B r straight from global memory
// (A-point transforms, twiddles w^(s j)), one exchange through shared memory, pass 2 (B points)
// stores s + A q straight to it. Neighbouring threads take neighbouring j, or s, where the array is
// line-major and neighbouring lines where it is x-major, so both sides move whole sectors. The lines' stride
// in shared memory is 9 modulo 16 elements: the 16 lines fall on distinct eight-byte banks in the
// one case, and consecutive j or s (B | 1 apart) do in the other. Bound by the latency of one
// round of loads and one of stores. E and E^H of 160 x 160 x 24, 14 coils, us together: 123 with the
// shared-memory Stockham passes of k_xfft (which read, transform and write in four to six phases
// with divisions by the runtime nx), 107 with this.
template <int A, int B, bool INV>
__global__ void __launch_bounds__(16 * (A > B ? A : B)) k_xfft_rows(const XfftArgs a) {
  constexpr int NX = A * B, BP = B | 1, RS = A * BP + (9 - A * BP % 16 + 16) % 16, NL = kXfftLines;
  __shared__ float2 buf[NL * RS];
  __shared__ float2 tw[NX];
  const Geom& g = a.g;
  const int tid = threadIdx.x, c = blockIdx.y, l0 = blockIdx.x * NL;
  for (int i = tid; i < NX; i += blockDim.x) tw[i] = a.tw_x[i / B * (i % B)];
  pdl_wait();   // the samples come from the preceding kernel
  const int m = a.persist->nlines;
  if (l0 >= m) return;
  const int nl = min(NL, m - l0), x0 = g.x0, nxl = g.nx;
  const long long lm = (long long)c * m * NX;                        // line-major: k-space [c][line][kx]
  const long long xm = (long long)c * g.mpad + l0, xs = (long long)g.ncoil * g.mpad;   // x-major: hybrid [x][c][line]
  __syncthreads();
  if (tid < NL * B) {
    const int l = INV ? tid / B : tid % NL, j = INV ? tid % B : tid / NL;
    float2 v[A];
    if (INV) {
      const float2* src = a.in + lm + (l < nl ? (long long)(a.raster ? a.raster[l0 + l] : l0 + l) * NX : 0) + j;
#pragma unroll
      for (int r = 0; r < A; ++r) v[r] = l < nl ? src[B * r] : make_float2(0.f, 0.f);
    } else {
      const float2* src = a.in + xm + l;
#pragma unroll
      for (int r = 0; r < A; ++r) {
        const int xl = j + B * r - x0;
        v[r] = l < nl && xl >= 0 && xl < nxl ? src[xl * xs] : make_float2(0.f, 0.f);
      }
    }
    dftr::dft<A, INV>(v);
#pragma unroll
    for (int s = 1; s < A; ++s) v[s] = INV ? cmulc(tw[s * B + j], v[s]) : cmul(v[s], tw[s * B + j]);
#pragma unroll
    for (int s = 0; s < A; ++s) buf[l * RS + BP * s + j] = v[s];
  }
  __syncthreads();
  if (tid < NL * A) {
    const int l = INV ? tid % NL : tid / A, s = INV ? tid / NL : tid % A;
    float2 w[B];
#pragma unroll
    for (int j = 0; j < B; ++j) w[j] = buf[l * RS + BP * s + j];
    dftr::dft<B, INV>(w);
    if (l >= nl) return;
    const float sc = g.scale_x;
    if (INV) {
#pragma unroll
      for (int q = 0; q < B; ++q) {
        const int xl = s + A * q - x0;
        if (xl >= 0 && xl < nxl) a.out[xm + l + xl * xs] = cscale(w[q], sc);
      }
    } else {
      float2* dst = a.out + lm + (long long)(a.raster ? a.raster[l0 + l] : l0 + l) * NX + s;
#pragma unroll
      for (int q = 0; q < B; ++q) dst[A * q] = cscale(w[q], sc);
    }
  }
}

// Launches the transform if nxt is in list I of dc_rows.cuh, else cudaErrorNotSupported.
template <int I>
cudaError_t launch_xfft_rows(const XfftArgs& a, cudaStream_t st);

}  // namespace lps

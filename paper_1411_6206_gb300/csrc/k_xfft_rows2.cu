// Readout transform (xfft_rows.cuh), row lengths of LPS_ROW_LIST_2.
#include "xfft_rows.cuh"

namespace lps {

template <>
cudaError_t launch_xfft_rows<2>(const XfftArgs& a, cudaStream_t st) {
  const dim3 grid((a.g.mpad + kXfftLines - 1) / kXfftLines, a.g.ncoil);
  cudaError_t e;
#define LPS_XFFT_CASE(NX, A, B)                                                                         \
  case NX:                                                                                              \
    e = a.inverse ? launch_pdl(k_xfft_rows<A, B, true>, grid, dim3(16 * (A > B ? A : B)), 0, st, a)     \
                  : launch_pdl(k_xfft_rows<A, B, false>, grid, dim3(16 * (A > B ? A : B)), 0, st, a);   \
    return e != cudaSuccess ? e : cudaGetLastError();
  switch (a.g.nxt) {
    LPS_ROW_LIST_2(LPS_XFFT_CASE)
    default: return cudaErrorNotSupported;
  }
#undef LPS_XFFT_CASE
}

}  // namespace lps

// Launchers of the runtime-sized data-consistency kernel k_dc (k_dc.cuh) and the choice among the
// data-consistency kernels.
#include "k_dc.cuh"

#include <algorithm>

namespace lps {

int dc_ept(const Geom& g) { return dc_ept_of(g.plane); }

size_t dc_smem_bytes(const Geom& g) {
  size_t b = 0;
  b += 2 * (size_t)g.planeP * sizeof(float2);
  if (!g.dc_direct) b += 2 * (size_t)g.plane * sizeof(float2);   // staged coil planes
  b += (size_t)(g.ny + g.nz + ((g.ny + g.nz) & 1)) * sizeof(float2);
  b += 3 * sizeof(uint64_t);
  b += 32 * sizeof(float);
  b += (size_t)g.nz * g.nz * sizeof(float2);   // W of the iteration form
  return b;
}

template <int MODE, bool STAGE, bool HALF>
static cudaError_t launch_dc_m(const DcArgs& a, cudaStream_t st) {
  const size_t smem = dc_smem_bytes(a.g);
  switch (dc_ept(a.g)) {
    case 1: return launch_dc_t<1, MODE, STAGE, HALF>(a, smem, st);
    case 2: return launch_dc_t<2, MODE, STAGE, HALF>(a, smem, st);
    case 4: return launch_dc_t<4, MODE, STAGE, HALF>(a, smem, st);
    case 8: return launch_dc_t<8, MODE, STAGE, HALF>(a, smem, st);
    case 16: return launch_dc_t<16, MODE, STAGE, HALF>(a, smem, st);
    case 24: return launch_dc_t<24, MODE, STAGE, HALF>(a, smem, st);
    default: return cudaErrorInvalidValue;
  }
}

// Staged coil planes are copied in float32 (the rounded maps); the direct variant of the update
// reads the half-precision copy when the plan keeps one.
template <int MODE>
static cudaError_t launch_dc_s(const DcArgs& a, cudaStream_t st) {
  if (!a.g.dc_direct) return launch_dc_m<MODE, true, false>(a, st);
  if constexpr (MODE == kDcUpdate) {
    if (a.coils_h) return launch_dc_m<MODE, false, true>(a, st);
  }
  return launch_dc_m<MODE, false, false>(a, st);
}

// One persistent launch over a batch's descriptor table (operator form of the update): each CTA
// takes (member, plane) items from an atomic counter, copies the member's arguments to shared
// memory and runs the plane with the runtime-sized body (coil maps read from L2, up to 24
// elements per thread, the shared memory of the largest member). No CTA waits on another.
__global__ void __launch_bounds__(kThreads, 1) k_dc_persist(const DcArgs* __restrict__ table,
                                                          const int* __restrict__ start, int nm, int* counter) {
  __shared__ DcArgs sa;
  __shared__ int item_s, member_s;
  const int total = start[nm];
  for (;;) {
    if (threadIdx.x == 0) {
      const int it = atomicAdd(counter, 1);
      int m = 0;
      while (m + 1 < nm && start[m + 1] <= it) ++m;
      item_s = it;
      member_s = m;
    }
    __syncthreads();
    const int it = item_s, m = member_s;
    if (it >= total) return;
    const int* src = reinterpret_cast<const int*>(table + m);
    int* dst = reinterpret_cast<int*>(&sa);
    for (int i = threadIdx.x; i < (int)(sizeof(DcArgs) / sizeof(int)); i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    dc_plane<24, kDcUpdate, false, false>(sa, it - start[m]);
    __syncthreads();
  }
}
static_assert(sizeof(DcArgs) % sizeof(int) == 0, "DcArgs copied as words");

// The persistent form needs planes of at most 24 * kThreads elements; smem: the largest
// member's runtime-sized direct layout.
bool dc_persist_fits(const Geom& g) {
  Geom gd = g;
  gd.dc_direct = 1;
  return g.plane <= 24 * kThreads && dc_smem_bytes(gd) + sizeof(DcArgs) + 64 <= 227 * 1024;
}

size_t dc_persist_smem(const Geom& g) {
  Geom gd = g;
  gd.dc_direct = 1;
  return dc_smem_bytes(gd);
}

cudaError_t launch_dc_persist(const DcArgs* table, const int* start, int nm, int* counter, size_t smem,
                              cudaStream_t st) {
  // the kernel's static shared memory (its argument copy) counts against the same 227 KB
  static SmemLimit limit;
  cudaError_t e = limit.raise(reinterpret_cast<const void*>(k_dc_persist), smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_dc_persist, kThreads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidValue;
  e = cudaMemsetAsync(counter, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  k_dc_persist<<<per_sm * sms, kThreads, smem, st>>>(table, start, nm, counter);
  return cudaGetLastError();
}

// The update of a 128 x 16 plane goes to the register-transform kernel (k_dc_reg) unless the
// plan selected another variant; the 32 x 8 plane to k_dc_fixed; planes that factor (dc_rows.cuh) to
// k_dc_rows; the rest, and plans that selected a runtime-sized variant, to k_dc.
cudaError_t launch_dc(const DcArgs& a, int mode, cudaStream_t st) {
  if (mode == kDcUpdate) {
    const cudaError_t er = launch_dc_reg(a, st);
    if (er != cudaErrorNotSupported) return er;
  }
  const cudaError_t ef = launch_dc_fixed(a, mode, st);
  if (ef != cudaErrorNotSupported) return ef;
  const cudaError_t ew = launch_dc_rows(a, mode, st);
  if (ew != cudaErrorNotSupported) return ew;
  if (dc_smem_bytes(a.g) > 227 * 1024) return cudaErrorInvalidValue;
  switch (mode) {
    case kDcUpdate: return launch_dc_s<kDcUpdate>(a, st);
    case kDcAdjoint: return launch_dc_s<kDcAdjoint>(a, st);
    case kDcForward: return launch_dc_s<kDcForward>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lps

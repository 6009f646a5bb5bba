// Declarations shared by the factored-row data-consistency kernel (k_dc_rows.cu) and its row
// and column transforms (dc_row_fn.cuh, dc_col_fn.cuh), which are separate device functions:
// any row length of the table below runs with any slice count up to 32 without a kernel per pair.
#pragma once

#include "lps_internal.cuh"

namespace lps {

// Row length ny = A B: pass 1 transforms y = j + B r over r (A points, B transforms a row),
// pass 2 the B points j of every s < A, so that ky = s + A q. B = 16 from 128 on (nz B and nz A
// tasks keep the CTA's ny threads busy in both passes from 16 slices on), 8 below it, an odd
// B beside A = 8 for the odd multiples of 8.
struct RowFactors {
  int A, B;
};
#define LPS_ROW_LIST_0(X) X(8, 4, 2) X(32, 4, 8) X(56, 8, 7) X(80, 10, 8) X(104, 8, 13) X(128, 8, 16) X(152, 8, 19) X(176, 11, 16)
#define LPS_ROW_LIST_1(X) X(16, 4, 4) X(40, 8, 5) X(64, 8, 8) X(88, 8, 11) X(112, 14, 8) X(136, 8, 17) X(160, 10, 16) X(184, 8, 23)
#define LPS_ROW_LIST_2(X) X(24, 8, 3) X(48, 6, 8) X(72, 8, 9) X(96, 12, 8) X(120, 8, 15) X(144, 9, 16) X(168, 12, 14) X(192, 12, 16)
#define LPS_ROW_LIST_3(X) X(200, 8, 25) X(208, 13, 16) X(216, 12, 18) X(224, 14, 16) X(240, 15, 16) X(256, 16, 16)
#define LPS_ROW_LIST(X) LPS_ROW_LIST_0(X) LPS_ROW_LIST_1(X) LPS_ROW_LIST_2(X) LPS_ROW_LIST_3(X)

__host__ __device__ constexpr RowFactors row_factors(int ny) {
#define LPS_ROW_CASE(NY, A, B) ny == NY ? RowFactors{A, B} :
  return LPS_ROW_LIST(LPS_ROW_CASE) RowFactors{0, 0};
#undef LPS_ROW_CASE
}

// Rows lie in shared memory with their blocks of B elements at the odd stride B | 1, element
// y = j + B r at (B | 1) r + j: the lanes of a half-warp then fall on the 16 eight-byte banks in pass 2
// (consecutive s, one block apart), as they do in pass 1 (consecutive j). Rows of blocks of up to
// 8 are spaced so that pass 1 runs over from row to row without conflicts.
__host__ __device__ constexpr int row_stride(int a, int b) {
  return b > 8 ? a * (b | 1) : a * (b | 1) + ((b - a * (b | 1)) % 16 + 16) % 16;
}
__host__ __device__ constexpr int row_pos(int b, int y) { return y / b * (b | 1) + y % b; }

// One task of pass 2, (kz, s): bit q of mask is set where (kz, ky = s + A q) is sampled; these
// lines are numbered base, base + 1, ... in the order of q. (The plan keeps its lines in the order
// of the tasks (kz, s) and q: a permutation of the user's raster order, see dc_row_tasks.)
struct RowTask {
  unsigned mask;
  int base;
};

#ifdef __CUDACC__
extern __shared__ __align__(16) unsigned char dc_dsm[];   // the rows start at its first byte

__device__ __forceinline__ void cp_async8(void* sdst, const void* gsrc) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Row transforms of all nz rows of one coil, between two barriers of the caller: forward passes
// (not for kDcAdjoint), the residual on the sampled lines (its energy is returned) or the samples
// (kDcAdjoint) or the samples' store to ho (kDcForward, which ends there), inverse passes.
// Bytes into dc_dsm: tw_off the twiddles w_ny^(s j) at [s B + j], task_off the tasks [nz][A],
// d_off the coil's samples (-1: they are read from dh, or dhh where that is not null).
template <int A, int B>
__device__ __noinline__ float row_phase(int mode, int nz, int tw_off, int task_off, int d_off, const float2* dh,
                                        const __half2* dhh, float2* ho);

// Column y of one coil, thread y. col_fwd: the thread's map column, which it has copied (cp.async) to
// its own slots of the rows (half-precision maps Ch are read here instead), times sc Z, transformed
// along z (not without fz), back to the slots. col_inv: the column transformed back, times
// conj(C), added to (first: stored in) the thread's column of the sums, acc_off bytes into
// dc_dsm at stride ny; the next coil's map column Cn (if any) is copied to the slots once they
// have been read.
template <int NZ>
__device__ __noinline__ void col_fwd(const __half2* Ch, const float2* Z, int xy, int rs, int pos, float sc, int fz);
template <int NZ>
__device__ __noinline__ void col_inv(const float2* C, const __half2* Ch, const float2* Cn, int xy, int rs, int pos,
                                     int acc_off, int ny, float sc, int fz, int first);
#endif

}  // namespace lps

// Launchers of the factored-row data-consistency kernel (k_dc_rows.cuh), its form for any plane, and
// the host side of its line order.
#include "k_dc_rows.cuh"

#include <algorithm>

namespace lps {

template <int MODE>
__global__ void __maxnreg__(128) k_dc_rows(const DcArgs a, const RowLaunch q) {
  dc_rows_plane<MODE, 0, 0>(a, q);
}

cudaError_t rows_launch(const void* kernel, const DcArgs& a, const RowLaunch& q, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.g.nx * q.kc);
  cfg.blockDim = dim3(q.nt);
  cfg.dynamicSmemBytes = q.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = q.kc * q.pc;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  void* args[2] = {const_cast<DcArgs*>(&a), const_cast<RowLaunch*>(&q)};
  cudaError_t e = cudaLaunchKernelExC(&cfg, kernel, args);
  return e != cudaSuccess ? e : cudaGetLastError();
}

namespace {

template <int MODE>
cudaError_t launch_any(const DcArgs& a, const RowLaunch& q, cudaStream_t st) {
  static SmemLimit limit;
  const void* kernel = reinterpret_cast<const void*>(k_dc_rows<MODE>);
  const cudaError_t e = limit.raise(kernel, 227 * 1024);
  return e != cudaSuccess ? e : rows_launch(kernel, a, q, st);
}

bool rows_fixed(const Geom& g) { return rows_fixed_ny(g.ny) && rows_fixed_nz(g.nz); }

// CTAs an SM holds (the any-plane form has 128 registers).
int rows_fit(const Geom& g) {
  if (rows_fixed(g)) return row_fit(g.ny, g.nz, false, false, 0);
  return std::max(1, std::min(228 * 1024 / (row_layout(g.ny, g.nz, false, false).d + 1024), 65536 / (128 * row_threads(g.ny))));
}

RowLaunch row_launch(const Geom& g, int kc, int pc) {
  RowLaunch q{};
  q.kc = kc;
  q.pc = pc;
  q.nt = row_threads(g.ny);
  q.lay = row_layout(g.ny, g.nz, rows_fixed(g) && row_z_shared(g.ny, g.nz), rows_fixed(g) && row_w_shared(g.ny, g.nz));
  q.smem = q.lay.d;
  // sample slots: as many as leave the CTAs that fit an SM without them
  const int room = std::min(227 * 1024, 228 * 1024 / rows_fit(g) - 1024) - q.smem;
  q.d_slots = room > 0 ? std::min(g.mpad + 2, room / (int)sizeof(float2)) : 0;
  q.smem += q.d_slots * (int)sizeof(float2);
  const int ych = ((g.ny + kc - 1) / kc + 7) & ~7, m_bytes = (8 * g.nz * (ych | 1) + 15) / 16 * 16;
  const bool behind = m_bytes + row_gram_bytes(g.ny, g.nz) <= q.lay.tw;
  q.gram_off = behind ? m_bytes : q.lay.acc;
  q.gram_sync = !behind && kc > 1;
  return q;
}

// CTAs per plane. The fullest of the 152 SMs works through n = nx kc / 152 CTAs in rounds of
// as many as it holds; a round takes its coils and about two coils' time for the prologue,
// epilogue and first loads, a fifth longer for every CTA that shares the SM. Over 13 planes this is 0.2 %
// from the fastest kc of each. Us per iteration at kc = 1, 2, 3, 4, 5, 7: 192 x 192 x 32, 12 coils 205, 191,
// 173, 195, 222, 250; 160 x 160 x 24, 14 coils 155, 120, 132, 123, 118, 134; 112 x 112 x 14, 15 coils 62, 53, 50,
// 50, 46, 60; 80 x 80 x 24, 13 coils 91, 77, 66, 67, 60, 58.
int rows_kc(const Geom& g) {
  const int fit = rows_fit(g);
  int best = 1;
  double least = 1e30;
  for (int kc = 1; kc <= std::min(8, g.ncoil); ++kc) {
    const int coils = (g.ncoil + kc - 1) / kc;
    double t = 0;
    for (int n = (g.nx * kc + 151) / 152; n > 0; n -= fit) {
      t += (coils + 2) * (0.8 + 0.2 * std::min(n, fit));
    }
    if (t < least) {
      least = t;
      best = kc;
    }
  }
  return best;
}

}  // namespace

bool dc_rows_geometry(const Geom& g) {
  if (g.cs != 1 || g.nz > 32 || row_factors(g.ny).A == 0) return false;
  return row_layout(g.ny, g.nz, false, false).d <= 227 * 1024;
}

// Number of Gram partials the data-consistency step leaves for the eigen kernel.
int dc_gram_parts(const Geom& g) {
  if (dc_reg_applies(g) || dc_small_applies(g)) return g.nx / 4;
  return g.nx;
}

// The benchmark planes, where lps_tune_result.dc_variant 0 names the default besides k_dc_reg (k_dc_fixed
// for 32 x 8, else the factored-row kernel).
bool dc_has_fixed(const Geom& g) {
  return dc_rows_geometry(g) &&
         ((g.ny == 128 && g.nz == 16) || (g.ny == 192 && g.nz == 32) || (g.ny == 32 && g.nz == 8));
}

bool dc_rows_applies(const Geom& g) { return g.dc_rows && !g.dc_generic && dc_rows_geometry(g); }

size_t dc_row_task_bytes(const Geom& g) { return (size_t)g.nz * row_factors(g.ny).A * sizeof(RowTask); }

// Tasks of a mask, its lines' positions kz nyp + ky in task order, and for each of them its number in
// the raster order of the mask. lines may be null.
void dc_row_tasks(const Geom& g, const unsigned char* mask, void* tasks, int* lines, unsigned short* raster) {
  const RowFactors f = row_factors(g.ny);
  RowTask* t = static_cast<RowTask*>(tasks);
  int l = 0, before = 0;   // before: sampled lines of the slices before z
  for (int z = 0; z < g.nz; ++z) {
    const unsigned char* row = mask + (size_t)z * g.ny;
    int number[1024], n = 0;
    for (int ky = 0; ky < g.ny; ++ky) number[ky] = row[ky] ? before + n++ : -1;
    for (int s = 0; s < f.A; ++s, ++t) {
      t->mask = 0;
      t->base = l;
      for (int q = 0; q < f.B; ++q) {
        const int ky = s + f.A * q;
        if (number[ky] < 0) continue;
        t->mask |= 1u << q;
        if (lines) lines[l] = z * g.nyp + ky;
        raster[l++] = (unsigned short)number[ky];
      }
    }
    before += n;
  }
}

cudaError_t launch_dc_rows(const DcArgs& a, int mode, cudaStream_t st) {
  if (!a.tasks || !dc_rows_applies(a.g)) return cudaErrorNotSupported;
  // as many planes a cluster as the eigen kernel expects to a partial (with k_dc_reg for the
  // update its four)
  const int pc = a.gram_part ? a.g.nx / dc_gram_parts(a.g) : 1;
  const RowLaunch q = row_launch(a.g, std::min(rows_kc(a.g), 8 / pc), pc);
  if (rows_fixed(a.g)) {
#define LPS_ROWS_CASE(NZ) \
  case NZ: return launch_dc_rows_nz<NZ>(a, mode, q, st);
    switch (a.g.nz) {
      LPS_ROWS_NZ_LIST(LPS_ROWS_CASE)
      default: break;
    }
#undef LPS_ROWS_CASE
  }
  switch (mode) {
    case kDcUpdate: return launch_any<kDcUpdate>(a, q, st);
    case kDcAdjoint: return launch_any<kDcAdjoint>(a, q, st);
    default: return launch_any<kDcForward>(a, q, st);
  }
}

}  // namespace lps

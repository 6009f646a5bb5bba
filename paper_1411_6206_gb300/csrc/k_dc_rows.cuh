// Data-consistency step (Algorithm 1 step 4, Sec. 3) and the acquisition operator both ways
// (Sec. 2) on x-planes of any slice count up to 32 and the row lengths of dc_rows.cuh, in the
// hybrid-space form of k_dc.cuh:
//     X = Z - sum_c conj(C_c) F_yz^H [ M F_yz (C_c Z) - d'_c ],     Z = L + S.
//
// One x-plane is worked on by a cluster of kc CTAs (one thread per pixel column each); CTA r
// takes the coils r, r + kc, ... and keeps their sum in its own shared memory. Per coil: the z
// transform of the thread's column in registers, the row transforms through shared memory with the
// residual in the middle (dc_row_body.cuh), the z transform back, the product with conj(C_c) and
// the sum; five barriers. Splitting the coils of a plane over CTAs rather than over groups of one
// CTA keeps the shared memory of a unit to one transform buffer and one sum, so that several units
// share an SM and hide each other's barriers and loads, and evens out the load when the planes
// are not a multiple of the SMs (192 planes of 12 coils on 152 SMs: 8 coil steps on the fullest SM
// instead of 12).
//
// What bounds it: the issue of the transforms' own instructions (about 140 a point and coil; 6,100
// cycles a coil and 192 x 32 plane of the 9,800 measured with two CTAs an SM), then the latency of
// the loads between its phases. The planes of the benchmark workloads are instantiated (a map column is then
// read once a coil and stays in registers); any other goes through functions of the row length and
// of the slice count, at about 1.6 times the time.
//
// Step (4) alone, us, before (shared-memory Stockham passes with 11 barriers a coil, or the
// 16-lane shuffle transforms that planes of ny = 16 Q had) and now: 192 x 192 x 32, 12 coils 202 and 98;
// 160 x 160 x 32, 12 coils 189 and 84; 160 x 160 x 24, 14 coils 157 and 71; 160 x 160 x 14, 16 coils 92 and 46;
// 120 x 104 x 15, 6 coils 128 and 23. E of 160 x 160 x 24, 14 coils 175 and 60, E^H 208 and 56 (with the
// kx transform).
//
// In the iteration form the CTAs of a plane first share out its pixel columns to form
// L_k = (X_{k-1} - S_{k-1}) W and Z = L_k + S_k, which is left in X (X_{k-1} has been consumed) for
// the cluster to read; in the end they share out the columns again to add the coil sums through
// distributed shared memory in rank order, write X_k and form the plane's Gram. A cluster holds
// pc planes, whose Grams are summed before they are written.
#pragma once

#include "dc_row_body.cuh"

#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace lps {

// Shared memory of a CTA, bytes into dc_dsm (the rows come first): twiddles, tasks, coil sums (also M
// or W in the prologue and the Gram's partial sums in the epilogue), Z (zs) and W (ws) of their own,
// scratch, sample slots.
struct RowLayout {
  int tw, task, acc, zs, w, red, d;
};
__host__ __device__ constexpr int row_max(int a, int b) { return a > b ? a : b; }
__host__ __device__ constexpr int row_min(int a, int b) { return a < b ? a : b; }
__host__ __device__ constexpr int row_threads(int ny) { return row_max(64, (ny + 31) / 32 * 32); }
__host__ __device__ constexpr int row_gram_bytes(int ny, int nz) {
  const int n4 = (nz + 3) / 4, np = n4 * (n4 + 1) / 2;
  return 8 * (nz * nz + 16 * np * (row_threads(ny) / np));
}
__host__ __device__ constexpr RowLayout row_layout(int ny, int nz, bool zs, bool ws) {
  const RowFactors f = row_factors(ny);
  const int w4 = 16 * nz * ((nz + 3) / 4 * 4);
  RowLayout l{};
  l.tw = (8 * nz * row_max(row_stride(f.A, f.B), ny + 1) + 15) / 16 * 16;
  l.task = l.tw + 8 * ny;
  l.acc = l.task + (8 * nz * f.A + 15) / 16 * 16;
  l.zs = l.acc + (row_max(8 * nz * (ws ? ny + 1 : ny), row_max(w4, row_gram_bytes(ny, nz))) + 15) / 16 * 16;
  l.w = l.zs + (zs ? 8 * nz * ny : 0);
  l.red = l.w + (ws ? w4 : 0);
  l.d = l.red + 100 * 4;
  return l;
}

// CTAs an SM holds, by shared memory (with `slots` samples of a coil) and by registers (a map column, a
// transform and its temporaries). Z is kept in shared memory where that and the samples of a
// fifth of the lines cost no CTA, and so is a place of its own for W (M then leaves the rows to the
// first coil's map column, which is copied before the wait).
__host__ __device__ constexpr int row_regs(int nz) { return (2 * nz + 88 + 7) / 8 * 8; }
__host__ __device__ constexpr int row_fit(int ny, int nz, bool zs, bool ws, int slots) {
  return row_max(1, row_min(228 * 1024 / (row_layout(ny, nz, zs, ws).d + 8 * slots + 1024),
                            65536 / (row_threads(ny) * row_regs(nz))));
}
__host__ __device__ constexpr bool row_z_shared(int ny, int nz) {
  return row_fit(ny, nz, true, false, ny * nz / 5) == row_fit(ny, nz, false, false, 0);
}
__host__ __device__ constexpr bool row_w_shared(int ny, int nz) {
  return row_fit(ny, nz, row_z_shared(ny, nz), true, ny * nz / 5) == row_fit(ny, nz, false, false, 0);
}

struct RowLaunch {
  int kc, pc;      // CTAs per plane, planes per cluster
  int nt;          // threads per CTA
  RowLayout lay;
  int d_slots;     // samples of a coil that fit at lay.d
  int gram_off;    // the Gram's partial sums, and whether they share the coil sums' memory with readers
  int gram_sync;
  int smem;
};

__device__ __forceinline__ float call_rows(int ny, int mode, int nz, int tw_off, int task_off, int d_off,
                                           const float2* dh, const __half2* dhh, float2* ho) {
#define LPS_ROW_CASE(NY, A, B) \
  case NY: return row_phase<A, B>(mode, nz, tw_off, task_off, d_off, dh, dhh, ho);
  switch (ny) {
    LPS_ROW_LIST(LPS_ROW_CASE)
    default: return 0.f;
  }
#undef LPS_ROW_CASE
}

#define LPS_COL_CASES(F)                                                                                   \
  F(1) F(2) F(3) F(4) F(5) F(6) F(7) F(8) F(9) F(10) F(11) F(12) F(13) F(14) F(15) F(16) F(17) F(18) F(19) \
  F(20) F(21) F(22) F(23) F(24) F(25) F(26) F(27) F(28) F(29) F(30) F(31) F(32)

__device__ __forceinline__ void call_col_fwd(int nz, const __half2* Ch, const float2* Z, int xy, int rs, int pos, float sc,
                                             int fz) {
#define LPS_COL_CASE(NZ) \
  case NZ: col_fwd<NZ>(Ch, Z, xy, rs, pos, sc, fz); break;
  switch (nz) {
    LPS_COL_CASES(LPS_COL_CASE)
    default: break;
  }
#undef LPS_COL_CASE
}

__device__ __forceinline__ void call_col_inv(int nz, const float2* C, const __half2* Ch, const float2* Cn, int xy, int rs,
                                             int pos, int acc_off, int ny, float sc, int fz, int first) {
#define LPS_COL_CASE(NZ) \
  case NZ: col_inv<NZ>(C, Ch, Cn, xy, rs, pos, acc_off, ny, sc, fz, first); break;
  switch (nz) {
    LPS_COL_CASES(LPS_COL_CASE)
    default: break;
  }
#undef LPS_COL_CASE
}

// Sums of three values over the block in a fixed order, in thread 0. red holds 3 * 32 floats.
__device__ __forceinline__ void block_sum3(float (&v)[3], float* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    v[i] = warp_sum(v[i]);
    if (lane == 0) red[32 * i + w] = v[i];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      v[i] = 0.f;
      for (int k = 0; k < nw; ++k) v[i] += red[32 * i + k];
    }
  }
}

// NY, NZ > 0: the plane is fixed at compile time, its transforms are inlined and the thread's map
// column stays in registers from the first product to the last. NY = 0: any plane, through the
// functions of dc_row_fn*.cu and dc_col_fn*.cu.
template <int MODE, int NY, int NZ>
__device__ __forceinline__ void dc_rows_plane(const DcArgs& a, const RowLaunch& q) {
  constexpr bool FIXED = NY > 0;
  constexpr bool ZS = FIXED && row_z_shared(NY, NZ);
  const Geom& g = a.g;
  const int nx = g.nx, ny = FIXED ? NY : g.ny, nz = FIXED ? NZ : g.nz, ncoil = g.ncoil;
  const int tid = threadIdx.x, nt = FIXED ? row_threads(NY) : blockDim.x;
  constexpr bool WS = FIXED && row_w_shared(NY, NZ);
  const RowLayout lay = FIXED ? row_layout(NY, NZ, ZS, WS) : q.lay;
  const int kc = q.kc, cl_size = kc * q.pc;
  const int crank = blockIdx.x % cl_size, pl = crank / kc, rank = crank - pl * kc;
  const int x = blockIdx.x / cl_size * q.pc + pl;
  const int xy = nx * ny, xo = x * ny;
  cg::cluster_group cl = cg::this_cluster();
  float2* buf = reinterpret_cast<float2*>(dc_dsm);
  float2* tw = reinterpret_cast<float2*>(dc_dsm + lay.tw);
  float2* acc = reinterpret_cast<float2*>(dc_dsm + lay.acc);
  float* red = reinterpret_cast<float*>(dc_dsm + lay.red);   // [96] scratch, [96..98] this CTA's statistics
  const RowFactors f = row_factors(ny);
  const int rs = row_stride(f.A, f.B);

  const int m = a.persist->nlines;
  for (int i = tid; i < ny; i += nt) {
    const int s = i / f.B, j = i - s * f.B;
    tw[i] = a.tw_y[s * j];
  }
  RowTask* tasks = reinterpret_cast<RowTask*>(dc_dsm + lay.task);
  for (int i = tid; i < nz * f.A; i += nt) tasks[i] = a.tasks[i];
  // this CTA's share of the plane's columns in the prologue and the epilogue: yc columns from y0,
  // thread (zl, yl) taking slices zl, zl + zs, ...
  const int ych = ((ny + kc - 1) / kc + 7) & ~7;
  const int y0 = min(ny, rank * ych), yc = min(ny, y0 + ych) - y0;
  const int zs = yc > 0 ? nt / yc : 1, zl = yc > 0 ? tid / yc : 0, yl = yc > 0 ? tid - zl * yc : 0;
  const bool mine = yc > 0 && zl < zs;
  const int ms = ych | 1;                     // column stride of M in buf
  const int yo = xo + y0 + yl;                // the thread's column in slice 0
  const bool early = MODE == kDcUpdate && a.W != nullptr;
  // The map column of the CTA's next coil goes to the thread's own slots of the rows, its samples
  // to the sample slots (where the mask's lines fit them), as soon as the previous coil has left
  // them; both have landed when the next coil begins.
  const bool col = tid < ny;
  const int pos = row_pos(f.B, tid);
  const float sc = g.scale_yz;
  const bool staged = MODE != kDcForward && m + 1 < q.d_slots;
  const bool half_maps = MODE == kDcUpdate && a.coils_h != nullptr;
  const bool half_data = MODE == kDcUpdate && a.dhyb_h != nullptr;
  float2* ds = reinterpret_cast<float2*>(dc_dsm + lay.d);
  auto row_of = [&](int c) { return ((long long)x * ncoil + c) * g.mpad; };
  auto stage_samples = [&](int c) {
    if (half_data) {
      const __half2* src = a.dhyb_h + row_of(c);
      for (int i = tid; i < m; i += nt) ds[i] = __half22float2(src[i]);
    } else {
      const float2* src = a.dhyb + row_of(c);
      for (int i = tid; 2 * i < m; i += nt) cp_async16(ds + 2 * i, src + 2 * i);   // rows of mpad (even) samples
    }
  };
  auto map_col = [&](int c) -> const float2* { return a.coils + (long long)c * g.N + xo + tid; };
  auto half_col = [&](int c) -> const __half2* {
    return half_maps ? a.coils_h + (long long)c * g.N + xo + tid : nullptr;
  };
  auto stage_map = [&](const float2* C) {
#pragma unroll
    for (int z = 0; z < nz; ++z) cp_async8(buf + z * rs + pos, C + z * xy);
  };
  // In a frame (ctrl) the maps and the samples were complete before its first kernel started: the
  // first coil's are copied before the wait, its map column unless the rows hold M first. A call of
  // one operator may directly follow the kernel that wrote them and copies them after it.
  float2* Msh = WS ? acc : buf;
  auto stage_first_map = [&]() {
    if (MODE != kDcAdjoint && col && !half_maps) stage_map(map_col(rank));
  };
  if (!a.ctrl) pdl_wait();
  if (staged) stage_samples(rank);
  if (WS || !early) stage_first_map();
  // Iteration form with W: this launch is released by the eigen kernel after that kernel's own
  // wait, so the outputs of the data-consistency kernel before it and of what that one waited for
  // (X_{k-1}, S_{k-1}, L_{k-1}) are read while it still runs: M_{k-1} into shared memory, Z_{k-1} of the
  // thread's first tasks into registers. (S_k is not: the sparse step beside the eigen kernel is a
  // programmatic predecessor too, which only the wait waits for.) They are read from L2: a launch
  // that starts before its predecessors have ended may find older lines in this SM's L1. A task is
  // one column and OT slices of L_k.
  constexpr int OT = 4, EARLY = 3;
  float2 Sk[EARLY][OT], Zo[EARLY][OT];
  auto load_prev = [&](int jb, float2 (&zo)[OT]) {
#pragma unroll
    for (int j = 0; j < OT; ++j) {
      const int gi = (jb + j) * xy + yo;
      zo[j] = jb + j < nz ? cadd(__ldcg(a.Lbuf + gi), __ldcg(a.Sprev + gi)) : make_float2(0.f, 0.f);
    }
  };
  auto load_sparse = [&](int jb, float2 (&sk)[OT]) {
#pragma unroll
    for (int j = 0; j < OT; ++j) sk[j] = jb + j < nz ? a.S[(jb + j) * xy + yo] : make_float2(0.f, 0.f);
  };
  if (early && mine) {
#pragma unroll 4
    for (int z = zl; z < nz; z += zs) Msh[z * ms + yl] = csub(__ldcg(a.X + z * xy + yo), __ldcg(a.Sprev + z * xy + yo));
#pragma unroll
    for (int k = 0; k < EARLY; ++k) load_prev(OT * (zl + k * zs), Zo[k]);
  }
  pdl_wait();
  if (a.ctrl && a.ctrl->converged) {
    cp_async_wait_all();
    return;
  }

  float dz2 = 0.f, z2 = 0.f, resid = 0.f;   // ||Z_k - Z_{k-1}||^2, ||Z_{k-1}||^2, ||E Z - d||^2: this thread's share
  const float2* Z = nullptr;
  float2* zsm = reinterpret_cast<float2*>(dc_dsm + lay.zs);
  const bool z_here = ZS && early && kc == 1;   // Z goes straight to this CTA's shared memory
  if (MODE == kDcUpdate) {
    Z = a.L;
    if (a.W) {
      if (mine) {
#pragma unroll
        for (int k = 0; k < EARLY; ++k) load_sparse(OT * (zl + k * zs), Sk[k]);
      }
      // W as (x, y, -y, x): a product is two packed multiply-adds on one 16-byte broadcast
      float4* W4 = reinterpret_cast<float4*>(WS ? dc_dsm + lay.w : dc_dsm + lay.acc);
      const int nzp = (nz + OT - 1) / OT * OT;
      for (int i0 = tid; i0 < nz * nzp; i0 += 6 * nt) {
        float2 w[6];
#pragma unroll
        for (int u = 0; u < 6; ++u) {
          const int i = i0 + u * nt, r = i / nzp, c = i - r * nzp;
          w[u] = r < nz && c < nz ? a.W[r * nz + c] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < 6; ++u)
          if (i0 + u * nt < nz * nzp) W4[i0 + u * nt] = make_float4(w[u].x, w[u].y, -w[u].y, w[u].x);
      }
      __syncthreads();
      auto task = [&](int jb, const float2 (&sk)[OT], const float2 (&zo)[OT]) {
        float2 o[OT];
#pragma unroll
        for (int j = 0; j < OT; ++j) o[j] = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int i = 0; i < nz; ++i) {
          const float2 mv = Msh[i * ms + yl];
#pragma unroll
          for (int j = 0; j < OT; ++j) {
            const float4 w = W4[i * nzp + jb + j];
            o[j] = dftr::axpy(make_float2(w.x, w.y), mv.x, dftr::axpy(make_float2(w.z, w.w), mv.y, o[j]));
          }
        }
#pragma unroll
        for (int j = 0; j < OT; ++j) {
          if (jb + j >= nz) break;
          const int gi = (jb + j) * xy + yo;
          a.Lbuf[gi] = o[j];
          if (z_here)
            zsm[(jb + j) * ny + y0 + yl] = cadd(o[j], sk[j]);
          else
            a.X[gi] = cadd(o[j], sk[j]);
          dz2 += cabs2(cadd(o[j], csub(sk[j], zo[j])));
          z2 += cabs2(zo[j]);
        }
      };
      if (mine) {
#pragma unroll
        for (int k = 0; k < EARLY; ++k)
          if (OT * (zl + k * zs) < nz) task(OT * (zl + k * zs), Sk[k], Zo[k]);
        for (int jb = OT * (zl + EARLY * zs); jb < nz; jb += OT * zs) {
          load_prev(jb, Zo[0]);
          load_sparse(jb, Sk[0]);
          task(jb, Sk[0], Zo[0]);
        }
      }
      Z = a.X;
    } else if (a.Lpre || a.S) {
      if (mine) {
#pragma unroll 4
        for (int z = zl; z < nz; z += zs) {
          const int gi = z * xy + yo;
          const float2 Sk = a.S[gi];
          if (a.Lpre) {
            const float2 Zo = cadd(a.Lbuf[gi], a.Sprev[gi]), Lk = a.Lpre[gi];
            a.Lbuf[gi] = Lk;
            a.X[gi] = cadd(Lk, Sk);
            dz2 += cabs2(cadd(Lk, csub(Sk, Zo)));
            z2 += cabs2(Zo);
          } else {
            a.X[gi] = cadd(a.L[gi], Sk);
          }
        }
      }
      Z = a.X;
    }
  } else if (MODE == kDcForward) {
    Z = a.L;
  }
  // Z is read by the whole cluster; M and W are done with
  if (Z == a.X && kc > 1)
    cl.sync();
  else
    __syncthreads();
  if (!WS && early) stage_first_map();

  // ---- coil loop ----------------------------------------------------------------------------
  if constexpr (FIXED) {
    constexpr RowFactors F = row_factors(NY);
    constexpr int RS = row_stride(F.A, F.B);
    float2* bc = buf + pos;
    float2* ac = acc + tid;
    float2* zc = zsm + tid;
    const float2* Zc = MODE == kDcAdjoint ? nullptr : Z + xo + tid;
    if (ZS && MODE != kDcAdjoint && col && !z_here) {
#pragma unroll
      for (int z = 0; z < NZ; ++z) zc[z * NY] = __ldcg(Zc + z * xy);   // this thread's column: no barrier
    }
    for (int c = rank; c < ncoil; c += kc) {
      const bool more = c + kc < ncoil;
      float2 cm[NZ];
      if (col && MODE == kDcAdjoint) {
        const float2* C = map_col(c);
#pragma unroll
        for (int z = 0; z < NZ; ++z) cm[z] = __ldg(C + z * xy);
      } else if (col) {
        float2 v[NZ];
#pragma unroll
        for (int z = 0; z < NZ; ++z) v[z] = ZS ? zc[z * NY] : __ldcg(Zc + z * xy);
        if (half_maps) {
          const __half2* Ch = half_col(c);
#pragma unroll
          for (int z = 0; z < NZ; ++z) cm[z] = __half22float2(__ldg(Ch + z * xy));
        } else {
          cp_async_wait_all();
#pragma unroll
          for (int z = 0; z < NZ; ++z) cm[z] = bc[z * RS];
        }
#pragma unroll
        for (int z = 0; z < NZ; ++z) v[z] = cscale(cmul(cm[z], v[z]), sc);
        if (g.fft_z) dftr::dft<NZ, false>(v);
#pragma unroll
        for (int z = 0; z < NZ; ++z) bc[z * RS] = v[z];
      }
      cp_async_wait_all();
      __syncthreads();
      resid += row_body<F.A, F.B>(MODE, NZ, row_threads(NY), buf, tw, tasks, staged ? ds : nullptr,
                                  MODE == kDcForward ? nullptr : a.dhyb + row_of(c),
                                  half_data ? a.dhyb_h + row_of(c) : nullptr,
                                  MODE == kDcForward ? a.hyb_out + row_of(c) : nullptr);
      __syncthreads();
      if (staged && more) stage_samples(c + kc);
      if (MODE == kDcForward) {
        if (col && more) stage_map(map_col(c + kc));
      } else if (col) {
        float2 v[NZ];
#pragma unroll
        for (int z = 0; z < NZ; ++z) v[z] = bc[z * RS];
        if (MODE == kDcUpdate && more && !half_maps) stage_map(map_col(c + kc));
        if (g.fft_z) dftr::dft<NZ, true>(v);
#pragma unroll
        for (int z = 0; z < NZ; ++z) {
          const float2 t = cmulc(cm[z], v[z]);
          const float2 s = c == rank ? make_float2(0.f, 0.f) : ac[z * NY];
          ac[z * NY] = make_float2(fmaf(t.x, sc, s.x), fmaf(t.y, sc, s.y));
        }
      }
    }
  } else {
    for (int c = rank; c < ncoil; c += kc) {
      const bool more = c + kc < ncoil;
      if (MODE != kDcAdjoint && col) call_col_fwd(nz, half_col(c), Z + xo + tid, xy, rs, pos, sc, g.fft_z);
      cp_async_wait_all();
      __syncthreads();
      resid += call_rows(ny, MODE, nz, lay.tw, lay.task, staged ? lay.d : -1,
                         MODE == kDcForward ? nullptr : a.dhyb + row_of(c), half_data ? a.dhyb_h + row_of(c) : nullptr,
                         MODE == kDcForward ? a.hyb_out + row_of(c) : nullptr);
      __syncthreads();
      if (staged && more) stage_samples(c + kc);
      if (MODE == kDcForward) {
        if (col && more) stage_map(map_col(c + kc));
      } else if (col) {
        call_col_inv(nz, map_col(c), half_col(c), MODE == kDcUpdate && !half_maps && more ? map_col(c + kc) : nullptr, xy,
                     rs, pos, lay.acc, ny, sc, g.fft_z, c == rank);
      }
    }
  }
  // (a thread's next coil writes the column that it has read: no barrier at the end of a coil)
  pdl_trigger();   // not earlier: the next kernels' CTAs would wait on the SMs through the coil loop
  if (MODE == kDcForward) return;

  // ---- epilogue: X_k = Z - sum over the CTAs of the plane, M = X_k - S_k ----------------------
  if (kc > 1)
    cl.sync();
  else
    __syncthreads();
  if (mine) {
    // four slices and the sums of four CTAs a round: their loads overlap
    constexpr int U = 4;
    for (int zb = zl; zb < nz; zb += U * zs) {
      float2 s[U], Zv[U], Sv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int z = zb + u * zs, gi = z * xy + yo;
        s[u] = Zv[u] = Sv[u] = make_float2(0.f, 0.f);
        if (z < nz && MODE == kDcUpdate) {
          Zv[u] = ZS ? zsm[z * ny + y0 + yl] : __ldcg(Z + gi);
          if (a.S) Sv[u] = a.S[gi];
        }
      }
      for (int r0 = 0; r0 < kc; r0 += 4) {
        float2 t[4][U];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float2* o = kc > 1 && r0 + r < kc ? cl.map_shared_rank(acc, pl * kc + r0 + r) : acc;
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int z = zb + u * zs;
            t[r][u] = z < nz && r0 + r < kc ? o[z * ny + y0 + yl] : make_float2(0.f, 0.f);
          }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int u = 0; u < U; ++u) s[u] = cadd(s[u], t[r][u]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int z = zb + u * zs, gi = z * xy + yo;
        if (z >= nz) break;
        float2 Xv = s[u];
        if (MODE == kDcUpdate) {
          Xv = csub(Zv[u], s[u]);
          if (a.recon) a.recon[gi] = Zv[u];
        } else {
          if (a.L_out) a.L_out[gi] = Xv;
          if (a.S_out) a.S_out[gi] = make_float2(0.f, 0.f);
        }
        a.X[gi] = Xv;
        buf[z * ms + yl] = csub(Xv, Sv[u]);
      }
    }
  }
  float* stat = red + 96;
  if (MODE == kDcUpdate && a.dc_part) {
    float t[3] = {resid, dz2, z2};
    block_sum3(t, red);
    if (tid == 0 && kc == 1) {
      reinterpret_cast<float4*>(a.dc_part)[x] = make_float4(t[0], t[1], t[2], 0.f);
    } else if (tid == 0) {
      stat[0] = t[0];
      stat[1] = t[1];
      stat[2] = t[2];
    }
  }
  // the Gram's partial sums lie behind M in the rows where they fit there, else in the place of the
  // coil sums, once every CTA of the plane has read them
  if (q.gram_sync)
    cl.sync();
  else
    __syncthreads();
  float2* gsm = reinterpret_cast<float2*>(dc_dsm + q.gram_off);   // [nz][nz]
  float2* gp = a.gram_part + (long long)(x / q.pc) * nz * nz;
  float2* gout = cl_size > 1 ? gsm : gp;
  if (a.gram_part) {
    // G[i][j] = sum_y conj(M[i][y]) M[j][y] over this CTA's columns: 4 x 4 entries a thread over
    // every ng-th column, the ng partial sums added in order
    float2* part = gsm + nz * nz;
    const int n4 = (nz + 3) / 4, np = n4 * (n4 + 1) / 2, ng = nt / np;
    const int grp = tid / np, p = tid - grp * np;
    int ti = 0, rem = p;
    while (rem >= n4 - ti) {
      rem -= n4 - ti;
      ++ti;
    }
    const int tj = ti + rem;
    if (grp < ng) {
      float2 s[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[i][j] = make_float2(0.f, 0.f);
      int ri[4], rj[4];   // rows past the last repeat it (their entries are not used)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        ri[i] = min(nz - 1, 4 * ti + i) * ms;
        rj[i] = min(nz - 1, 4 * tj + i) * ms;
      }
      for (int y = grp; y < yc; y += ng) {
        float2 u[4], v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          u[i] = buf[ri[i] + y];
          v[i] = buf[rj[i] + y];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            s[i][j].x = fmaf(u[i].x, v[j].x, fmaf(u[i].y, v[j].y, s[i][j].x));
            s[i][j].y = fmaf(u[i].x, v[j].y, fmaf(-u[i].y, v[j].x, s[i][j].y));
          }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) part[(i * 4 + j) * (np * ng) + tid] = s[i][j];
    }
    __syncthreads();
    for (int e = tid; e < nz * nz; e += nt) {
      const int i = e / nz, j = e - i * nz;
      if (i > j) continue;
      const int bi = i >> 2, bj = j >> 2;
      const float2* src = part + ((i & 3) * 4 + (j & 3)) * (np * ng) + bi * n4 - bi * (bi - 1) / 2 + (bj - bi);
      float2 s = src[0];
      for (int r = 1; r < ng; ++r) s = cadd(s, src[r * np]);
      gout[i * nz + j] = s;
      if (i != j) gout[j * nz + i] = cconj(s);
    }
  }
  if (cl_size == 1) return;
  cl.sync();
  if (a.gram_part) {
    for (int e = crank + cl_size * tid; e < nz * nz; e += cl_size * nt) {
      float2 t[8];   // clusters hold at most 8 CTAs
#pragma unroll
      for (int r = 0; r < 8; ++r)
        t[r] = r < cl_size ? cl.map_shared_rank(gsm, r)[e] : make_float2(0.f, 0.f);
      float2 s = t[0];
#pragma unroll
      for (int r = 1; r < 8; ++r) s = cadd(s, t[r]);
      gp[e] = s;
    }
  }
  if (MODE == kDcUpdate && a.dc_part && kc > 1 && rank == 0 && tid < 32) {
    // lane r < kc reads CTA r's statistics; added in rank order
    const float* o = cl.map_shared_rank(stat, pl * kc + min(tid, kc - 1));
    const float r2 = o[0], d2 = o[1], o2 = o[2];
    float4 t = make_float4(r2, d2, o2, 0.f);
    for (int r = 1; r < kc; ++r) {
      t.x += __shfl_sync(0xffffffffu, r2, r);
      t.y += __shfl_sync(0xffffffffu, d2, r);
      t.z += __shfl_sync(0xffffffffu, o2, r);
    }
    if (tid == 0) reinterpret_cast<float4*>(a.dc_part)[x] = t;
  }
  cl.sync();   // no CTA leaves while another still reads its shared memory
}

// Launch of a kernel with the cluster shape of q (k_dc_rows.cu).
cudaError_t rows_launch(const void* kernel, const DcArgs& a, const RowLaunch& q, cudaStream_t st);

// Slice counts with compile-time planes, one translation unit each.
#define LPS_ROWS_NZ_LIST(X) X(8) X(10) X(12) X(14) X(16) X(20) X(24) X(28) X(32)
__host__ __device__ constexpr bool rows_fixed_nz(int nz) {
#define LPS_ROWS_NZ_IS(NZ) nz == NZ ||
  return LPS_ROWS_NZ_LIST(LPS_ROWS_NZ_IS) false;
#undef LPS_ROWS_NZ_IS
}

template <int MODE, int NY, int NZ>
__global__ void __launch_bounds__(row_threads(NY), row_fit(NY, NZ, false, false, 0))
    k_dc_rows_fixed(const DcArgs a, const RowLaunch q) {
  dc_rows_plane<MODE, NY, NZ>(a, q);
}

template <int MODE, int NY, int NZ>
cudaError_t launch_rows_fixed_mode(const DcArgs& a, const RowLaunch& q, cudaStream_t st) {
  static SmemLimit limit;
  const void* kernel = reinterpret_cast<const void*>(k_dc_rows_fixed<MODE, NY, NZ>);
  const cudaError_t e = limit.raise(kernel, 227 * 1024);
  return e != cudaSuccess ? e : rows_launch(kernel, a, q, st);
}

template <int NY, int NZ>
cudaError_t launch_rows_fixed(const DcArgs& a, int mode, const RowLaunch& q, cudaStream_t st) {
  switch (mode) {
    case kDcUpdate: return launch_rows_fixed_mode<kDcUpdate, NY, NZ>(a, q, st);
    case kDcAdjoint: return launch_rows_fixed_mode<kDcAdjoint, NY, NZ>(a, q, st);
    default: return launch_rows_fixed_mode<kDcForward, NY, NZ>(a, q, st);
  }
}

// Row lengths with compile-time planes: those of the benchmark workloads and of the uneven mix.
#define LPS_ROWS_NY_LIST(X) X(32) X(64) X(80) X(96) X(112) X(128) X(144) X(160) X(192)
__host__ __device__ constexpr bool rows_fixed_ny(int ny) {
#define LPS_ROWS_NY_IS(NY) ny == NY ||
  return LPS_ROWS_NY_LIST(LPS_ROWS_NY_IS) false;
#undef LPS_ROWS_NY_IS
}

template <int NZ>
cudaError_t launch_dc_rows_nz(const DcArgs& a, int mode, const RowLaunch& q, cudaStream_t st) {
#define LPS_ROWS_CASE(NY) \
  case NY: return launch_rows_fixed<NY, NZ>(a, mode, q, st);
  switch (a.g.ny) {
    LPS_ROWS_NY_LIST(LPS_ROWS_CASE)
    default: return cudaErrorNotSupported;
  }
#undef LPS_ROWS_CASE
}
#define LPS_ROWS_NZ_EXTERN(NZ) \
  extern template cudaError_t launch_dc_rows_nz<NZ>(const DcArgs&, int, const RowLaunch&, cudaStream_t);
LPS_ROWS_NZ_LIST(LPS_ROWS_NZ_EXTERN)
#undef LPS_ROWS_NZ_EXTERN

}  // namespace lps

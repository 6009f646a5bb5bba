// Float32 forms of the two contractions of the singular-value step (steps (1)-(2), Sec. 3) as
// stand-alone kernels: the Casorati Gram G = M^H M, M = X - S, and the reprojection L = M W. (Inside a
// frame the data-consistency kernels form both on the plane they hold.)
#include "lps_internal.cuh"

#include <algorithm>

namespace lps {

namespace {

constexpr int kGramThreads = 512;
constexpr int kGramRows = 256;   // voxels of a column that a CTA of k_gram_f32 holds at a time

}  // namespace

// Partials of the Gram, one per CTA: the CTA's chunks of 256 voxels of every column go through
// shared memory, and each thread keeps a 4 x 4 tile of entries (i, j), i <= j, over every ng-th voxel
// (ng = 512 threads / tiles); the ng sums are added in order at the end. Bound by the latency of one
// round of loads and by the 8 shared loads per 64 multiply-adds: 19 MB in 13 us at 192 x 192 x 32 (a
// thread per entry, all voxels of a plane in a row: 33 us).
__global__ void __launch_bounds__(kGramThreads) k_gram_f32(const float2* X, const float2* S, int nc, long long nr,
                                                           long long per, float2* gram_part) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int R = kGramRows, ms = R | 1;
  float2* M = reinterpret_cast<float2*>(smem);   // [nc][ms], in the end the partial sums [16][512]
  const int tid = threadIdx.x;
  const int n4 = (nc + 3) / 4, np = n4 * (n4 + 1) / 2, ng = kGramThreads / np;
  const int grp = tid / np, p = tid - grp * np;
  int ti = 0, rem = p;
  while (rem >= n4 - ti) {
    rem -= n4 - ti;
    ++ti;
  }
  const int tj = ti + rem;
  float2 s[4][4];
  int ri[4], rj[4];   // columns past the last repeat it (their entries are not used)
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    ri[i] = min(nc - 1, 4 * ti + i) * ms;
    rj[i] = min(nc - 1, 4 * tj + i) * ms;
#pragma unroll
    for (int j = 0; j < 4; ++j) s[i][j] = make_float2(0.f, 0.f);
  }
  const long long r0 = blockIdx.x * per, r1 = min(nr, r0 + per);
  constexpr int zstep = kGramThreads / R;
  const int yl = tid % R, zl = tid / R;
  pdl_trigger();
  pdl_wait();   // the images may come from the preceding kernel
  for (long long c0 = r0; c0 < r1; c0 += R) {
    const int rows = (int)min((long long)R, r1 - c0);
    __syncthreads();
    if (yl < rows) {
      constexpr int U = 16;   // every column of this thread: one round of loads
      float2 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int z = zl + u * zstep;
        v[u] = z < nc ? X[z * nr + c0 + yl] : make_float2(0.f, 0.f);
      }
      if (S) {
        float2 w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int z = zl + u * zstep;
          w[u] = z < nc ? S[z * nr + c0 + yl] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = csub(v[u], w[u]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (zl + u * zstep < nc) M[(zl + u * zstep) * ms + yl] = v[u];
    }
    __syncthreads();
    if (grp < ng) {
      for (int y = grp; y < rows; y += ng) {
        float2 u[4], v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          u[i] = M[ri[i] + y];
          v[i] = M[rj[i] + y];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            s[i][j].x = fmaf(u[i].x, v[j].x, fmaf(u[i].y, v[j].y, s[i][j].x));
            s[i][j].y = fmaf(u[i].x, v[j].y, fmaf(-u[i].y, v[j].x, s[i][j].y));
          }
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) M[(i * 4 + j) * kGramThreads + tid] = s[i][j];
  __syncthreads();
  float2* gp = gram_part + (long long)blockIdx.x * nc * nc;
  for (int e = tid; e < nc * nc; e += kGramThreads) {
    const int i = e / nc, j = e - i * nc;
    if (i > j) continue;
    const int bi = i >> 2, bj = j >> 2;
    const float2* src = M + ((i & 3) * 4 + (j & 3)) * kGramThreads + bi * n4 - bi * (bi - 1) / 2 + (bj - bi);
    float2 t = src[0];
    for (int r = 1; r < ng; ++r) t = cadd(t, src[r * np]);
    if (i == j) t.y = 0.f;   // exactly real diagonal
    gp[i * nc + j] = t;
    if (i != j) gp[j * nc + i] = cconj(t);
  }
}
static_assert(kGramThreads / kGramRows * 16 >= kMaxNc, "one round of loads covers the columns");

// G = sum of the nparts partials: a CTA takes 32 entries, warp w the partials w, w + 16, ..., and the
// sixteen sums are added in order. 192 partials of 32 x 32: 3.5 us (a thread per entry, all partials in
// a row: 21 us).
__global__ void __launch_bounds__(512) k_gram_sum(const float2* part, int nparts, int nn, float2* G) {
  __shared__ float2 sub[16][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
  pdl_trigger();
  pdl_wait();
  float2 s = make_float2(0.f, 0.f);
  if (e < nn) {
    constexpr int U = 12;
    for (int p0 = w; p0 < nparts; p0 += 16 * U) {
      float2 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        v[u] = p0 + 16 * u < nparts ? part[(long long)(p0 + 16 * u) * nn + e] : make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < U; ++u) s = cadd(s, v[u]);
    }
  }
  sub[w][lane] = s;
  __syncthreads();
  if (w == 0 && e < nn) {
#pragma unroll
    for (int q = 1; q < 16; ++q) s = cadd(s, sub[q][lane]);
    G[e] = s;
  }
}

// L[j][r] = sum_i (X - S)[i][r] W[i][j]. A CTA holds M of 4 PG voxels and W, as (x, y, -y, x), in shared
// memory; a thread forms 8 outputs of 4 voxels, a product being two packed multiply-adds: 12 shared
// loads (the 8 of W broadcast) per 64 of them. NG: groups of 8 outputs (nc <= 8 NG). Bound by the
// multiply-adds (4 nc a value) and by the shared loads of W, 16 bytes a lane, about alike: 28 MB in
// 14.6 us at 192 x 192 x 32 (a voxel a thread, W through the cache, scalar products: 74 us; a voxel a
// thread with W in shared memory: 20 us, 16 of them the broadcasts of W).
constexpr __host__ __device__ int reproj_pg(int ng) { return ng == 1 ? 256 : ng == 2 ? 128 : 64; }
template <int NG>
__global__ void __launch_bounds__(NG* reproj_pg(NG)) k_reproj_f32(const float2* X, const float2* S, const float2* W,
                                                                   float2* L, int nc, long long nr) {
  constexpr int PG = reproj_pg(NG), NT = NG * PG, NC = 8 * NG, P = 4 * PG;
  extern __shared__ __align__(16) unsigned char smem[];
  float4* W4 = reinterpret_cast<float4*>(smem);         // [NC][NC]
  float2* M = reinterpret_cast<float2*>(W4 + NC * NC);   // [NC][P]
  const int tid = threadIdx.x;
  const long long r0 = (long long)blockIdx.x * P;
  pdl_trigger();
  pdl_wait();   // the images and W may come from the preceding kernel
  for (int e = tid; e < NC * NC; e += NT) {
    const int i = e / NC, j = e % NC;
    const float2 w = i < nc && j < nc ? W[i * nc + j] : make_float2(0.f, 0.f);
    W4[e] = make_float4(w.x, w.y, -w.y, w.x);
  }
  // voxel tid, tid + NT, ... of each column, 8 columns a round
  for (int y = tid; y < P; y += NT) {
    const bool in = r0 + y < nr;
#pragma unroll 1
    for (int z0 = 0; z0 < NC; z0 += 8) {
      float2 v[8], w[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = in && z0 + u < nc ? X[(z0 + u) * nr + r0 + y] : make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 8; ++u) w[u] = S && in && z0 + u < nc ? S[(z0 + u) * nr + r0 + y] : make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 8; ++u) M[(z0 + u) * P + y] = csub(v[u], w[u]);
    }
  }
  __syncthreads();
  const int pg = tid % PG, j0 = tid / PG * 8;   // PG is a multiple of 32: a warp shares its outputs
  float2 o[4][8];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 8; ++j) o[k][j] = make_float2(0.f, 0.f);
#pragma unroll 2
  for (int i = 0; i < nc; ++i) {
    float2 m[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) m[k] = M[i * P + pg + PG * k];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float4 w = W4[i * NC + j0 + j];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        o[k][j] = fma2(make_float2(w.x, w.y), m[k].x, fma2(make_float2(w.z, w.w), m[k].y, o[k][j]));
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const long long r = r0 + pg + PG * k;
    if (r < nr) {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j0 + j < nc) L[(j0 + j) * nr + r] = o[k][j];
    }
  }
}

cudaError_t launch_gram_f32(const float2* X, const float2* S, const Geom& g, float2* gram_part, int nparts,
                            cudaStream_t st) {
  const long long nr = g.N / g.nc;
  if (nparts <= 0) return cudaErrorInvalidValue;
  const size_t smem = std::max((size_t)g.nc * (kGramRows | 1), (size_t)16 * kGramThreads) * sizeof(float2);
  static SmemLimit limit;
  cudaError_t e = limit.raise(reinterpret_cast<const void*>(k_gram_f32), smem);
  if (e != cudaSuccess) return e;
  e = launch_pdl(k_gram_f32, dim3(nparts), dim3(kGramThreads), smem, st, X, S, g.nc, nr,
                 (nr + nparts - 1) / nparts, gram_part);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_gram_sum(const float2* part, int nparts, int nc, float2* G, cudaStream_t st) {
  const int nn = nc * nc;
  const cudaError_t e = launch_pdl(k_gram_sum, dim3((nn + 31) / 32), dim3(512), 0, st, part, nparts, nn, G);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int NG>
static cudaError_t launch_reproj_ng(const float2* X, const float2* S, const float2* W, float2* L, const Geom& g,
                                    cudaStream_t st) {
  const long long nr = g.N / g.nc;
  constexpr int P = 4 * reproj_pg(NG), NC = 8 * NG;
  constexpr size_t smem = NC * NC * sizeof(float4) + (size_t)NC * P * sizeof(float2);
  static SmemLimit limit;
  cudaError_t e = limit.raise(reinterpret_cast<const void*>(k_reproj_f32<NG>), smem);
  if (e != cudaSuccess) return e;
  e = launch_pdl(k_reproj_f32<NG>, dim3((unsigned)((nr + P - 1) / P)), dim3(NG * reproj_pg(NG)), smem, st, X, S, W, L,
                 g.nc, nr);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_reproj_f32(const float2* X, const float2* S, const float2* W, float2* L, const Geom& g,
                              cudaStream_t st) {
  switch ((g.nc + 7) / 8) {
    case 1: return launch_reproj_ng<1>(X, S, W, L, g, st);
    case 2: return launch_reproj_ng<2>(X, S, W, L, g, st);
    case 3: return launch_reproj_ng<3>(X, S, W, L, g, st);
    default: return launch_reproj_ng<4>(X, S, W, L, g, st);
  }
}

}  // namespace lps

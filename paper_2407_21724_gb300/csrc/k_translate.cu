// FP32 translation of one right-hand side (Eqs. 22-23):
//   in[b][k] = sum over (b', o) in the interaction list of b of T[o][k] out[b'][k].
//
// A thread owns one direction (its two fields, 16 bytes) for a tile of
// 4x4 target boxes (2x2 parents), whose sources lie in the 8x8 window around
// it: it reads each source once, row by row of the window, and adds it to all
// targets that list it, with the seven translation factors of the row pair in
// registers.  64 loads and about 170 shared-memory reads of factors then serve
// 432 complex multiply-adds of two fields, which are the bound: FP32 issue, 60 %
// busy, the rest waits for the sources (13 GFLOP over the levels of the 200x200
// lens, 0.17 ms at the measured FP32 peak; seven levels 503 us, level 0 131 us).
// With four fields a direction it took 850 us (level 0 229), a kernel that staged a
// 12x12 window and the factors for 8x8 targets in shared memory and read one factor
// per multiply-add from there 1057 (282) us.  Loading the next window row ahead takes 163 registers and
// loses more to the fourth CTA per SM than it hides (1028 against 847 us).  A CTA
// keeps its chunk of 64 directions and their factors and walks over tiles, one
// for each half of its threads (one tile at a time for 64 threads: 526 us, and the
// small levels of a 40x40 array 16 to 22 us each instead of 12 to 18: the factors are
// loaded by half as many threads).
#include <algorithm>

#include "smr_internal.h"

namespace smr {

namespace {

constexpr int TRL_THREADS = 128, TRL_DIRS = TRL_THREADS / 2;

__device__ __forceinline__ void cmadd(float4& a, float2 t, const float4& v) {
  a.x = fmaf(t.x, v.x, a.x); a.x = fmaf(-t.y, v.y, a.x);
  a.y = fmaf(t.x, v.y, a.y); a.y = fmaf(t.y, v.x, a.y);
  a.z = fmaf(t.x, v.z, a.z); a.z = fmaf(-t.y, v.w, a.z);
  a.w = fmaf(t.x, v.w, a.w); a.w = fmaf(t.y, v.z, a.w);
}

// One target row against one source row of the window: t[dx + 3], NEAR: the
// rows are at most one apart, so boxes at most one apart are neighbours.
template <int P, bool NEAR>
__device__ __forceinline__ void row_pair(float4* acc, const float2* t, const float4* v) {
#pragma unroll
  for (int tx = 0; tx < 2 * P; ++tx)
#pragma unroll
    for (int sx = (tx & 2); sx < (tx & 2) + 6; ++sx) {
      const int dx = tx + 2 - sx;
      if (NEAR && dx >= -1 && dx <= 1) continue;
      cmadd(acc[tx], t[dx + 3], v[sx]);
    }
}

// tab[tile][80]: the 8x8 window's source boxes (row by row, -1 if absent), then
// the 4x4 target boxes.  Tt[49][K]: factors by offset (dx + 3) * 7 + dy + 3.
// The offsets lie in the plane, so a factor is the same at theta and pi - theta:
// only the upper half of the table is read.  P parents per side: 2, the whole
// tile, or 1, one parent of the tile per half CTA and blockIdx.z (2x2 targets, a
// 6x6 window).
template <int P>
__global__ void __launch_bounds__(TRL_THREADS, 4) k_translate_tile(int K, int nth, int nph, int ntile,
                                                                   const int* __restrict__ tab,
                                                                   const float2* __restrict__ Tt,
                                                                   const float4* __restrict__ out,
                                                                   float4* __restrict__ in) {
  constexpr int NT = 2 * P, NW = NT + 4;        // targets and window boxes per side
  __shared__ float2 Ts[49][TRL_DIRS];
  const int k0 = blockIdx.x * TRL_DIRS, kl = threadIdx.x & (TRL_DIRS - 1), half = threadIdx.x / TRL_DIRS;
  // all lanes stay for the exchange of box ids; those past the last direction
  // repeat its part and store nothing
  const bool ok = k0 + kl < K;
  const unsigned stride = K;                    // directions of a box
  const unsigned u = ok ? k0 + kl : K - 1;
  const float4* src = out + u;
  float4* dst = in + u;
  const int ox = P == 2 ? 0 : 2 * half, oy = P == 2 ? 0 : 2 * blockIdx.z;
  // a tile's 80 ids over the warp's lanes, the next tile's on their way
  const int lane = threadIdx.x & 31;
  int n0 = -1, n1 = -1, n2 = -1;
  auto fetch = [&](int tile) {
    if (tile < ntile) {
      const int* id = tab + (size_t)tile * 80 + lane;
      n0 = __ldg(id);
      n1 = __ldg(id + 32);
      if (lane < 16) n2 = __ldg(id + 64);
    }
  };
  const int first = P == 2 ? 2 * blockIdx.y + half : blockIdx.y, step = P == 2 ? 2 * gridDim.y : gridDim.y;
  fetch(first);
  {
    const int d = threadIdx.x & (TRL_DIRS - 1), k = min(k0 + d, K - 1);
    const int i = k / nph, kk = min(i, nth - 1 - i) * nph + (k - i * nph);
    constexpr unsigned long long NEIGHBOURS = 0x7ull << 16 | 0x7ull << 23 | 0x7ull << 30;   // never read
#pragma unroll 5
    for (int o = threadIdx.x / TRL_DIRS; o < 49; o += TRL_THREADS / TRL_DIRS)
      if (!(NEIGHBOURS >> o & 1u)) Ts[o][d] = __ldg(Tt + (size_t)o * K + kk);
  }
  __syncthreads();
  for (int tile = first; tile < ntile; tile += step) {
    const int i0 = n0, i1 = n1, i2 = n2;
    const unsigned m0 = __ballot_sync(0xffffffffu, i0 >= 0), m1 = __ballot_sync(0xffffffffu, i1 >= 0);
    fetch(tile + step);
    float4 acc[NT][NT];
#pragma unroll
    for (int y = 0; y < NT; ++y)
#pragma unroll
      for (int x = 0; x < NT; ++x) acc[y][x] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int sy = 0; sy < NW; ++sy) {
      constexpr unsigned ALL = (1u << NW) - 1;
      const int wy = sy + oy, w0 = 8 * (wy & 3) + ox;
      const unsigned have = (wy < 4 ? m0 : m1) >> w0 & ALL;
      if (have == 0) continue;                  // no source in this row
      float4 v[NW];
      const int is = wy < 4 ? i0 : i1;
#pragma unroll
      for (int x = 0; x < NW; ++x) {
        const int n = __shfl_sync(0xffffffffu, is, w0 + x);
        if (have == ALL) v[x] = __ldg(src + (size_t)((unsigned)n) * stride);
        else v[x] = n >= 0 ? __ldg(src + (size_t)((unsigned)n) * stride) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int ty = 0; ty < NT; ++ty) {
        // sources of ty's parent row: window rows (ty & 2) .. (ty & 2) + 5
        if (sy >= (ty & 2) && sy < (ty & 2) + 6) {
          const int dy = ty + 2 - sy;
          float2 t[7];
#pragma unroll
          for (int x = 0; x < 7; ++x) t[x] = Ts[7 * x + dy + 3][kl];
          if (dy >= -1 && dy <= 1) row_pair<P, true>(acc[ty], t, v);
          else row_pair<P, false>(acc[ty], t, v);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < NT * NT; ++q) {
      const int n = __shfl_sync(0xffffffffu, i2, 4 * (q / NT + oy) + q % NT + ox);
      if (ok && n >= 0) dst[(size_t)((unsigned)n) * stride] = acc[q / NT][q % NT];
    }
  }
}

}  // namespace

// Source and target boxes of the level's non-empty 4x4 tiles
int build_translate_tiles(Ctx* c, Level& L, const std::vector<int>& tiles, const std::vector<int>& boxmap) {
  std::vector<int> tab(tiles.size() * 80, -1);
  auto box = [&](int x, int y) {
    x -= L.map_x0;
    y -= L.map_y0;
    return x >= 0 && y >= 0 && x < L.map_w && y < L.map_h ? boxmap[(size_t)y * L.map_w + x] : -1;
  };
  for (size_t t = 0; t < tiles.size(); ++t) {
    const int x0 = ((L.map_x0 >> 2) + tiles[t] % L.ntile_x) * 4, y0 = ((L.map_y0 >> 2) + tiles[t] / L.ntile_x) * 4;
    for (int s = 0; s < 64; ++s) tab[t * 80 + s] = box(x0 - 2 + (s & 7), y0 - 2 + (s >> 3));
    for (int s = 0; s < 16; ++s) tab[t * 80 + 64 + s] = box(x0 + (s & 3), y0 + (s >> 2));
  }
  return upload(c, &L.d_tile_tab, tab);
}

int run_translate_tiles(Ctx* c, int s, cudaStream_t st) {
  const Level& L = c->lev[s];
  const int nk = (L.K + TRL_DIRS - 1) / TRL_DIRS;
  if (nk * L.ntile_ne <= 152) {
    // too few tiles to fill the SMs: one parent per half CTA, a shorter chain of
    // rows (24x24 array: four levels 59 us by whole tiles, 47 by parents;
    // with up to 304, 40x40 levels 1 and 2 16 against 14 us alone, but the product,
    // where they run beside the interpolation, 208 against 210)
    k_translate_tile<1><<<dim3(nk, L.ntile_ne, 2), TRL_THREADS, 0, st>>>(
        L.K, L.nth, L.nph, L.ntile_ne, L.d_tile_tab, L.d_T32, (const float4*)L.d_out, (float4*)L.d_in);
    SMR_LAUNCH(c);
    return SMR_OK;
  }
  // CTAs along the tiles: the number that finishes first with four CTAs per SM
  // at a time, staging the factors costing about 0.7 of a tile
  int ny = 1;
  double best = 1e30;
  const int pairs = (L.ntile_ne + 1) / 2;
  for (int y = 1; y <= pairs && (y == 1 || (long long)y * nk <= 16 * 152); ++y) {
    const double cost = ((nk * (long long)y + 607) / 608) * (0.7 + (pairs + y - 1) / y);
    if (cost <= best) {
      best = cost;
      ny = y;
    }
  }
  k_translate_tile<2><<<dim3(nk, ny), TRL_THREADS, 0, st>>>(L.K, L.nth, L.nph, L.ntile_ne, L.d_tile_tab, L.d_T32,
                                                           (const float4*)L.d_out, (float4*)L.d_in);
  SMR_LAUNCH(c);
  return SMR_OK;
}

}  // namespace smr

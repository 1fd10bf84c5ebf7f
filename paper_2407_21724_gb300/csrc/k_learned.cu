// Learned initial guess for the GMRES solve: per-scatterer features, a 4-layer
// MLP (BF16 weights, FP32 activations and accumulation, FP32 Adam master
// weights) trained on solutions of the plain solver, and the re-phasing that
// turns its output into coefficients.
//
// Features of particle mu (F = 448):
//   for each of the 48 lattice neighbours within 2 wavelengths (0 < dx^2+dy^2 <= 16
//   cells at pitch 0.5, fixed order by distance then angle): one-hot shape (8)
//   and presence (1); own shape one-hot (8); incidence direction (3) and the
//   real polarisation vector (3); 2 zeros of padding.
// Output (O = 4 n_psi): real and imaginary parts of the de-phased coefficients
//   abar_mu = alpha_mu exp(+j k khat . r_mu) / scale, [Re(e,m modes) | Im(e,m modes)].
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "smr_internal.h"

namespace smr {

namespace {

constexpr int kSlots = 48;
constexpr int kShapesMax = 8;

__device__ __forceinline__ float silu(float z) { return z / (1.f + __expf(-z)); }
__device__ __forceinline__ float dsilu(float z) {
  float s = 1.f / (1.f + __expf(-z));
  return s * (1.f + z * (1.f - s));
}
// ------------------------------------------------------------------ GEMMs
// C tile of 64 x 64 per CTA, 256 threads of 4 x 4 results each, K in steps of 32
// through two shared-memory buffers (the next step's values are loaded into
// registers while this one is multiplied).  FP32 multiply-adds: a split-TF32
// mma.sync version took 288 us a batch (below) against 323, but its one accumulator a
// result rounds toward zero, which over a batch's rows put the gradient 6.3e-6 off,
// against 1.7e-7; several accumulators, as in k_tc.cu, were not tried.
// Bound: the grids are small (4,096 rows at width 256 make 256 such tiles), so
// few warps per scheduler hide the shared-memory latency of two reads per 16
// multiply-adds.  A 4096 x 256 x 256 layer takes 27 us; 8 x 4 results per
// thread and half the threads 38 us, 8 x 8 (128 tiles of 128 x 64) 45 us.  A
// batch (4,096 rows, width 256, loss and gradient to the host): 2.68 -> 0.32 ms,
// against no prefetch, one CTA per tile of the weight gradients (28 CTAs) and
// serial column and loss sums.
constexpr int GT = 64, GK = 32, GTHREADS = 256, GP = GT + 4;

// A tile's loader: 64 (rows of the tile) x 32 (k), 8 values per thread in two
// runs of four.  KC: k is the contiguous index of the matrix, a run is (row
// q / 8, k 4 (q % 8)); else the tile's row is, a run is (k q / 16, rows
// 4 (q % 16)).  V4: rows are 16-byte (BF16: 8-byte) aligned and a multiple of
// four long.
template <typename T, bool KC, bool V4>
struct TileLoad {
  const T* p[2];                               // KC: the run's row; else its column in row 0
  const int* idx;                              // gathered rows (not KC)
  int ld, left[2];                             // KC: -1 where the row is outside; else values in the row
  float v[8];
  __device__ __forceinline__ TileLoad(const T* src, const int* gather, int ld_, int nrow, int row0)
      : idx(gather), ld(ld_) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int q = threadIdx.x + u * GTHREADS, r = row0 + (KC ? q >> 3 : 4 * (q & 15));
      left[u] = KC ? (r < nrow ? 4 : -1) : nrow - r;
      p[u] = KC ? src + (size_t)(r < nrow ? (gather ? gather[r] : r) : 0) * ld + 4 * (q & 7) : src + r;
    }
  }
  static __device__ __forceinline__ float one(const float* a) { return *a; }
  static __device__ __forceinline__ float one(const __nv_bfloat16* a) { return __bfloat162float(*a); }
  // four values from a, of which n exist
  static __device__ __forceinline__ void run(const T* a, int n, float* o) {
    if (V4 && n >= 4) {
      if constexpr (sizeof(T) == 4) {
        const float4 x = *reinterpret_cast<const float4*>(a);
        o[0] = x.x; o[1] = x.y; o[2] = x.z; o[3] = x.w;
      } else {
        const uint2 x = *reinterpret_cast<const uint2*>(a);
        o[0] = __uint_as_float(x.x << 16); o[1] = __uint_as_float(x.x & 0xffff0000u);
        o[2] = __uint_as_float(x.y << 16); o[3] = __uint_as_float(x.y & 0xffff0000u);
      }
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = e < n ? one(a + e) : 0.f;
    }
  }
  __device__ __forceinline__ void load(int k0, int k1) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int q = threadIdx.x + u * GTHREADS;
      if (KC) {
        run(p[u] + k0, left[u] < 0 ? 0 : k1 - k0 - 4 * (q & 7), v + 4 * u);
      } else {
        const int k = k0 + (q >> 4);
        const bool in = k < k1;
        run(p[u] + (size_t)(in ? (idx ? idx[k] : k) : 0) * ld, in ? left[u] : 0, v + 4 * u);
      }
    }
  }
  __device__ __forceinline__ void store(float (*S)[GP]) const {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int q = threadIdx.x + u * GTHREADS;
      if (KC) {
#pragma unroll
        for (int e = 0; e < 4; ++e) S[4 * (q & 7) + e][q >> 3] = v[4 * u + e];
      } else {
        *reinterpret_cast<float4*>(&S[q >> 4][4 * (q & 15)]) =
            make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
      }
    }
  }
};

typedef float TileS[GK][GP];

// This thread's 4 x 4 results: rows 4 (thread / 16) + i, columns 4 (thread % 16) + j
struct Tile {
  float2 d[4][2];
  // f(row, column, value) for every result
  template <typename Fn> __device__ __forceinline__ void each(Fn f) const {
    const int r = threadIdx.x >> 4 << 2, c = (threadIdx.x & 15) << 2;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        f(r + i, c + 2 * j, d[i][j].x);
        f(r + i, c + 2 * j + 1, d[i][j].y);
      }
  }
};

// C += A B over k in [k0, k1); with colsum, db += the sums over k of B's
// column threadIdx.x
template <typename LA, typename LB>
__device__ __forceinline__ void tile_mma(LA& a, LB& b, int k0, int k1, TileS* As, TileS* Bs, Tile& c, bool colsum,
                                         float* db) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  a.load(k0, k1);
  b.load(k0, k1);
  int buf = 0;
  for (int k = k0; k < k1; k += GK, buf ^= 1) {
    a.store(As[buf]);
    b.store(Bs[buf]);
    __syncthreads();
    if (k + GK < k1) {
      a.load(k + GK, k1);
      b.load(k + GK, k1);
    }
#pragma unroll
    for (int q = 0; q < GK; ++q) {
      const float4 x = *reinterpret_cast<const float4*>(&As[buf][q][4 * ty]);
      const float4 y = *reinterpret_cast<const float4*>(&Bs[buf][q][4 * tx]);
      const float2 y0 = make_float2(y.x, y.y), y1 = make_float2(y.z, y.w);
      const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 xx = make_float2(xs[i], xs[i]);
        c.d[i][0] = __ffma2_rn(xx, y0, c.d[i][0]);
        c.d[i][1] = __ffma2_rn(xx, y1, c.d[i][1]);
      }
    }
    if (colsum && threadIdx.x < GT) {
#pragma unroll
      for (int q = 0; q < GK; ++q) *db += Bs[buf][q][threadIdx.x];
    }
  }
}

// Forward layer: Z = A W + b, and A' = silu(Z) (act), or for the last layer
// with targets dZ = 2 (Z - T) / (n O) and the CTA's sum of (Z - T)^2.
template <bool V4>
__global__ void __launch_bounds__(GTHREADS) k_fwd(int n, int N, int K, const float* __restrict__ A,
                                                  const int* __restrict__ aidx, const __nv_bfloat16* __restrict__ W,
                                                  const float* __restrict__ bias, float* __restrict__ Z,
                                                  float* __restrict__ act, const float* __restrict__ T,
                                                  const int* __restrict__ tidx, float* __restrict__ dZ,
                                                  double* __restrict__ part) {
  __shared__ __align__(16) TileS As[2], Bs[2];
  __shared__ double red[GTHREADS];
  const int m0 = blockIdx.y * GT, n0 = blockIdx.x * GT;
  TileLoad<float, true, V4> a(A, aidx, K, n, m0);
  TileLoad<__nv_bfloat16, false, V4> b(W, nullptr, N, N, n0);
  Tile acc = {};
  tile_mma(a, b, 0, K, As, Bs, acc, false, nullptr);
  double e2 = 0.0;
  const float scale = (float)n * (float)N;
  acc.each([&](int i, int j, float v) {
    const int m = m0 + i, c = n0 + j;
    if (m >= n || c >= N) return;
    const float z = v + bias[c];
    Z[(size_t)m * N + c] = z;
    if (act) act[(size_t)m * N + c] = silu(z);
    if (T) {
      const float d = z - T[(size_t)(tidx ? tidx[m] : m) * N + c];
      dZ[(size_t)m * N + c] = 2.f * d / scale;
      e2 += (double)d * d;
    }
  });
  if (!T) return;
  red[threadIdx.x] = e2;
  __syncthreads();
  for (int h = GTHREADS / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.y * gridDim.x + blockIdx.x] = red[0];
}

// dZ_{l-1} = (dZ_l W_l^T) silu'(Z_{l-1});  dZ_l [n][K], W_l [N][K]
template <bool V4>
__global__ void __launch_bounds__(GTHREADS) k_dx(int n, int N, int K, const float* __restrict__ dZl,
                                                 const __nv_bfloat16* __restrict__ W, const float* __restrict__ Z,
                                                 float* __restrict__ out) {
  __shared__ __align__(16) TileS As[2], Bs[2];
  const int m0 = blockIdx.y * GT, n0 = blockIdx.x * GT;
  TileLoad<float, true, V4> a(dZl, nullptr, K, n, m0);
  TileLoad<__nv_bfloat16, true, V4> b(W, nullptr, K, N, n0);
  Tile acc = {};
  tile_mma(a, b, 0, K, As, Bs, acc, false, nullptr);
  acc.each([&](int i, int j, float v) {
    const int m = m0 + i, c = n0 + j;
    if (m < n && c < N) out[(size_t)m * N + c] = v * dsilu(Z[(size_t)m * N + c]);
  });
}

// Weight gradients of all layers in one launch: dW_l = A_l^T dZ_l and db_l =
// the column sums of dZ_l over the rows of split blockIdx.y, into that split's
// copy of the parameter layout.  Tiles t0[l] .. t0[l + 1] belong to layer l.
struct GradArgs {
  const float* A[4];
  const float* dZ[4];
  const int* idx;                              // rows of layer 0's input
  int in[4], out[4], t0[5];
  long long off[4], np;
};
template <bool V4>
__global__ void __launch_bounds__(GTHREADS) k_dw(GradArgs g, int n, int rows, float* __restrict__ part) {
  __shared__ __align__(16) TileS As[2], Bs[2];
  int l = 0;
  while (l < 3 && (int)blockIdx.x >= g.t0[l + 1]) ++l;
  const int t = blockIdx.x - g.t0[l], M = g.in[l], N = g.out[l], nx = (N + GT - 1) / GT;
  const int m0 = t / nx * GT, n0 = t % nx * GT;
  const int k0 = blockIdx.y * rows, k1 = min(n, k0 + rows);
  TileLoad<float, false, V4> a(g.A[l], l == 0 ? g.idx : nullptr, M, M, m0);
  TileLoad<float, false, V4> b(g.dZ[l], nullptr, N, N, n0);
  Tile acc = {};
  float db = 0.f;
  if (k0 < k1) tile_mma(a, b, k0, k1, As, Bs, acc, m0 == 0, &db);
  float* o = part + (size_t)blockIdx.y * g.np + g.off[l];
  acc.each([&](int i, int j, float v) {
    const int m = m0 + i, c = n0 + j;
    if (m < M && c < N) o[(size_t)m * N + c] = v;
  });
  if (m0 == 0 && threadIdx.x < GT && n0 + threadIdx.x < N) o[(size_t)M * N + n0 + threadIdx.x] = db;
}

// gradient = sum of the splits, in split order
__global__ void k_split_sum(long long np, int S, const float* __restrict__ part, float* __restrict__ g) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= np) return;
  float s = part[i];
  for (int q = 1; q < S; ++q) s += part[(size_t)q * np + i];
  g[i] = s;
}

// loss = scale x the sum of the partial sums (one CTA of 256)
__global__ void k_sum(int n, const double* __restrict__ part, double scale, double* __restrict__ out) {
  __shared__ double red[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) s += part[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0] * scale;
}

__global__ void k_adam(long long n, float* __restrict__ p, __nv_bfloat16* __restrict__ w16,
                       const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v, float lr,
                       float b1, float b2, float eps, float bc1, float bc2) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= n) return;
  float gt = g[t];
  float mt = b1 * m[t] + (1.f - b1) * gt;
  float vt = b2 * v[t] + (1.f - b2) * gt * gt;
  m[t] = mt;
  v[t] = vt;
  float pt = p[t] - lr * (mt / bc1) / (sqrtf(vt / bc2) + eps);
  p[t] = pt;
  w16[t] = __float2bfloat16(pt);
}

__global__ void k_to_bf16(long long n, const float* __restrict__ p, __nv_bfloat16* __restrict__ w16) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t < n) w16[t] = __float2bfloat16(p[t]);
}

// features, one thread per particle
__global__ void k_features(int p, int F, const int* __restrict__ sid, const int* __restrict__ arr,
                           const int* __restrict__ pi, const int* __restrict__ pj, int map_x0, int map_y0,
                           int map_w, int map_h, const int* __restrict__ boxmap, const int* __restrict__ slots,
                           const double* __restrict__ khat, const double* __restrict__ pol,
                           float* __restrict__ feat) {
  int mu = blockIdx.x * blockDim.x + threadIdx.x;
  if (mu >= p) return;
  float* f = feat + (size_t)mu * F;
  for (int i = 0; i < F; ++i) f[i] = 0.f;
  for (int s = 0; s < kSlots; ++s) {
    int x = pi[mu] + slots[2 * s] - map_x0, y = pj[mu] + slots[2 * s + 1] - map_y0;
    if (x < 0 || y < 0 || x >= map_w || y >= map_h) continue;
    int nu = boxmap[y * map_w + x];
    if (nu < 0) continue;
    f[s * 9 + sid[nu]] = 1.f;
    f[s * 9 + 8] = 1.f;
  }
  f[kSlots * 9 + sid[mu]] = 1.f;
  int a = arr[mu];
  for (int d = 0; d < 3; ++d) {
    f[kSlots * 9 + 8 + d] = (float)khat[3 * a + d];
    f[kSlots * 9 + 11 + d] = (float)pol[6 * a + 2 * d];
  }
}

// targets: de-phased coefficients / scale
__global__ void k_targets(int p, int npsi, const int* __restrict__ arr, const double* __restrict__ cen,
                          const double* __restrict__ khat, const double2* __restrict__ x, double kw,
                          double inv_scale, float* __restrict__ tgt) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  int n2 = 2 * npsi;
  if (t >= (long long)p * n2) return;
  int mu = (int)(t / n2), i = (int)(t % n2);
  const double* kh = khat + 3 * arr[mu];
  const double* r = cen + 3 * mu;
  double sn, cs;
  sincos(kw * (kh[0] * r[0] + kh[1] * r[1] + kh[2] * r[2]), &sn, &cs);
  double2 v = x[(size_t)mu * n2 + i];
  tgt[(size_t)mu * 2 * n2 + i] = (float)((v.x * cs - v.y * sn) * inv_scale);
  tgt[(size_t)mu * 2 * n2 + n2 + i] = (float)((v.x * sn + v.y * cs) * inv_scale);
}

// re-phase the network output into coefficients x0
__global__ void k_rephase(int p, int npsi, int row0, int rows, const int* __restrict__ arr,
                          const double* __restrict__ cen, const double* __restrict__ khat,
                          const float* __restrict__ Y, double kw, double scale, double2* __restrict__ x0) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  int n2 = 2 * npsi;
  if (t >= (long long)rows * n2) return;
  int m = (int)(t / n2), i = (int)(t % n2);
  int mu = row0 + m;
  const double* kh = khat + 3 * arr[mu];
  const double* r = cen + 3 * mu;
  double sn, cs;
  sincos(-kw * (kh[0] * r[0] + kh[1] * r[1] + kh[2] * r[2]), &sn, &cs);
  double re = scale * Y[(size_t)m * 2 * n2 + i], im = scale * Y[(size_t)m * 2 * n2 + n2 + i];
  x0[(size_t)mu * n2 + i] = make_double2(re * cs - im * sn, re * sn + im * cs);
}

uint64_t splitmix(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ULL);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

long long woff(const NN& nn, int l) {
  long long o = 0;
  for (int q = 0; q < l; ++q) o += (long long)nn.dims[q] * nn.dims[q + 1] + nn.dims[q + 1];
  return o;
}

}  // namespace

void nn_free(Ctx* c) {
  NN& nn = c->nn;
  cudaFree(nn.p32); cudaFree(nn.w16); cudaFree(nn.m); cudaFree(nn.v); cudaFree(nn.g);
  cudaFree(nn.act); cudaFree(nn.dact); cudaFree(nn.part); cudaFree(nn.d_loss); cudaFree(nn.d_slots);
  nn = NN();
}

int nn_init(Ctx* c, int width, unsigned long long seed) {
  if (c->npsi <= 0) { c->err = "set the scene before smr_nn_init (output size is 4 n_psi)"; return SMR_E_STATE; }
  if (width < 1 || width > 4096) { c->err = "width must be in 1..4096"; return SMR_E_INVALID_ARG; }
  nn_free(c);
  NN& nn = c->nn;
  nn.H = width;
  nn.O = 4 * c->npsi;
  int dims[5] = {nn.F, width, width, width, nn.O};
  for (int i = 0; i < 5; ++i) nn.dims[i] = dims[i];
  nn.np = woff(nn, 4);
  std::vector<float> p((size_t)nn.np, 0.f);
  uint64_t s = seed;
  for (int l = 0; l < 4; ++l) {
    long long o = woff(nn, l);
    double a = std::sqrt(6.0 / (nn.dims[l] + nn.dims[l + 1]));
    for (long long i = 0; i < (long long)nn.dims[l] * nn.dims[l + 1]; ++i) {
      double u = (double)(splitmix(s) >> 11) * (1.0 / 9007199254740992.0);
      p[o + i] = (float)((2.0 * u - 1.0) * a);
    }
  }
  nn.cap = 8192;
  size_t abytes = (size_t)nn.cap * (6 * (size_t)width + nn.O) * sizeof(float);
  SMR_CUDA(c, cudaMalloc((void**)&nn.p32, nn.np * sizeof(float)));
  SMR_CUDA(c, cudaMalloc((void**)&nn.w16, nn.np * sizeof(__nv_bfloat16)));
  SMR_CUDA(c, cudaMalloc((void**)&nn.m, nn.np * sizeof(float)));
  SMR_CUDA(c, cudaMalloc((void**)&nn.v, nn.np * sizeof(float)));
  SMR_CUDA(c, cudaMalloc((void**)&nn.g, nn.np * sizeof(float)));
  SMR_CUDA(c, cudaMalloc((void**)&nn.act, abytes));
  SMR_CUDA(c, cudaMalloc((void**)&nn.dact, (size_t)nn.cap * (3 * (size_t)width + nn.O) * sizeof(float)));
  SMR_CUDA(c, cudaMalloc((void**)&nn.d_loss, ((size_t)(nn.cap / GT) * ((nn.O + GT - 1) / GT) + 1) * sizeof(double)));
  SMR_CUDA(c, cudaMemcpy(nn.p32, p.data(), nn.np * sizeof(float), cudaMemcpyHostToDevice));
  SMR_CUDA(c, cudaMemset(nn.m, 0, nn.np * sizeof(float)));
  SMR_CUDA(c, cudaMemset(nn.v, 0, nn.np * sizeof(float)));
  k_to_bf16<<<(unsigned)((nn.np + 255) / 256), 256>>>(nn.np, nn.p32, nn.w16);
  SMR_LAUNCH(c);
  // neighbour slots within 2 wavelengths, by distance then angle
  std::vector<std::pair<std::pair<int, double>, std::pair<int, int>>> sl;
  for (int dy = -4; dy <= 4; ++dy)
    for (int dx = -4; dx <= 4; ++dx) {
      int d2 = dx * dx + dy * dy;
      if (d2 == 0 || d2 > 16) continue;
      sl.push_back({{d2, std::atan2((double)dy, (double)dx)}, {dx, dy}});
    }
  std::sort(sl.begin(), sl.end());
  std::vector<int> slots;
  for (auto& e : sl) { slots.push_back(e.second.first); slots.push_back(e.second.second); }
  int rc = upload(c, &nn.d_slots, slots);
  if (rc) return rc;
  SMR_CUDA(c, cudaDeviceSynchronize());
  return SMR_OK;
}

int nn_features(Ctx* c, const double* d_khat, const double* d_pol, float* feat, cudaStream_t st) {
  if (!c->nn.p32) { c->err = "call smr_nn_init first"; return SMR_E_STATE; }
  if (c->S > kShapesMax) { c->err = "learned features support at most 8 shapes"; return SMR_E_INVALID_ARG; }
  if (c->multi) { c->err = "learned features need at most one particle per lattice cell"; return SMR_E_INVALID_ARG; }
  Level& L0 = c->lev[0];
  // lattice indices of particles (level-0 boxes are the particles)
  int* d_pi = nullptr;
  int* d_pj = nullptr;
  int rc;
  if ((rc = upload(c, &d_pi, c->pi)) || (rc = upload(c, &d_pj, c->pj))) return rc;
  k_features<<<(c->p + 127) / 128, 128, 0, st>>>(c->p, c->nn.F, c->d_sid, c->d_arr, d_pi, d_pj, L0.map_x0,
                                                  L0.map_y0, L0.map_w, L0.map_h, L0.d_boxmap, c->nn.d_slots,
                                                  d_khat, d_pol, feat);
  SMR_LAUNCH(c);
  SMR_CUDA(c, cudaStreamSynchronize(st));
  cudaFree(d_pi);
  cudaFree(d_pj);
  return SMR_OK;
}

int nn_targets(Ctx* c, const double* d_khat, const double2* x, double scale, float* tgt, cudaStream_t st) {
  long long n = (long long)c->p * 2 * c->npsi;
  k_targets<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(c->p, c->npsi, c->d_arr, c->d_centres, d_khat, x, c->k,
                                                         1.0 / scale, tgt);
  SMR_LAUNCH(c);
  return SMR_OK;
}

// Forward (and backward into nn.g) over n rows of feat (rows idx[] if given).
int nn_forward_backward(Ctx* c, int n, const float* feat, const int* idx, const float* tgt, bool backward,
                        double* loss_host, cudaStream_t st) {
  NN& nn = c->nn;
  if (!nn.p32) { c->err = "call smr_nn_init first"; return SMR_E_STATE; }
  if (n < 1 || n > nn.cap) { c->err = "batch must be 1..8192 rows"; return SMR_E_INVALID_ARG; }
  const int H = nn.H, O = nn.O;
  // buffers: pre-activations Z and activations A of the three hidden layers,
  // the output, and the gradients with respect to the pre-activations
  float *Z[4], *A[4] = {nullptr, nullptr, nullptr, nullptr}, *dZ[4];
  for (int l = 0; l < 3; ++l) {
    Z[l] = nn.act + (size_t)(2 * l) * nn.cap * H;
    A[l] = nn.act + (size_t)(2 * l + 1) * nn.cap * H;
    dZ[l] = nn.dact + (size_t)nn.cap * O + (size_t)l * nn.cap * H;
  }
  Z[3] = nn.act + (size_t)6 * nn.cap * H;
  dZ[3] = nn.dact;
  // 16-byte loads where every row of every operand is aligned for them
  const bool v4 = nn.F % 4 == 0 && H % 4 == 0 && O % 4 == 0 && ((uintptr_t)feat & 15) == 0;
  const int my = (n + GT - 1) / GT;
  int nb = 0;
  for (int l = 0; l < 4; ++l) {
    const int in = nn.dims[l], out = nn.dims[l + 1];
    const __nv_bfloat16* W = nn.w16 + woff(nn, l);
    const float* b = nn.p32 + woff(nn, l) + (long long)in * out;
    const dim3 g((out + GT - 1) / GT, my);
    const bool last = l == 3;
    if (last) nb = (int)(g.x * g.y);
    auto k = v4 ? k_fwd<true> : k_fwd<false>;
    k<<<g, GTHREADS, 0, st>>>(n, out, in, l ? A[l - 1] : feat, l ? nullptr : idx, W, b, Z[l], A[l],
                              last ? tgt : nullptr, idx, dZ[3], nn.d_loss + 1);
    SMR_LAUNCH(c);
  }
  if (!tgt) return SMR_OK;                      // inference only
  k_sum<<<1, 256, 0, st>>>(nb, nn.d_loss + 1, 1.0 / ((double)n * O), nn.d_loss);
  SMR_LAUNCH(c);
  if (backward) {
    for (int l = 3; l > 0; --l) {
      const int in = nn.dims[l], out = nn.dims[l + 1];
      auto k = v4 ? k_dx<true> : k_dx<false>;
      k<<<dim3((in + GT - 1) / GT, my), GTHREADS, 0, st>>>(n, in, out, dZ[l], nn.w16 + woff(nn, l), Z[l - 1],
                                                           dZ[l - 1]);
      SMR_LAUNCH(c);
    }
    GradArgs g;
    g.idx = idx;
    g.np = nn.np;
    g.t0[0] = 0;
    for (int l = 0; l < 4; ++l) {
      g.A[l] = l ? A[l - 1] : feat;
      g.dZ[l] = dZ[l];
      g.in[l] = nn.dims[l];
      g.out[l] = nn.dims[l + 1];
      g.off[l] = woff(nn, l);
      g.t0[l + 1] = g.t0[l] + (g.in[l] + GT - 1) / GT * ((g.out[l] + GT - 1) / GT);
    }
    // the batch's rows in splits: about three CTAs per SM in all, at least 64
    // rows each (68 tiles at width 256: six splits)
    int S = std::max(1, std::min(3 * 152 / g.t0[4], n / 64));
    const int rows = ((n + S - 1) / S + GK - 1) / GK * GK;
    S = (n + rows - 1) / rows;
    const size_t need = (size_t)S * nn.np;
    if (S > 1 && nn.part_elems < need) {
      cudaFree(nn.part);
      nn.part = nullptr;
      nn.part_elems = 0;
      SMR_CUDA(c, cudaMalloc((void**)&nn.part, need * sizeof(float)));
      nn.part_elems = need;
    }
    auto k = v4 ? k_dw<true> : k_dw<false>;
    k<<<dim3(g.t0[4], S), GTHREADS, 0, st>>>(g, n, rows, S > 1 ? nn.part : nn.g);
    SMR_LAUNCH(c);
    if (S > 1) {
      k_split_sum<<<(unsigned)((nn.np + 255) / 256), 256, 0, st>>>(nn.np, S, nn.part, nn.g);
      SMR_LAUNCH(c);
    }
  }
  if (loss_host) {
    SMR_CUDA(c, cudaMemcpyAsync(loss_host, nn.d_loss, sizeof(double), cudaMemcpyDeviceToHost, st));
    SMR_CUDA(c, cudaStreamSynchronize(st));
  }
  return SMR_OK;
}

int nn_adam(Ctx* c, float lr, cudaStream_t st) {
  NN& nn = c->nn;
  nn.step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  float bc1 = 1.f - std::pow(b1, (float)nn.step), bc2 = 1.f - std::pow(b2, (float)nn.step);
  k_adam<<<(unsigned)((nn.np + 255) / 256), 256, 0, st>>>(nn.np, nn.p32, nn.w16, nn.g, nn.m, nn.v, lr, b1, b2,
                                                         1e-8f, bc1, bc2);
  SMR_LAUNCH(c);
  return SMR_OK;
}

int nn_predict(Ctx* c, const double* d_khat, const double* d_pol, double scale, double2* x0, cudaStream_t st) {
  NN& nn = c->nn;
  float* feat = nullptr;
  SMR_CUDA(c, cudaMalloc((void**)&feat, (size_t)c->p * nn.F * sizeof(float)));
  int rc = nn_features(c, d_khat, d_pol, feat, st);
  for (int r0 = 0; rc == SMR_OK && r0 < c->p; r0 += nn.cap) {
    int rows = std::min(nn.cap, c->p - r0);
    rc = nn_forward_backward(c, rows, feat + (size_t)r0 * nn.F, nullptr, nullptr, false, nullptr, st);
    if (rc) break;
    float* Y = nn.act + (size_t)6 * nn.cap * nn.H;
    long long ne = (long long)rows * 2 * c->npsi;
    k_rephase<<<(unsigned)((ne + 255) / 256), 256, 0, st>>>(c->p, c->npsi, r0, rows, c->d_arr, c->d_centres, d_khat,
                                                           Y, c->k, scale, x0);
    SMR_LAUNCH(c);
  }
  cudaStreamSynchronize(st);
  cudaFree(feat);
  return rc;
}

// Learned local-coupling preconditioner: per unknown, the ratio of the
// network's predicted coefficient to the isolated-particle response
// (blockdiag(Z_s^-1) b), with its magnitude clamped to [0.1, 10] (a zero or
// undefined ratio becomes 0.1).
__global__ void k_lpc_ratio(long long n, const double2* __restrict__ xp, const double2* __restrict__ zi,
                            double2* __restrict__ D) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double2 a = xp[i], b = zi[i];
  double bb = b.x * b.x + b.y * b.y;
  double2 r = make_double2(0.0, 0.0);
  if (bb > 0) r = make_double2((a.x * b.x + a.y * b.y) / bb, (a.y * b.x - a.x * b.y) / bb);
  double m = sqrt(r.x * r.x + r.y * r.y);
  if (!(m > 0.1)) {
    r = (m > 0) ? make_double2(0.1 * r.x / m, 0.1 * r.y / m) : make_double2(0.1, 0.0);
  } else if (m > 10.0) {
    r = make_double2(10.0 * r.x / m, 10.0 * r.y / m);
  }
  D[i] = r;
}

// z[i] *= D[i]
__global__ void k_lpc_apply(long long n, const double2* __restrict__ D, double2* __restrict__ z) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double2 d = D[i], v = z[i];
  z[i] = make_double2(d.x * v.x - d.y * v.y, d.x * v.y + d.y * v.x);
}

int nn_precond(Ctx* c, const double* d_khat, const double* d_pol, double scale, const double2* b, cudaStream_t st) {
  long long n = 2LL * c->npsi * c->p;
  double2 *xp = nullptr, *zi = nullptr;
  if (!c->d_lpc) SMR_CUDA(c, cudaMalloc((void**)&c->d_lpc, n * sizeof(double2)));
  SMR_CUDA(c, cudaMalloc((void**)&xp, n * sizeof(double2)));
  if (cudaMalloc((void**)&zi, n * sizeof(double2)) != cudaSuccess) {
    cudaFree(xp);
    c->err = "out of device memory";
    return SMR_E_OOM;
  }
  int rc = nn_predict(c, d_khat, d_pol, scale, xp, st);
  if (!rc) rc = run_precond(c, 1, SMR_PREC_FP64, b, zi, st);
  if (!rc) {
    k_lpc_ratio<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, xp, zi, c->d_lpc);
    if (cudaGetLastError() != cudaSuccess) { c->err = "lpc kernel launch"; rc = SMR_E_CUDA; }
  }
  cudaStreamSynchronize(st);
  cudaFree(xp);
  cudaFree(zi);
  c->lpc_ready = (rc == SMR_OK);
  return rc;
}

int lpc_apply(Ctx* c, double2* z, cudaStream_t st) {
  long long n = 2LL * c->npsi * c->p;
  k_lpc_apply<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, c->d_lpc, z);
  SMR_LAUNCH(c);
  return SMR_OK;
}

}  // namespace smr

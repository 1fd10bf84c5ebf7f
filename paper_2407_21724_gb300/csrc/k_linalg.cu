// FP64 Krylov kernels and the GMRES solver (Sec. V, stage v).
//
// Vectors are complex FP64 [n][R] (R right-hand sides innermost).  The R
// systems advance in lockstep: one R-column product per Arnoldi step, classical
// Gram-Schmidt with a second pass whenever a column's norm falls below 1/sqrt(10)
// of its value before projection, Givens rotations and the small least-squares
// problems on the host in FP64.  One device->host copy per step (two when the
// second pass runs) carries the Hessenberg column of every right-hand side.
#include <chrono>
#include <cmath>

#include "smr_internal.h"

namespace smr {

// partial[j][chunk][r] = sum over rows in chunk of conj(V_j[i][r]) w[i][r]
__global__ void k_multidot_part(int J, long long n, int R, int rl, int nchunk, long long rows_per,
                                const double2* __restrict__ V, long long ldv,
                                const double2* __restrict__ w, double2* __restrict__ part) {
  int j = blockIdx.y, chunk = blockIdx.x;
  int a = threadIdx.x / R, r = threadIdx.x % R;
  double2 acc = make_double2(0, 0);
  if (a < rl) {
    const double2* v = V + (size_t)j * ldv;
    long long i0 = chunk * rows_per, i1 = min(n, i0 + rows_per);
    for (long long i = i0 + a; i < i1; i += rl) {
      double2 x = v[i * R + r], y = w[i * R + r];
      acc.x = fma(x.y, y.y, fma(x.x, y.x, acc.x));
      acc.y = fma(-x.y, y.x, fma(x.x, y.y, acc.y));
    }
  }
  __shared__ double2 red[256];
  red[threadIdx.x] = acc;
  __syncthreads();
  if (a == 0 && r < R) {
    double2 s = make_double2(0, 0);
    for (int q = 0; q < rl; ++q) {
      double2 t = red[q * R + r];
      s.x += t.x;
      s.y += t.y;
    }
    part[((size_t)j * nchunk + chunk) * R + r] = s;
  }
}

__global__ void k_multidot_final(int J, int R, int nchunk, const double2* __restrict__ part,
                                 double2* __restrict__ h) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= J * R) return;
  int j = t / R, r = t % R;
  double2 s = make_double2(0, 0);
  for (int c = 0; c < nchunk; ++c) {
    double2 v = part[((size_t)j * nchunk + c) * R + r];
    s.x += v.x;
    s.y += v.y;
  }
  h[t] = s;
}

// w[i][r] += sign * sum_j V_j[i][r] h[j][r]
__global__ void k_multi_axpy(int J, long long n, int R, const double2* __restrict__ V, long long ldv,
                             const double2* __restrict__ h, double2* __restrict__ w, double sign) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= n * R) return;
  int r = (int)(t % R);
  double2 acc = make_double2(0, 0), acc2 = make_double2(0, 0);
  int j = 0;
  for (; j + 4 <= J; j += 4) {
    double2 v0 = V[(size_t)j * ldv + t], v1 = V[(size_t)(j + 1) * ldv + t];
    double2 v2 = V[(size_t)(j + 2) * ldv + t], v3 = V[(size_t)(j + 3) * ldv + t];
    double2 c0 = h[(size_t)j * R + r], c1 = h[(size_t)(j + 1) * R + r];
    double2 c2 = h[(size_t)(j + 2) * R + r], c3 = h[(size_t)(j + 3) * R + r];
    acc.x = fma(-v1.y, c1.y, fma(v1.x, c1.x, fma(-v0.y, c0.y, fma(v0.x, c0.x, acc.x))));
    acc.y = fma(v1.y, c1.x, fma(v1.x, c1.y, fma(v0.y, c0.x, fma(v0.x, c0.y, acc.y))));
    acc2.x = fma(-v3.y, c3.y, fma(v3.x, c3.x, fma(-v2.y, c2.y, fma(v2.x, c2.x, acc2.x))));
    acc2.y = fma(v3.y, c3.x, fma(v3.x, c3.y, fma(v2.y, c2.x, fma(v2.x, c2.y, acc2.y))));
  }
  for (; j < J; ++j) {
    double2 v = V[(size_t)j * ldv + t], c = h[(size_t)j * R + r];
    acc.x = fma(-v.y, c.y, fma(v.x, c.x, acc.x));
    acc.y = fma(v.y, c.x, fma(v.x, c.y, acc.y));
  }
  acc.x += acc2.x;
  acc.y += acc2.y;
  double2 o = w[t];
  o.x += sign * acc.x;
  o.y += sign * acc.y;
  w[t] = o;
}

// y = a[r] x + b[r] y
__global__ void k_axpby(long long n, int R, const double2* __restrict__ a, const double2* __restrict__ x,
                        const double2* __restrict__ b, double2* __restrict__ y) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= n * R) return;
  int r = (int)(t % R);
  double2 xa = x[t], yb = y[t], ca = a[r], cb = b[r];
  y[t] = make_double2(ca.x * xa.x - ca.y * xa.y + cb.x * yb.x - cb.y * yb.y,
                      ca.x * xa.y + ca.y * xa.x + cb.x * yb.y + cb.y * yb.x);
}

// y = a[r] x
__global__ void k_scale(long long n, int R, const double2* __restrict__ a, const double2* __restrict__ x,
                        double2* __restrict__ y) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= n * R) return;
  int r = R == 1 ? 0 : (int)(t % R);
  double2 xa = x[t], ca = a[r];
  y[t] = make_double2(ca.x * xa.x - ca.y * xa.y, ca.x * xa.y + ca.y * xa.x);
}

static void chunking(long long n, int R, int* rl, int* nchunk, long long* rows_per) {
  *rl = std::max(1, 256 / R);
  long long per = std::max<long long>(1024, (n + 511) / 512);
  *rows_per = per;
  *nchunk = (int)((n + per - 1) / per);
}

static int red_buffer(Ctx* c, size_t bytes) {
  if (c->red_bytes >= bytes) return SMR_OK;
  if (c->d_red) cudaFree(c->d_red);
  if (c->h_red) cudaFreeHost(c->h_red);
  c->d_red = nullptr;
  c->h_red = nullptr;
  SMR_CUDA(c, cudaMalloc((void**)&c->d_red, bytes));
  SMR_CUDA(c, cudaMallocHost((void**)&c->h_red, bytes));
  c->red_bytes = bytes;
  return SMR_OK;
}

// ---- single right-hand side Gram-Schmidt passes ----------------------------
// Warp g owns rows [GS_SEG g, GS_SEG (g+1)) and keeps its slice of w in
// registers; lane l holds rows GS_SEG g + l + 32 q, q < GS_RPL, so every load
// instruction of the warp is one coalesced 512-byte segment.  Two basis
// vectors are read per step (16 independent loads in flight per lane).
// Partial sums go to part[row][g] and a second kernel adds them up in a
// fixed order, so the results are deterministic.
constexpr int GS_RPL = 8;
constexpr int GS_SEG = 32 * GS_RPL;

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// part[j][g] = sum over the warp's rows of conj(V_j) w (j < J); with
// with_norm, part[J][g] = sum |w|^2.
__global__ void __launch_bounds__(256) k_gs_dot(int J, long long n, const double2* __restrict__ V,
                                                long long ldv, const double2* __restrict__ w,
                                                double2* __restrict__ part, int nseg, int with_norm) {
  int g = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  int lane = threadIdx.x & 31;
  if (g >= nseg) return;
  long long i0 = (long long)g * GS_SEG + lane;
  bool full = (long long)(g + 1) * GS_SEG <= n;
  double2 wr[GS_RPL];
#pragma unroll
  for (int q = 0; q < GS_RPL; ++q) {
    long long i = i0 + 32 * q;
    wr[q] = (full || i < n) ? w[i] : make_double2(0, 0);
  }
  if (with_norm && blockIdx.y == 0) {
    double s = 0;
#pragma unroll
    for (int q = 0; q < GS_RPL; ++q) s += wr[q].x * wr[q].x + wr[q].y * wr[q].y;
    s = warp_sum(s);
    if (lane == 0) part[(size_t)J * nseg + g] = make_double2(s, 0);
  }
  const int G = gridDim.y, per = 2 * (((J + 1) / 2 + G - 1) / G), j1 = min(J, per * ((int)blockIdx.y + 1));
  int j = per * blockIdx.y;
  for (; j + 2 <= j1; j += 2) {
    const double2* v0 = V + (size_t)j * ldv + i0;
    const double2* v1 = v0 + ldv;
    double2 a[GS_RPL], b[GS_RPL];
    if (full) {
#pragma unroll
      for (int q = 0; q < GS_RPL; ++q) {
        a[q] = v0[32 * q];
        b[q] = v1[32 * q];
      }
    } else {
#pragma unroll
      for (int q = 0; q < GS_RPL; ++q) {
        bool in = i0 + 32 * q < n;
        a[q] = in ? v0[32 * q] : make_double2(0, 0);
        b[q] = in ? v1[32 * q] : make_double2(0, 0);
      }
    }
    double ax = 0, ay = 0, bx = 0, by = 0;
#pragma unroll
    for (int q = 0; q < GS_RPL; ++q) {
      ax = fma(a[q].y, wr[q].y, fma(a[q].x, wr[q].x, ax));
      ay = fma(-a[q].y, wr[q].x, fma(a[q].x, wr[q].y, ay));
      bx = fma(b[q].y, wr[q].y, fma(b[q].x, wr[q].x, bx));
      by = fma(-b[q].y, wr[q].x, fma(b[q].x, wr[q].y, by));
    }
    ax = warp_sum(ax);
    ay = warp_sum(ay);
    bx = warp_sum(bx);
    by = warp_sum(by);
    if (lane == 0) {
      part[(size_t)j * nseg + g] = make_double2(ax, ay);
      part[(size_t)(j + 1) * nseg + g] = make_double2(bx, by);
    }
  }
  if (j < j1) {
    const double2* v0 = V + (size_t)j * ldv + i0;
    double ax = 0, ay = 0;
#pragma unroll
    for (int q = 0; q < GS_RPL; ++q) {
      double2 a = (full || i0 + 32 * q < n) ? v0[32 * q] : make_double2(0, 0);
      ax = fma(a.y, wr[q].y, fma(a.x, wr[q].x, ax));
      ay = fma(-a.y, wr[q].x, fma(a.x, wr[q].y, ay));
    }
    ax = warp_sum(ax);
    ay = warp_sum(ay);
    if (lane == 0) part[(size_t)j * nseg + g] = make_double2(ax, ay);
  }
}

// w += sign * sum_j V_j h[j] on the warp's rows; with part_norm, also
// part_norm[g] = sum |w_new|^2 over those rows.  A lane holds RPL rows and reads
// 16 / RPL basis vectors at a time.
template <int RPL>
__global__ void __launch_bounds__(256) k_gs_axpy(int J, long long n, const double2* __restrict__ V,
                                                 long long ldv, const double2* __restrict__ h,
                                                 double2* __restrict__ w, double sign,
                                                 double2* __restrict__ part_norm, int nseg) {
  constexpr int JU = 16 / RPL, SEG = 32 * RPL;
  int g = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  int lane = threadIdx.x & 31;
  if (g >= nseg) return;
  long long i0 = (long long)g * SEG + lane;
  bool full = (long long)(g + 1) * SEG <= n;
  double2 acc[RPL];
#pragma unroll
  for (int q = 0; q < RPL; ++q) acc[q] = make_double2(0, 0);
  auto ld = [&](int jj, int q) {
    return full || i0 + 32 * q < n ? V[(size_t)jj * ldv + i0 + 32 * q] : make_double2(0, 0);
  };
  auto add = [&](double2& o, double2 a, double2 c0) {
    o.x = fma(-a.y, c0.y, fma(a.x, c0.x, o.x));
    o.y = fma(a.y, c0.x, fma(a.x, c0.y, o.y));
  };
  int j = 0;
  for (; j + JU <= J; j += JU) {
    double2 a[JU][RPL];
#pragma unroll
    for (int u = 0; u < JU; ++u)
#pragma unroll
      for (int q = 0; q < RPL; ++q) a[u][q] = ld(j + u, q);
#pragma unroll
    for (int u = 0; u < JU; ++u) {
      const double2 c0 = h[j + u];
#pragma unroll
      for (int q = 0; q < RPL; ++q) add(acc[q], a[u][q], c0);
    }
  }
  for (; j < J; ++j) {
    const double2 c0 = h[j];
#pragma unroll
    for (int q = 0; q < RPL; ++q) add(acc[q], ld(j, q), c0);
  }
  double s = 0;
#pragma unroll
  for (int q = 0; q < RPL; ++q) {
    long long i = i0 + 32 * q;
    if (full || i < n) {
      double2 o = w[i];
      o.x += sign * acc[q].x;
      o.y += sign * acc[q].y;
      w[i] = o;
      s += o.x * o.x + o.y * o.y;
    }
  }
  if (part_norm) {
    s = warp_sum(s);
    if (lane == 0) part_norm[g] = make_double2(s, 0);
  }
}

// out[r] = sum_g part[r][g] for r < rows (r < na goes to out_a[r], the rest
// to out_b[r - na]); one CTA per row, fixed summation order.
__global__ void k_gs_final(int nseg, const double2* __restrict__ part, int na, double2* __restrict__ out_a,
                           double2* __restrict__ out_b, float2* __restrict__ out_f) {
  __shared__ double2 red[256];
  int r = blockIdx.x;
  double2 s = make_double2(0, 0);
  for (int c = threadIdx.x; c < nseg; c += blockDim.x) {
    double2 v = part[(size_t)r * nseg + c];
    s.x += v.x;
    s.y += v.y;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int hh = blockDim.x / 2; hh > 0; hh >>= 1) {
    if ((int)threadIdx.x < hh) {
      red[threadIdx.x].x += red[threadIdx.x + hh].x;
      red[threadIdx.x].y += red[threadIdx.x + hh].y;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (r < na) {
      out_a[r] = red[0];
      if (out_f) out_f[r] = make_float2((float)red[0].x, (float)red[0].y);
    } else {
      out_b[r - na] = red[0];
    }
  }
}

static inline int gs_nseg(long long n) { return (int)((n + GS_SEG - 1) / GS_SEG); }
static inline unsigned gs_grid(int nseg) { return (unsigned)((nseg + 7) / 8); }

// CTAs along the basis vectors of an inner-product pass: as many as make two CTAs an
// SM, at most one per `most` units.  A solve of 1,600 particles, 107 steps on an FP32
// basis: 9.6 ms of Gram-Schmidt with 25 CTAs for all vectors, 5.3 with the split and
// with one row pair a lane in the update below 152 CTAs of eight
static inline unsigned gs_split(unsigned ctas, int most) {
  return std::max(1u, std::min((unsigned)std::max(1, most), 304u / std::max(1u, ctas)));
}

// h[0..J) = V^H w and, when d_norm is given, *d_norm = ||w||^2 (one pass).
static int gs_dot(Ctx* c, int J, long long n, const double2* V, long long ldv, const double2* w,
                  double2* d_h, double2* d_norm, double2* d_part, cudaStream_t st) {
  int nseg = gs_nseg(n);
  int rows = J + (d_norm ? 1 : 0);
  if (rows == 0) return SMR_OK;
  const dim3 grid(gs_grid(nseg), gs_split(gs_grid(nseg), (J + 1) / 2));
  k_gs_dot<<<grid, 256, 0, st>>>(J, n, V, ldv, w, d_part, nseg, d_norm ? 1 : 0);
  SMR_LAUNCH(c);
  k_gs_final<<<rows, 256, 0, st>>>(nseg, d_part, J, d_h, d_norm, nullptr);
  SMR_LAUNCH(c);
  return SMR_OK;
}

// w += sign V h and, when d_norm is given, *d_norm = ||w_new||^2 (one pass).
static int gs_axpy(Ctx* c, int J, long long n, const double2* V, long long ldv, const double2* d_h,
                   double2* w, double sign, double2* d_norm, double2* d_part, cudaStream_t st) {
  // one row a lane where eight leave SMs idle (as in gs32_axpy)
  const bool few = gs_grid(gs_nseg(n)) < 152;
  const int nseg = few ? (int)((n + 31) / 32) : gs_nseg(n);
  auto k = few ? k_gs_axpy<1> : k_gs_axpy<GS_RPL>;
  k<<<gs_grid(nseg), 256, 0, st>>>(J, n, V, ldv, d_h, w, sign, d_norm ? d_part : nullptr, nseg);
  SMR_LAUNCH(c);
  if (d_norm) {
    k_gs_final<<<1, 256, 0, st>>>(nseg, d_part, 0, nullptr, d_norm, nullptr);
    SMR_LAUNCH(c);
  }
  return SMR_OK;
}

// ---- single right-hand side with an FP32 Krylov basis ----------------------
// The FP64 passes above are bound by the FP64 units (four DFMA per complex
// element, a ~1.2 TFLOP/s rate), not by HBM.  With the basis in FP32 the
// products run on the FP32 pipes and the bytes halve.  Lane l of warp g holds
// complex rows G32_SEG g + 2 l + 64 q + {0, 1}, q < G32_RPL, read as one
// float4 per basis vector (a 512-byte segment per warp instruction); the
// in-warp sums are FP32, the sums over warps FP64.  The new w stays FP64.
constexpr int G32_RPL = 8;
constexpr int G32_SEG = 64 * G32_RPL;

__device__ __forceinline__ float warp_sumf(float v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// float4 holding complex rows i, i + 1 of v (zero beyond n)
__device__ __forceinline__ float4 ld_pair(const float2* __restrict__ v, long long i, long long n, bool full) {
  if (full || i + 1 < n) return *reinterpret_cast<const float4*>(v + i);
  if (i < n) {
    float2 a = v[i];
    return make_float4(a.x, a.y, 0.f, 0.f);
  }
  return make_float4(0.f, 0.f, 0.f, 0.f);
}

// part[j][g] = conj(V_j) . w over the warp's rows (j < J); with with_norm,
// part[J][g] = sum |w|^2 (FP64).  The basis vectors are divided over blockIdx.y: with
// a warp per segment for all of them, short vectors leave most SMs idle (1,600
// particles: 200 warps; figures at gs_split).
__global__ void __launch_bounds__(256) k_gs32_dot(int J, long long n, const float2* __restrict__ V,
                                                  long long ldv, const double2* __restrict__ w,
                                                  double2* __restrict__ part, int nseg, int with_norm) {
  const int g = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  int lane = threadIdx.x & 31;
  if (g >= nseg) return;
  long long i0 = (long long)g * G32_SEG + 2 * lane;
  bool full = (long long)(g + 1) * G32_SEG <= n;
  float4 wf[G32_RPL];
  double s = 0;
#pragma unroll
  for (int q = 0; q < G32_RPL; ++q) {
    long long i = i0 + 64 * q;
    double2 w0 = (full || i < n) ? w[i] : make_double2(0, 0);
    double2 w1 = (full || i + 1 < n) ? w[i + 1] : make_double2(0, 0);
    s += w0.x * w0.x + w0.y * w0.y + w1.x * w1.x + w1.y * w1.y;
    wf[q] = make_float4((float)w0.x, (float)w0.y, (float)w1.x, (float)w1.y);
  }
  if (with_norm && blockIdx.y == 0) {
    s = warp_sum(s);
    if (lane == 0) part[(size_t)J * nseg + g] = make_double2(s, 0);
  }
  // this CTA's basis vectors, an even number of them but for the last
  const int G = gridDim.y, per = 2 * (((J + 1) / 2 + G - 1) / G), j1 = min(J, per * ((int)blockIdx.y + 1));
  int j = per * blockIdx.y;
  for (; j + 2 <= j1; j += 2) {
    const float2* v0 = V + (size_t)j * ldv;
    const float2* v1 = v0 + ldv;
    float4 a[G32_RPL], b[G32_RPL];
#pragma unroll
    for (int q = 0; q < G32_RPL; ++q) {
      a[q] = ld_pair(v0, i0 + 64 * q, n, full);
      b[q] = ld_pair(v1, i0 + 64 * q, n, full);
    }
    float ax = 0, ay = 0, bx = 0, by = 0;
#pragma unroll
    for (int q = 0; q < G32_RPL; ++q) {
      float4 u = wf[q];
      ax = fma(a[q].w, u.w, fma(a[q].z, u.z, fma(a[q].y, u.y, fma(a[q].x, u.x, ax))));
      ay = fma(-a[q].w, u.z, fma(a[q].z, u.w, fma(-a[q].y, u.x, fma(a[q].x, u.y, ay))));
      bx = fma(b[q].w, u.w, fma(b[q].z, u.z, fma(b[q].y, u.y, fma(b[q].x, u.x, bx))));
      by = fma(-b[q].w, u.z, fma(b[q].z, u.w, fma(-b[q].y, u.x, fma(b[q].x, u.y, by))));
    }
    ax = warp_sumf(ax);
    ay = warp_sumf(ay);
    bx = warp_sumf(bx);
    by = warp_sumf(by);
    if (lane == 0) {
      part[(size_t)j * nseg + g] = make_double2(ax, ay);
      part[(size_t)(j + 1) * nseg + g] = make_double2(bx, by);
    }
  }
  if (j < j1) {
    const float2* v0 = V + (size_t)j * ldv;
    float ax = 0, ay = 0;
#pragma unroll
    for (int q = 0; q < G32_RPL; ++q) {
      float4 a = ld_pair(v0, i0 + 64 * q, n, full), u = wf[q];
      ax = fma(a.w, u.w, fma(a.z, u.z, fma(a.y, u.y, fma(a.x, u.x, ax))));
      ay = fma(-a.w, u.z, fma(a.z, u.w, fma(-a.y, u.x, fma(a.x, u.y, ay))));
    }
    ax = warp_sumf(ax);
    ay = warp_sumf(ay);
    if (lane == 0) part[(size_t)j * nseg + g] = make_double2(ax, ay);
  }
}

// w += sign * sum_j V_j hf[j] (FP32 products and sums, FP64 update of w);
// with part_norm, part_norm[g] = sum |w_new|^2 over the warp's rows.  A lane holds
// RPL row pairs and reads 16 / RPL basis vectors at a time.
template <int RPL>
__global__ void __launch_bounds__(256) k_gs32_axpy(int J, long long n, const float2* __restrict__ V,
                                                   long long ldv, const float2* __restrict__ hf,
                                                   double2* __restrict__ w, double sign,
                                                   double2* __restrict__ part_norm, int nseg) {
  constexpr int JU = 16 / RPL, SEG = 64 * RPL;
  int g = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  int lane = threadIdx.x & 31;
  if (g >= nseg) return;
  long long i0 = (long long)g * SEG + 2 * lane;
  bool full = (long long)(g + 1) * SEG <= n;
  float4 acc[RPL];
#pragma unroll
  for (int q = 0; q < RPL; ++q) acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  auto add = [&](float4& o, float4 a, float2 c0) {
    o.x = fma(-a.y, c0.y, fma(a.x, c0.x, o.x));
    o.y = fma(a.y, c0.x, fma(a.x, c0.y, o.y));
    o.z = fma(-a.w, c0.y, fma(a.z, c0.x, o.z));
    o.w = fma(a.w, c0.x, fma(a.z, c0.y, o.w));
  };
  int j = 0;
  for (; j + JU <= J; j += JU) {
    float4 a[JU][RPL];
#pragma unroll
    for (int u = 0; u < JU; ++u)
#pragma unroll
      for (int q = 0; q < RPL; ++q) a[u][q] = ld_pair(V + (size_t)(j + u) * ldv, i0 + 64 * q, n, full);
#pragma unroll
    for (int u = 0; u < JU; ++u) {
      const float2 c0 = hf[j + u];
#pragma unroll
      for (int q = 0; q < RPL; ++q) add(acc[q], a[u][q], c0);
    }
  }
  for (; j < J; ++j) {
    const float2 c0 = hf[j];
#pragma unroll
    for (int q = 0; q < RPL; ++q) add(acc[q], ld_pair(V + (size_t)j * ldv, i0 + 64 * q, n, full), c0);
  }
  double s = 0;
#pragma unroll
  for (int q = 0; q < RPL; ++q) {
    long long i = i0 + 64 * q;
    if (full || i < n) {
      double2 o = w[i];
      o.x += sign * (double)acc[q].x;
      o.y += sign * (double)acc[q].y;
      w[i] = o;
      s += o.x * o.x + o.y * o.y;
    }
    if (full || i + 1 < n) {
      double2 o = w[i + 1];
      o.x += sign * (double)acc[q].z;
      o.y += sign * (double)acc[q].w;
      w[i + 1] = o;
      s += o.x * o.x + o.y * o.y;
    }
  }
  if (part_norm) {
    s = warp_sum(s);
    if (lane == 0) part_norm[g] = make_double2(s, 0);
  }
}

// v = (float) (a[0] w)
__global__ void k_narrow_scale(long long n, const double2* __restrict__ a, const double2* __restrict__ w,
                               float2* __restrict__ v) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= n) return;
  double2 x = w[t], c = a[0];
  v[t] = make_float2((float)(c.x * x.x - c.y * x.y), (float)(c.x * x.y + c.y * x.x));
}

__global__ void k_widen(long long n, const float2* __restrict__ v, double2* __restrict__ u) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= n) return;
  float2 x = v[t];
  u[t] = make_double2(x.x, x.y);
}

// ---- several right-hand sides with an FP32 Krylov basis (vectors [n][R])
// part[j][chunk][r] = conj(V_j) . w over the chunk's rows, FP32 products and
// per-thread sums, FP64 sums across the CTA
__global__ void k_gsr_dot(int J, long long n, int R, int rl, int nchunk, long long rows_per,
                          const float2* __restrict__ V, long long ldv, const double2* __restrict__ w,
                          double2* __restrict__ part) {
  int j = blockIdx.y, chunk = blockIdx.x;
  int a = threadIdx.x / R, r = threadIdx.x % R;
  float ax = 0.f, ay = 0.f;
  if (a < rl) {
    const float2* v = V + (size_t)j * ldv;
    long long i0 = chunk * rows_per, i1 = min(n, i0 + rows_per);
    for (long long i = i0 + a; i < i1; i += rl) {
      float2 x = v[i * R + r];
      double2 yd = w[i * R + r];
      float2 y = make_float2((float)yd.x, (float)yd.y);
      ax = fma(x.y, y.y, fma(x.x, y.x, ax));
      ay = fma(-x.y, y.x, fma(x.x, y.y, ay));
    }
  }
  __shared__ double2 red[256];
  red[threadIdx.x] = make_double2(ax, ay);
  __syncthreads();
  if (a == 0 && r < R) {
    double2 s = make_double2(0, 0);
    for (int q = 0; q < rl; ++q) {
      double2 t = red[q * R + r];
      s.x += t.x;
      s.y += t.y;
    }
    part[((size_t)j * nchunk + chunk) * R + r] = s;
  }
}

// h[j][r] (FP64) and hf[j][r] (FP32) = sum over chunks of part[j][chunk][r]
__global__ void k_gsr_final(int J, int R, int nchunk, const double2* __restrict__ part, double2* __restrict__ h,
                            float2* __restrict__ hf) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= J * R) return;
  int j = t / R, r = t % R;
  double2 s = make_double2(0, 0);
  for (int c = 0; c < nchunk; ++c) {
    double2 v = part[((size_t)j * nchunk + c) * R + r];
    s.x += v.x;
    s.y += v.y;
  }
  h[t] = s;
  hf[t] = make_float2((float)s.x, (float)s.y);
}

// w[i][r] += sign * sum_j V_j[i][r] hf[j][r] (FP32 products and sums)
__global__ void k_gsr_axpy(int J, long long n, int R, const float2* __restrict__ V, long long ldv,
                           const float2* __restrict__ hf, double2* __restrict__ w, double sign) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= n * R) return;
  int r = (int)(t % R);
  float ax = 0.f, ay = 0.f, bx = 0.f, by = 0.f;
  int j = 0;
  for (; j + 2 <= J; j += 2) {
    float2 v0 = V[(size_t)j * ldv + t], v1 = V[(size_t)(j + 1) * ldv + t];
    float2 c0 = hf[(size_t)j * R + r], c1 = hf[(size_t)(j + 1) * R + r];
    ax = fma(-v0.y, c0.y, fma(v0.x, c0.x, ax));
    ay = fma(v0.y, c0.x, fma(v0.x, c0.y, ay));
    bx = fma(-v1.y, c1.y, fma(v1.x, c1.x, bx));
    by = fma(v1.y, c1.x, fma(v1.x, c1.y, by));
  }
  if (j < J) {
    float2 v0 = V[(size_t)j * ldv + t], c0 = hf[(size_t)j * R + r];
    ax = fma(-v0.y, c0.y, fma(v0.x, c0.x, ax));
    ay = fma(v0.y, c0.x, fma(v0.x, c0.y, ay));
  }
  double2 o = w[t];
  o.x += sign * ((double)ax + (double)bx);
  o.y += sign * ((double)ay + (double)by);
  w[t] = o;
}

// v[i][r] = (float) (a[r] w[i][r])
__global__ void k_narrow_scale_r(long long n, int R, const double2* __restrict__ a, const double2* __restrict__ w,
                                 float2* __restrict__ v) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= n * R) return;
  double2 x = w[t], c = a[t % R];
  v[t] = make_float2((float)(c.x * x.x - c.y * x.y), (float)(c.x * x.y + c.y * x.x));
}

static inline int g32_nseg(long long n) { return (int)((n + G32_SEG - 1) / G32_SEG); }

// h = V^H w (FP64 d_h and FP32 d_hf copies) and optionally ||w||^2
static int gs32_dot(Ctx* c, int J, long long n, const float2* V, long long ldv, const double2* w,
                    double2* d_h, float2* d_hf, double2* d_norm, double2* d_part, cudaStream_t st) {
  int nseg = g32_nseg(n);
  int rows = J + (d_norm ? 1 : 0);
  if (rows == 0) return SMR_OK;
  const dim3 grid(gs_grid(nseg), gs_split(gs_grid(nseg), (J + 1) / 2));
  k_gs32_dot<<<grid, 256, 0, st>>>(J, n, V, ldv, w, d_part, nseg, d_norm ? 1 : 0);
  SMR_LAUNCH(c);
  k_gs_final<<<rows, 256, 0, st>>>(nseg, d_part, J, d_h, d_norm, d_hf);
  SMR_LAUNCH(c);
  return SMR_OK;
}

static int gs32_axpy(Ctx* c, int J, long long n, const float2* V, long long ldv, const float2* d_hf,
                     double2* w, double sign, double2* d_norm, double2* d_part, cudaStream_t st) {
  // one row pair a lane where eight leave SMs idle (figures at gs_split)
  const bool few = gs_grid(g32_nseg(n)) < 152;
  const int nseg = few ? (int)((n + 63) / 64) : g32_nseg(n);
  auto k = few ? k_gs32_axpy<1> : k_gs32_axpy<G32_RPL>;
  k<<<gs_grid(nseg), 256, 0, st>>>(J, n, V, ldv, d_hf, w, sign, d_norm ? d_part : nullptr, nseg);
  SMR_LAUNCH(c);
  if (d_norm) {
    k_gs_final<<<1, 256, 0, st>>>(nseg, d_part, 0, nullptr, d_norm, nullptr);
    SMR_LAUNCH(c);
  }
  return SMR_OK;
}

// partial-sum area (double2 elements) that J inner products need
static size_t part_elems(long long n, int R, int J) {
  int rl, nchunk;
  long long per;
  chunking(n, R, &rl, &nchunk, &per);
  return std::max(std::max((size_t)J * nchunk * R, (size_t)(J + 1) * gs_nseg(n)), (size_t)((n + 31) / 32));
}

// d_h[J][R] on the device.
static int multidot_dev(Ctx* c, int J, long long n, int R, const double2* V, long long ldv,
                        const double2* w, double2* d_h, double2* d_part, cudaStream_t st) {
  if (R == 1) return gs_dot(c, J, n, V, ldv, w, d_h, nullptr, d_part, st);
  int rl, nchunk;
  long long per;
  chunking(n, R, &rl, &nchunk, &per);
  dim3 g(nchunk, J);
  k_multidot_part<<<g, 256, 0, st>>>(J, n, R, rl, nchunk, per, V, ldv, w, d_part);
  SMR_LAUNCH(c);
  k_multidot_final<<<(J * R + 127) / 128, 128, 0, st>>>(J, R, nchunk, d_part, d_h);
  SMR_LAUNCH(c);
  return SMR_OK;
}

int multidot(Ctx* c, int J, long long n, int R, const double2* V, long long ldv, const double2* w,
             double2* h_host, cudaStream_t st) {
  int rl, nchunk;
  long long per;
  chunking(n, R, &rl, &nchunk, &per);
  size_t np = part_elems(n, R, J);
  size_t need = (np + (size_t)J * R) * sizeof(double2);
  int rc = red_buffer(c, need);
  if (rc) return rc;
  double2* d_part = (double2*)c->d_red;
  double2* d_h = d_part + np;
  rc = multidot_dev(c, J, n, R, V, ldv, w, d_h, d_part, st);
  if (rc) return rc;
  SMR_CUDA(c, cudaMemcpyAsync(h_host, d_h, (size_t)J * R * sizeof(double2), cudaMemcpyDeviceToHost, st));
  SMR_CUDA(c, cudaStreamSynchronize(st));
  return SMR_OK;
}

int multi_axpy(Ctx* c, int J, long long n, int R, const double2* V, long long ldv, const double2* d_h,
               double2* w, double sign, cudaStream_t st) {
  if (R == 1) return gs_axpy(c, J, n, V, ldv, d_h, w, sign, nullptr, nullptr, st);
  long long tot = n * R;
  k_multi_axpy<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(J, n, R, V, ldv, d_h, w, sign);
  SMR_LAUNCH(c);
  return SMR_OK;
}

int col_norms(Ctx* c, long long n, int R, const double2* v, double* norms_host, cudaStream_t st) {
  std::vector<double2> h(R);
  int rc = multidot(c, 1, n, R, v, 0, v, h.data(), st);
  if (rc) return rc;
  // NaN stays NaN (std::max(0.0, NaN) would hide it)
  for (int r = 0; r < R; ++r) norms_host[r] = std::isnan(h[r].x) ? h[r].x : std::sqrt(std::max(0.0, h[r].x));
  return SMR_OK;
}

int col_axpby(long long n, int R, const double2* d_a, const double2* x, const double2* d_b, double2* y,
              cudaStream_t st) {
  long long tot = n * R;
  k_axpby<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(n, R, d_a, x, d_b, y);
  return cudaGetLastError() == cudaSuccess ? SMR_OK : SMR_E_CUDA;
}

// ------------------------------------------------------------------ GMRES
namespace {

struct Work {
  bool f32 = false;        // Krylov basis in FP32 (one right-hand side, FP32 operator)
  void* V = nullptr;       // [m+1][n][R] basis, double2 or float2
  double2* u = nullptr;    // [n][R] residual r0; FP64 copy of v_j for the preconditioner
  double2* w = nullptr;    // [n][R]
  double2* t = nullptr;    // [n][R]
  double2* coef = nullptr; // device [4][m+2][R] coefficients
  float2* coef_f = nullptr;  // device [3][m+2] FP32 coefficient copies
  double2* part = nullptr; // reduction partials
  double2* hpin = nullptr; // pinned host copy of the coefficient area read each iteration
  cudaEvent_t ev[6] = {};
  double t_pc = 0, t_mv = 0, t_or = 0;   // seconds in preconditioner, products, Gram-Schmidt
};

}  // namespace

static int apply_A(Ctx* c, int R, int prec, const double2* x, double2* y, cudaStream_t st) {
  return run_product(c, R, prec, x, y, st);
}

// y += a x for a complex scalar a
__global__ void k_caxpy(long long n, double2 a, const double2* __restrict__ x, double2* __restrict__ y) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) {
    const double2 v = x[i];
    double2 o = y[i];
    o.x += a.x * v.x - a.y * v.y;
    o.y += a.x * v.y + a.y * v.x;
    y[i] = o;
  }
}

__global__ void k_sweep_update(long long n, double2* __restrict__ z, const double2* __restrict__ t,
                               const double2* __restrict__ u) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) {
    double2 a = z[i], b = t[i], d = u[i];
    z[i] = make_double2(a.x + b.x - d.x, a.y + b.y - d.y);
  }
}

// z = M^-1 v: the block-diagonal preconditioner D^-1, scaled per unknown by
// the learned diagonal for SMR_PRECOND_LEARNED, followed for
// SMR_PRECOND_NEAR by c->pc_sweeps Jacobi sweeps over the near field
// (z <- z + D^-1 v - D^-1 Z_near z), the cluster block-Jacobi inverse for
// SMR_PRECOND_CLUSTER, or a copy for SMR_PRECOND_NONE

typedef std::complex<double> zc;

// Eigenvalues of an upper Hessenberg complex matrix A (n x n, column-major)
// by the shifted QR algorithm: Wilkinson shifts from the trailing 2 x 2 of
// the active block, Givens rotations, deflation at negligible subdiagonals.
static bool hess_eigvals(int n, std::vector<zc> A, std::vector<zc>& ev) {
  auto a = [&](int i, int j) -> zc& { return A[(size_t)j * n + i]; };
  ev.assign(n, zc(0, 0));
  int hi = n - 1, iter = 0;
  while (hi >= 0) {
    if (hi == 0) { ev[0] = a(0, 0); break; }
    int l = hi;
    for (; l > 0; --l) {
      const double sc = std::abs(a(l - 1, l - 1)) + std::abs(a(l, l));
      if (std::abs(a(l, l - 1)) <= 1e-15 * (sc > 0 ? sc : 1.0)) { a(l, l - 1) = 0; break; }
    }
    if (l == hi) { ev[hi] = a(hi, hi); --hi; iter = 0; continue; }
    if (++iter > 300) return false;
    const zc p = a(hi - 1, hi - 1), q = a(hi - 1, hi), r = a(hi, hi - 1), t = a(hi, hi);
    const zc tr = p + t, det = p * t - q * r, disc = std::sqrt(tr * tr / 4.0 - det);
    const zc m1 = tr / 2.0 + disc, m2 = tr / 2.0 - disc;
    zc mu = std::abs(m1 - t) < std::abs(m2 - t) ? m1 : m2;
    if (iter % 11 == 10) mu = t + zc(std::abs(a(hi, hi - 1)), 0.0);   // exceptional shift
    for (int k = l; k <= hi; ++k) a(k, k) -= mu;
    std::vector<zc> cs(hi - l), sn(hi - l);
    for (int k = l; k < hi; ++k) {
      const zc x = a(k, k), y = a(k + 1, k);
      const double rr = std::sqrt(std::norm(x) + std::norm(y));
      const zc cc = rr > 0 ? x / rr : zc(1, 0), ss = rr > 0 ? y / rr : zc(0, 0);
      for (int j = k; j <= hi; ++j) {                // rows k, k+1 <- G [rows]
        const zc t1 = a(k, j), t2 = a(k + 1, j);
        a(k, j) = std::conj(cc) * t1 + std::conj(ss) * t2;
        a(k + 1, j) = -ss * t1 + cc * t2;
      }
      cs[k - l] = cc;
      sn[k - l] = ss;
    }
    for (int k = l; k < hi; ++k) {                    // columns k, k+1 <- [columns] G^H
      const zc cc = cs[k - l], ss = sn[k - l];
      for (int i = l; i <= std::min(k + 1, hi); ++i) {
        const zc t1 = a(i, k), t2 = a(i, k + 1);
        a(i, k) = t1 * cc + t2 * ss;
        a(i, k + 1) = -t1 * std::conj(ss) + t2 * std::conj(cc);
      }
    }
    for (int k = l; k <= hi; ++k) a(k, k) += mu;
  }
  return true;
}

// Harmonic Ritz values of the d-step Arnoldi relation with the (d+1) x d
// Hessenberg Hb (column-major, leading dimension ld): the eigenvalues of
// H_d + |h_{d+1,d}|^2 f e_d^T with H_d^H f = e_d -- the roots of the GMRES
// residual polynomial of degree d.
static bool harmonic_ritz(int d, const std::vector<zc>& Hb, int ldh, std::vector<zc>& th) {
  std::vector<zc> Hd((size_t)d * d), M((size_t)d * d), f(d, zc(0, 0));
  for (int j = 0; j < d; ++j)
    for (int i = 0; i < d; ++i) Hd[(size_t)j * d + i] = Hb[(size_t)j * ldh + i];
  const zc h = Hb[(size_t)(d - 1) * ldh + d];
  // solve H_d^H f = e_d by Gaussian elimination with partial pivoting
  for (int j = 0; j < d; ++j)
    for (int i = 0; i < d; ++i) M[(size_t)j * d + i] = std::conj(Hd[(size_t)i * d + j]);
  f[d - 1] = 1.0;
  for (int k = 0; k < d; ++k) {
    int piv = k;
    for (int i = k + 1; i < d; ++i)
      if (std::abs(M[(size_t)k * d + i]) > std::abs(M[(size_t)k * d + piv])) piv = i;
    if (std::abs(M[(size_t)k * d + piv]) == 0.0) return false;
    if (piv != k) {
      for (int j = 0; j < d; ++j) std::swap(M[(size_t)j * d + k], M[(size_t)j * d + piv]);
      std::swap(f[k], f[piv]);
    }
    for (int i = k + 1; i < d; ++i) {
      const zc fac = M[(size_t)k * d + i] / M[(size_t)k * d + k];
      for (int j = k; j < d; ++j) M[(size_t)j * d + i] -= fac * M[(size_t)j * d + k];
      f[i] -= fac * f[k];
    }
  }
  for (int i = d - 1; i >= 0; --i) {
    zc sum = f[i];
    for (int j = i + 1; j < d; ++j) sum -= M[(size_t)j * d + i] * f[j];
    f[i] = sum / M[(size_t)i * d + i];
  }
  for (int i = 0; i < d; ++i) Hd[(size_t)(d - 1) * d + i] += std::norm(h) * f[i];
  if (!hess_eigvals(d, Hd, th)) return false;
  for (const zc& z : th)
    if (!std::isfinite(z.real()) || !std::isfinite(z.imag()) || std::abs(z) == 0.0) return false;
  return true;
}

// Leja order: the largest root first, then each next root maximises the
// product of its distances to the roots already taken.
static void leja_order(std::vector<zc>& th) {
  const int n = (int)th.size();
  std::vector<zc> out;
  std::vector<char> used(n, 0);
  for (int k = 0; k < n; ++k) {
    int best = -1;
    double bs = -1e300;
    for (int i = 0; i < n; ++i) {
      if (used[i]) continue;
      double sc = 0;
      if (out.empty()) sc = std::abs(th[i]);
      else
        for (const zc& z : out) sc += std::log(std::max(std::abs(th[i] - z), 1e-300));
      if (sc > bs) { bs = sc; best = i; }
    }
    used[best] = 1;
    out.push_back(th[best]);
  }
  th = out;
}

static int apply_M(Ctx* c, int R, int prec, int precond, const double2* v, double2* z, cudaStream_t st);

// z = M^-1 p(B) v with B = A M^-1 and p the polynomial preconditioner in
// root form: 1 - x p(x) = prod_i (1 - x / theta_i), the roots in Leja order
// (prod <- v; for each root but the last: y += prod / theta_i, prod -= B prod
// / theta_i; y += prod / theta_last; z = M^-1 y)
static int apply_poly(Ctx* c, int R, int prec, int precond, const double2* v, double2* z, cudaStream_t st) {
  const long long ld = 2LL * c->npsi * c->p * R;
  const unsigned nb = (unsigned)((ld + 255) / 256);
  double2* prod = c->d_polyw;
  double2* y = c->d_polyw + ld;
  double2* t = c->d_polyw + 2 * ld;
  double2* w = c->d_polyw + 3 * ld;
  const auto& th = c->poly_roots;
  const int dp = (int)th.size();
  SMR_CUDA(c, cudaMemcpyAsync(prod, v, (size_t)ld * sizeof(double2), cudaMemcpyDeviceToDevice, st));
  SMR_CUDA(c, cudaMemsetAsync(y, 0, (size_t)ld * sizeof(double2), st));
  int rc = SMR_OK;
  for (int i = 0; i < dp && !rc; ++i) {
    const std::complex<double> inv = 1.0 / th[i];
    k_caxpy<<<nb, 256, 0, st>>>(ld, make_double2(inv.real(), inv.imag()), prod, y);
    SMR_CUDA(c, cudaGetLastError());
    if (i + 1 == dp) break;
    rc = apply_M(c, R, prec, precond, prod, t, st);
    if (!rc) rc = run_matvec_graph(c, R, prec, t, w, st);
    if (!rc) {
      k_caxpy<<<nb, 256, 0, st>>>(ld, make_double2(-inv.real(), -inv.imag()), w, prod);
      SMR_CUDA(c, cudaGetLastError());
      ++c->poly_mv;
    }
  }
  if (!rc) rc = apply_M(c, R, prec, precond, y, z, st);
  return rc;
}

static int apply_M(Ctx* c, int R, int prec, int precond, const double2* v, double2* z, cudaStream_t st) {
  const long long ld = 2LL * c->npsi * c->p * R;
  if (!c->poly_roots.empty() && !c->poly_busy) {
    c->poly_busy = true;                      // the base preconditioner inside
    int rc = apply_poly(c, R, prec, precond, v, z, st);
    c->poly_busy = false;
    return rc;
  }
  if (precond == SMR_PRECOND_NONE) {
    SMR_CUDA(c, cudaMemcpyAsync(z, v, (size_t)ld * sizeof(double2), cudaMemcpyDeviceToDevice, st));
    return SMR_OK;
  }
  if (precond == SMR_PRECOND_NEAR) {
    if (!c->d_pcw || c->pcw_elems < (size_t)3 * ld) {
      c->err = "near-field preconditioner work vectors missing";
      return SMR_E_STATE;
    }
    double2* t = c->d_pcw;                    // D^-1 v
    double2* y = c->d_pcw + ld;               // Z_near z
    double2* u = c->d_pcw + 2 * ld;           // D^-1 Z_near z
    int rc = run_precond(c, R, prec, v, t, st);
    if (rc) return rc;
    SMR_CUDA(c, cudaMemcpyAsync(z, t, (size_t)ld * sizeof(double2), cudaMemcpyDeviceToDevice, st));
    for (int k = 0; k < c->pc_sweeps && !rc; ++k) {
      c->x32_of = nullptr;                    // z changed: the FP32 copy of x is stale
      rc = run_near(c, R, prec, z, y, st);
      if (!rc) rc = run_precond(c, R, prec, y, u, st);
      if (!rc) {
        k_sweep_update<<<(unsigned)((ld + 255) / 256), 256, 0, st>>>(ld, z, t, u);
        SMR_CUDA(c, cudaGetLastError());
      }
    }
    return rc;
  }
  if (precond == SMR_PRECOND_CLUSTER) return run_cluster(c, R, prec, v, z, st);
  int rc = run_precond(c, R, prec, v, z, st);
  if (rc || precond != SMR_PRECOND_LEARNED) return rc;
  return lpc_apply(c, z, st);
}

static float elapsed_s(cudaEvent_t a, cudaEvent_t b) {
  float ms = 0;
  cudaEventElapsedTime(&ms, a, b);
  return ms * 1e-3f;
}

// One Gram-Schmidt pass of w against v_0..v_{J-1}: h = V^H w, w -= V h,
// *d_nr = ||w||^2 after the pass, and (when d_n0 is given) ||w||^2 before it.
static int gs_pass(Ctx* c, Work& W, int J, long long n, int R, long long ld, double2* d_h, float2* d_hf,
                   double2* d_n0, double2* d_nr, cudaStream_t st) {
  int rc;
  if (W.f32 && R == 1) {
    rc = gs32_dot(c, J, n, (const float2*)W.V, ld, W.w, d_h, d_hf, d_n0, W.part, st);
    if (rc) return rc;
    return gs32_axpy(c, J, n, (const float2*)W.V, ld, d_hf, W.w, -1.0, d_nr, W.part, st);
  }
  if (W.f32) {
    if (d_n0) {
      rc = multidot_dev(c, 1, n, R, W.w, 0, W.w, d_n0, W.part, st);
      if (rc) return rc;
    }
    int rl, nchunk;
    long long per;
    chunking(n, R, &rl, &nchunk, &per);
    dim3 g(nchunk, J);
    k_gsr_dot<<<g, 256, 0, st>>>(J, n, R, rl, nchunk, per, (const float2*)W.V, ld, W.w, W.part);
    SMR_LAUNCH(c);
    k_gsr_final<<<(J * R + 127) / 128, 128, 0, st>>>(J, R, nchunk, W.part, d_h, d_hf);
    SMR_LAUNCH(c);
    k_gsr_axpy<<<(unsigned)((ld + 255) / 256), 256, 0, st>>>(J, n, R, (const float2*)W.V, ld, d_hf, W.w, -1.0);
    SMR_LAUNCH(c);
    return multidot_dev(c, 1, n, R, W.w, 0, W.w, d_nr, W.part, st);
  }
  const double2* V = (const double2*)W.V;
  if (R == 1) {
    rc = gs_dot(c, J, n, V, ld, W.w, d_h, d_n0, W.part, st);
    if (rc) return rc;
    return gs_axpy(c, J, n, V, ld, d_h, W.w, -1.0, d_nr, W.part, st);
  }
  if (d_n0) {
    rc = multidot_dev(c, 1, n, R, W.w, 0, W.w, d_n0, W.part, st);
    if (rc) return rc;
  }
  rc = multidot_dev(c, J, n, R, V, ld, W.w, d_h, W.part, st);
  if (rc) return rc;
  rc = multi_axpy(c, J, n, R, V, ld, d_h, W.w, -1.0, st);
  if (rc) return rc;
  return multidot_dev(c, 1, n, R, W.w, 0, W.w, d_nr, W.part, st);
}

// Solve A d = rhs from d = d0 (in d) to per-column relative residual tol_col[r]
// (relative to ||rhs_r||) with right preconditioning, x = d0 + M^-1 V y;
// A and the preconditioner in precision `prec`.  Iterations add to *its.
static int gmres_core(Ctx* c, int R, int prec, int precond, const double2* rhs, double2* d,
                      bool have_d0, const std::vector<double>& tol_col, int maxit, int restart,
                      Work& W, int* its, int* nmv, int* n_reorth, std::vector<double>& rel_out,
                      cudaStream_t st, std::vector<std::complex<double>>* Hout = nullptr) {
  long long n = 2LL * c->npsi * c->p;
  long long ld = n * R;
  int m = restart;
  size_t eb = W.f32 ? sizeof(float2) : sizeof(double2);
  auto Vj = [&](int j) { return (void*)((char*)W.V + (size_t)j * ld * eb); };
  unsigned nb = (unsigned)((ld + 255) / 256);
  std::vector<double> bn(R), beta(R);
  int rc = col_norms(c, n, R, rhs, bn.data(), st);
  if (rc) return rc;
  for (int r = 0; r < R; ++r)
    if (bn[r] == 0.0) bn[r] = 1.0;
  // r0 = rhs - A d0  (in W.u)
  double2* r0 = W.u;
  auto residual = [&]() -> int {
    int e = apply_A(c, R, prec, d, W.w, st);
    if (e) return e;
    ++*nmv;
    SMR_CUDA(c, cudaMemcpyAsync(r0, rhs, ld * sizeof(double2), cudaMemcpyDeviceToDevice, st));
    std::vector<double2> mone(R, make_double2(-1, 0)), one(R, make_double2(1, 0));
    SMR_CUDA(c, cudaMemcpyAsync(W.coef, mone.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
    SMR_CUDA(c, cudaMemcpyAsync(W.coef + R, one.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
    e = col_axpby(n, R, W.coef, W.w, W.coef + R, r0, st);
    if (e) c->err = "axpby launch";
    return e;
  };
  if (have_d0) {
    rc = residual();
    if (rc) return rc;
  } else {
    SMR_CUDA(c, cudaMemcpyAsync(r0, rhs, ld * sizeof(double2), cudaMemcpyDeviceToDevice, st));
    SMR_CUDA(c, cudaMemsetAsync(d, 0, ld * sizeof(double2), st));
  }
  std::vector<int> done(R, 0);
  // columns whose Krylov space became invariant (Arnoldi breakdown); if the
  // true residual is still above the tolerance after that cycle's update,
  // no further iteration can lower it and the solve stops with BREAKDOWN
  std::vector<int> broke(R, 0);
  rel_out.assign(R, 1.0);
  // coefficient areas on the device
  double2* dh1 = W.coef;                                    // [m+1][R]
  double2* dh2 = W.coef + (size_t)(m + 1) * R;              // [m+1][R]
  double2* dnr = W.coef + (size_t)2 * (m + 1) * R;          // ||w'||^2  [R]
  double2* dn0 = dnr + R;                                   // ||w||^2   [R]
  double2* dsc = W.coef + (size_t)3 * (m + 1) * R;          // scale     [R]
  float2* dh1f = W.coef_f;
  float2* dh2f = W.coef_f + (size_t)(m + 1) * R;
  float2* dyf = W.coef_f + (size_t)2 * (m + 1) * R;
  // host Hessenberg storage (rotated), rotations, rhs g.  Column j of right-hand side
  // r has j + 2 entries and the columns are packed as they come: with the full
  // (m + 1) x m an unrestarted solve (m = maxit = 2,000) clears 64 MB for each
  // right-hand side, 3.6 ms each
  std::vector<std::complex<double>> H, g((size_t)(m + 1) * R);
  auto hcol = [&](int r, int j) { return (size_t)R * j * (j + 3) / 2 + (size_t)r * (j + 2); };
  std::vector<std::complex<double>> cs((size_t)m * R), sn((size_t)m * R);
  // pinned host mirror of the coefficient area; each iteration copies only
  // the live part (j + 1 coefficients per column and the two norms)
  double2* hbuf = W.hpin;
  const size_t onrm = (size_t)2 * (m + 1) * R;             // dnr, dn0 in the area
  // v_j <- a * src (per column a[r] on the device at dsc)
  auto store_basis = [&](int j, const double2* src) -> int {
    if (W.f32 && R == 1) k_narrow_scale<<<nb, 256, 0, st>>>(n, dsc, src, (float2*)Vj(j));
    else if (W.f32) k_narrow_scale_r<<<nb, 256, 0, st>>>(n, R, dsc, src, (float2*)Vj(j));
    else k_scale<<<nb, 256, 0, st>>>(n, R, dsc, src, (double2*)Vj(j));
    SMR_LAUNCH(c);
    return SMR_OK;
  };
  while (true) {
    rc = col_norms(c, n, R, r0, beta.data(), st);
    if (rc) return rc;
    bool all = true;
    for (int r = 0; r < R; ++r) {
      rel_out[r] = beta[r] / bn[r];
      if (!std::isfinite(beta[r])) { c->err = "NaN in residual"; return SMR_E_NAN; }
      if (rel_out[r] <= tol_col[r]) done[r] = 1;
      all = all && done[r];
    }
    for (int r = 0; r < R; ++r)
      if (broke[r] && !done[r]) {
        c->err = "Arnoldi breakdown: the Krylov space of right-hand side " + std::to_string(r) +
                 " became invariant with the true relative residual at " + std::to_string(rel_out[r]) +
                 " (singular or nearly singular operator)";
        return SMR_E_BREAKDOWN;
      }
    if (all || *its >= maxit) return all ? SMR_OK : SMR_E_NOT_CONVERGED;
    std::vector<double2> sc(R);
    for (int r = 0; r < R; ++r) sc[r] = make_double2(beta[r] > 0 ? 1.0 / beta[r] : 0.0, 0);
    SMR_CUDA(c, cudaMemcpyAsync(dsc, sc.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
    rc = store_basis(0, r0);
    if (rc) return rc;
    std::fill(g.begin(), g.end(), std::complex<double>(0, 0));
    for (int r = 0; r < R; ++r) g[(size_t)r * (m + 1)] = beta[r];
    std::vector<int> jend(R, 0), active(R, 0);
    for (int r = 0; r < R; ++r) active[r] = !done[r];
    int j = 0;
    for (; j < m && *its < maxit; ++j) {
      cudaEventRecord(W.ev[0], st);
      // t = M^-1 v_j (W.t has a fixed address, so one captured graph serves
      // every product of the solve)
      const double2* vj = (const double2*)Vj(j);
      if (W.f32) {
        k_widen<<<nb, 256, 0, st>>>(ld, (const float2*)Vj(j), W.u);
        SMR_LAUNCH(c);
        vj = W.u;
      }
      rc = apply_M(c, R, prec, precond, vj, W.t, st);
      if (rc) return rc;
      cudaEventRecord(W.ev[1], st);
      rc = run_matvec_graph(c, R, prec, W.t, W.w, st);
      if (rc) return rc;
      cudaEventRecord(W.ev[2], st);
      ++*nmv;
      ++*its;
      // classical Gram-Schmidt against v_0..v_j, repeated once when the norm
      // drops below 1/sqrt(10) of its value before the projection (a single
      // pass then loses at most ~3x the working precision in orthogonality);
      // the coefficients and norms are summed in FP64
      rc = gs_pass(c, W, j + 1, n, R, ld, dh1, dh1f, dn0, dnr, st);
      if (rc) return rc;
      cudaEventRecord(W.ev[3], st);
      SMR_CUDA(c, cudaMemcpyAsync(hbuf, W.coef, (size_t)(j + 1) * R * sizeof(double2), cudaMemcpyDeviceToHost, st));
      SMR_CUDA(c, cudaMemcpyAsync(hbuf + onrm, W.coef + onrm, (size_t)2 * R * sizeof(double2),
                                  cudaMemcpyDeviceToHost, st));
      SMR_CUDA(c, cudaStreamSynchronize(st));
      W.t_pc += elapsed_s(W.ev[0], W.ev[1]);
      W.t_mv += elapsed_s(W.ev[1], W.ev[2]);
      W.t_or += elapsed_s(W.ev[2], W.ev[3]);
      bool reorth = false;
      for (int r = 0; r < R; ++r) {
        double a0 = hbuf[(size_t)2 * (m + 1) * R + R + r].x, a1 = hbuf[(size_t)2 * (m + 1) * R + r].x;
        if (active[r] && a1 < 0.1 * a0) reorth = true;
      }
      if (reorth) {
        ++*n_reorth;
        cudaEventRecord(W.ev[4], st);
        rc = gs_pass(c, W, j + 1, n, R, ld, dh2, dh2f, nullptr, dnr, st);
        if (rc) return rc;
        cudaEventRecord(W.ev[5], st);
        SMR_CUDA(c, cudaMemcpyAsync(hbuf + (size_t)(m + 1) * R, dh2, (size_t)(j + 1) * R * sizeof(double2),
                                    cudaMemcpyDeviceToHost, st));
        SMR_CUDA(c, cudaMemcpyAsync(hbuf + onrm, dnr, (size_t)R * sizeof(double2), cudaMemcpyDeviceToHost, st));
        SMR_CUDA(c, cudaStreamSynchronize(st));
        W.t_or += elapsed_s(W.ev[4], W.ev[5]);
      } else {
        for (size_t q = 0; q < (size_t)(j + 1) * R; ++q) hbuf[(size_t)(m + 1) * R + q] = make_double2(0, 0);
      }
      // next basis vector v_{j+1} = w / ||w||
      std::vector<double2> inv(R);
      std::vector<double> hn(R);
      for (int r = 0; r < R; ++r) {
        const double n2 = hbuf[(size_t)2 * (m + 1) * R + r].x;
        hn[r] = std::isnan(n2) ? n2 : std::sqrt(std::max(0.0, n2));
        inv[r] = make_double2(hn[r] > 0 ? 1.0 / hn[r] : 0.0, 0);
      }
      SMR_CUDA(c, cudaMemcpyAsync(dsc, inv.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
      rc = store_basis(j + 1, W.w);
      if (rc) return rc;
      bool any = false;
      if (H.size() < hcol(0, j + 1)) H.resize(std::max(2 * H.size(), hcol(0, j + 1)));
      for (int r = 0; r < R; ++r) {
        if (!active[r]) continue;
        std::complex<double>* Hc = &H[hcol(r, j)];
        for (int i = 0; i <= j; ++i) {
          double2 a = hbuf[(size_t)i * R + r], b = hbuf[(size_t)(m + 1) * R + (size_t)i * R + r];
          Hc[i] = std::complex<double>(a.x + b.x, a.y + b.y);
        }
        Hc[j + 1] = hn[r];
        if (Hout && r == 0 && Hout->size() >= (size_t)(m + 1) * m)   // the unrotated column (first cycle)
          for (int i = 0; i <= j + 1; ++i) (*Hout)[(size_t)j * (m + 1) + i] = Hc[i];
        for (int i = 0; i < j; ++i) {
          std::complex<double> ci = cs[(size_t)r * m + i], si = sn[(size_t)r * m + i];
          std::complex<double> t = ci * Hc[i] + si * Hc[i + 1];
          Hc[i + 1] = -std::conj(si) * Hc[i] + ci * Hc[i + 1];
          Hc[i] = t;
        }
        std::complex<double> a = Hc[j], b = Hc[j + 1];
        double den = std::sqrt(std::norm(a) + std::norm(b));
        std::complex<double> ci, si;
        if (den == 0.0) { ci = 1.0; si = 0.0; }
        else if (std::abs(a) == 0.0) { ci = 0.0; si = std::conj(b) / std::abs(b); }
        else { ci = std::abs(a) / den; si = (a / std::abs(a)) * std::conj(b) / den; }
        cs[(size_t)r * m + j] = ci;
        sn[(size_t)r * m + j] = si;
        Hc[j] = ci * a + si * b;
        Hc[j + 1] = 0.0;
        std::complex<double>* gr = &g[(size_t)r * (m + 1)];
        gr[j + 1] = -std::conj(si) * gr[j];
        gr[j] = ci * gr[j];
        jend[r] = j + 1;
        double est = std::abs(gr[j + 1]) / bn[r];
        rel_out[r] = est;
        if (!std::isfinite(est)) { c->err = "NaN in Givens update"; return SMR_E_NAN; }
        // breakdown: the new direction vanishes against the norm of A M^-1 v_j
        // (exactly, or to 1e-13 of it in FP64, where projection noise is ~1e-16)
        const double w0 = std::sqrt(std::max(0.0, hbuf[(size_t)2 * (m + 1) * R + R + r].x));
        if (hn[r] == 0.0 || (!W.f32 && hn[r] <= 1e-13 * w0)) broke[r] = 1;
        if (est <= tol_col[r] || broke[r]) active[r] = 0;
        any = any || active[r];
      }
      if (!any) { ++j; break; }
    }
    // y per column by back substitution, then d += M^-1 (V y)
    int jmax = 0;
    for (int r = 0; r < R; ++r) jmax = std::max(jmax, jend[r]);
    std::vector<double2> ycoef((size_t)std::max(jmax, 1) * R, make_double2(0, 0));
    for (int r = 0; r < R; ++r) {
      int J = jend[r];
      std::vector<std::complex<double>> y(J);
      for (int i = J - 1; i >= 0; --i) {
        std::complex<double> s = g[(size_t)r * (m + 1) + i];
        for (int q = i + 1; q < J; ++q) s -= H[hcol(r, q) + i] * y[q];
        std::complex<double> diag = H[hcol(r, i) + i];
        y[i] = (diag != 0.0) ? s / diag : 0.0;
      }
      for (int i = 0; i < J; ++i) ycoef[(size_t)i * R + r] = make_double2(y[i].real(), y[i].imag());
    }
    if (jmax > 0) {
      SMR_CUDA(c, cudaMemsetAsync(W.w, 0, ld * sizeof(double2), st));
      if (W.f32) {
        std::vector<float2> yf((size_t)jmax * R);
        for (size_t i = 0; i < yf.size(); ++i) yf[i] = make_float2((float)ycoef[i].x, (float)ycoef[i].y);
        SMR_CUDA(c, cudaMemcpyAsync(dyf, yf.data(), yf.size() * sizeof(float2), cudaMemcpyHostToDevice, st));
        if (R == 1) {
          rc = gs32_axpy(c, jmax, n, (const float2*)W.V, ld, dyf, W.w, 1.0, nullptr, nullptr, st);
        } else {
          k_gsr_axpy<<<(unsigned)((ld + 255) / 256), 256, 0, st>>>(jmax, n, R, (const float2*)W.V, ld, dyf, W.w,
                                                                 1.0);
          rc = cudaGetLastError() == cudaSuccess ? SMR_OK : SMR_E_CUDA;
        }
      } else {
        SMR_CUDA(c, cudaMemcpyAsync(W.coef, ycoef.data(), (size_t)jmax * R * sizeof(double2),
                                    cudaMemcpyHostToDevice, st));
        rc = multi_axpy(c, jmax, n, R, (const double2*)W.V, ld, W.coef, W.w, 1.0, st);
      }
      if (rc) return rc;
      rc = apply_M(c, R, prec, precond, W.w, W.t, st);
      if (rc) return rc;
      std::vector<double2> one(R, make_double2(1, 0));
      SMR_CUDA(c, cudaMemcpyAsync(W.coef, one.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
      rc = col_axpby(n, R, W.coef, W.t, W.coef, d, st);
      if (rc) return rc;
    }
    // true residual of this operator
    rc = residual();
    if (rc) return rc;
  }
}

int solve(Ctx* c, int R, const double2* b, double2* x, const smr_solve_opts* o, smr_solve_stats* stats,
          cudaStream_t st) {
  auto t0 = std::chrono::steady_clock::now();
  long long n = 2LL * c->npsi * c->p;
  long long ld = n * R;
  int maxit = o->maxit > 0 ? o->maxit : 2000;
  int m = (o->restart > 0) ? std::min(o->restart, maxit) : maxit;
  // cap the Krylov dimension by device memory (60% of what is free); the
  // FP32 operator keeps its basis in FP32
  size_t freeb = 0, totb = 0;
  cudaMemGetInfo(&freeb, &totb);
  Work W;
  W.f32 = (o->precision == SMR_PREC_FP32 && n % 2 == 0);
  size_t eb = W.f32 ? sizeof(float2) : sizeof(double2);
  double per = (double)ld * eb;
  int mcap = (int)std::max(2.0, 0.6 * (double)freeb / per - 4);
  m = std::max(1, std::min(m, mcap));
  auto cleanup = [&]() {
    cudaFree(W.V); cudaFree(W.u); cudaFree(W.w); cudaFree(W.t); cudaFree(W.coef); cudaFree(W.coef_f);
    cudaFree(W.part);
    if (W.hpin) cudaFreeHost(W.hpin);
    for (int q = 0; q < 6; ++q)
      if (W.ev[q]) cudaEventDestroy(W.ev[q]);
  };
  bool ok = cudaMalloc(&W.V, (size_t)(m + 1) * ld * eb) == cudaSuccess &&
            cudaMalloc((void**)&W.u, ld * sizeof(double2)) == cudaSuccess &&
            cudaMalloc((void**)&W.w, ld * sizeof(double2)) == cudaSuccess &&
            cudaMalloc((void**)&W.t, ld * sizeof(double2)) == cudaSuccess &&
            cudaMalloc((void**)&W.coef, (size_t)4 * (m + 2) * R * sizeof(double2)) == cudaSuccess &&
            cudaMalloc((void**)&W.coef_f, (size_t)3 * (m + 2) * R * sizeof(float2)) == cudaSuccess &&
            cudaMalloc((void**)&W.part, part_elems(n, R, m + 2) * sizeof(double2)) == cudaSuccess &&
            cudaMallocHost((void**)&W.hpin, (size_t)(2 * (m + 1) + 2) * R * sizeof(double2)) == cudaSuccess;
  for (int q = 0; q < 6 && ok; ++q) ok = cudaEventCreate(&W.ev[q]) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    cleanup();
    c->err = "solve: device allocation of the Krylov workspace failed";
    return SMR_E_OOM;
  }
  int its = 0, mv64 = 0, mv32 = 0, outer = 0, nreo = 0, rc = SMR_OK;
  int fb_x0 = 0, fb_pc = 0, its_learned = 0;
  int precond = o->precond;
  const bool learned = precond == SMR_PRECOND_LEARNED && o->fallback_iters > 0;
  if (precond == SMR_PRECOND_NEAR) {
    c->pc_sweeps = o->near_sweeps;
    if (c->pcw_elems < (size_t)3 * ld) {
      if (c->d_pcw) cudaFree(c->d_pcw);
      c->d_pcw = nullptr;
      c->pcw_elems = 0;
      if (cudaMalloc((void**)&c->d_pcw, (size_t)3 * ld * sizeof(double2)) != cudaSuccess) {
        cudaGetLastError();
        cleanup();
        c->err = "solve: device allocation of the near-field preconditioner's work vectors failed";
        return SMR_E_OOM;
      }
      c->pcw_elems = (size_t)3 * ld;
    }
  }
  // polynomial preconditioner: roots from d Arnoldi steps on the operator the
  // iterations use (the FP32 one for the refinement), started from b
  c->poly_roots.clear();
  c->poly_mv = 0;
  int its_poly = 0;
  if (o->poly_degree >= 2 && R == 1) {
    const int dp = std::min(o->poly_degree, m);
    if (c->polyw_elems < (size_t)4 * ld) {
      if (c->d_polyw) cudaFree(c->d_polyw);
      c->d_polyw = nullptr;
      c->polyw_elems = 0;
      if (cudaMalloc((void**)&c->d_polyw, (size_t)4 * ld * sizeof(double2)) != cudaSuccess) {
        cudaGetLastError();
        cleanup();
        c->err = "solve: device allocation of the polynomial preconditioner's work vectors failed";
        return SMR_E_OOM;
      }
      c->polyw_elems = (size_t)4 * ld;
    }
    const int pprec = o->precision == SMR_PREC_FP64 ? SMR_PREC_FP64 : SMR_PREC_FP32;
    std::vector<zc> Hb((size_t)(dp + 1) * dp, zc(0, 0));
    std::vector<double> tnever(R, 0.0), relp(R);
    int mvp = 0, nrp = 0;
    double2* xp = c->d_polyw;                 // scratch solution of the Arnoldi run
    int rp = gmres_core(c, R, pprec, precond, b, xp, false, tnever, dp, dp, W, &its_poly, &mvp, &nrp, relp, st, &Hb);
    if (rp && rp != SMR_E_NOT_CONVERGED && rp != SMR_E_BREAKDOWN) {
      cleanup();
      return rp;
    }
    (pprec == SMR_PREC_FP64 ? mv64 : mv32) += mvp;
    std::vector<zc> th;
    const int deff = std::min(its_poly, dp);
    if (deff >= 2 && harmonic_ritz(deff, Hb, dp + 1, th)) {
      leja_order(th);
      c->poly_roots = th;
    }
  }
  std::vector<double> rel;
  double tol = o->tol > 0 ? o->tol : 1e-4;
  // columns of x set to a * x (a = 0 or 1 per column, host values)
  auto scale_cols = [&](double2* v, const std::vector<int>& keep) -> int {
    std::vector<double2> zero(R, make_double2(0, 0)), k(R);
    for (int q = 0; q < R; ++q) k[q] = make_double2(keep[q] ? 1.0 : 0.0, 0.0);
    SMR_CUDA(c, cudaMemcpyAsync(W.coef, zero.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
    SMR_CUDA(c, cudaMemcpyAsync(W.coef + R, k.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
    return col_axpby(n, R, W.coef, v, W.coef + R, v, st);
  };
  if (o->precision == SMR_PREC_FP64) {
    std::vector<double> tc(R, tol), rel0(R, 1.0);
    bool have_x0 = o->use_x0 != 0;
    if (have_x0) {
      // a guess worse than zero (true residual above ||b||) is dropped
      std::vector<double> bn(R), rn(R);
      rc = apply_A(c, R, SMR_PREC_FP64, x, W.w, st);
      ++mv64;
      std::vector<double2> mone(R, make_double2(-1, 0)), one(R, make_double2(1, 0));
      if (!rc) {
        SMR_CUDA(c, cudaMemcpyAsync(W.u, b, ld * sizeof(double2), cudaMemcpyDeviceToDevice, st));
        SMR_CUDA(c, cudaMemcpyAsync(W.coef, mone.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
        SMR_CUDA(c, cudaMemcpyAsync(W.coef + R, one.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
        rc = col_axpby(n, R, W.coef, W.w, W.coef + R, W.u, st);
      }
      if (!rc) rc = col_norms(c, n, R, b, bn.data(), st);
      if (!rc) rc = col_norms(c, n, R, W.u, rn.data(), st);
      std::vector<int> keep(R, 1);
      for (int q = 0; q < R && !rc; ++q) {
        const double bq = bn[q] > 0 ? bn[q] : 1.0;
        if (std::isfinite(rn[q]) && rn[q] > bq) { keep[q] = 0; ++fb_x0; }
        else rel0[q] = rn[q] / bq;
      }
      if (!rc && fb_x0) rc = scale_cols(x, keep);
    }
    if (!rc && learned) {
      // probe: up to fallback_iters iterations with the learned preconditioner
      rc = gmres_core(c, R, SMR_PREC_FP64, precond, b, x, have_x0, tc, std::min(maxit, o->fallback_iters), m, W,
                      &its, &mv64, &nreo, rel, st);
      its_learned = its;
      if (rc == SMR_E_NOT_CONVERGED) {
        bool dropped = true;
        for (int q = 0; q < R; ++q) dropped = dropped && rel[q] <= 0.1 * rel0[q];
        if (!dropped) { precond = SMR_PRECOND_BLOCKDIAG; fb_pc = 1; }
        have_x0 = true;
        rc = SMR_OK;
      } else if (rc == SMR_OK) {
        have_x0 = false;               // converged: skip the second call
        maxit = its;
      }
    }
    if (!rc && its < maxit) {
      const int its0 = its;
      rc = gmres_core(c, R, SMR_PREC_FP64, precond, b, x, have_x0, tc, maxit, m, W, &its, &mv64, &nreo, rel, st);
      if (precond == SMR_PRECOND_LEARNED) its_learned += its - its0;
    }
  } else {
    // iterative refinement: outer FP64 residual, inner GMRES on the FP32 operator
    double2 *r = nullptr, *dlt = nullptr;
    SMR_CUDA(c, cudaMalloc((void**)&r, ld * sizeof(double2)));
    SMR_CUDA(c, cudaMalloc((void**)&dlt, ld * sizeof(double2)));
    std::vector<double> bn(R), rn(R), rn_probe;
    rc = col_norms(c, n, R, b, bn.data(), st);
    if (!o->use_x0) SMR_CUDA(c, cudaMemsetAsync(x, 0, ld * sizeof(double2), st));
    int max_outer = o->max_outer > 0 ? o->max_outer : 8;
    bool probe = learned, check = false;
    while (rc == SMR_OK) {
      // r = b - A64 x
      if (outer == 0 && !o->use_x0) {
        SMR_CUDA(c, cudaMemcpyAsync(r, b, ld * sizeof(double2), cudaMemcpyDeviceToDevice, st));
      } else {
        rc = apply_A(c, R, SMR_PREC_FP64, x, W.w, st);
        if (rc) break;
        ++mv64;
        SMR_CUDA(c, cudaMemcpyAsync(r, b, ld * sizeof(double2), cudaMemcpyDeviceToDevice, st));
        std::vector<double2> mone(R, make_double2(-1, 0)), one(R, make_double2(1, 0));
        SMR_CUDA(c, cudaMemcpyAsync(W.coef, mone.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
        SMR_CUDA(c, cudaMemcpyAsync(W.coef + R, one.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
        rc = col_axpby(n, R, W.coef, W.w, W.coef + R, r, st);
        if (rc) break;
      }
      rc = col_norms(c, n, R, r, rn.data(), st);
      if (rc) break;
      if (outer == 0 && o->use_x0) {
        // a guess worse than zero (true residual above ||b||) is dropped:
        // x = 0 and r = b in those columns
        std::vector<int> keep(R, 1);
        for (int q = 0; q < R; ++q) {
          const double bq = bn[q] > 0 ? bn[q] : 1.0;
          if (std::isfinite(rn[q]) && rn[q] > bq) { keep[q] = 0; ++fb_x0; }
        }
        if (fb_x0) {
          if ((rc = scale_cols(x, keep))) break;
          std::vector<double2> a(R), bb(R);
          for (int q = 0; q < R; ++q) {
            a[q] = make_double2(keep[q] ? 0.0 : 1.0, 0.0);
            bb[q] = make_double2(keep[q] ? 1.0 : 0.0, 0.0);
            if (!keep[q]) rn[q] = bn[q];
          }
          SMR_CUDA(c, cudaMemcpyAsync(W.coef, a.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
          SMR_CUDA(c, cudaMemcpyAsync(W.coef + R, bb.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
          if ((rc = col_axpby(n, R, W.coef, b, W.coef + R, r, st))) break;
        }
      }
      if (check) {
        // the probe with the learned preconditioner must have cut the true
        // residual tenfold; otherwise the block-diagonal one takes over
        bool dropped = true;
        for (int q = 0; q < R; ++q) dropped = dropped && rn[q] <= 0.1 * rn_probe[q];
        if (!dropped) { precond = SMR_PRECOND_BLOCKDIAG; fb_pc = 1; }
        check = false;
      }
      bool finite = true;
      for (int q = 0; q < R; ++q) finite = finite && std::isfinite(rn[q]);
      if (!finite) {
        c->err = "NaN or Inf in the residual (right-hand side or initial guess)";
        rel.assign(R, std::nan(""));
        rc = SMR_E_NAN;
        break;
      }
      bool all = true;
      std::vector<double> tc(R);
      rel.assign(R, 0.0);
      for (int q = 0; q < R; ++q) {
        double bq = bn[q] > 0 ? bn[q] : 1.0;
        rel[q] = rn[q] / bq;
        all = all && rel[q] <= tol;
        // inner target: 90% of the remaining tolerance (the FP32 product error
        // is ~1e-6 relative, far below the rest)
        tc[q] = (rn[q] > 0) ? std::max(0.9 * tol * bq / rn[q], 1e-7) : 1.0;
      }
      if (all) break;
      if (outer >= max_outer || its >= maxit) { rc = SMR_E_NOT_CONVERGED; break; }
      std::vector<double> rel_in;
      int lim = maxit - its;
      if (probe) {
        lim = std::min(lim, o->fallback_iters);
        rn_probe = rn;
        probe = false;
        check = true;
      }
      const int its0 = its;
      int rci = gmres_core(c, R, SMR_PREC_FP32, precond, r, dlt, false, tc, its + lim, m, W,
                           &its, &mv32, &nreo, rel_in, st);
      if (precond == SMR_PRECOND_LEARNED) its_learned += its - its0;
      if (rci && rci != SMR_E_NOT_CONVERGED) { rc = rci; break; }
      std::vector<double2> one(R, make_double2(1, 0));
      SMR_CUDA(c, cudaMemcpyAsync(W.coef, one.data(), R * sizeof(double2), cudaMemcpyHostToDevice, st));
      rc = col_axpby(n, R, W.coef, dlt, W.coef, x, st);
      ++outer;
    }
    cudaFree(r);
    cudaFree(dlt);
  }
  SMR_CUDA(c, cudaStreamSynchronize(st));
  cleanup();
  if (stats) {
    stats->iters = its + its_poly;
    stats->matvecs_fp64 = mv64 + (o->precision == SMR_PREC_FP64 ? c->poly_mv : 0);
    stats->matvecs_fp32 = mv32 + (o->precision == SMR_PREC_FP64 ? 0 : c->poly_mv);
    stats->outer = outer;
    stats->reorth = nreo;
    stats->seconds_product = W.t_mv;
    stats->seconds_precond = W.t_pc;
    stats->seconds_orth = W.t_or;
    stats->fallback_x0 = fb_x0;
    stats->fallback_precond = fb_pc;
    stats->iters_learned = its_learned;
    double mx = 0;
    for (double v : rel) mx = (std::isnan(v) || std::isnan(mx)) ? std::nan("") : std::max(mx, v);
    stats->resid_true = mx;
    stats->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  }
  c->poly_roots.clear();
  return rc;
}

}  // namespace smr

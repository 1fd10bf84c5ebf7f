// Hot path of the MLFMA-SMR product (Sec. IV): near block-sparse product,
// aggregation, interpolation, translation, anterpolation and receive.
// Every kernel is templated on the arithmetic type (double / float); the
// unknown vectors stay complex FP64 and are converted on load / store.
//
// Layouts (complex, interleaved):
//   x, y              [p][2][n_psi][R]
//   patterns Pd, Pm   [S][2][n_psi][K0 / 2], [S][2][K0 / 2][n_psi]  (P_th +- j P_ph, Eq. 26)
//   spectra out/in    [n_box][K_s][NF][R]     circular fields (smr_internal.h)
//   translation T     [n_offset][K_s]         (Eq. 23)
//   self blocks       [S][2 n_psi (col j)][2 n_psi (row i)]  (transposed)
//   exterior blocks   [n_blk - S][n_psi (col j)][+, -][n_psi (row i)]  (k_near_rows)
#include <algorithm>

#include "smr_internal.h"

namespace smr {

template <typename T> struct CV;
template <> struct CV<double> { typedef double2 V; };
template <> struct CV<float> { typedef float2 V; };

__device__ __forceinline__ double2 mkc(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ float2 mkc(float a, float b) { return make_float2(a, b); }
template <typename V> __device__ __forceinline__ V czero();
template <> __device__ __forceinline__ double2 czero<double2>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ float2 czero<float2>() { return make_float2(0.f, 0.f); }
__device__ __forceinline__ double2 cvt2(double2 v, double2) { return v; }
__device__ __forceinline__ float2 cvt2(double2 v, float2) { return make_float2((float)v.x, (float)v.y); }
__device__ __forceinline__ float2 cvt2(float2 v, float2) { return v; }
__device__ __forceinline__ double2 to64(double2 v) { return v; }
__device__ __forceinline__ double2 to64(float2 v) { return make_double2(v.x, v.y); }

// acc += a * b
template <typename V> __device__ __forceinline__ void cfma(V& acc, V a, V b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}
// acc += conj(a) * b
template <typename V> __device__ __forceinline__ void cfmac(V& acc, V a, V b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(-a.y, b.x, acc.y);
}
// acc += w * b  (w real)
template <typename V, typename T> __device__ __forceinline__ void rfma(V& acc, T w, V b) {
  acc.x = fma(w, b.x, acc.x);
  acc.y = fma(w, b.y, acc.y);
}
template <typename V> __device__ __forceinline__ V cmul(V a, V b) {
  V r;
  r.x = a.x * b.x - a.y * b.y;
  r.y = a.x * b.y + a.y * b.x;
  return r;
}

// ------------------------------------------------------------------ 16-byte direction parts
// The gather kernels work on 16-byte parts of a direction (one field in FP64, two in
// FP32), so that a warp instruction reads or writes contiguous runs and shared memory
// is accessed without bank conflicts.  NT parts make the fields of one column.
template <typename T> struct Part;
template <> struct Part<double> {
  typedef double2 H;
  static constexpr int NT = NF;
  static __device__ __forceinline__ H zero() { return make_double2(0.0, 0.0); }
  static __device__ __forceinline__ void rfma(H& a, double w, H v) { a.x = fma(w, v.x, a.x); a.y = fma(w, v.y, a.y); }
  static __device__ __forceinline__ void cfma(H& a, double2 s, H v) {
    a.x = fma(s.x, v.x, a.x); a.x = fma(-s.y, v.y, a.x);
    a.y = fma(s.x, v.y, a.y); a.y = fma(s.y, v.x, a.y);
  }
  static __device__ __forceinline__ void add(H& a, H v) { a.x += v.x; a.y += v.y; }
  static __device__ __forceinline__ void w4(const double* p, double* w) {
    double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
    w[0] = a.x; w[1] = a.y; w[2] = b.x; w[3] = b.y;
  }
};
template <> struct Part<float> {
  typedef float4 H;
  static constexpr int NT = NF / 2;
  static __device__ __forceinline__ H zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ void rfma(H& a, float w, H v) {
    a.x = fmaf(w, v.x, a.x); a.y = fmaf(w, v.y, a.y); a.z = fmaf(w, v.z, a.z); a.w = fmaf(w, v.w, a.w);
  }
  static __device__ __forceinline__ void cfma(H& a, float2 s, H v) {
    a.x = fmaf(s.x, v.x, a.x); a.x = fmaf(-s.y, v.y, a.x);
    a.y = fmaf(s.x, v.y, a.y); a.y = fmaf(s.y, v.x, a.y);
    a.z = fmaf(s.x, v.z, a.z); a.z = fmaf(-s.y, v.w, a.z);
    a.w = fmaf(s.x, v.w, a.w); a.w = fmaf(s.y, v.z, a.w);
  }
  static __device__ __forceinline__ void add(H& a, H v) { a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w; }
  static __device__ __forceinline__ void w4(const float* p, float* w) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
  }
};
template <typename T>
__device__ __forceinline__ typename Part<T>::H ldp(const typename CV<T>::V* base, size_t dir, int h) {
  return reinterpret_cast<const typename Part<T>::H*>(base + dir * NF)[h];
}
template <typename T>
__device__ __forceinline__ void stp(typename CV<T>::V* base, size_t dir, int h, typename Part<T>::H v) {
  reinterpret_cast<typename Part<T>::H*>(base + dir * NF)[h] = v;
}

// ------------------------------------------------------------------ aggregation
// out0[mu][k][f][r] = shift * sum_n conj(P_f[s][n][k]) (e_n +- (j/z) m_n), e and m
// the particle's electric and magnetic coefficients, P_+- = P_th +- j P_ph.
// The modes are real, so the pattern of the opposite direction k' is the
// conjugate one: with P = a + j b and x = u + j v the sums of a u, b v, a v and
// b u give both directions, 8 real multiply-adds a mode and pair of directions
// (both fields) where 4 fields of every direction take 32.
// CTA = one column (particle, r) x 128 pairs of directions, the modes in two
// halves: what bounds it in FP64 is the FP64 rate, and a CTA per column keeps
// every SM at it from some 100 columns on (64 particles: 104 us on 16 CTAs of 16
// columns and 4 fields before, 12.3 us now; 1,600 particles 424 and 105 us).
constexpr int AGC_PAIRS = 128;
template <typename T>
__global__ void __launch_bounds__(2 * AGC_PAIRS) k_aggregate(
    int K0, int nph, int npsi, int R, int nchunk, const int* __restrict__ perm, const int* __restrict__ sid,
    const double2* __restrict__ x, const typename CV<T>::V* __restrict__ Pd, const double* __restrict__ dshift,
    int any_dshift, const double* __restrict__ khat, double k, double iz, typename CV<T>::V* __restrict__ out) {
  typedef typename CV<T>::V V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* xs = reinterpret_cast<V*>(smem_raw);          // [npsi][2]
  V* red = xs + 2 * npsi;                          // [2 halves][4][AGC_PAIRS]
  const int chunk = blockIdx.x % nchunk, col = blockIdx.x / nchunk;
  const int mu = perm[col / R], r = col % R, s = sid[mu];
  for (int n = threadIdx.x; n < npsi; n += blockDim.x) {
    const double2 e = x[((size_t)mu * 2 * npsi + n) * R + r], m = x[((size_t)mu * 2 * npsi + npsi + n) * R + r];
    xs[2 * n] = cvt2(make_double2(fma(-iz, m.y, e.x), fma(iz, m.x, e.y)), V());
    xs[2 * n + 1] = cvt2(make_double2(fma(iz, m.y, e.x), fma(-iz, m.x, e.y)), V());
  }
  __syncthreads();
  const int K2 = K0 / 2, kl = threadIdx.x % AGC_PAIRS, half = threadIdx.x / AGC_PAIRS;
  const int q = chunk * AGC_PAIRS + kl;
  {
    const V* Pp = Pd + (size_t)s * 2 * npsi * K2 + min(q, K2 - 1);
    const V* Pm = Pp + (size_t)npsi * K2;
    V ap = czero<V>(), bp = czero<V>(), am = czero<V>(), bm = czero<V>();   // a x, b x of both fields
#pragma unroll 4
    for (int n = half; n < npsi; n += 2) {
      const V p = Pp[(size_t)n * K2], m = Pm[(size_t)n * K2], xp = xs[2 * n], xm = xs[2 * n + 1];
      rfma(ap, p.x, xp);
      rfma(bp, p.y, xp);
      rfma(am, m.x, xm);
      rfma(bm, m.y, xm);
    }
    V* o = red + (size_t)half * 4 * AGC_PAIRS + kl;
    o[0] = ap; o[AGC_PAIRS] = bp; o[2 * AGC_PAIRS] = am; o[3 * AGC_PAIRS] = bm;
  }
  __syncthreads();
  if (q >= K2) return;
  V t[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const V a = red[i * AGC_PAIRS + kl], b = red[(4 + i) * AGC_PAIRS + kl];
    t[i] = mkc(a.x + b.x, a.y + b.y);
  }
  // one half of the threads takes the directions of the table, the other their opposites
  const T sg = half ? (T)-1 : (T)1;                // conj(P) x = (au + bv) + j (av - bu); P x the other signs
  V w0 = mkc(t[0].x + sg * t[1].y, t[0].y - sg * t[1].x), w1 = mkc(t[2].x + sg * t[3].y, t[2].y - sg * t[3].x);
  const int i = q / nph, j = q - i * nph;
  const int kk = half ? (K0 / nph - 1 - i) * nph + (j + nph / 2 < nph ? j + nph / 2 : j - nph / 2) : q;
  if (any_dshift) {
    const double* d = dshift + 3 * mu;
    const double* kh = khat + 3 * kk;
    double sn, cs;
    sincos(k * (kh[0] * d[0] + kh[1] * d[1] + kh[2] * d[2]), &sn, &cs);
    const V sh = mkc((T)cs, (T)sn);
    w0 = cmul(w0, sh);
    w1 = cmul(w1, sh);
  }
  V* o = out + ((size_t)mu * K0 + kk) * NF * R + r;
  o[0] = w0;
  o[R] = w1;
}

// ------------------------------------------------------------------ FP64 interpolation, one right-hand side
// The FP64 rate is the bound (two FP64 multiply-adds per clock and SM), and the
// theta pass first needs the fewest of them: it runs on the child's columns,
// and rows past a pole cost no extra passes.  CTA = (parent box, tile of TR parent theta rows);
// each thread owns up to EM1 parent direction parts of the tile across the
// loop over the children.  Per child: theta pass of the tile's rows into
// shared memory G[TR][nphC][NF] (4 taps, tables read as 16-byte vectors), then
// phi pass, shift and child sum in registers.
constexpr int EM1 = 6;                           // direction parts per thread, at most
__global__ void __launch_bounds__(256, 2) k_interp1(int nthP, int nphP, unsigned mP, int nphC, int Kc, int TR, int nrt,
                                                 const int* __restrict__ ch_ptr, const int* __restrict__ ch_idx,
                                                 const int* __restrict__ ch_quad, const int* __restrict__ th_pk,
                                                 const double* __restrict__ th_w,
                                                 const int* __restrict__ ph_src, const double* __restrict__ ph_w,
                                                 const double2* __restrict__ shift,
                                                 const double2* __restrict__ F,
                                                 double2* __restrict__ out) {
  typedef double T;
  typedef double2 V;
  typedef Part<T> P;
  typedef P::H H;
  constexpr int NT = P::NT, EM = EM1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* G = reinterpret_cast<V*>(smem_raw);           // [TR][nphC][NF]
  int B = blockIdx.x / nrt, rt = blockIdx.x - (blockIdx.x / nrt) * nrt;
  int tp0 = rt * TR, ntr = min(TR, nthP - tp0);
  int Kp = nthP * nphP;
  int nout = ntr * nphP * NT;
  int half = nphC >> 1;
  // (row, column) of this thread's tasks, stepped by the NTH tasks of one
  // sweep of the CTA without dividing per task
  const int NTH = blockDim.x / NT, task0 = threadIdx.x / NT, h = threadIdx.x % NT;
  const int trG0 = task0 / nphC, jG0 = task0 - trG0 * nphC;
  const int dqG = NTH / nphC, drG = NTH - dqG * nphC;
  H acc[EM];
#pragma unroll
  for (int i = 0; i < EM; ++i) acc[i] = P::zero();
  for (int e = ch_ptr[B]; e < ch_ptr[B + 1]; ++e) {
    const V* src = F + (size_t)ch_idx[e] * Kc * NF;
    const V* sh = shift + (size_t)ch_quad[e] * Kp + (size_t)tp0 * nphP;
    __syncthreads();
    for (int tr = trG0, j = jG0, task = task0; tr < ntr; task += NTH) {
      int tp = tp0 + tr;
      int jr = j + half;
      jr = jr >= nphC ? jr - nphC : jr;
      int4 pk = *reinterpret_cast<const int4*>(th_pk + tp * 4);
      T w[4];
      P::w4(th_w + tp * 4, w);
      H a = P::zero();
      P::rfma(a, w[0], ldp<T>(src, (size_t)(pk.x & 0xffff) * nphC + ((pk.x >> 16) ? jr : j), h));
      P::rfma(a, w[1], ldp<T>(src, (size_t)(pk.y & 0xffff) * nphC + ((pk.y >> 16) ? jr : j), h));
      P::rfma(a, w[2], ldp<T>(src, (size_t)(pk.z & 0xffff) * nphC + ((pk.z >> 16) ? jr : j), h));
      P::rfma(a, w[3], ldp<T>(src, (size_t)(pk.w & 0xffff) * nphC + ((pk.w >> 16) ? jr : j), h));
      stp<T>(G, task, h, a);
      j += drG;
      tr += dqG;
      if (j >= nphC) { j -= nphC; ++tr; }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < EM; ++i) {
      // task / nphP as a multiply-high by ceil(2^32 / nphP): exact while task * nphP < 2^32
      const unsigned task = (unsigned)(task0 + i * NTH);
      const int tr = (int)__umulhi(task, mP), jp = (int)task - tr * nphP;
      if (tr < ntr) {
        int4 cs = *reinterpret_cast<const int4*>(ph_src + jp * 4);
        T w[4];
        P::w4(ph_w + jp * 4, w);
        size_t rb = (size_t)tr * nphC;
        H sm = P::zero();
        P::rfma(sm, w[0], ldp<T>(G, rb + cs.x, h));
        P::rfma(sm, w[1], ldp<T>(G, rb + cs.y, h));
        P::rfma(sm, w[2], ldp<T>(G, rb + cs.z, h));
        P::rfma(sm, w[3], ldp<T>(G, rb + cs.w, h));
        P::cfma(acc[i], sh[tr * nphP + jp], sm);
      }
    }
  }
  V* dst = out + ((size_t)B * Kp + (size_t)tp0 * nphP) * NF;
#pragma unroll
  for (int i = 0; i < EM; ++i) {
    int t = threadIdx.x + i * blockDim.x;
    if (t < nout) stp<T>(dst, t / NT, t % NT, acc[i]);
  }
}
// ------------------------------------------------------------------ translation
// in[b][k] = sum_{(b', o) in IL(b)} T[o][k] out[b'][k]   (Eqs. 22-23)
// FP32, several columns (one column: k_translate.cu).  One CTA = 4x4 target boxes of the lattice x a chunk of directions; the 8x8
// source halo and the table rows of the chunk are staged in shared memory,
// so each source spectrum is fetched about 4 times instead of 27.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, int src_bytes) {
  unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(src_bytes));
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\n" ::);
  asm volatile("cp.async.wait_group 0;\n" ::);
}

__global__ void k_translate(int K, int R, int RC, int KC, int ntx, int ntile, const int* __restrict__ tiles,
                            int map_x0, int map_y0, int map_w, int map_h, int noff,
                            const int* __restrict__ boxmap, const int* __restrict__ offid,
                            const float2* __restrict__ Tt, const float2* __restrict__ out,
                            float2* __restrict__ in) {
  typedef float2 V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int nrc = (R + RC - 1) / RC;
  int tile = tiles[blockIdx.x % ntile];
  int rest = blockIdx.x / ntile;
  int rch = rest % nrc, kch = rest / nrc;
  int tx = tile % ntx, ty = tile / ntx;
  // absolute lattice origin of the tile, aligned to multiples of 4
  int ax0 = ((map_x0 >> 2) + tx) * 4, ay0 = ((map_y0 >> 2) + ty) * 4;
  int k0 = kch * KC, r0 = rch * RC;
  int nk = min(KC, K - k0), nr = min(RC, R - r0);
  int W = KC * NF * RC;                               // V per source box in the chunk
  V* S = reinterpret_cast<V*>(smem_raw);              // [64 sources][KC][NF][RC]
  V* Ts = S + 64 * W;                                 // [noff][KC]
  int* bid = reinterpret_cast<int*>(Ts + max(noff, 1) * KC);   // [64] source box ids
  int* tgt = bid + 64;                                // [16] target box ids
  int* cnt = tgt + 16;                                // [16] candidate counts
  int2* lst = reinterpret_cast<int2*>(cnt + 16);      // [16][27] (source slot, table row)
  for (int t = threadIdx.x; t < 64; t += blockDim.x) {
    int sx = ax0 - 2 + (t & 7), sy = ay0 - 2 + (t >> 3);
    int lx = sx - map_x0, ly = sy - map_y0;
    bid[t] = (lx >= 0 && ly >= 0 && lx < map_w && ly < map_h) ? boxmap[ly * map_w + lx] : -1;
  }
  __syncthreads();
  if (RC == R) {
    // each source box's chunk is contiguous in global memory: asynchronous
    // 16-byte copies, zero-filled for missing boxes and past the last direction
    int per = W * (int)sizeof(V) / 16;
    int valid = nk * NF * R * (int)sizeof(V);
    for (int t = threadIdx.x; t < 64 * per; t += blockDim.x) {
      int sb = t / per, pc = t - sb * per;
      int b = bid[sb];
      const char* g = reinterpret_cast<const char*>(out);
      int nb = 0;
      if (b >= 0 && pc * 16 < valid) {
        g += ((size_t)b * K + k0) * NF * R * sizeof(V) + (size_t)pc * 16;
        nb = 16;
      }
      cp_async16(reinterpret_cast<char*>(S + (size_t)sb * W) + pc * 16, g, nb);
    }
  } else if ((R * (int)sizeof(V)) % 16 == 0 && (RC * (int)sizeof(V)) % 16 == 0) {
    // asynchronous 16-byte copies of each (source, direction, field) run of RC
    // columns (aligned: R and RC span whole 16-byte pieces), zero-filled for
    // missing boxes, past the last direction and past the last column
    int pr = RC * (int)sizeof(V) / 16;               // pieces per run
    int per = KC * NF * pr;                          // pieces per source box
    for (int t = threadIdx.x; t < 64 * per; t += blockDim.x) {
      int sb = t / per, e = t - sb * per;
      int run = e / pr, pc = e - run * pr;           // run = kl * NF + f
      int kl = run / NF;
      int b = bid[sb];
      const char* g = reinterpret_cast<const char*>(out);
      int nb = 0;
      int col = pc * 16 / (int)sizeof(V);            // first column of the piece
      if (b >= 0 && kl < nk && col < nr) {
        g += ((((size_t)b * K + k0 + kl) * NF + run % NF) * R + r0) * sizeof(V) + (size_t)pc * 16;
        nb = 16;
      }
      cp_async16(reinterpret_cast<char*>(S + (size_t)sb * W + (size_t)run * RC) + pc * 16, g, nb);
    }
  } else {
    for (int t = threadIdx.x; t < 64 * W; t += blockDim.x) {
      int sb = t / W, e = t % W;
      int rl = e % RC, kl = e / (NF * RC), f = (e / RC) % NF;
      int b = bid[sb];
      S[t] = (b >= 0 && kl < nk && rl < nr) ? out[(((size_t)b * K + k0 + kl) * NF + f) * R + r0 + rl]
                                           : czero<V>();
    }
  }
  for (int t = threadIdx.x; t < noff * KC; t += blockDim.x) {
    int o = t / KC, kl = t % KC;
    Ts[t] = (kl < nk) ? Tt[(size_t)o * K + k0 + kl] : czero<V>();
  }
  if (threadIdx.x < 16) {
    int tg = threadIdx.x;
    int ix = ax0 + (tg & 3), iy = ay0 + (tg >> 2);
    int lx = ix - map_x0, ly = iy - map_y0;
    int b = (lx >= 0 && ly >= 0 && lx < map_w && ly < map_h) ? boxmap[ly * map_w + lx] : -1;
    tgt[tg] = b;
    int n = 0;
    if (b >= 0) {
      int px = ix >> 1, py = iy >> 1;
      for (int cy = 2 * py - 2; cy <= 2 * py + 3; ++cy)
        for (int cx = 2 * px - 2; cx <= 2 * px + 3; ++cx) {
          int dx = ix - cx, dy = iy - cy;
          if (dx >= -1 && dx <= 1 && dy >= -1 && dy <= 1) continue;
          int sb = (cy - ay0 + 2) * 8 + (cx - ax0 + 2);
          int o = offid[(dx + 3) * 7 + (dy + 3)];
          if (bid[sb] < 0 || o < 0 || n >= 27) continue;
          lst[tg * 27 + n] = make_int2(sb * W, o * KC);
          ++n;
        }
    }
    cnt[tg] = n;
  }
  cp_async_wait_all();
  __syncthreads();
  // outputs: 16 targets x nk directions x nr columns, NF fields each
  int nout = 16 * nk * nr;
  for (int t = threadIdx.x; t < nout; t += blockDim.x) {
    int rl = t % nr, kl = (t / nr) % nk, tg = t / (nr * nk);
    int b = tgt[tg];
    if (b < 0) continue;
    V acc[NF] = {czero<V>(), czero<V>()};
    int n = cnt[tg];
    const int2* L = lst + tg * 27;
    int kr = kl * NF * RC + rl;
    for (int e = 0; e < n; ++e) {
      int2 so = L[e];
      V tv = Ts[so.y + kl];
      const V* sv = S + so.x + kr;
      cfma(acc[0], tv, sv[0]);
      cfma(acc[1], tv, sv[RC]);
    }
    V* o = in + ((size_t)b * K + k0 + kl) * NF * R + r0 + rl;
    for (int f = 0; f < NF; ++f) o[f * R] = acc[f];
  }
}

// FP64, straight from the interaction lists: thread = one complex value (direction,
// field, column) of one target box, the sources' values and the factors read through
// the L2.  Bound by the FP64 rate: 32 bytes for four FP64 multiply-adds are no burden
// at two of them per clock and SM, so nothing has to be staged, and every level
// splits into enough CTAs.  Levels of the 40x40 array 170 + 143 + 133 + 39 + 18 us in
// kernels that staged 8x8 tiles or ran along the directions of 8 boxes, 141 + 90 + 51 +
// 27 + 14 now; 8x8 87 -> 22; 200x200 10.6 -> 9.6 ms; four right-hand sides on 20x20 337
// -> 247 us.  il_pk: source box * 64 + table row.
__global__ void __launch_bounds__(128) k_translate_il(int K, int NR, int nch, const int* __restrict__ il_ptr,
                                                      const int* __restrict__ il_pk, const double2* __restrict__ Tg,
                                                      const double2* __restrict__ out, double2* __restrict__ in) {
  const int b = blockIdx.x / nch;
  const unsigned n = (unsigned)K * NR, e = (blockIdx.x - b * nch) * 128u + threadIdx.x;
  if (e >= n) return;
  const unsigned k = e / NR;
  const int l1 = il_ptr[b + 1];
  double2 a = make_double2(0.0, 0.0);
#pragma unroll 6
  for (int l = il_ptr[b]; l < l1; ++l) {
    const int pk = __ldg(il_pk + l);
    cfma(a, __ldg(Tg + (size_t)(pk & 63) * K + k), __ldg(out + (size_t)(pk >> 6) * n + e));
  }
  in[(size_t)b * n + e] = a;
}

// ------------------------------------------------------------------ anterpolation by gathering
// For the levels where it is ahead of the marching kernel (gather_anterp).
// Both adjoint passes fused.  CTA = (child c, tile of
// child theta rows [i0, i0 + TI), column chunk [j0, j0 + JC) of the first
// half of the phi grid together with the same chunk shifted by N/2, so that
// the pole reflection j -> j + N/2 stays inside the CTA), one right-hand side
// per blockIdx.y (MC).  The parent rows
// [lo, hi) the tile draws on get the phi-transposed pass (conjugate shift and
// parent theta weight) into shared memory; then the theta-transposed pass adds
// into the child's incoming spectrum.  A thread takes all fields of a direction.
// Transposed taps are padded to PM / TM
// per child column / row (zero weights), packed as (tp | refl << 16).
// PMC > 0: tap tables padded to 8 per row (PM = TM = 8) and at most PMC
// real taps per row, known at compile time (tap loops unrolled)
template <typename T, int PMC, bool MC>
__global__ void __launch_bounds__(256) k_anterp1(int nthC, int nphC, int nthP, int nphP, int R, int TI, int nit,
                                                 int JC, int njc, const int* __restrict__ parent,
                                                 const int* __restrict__ quad, const int* __restrict__ lo_row,
                                                 int PM, const int* __restrict__ pjp, const T* __restrict__ pw,
                                                 const T* __restrict__ wthp,
                                                 const typename CV<T>::V* __restrict__ shift,
                                                 const typename Part<T>::H* __restrict__ inP, int TM,
                                                 const int* __restrict__ ttp, const T* __restrict__ tw,
                                                 typename Part<T>::H* __restrict__ inC) {
  typedef typename CV<T>::V V;
  typedef Part<T> P;
  typedef typename P::H H;
  constexpr int NT = P::NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  H* Gt = reinterpret_cast<H*>(smem_raw);          // [GR][2 JC][NT]
  const int nt = MC ? NT * R : NT;                 // parts of a direction
  int blk = blockIdx.x;
  int jcb = blk % njc;
  blk /= njc;
  int it = blk % nit, c = blk / nit;
  int i0 = it * TI, ni = min(TI, nthC - i0);
  int half = nphC >> 1;
  int j0 = jcb * JC, nj = min(JC, half - j0);
  int lo = lo_row[it], hi = lo_row[nit + it];
  int nr = hi - lo, W = 2 * nj;
  int Kp = nthP * nphP, Kc = nthC * nphC;
  const H* srcP = inP + (size_t)parent[c] * Kp * nt;
  if (MC) {
    srcP += blockIdx.y * NT;
    inC += blockIdx.y * NT;
  }
  const V* sh = shift + (size_t)quad[c] * Kp;
  // (row, column) of a thread's tasks stepped by the tasks of one sweep of the
  // CTA without dividing per task
  const int NTH = blockDim.x, task0 = threadIdx.x;
  const int r0 = task0 / W, u0 = task0 - r0 * W;
  const int dq = NTH / W, dr = NTH - dq * W;
  for (int r = r0, u = u0, task = task0; r < nr; task += NTH) {
    int j = (u < nj) ? j0 + u : j0 + half + (u - nj);
    int tp = lo + r;
    T wt = wthp[tp];
    const H* prow = srcP + (size_t)tp * nphP * nt;
    const V* srow = sh + (size_t)tp * nphP;
    H a[NT];
#pragma unroll
    for (int h = 0; h < NT; ++h) a[h] = P::zero();
    const int pm = PMC > 0 ? 8 : PM;
#pragma unroll
    for (int q = 0; q < (PMC > 0 ? PMC : PM); q += 4) {
      int4 jj = *reinterpret_cast<const int4*>(pjp + (size_t)j * pm + q);
      T w[4];
      P::w4(pw + (size_t)j * pm + q, w);
      int js[4] = {jj.x, jj.y, jj.z, jj.w};
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        if (PMC > 0 && q + b >= PMC) break;
        V s = srow[js[b]];
        T ww = w[b] * wt;
        const V cw = mkc(ww * s.x, -ww * s.y);
#pragma unroll
        for (int h = 0; h < NT; ++h) P::cfma(a[h], cw, prow[(size_t)js[b] * nt + h]);
      }
    }
#pragma unroll
    for (int h = 0; h < NT; ++h) Gt[task * NT + h] = a[h];
    u += dr;
    r += dq;
    if (u >= W) { u -= W; ++r; }
  }
  __syncthreads();
  for (int il = r0, u = u0; il < ni;) {
    int ur = u < nj ? u + nj : u - nj;             // column j + N/2 (mod N)
    int j = (u < nj) ? j0 + u : j0 + half + (u - nj);
    int i = i0 + il;
    H a[NT];
#pragma unroll
    for (int h = 0; h < NT; ++h) a[h] = P::zero();
    const int tm = PMC > 0 ? 8 : TM;
#pragma unroll
    for (int q = 0; q < (PMC > 0 ? PMC : TM); q += 4) {
      int4 pk = *reinterpret_cast<const int4*>(ttp + (size_t)i * tm + q);
      T w[4];
      P::w4(tw + (size_t)i * tm + q, w);
      int ps[4] = {pk.x, pk.y, pk.z, pk.w};
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        if (PMC > 0 && q + b >= PMC) break;
        int r = (ps[b] & 0xffff) - lo;
        const H* g = Gt + (size_t)(r * W + ((ps[b] >> 16) ? ur : u)) * NT;
#pragma unroll
        for (int h = 0; h < NT; ++h) P::rfma(a[h], w[b], g[h]);
      }
    }
    H* d = inC + ((size_t)c * Kc + (size_t)i * nphC + j) * nt;
#pragma unroll
    for (int h = 0; h < NT; ++h) {
      H cur = d[h];
      P::add(cur, a[h]);
      d[h] = cur;
    }
    u += dr;
    il += dq;
    if (u >= W) { u -= W; ++il; }
  }
}
// ------------------------------------------------------------------ receive
// Y_f[n] = sum_k w conj(sh) P_f[n][k] W_f[k];  y_e += -jk z (Y_+ + Y_-) / 2,
// y_m += -(k / 2) (Y_+ - Y_-)   (Eqs. 24-25 in the circular components).
// Opposite directions k, k' together: P W + conj(P) W' = a (W + W') + j b (W - W'),
// 8 real multiply-adds a mode and pair of directions.  CTA = one column; threads
// are (mode, every KS-th pair), the sums and differences of 64 pairs staged in
// shared memory.  Bound by the FP64 rate (64 particles 426 us on 4 CTAs of 16
// columns and 4 fields before, 16.4 us now; 1,600 particles 543 and 102 us).
constexpr int RCV_PAIRS = 64;
template <typename T>
__global__ void k_receive(int K0, int nph, int npsi, int R, const int* __restrict__ perm, const int* __restrict__ sid,
                          const typename CV<T>::V* __restrict__ in0, const typename CV<T>::V* __restrict__ Pm,
                          const double* __restrict__ w0, const double* __restrict__ dshift, int any_dshift,
                          const double* __restrict__ khat, double k, double zeta, double2* __restrict__ y,
                          int accumulate) {
  typedef typename CV<T>::V V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* sd = reinterpret_cast<V*>(smem_raw);          // [RCV_PAIRS][2 fields][sum, difference]
  V* red = sd + 4 * RCV_PAIRS;                     // [2 fields][threads]
  const int mu = perm[blockIdx.x / R], r = blockIdx.x % R, s = sid[mu];
  const int K2 = K0 / 2, KS = blockDim.x / npsi, m = threadIdx.x % npsi, ks = threadIdx.x / npsi;
  const V* Pp = Pm + (size_t)s * 2 * K2 * npsi + m;
  const V* Pn = Pp + (size_t)K2 * npsi;
  V yp = czero<V>(), yn = czero<V>();
  for (int q0 = 0; q0 < K2; q0 += RCV_PAIRS) {
    const int nq = min(RCV_PAIRS, K2 - q0);
    __syncthreads();
    for (int t = threadIdx.x; t < 2 * nq; t += blockDim.x) {
      const int f = t & 1, q = q0 + (t >> 1), i = q / nph, j = q - i * nph;
      const int kk = (K0 / nph - 1 - i) * nph + (j + nph / 2 < nph ? j + nph / 2 : j - nph / 2);
      V a = in0[(((size_t)mu * K0 + q) * NF + f) * R + r], b = in0[(((size_t)mu * K0 + kk) * NF + f) * R + r];
      if (any_dshift) {
        const double* d = dshift + 3 * mu;
        const double* kh = khat + 3 * q;
        double sn, cs;
        sincos(-k * (kh[0] * d[0] + kh[1] * d[1] + kh[2] * d[2]), &sn, &cs);
        a = cmul(a, mkc((T)cs, (T)sn));
        b = cmul(b, mkc((T)cs, (T)-sn));
      }
      const T w = (T)w0[q];
      sd[2 * t] = mkc(w * (a.x + b.x), w * (a.y + b.y));
      sd[2 * t + 1] = mkc(w * (a.x - b.x), w * (a.y - b.y));
    }
    __syncthreads();
#pragma unroll 4
    for (int q = ks; q < nq; q += KS) {
      const V p = Pp[(size_t)(q0 + q) * npsi], n = Pn[(size_t)(q0 + q) * npsi];
      const V* c = sd + 4 * q;
      rfma(yp, p.x, c[0]);
      yp.x = fma(-p.y, c[1].y, yp.x);
      yp.y = fma(p.y, c[1].x, yp.y);
      rfma(yn, n.x, c[2]);
      yn.x = fma(-n.y, c[3].y, yn.x);
      yn.y = fma(n.y, c[3].x, yn.y);
    }
  }
  red[threadIdx.x] = yp;
  red[blockDim.x + threadIdx.x] = yn;
  __syncthreads();
  if (ks) return;
  for (int t = 1; t < KS; ++t) {
    const V a = red[t * npsi + m], b = red[blockDim.x + t * npsi + m];
    yp.x += a.x; yp.y += a.y;
    yn.x += b.x; yn.y += b.y;
  }
  const double h = 0.5 * k, hz = h * zeta;
  const double2 p = to64(yp), n = to64(yn);
  double2 oe = make_double2(hz * (p.y + n.y), -hz * (p.x + n.x));
  double2 om = make_double2(-h * (p.x - n.x), -h * (p.y - n.y));
  double2* pe = y + ((size_t)mu * 2 * npsi + m) * R + r;
  double2* pm = pe + (size_t)npsi * R;
  if (accumulate) {
    const double2 a = *pe, b = *pm;
    oe.x += a.x; oe.y += a.y; om.x += b.x; om.y += b.y;
  }
  *pe = oe;
  *pm = om;
}

// ------------------------------------------------------------------ near product
// y[mu] = sum_{e in row mu} B[blk_e] x[col_e].  An exterior block [z T, K; -K, T / z]
// couples the circular combinations x_+- = e +- (j/z) m and Y_+- = y_e / z +- j y_m
// only with themselves, Y_+- = (T -+ j K) x_+-: half the multiply-adds and half the
// block.  Self blocks (blk < S) carry the interior medium as well and stay whole.
// CTA = one row (particle, r); threads are (output row, every KS-th column), the
// vectors of up to NR_PAIRS pairs staged in shared memory.  Bound in FP64 by the
// FP64 rate (1,600 particles 428 -> 236 us, 64 particles 94 -> 27), with one block a pair (displaced particles) by the blocks' bytes
// (24x24 in FP32 84.6 -> 27.5 us).
constexpr int NR_PAIRS = 9;
template <typename T, typename XV>
__global__ void k_near_rows(int n, int R, int S, const int* __restrict__ ptr, const int* __restrict__ col,
                            const int* __restrict__ blk, const typename CV<T>::V* __restrict__ Bs,
                            const typename CV<T>::V* __restrict__ Bc, double zeta, const XV* __restrict__ x,
                            double2* __restrict__ y) {
  typedef typename CV<T>::V V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n2 = 2 * n, KS = blockDim.x / n2, t = threadIdx.x % n2, ks = threadIdx.x / n2;
  V* xs = reinterpret_cast<V*>(smem_raw);          // [NR_PAIRS][2][n]: + and -, or e and m
  V* red = xs + NR_PAIRS * n2;                     // [2][threads]
  const int mu = blockIdx.x / R, r = blockIdx.x % R;
  const double iz = 1.0 / zeta;
  const int sg = t >= n ? n : 0;                   // this row's circular component
  V full = czero<V>(), circ = czero<V>();
  const int e1 = ptr[mu + 1];
  for (int e0 = ptr[mu]; e0 < e1; e0 += NR_PAIRS) {
    const int ne = min(NR_PAIRS, e1 - e0);
    __syncthreads();
    for (int u = threadIdx.x; u < ne * n; u += blockDim.x) {
      const int q = u / n, j = u - q * n;
      const XV* xv = x + (size_t)col[e0 + q] * n2 * R + r;
      const double2 a = to64(xv[(size_t)j * R]), b = to64(xv[(size_t)(n + j) * R]);
      const bool self = blk[e0 + q] < S;
      xs[q * n2 + j] = cvt2(self ? a : make_double2(fma(-iz, b.y, a.x), fma(iz, b.x, a.y)), V());
      xs[q * n2 + n + j] = cvt2(self ? b : make_double2(fma(iz, b.y, a.x), fma(-iz, b.x, a.y)), V());
    }
    __syncthreads();
    for (int q = 0; q < ne; ++q) {
      const int b = blk[e0 + q];
      if (b < S) {
        const V* B = Bs + (size_t)b * n2 * n2 + t;
#pragma unroll 4
        for (int j = ks; j < n2; j += KS) cfma(full, B[(size_t)j * n2], xs[q * n2 + j]);
      } else {
        const V* B = Bc + (size_t)(b - S) * n * n2 + t;
#pragma unroll 8
        for (int j = ks; j < n; j += KS) cfma(circ, B[(size_t)j * n2], xs[q * n2 + sg + j]);
      }
    }
  }
  red[threadIdx.x] = full;
  red[blockDim.x + threadIdx.x] = circ;
  __syncthreads();
  if (threadIdx.x >= n) return;
  double2 f[2] = {}, c[2] = {};
  for (int h = 0; h < 2; ++h)
    for (int k = 0; k < KS; ++k) {
      const double2 a = to64(red[k * n2 + h * n + t]), b = to64(red[blockDim.x + k * n2 + h * n + t]);
      f[h].x += a.x; f[h].y += a.y;
      c[h].x += b.x; c[h].y += b.y;
    }
  const double hz = 0.5 * zeta;
  double2* o = y + ((size_t)mu * n2 + t) * R + r;
  o[0] = make_double2(fma(hz, c[0].x + c[1].x, f[0].x), fma(hz, c[0].y + c[1].y, f[0].y));
  o[(size_t)n * R] = make_double2(fma(0.5, c[0].y - c[1].y, f[1].x), fma(-0.5, c[0].x - c[1].x, f[1].y));
}

// ------------------------------------------------------------------ block-sparse product
// y[mu][i][r] (+)= sum_{e in row mu} sum_j B[blk_e][i][j] x[col_e][j][r]
template <typename T>
__global__ void k_blocksparse(int nrow, int n2, int R, int rc, int nrc, const int* __restrict__ ptr,
                              const int* __restrict__ col, const int* __restrict__ blk,
                              const typename CV<T>::V* __restrict__ Bt,
                              const double2* __restrict__ x, double2* __restrict__ y,
                              int accumulate) {
  typedef typename CV<T>::V V;
  extern __shared__ unsigned char smem_raw[];
  V* xs = reinterpret_cast<V*>(smem_raw);            // [n2][rc]
  int mu = blockIdx.x / nrc, r0 = (blockIdx.x % nrc) * rc;
  int nr = min(rc, R - r0);
  int i = threadIdx.x / rc, rl = threadIdx.x % rc;
  bool active = (i < n2) && (rl < nr);
  V acc = czero<V>();
  for (int e = ptr[mu]; e < ptr[mu + 1]; ++e) {
    const double2* xv = x + (size_t)col[e] * n2 * R + r0;
    __syncthreads();
    for (int t = threadIdx.x; t < n2 * nr; t += blockDim.x) {
      int jl = t / nr, q = t % nr;
      xs[jl * rc + q] = cvt2(xv[(size_t)jl * R + q], V());
    }
    __syncthreads();
    if (active) {
      const V* Bb = Bt + (size_t)blk[e] * n2 * n2 + i;
      for (int j = 0; j < n2; ++j) cfma(acc, Bb[(size_t)j * n2], xs[j * rc + rl]);
    }
  }
  if (!active) return;
  double2* yp = y + ((size_t)mu * n2 + i) * R + r0 + rl;
  double2 o = to64(acc);
  if (accumulate) {
    double2 a = *yp;
    o.x += a.x;
    o.y += a.y;
  }
  *yp = o;
}

// ------------------------------------------------------------------ host drivers
// Destroys the captured products for which stale(entry) holds: a graph replays on the
// addresses of its capture, so it goes before the buffers it was built on do.
template <typename F> static void drop_graphs(Ctx* c, F stale) {
  for (size_t i = 0; i < c->graphs.size();) {
    if (stale(c->graphs[i])) {
      cudaGraphExecDestroy(c->graphs[i].exec);
      c->graphs.erase(c->graphs.begin() + i);
    } else {
      ++i;
    }
  }
}
// products that run column by column, on d_split and the lanes' buffers
static void drop_split_graphs(Ctx* c) {
  drop_graphs(c, [](const Ctx::GraphEntry& g) { return g.prec == SMR_PREC_FP32 && g.R > 1; });
}

int ensure_spectra(Ctx* c, int R, int prec) {
  int p = (prec == SMR_PREC_FP64) ? 0 : 1;
  if (c->buf_R[p] != R) {
    // (re)allocate this precision's spectra; graphs built on them are dropped
    drop_graphs(c, [&](const Ctx::GraphEntry& g) { return g.prec == prec; });
    size_t es = (p == 0) ? sizeof(double2) : sizeof(float2);
    c->buf_R[p] = 0;
    for (int s = 0; s < c->nlev; ++s) {
      Level& L = c->lev[s];
      if (L.buf_out[p]) cudaFree(L.buf_out[p]);
      if (L.buf_in[p]) cudaFree(L.buf_in[p]);
      L.buf_out[p] = L.buf_in[p] = nullptr;
      size_t bytes = (size_t)L.nbox * L.K * NF * R * es;
      if (cudaMalloc(&L.buf_out[p], bytes) != cudaSuccess || cudaMalloc(&L.buf_in[p], bytes) != cudaSuccess) {
        c->err = "out of device memory for level spectra";
        c->spec_prec = -1;
        return SMR_E_OOM;
      }
      L.buf_bytes[p] = bytes;
    }
    if (c->pspec[p]) cudaFree(c->pspec[p]);
    c->pspec[p] = nullptr;
    if ((c->multi || c->any_dshift) &&
        cudaMalloc(&c->pspec[p], (size_t)c->p * c->lev[0].K * NF * R * es) != cudaSuccess) {
      c->err = "out of device memory for the per-particle spectra";
      c->spec_prec = -1;
      return SMR_E_OOM;
    }
    if (c->d_xs[p]) cudaFree(c->d_xs[p]);
    c->d_xs[p] = nullptr;
    if (cudaMalloc((void**)&c->d_xs[p], (size_t)c->p * 2 * c->npsi * R * sizeof(double2)) != cudaSuccess) {
      cudaGetLastError();
      c->err = "out of device memory for the spectra's coefficients";
      c->spec_prec = -1;
      return SMR_E_OOM;
    }
    c->buf_R[p] = R;
  }
  for (auto& L : c->lev) {
    L.d_out = L.buf_out[p];
    L.d_in = L.buf_in[p];
    L.spec_bytes = L.buf_bytes[p];
  }
  c->spec_R = R;
  c->spec_prec = prec;
  return SMR_OK;
}

// FP64, one right-hand side: the gather kernels above, or the marching kernels
// (k_march.cu) where they do less.  All are bound by the FP64 rate.
// Interpolation: the gather kernel does fewer operations (200x200 lens, level
// 0: 1.57 ms against 2.16 ms).  Anterpolation: the marching kernel does fewer, but a
// CTA costs some seven rows more than it has and short rows leave it few threads.
// On rows of 22 columns (level 0) the gather kernel is ahead at every size (60x60
// 256 against 272 us, 200x200 2.74 against 2.84 ms), on 36 columns up to some 2
// million parent directions (boxes x K; 100x100 448 against 510 us, 200x200 1.75
// against 1.63 ms), on longer rows up to 240,000 (40x40 68 against 84 us at 139,000,
// 60x60 147 against 133 us at 248,000).
static bool march_interp(int v) { return v > 2; }
static bool march_anterp(const Level& Lc, const Level& Lp, int v) {
  if (v != 0) return v > 2;
  return Lc.nph > 24 && (size_t)Lp.nbox * Lp.K >= (Lc.nph <= 40 ? 2000000u : 240000u);
}
// FP32, or several columns: the marching kernel but for stencils wider than it is
// compiled for (ant_wide), whose taps its threads walk one by one for every parent row
// in turn, a chain that few boxes cannot hide.  The gather kernel's time grows with the
// child boxes and the columns, the chain's with the taps: they cross near nbox K_p R =
// 300,000 taps (FP32, orders 10 -> 38: 576 boxes 35 us against 78, 2,304 boxes 113
// against 98; 16 -> 68: 144 boxes 43 against 104, 576 boxes 127 against 115; 2 -> 68:
// 144 boxes 37 against 950; FP64, three columns, 4 -> 17: 576 boxes 125 against 227;
// 12 -> 48: 576 boxes 798 against 650).  In FP64 rows of up to 10 columns leave the
// marching kernel too few threads at any size (2 -> 11, 25,600 boxes, three columns:
// 3.05 against 4.93 ms).
constexpr size_t ANT_SMEM = 200 * 1024;
static bool gather_anterp(const Level& Lc, const Level& Lp, bool f64, int R, int v) {
  if (f64 && R == 1) return !march_anterp(Lc, Lp, v);
  const bool few = (f64 && Lc.nph <= 10) || (double)Lc.nbox * Lp.K * R < 300000.0 * Lc.ma_pm;
  return Lc.ant_wide && v <= 2 && (few || (v && !f64)) &&      // FP64's variant is for one column
         (size_t)Lc.ant_GR * 2 * NF * (f64 ? 16 : 8) <= ANT_SMEM;
}

// anterpolation of level Lp into Lc by gathering
template <typename T> static int run_anterp_gather(Ctx* c, const Level& Lc, const Level& Lp, int R, int an, cudaStream_t st) {
  typedef typename CV<T>::V V;
  typedef typename Part<T>::H H;
  const bool f64 = sizeof(T) == 8, one = f64 && R == 1;
  // column chunk: half of the table's where rows are long (40x40 level 1: 123 ->
  // 78 us; level 0, 11 columns: 121 -> 133) or boxes fewer than SMs (40x40 level 3:
  // 90 -> 68 us); for wide stencils as many chunks as make two CTAs an SM
  int JC = Lc.ant_JC;
  if (an == 1 || (an == 0 && one && (JC > 12 || Lc.nbox < 152))) JC = std::max(1, JC / 2);
  if (!one) JC = (int)std::max<long long>(1, std::min<long long>(JC, (long long)Lc.nph / 2 * Lc.nbox * Lc.ant_nit * R / 304));
  const int njc = (Lc.nph / 2 + JC - 1) / JC;
  const size_t sm = (size_t)Lc.ant_GR * 2 * JC * NF * sizeof(V);
  const int thr = (an == 2 || (an == 0 && Lc.nph <= 24) || Lc.ant_GR * 2 * JC >= 2048) ? 256 : 128;
  auto k = k_anterp1<T, 0, true>;
  if constexpr (sizeof(T) == 8) {
    if (one) {
      k = k_anterp1<T, 0, false>;
      if (Lc.ant_PM == 8 && Lc.ant_TM == 8) k = std::max(Lc.ant_PMx, Lc.ant_TMx) <= 7 ? k_anterp1<T, 7, false> : k_anterp1<T, 8, false>;
    }
  }
  if (!one) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ANT_SMEM);
  k<<<dim3((unsigned)(Lc.nbox * Lc.ant_nit * njc), (unsigned)R), thr, sm, st>>>(
      Lc.nth, Lc.nph, Lp.nth, Lp.nph, R, Lc.ant_TI, Lc.ant_nit, JC, njc, Lc.d_parent, Lc.d_quad, Lc.d_ant_lo,
      Lc.ant_PM, Lc.d_ant_pjp, (const T*)(f64 ? (void*)Lc.d_ant_pw64 : (void*)Lc.d_ant_pw32),
      (const T*)(f64 ? (void*)Lc.d_wthp64 : (void*)Lc.d_wthp32),
      (const V*)(f64 ? (void*)Lc.d_shift64 : (void*)Lc.d_shift32), (const H*)Lp.d_in, Lc.ant_TM, Lc.d_ant_ttp,
      (const T*)(f64 ? (void*)Lc.d_ant_tw64 : (void*)Lc.d_ant_tw32), (H*)Lc.d_in);
  SMR_LAUNCH(c);
  return SMR_OK;
}

// Finest boxes made of cells.  Box b's outgoing spectrum is the sum of its
// particles' spectra, and each particle receives its box's incoming
// spectrum; a row is one box's or one particle's [K0][NF][R] spectrum.  With
// `shift` set the kernels also carry each particle's displacement d from
// its box centre: e^{+jk khat.d} into the sum, e^{-jk khat.d} out of the
// broadcast (the tensor-core aggregation and receive work on unshifted
// per-particle spectra).  Grid: (boxes or particles, row chunks of 256
// elements); both kernels guard the row end.
template <typename T>
__device__ __forceinline__ typename CV<T>::V shift_phase(const double* d, const double* kh, double k, double sgn) {
  const double ph = sgn * k * (kh[0] * d[0] + kh[1] * d[1] + kh[2] * d[2]);
  T sn, cs;
  if (sizeof(T) == 8) {
    double s8, c8;
    sincos(ph, &s8, &c8);
    sn = (T)s8;
    cs = (T)c8;
  } else {
    float s4, c4;
    sincosf((float)ph, &s4, &c4);
    sn = (T)s4;
    cs = (T)c4;
  }
  return mkc(cs, sn);
}

template <typename T>
__global__ void k_cell_sum(int nbox, long long row, int R, const int* __restrict__ ptr,
                           const int* __restrict__ idx, int shift, const double* __restrict__ dshift,
                           const double* __restrict__ khat, double k,
                           const typename CV<T>::V* __restrict__ part, typename CV<T>::V* __restrict__ box) {
  typedef typename CV<T>::V V;
  const int b = blockIdx.x;
  const long long e = blockIdx.y * (long long)blockDim.x + threadIdx.x;
  if (b >= nbox || e >= row) return;
  const int kk = (int)(e / ((long long)NF * R));
  V acc = mkc((T)0, (T)0);
  for (int t = ptr[b]; t < ptr[b + 1]; ++t) {
    const int mu = idx[t];
    V v = part[(size_t)mu * row + e];
    if (shift) v = cmul(v, shift_phase<T>(dshift + 3 * mu, khat + 3 * kk, k, 1.0));
    acc.x += v.x;
    acc.y += v.y;
  }
  box[(size_t)b * row + e] = acc;
}

template <typename T>
__global__ void k_cell_bcast(int p, long long row, int R, const int* __restrict__ cell, int shift,
                             const double* __restrict__ dshift, const double* __restrict__ khat, double k,
                             const typename CV<T>::V* __restrict__ box, typename CV<T>::V* __restrict__ part) {
  typedef typename CV<T>::V V;
  const int mu = blockIdx.x;
  const long long e = blockIdx.y * (long long)blockDim.x + threadIdx.x;
  if (mu >= p || e >= row) return;
  V v = box[(size_t)cell[mu] * row + e];
  if (shift) v = cmul(v, shift_phase<T>(dshift + 3 * mu, khat + 3 * (int)(e / ((long long)NF * R)), k, -1.0));
  part[(size_t)mu * row + e] = v;
}

template <typename T>
static int far_impl(Ctx* c, int R, const double2* x, double2* y, bool accumulate, cudaStream_t st) {
  typedef typename CV<T>::V V;
  const bool f64 = sizeof(T) == 8;
  const double es = sizeof(V), R_ = R;
  Level& L0 = c->lev[0];
  // Overlap: the translation of each level runs on a side stream after an
  // event that marks its outgoing spectra, and the anterpolation into a level
  // waits for that level's translation; the receive waits for the near
  // product when run_product put it on a side stream (c->near_ev).
  Ctx::Side* sd = (c->overlap && !c->prof && c->cur_side < (int)c->side.size()) ? &c->side[c->cur_side] : nullptr;
  if (sd && (!sd->tr || c->nlev > (int)sd->eout.size())) sd = nullptr;
  // the coefficients stay with the spectra (smr_copy_level's fields come from both)
  if (!c->keep_x) {
    const size_t bytes = (size_t)c->p * 2 * c->npsi * R * sizeof(double2);
    if (sd) {
      SMR_CUDA(c, cudaEventRecord(sd->efork, st));
      SMR_CUDA(c, cudaStreamWaitEvent(sd->tr, sd->efork, 0));
    }
    pbeg(c, st, "keep", -1, 2.0 * bytes, 0.0);
    SMR_CUDA(c, cudaMemcpyAsync(c->d_xs[f64 ? 0 : 1], x, bytes, cudaMemcpyDeviceToDevice, sd ? sd->tr : st));
    pend(c, st);
  }
  // translation at every level (in the upward loop when it overlaps)
  auto translate = [&](int s, cudaStream_t ts) -> int {
    Level& L = c->lev[s];
    if (L.off_dx.empty()) {                  // no interaction list at this level
      SMR_CUDA(c, cudaMemsetAsync(L.d_in, 0, L.spec_bytes, ts));
      return SMR_OK;
    }
    pbeg(c, ts, "translate", s,
         2.0 * L.nbox * L.K * NF * R_ * es + (double)L.off_dx.size() * L.K * es,
         8.0 * L.il_src.size() * L.K * NF * R_);
    if (!f64 && R == 1) {
      int rc = run_translate_tiles(c, s, ts);
      pend(c, ts);
      return rc;
    }
    if (f64) {
      const int NR = NF * R, nch = (int)(((long long)L.K * NR + 127) / 128);
      k_translate_il<<<(unsigned)((long long)L.nbox * nch), 128, 0, ts>>>(
          L.K, NR, nch, L.d_il_ptr, L.d_il_pk, L.d_T64, (const double2*)L.d_out, (double2*)L.d_in);
      SMR_LAUNCH(c);
      pend(c, ts);
      return SMR_OK;
    }
    // FP32, several columns at once
    const int noff = 49;                     // tables by lattice offset (7 x 7 grid)
    const int cap = 32;                      // directions x columns staged per CTA
    const int RCt = std::min(R, cap), KC = std::max(1, cap / RCt);
    const int nkch = (L.K + KC - 1) / KC, nrct = (R + RCt - 1) / RCt;
    const size_t sm = ((size_t)64 * KC * NF * RCt + (size_t)noff * KC) * sizeof(float2) + (64 + 16 + 16) * sizeof(int) +
                      16 * 27 * sizeof(int2);
    cudaFuncSetAttribute(k_translate, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    k_translate<<<(unsigned)(L.ntile_ne * nkch * nrct), 256, sm, ts>>>(
        L.K, R, RCt, KC, L.ntile_x, L.ntile_ne, L.d_tiles, L.map_x0, L.map_y0, L.map_w, L.map_h, noff, L.d_boxmap,
        L.d_offid, L.d_T32, (const float2*)L.d_out, (float2*)L.d_in);
    SMR_LAUNCH(c);
    pend(c, ts);
    return SMR_OK;
  };
  auto fork_translate = [&](int s) -> int {
    SMR_CUDA(c, cudaEventRecord(sd->eout[s], st));
    SMR_CUDA(c, cudaStreamWaitEvent(sd->tr, sd->eout[s], 0));
    int rc = translate(s, sd->tr);
    if (rc) return rc;
    SMR_CUDA(c, cudaEventRecord(sd->etr[s], sd->tr));
    return SMR_OK;
  };
  // aggregation
  {
    pbeg(c, st, "aggregate", 0,
         (double)c->p * 2 * c->npsi * R_ * 16 + (double)c->S * c->npsi * 2 * L0.K * es +
             (double)c->p * L0.K * NF * R_ * es,
         16.0 * c->npsi * c->p * L0.K * R_);
    // per-particle spectra go through the box sum where boxes hold several
    // particles, or where the tensor cores aggregate displaced particles
    // (the sum then applies the displacement shifts)
    const bool tc = !f64 && tc_aggregate_ok(c, R) && c->tune_tc_agg != 0;
    const bool cells = c->multi || (tc && c->any_dshift);
    V* agg = (V*)(cells ? c->pspec[f64 ? 0 : 1] : L0.d_out);
    if (tc) {
      int rc = run_aggregate_tc(c, x, c->x32_of == x ? c->d_x32 : nullptr, (float2*)agg, st);
      if (rc) {
        pend(c, st);
        return rc;
      }
    } else {
      const int nchunk = (L0.K / 2 + AGC_PAIRS - 1) / AGC_PAIRS;
      const size_t sm = (size_t)(2 * c->npsi + 8 * AGC_PAIRS) * sizeof(V);
      k_aggregate<T><<<(unsigned)((long long)c->p * R * nchunk), 2 * AGC_PAIRS, sm, st>>>(
          L0.K, L0.nph, c->npsi, R, nchunk, c->d_perm, c->d_sid, x,
          (const V*)(f64 ? (void*)c->d_Pd64 : (void*)c->d_Pd32), c->d_dshift, c->any_dshift, L0.d_khat, c->k,
          1.0 / c->zeta, agg);
      SMR_LAUNCH(c);
    }
    if (cells) {
      const long long row = (long long)L0.K * NF * R;
      k_cell_sum<T><<<dim3((unsigned)L0.nbox, (unsigned)((row + 255) / 256)), 256, 0, st>>>(
          L0.nbox, row, R, c->d_cell_ptr, c->d_cell_idx, (tc && c->any_dshift) ? 1 : 0, c->d_dshift,
          L0.d_khat, c->k, agg, (V*)L0.d_out);
      SMR_LAUNCH(c);
    }
    pend(c, st);
  }
  // upward: interpolation, shift and child sum
  for (int s = 0; s + 1 < c->nlev; ++s) {
    if (sd) {
      int rc = fork_translate(s);              // level s's outgoing spectra are complete
      if (rc) return rc;
    }
    Level &Lc = c->lev[s], &Lp = c->lev[s + 1];
    pbeg(c, st, "interpolate", s,
         ((double)Lc.nbox * Lc.K + (double)Lp.nbox * Lp.K) * NF * R_ * es + 4.0 * Lp.K * es,
         (double)Lc.nbox * Lp.nth * Lc.nph * NF * R_ * 16.0 + (double)Lc.nbox * Lp.K * NF * R_ * 24.0);
    if (!f64 || R > 1 || march_interp(Lc.tune_ip) || Lp.nph * Part<double>::NT > 256 * EM1) {
      int rc = run_interp(c, s, R, f64 ? SMR_PREC_FP64 : SMR_PREC_FP32, st);
      if (rc) return rc;
    } else {
      // parent rows of a CTA: whole tiles (variants 1, 2: half), or the split that finishes
      // first with two CTAs an SM at a time, a CTA costing about two rows more than it
      // has (levels of the 20x20 array 33 + 35 + 32 us with whole tiles, 23 + 21 + 19 so;
      // 40x40 80 + 60 + 56 + 44 and 79 + 49 + 42 + 36)
      const int most = std::max(1, std::min(Lp.nth, (256 * EM1) / (Lp.nph * Part<double>::NT)));
      int TR = Lc.tune_ip == 2 ? std::max(1, most / 2) : most;
      if (Lc.tune_ip == 0) {
        long long cost = -1;
        for (int t = most; t >= 1; --t) {
          const long long w = ((long long)Lp.nbox * ((Lp.nth + t - 1) / t) + 303) / 304 * (t + 2);
          if (cost < 0 || w < cost) {
            cost = w;
            TR = t;
          }
        }
      }
      int nrt = (Lp.nth + TR - 1) / TR;
      size_t sm1 = (size_t)TR * Lc.nph * NF * sizeof(double2);
      cudaFuncSetAttribute(k_interp1, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
      const unsigned mP = (unsigned)(((1ull << 32) + (unsigned)Lp.nph - 1) / (unsigned)Lp.nph);
      k_interp1<<<(unsigned)(Lp.nbox * nrt), 256, sm1, st>>>(
          Lp.nth, Lp.nph, mP, Lc.nph, Lc.K, TR, nrt, Lp.d_ch_ptr, Lp.d_ch_idx, Lp.d_ch_quad, Lc.d_th_pk,
          Lc.d_th_ws64, Lc.d_ph_src, Lc.d_ph_w64, Lc.d_shift64, (const double2*)Lc.d_out, (double2*)Lp.d_out);
      SMR_LAUNCH(c);
    }
    pend(c, st);
  }
  if (sd) {
    int rc = fork_translate(c->nlev - 1);      // the top level
    if (rc) return rc;
  } else {
    for (int s = 0; s < c->nlev; ++s) {
      int rc = translate(s, st);
      if (rc) return rc;
    }
  }
  // downward: the weighted adjoint (accumulates)
  for (int s = c->nlev - 2; s >= 0; --s) {
    if (sd) {
      // the parent level's incoming spectra and this level's translation
      SMR_CUDA(c, cudaStreamWaitEvent(st, sd->etr[s + 1], 0));
      SMR_CUDA(c, cudaStreamWaitEvent(st, sd->etr[s], 0));
    }
    Level &Lc = c->lev[s], &Lp = c->lev[s + 1];
    pbeg(c, st, "anterpolate", s,
         ((double)Lp.nbox * Lp.K + 2.0 * Lc.nbox * Lc.K) * NF * R_ * es + 4.0 * Lp.K * es,
         (double)Lc.nbox * Lp.nth * Lc.nph * NF * R_ * 8.0 * 2 * (double)Lp.nph / Lc.nph * 4.0 / 4.0 +
             (double)Lc.nbox * Lc.K * NF * R_ * 16.0 * (double)Lp.nth / Lc.nth);
    const int an = Lc.tune_an[f64 ? 0 : 1];
    int rc;
    if (gather_anterp(Lc, Lp, f64, R, an)) rc = run_anterp_gather<T>(c, Lc, Lp, R, f64 && R > 1 ? 0 : an, st);
    else rc = run_anterp(c, s, R, f64 ? SMR_PREC_FP64 : SMR_PREC_FP32, st);
    if (rc) return rc;
    pend(c, st);
  }
  // receive
  if (sd) SMR_CUDA(c, cudaStreamWaitEvent(st, sd->etr[0], 0));
  {
    pbeg(c, st, "receive", 0,
         (double)c->p * L0.K * NF * R_ * es + (double)c->S * c->npsi * 2 * L0.K * es +
             (accumulate ? 2.0 : 1.0) * c->p * 2 * c->npsi * R_ * 16,
         16.0 * c->p * c->npsi * L0.K * R_);
    // per-particle incoming spectra where boxes hold several particles, or
    // where the tensor cores receive for displaced particles (the broadcast
    // then applies the displacement shifts)
    const bool tc = !f64 && tc_receive_ok(c, R) && c->tune_tc_rec != 0;
    const bool cells = c->multi || (tc && c->any_dshift);
    const V* inc = (const V*)L0.d_in;
    if (cells) {
      const long long row = (long long)L0.K * NF * R;
      V* part = (V*)c->pspec[f64 ? 0 : 1];
      k_cell_bcast<T><<<dim3((unsigned)c->p, (unsigned)((row + 255) / 256)), 256, 0, st>>>(
          c->p, row, R, c->d_cell_of, (tc && c->any_dshift) ? 1 : 0, c->d_dshift, L0.d_khat, c->k,
          (const V*)L0.d_in, part);
      SMR_LAUNCH(c);
      inc = part;
    }
    if (tc) {
      int rc = run_receive_tc(c, (const float2*)inc, y, accumulate, c->near_ev, st);
      pend(c, st);
      return rc;
    }
    if (c->near_ev) SMR_CUDA(c, cudaStreamWaitEvent(st, c->near_ev, 0));
    const int thr = c->npsi * std::max(1, 256 / c->npsi);
    k_receive<T><<<(unsigned)((long long)c->p * R), thr, (size_t)(4 * RCV_PAIRS + 2 * thr) * sizeof(V), st>>>(
        L0.K, L0.nph, c->npsi, R, c->d_perm, c->d_sid, inc, (const V*)(f64 ? (void*)c->d_Pm64 : (void*)c->d_Pm32),
        L0.d_w, c->d_dshift, c->any_dshift, L0.d_khat, c->k, c->zeta, y, accumulate ? 1 : 0);
    SMR_LAUNCH(c);
    pend(c, st);
  }
  return SMR_OK;
}

int run_far(Ctx* c, int R, int prec, const double2* x, double2* y, bool accumulate,
            cudaStream_t st) {
  int rc = ensure_spectra(c, R, prec);
  if (rc) return rc;
  return prec == SMR_PREC_FP64 ? far_impl<double>(c, R, x, y, accumulate, st)
                               : far_impl<float>(c, R, x, y, accumulate, st);
}

template <typename T>
static int bs_impl(Ctx* c, int nrow, int R, const int* ptr, const int* col, const int* blk,
                   const void* Bt, const double2* x, double2* y, bool acc, cudaStream_t st) {
  typedef typename CV<T>::V V;
  int n2 = 2 * c->npsi;
  int rc = std::min(R, std::max(1, 256 / n2));
  int nrc = (R + rc - 1) / rc;
  size_t sm = (size_t)n2 * rc * sizeof(V);
  k_blocksparse<T><<<(unsigned)(nrow * nrc), n2 * rc, sm, st>>>(nrow, n2, R, rc, nrc, ptr, col, blk,
                                                               (const V*)Bt, x, y, acc ? 1 : 0);
  SMR_LAUNCH(c);
  return SMR_OK;
}

__global__ void k_x32f(long long n, const double2* __restrict__ a, float2* __restrict__ b) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) b[i] = make_float2((float)a[i].x, (float)a[i].y);
}

// The FP32 single right-hand-side product converts x to FP32 once (the
// conversion runs on the FP64 units, 1/64 of the FP32 rate) for the near
// gathers and the tensor-core aggregation; c->x32_of records which x the
// copy holds, so a step that finds another x reads the FP64 one.  The record
// lives for one product call: the callers clear it before they return, and
// graph capture clears it (a capture converts nothing).
int prep_x32(Ctx* c, int R, int prec, const double2* x, cudaStream_t st) {
  c->x32_of = nullptr;
  if (prec != SMR_PREC_FP32 || R != 1 || !c->d_x32) return SMR_OK;
  const long long n = (long long)c->p * 2 * c->npsi;
  pbeg(c, st, "convert", -1, (double)n * 24.0, 0.0);
  k_x32f<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, x, c->d_x32);
  SMR_LAUNCH(c);
  pend(c, st);
  c->x32_of = x;
  return SMR_OK;
}

int run_near(Ctx* c, int R, int prec, const double2* x, double2* y, cudaStream_t st) {
  if (prec == SMR_PREC_FP32 && tc_near_ok(c, R) && c->tune_tc_near != 0) {
    if (c->x32_of != x) {
      int rc = prep_x32(c, R, prec, x, st);
      if (rc) return rc;
    }
    return run_near_tc(c, y, st);
  }
  double n2 = 2.0 * c->npsi, es = prec == SMR_PREC_FP64 ? 16 : 8;
  const bool x32 = prec == SMR_PREC_FP32 && R == 1 && c->x32_of == x;
  pbeg(c, st, "near", -1, c->p * n2 * R * (x32 ? 8 + 16 : 16 + 16) + (c->nblk + c->S) * 0.5 * n2 * n2 * es,
       4.0 * n2 * n2 * (c->nr_col.size() + c->p) * R);
  const int n = c->npsi, thr = 2 * n * std::max(1, 256 / (2 * n));
  const size_t vb = prec == SMR_PREC_FP64 ? sizeof(double2) : sizeof(float2);
  const size_t sm = ((size_t)NR_PAIRS * 2 * n + 2 * thr) * vb;
  const unsigned g = (unsigned)((long long)c->p * R);
  if (prec == SMR_PREC_FP64)
    k_near_rows<double, double2><<<g, thr, sm, st>>>(n, R, c->S, c->d_nr_ptr, c->d_nr_col, c->d_nr_blk, c->d_Bs64,
                                                     c->d_Bc64, c->zeta, x, y);
  else if (x32)
    k_near_rows<float, float2><<<g, thr, sm, st>>>(n, R, c->S, c->d_nr_ptr, c->d_nr_col, c->d_nr_blk, c->d_Bs32,
                                                   c->d_Bc32, c->zeta, c->d_x32, y);
  else
    k_near_rows<float, double2><<<g, thr, sm, st>>>(n, R, c->S, c->d_nr_ptr, c->d_nr_col, c->d_nr_blk, c->d_Bs32,
                                                    c->d_Bc32, c->zeta, x, y);
  SMR_LAUNCH(c);
  pend(c, st);
  return SMR_OK;
}

// out[c][i] = in[i][c] for in [rows][cols] (tiles of 32 x 32 through shared
// memory); grid x runs over the longer of the two dimensions
__global__ void k_transpose_c128(long long rows, long long cols, const double2* __restrict__ in,
                                 double2* __restrict__ out) {
  __shared__ double2 t[32][33];
  const bool rx = rows >= cols;
  const long long i0 = (long long)(rx ? blockIdx.x : blockIdx.y) * 32;
  const long long c0 = (long long)(rx ? blockIdx.y : blockIdx.x) * 32;
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    long long i = i0 + k, cc = c0 + threadIdx.x;
    if (i < rows && cc < cols) t[k][threadIdx.x] = in[i * cols + cc];
  }
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    long long cc = c0 + k, i = i0 + threadIdx.x;
    if (i < rows && cc < cols) out[cc * rows + i] = t[threadIdx.x][k];
  }
}

static int transpose_c128(Ctx* c, long long rows, long long cols, const double2* in, double2* out,
                          cudaStream_t st) {
  long long a = (rows + 31) / 32, b = (cols + 31) / 32;
  dim3 g((unsigned)std::max(a, b), (unsigned)std::min(a, b));
  k_transpose_c128<<<g, dim3(32, 8), 0, st>>>(rows, cols, in, out);
  SMR_LAUNCH(c);
  return SMR_OK;
}

bool split_columns(const Ctx* c, int R, int prec) { return R > 1 && prec == SMR_PREC_FP32 && c->split_cols; }

// column buffers [R][N] for split products (allocated outside graph capture)
int ensure_split(Ctx* c, int R) {
  size_t need = (size_t)2 * R * 2 * c->npsi * c->p;
  if (c->split_elems >= need) return SMR_OK;
  drop_split_graphs(c);
  if (c->d_split) cudaFree(c->d_split);
  c->d_split = nullptr;
  c->split_elems = 0;
  if (cudaMalloc((void**)&c->d_split, need * sizeof(double2)) != cudaSuccess) {
    cudaGetLastError();
    c->err = "out of device memory for the column buffers of a split product";
    return SMR_E_OOM;
  }
  c->split_elems = need;
  return SMR_OK;
}

void free_lanes(Ctx* c) {
  drop_split_graphs(c);
  for (size_t j = 1; j < c->lanes.size(); ++j) {
    Ctx::Lane& a = c->lanes[j];
    for (void* q : a.out) if (q) cudaFree(q);
    for (void* q : a.in) if (q) cudaFree(q);
    if (a.x32) cudaFree(a.x32);
    if (a.tcn_part) cudaFree(a.tcn_part);
    if (a.tc_part) cudaFree(a.tc_part);
    if (a.s) cudaStreamDestroy(a.s);
  }
  for (auto& a : c->lanes)
    if (a.ev) cudaEventDestroy(a.ev);
  c->lanes.clear();
  if (c->lane_fork) cudaEventDestroy(c->lane_fork);
  c->lane_fork = nullptr;
}

// Work buffers of nl column lanes for FP32 single-column products (outside
// graph capture; lanes that exist are kept and grown only).
int ensure_lanes(Ctx* c, int nl) {
  int rc = ensure_spectra(c, 1, SMR_PREC_FP32);
  if (rc) return rc;
  if ((int)c->lanes.size() < nl) c->lanes.resize(nl);
  if (!c->lane_fork) SMR_CUDA(c, cudaEventCreateWithFlags(&c->lane_fork, cudaEventDisableTiming));
  Ctx::Lane& l0 = c->lanes[0];                 // the context's own buffers
  l0.out.assign(c->nlev, nullptr);
  l0.in.assign(c->nlev, nullptr);
  for (int s = 0; s < c->nlev; ++s) {
    l0.out[s] = c->lev[s].buf_out[1];
    l0.in[s] = c->lev[s].buf_in[1];
  }
  l0.x32 = c->d_x32;
  l0.tcn_part = c->d_tcn_part;
  l0.tc_part = c->d_tc_part;
  for (int j = 0; j < nl; ++j) {
    Ctx::Lane& a = c->lanes[j];
    if (!a.ev) SMR_CUDA(c, cudaEventCreateWithFlags(&a.ev, cudaEventDisableTiming));
    if (j == 0) continue;
    if (!a.s) SMR_CUDA(c, cudaStreamCreateWithFlags(&a.s, cudaStreamNonBlocking));
    if ((int)a.out.size() != c->nlev) {
      a.out.assign(c->nlev, nullptr);
      a.in.assign(c->nlev, nullptr);
    }
    bool ok = true;
    for (int s = 0; s < c->nlev && ok; ++s) {
      const size_t b = c->lev[s].buf_bytes[1];
      ok = (a.out[s] || cudaMalloc(&a.out[s], b) == cudaSuccess) &&
           (a.in[s] || cudaMalloc(&a.in[s], b) == cudaSuccess);
    }
    if (ok && c->d_x32 && !a.x32)
      ok = cudaMalloc((void**)&a.x32, (size_t)c->p * 2 * c->npsi * sizeof(float2)) == cudaSuccess;
    if (ok && c->d_tc_part && !a.tc_part) ok = cudaMalloc((void**)&a.tc_part, c->tc_part_bytes) == cudaSuccess;
    if (ok && c->d_tcn_part && !a.tcn_part) ok = cudaMalloc((void**)&a.tcn_part, c->tcn_part_bytes) == cudaSuccess;
    if (!ok) {
      cudaGetLastError();
      free_lanes(c);
      c->err = "out of device memory for the column lanes of a split product";
      return SMR_E_OOM;
    }
  }
  return SMR_OK;
}

// Points the FP32 single-column work buffers at lane j's.
static void use_lane(Ctx* c, int j) {
  const Ctx::Lane& a = c->lanes[j];
  for (int s = 0; s < c->nlev; ++s) {
    c->lev[s].d_out = a.out[s];
    c->lev[s].d_in = a.in[s];
  }
  c->d_x32 = a.x32;
  c->d_tcn_part = a.tcn_part;
  c->d_tc_part = a.tc_part;
}

// one lane where products use the shared per-particle spectra (several
// particles per box, or displaced particles)
int lanes_for(const Ctx* c, int R) {
  return (c->prof || c->multi || c->any_dshift) ? 1 : std::max(1, std::min(R, c->n_lanes));
}

// Side streams and events of lanes 0 .. n-1 for the overlapped product
// (created outside graph capture, kept until the context goes).
int ensure_side(Ctx* c, int n) {
  if (!c->overlap) return SMR_OK;
  if ((int)c->side.size() < n) c->side.resize(n);
  for (int j = 0; j < n; ++j) {
    Ctx::Side& d = c->side[j];
    if (d.tr) continue;
    SMR_CUDA(c, cudaStreamCreateWithFlags(&d.tr, cudaStreamNonBlocking));
    SMR_CUDA(c, cudaStreamCreateWithFlags(&d.nr, cudaStreamNonBlocking));
    SMR_CUDA(c, cudaEventCreateWithFlags(&d.ex, cudaEventDisableTiming));
    SMR_CUDA(c, cudaEventCreateWithFlags(&d.enear, cudaEventDisableTiming));
    SMR_CUDA(c, cudaEventCreateWithFlags(&d.efork, cudaEventDisableTiming));
    d.eout.assign(32, nullptr);
    d.etr.assign(32, nullptr);
    for (int s = 0; s < 32; ++s) {
      SMR_CUDA(c, cudaEventCreateWithFlags(&d.eout[s], cudaEventDisableTiming));
      SMR_CUDA(c, cudaEventCreateWithFlags(&d.etr[s], cudaEventDisableTiming));
    }
  }
  return SMR_OK;
}

void free_side(Ctx* c) {
  for (auto& d : c->side) {
    if (d.tr) cudaStreamDestroy(d.tr);
    if (d.nr) cudaStreamDestroy(d.nr);
    if (d.ex) cudaEventDestroy(d.ex);
    if (d.enear) cudaEventDestroy(d.enear);
    if (d.efork) cudaEventDestroy(d.efork);
    for (auto e : d.eout) if (e) cudaEventDestroy(e);
    for (auto e : d.etr) if (e) cudaEventDestroy(e);
  }
  c->side.clear();
}

// The near product of lane j: on the lane's side stream after an event on
// st (x and its FP32 copy ready), with c->near_ev for the receive to wait on;
// on st itself when the product does not overlap.
static int near_step(Ctx* c, int R, int prec, const double2* x, double2* y, cudaStream_t st, int j) {
  c->near_ev = nullptr;
  if (!c->overlap || c->prof || j >= (int)c->side.size() || !c->side[j].nr) return run_near(c, R, prec, x, y, st);
  Ctx::Side& d = c->side[j];
  SMR_CUDA(c, cudaEventRecord(d.ex, st));
  SMR_CUDA(c, cudaStreamWaitEvent(d.nr, d.ex, 0));
  int rc = run_near(c, R, prec, x, y, d.nr);
  SMR_CUDA(c, cudaEventRecord(d.enear, d.nr));
  if (rc) {
    SMR_CUDA(c, cudaStreamWaitEvent(st, d.enear, 0));   // joined even on failure
    return rc;
  }
  c->near_ev = d.enear;
  return SMR_OK;
}

// y = Z x for R right-hand sides [N][R].  FP32 products with several
// right-hand sides run column by column on the single right-hand-side kernels
// (16-byte parts, tensor-core aggregation and receive), which are faster per
// column than the batched kernels: x is transposed to [R][N], each column is
// multiplied, and y is transposed back.  The columns are dealt to the lanes
// round-robin; lane j > 0 runs on its own stream, forked from st after the
// transpose and joined before the transpose back, so a graph captured on st
// holds n_lanes independent chains of single-column products.
int run_product(Ctx* c, int R, int prec, const double2* x, double2* y, cudaStream_t st) {
  if (!split_columns(c, R, prec)) {
    int rc = ensure_side(c, 1);
    c->cur_side = 0;
    if (!rc) rc = prep_x32(c, R, prec, x, st);
    if (!rc) rc = near_step(c, R, prec, x, y, st, 0);
    if (!rc) rc = run_far(c, R, prec, x, y, true, st);
    c->near_ev = nullptr;
    c->x32_of = nullptr;                        // the FP32 copy lives for one product only
    return rc;
  }
  const int nl = lanes_for(c, R);
  int rc = ensure_split(c, R);
  if (!rc) rc = ensure_lanes(c, nl);
  if (!rc) rc = ensure_side(c, nl);
  if (rc) return rc;
  const long long n = 2LL * c->npsi * c->p;
  double2* xs = c->d_split;
  double2* ys = c->d_split + (size_t)R * n;
  pbeg(c, st, "transpose", -1, 2.0 * n * R * 16, 0.0);
  rc = transpose_c128(c, n, R, x, xs, st);
  pend(c, st);
  if (rc) return rc;
  if (nl > 1) {
    SMR_CUDA(c, cudaEventRecord(c->lane_fork, st));
    for (int j = 1; j < nl; ++j) SMR_CUDA(c, cudaStreamWaitEvent(c->lanes[j].s, c->lane_fork, 0));
  }
  for (int r = 0; r < R && !rc; ++r) {
    const int j = r % nl;
    cudaStream_t sj = j ? c->lanes[j].s : st;
    use_lane(c, j);
    c->cur_side = j;
    c->keep_x = j > 0 || r + nl < R;             // lane 0's last column is the one that stays
    rc = prep_x32(c, 1, prec, xs + (size_t)r * n, sj);
    if (!rc) rc = near_step(c, 1, prec, xs + (size_t)r * n, ys + (size_t)r * n, sj, j);
    if (!rc) rc = far_impl<float>(c, 1, xs + (size_t)r * n, ys + (size_t)r * n, true, sj);
    c->near_ev = nullptr;
  }
  use_lane(c, 0);
  c->cur_side = 0;
  c->keep_x = false;
  c->x32_of = nullptr;
  // every forked lane is joined, also after an error, so that a capture ends cleanly
  for (int j = 1; j < nl; ++j) {
    cudaError_t e = cudaEventRecord(c->lanes[j].ev, c->lanes[j].s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, c->lanes[j].ev, 0);
    if (e != cudaSuccess && !rc) {
      c->err = std::string("joining column lanes: ") + cudaGetErrorString(e);
      rc = SMR_E_CUDA;
    }
  }
  if (rc) return rc;
  pbeg(c, st, "transpose", -1, 2.0 * n * R * 16, 0.0);
  rc = transpose_c128(c, R, n, ys, y, st);
  pend(c, st);
  return rc;
}

void free_graphs(Ctx* c) {
  for (auto& g : c->graphs) cudaGraphExecDestroy(g.exec);
  c->graphs.clear();
  if (c->capture_stream) cudaStreamDestroy(c->capture_stream);
  c->capture_stream = nullptr;
}

int run_matvec_graph(Ctx* c, int R, int prec, const double2* x, double2* y, cudaStream_t st) {
  const bool split = split_columns(c, R, prec);
  for (auto& g : c->graphs)
    if (g.x == x && g.y == y && g.R == R && g.prec == prec) {
      SMR_CUDA(c, cudaGraphLaunch(g.exec, st));
      // the last product's spectra are the replay's (its buffers are still the
      // context's: a reallocation would have dropped the graph)
      return ensure_spectra(c, split ? 1 : R, prec);
    }
  // allocations happen outside the capture
  int rc = ensure_spectra(c, split ? 1 : R, prec);
  if (!rc && split) rc = ensure_split(c, R);
  if (!rc && split) rc = ensure_lanes(c, lanes_for(c, R));
  if (!rc) rc = ensure_side(c, split ? lanes_for(c, R) : 1);
  if (rc) return rc;
  if (!c->capture_stream) SMR_CUDA(c, cudaStreamCreateWithFlags(&c->capture_stream, cudaStreamNonBlocking));
  cudaStream_t cs = c->capture_stream;
  // order the capture stream after work already queued on the caller's stream
  cudaEvent_t ev;
  SMR_CUDA(c, cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
  SMR_CUDA(c, cudaEventRecord(ev, st));
  SMR_CUDA(c, cudaStreamWaitEvent(cs, ev, 0));
  SMR_CUDA(c, cudaStreamSynchronize(cs));
  cudaEventDestroy(ev);
  std::vector<ProfRec>* prof = c->prof;
  c->prof = nullptr;
  SMR_CUDA(c, cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
  rc = run_product(c, R, prec, x, y, cs);
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamEndCapture(cs, &graph);
  c->prof = prof;
  c->x32_of = nullptr;                          // the capture converted nothing
  if (rc) {
    if (graph) cudaGraphDestroy(graph);
    return rc;
  }
  if (e != cudaSuccess) {
    c->err = std::string("graph capture: ") + cudaGetErrorString(e);
    return SMR_E_CUDA;
  }
  cudaGraphExec_t exec = nullptr;
  e = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) {
    c->err = std::string("graph instantiate: ") + cudaGetErrorString(e);
    return SMR_E_CUDA;
  }
  if (c->graphs.size() >= 16) {                  // keep a handful of recent products
    cudaGraphExecDestroy(c->graphs.front().exec);
    c->graphs.erase(c->graphs.begin());
  }
  c->graphs.push_back({x, y, R, prec, exec});
  SMR_CUDA(c, cudaGraphLaunch(exec, st));
  return SMR_OK;
}

int run_precond(Ctx* c, int R, int prec, const double2* r, double2* z, cudaStream_t st) {
  if (!c->pinv_ok) {
    c->err = "a self block is singular: the block-diagonal preconditioner is undefined";
    return SMR_E_INVALID_ARG;
  }
  if (prec == SMR_PREC_FP64)
    return bs_impl<double>(c, c->p, R, c->d_pc_ptr, c->d_pc_col, c->d_pc_blk, c->d_Pinv64, r, z, false, st);
  return bs_impl<float>(c, c->p, R, c->d_pc_ptr, c->d_pc_col, c->d_pc_blk, c->d_Pinv32, r, z, false, st);
}

// current `cur`'s coefficients of x, zeros for the other's
__global__ void k_one_current(long long n, int run, int cur, const double2* __restrict__ x, double2* __restrict__ o) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) o[i] = (int)(i / run & 1) == cur ? x[i] : make_double2(0.0, 0.0);
}

// A level's spectra of the last product in the four fields (theta and phi of
// the electric and of the magnetic current's radiation), which the two circular
// fields do not tell apart: the far pass once more for each current alone, in
// scratch spectra, so that the product's stay as they are.  What the two passes
// differ by from the stored fields is divided between the currents: the fields
// returned combine to the spectra that the product left, whatever ran it.
int copy_fields(Ctx* c, int level, int kind, double* out) {
  const int prec = c->spec_prec, R = c->spec_R, p = prec == SMR_PREC_FP64 ? 0 : 1;
  const Level& L = c->lev[level];
  const long long n = (long long)c->p * 2 * c->npsi * R;
  const size_t elems = (size_t)L.nbox * L.K * NF * R;
  std::vector<double2> w[3];                     // electric current, magnetic current, as stored
  auto read = [&](std::vector<double2>& v) -> int {
    const void* src = kind == 0 ? L.d_out : L.d_in;
    v.resize(elems);
    if (p == 0) {
      SMR_CUDA(c, cudaMemcpy(v.data(), src, elems * sizeof(double2), cudaMemcpyDeviceToHost));
      return SMR_OK;
    }
    std::vector<float2> t(elems);
    SMR_CUDA(c, cudaMemcpy(t.data(), src, elems * sizeof(float2), cudaMemcpyDeviceToHost));
    for (size_t i = 0; i < elems; ++i) v[i] = make_double2(t[i].x, t[i].y);
    return SMR_OK;
  };
  SMR_CUDA(c, cudaDeviceSynchronize());
  int rc = read(w[2]);
  if (!rc) rc = ensure_side(c, 1);
  if (rc) return rc;
  // scratch: the outgoing and incoming spectra of every level, x and y
  std::vector<void*> own, scratch;
  for (auto& l : c->lev) {
    own.push_back(l.d_out);
    own.push_back(l.d_in);
  }
  for (size_t i = 0; i <= own.size() && !rc; ++i) {
    void* q = nullptr;
    if (cudaMalloc(&q, i < own.size() ? c->lev[i / 2].buf_bytes[p] : 2 * n * sizeof(double2)) != cudaSuccess) {
      cudaGetLastError();
      c->err = "out of device memory for a level's fields";
      rc = SMR_E_OOM;
    }
    scratch.push_back(q);
  }
  auto use = [&](const std::vector<void*>& b) {
    for (size_t s = 0; s < c->lev.size(); ++s) {
      c->lev[s].d_out = b[2 * s];
      c->lev[s].d_in = b[2 * s + 1];
    }
  };
  std::vector<ProfRec>* prof = c->prof;
  if (!rc) use(scratch);
  c->prof = nullptr;
  c->cur_side = 0;
  c->keep_x = true;
  double2* buf = (double2*)scratch.back();
  for (int cur = 0; cur < 2 && !rc; ++cur) {
    k_one_current<<<(unsigned)((n + 255) / 256), 256>>>(n, c->npsi * R, cur, c->d_xs[p], buf);
    rc = p == 0 ? far_impl<double>(c, R, buf, buf + n, false, nullptr)
                : far_impl<float>(c, R, buf, buf + n, false, nullptr);
    const cudaError_t e = cudaDeviceSynchronize();
    if (!rc && e != cudaSuccess) {
      c->err = std::string("level fields: ") + cudaGetErrorString(e);
      rc = SMR_E_CUDA;
    }
    if (!rc) rc = read(w[cur]);
  }
  use(own);
  c->keep_x = false;
  c->prof = prof;
  for (void* q : scratch) cudaFree(q);
  if (rc) return rc;
  for (size_t i = 0; i < elems; ++i) {
    const double2 d = make_double2(0.5 * (w[2][i].x - w[0][i].x - w[1][i].x), 0.5 * (w[2][i].y - w[0][i].y - w[1][i].y));
    for (int cur = 0; cur < 2; ++cur) {
      w[cur][i].x += d.x;
      w[cur][i].y += d.y;
    }
  }
  // electric current: W_+- = B0 -+ j B1; magnetic: W_+- = +-(j / z) (B2 -+ j B3)
  for (size_t d = 0; d < (size_t)L.nbox * L.K; ++d)
    for (int r = 0; r < R; ++r) {
      double* o = out + 2 * (d * 4 * R + r);
      for (int cur = 0; cur < 2; ++cur) {
        double2 p = w[cur][d * NF * R + r], q = w[cur][(d * NF + 1) * R + r];
        if (cur) {
          p = make_double2(c->zeta * p.y, -c->zeta * p.x);    // -j z W_+
          q = make_double2(-c->zeta * q.y, c->zeta * q.x);    // +j z W_-
        }
        const double2 v[2] = {make_double2(0.5 * (p.x + q.x), 0.5 * (p.y + q.y)),
                              make_double2(0.5 * (q.y - p.y), -0.5 * (q.x - p.x))};
        for (int f = 0; f < 2; ++f) {
          o[2 * (size_t)(2 * cur + f) * R] = v[f].x;
          o[2 * (size_t)(2 * cur + f) * R + 1] = v[f].y;
        }
      }
    }
  return SMR_OK;
}

}  // namespace smr

// Level steps of the product that move spectra between the quadtree's grids:
// interpolation (Sec. V, "4x4 Lagrange", child grid -> parent grid, shift,
// child sum) and its weighted adjoint, anterpolation.
//
// Both stencils are separable, real and narrow: 4 theta rows times 4 phi
// columns.  A thread owns one phi column of its output grid (one 16-byte part
// of it: part h of the NT parts a direction's NF R complex fields make) for
// the four children of a parent box, and marches along theta with the 4-row
// stencil window in registers, so every theta tap after the first is a
// register read.  All lanes are at the same theta position, which makes the
// window's rotation (four rows, unrolled four-fold) and all theta weights
// uniform.  The input rows stream through a ring of four shared-memory rows
// filled by asynchronous 16-byte copies three rows ahead; the phi taps are
// shared-memory reads at consecutive columns (the copies unwrap the period).
//
// The children's shifts come in conjugate pairs, s_3 = conj(s_0) and s_2 =
// conj(s_1) (children sit at (+-1/2, +-1/2) box from the parent's centre), so
//   s_0 a + s_3 b = Re(s_0) (a + b) + Im(s_0) i (a - b):
// the windows hold the sums and the differences of opposite children, a
// complex shift becomes two real weights, and the adjoint accumulates Re and
// Im parts once per pair instead of once per child.
//
// Bound: instruction issue and shared-memory reads, both near half of their
// peak with 12 to 16 warps per SM (the windows take the registers).  On the
// 200x200 lens in FP32 (algorithmic bytes 259 and 414 MB at level 0, of
// measured 6.68 TB/s): interpolation level 0 88 us, six levels 313 us;
// anterpolation level 0 111 us, six levels 378 us.  With four fields a direction
// these took 168, 597, 235 and 808 us, and kernels that kept the phi-pass rows in
// shared memory (a barrier and a round trip per row, 7 gathered taps per output)
// 262, 955, 356 and 1369 us.  Measured with four fields: a thread per child pair
// instead of four children (half the registers, twice the warps) 696 and 1021
// us; CTAs that run on over several boxes 873 and 1062 us, the ring's
// bookkeeping costing more than its restarts.  The adjoint's shifts, read by every
// tap, stay packed as they lie in memory (Mp<float>::G): staged as the weight pairs
// the packed multiply-add takes for two fields they took 649 us.
#include <algorithm>

#include "march_tile.h"
#include "smr_internal.h"

namespace smr {

namespace {

// threads of a CTA (at most), resident CTAs the register budget is set for,
// copies of one input row per thread (at most)
// by precision: more and smaller CTAs wait less at their barriers (FP32, 200x200
// lens: interpolation 352 us with 2 x 224 threads, 313 with 4 x 128; anterpolation 403
// with 2 x 192, 378 with 3 x 128), in FP64 their shared rows cost more than that
// (20x20, four columns, product: 1.24 ms with 4 x 128, 1.21 with 2 x 224)
template <typename T> constexpr int INTERP_THREADS = sizeof(T) == 8 ? 224 : 128;
template <typename T> constexpr int INTERP_CTAS = sizeof(T) == 8 ? 2 : 4;
template <typename T> constexpr int ANTERP_THREADS = sizeof(T) == 8 ? 192 : 128;
template <typename T> constexpr int ANTERP_CTAS = sizeof(T) == 8 ? 2 : 3;
constexpr int INTERP_NK = 3, ANTERP_NK = 4;
constexpr int MARCH_ROWS = 64;                 // parent rows of an interpolation tile, at most

// 16 bytes global -> shared
__device__ __forceinline__ void copy16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the newest two groups have landed
__device__ __forceinline__ void copies_wait2() { asm volatile("cp.async.wait_group 2;" ::: "memory"); }

template <typename T> struct Mp;
template <> struct Mp<float> {
  typedef float4 H;                            // one 16-byte part: two complex fields
  typedef float2 W;                            // a weight as the pair the packed multiply-add takes
  typedef float2 C;                            // a complex value
  typedef float4 S;                            // a direction's two shifts
  // Re and Im sums of both conjugate pairs, [component][pair]: the packed
  // multiply-add takes a pair's Re and Im weights as they lie in memory, where one
  // weight for both fields would have to be read or moved into a pair first
  struct G { float2 c[4][2]; };
  static __device__ __forceinline__ void gzero(G& g) {
#pragma unroll
    for (int i = 0; i < 4; ++i) g.c[i][0] = g.c[i][1] = make_float2(0.f, 0.f);
  }
  // g += (Re, Im of both shifts) w v
  static __device__ __forceinline__ void tap(G& g, float w, H v, const S* sp) {
    const float4 s = *sp;
    const float e[4] = {w * v.x, w * v.y, w * v.z, w * v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 d = make_float2(e[i], e[i]);
      g.c[i][0] = __ffma2_rn(d, make_float2(s.x, s.y), g.c[i][0]);
      g.c[i][1] = __ffma2_rn(d, make_float2(s.z, s.w), g.c[i][1]);
    }
  }
  static __device__ __forceinline__ void scatter(G& a, float w, const G& g) {
    const float2 w2 = make_float2(w, w);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      a.c[i][0] = __ffma2_rn(w2, g.c[i][0], a.c[i][0]);
      a.c[i][1] = __ffma2_rn(w2, g.c[i][1], a.c[i][1]);
    }
  }
  // conj(s_q) v of the four children: Re - i Im for 0 and 1, Re + i Im for 3 and 2
  static __device__ __forceinline__ void children(const G& a, H* d) {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const float2 x = a.c[0][p], y = a.c[1][p], z = a.c[2][p], w = a.c[3][p];
      d[p] = make_float4(x.x + y.y, y.x - x.y, z.x + w.y, w.x - z.y);
      d[3 - p] = make_float4(x.x - y.y, y.x + x.y, z.x - w.y, w.x + z.y);
    }
  }
  // the four children's values += d, as reductions in the L2 (one addend per
  // element, so the result does not depend on their order)
  static __device__ __forceinline__ void add_to(const bool* has, H* base, const unsigned* kid, unsigned ro, int NT,
                                                const H* d) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (has[q]) {
        H* p = base + (size_t)(kid[q] + ro) * NT;
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(d[q].x), "f"(d[q].y), "f"(d[q].z),
                     "f"(d[q].w)
                     : "memory");
      }
  }
  static __device__ __forceinline__ void unpack(const S* p, float* s) {
    const float4 v = *p;
    s[0] = v.x; s[1] = v.y; s[2] = v.z; s[3] = v.w;
  }
  static constexpr int HN = NF / 2;            // parts of a direction a CTA takes (R = 1: all of them)
  static __device__ __forceinline__ H zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ W wt(float w) { return make_float2(w, w); }
  static __device__ __forceinline__ void fma(H& a, W w, H v) {
    const float2 lo = __ffma2_rn(w, make_float2(v.x, v.y), make_float2(a.x, a.y));
    const float2 hi = __ffma2_rn(w, make_float2(v.z, v.w), make_float2(a.z, a.w));
    a = make_float4(lo.x, lo.y, hi.x, hi.y);
  }
  // one-off weights: a scalar multiply-add needs no pair
  static __device__ __forceinline__ void fma1(H& a, float w, H v) {
    a.x = fmaf(w, v.x, a.x); a.y = fmaf(w, v.y, a.y); a.z = fmaf(w, v.z, a.z); a.w = fmaf(w, v.w, a.w);
  }
  // a += i w v
  static __device__ __forceinline__ void fmai(H& a, float w, H v) {
    a.x = fmaf(-w, v.y, a.x); a.y = fmaf(w, v.x, a.y); a.z = fmaf(-w, v.w, a.z); a.w = fmaf(w, v.z, a.w);
  }
  static __device__ __forceinline__ H add(H a, H b) {
    const float2 lo = __fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
    const float2 hi = __fadd2_rn(make_float2(a.z, a.w), make_float2(b.z, b.w));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
  }
  static __device__ __forceinline__ H sub(H a, H b) {
    const float2 m = make_float2(-1.f, -1.f);
    const float2 lo = __ffma2_rn(m, make_float2(b.x, b.y), make_float2(a.x, a.y));
    const float2 hi = __ffma2_rn(m, make_float2(b.z, b.w), make_float2(a.z, a.w));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
  }
  static __device__ __forceinline__ H itimes(H a) { return make_float4(-a.y, a.x, -a.w, a.z); }
  static __device__ __forceinline__ void t4(const float* p, float* w) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p));
    w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
  }
  static __device__ __forceinline__ void w4(const W* p, W* w) {
    const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
    w[0] = make_float2(a.x, a.y); w[1] = make_float2(a.z, a.w);
    w[2] = make_float2(b.x, b.y); w[3] = make_float2(b.z, b.w);
  }
};
template <> struct Mp<double> {
  typedef double2 H;
  typedef double W;
  typedef double2 C;
  struct S { double2 a, b; };
  struct G { double2 x[4]; };                  // Re 03, Im 03, Re 12, Im 12
  static __device__ __forceinline__ void gzero(G& g) {
#pragma unroll
    for (int x = 0; x < 4; ++x) g.x[x] = zero();
  }
  static __device__ __forceinline__ void tap(G& g, double w, H r, const S* sp) {
    double s[4];
    unpack(sp, s);
    const H v = make_double2(w * r.x, w * r.y);
#pragma unroll
    for (int x = 0; x < 4; ++x) fma(g.x[x], s[x], v);
  }
  static __device__ __forceinline__ void scatter(G& a, double w, const G& g) {
#pragma unroll
    for (int x = 0; x < 4; ++x) fma(a.x[x], w, g.x[x]);
  }
  static __device__ __forceinline__ void children(const G& a, H* d) {
    const H i03 = itimes(a.x[1]), i12 = itimes(a.x[3]);
    d[0] = sub(a.x[0], i03); d[1] = sub(a.x[2], i12); d[2] = add(a.x[2], i12); d[3] = add(a.x[0], i03);
  }
  static __device__ __forceinline__ void add_to(const bool* has, H* base, const unsigned* kid, unsigned ro, int NT,
                                                const H* d) {
    H cur[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) cur[q] = has[q] ? base[(size_t)(kid[q] + ro) * NT] : zero();
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (has[q]) base[(size_t)(kid[q] + ro) * NT] = add(cur[q], d[q]);
  }
  static __device__ __forceinline__ void unpack(const S* p, double* s) {
    const double2 a = p->a, b = p->b;
    s[0] = a.x; s[1] = a.y; s[2] = b.x; s[3] = b.y;
  }
  static constexpr int HN = NF;
  static __device__ __forceinline__ H zero() { return make_double2(0.0, 0.0); }
  static __device__ __forceinline__ W wt(double w) { return w; }
  static __device__ __forceinline__ void fma(H& a, W w, H v) { a.x = ::fma(w, v.x, a.x); a.y = ::fma(w, v.y, a.y); }
  static __device__ __forceinline__ void fma1(H& a, double w, H v) { fma(a, w, v); }
  static __device__ __forceinline__ void fmai(H& a, double w, H v) { a.x = ::fma(-w, v.y, a.x); a.y = ::fma(w, v.x, a.y); }
  static __device__ __forceinline__ H add(H a, H b) { return make_double2(a.x + b.x, a.y + b.y); }
  static __device__ __forceinline__ H sub(H a, H b) { return make_double2(a.x - b.x, a.y - b.y); }
  static __device__ __forceinline__ H itimes(H a) { return make_double2(-a.y, a.x); }
  static __device__ __forceinline__ void t4(const double* p, double* w) {
    const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p) + 1);
    w[0] = a.x; w[1] = a.y; w[2] = b.x; w[3] = b.y;
  }
  static __device__ __forceinline__ void w4(const W* p, W* w) {
    const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
    w[0] = a.x; w[1] = a.y; w[2] = b.x; w[3] = b.y;
  }
};

__device__ __forceinline__ unsigned div_by(unsigned x, unsigned magic) { return magic ? __umulhi(x, magic) : x; }

// A thread's copies of every input row: NK 16-byte chunks at ring offsets
// 16 (tid + k T).  at[k]: chunk k of the next direct row; have, over: bit k
// set where chunk k exists (else it stays zero) and where half a turn around
// phi leaves the row.
template <int NK> struct RowCopies {
  const char* at[NK];
  unsigned have, over;
};

template <int NK>
__device__ __forceinline__ void stage_direct(RowCopies<NK>& rc, int rowb, uint32_t dst, uint32_t step) {
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    if (rc.have >> k & 1u) copy16(dst + k * step, rc.at[k]);
    rc.at[k] += rowb;
  }
}
// a reflected row `ahead` rows past (or before) the next direct one
template <int NK>
__device__ __forceinline__ void stage_turned(const RowCopies<NK>& rc, int rowb, int ahead, uint32_t dst, uint32_t step) {
#pragma unroll
  for (int k = 0; k < NK; ++k)
    if (rc.have >> k & 1u)
      copy16(dst + k * step, rc.at[k] + (long long)ahead * rowb + ((rc.over >> k & 1u) ? -(rowb >> 1) : rowb >> 1));
}

// Interpolation s -> s + 1.  Grid: x over (box group, column chunk, part
// chunk), y over ranges of TR parent rows.  vlast[tp]: the last of the four
// virtual child rows of parent row tp's stencil; virtual row v < 0 is child row
// -1 - v and v >= nthC child row 2 nthC - 1 - v, both half a turn around phi
// (the pole reflection, its sign folded into th_w).  ph_src[4 jp + 1]: the
// child column at or before column jp.
template <typename T>
__global__ void __launch_bounds__(INTERP_THREADS<T>, INTERP_CTAS<T>) k_interp_march(
    int nbox, int nthC, int nphC, int nthP, int nphP, int NT, int TR, MarchTile m, const int4* __restrict__ ch4,
    const int* __restrict__ vlast, const T* __restrict__ th_w, const int* __restrict__ ph_src,
    const T* __restrict__ ph_w, const typename Mp<T>::C* __restrict__ shift,
    const typename Mp<T>::H* __restrict__ F, typename Mp<T>::H* __restrict__ out) {
  typedef Mp<T> P;
  typedef typename P::H H;
  typedef typename P::W W;
  typedef typename P::S S;
  constexpr int HN = P::HN, NK = INTERP_NK;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(16) W sw[MARCH_ROWS * 4];  // the range's theta weights
  __shared__ int sv[MARCH_ROWS + 2];             // and last virtual rows, ended by two sentinels
  const int tid = threadIdx.x;
  const int tp0 = blockIdx.y * TR, ntr = min(nthP, tp0 + TR) - tp0;
  for (int t = tid; t < 4 * ntr; t += m.T) sw[t] = P::wt(th_w[4 * tp0 + t]);
  for (int t = tid; t < ntr + 2; t += m.T) sv[t] = t < ntr ? vlast[tp0 + t] : 1 << 30;
  int bx = blockIdx.x;
  const int bg = bx / (m.nck * m.nhk);
  bx -= bg * m.nck * m.nhk;
  const int ck = bx / m.nhk, h0 = (bx - ck * m.nhk) * HN, p0 = ck * m.ncol, B0 = bg * m.nbx;
  const int jc0 = ph_src[4 * p0 + 1] - 1;       // first staged child column (before wrapping)
  const int v0 = vlast[tp0] - 3, v1 = vlast[tp0 + ntr - 1];
  const int rowP = nphP * NT, rowb = nphC * NT * 16;
  // chunk e of a row = ((box, child), column, part); HN divides T, so all of
  // a thread's chunks are part h
  const int h = tid & (HN - 1);
  const int E = m.nbx * 4 * m.cc * HN;
  int r0 = max(v0, 0);                          // the next direct row
  RowCopies<NK> rc;
  rc.have = rc.over = 0;
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    const unsigned e = tid + k * m.T, ec = e / HN, bq = div_by(ec, m.mcc), B = B0 + (bq >> 2);
    int j = jc0 + (int)(ec - bq * m.cc);
    j = j < 0 ? j + nphC : j >= nphC ? j - nphC : j;
    const int child =
        (e < (unsigned)E && B < (unsigned)nbox && j < nphC) ? reinterpret_cast<const int*>(ch4 + B)[bq & 3] : -1;
    rc.at[k] = reinterpret_cast<const char*>(F + ((size_t)max(child, 0) * nthC * nphC + j) * NT + h0 + h) +
               (size_t)r0 * rowb;
    if (child >= 0) rc.have |= 1u << k;
    if (j >= (nphC >> 1)) rc.over |= 1u << k;
    if (child < 0 && e < (unsigned)E)
      for (int q = 0; q < 4; ++q) reinterpret_cast<H*>(smem)[q * E + e] = P::zero();
  }
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem) + 16u * tid;
  auto stage = [&](int v, int slot) {
    const uint32_t dst = sbase + slot * 16u * E, step = 16u * m.T;
    if (v <= v1) {                              // uniform
      if (v >= 0 && v < nthC) {
        stage_direct(rc, rowb, dst, step);
        ++r0;
      } else {
        stage_turned(rc, rowb, (v < 0 ? -1 - v : 2 * nthC - 1 - v) - r0, dst, step);
      }
    }
    copies_commit();
  };
  for (int k = 0; k < 3; ++k) stage(v0 + k, k);
  // this thread's output column
  const unsigned uc = tid / HN;
  const int lb = (int)div_by(uc, m.mper), lc = (int)uc - lb * m.ncol;
  const int jp = p0 + lc, B = B0 + lb;
  const bool act = lb < m.nbx && B < nbox && jp < nphP;
  const int jq = act ? jp : p0;
  W pw[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) pw[b] = P::wt(ph_w[4 * jq + b]);
  const H* tap = reinterpret_cast<const H*>(smem) +
                 ((act ? lb : 0) * 4 * m.cc + (ph_src[4 * jq + 1] - 1 - jc0)) * HN + h;
  const int kid = m.cc * HN;
  H* dst = out + ((size_t)(act ? B : B0) * nthP + tp0) * rowP + jq * NT + h0 + h;
  const S* shp = reinterpret_cast<const S*>(shift) + (size_t)tp0 * nphP + jq;
  H win[4][4];                                  // [row mod 4][sum 03, difference 03, sum 12, difference 12]
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int x = 0; x < 4; ++x) win[a][x] = P::zero();
  T s[4];
  P::unpack(shp, s);
  __syncthreads();
  const W* wt = sw;
  const int* pv = sv + 2;
  int vn = sv[0], vm = sv[1];
  // virtual row v = vb + ph: ph the window and ring slot
  for (int vb = v0;; vb += 4) {
#pragma unroll
    for (int ph = 0; ph < 4; ++ph) {
      const int v = vb + ph;
      if (v > v1) return;                       // uniform
      copies_wait2();
      __syncthreads();                          // this row landed; the previous row's slot is free
      stage(v + 3, (ph + 3) & 3);
      const H* r = tap + ph * E;
      H g[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        g[q] = P::zero();
#pragma unroll
        for (int b = 0; b < 4; ++b) P::fma(g[q], pw[b], r[b * HN]);
        r += kid;
      }
      win[ph][0] = P::add(g[0], g[3]);
      win[ph][1] = P::sub(g[0], g[3]);
      win[ph][2] = P::add(g[1], g[2]);
      win[ph][3] = P::sub(g[1], g[2]);
      while (vn == v) {                         // every parent row whose stencil ends here
        W w[4];
        P::w4(wt, w);
        wt += 4;
        vn = vm;
        vm = *pv++;
        H o = P::zero();
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          H z = P::zero();
#pragma unroll
          for (int a = 0; a < 4; ++a) P::fma(z, w[a], win[(ph + 1 + a) & 3][x]);
          if (x & 1) P::fmai(o, s[x], z);
          else P::fma1(o, s[x], z);
        }
        if (vn < (1 << 30)) P::unpack(shp += nphP, s);   // the next row's shifts
        if (act) *dst = o;
        dst += rowP;
      }
    }
  }
}

// Anterpolation s + 1 -> s.  Grid: x over (box group, column chunk, part
// chunk), y over ranges of TI child rows.  The parent rows arrive in the order
// of the child rows their theta stencils start at (entries ent: parent row |
// reflected << 16; entw the weights of child rows b .. b + 3 for the entries
// ent_ptr[b] .. ent_ptr[b + 1], the parent's quadrature weight and the
// child's inverse one folded in).  A stencil that reaches past a pole is a
// second, reflected entry, half a turn around phi.  Per entry the
// phi-transposed taps (consecutive parent columns from pst[j] + q0, weights
// ptw [nph][pm]; PM of them, or `taps` if PM is 0) give the thread's child
// column the Re- and Im-weighted sums of both conjugate pairs; the window
// scatters them to four child rows, and a row that no later entry reaches is
// added to the four children's incoming spectra.
template <typename T, int PM, int NK = ANTERP_NK>
__global__ void __launch_bounds__(ANTERP_THREADS<T>, ANTERP_CTAS<T>) k_anterp_march(
    int nbox, int nthC, int nphC, int nthP, int nphP, int NT, int TI, MarchTile m, const int4* __restrict__ ch4,
    const int* __restrict__ ent_ptr, const int* __restrict__ ent, const T* __restrict__ entw,
    const int* __restrict__ pst, const T* __restrict__ ptw, int pm, int taps, int q0,
    const typename Mp<T>::S* __restrict__ shift, const typename Mp<T>::H* __restrict__ inP,
    typename Mp<T>::H* __restrict__ inC) {
  typedef Mp<T> P;
  typedef typename P::H H;
  typedef typename P::S S;
  typedef typename P::G G;
  constexpr int HN = P::HN;
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x;
  const int i0 = blockIdx.y * TI, i1 = min(nthC, i0 + TI);
  int bx = blockIdx.x;
  const int bg = bx / (m.nck * m.nhk);
  bx -= bg * m.nck * m.nhk;
  const int ck = bx / m.nhk, h0 = (bx - ck * m.nhk) * HN, p0 = ck * m.ncol, B0 = bg * m.nbx;
  const int jp0 = pst[p0] + q0;                 // first staged parent column (before wrapping)
  constexpr int SP = sizeof(S) / 16;            // 16-byte pieces of a direction's shifts
  const int h = tid & (HN - 1);
  // chunk e of a row = (box, column, part), then the row's shifts
  const int Ev = m.nbx * m.cc * HN, E = Ev + m.cc * SP;
  const int b0 = max(0, i0 - 3), nb = max(1, nthC - 3);
  int e = ent_ptr[min(b0, nb)];
  const int e_end = ent_ptr[min(i1, nb)];
  int pk = e < e_end ? ent[e] : 0;              // the next entry to stage
  const int rowb = nphP * NT * 16, rows = nphP * SP * 16;
  RowCopies<NK> rc;
  unsigned shb = 0;                             // bit k: chunk k is of the shifts
  rc.have = rc.over = 0;
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    const unsigned c = tid + k * m.T;
    const bool sh = c >= (unsigned)Ev;
    const unsigned ec = sh ? (c - Ev) / SP : c / HN, lb = sh ? 0u : div_by(ec, m.mcc);
    int j = jp0 + (int)(ec - lb * m.cc);
    j = j < 0 ? j + nphP : j >= nphP ? j - nphP : j;
    const bool ok = c < (unsigned)E && B0 + (int)lb < nbox && j >= 0 && j < nphP;
    rc.at[k] = sh ? reinterpret_cast<const char*>(shift + j) + (c - Ev) % SP * 16
                  : reinterpret_cast<const char*>(inP + ((size_t)(B0 + lb) * nthP * nphP + j) * NT + h0 + h);
    if (ok) rc.have |= 1u << k;
    if (j >= (nphP >> 1)) rc.over |= 1u << k;
    if (sh) shb |= 1u << k;
    if (!ok && c < (unsigned)E)
      for (int q = 0; q < 4; ++q) reinterpret_cast<H*>(smem)[q * E + c] = P::zero();
  }
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem) + 16u * tid;
  auto stage = [&](int i) {                     // entry i, packed in pk
    if (i < e_end) {                            // uniform
      const uint32_t dst = sbase + (i & 3) * 16u * E, step = 16u * m.T;
      const int tp = pk & 0xffff;
      if (!(pk >> 16)) {
        const long long ov = (long long)tp * rowb, os = (long long)tp * rows;
#pragma unroll
        for (int k = 0; k < NK; ++k)
          if (rc.have >> k & 1u) copy16(dst + k * step, rc.at[k] + ((shb >> k & 1u) ? os : ov));
      } else {
#pragma unroll
        for (int k = 0; k < NK; ++k)
          if (rc.have >> k & 1u) {
            const int len = (shb >> k & 1u) ? rows : rowb;
            copy16(dst + k * step, rc.at[k] + (long long)tp * len + ((rc.over >> k & 1u) ? -(len >> 1) : len >> 1));
          }
      }
    }
    copies_commit();
    if (i + 1 < e_end) pk = ent[i + 1];
  };
  for (int k = 0; k < 3; ++k) stage(e + k);
  // this thread's child column
  const unsigned uc = tid / HN;
  const int lb = (int)div_by(uc, m.mper), lc = (int)uc - lb * m.ncol;
  const int B = B0 + lb;
  const bool act = lb < m.nbx && B < nbox && p0 + lc < nphC;
  const int j = act ? p0 + lc : p0;
  const int4 c4 = act ? ch4[B] : make_int4(-1, -1, -1, -1);
  const unsigned Kc = (unsigned)(nthC * nphC);
  H* Ch = inC + h0 + h;
  const unsigned kid[4] = {(unsigned)c4.x * Kc + j, (unsigned)c4.y * Kc + j, (unsigned)c4.z * Kc + j,
                           (unsigned)c4.w * Kc + j};
  const bool has[4] = {c4.x >= 0, c4.y >= 0, c4.z >= 0, c4.w >= 0};
  const int tcol = pst[j] + q0 - jp0;
  const H* tap = reinterpret_cast<const H*>(smem) + ((act ? lb : 0) * m.cc + tcol) * HN + h;
  const int stap = (Ev - ((act ? lb : 0) * m.cc + tcol) * HN - h) * 16 + tcol * (int)sizeof(S);
  T w[PM > 0 ? PM : 1];
  if (PM > 0) {
#pragma unroll
    for (int q = 0; q < PM; ++q) w[q] = ptw[(size_t)j * pm + q];
  }
  G acc[4];                                     // [child row mod 4]
#pragma unroll
  for (int a = 0; a < 4; ++a) P::gzero(acc[a]);
  int e1 = ent_ptr[min(b0 + 1, nb)];
  // child row b = bb + ph: ph the window slot
  for (int bb = b0;; bb += 4) {
#pragma unroll
    for (int ph = 0; ph < 4; ++ph) {
      const int b = bb + ph;
      if (b >= i1) return;                      // uniform
      const int e2 = ent_ptr[min(b + 2, nb)];
      for (; e < e1; ++e) {
        T tw[4];
        P::t4(entw + 4 * (size_t)e, tw);
        copies_wait2();
        __syncthreads();                        // this entry's row landed; the previous one's slot is free
        stage(e + 3);
        const H* r = tap + (e & 3) * E;
        const S* rs = reinterpret_cast<const S*>(reinterpret_cast<const char*>(r) + stap);
        G g;
        P::gzero(g);
#pragma unroll
        for (int q = 0; q < (PM > 0 ? PM : taps); ++q)
          P::tap(g, PM > 0 ? w[PM > 0 ? q : 0] : ptw[(size_t)j * pm + q], r[q * HN], rs + q);
#pragma unroll
        for (int a = 0; a < 4; ++a) P::scatter(acc[(ph + a) & 3], tw[a], g);
      }
      e1 = e2;
      if (b >= i0) {
        const unsigned ro = (unsigned)(b * nphC);
        H d[4];
        P::children(acc[ph], d);
        P::add_to(has, Ch, kid, ro, NT, d);
      }
      P::gzero(acc[ph]);
    }
  }
}

template <typename T>
int interp_impl(Ctx* c, int s, int R, cudaStream_t st) {
  typedef Mp<T> P;
  const bool f64 = sizeof(T) == 8;
  const Level &Lc = c->lev[s], &Lp = c->lev[s + 1];
  const int NT = P::HN * R;
  const MarchTile m = march_tile(INTERP_THREADS<T>, INTERP_NK, P::HN, P::HN, !f64, Lp.nbox, Lp.nph, NT, Lc.mi_start, 4, 4, 0);
  // FP64: the two FP64 lanes of an SM are the bound, CTAs of one SM take turns
  const int TR = march_rows(m, Lp.nth, f64 ? 1 : 65536 / (128 * m.T), MARCH_ROWS);
  const size_t sm = (size_t)4 * 16 * m.nbx * 4 * m.cc * P::HN;
  cudaFuncSetAttribute(k_interp_march<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
  dim3 g((unsigned)((long long)m.nbg * m.nck * m.nhk), (unsigned)((Lp.nth + TR - 1) / TR));
  k_interp_march<T><<<g, m.T, sm, st>>>(
      Lp.nbox, Lc.nth, Lc.nph, Lp.nth, Lp.nph, NT, TR, m, (const int4*)Lp.d_ch4, Lc.d_mi_vlast,
      (const T*)(f64 ? (void*)Lc.d_th_ws64 : (void*)Lc.d_th_ws32), Lc.d_ph_src,
      (const T*)(f64 ? (void*)Lc.d_ph_w64 : (void*)Lc.d_ph_w32),
      (const typename P::C*)(f64 ? (void*)Lc.d_shiftp64 : (void*)Lc.d_shiftp32),
      (const typename P::H*)Lc.d_out, (typename P::H*)Lp.d_out);
  SMR_LAUNCH(c);
  return SMR_OK;
}

template <typename T>
int anterp_impl(Ctx* c, int s, int R, cudaStream_t st) {
  typedef Mp<T> P;
  const bool f64 = sizeof(T) == 8;
  const Level &Lc = c->lev[s], &Lp = c->lev[s + 1];
  const int NT = P::HN * R, sp = (int)sizeof(typename P::S) / 16;
  int taps;
  const MarchTile m = anterp_tile(ANTERP_THREADS<T>, Lc.ma_pm <= 8 ? ANTERP_NK : 16, P::HN, P::HN, !f64, Lp.nbox,
                                  Lc.nph, NT, Lc.ma_start, Lc.ma_pm, sp, &taps);
  const int TI = march_rows(m, Lc.nth, f64 ? 1 : 65536 / (168 * m.T), Lc.nth);
  const size_t sm = (size_t)4 * 16 * m.cc * (m.nbx * P::HN + sp);
  auto k = Lc.ma_pm == 7 ? k_anterp_march<T, 7> : Lc.ma_pm == 8 ? k_anterp_march<T, 8> : k_anterp_march<T, 0, 16>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  dim3 g((unsigned)((long long)m.nbg * m.nck * m.nhk), (unsigned)((Lc.nth + TI - 1) / TI));
  // one launch but for stencils too wide for a CTA (above 768 parent columns in
  // FP64, 1,024 in FP32), whose taps are divided: every launch adds its part
  for (int q0 = 0; q0 < Lc.ma_pm; q0 += taps) {
    k<<<g, m.T, sm, st>>>(Lp.nbox, Lc.nth, Lc.nph, Lp.nth, Lp.nph, NT, TI, m, (const int4*)Lp.d_ch4, Lc.d_ma_ptr,
                          Lc.d_ma_ent, (const T*)(f64 ? (void*)Lc.d_ma_w64 : (void*)Lc.d_ma_w32), Lc.d_ma_pst,
                          (const T*)(f64 ? (void*)Lc.d_ma_pw64 : (void*)Lc.d_ma_pw32) + q0, Lc.ma_pm,
                          std::min(taps, Lc.ma_pm - q0), q0,
                          (const typename P::S*)(f64 ? (void*)Lc.d_shiftp64 : (void*)Lc.d_shiftp32),
                          (const typename P::H*)Lp.d_in, (typename P::H*)Lc.d_in);
    SMR_LAUNCH(c);
  }
  return SMR_OK;
}

}  // namespace

int run_interp(Ctx* c, int s, int R, int prec, cudaStream_t st) {
  return prec == SMR_PREC_FP64 ? interp_impl<double>(c, s, R, st) : interp_impl<float>(c, s, R, st);
}

int run_anterp(Ctx* c, int s, int R, int prec, cudaStream_t st) {
  return prec == SMR_PREC_FP64 ? anterp_impl<double>(c, s, R, st) : anterp_impl<float>(c, s, R, st);
}

}  // namespace smr

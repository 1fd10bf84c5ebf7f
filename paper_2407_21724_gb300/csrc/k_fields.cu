// Fields of a solution: far-field amplitudes, cross sections, near fields.  All
// in FP64, whose rate (2 FMA per clock and SM, 64 clocks between the
// instructions of a warp scheduler) bounds every kernel here: what counts is the
// number of FP64 instructions, and memory and integer work hide behind them.
#include <cmath>
#include <cstring>

#include "smr_internal.h"

namespace smr {

namespace {

// length of u, unit vector t along it (z for a zero vector), and e1, e2 with
// e1 x e2 = t
__device__ double dir_basis(const double* u, double* t, double* e1, double* e2) {
  const double n = sqrt(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
  t[0] = 0; t[1] = 0; t[2] = 1;
  if (n != 0)
    for (int i = 0; i < 3; ++i) t[i] = u[i] / n;
  if (fabs(t[2]) < 0.9) {
    const double h = 1.0 / sqrt(t[0] * t[0] + t[1] * t[1]);
    e1[0] = -t[1] * h; e1[1] = t[0] * h; e1[2] = 0;
  } else {
    const double h = 1.0 / sqrt(t[1] * t[1] + t[2] * t[2]);
    e1[0] = 0; e1[1] = -t[2] * h; e1[2] = t[1] * h;
  }
  e2[0] = t[1] * e1[2] - t[2] * e1[1];
  e2[1] = t[2] * e1[0] - t[0] * e1[2];
  e2[2] = t[0] * e1[1] - t[1] * e1[0];
  return n;
}

// a direction whose length is 1 up to rounding needs no radial component
__device__ __forceinline__ bool not_unit(double n) { return !(fabs(1.0 - n * n) <= 1e-14); }

__device__ __forceinline__ void cfma(double2& a, double2 x, double2 y) {
  a.x = fma(x.x, y.x, a.x); a.x = fma(-x.y, y.y, a.x);
  a.y = fma(x.x, y.y, a.y); a.y = fma(x.y, y.x, a.y);
}

}  // namespace

// ------------------------------------------------------------------ far field
// Rv[s][n][i][d] = sum_q w psi_n(q) exp(+j k u_d . r_q), the radiation vectors
// along e1, e2 and u_d.  CTA = D directions x 32 modes (4 per thread) of one
// shape; the threads of a direction and a mode group are T / (8 D) and take
// every so manieth surface point.  The phases of 64 surface points are computed
// once per CTA into shared memory: a thread per (mode, direction) that recomputes
// them for each mode spends 8 times more instructions on them than on the sums.
// With few directions the surface points are also divided over blockIdx.y, one
// slice of Rv each (a CTA's 512 points take some 0.5 ms whatever the number of
// CTAs).  D = 16 spends the FP64 rate on absent directions too; D = 4 is taken
// where it spends it on at least an eighth fewer: 300 shapes of 32 modes, one
// direction 1.41 -> 0.69 ms (20 directions 2.3 -> 1.6), a thread per mode and
// direction 1.18.
constexpr int RV_N = 4, RV_T = 128, RV_Q = 64, RV_M = 8 * RV_N;

template <int D>
__global__ void __launch_bounds__(RV_T) k_radvec(int npsi, int Q, int nd, int ndt, int nng,
                                                 const double* __restrict__ modes, const double* __restrict__ rq,
                                                 const double* __restrict__ dirs, double kw, size_t slice,
                                                 double2* __restrict__ Rv) {
  constexpr int SL = RV_T / (8 * D);               // threads that share a direction and a mode group
  __shared__ double2 ph[RV_Q][D];
  const int dt = blockIdx.x % ndt, g = (blockIdx.x / ndt) % nng, s = blockIdx.x / (ndt * nng);
  const int dl = threadIdx.x % D, d = min(dt * D + dl, nd - 1), sl = threadIdx.x / (8 * D);
  const int n0 = g * RV_M + threadIdx.x / D % 8 * RV_N;
  const double u[3] = {dirs[3 * d], dirs[3 * d + 1], dirs[3 * d + 2]};
  const double* Rr = rq + (size_t)s * Q * 4;
  const double* M[RV_N];
#pragma unroll
  for (int i = 0; i < RV_N; ++i) M[i] = modes + ((size_t)s * npsi + min(n0 + i, npsi - 1)) * Q * 4;
  double2 a[RV_N][3] = {};
  const int nch = (Q + RV_Q - 1) / RV_Q;
  const int qe = min(Q, (int)((long long)nch * (blockIdx.y + 1) / gridDim.y) * RV_Q);
  for (int q0 = (int)((long long)nch * blockIdx.y / gridDim.y) * RV_Q; q0 < qe; q0 += RV_Q) {
    const int nq = min(RV_Q, qe - q0);
    __syncthreads();
    for (int q = threadIdx.x / D; q < nq; q += RV_T / D) {
      const double* p = Rr + 4 * (q0 + q);
      double sn, cs;
      sincos(kw * (u[0] * p[0] + u[1] * p[1] + u[2] * p[2]), &sn, &cs);
      ph[q][dl] = make_double2(p[3] * cs, p[3] * sn);
    }
    __syncthreads();
#pragma unroll 2
    for (int q = sl; q < nq; q += SL) {
      const double2 e = ph[q][dl];
#pragma unroll
      for (int i = 0; i < RV_N; ++i) {
        const double2 m0 = *reinterpret_cast<const double2*>(M[i] + 4 * (q0 + q));
        const double m2 = M[i][4 * (q0 + q) + 2];
        a[i][0].x = fma(m0.x, e.x, a[i][0].x); a[i][0].y = fma(m0.x, e.y, a[i][0].y);
        a[i][1].x = fma(m0.y, e.x, a[i][1].x); a[i][1].y = fma(m0.y, e.y, a[i][1].y);
        a[i][2].x = fma(m2, e.x, a[i][2].x); a[i][2].y = fma(m2, e.y, a[i][2].y);
      }
    }
  }
  if constexpr (SL > 1) {
    __shared__ double2 red[SL][RV_N * 3][8 * D];
    const int t = threadIdx.x % (8 * D);
#pragma unroll
    for (int i = 0; i < RV_N * 3; ++i) red[sl][i][t] = a[i / 3][i % 3];
    __syncthreads();
    if (sl) return;
#pragma unroll
    for (int i = 0; i < RV_N * 3; ++i)
      for (int k = 1; k < SL; ++k) {
        a[i / 3][i % 3].x += red[k][i][t].x;
        a[i / 3][i % 3].y += red[k][i][t].y;
      }
  }
  if (dt * D + dl >= nd) return;
  double t[3], e1[3], e2[3];
  dir_basis(u, t, e1, e2);
#pragma unroll
  for (int i = 0; i < RV_N; ++i) {
    if (n0 + i >= npsi) break;
    double2* o = Rv + blockIdx.y * slice + ((size_t)s * npsi + n0 + i) * 3 * nd + d;
    o[0] = make_double2(e1[0] * a[i][0].x + e1[1] * a[i][1].x + e1[2] * a[i][2].x,
                        e1[0] * a[i][0].y + e1[1] * a[i][1].y + e1[2] * a[i][2].y);
    o[nd] = make_double2(e2[0] * a[i][0].x + e2[1] * a[i][1].x + e2[2] * a[i][2].x,
                         e2[0] * a[i][0].y + e2[1] * a[i][1].y + e2[2] * a[i][2].y);
    o[2 * (size_t)nd] = make_double2(t[0] * a[i][0].x + t[1] * a[i][1].x + t[2] * a[i][2].x,
                                     t[0] * a[i][0].y + t[1] * a[i][1].y + t[2] * a[i][2].y);
  }
}

// slice 0 of Rv += the other slices
__global__ void k_rv_sum(size_t n, int ns, double2* __restrict__ Rv) {
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  double2 v = Rv[t];
  for (int i = 1; i < ns; ++i) {
    const double2 w = Rv[t + i * n];
    v.x += w.x;
    v.y += w.y;
  }
  Rv[t] = v;
}

// part[unit][d][i][r]: the amplitude's components along e1, e2 and u from C
// consecutive particles of the list sorted by shape.  CTA = 32 directions
// (lanes); a warp sums exp(+j k u.c) x over the particles of one shape for 16
// coefficients in registers and multiplies by the shape's radiation vectors when
// the shape changes: 8 FMA a mode and direction (both currents) where a product
// with the radiation vectors for each particle takes 24.  Cross sections of 40x40
// particles over 1,153 directions: 15.3 ms with a CTA per direction reading all
// coefficients with a stride and recomputed phases, 3.2 ms so.
constexpr int FF_T = 128, FF_P = 16, FF_C = 16;

__global__ void __launch_bounds__(FF_T) k_farfield(int p, int npsi, int nd, int R, int C,
                                                   const int* __restrict__ order, const int* __restrict__ sid,
                                                   const double* __restrict__ cen, const double* __restrict__ dirs,
                                                   const double2* __restrict__ Rv, const double2* __restrict__ x,
                                                   double kw, double zeta, double2* __restrict__ part) {
  __shared__ double2 ph[FF_P][32];
  __shared__ int smu[FF_P], ssh[FF_P];
  __shared__ double2 red[FF_T / 32][3][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = blockIdx.x / R, r = blockIdx.x % R, unit = blockIdx.y;
  const int dd = tile * 32 + lane, d = min(dd, nd - 1);
  const double u[3] = {dirs[3 * d], dirs[3 * d + 1], dirs[3 * d + 2]};
  const double len = sqrt(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
  const bool radial = not_unit(len);
  const int e0 = unit * C, e1 = min(p, e0 + C), n2 = 2 * npsi;
  double2 f[3] = {};
  for (int c0 = 0; c0 < n2; c0 += FF_C * FF_T / 32) {
    const int cb = c0 + FF_C * warp;
    double2 Y[FF_C] = {};
    int cur = -1;
    auto flush = [&]() {
      if (cur < 0) return;
#pragma unroll
      for (int i = 0; i < FF_C; ++i) {
        const int ci = cb + i;
        if (ci < n2) {
          const int m = ci >= npsi;
          const double sc = m ? len : zeta;
          const double2 y = make_double2(sc * Y[i].x, sc * Y[i].y);
          const double2* v = Rv + ((size_t)cur * npsi + ci - m * npsi) * 3 * nd + d;
          const double2 v1 = v[0], v2 = v[nd];
          if (!m) {                                     // zeta J - u (u . J)
            cfma(f[0], y, v1);
            cfma(f[1], y, v2);
            if (radial) cfma(f[2], y, v[2 * (size_t)nd]);
          } else {                                      // - u x M
            cfma(f[0], y, v2);
            cfma(f[1], y, make_double2(-v1.x, -v1.y));
          }
        }
        Y[i] = make_double2(0, 0);
      }
    };
    for (int b0 = e0; b0 < e1; b0 += FF_P) {
      const int nb = min(FF_P, e1 - b0);
      __syncthreads();
      for (int j = warp; j < nb; j += FF_T / 32) {
        const int mu = order[b0 + j];
        const double* cc = cen + 3 * mu;
        double sn, cs;
        sincos(kw * (u[0] * cc[0] + u[1] * cc[1] + u[2] * cc[2]), &sn, &cs);
        ph[j][lane] = make_double2(cs, sn);
        if (lane == 0) {
          smu[j] = mu;
          ssh[j] = sid[mu];
        }
      }
      __syncthreads();
      if (cb < n2)
        for (int j = 0; j < nb; ++j) {
          if (ssh[j] != cur) {
            flush();
            cur = ssh[j];
          }
          const double2 e = ph[j][lane];
          const double2* xr = x + (size_t)smu[j] * n2 * R + r;
#pragma unroll
          for (int i = 0; i < FF_C; ++i) cfma(Y[i], xr[(size_t)min(cb + i, n2 - 1) * R], e);
        }
    }
    if (cb < n2) flush();
  }
  for (int i = 0; i < 3; ++i) red[warp][i][lane] = f[i];
  __syncthreads();
  if (warp < 3 && dd < nd) {
    double2 v = red[0][warp][lane];
    for (int w = 1; w < FF_T / 32; ++w) {
      v.x += red[w][warp][lane].x;
      v.y += red[w][warp][lane].y;
    }
    part[(((size_t)unit * nd + dd) * 3 + warp) * R + r] = v;
  }
}

// F[d][3][r] = j k / (4 pi) times the sum of the units' parts, in Cartesian
// components; the part along u, zeta (1 - u.u) J, vanishes for unit directions
__global__ void k_far_sum(int nd, int R, int nu, const double* __restrict__ dirs, const double2* __restrict__ part,
                          double kw, double2* __restrict__ F) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)nd * R) return;
  const int d = (int)(t / R), r = (int)(t % R);
  double2 f[3] = {};
  for (int u = 0; u < nu; ++u)
    for (int i = 0; i < 3; ++i) {
      const double2 v = part[(((size_t)u * nd + d) * 3 + i) * R + r];
      f[i].x += v.x;
      f[i].y += v.y;
    }
  double b[3][3];
  const double len = dir_basis(dirs + 3 * (size_t)d, b[2], b[0], b[1]);
  const double w3 = not_unit(len) ? 1.0 - len * len : 0.0, pre = kw / (4.0 * M_PI);
  for (int i = 0; i < 3; ++i)
    F[((size_t)d * 3 + i) * R + r] =
        make_double2(-pre * (b[0][i] * f[0].y + b[1][i] * f[1].y + w3 * b[2][i] * f[2].y),
                     pre * (b[0][i] * f[0].x + b[1][i] * f[1].x + w3 * b[2][i] * f[2].x));
}

int launch_far_field(Ctx* c, int R, const double2* x, int nd, const double* d_dirs, double2* F,
                     cudaStream_t st) {
  // units of at least FF_P particles, as many as fill the 152 SMs with 8 CTAs
  // each: smaller ones spend more on the products with the radiation vectors than
  // on the sums.  Splits of the surface points up to 4 CTAs an SM (64 directions
  // of 40x40 particles: far field 0.93 ms without, 0.51 with).
  const int tiles = (nd + 31) / 32;
  const int want = (int)std::min<long long>((c->p + FF_P - 1) / FF_P,
                                            std::max<long long>(1, 1216 / ((long long)tiles * R)));
  const int C = (c->p + want - 1) / want, nu = (c->p + C - 1) / C;
  double2 *Rv = nullptr, *part = nullptr;
  const int d4 = (nd + 3) / 4 * 4, d16 = (nd + 15) / 16 * 16, D = 8 * d16 > 9 * d4 ? 4 : 16;
  const int ndt = (nd + D - 1) / D, nng = (c->npsi + RV_M - 1) / RV_M;
  const long long ctas = (long long)c->S * nng * ndt;
  const int nqs = std::min((c->Q + RV_Q - 1) / RV_Q, ctas < 608 ? (int)(608 / ctas) : 1);
  const size_t slice = (size_t)c->S * c->npsi * nd * 3;
  SMR_CUDA(c, cudaMallocAsync((void**)&Rv, nqs * slice * sizeof(double2), st));
  const cudaError_t e = cudaMallocAsync((void**)&part, (size_t)nu * nd * 3 * R * sizeof(double2), st);
  if (e != cudaSuccess) cudaFreeAsync(Rv, st);
  SMR_CUDA(c, e);
  const dim3 gr((unsigned)ctas, (unsigned)nqs);
  auto k = D == 4 ? k_radvec<4> : k_radvec<16>;
  k<<<gr, RV_T, 0, st>>>(c->npsi, c->Q, nd, ndt, nng, c->d_modes, c->d_rq, d_dirs, c->k, slice, Rv);
  SMR_LAUNCH(c);
  if (nqs > 1) {
    k_rv_sum<<<(unsigned)((slice + 255) / 256), 256, 0, st>>>(slice, nqs, Rv);
    SMR_LAUNCH(c);
  }
  const dim3 gf((unsigned)tiles * (unsigned)R, (unsigned)nu);
  k_farfield<<<gf, FF_T, 0, st>>>(
      c->p, c->npsi, nd, R, C, c->d_perm, c->d_sid, c->d_centres, d_dirs, Rv, x, c->k, c->zeta, part);
  SMR_LAUNCH(c);
  k_far_sum<<<(unsigned)(((long long)nd * R + 127) / 128), 128, 0, st>>>(nd, R, nu, d_dirs, part, c->k, F);
  SMR_LAUNCH(c);
  SMR_CUDA(c, cudaFreeAsync(part, st));
  SMR_CUDA(c, cudaFreeAsync(Rv, st));
  return SMR_OK;
}

// Cross sections from far-field amplitudes F[nd][3][R].  CTA per column r:
// the first n_sca directions carry quadrature weights W (scattered power
// over the sphere, Sec. V); direction n_sca + r is column r's own incident
// direction, where the optical theorem gives the extinction.  cs[2r] = C_sca,
// cs[2r + 1] = C_ext.
__global__ void k_cross_sections(int n_sca, int R, const double2* __restrict__ F,
                                 const double* __restrict__ W, const double2* __restrict__ pol,
                                 double kw, double* __restrict__ cs) {
  __shared__ double red[256];
  int r = blockIdx.x;
  double acc = 0;
  for (int d = threadIdx.x; d < n_sca; d += blockDim.x) {
    double e = 0;
    for (int i = 0; i < 3; ++i) {
      double2 f = F[((size_t)d * 3 + i) * R + r];
      e += f.x * f.x + f.y * f.y;
    }
    acc += W[d] * e;
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    // Im(conj(e) . F) / |e|^2 at the forward direction.
    double im = 0, nn = 0;
    for (int i = 0; i < 3; ++i) {
      double2 e = pol[(size_t)r * 3 + i];
      double2 f = F[((size_t)(n_sca + r) * 3 + i) * R + r];
      im += e.x * f.y - e.y * f.x;
      nn += e.x * e.x + e.y * e.y;
    }
    cs[2 * r] = red[0];
    cs[2 * r + 1] = -(4.0 * M_PI / kw) * im / nn;
  }
}

int launch_cross_sections(Ctx* c, int R, const double2* x, int n_sca, const double* d_dirs,
                          const double* d_w, const double2* d_pol, double* d_cs, cudaStream_t st) {
  int nd = n_sca + R;
  double2* F = nullptr;
  SMR_CUDA(c, cudaMallocAsync((void**)&F, (size_t)nd * 3 * R * sizeof(double2), st));
  int rc = launch_far_field(c, R, x, nd, d_dirs, F, st);
  if (rc == SMR_OK) {
    k_cross_sections<<<R, 256, 0, st>>>(n_sca, R, F, d_w, d_pol, c->k, d_cs);
    SMR_LAUNCH(c);
  }
  SMR_CUDA(c, cudaFreeAsync(F, st));
  return rc;
}

// ------------------------------------------------------------------ near field
// E = j k zeta sum G [J + c (d (div J) / k + d x M')],
// H = -k sum G [M' + c (d (div M') / k + d x J)], M' = M / (j zeta),
// over all surface points, d = point - source, G = w exp(-j k R) / (4 pi R) and
// c = -(1 / (k R^2) + j / R): both operators of both currents with 84 FMA.
// Units (particle, NF_Q surface points): a unit's currents J, div J / k, M',
// div M' / k times w / (4 pi) are staged in shared memory; thread = one of tp
// field points and every (256 / tp)-th surface point, sums in registers, added
// over the threads and to EH once per CTA.  Phases and distances take 27 FP64
// instructions: 1/R by one Halley step x + x e (1/2 + 3/8 e), e = 1 - R^2 x^2,
// from a single-precision seed (error ~ e^3 ~ 1e-20) and R = R^2 / R with one
// Newton correction, exp(-j k R) by rotating
// the nearest of 512 tabulated phases (table-driven reduction, P. T. P. Tang
// 1989) by a Taylor polynomial (|r| < 0.0062: r^7 / 5040 and r^6 / 720 stay below
// 1e-16); library sqrt, divide and sincos took some 70 and the divisions by k and
// zeta inside the loop 180 more.  1,600 particles, 128 points: 69.7 ms before,
// 22.2 now, 118 instructions a pair at the FP64 rate being 21.3.
constexpr int NF_T = 256, NF_Q = 128, NF_TAB = 512;

__global__ void __launch_bounds__(NF_T, 2) k_nearfield(int p, int npsi, int Q, int npt, int R, int tp, int gx,
                                                       unsigned hi0, unsigned hspan, const int* __restrict__ sid,
                                                       const double* __restrict__ cen,
                                                       const double* __restrict__ modes,
                                                       const double* __restrict__ rq, const double2* __restrict__ x,
                                                       const double* __restrict__ pts, double kw, double zeta,
                                                       double* __restrict__ EH) {
  __shared__ double2 cur[NF_Q * 8 + NF_Q * 2];        // [q][J xyz, div J, M' xyz, div M'], [q][point]
  __shared__ double2 tab[NF_TAB];
  double* pq = reinterpret_cast<double*>(cur + NF_Q * 8);
  const int tid = threadIdx.x;
  const int i0 = blockIdx.x % gx, r = blockIdx.x / gx % R;
  const long long g0 = (long long)(blockIdx.x / gx / R) * tp;
  const int nsub = NF_T / tp, sub = tid / tp;
  const long long ip = g0 + tid % tp;
  const double* pt = pts + 3 * min(ip, (long long)npt - 1);
  const double P0 = pt[0], P1 = pt[1], P2 = pt[2];
  for (int i = tid; i < NF_TAB; i += NF_T) {
    double sn, cs;
    sincospi(i * (2.0 / NF_TAB), &sn, &cs);
    tab[i] = make_double2(cs, -sn);
  }
  const double step = NF_TAB / (2.0 * M_PI), s1 = 2.0 * M_PI / NF_TAB, s2 = 2.4492935982947064e-16 / NF_TAB;
  const double nik = -1.0 / kw, w4 = 1.0 / (4.0 * M_PI), iz = 1.0 / zeta, ik = 1.0 / kw;
  double2 E[3] = {}, H[3] = {};
  const int nch = (Q + NF_Q - 1) / NF_Q;
  for (long long un = i0; un < (long long)p * nch; un += gx) {
    const int mu = (int)(un / nch), q0 = (int)(un % nch) * NF_Q, nq = min(NF_Q, Q - q0);
    const int s = sid[mu];
    __syncthreads();
    {
      // half the threads stage J, half M
      const int q = tid % NF_Q, m = tid / NF_Q;
      if (q < nq) {
        const double* Ms = modes + (size_t)s * npsi * Q * 4 + (size_t)(q0 + q) * 4;
        const double2* xr = x + ((size_t)mu * 2 + m) * npsi * R + r;
        double2 a[4] = {};
#pragma unroll 4
        for (int n = 0; n < npsi; ++n) {
          const double2 v = xr[(size_t)n * R];
          const double2 ma = *reinterpret_cast<const double2*>(Ms + (size_t)n * Q * 4);
          const double2 mb = *reinterpret_cast<const double2*>(Ms + (size_t)n * Q * 4 + 2);
          a[0].x = fma(v.x, ma.x, a[0].x); a[0].y = fma(v.y, ma.x, a[0].y);
          a[1].x = fma(v.x, ma.y, a[1].x); a[1].y = fma(v.y, ma.y, a[1].y);
          a[2].x = fma(v.x, mb.x, a[2].x); a[2].y = fma(v.y, mb.x, a[2].y);
          a[3].x = fma(v.x, mb.y, a[3].x); a[3].y = fma(v.y, mb.y, a[3].y);
        }
        const double* rr = rq + ((size_t)s * Q + q0 + q) * 4;
        const double w = rr[3] * w4 * (m ? iz : 1.0);
        for (int i = 0; i < 4; ++i) {
          const double wi = i == 3 ? w * ik : w;
          cur[q * 8 + 4 * m + i] = m ? make_double2(wi * a[i].y, -wi * a[i].x) : make_double2(wi * a[i].x, wi * a[i].y);
        }
        if (!m)
          for (int i = 0; i < 3; ++i) pq[4 * q + i] = rr[i] + cen[3 * mu + i];
      }
    }
    __syncthreads();
    for (int q = sub; q < nq; q += nsub) {
      const double2 pa = *reinterpret_cast<const double2*>(pq + 4 * q);
      const double d0 = P0 - pa.x, d1 = P1 - pa.y, d2 = P2 - pq[4 * q + 2];
      const double R2 = fma(d2, d2, fma(d1, d1, d0 * d0));
      const unsigned hi = (unsigned)__double2hiint(R2), lo = (unsigned)__double2loint(R2);
      double iR, ex, ey;
      if (hi - hi0 < hspan) {
        const float sf = rsqrtf(__uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29)));
        const unsigned sb = __float_as_uint(sf);
        const double y = __hiloint2double((int)((sb >> 3) + 0x38000000u), (int)(sb << 29));
        const double e = fma(-(R2 * y), y, 1.0);
        iR = fma(y * e, fma(e, 0.375, 0.5), y);
        const double Ra = R2 * iR, Rr = fma(fma(-Ra, Ra, R2), 0.5 * iR, Ra), ph = kw * Rr;
        const double t = fma(ph, step, 6755399441055744.0), n = t - 6755399441055744.0;
        const double rr = fma(-n, s2, fma(-n, s1, ph)), r2 = rr * rr;
        const double sn = fma(rr * r2, fma(r2, 1.0 / 120.0, -1.0 / 6.0), rr), c1 = r2 * fma(r2, 1.0 / 24.0, -0.5);
        const double2 T = tab[__double2loint(t) & (NF_TAB - 1)];
        ex = fma(T.x, c1, fma(T.y, sn, T.x));
        ey = fma(T.y, c1, fma(-T.x, sn, T.y));
      } else {                                         // out of the seed's range, or phases beyond 1e9
        const double Rr = sqrt(R2);
        double sn;
        iR = 1.0 / Rr;
        sincos(-kw * Rr, &sn, &ex);
        ey = sn;
      }
      const double gx_ = iR * ex, gy_ = iR * ey, ca = nik * iR * iR;
      const double2* c8 = cur + q * 8;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const double2 *X = c8 + 4 * h, *Z = c8 + 4 * (1 - h);
        const double2 z0 = Z[0], z1 = Z[1], z2 = Z[2], dv = X[3];
        double2 V[3];
        V[0] = make_double2(fma(d0, dv.x, fma(d1, z2.x, -d2 * z1.x)), fma(d0, dv.y, fma(d1, z2.y, -d2 * z1.y)));
        V[1] = make_double2(fma(d1, dv.x, fma(d2, z0.x, -d0 * z2.x)), fma(d1, dv.y, fma(d2, z0.y, -d0 * z2.y)));
        V[2] = make_double2(fma(d2, dv.x, fma(d0, z1.x, -d1 * z0.x)), fma(d2, dv.y, fma(d0, z1.y, -d1 * z0.y)));
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const double2 Xi = X[i];
          const double2 T = make_double2(fma(ca, V[i].x, fma(iR, V[i].y, Xi.x)), fma(ca, V[i].y, fma(-iR, V[i].x, Xi.y)));
          cfma(h ? H[i] : E[i], make_double2(gx_, gy_), T);
        }
      }
    }
  }
  // sums over the threads of a field point
  double2* red = cur;                                  // [3][NF_T] at a time
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    __syncthreads();
    for (int i = 0; i < 3; ++i) red[i * NF_T + tid] = h ? H[i] : E[i];
    __syncthreads();
    for (int w = NF_T / 2; w >= tp; w >>= 1) {
      if (tid < w)
        for (int i = 0; i < 3; ++i) {
          red[i * NF_T + tid].x += red[i * NF_T + tid + w].x;
          red[i * NF_T + tid].y += red[i * NF_T + tid + w].y;
        }
      __syncthreads();
    }
    if (tid < tp && ip < npt)
      for (int i = 0; i < 3; ++i) {
        const double2 v = red[i * NF_T + tid];
        double* o = EH + (((size_t)ip * 6 + 3 * h + i) * R + r) * 2;
        atomicAdd(o, h ? -kw * v.x : -kw * zeta * v.y);
        atomicAdd(o + 1, h ? -kw * v.y : kw * zeta * v.x);
      }
  }
}

int launch_near_field(Ctx* c, int R, const double2* x, int npt, const double* d_pts, double2* EH,
                      cudaStream_t st) {
  SMR_CUDA(c, cudaMemsetAsync(EH, 0, (size_t)npt * 6 * R * sizeof(double2), st));
  // up to 128 field points a CTA: a unit's currents are computed once for them
  int tp = 8;
  while (tp < 128 && tp < npt) tp *= 2;
  const long long groups = ((long long)npt + tp - 1) / tp * R;
  const long long units = (long long)c->p * ((c->Q + NF_Q - 1) / NF_Q);
  // two CTAs an SM stay resident and share a few groups' units evenly; with many
  // groups, four times as many are left to the scheduler
  const int gx = (int)std::min<long long>(units, groups < 4 ? 304 / groups : (1216 + groups - 1) / groups);
  // R^2 in the single-precision seed's range and phases below 1e9: bounds on the
  // high word of R^2
  auto hiword = [](double v) {
    unsigned long long b;
    std::memcpy(&b, &v, 8);
    return (unsigned)(b >> 32);
  };
  const double rmax = 1e9 / c->k;
  const unsigned hi0 = hiword(1e-30), hi1 = hiword(std::min(1e30, rmax * rmax));
  k_nearfield<<<(unsigned)(groups * gx), NF_T, 0, st>>>(c->p, c->npsi, c->Q, npt, R, tp, gx, hi0,
                                                        hi1 > hi0 ? hi1 - hi0 : 0u, c->d_sid, c->d_centres,
                                                        c->d_modes, c->d_rq, x, d_pts, c->k, c->zeta, (double*)EH);
  SMR_LAUNCH(c);
  return SMR_OK;
}

}  // namespace smr

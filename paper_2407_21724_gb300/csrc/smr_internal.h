// Internal declarations of libsmr: context, per-level tables, kernel launchers.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <complex>
#include <cstdint>
#include <string>
#include <vector>

#include "../../include/smr.h"

namespace smr {

// Fields of a direction's spectrum.  A particle's radiation has four, the theta
// and phi components of both currents' (B0, B1 electric, B2, B3 magnetic), and the
// receive takes them in two combinations only, v = B0 + B3 / z and u = -B1 + B2 / z
// (Eqs. 24-25).  The product carries the circular ones, W_+- = v +- j u: every step
// between is the same linear map for all fields, the patterns of the aggregation and
// the receive become P_th +- j P_ph, and the two never mix.
constexpr int NF = 2;

typedef std::complex<double> cd;

// ------------------------------------------------------------------ host math
namespace hm {
// n-point Gauss-Legendre rule on [-1,1], nodes descending (theta ascending).
void gauss_legendre(int n, std::vector<double>& x, std::vector<double>& w);
// Real orthonormal Y_lm (m >= 0, kind 0 = cos, 1 = sin) and its surface
// gradient components dY/dtheta, (1/sin theta) dY/dphi.
void real_ylm(int l, int m, int kind, double theta, double phi, double* Y, double* Yt, double* Yp);
// Spherical Bessel j_l, y_l for l = 0..L at real x > 0 (Miller downward for j,
// upward for y).
void sph_bessel(int L, double x, std::vector<double>& j, std::vector<double>& y);
// Riccati psi_l(x) = x j_l, xi_l(x) = x h^(2)_l and derivatives.
void riccati(int l, double x, double* psi, double* dpsi, cd* xi, cd* dxi);
// In-place inverse of an n x n complex row-major matrix (partial pivoting).
bool invert(int n, std::vector<cd>& a);
// Modes of a sphere shell list: (l, m, kind) for the first n modes.
void mode_list(int n, std::vector<int>& l, std::vector<int>& m, std::vector<int>& kind);
}  // namespace hm

// ------------------------------------------------------------------ data
// Static modes of a meshed shape (smr_add_shape_mesh): the mode -> RWG
// matrix of Eq. 20, the kept eigenvalues, the geometry, per triangle and
// mode the affine field psi = alpha r - beta ([nt][n_psi][alpha, beta xyz]),
// and the 3-point samples handed to the solver like a sampled shape.
struct MeshModes {
  int ne = 0, nt = 0, nq = 0;
  std::vector<double> M, gamma;
  std::vector<double> geo_V;
  std::vector<int> geo_T;
  std::vector<double> area, nrm, ab;
  std::vector<double> rq, modes;
};

struct Shape {
  double a;                               // sphere radius, or bounding radius of a sampled shape
  int n_perp, n_par;
  int n_psi() const { return n_perp + n_par; }
  // shape given as data (smr_add_shape_sampled): points and weights [nq][4],
  // mode fields and divergences [n_psi][nq][4], self block [2n][2n]
  bool sampled = false;
  int nq = 0;
  std::vector<double> rq, modes;
  std::vector<cd> Z;
  // meshed shape: the self block is assembled for the scene's media
  bool mesh = false;
  MeshModes mm;
  double lateral = 0;                     // largest distance of a point from the z axis
  // rotated copy of another shape (about the z axis): the shape whose self
  // block it shares (rotation leaves Z_s unchanged), -1 if none
  int rot_base = -1;
  double rot_angle = 0;
};

struct Level {
  int L = 0, K = 0, nth = 0, nph = 0, nbox = 0;
  double box = 0;
  std::vector<double> khat, w;          // [K][3], [K]
  std::vector<int> bi, bj;               // box integer coordinates
  std::vector<double> centre;            // [nbox][3]
  std::vector<int> il_ptr, il_src, il_off;  // interaction list CSR by target box
  std::vector<int> off_dx, off_dy;       // unique offsets (box units)
  std::vector<int> parent, quad;         // to level s+1
  std::vector<int> ch_ptr, ch_idx, ch_quad;  // children at level s-1 (s >= 1)
  // device
  double* d_khat = nullptr;
  double* d_w = nullptr;
  int* d_il_ptr = nullptr;
  int* d_il_pk = nullptr;                // [n_il] source box * 64 + table row (FP64 translation)
  double2* d_T64 = nullptr;              // [noff][K]
  float2* d_T32 = nullptr;
  int* d_parent = nullptr;
  int* d_quad = nullptr;
  int* d_ch4 = nullptr;                  // [nbox][4] child box per quadrant, -1 if absent
  int* d_ch_ptr = nullptr;
  int* d_ch_idx = nullptr;
  int* d_ch_quad = nullptr;
  // interpolation from this level (child) to s+1 (parent) -- stored on the child
  int* d_th_pk = nullptr;                 // [nth_parent][4] source row | reflected << 16
  double* d_th_ws64 = nullptr;            // [nth_parent][4] weights, reflection sign folded in
  float* d_th_ws32 = nullptr;
  int* d_ph_src = nullptr;               // [nph_p][4]
  double* d_ph_w64 = nullptr;
  float* d_ph_w32 = nullptr;
  double2* d_shift64 = nullptr;          // [4][K_p] exp(j k khat_p.(c_c - c_p))
  // marching kernels (k_march.cu), stored on the child level: the shifts of
  // quadrants 0 and 1 per parent direction ([K_p][2]; 3 and 2 are their
  // conjugates); the last virtual child row of every parent row's stencil;
  // the adjoint's entries (parent row | reflected << 16) by first child row
  // with the weights of four child rows
  double2* d_shiftp64 = nullptr;
  float2* d_shiftp32 = nullptr;
  int* d_mi_vlast = nullptr;
  int* d_ma_ptr = nullptr;
  int* d_ma_ent = nullptr;
  std::vector<int> mi_start;             // [nph_p] child column before the first phi tap (unwrapped)
  // phi-transposed taps: ma_pm consecutive parent columns from ma_start[j]
  // (unwrapped) per child column j, weights [nph][ma_pm]
  std::vector<int> ma_start;
  int ma_pm = 0;
  int* d_ma_pst = nullptr;
  double* d_ma_pw64 = nullptr;
  float* d_ma_pw32 = nullptr;
  double* d_ma_w64 = nullptr;
  float* d_ma_w32 = nullptr;
  double* d_wthp64 = nullptr;            // [nth_p] parent theta weights (stored on the child level)
  // dense lattice map of the boxes of this level (translation tiles)
  int map_x0 = 0, map_y0 = 0, map_w = 0, map_h = 0;
  int* d_boxmap = nullptr;               // [map_h][map_w] box index or -1
  int* d_offid = nullptr;                // [7][7] offset (dx+3, dy+3) -> table row or -1
  int ntile_x = 0, ntile_y = 0, ntile_ne = 0;
  int* d_tiles = nullptr;                // non-empty 4x4 translation tiles (ty * ntile_x + tx)
  int* d_tile_tab = nullptr;             // per non-empty 4x4 tile: 64 source and 16 target boxes (k_translate.cu)
  // gather anterpolation into this level (k_anterp1):
  // child theta rows in nit tiles of TI, parent rows [lo, hi) per tile
  // ([2][nit]), GR the widest range, JC the column chunk
  int ant_TI = 0, ant_nit = 0, ant_GR = 0, ant_JC = 0;
  int* d_ant_lo = nullptr;
  // launch variants (smr_set_variant; smr_autotune chooses FP64's), one right-hand
  // side: 0 = built-in rule.  FP64 interpolation into the parent level: 1 / 2
  // the gather kernel with the full / half theta-row tile, 3 the marching kernel.
  int tune_ip = 0;
  // anterpolation into this level (FP64, FP32): 1 / 2 = the gather kernel with half
  // the column chunk / with 256 threads, 4 and 5 the marching kernel
  int tune_an[2] = {0, 0};
  // the transposed taps padded to fixed widths (multiples of 4, zero weights):
  // phi by child column [nph][PM] (parent column, weight x dphi_p / dphi_c),
  // theta by child row [nth][TM] (parent row | refl << 16, sign x weight / w_theta)
  int ant_PM = 0, ant_TM = 0;             // padded transposed taps per child column / row
  int ant_PMx = 0, ant_TMx = 0;           // real maxima
  int* d_ant_pjp = nullptr;
  double* d_ant_pw64 = nullptr;
  int* d_ant_ttp = nullptr;
  double* d_ant_tw64 = nullptr;
  // stencils of more than 8 taps, wider than the marching kernel's compiled
  // ones: the same tables in FP32, the parent's theta weights, the shifts
  bool ant_wide = false;
  float *d_ant_pw32 = nullptr, *d_ant_tw32 = nullptr, *d_wthp32 = nullptr;
  float2* d_shift32 = nullptr;
  // spectra (allocated for the current R and precision)
  void* d_out = nullptr;                 // active spectra (the last product's precision)
  void* d_in = nullptr;
  size_t spec_bytes = 0;
  void* buf_out[2] = {nullptr, nullptr};   // per precision (SMR_PREC_FP64, SMR_PREC_FP32)
  void* buf_in[2] = {nullptr, nullptr};
  size_t buf_bytes[2] = {0, 0};
};

struct NN {
  int F = 448, H = 0, O = 0, nl = 4;
  int dims[5] = {0, 0, 0, 0, 0};
  long long np = 0;                     // parameter count
  float* p32 = nullptr;                 // master parameters (W_l [in][out] then b_l [out], per layer)
  __nv_bfloat16* w16 = nullptr;         // BF16 copies of the weight matrices (same offsets)
  float *m = nullptr, *v = nullptr, *g = nullptr;
  long long step = 0;
  int cap = 0;                          // rows of the activation buffers
  float* act = nullptr;                 // activations and pre-activations
  float* dact = nullptr;
  float* part = nullptr;                // weight gradients per split of the batch's rows
  size_t part_elems = 0;
  double* d_loss = nullptr;
  int* d_slots = nullptr;               // [48][2] neighbour offsets, sorted
};

// one profiled launch: algorithmic bytes / flops and CUDA events around it
struct ProfRec {
  const char* name;
  int level;
  double bytes, flops;
  cudaEvent_t a, b;
};

struct Ctx {
  smr_opts opts;
  std::vector<ProfRec>* prof = nullptr;   // non-null while smr_profile_matvec runs
  std::string err;
  int device = 0;
  std::vector<Shape> shapes;
  bool have_scene = false;
  // scene
  int p = 0, npsi = 0, S = 0, nlev = 0, n_arrays = 1;
  double k = 0, zeta = 1, k_in = 0, zeta_in = 1;
  std::vector<double> centres;          // [p][3]
  std::vector<int> sid;                 // [p]
  std::vector<int> pi, pj;              // lattice indices
  double origin[2] = {0, 0}, z0 = 0;
  std::vector<Level> lev;
  // surface rule (shared by all shapes, scaled by radius)
  int Q = 0;
  std::vector<double> rule_th, rule_ph, rule_w1;  // unit-sphere rule
  double* d_modes = nullptr;            // [S][npsi][Q][4]: psi xyz, div
  double* d_rq = nullptr;               // [S][Q][4]: point xyz, weight
  // patterns [S][npsi][2][K0]
  double2* d_P64 = nullptr;
  // circular patterns P_th +- j P_ph, half of the directions: [S][2][npsi][K0 / 2]
  // and [S][2][K0 / 2][npsi]
  double2 *d_Pd64 = nullptr, *d_Pm64 = nullptr;
  float2 *d_Pd32 = nullptr, *d_Pm32 = nullptr;
  // particles
  int* d_sid = nullptr;
  std::vector<int> arr;                 // [p] array id of each particle
  int* d_arr = nullptr;
  double* d_centres = nullptr;          // [p][3]
  double* d_dshift = nullptr;           // [p][3] r_mu - c_box (finest level)
  int any_dshift = 0;
  // several particles in one finest box: the boxes are the occupied cells,
  // aggregation sums each box's particles and receive reads its box
  int multi = 0;
  std::vector<int> cell_of;              // [p] finest box of each particle
  int* d_cell_of = nullptr;
  int* d_cell_ptr = nullptr;             // [nbox0 + 1] CSR of each box's particles
  int* d_cell_idx = nullptr;             // [p]
  void* pspec[2] = {nullptr, nullptr};   // per-particle level-0 spectra (FP64, FP32)
  // near SpMV: CSR by particle, block ids; blocks stored transposed [nb][2n][2n]
  std::vector<int> nr_ptr, nr_col, nr_blk;
  int* d_nr_ptr = nullptr;
  int* d_nr_col = nullptr;
  int* d_nr_blk = nullptr;
  int nblk = 0;
  std::vector<int> blk_sm, blk_sn, blk_dx, blk_dy;  // key of each block
  std::vector<double> blk_off;            // [nblk][3] r_mu - r_nu of each block
  // self blocks [S][2 npsi (col)][2 npsi (row)], and the circular halves of the exterior
  // ones [nblk - S][npsi (col)][+, -][npsi (row)] (k_near_rows)
  double2 *d_Bs64 = nullptr, *d_Bc64 = nullptr;
  float2 *d_Bs32 = nullptr, *d_Bc32 = nullptr;
  // preconditioner: inverse self blocks, transposed [S][2n][2n]
  bool pinv_ok = true;                  // every self block was invertible
  double2* d_Pinv64 = nullptr;
  float2* d_Pinv32 = nullptr;
  int* d_pc_ptr = nullptr;              // identity CSR for the block kernel
  int* d_pc_col = nullptr;
  int* d_pc_blk = nullptr;
  int* d_perm = nullptr;                // particles sorted by shape
  NN nn;
  // captured products: (x, y, R, precision) -> executable graph
  struct GraphEntry {
    const void* x;
    void* y;
    int R, prec;
    cudaGraphExec_t exec;
  };
  std::vector<GraphEntry> graphs;
  cudaStream_t capture_stream = nullptr;
  // work buffers
  int buf_R[2] = {0, 0};
  int spec_R = 0, spec_prec = -1;
  double2* d_xs[2] = {nullptr, nullptr}; // per precision: the coefficients the spectra belong to
  bool keep_x = false;                   // a product that leaves d_xs alone
  double2* d_tmp = nullptr;             // [N][R] scratch for split products
  size_t tmp_elems = 0;
  // solver scratch
  void* d_sol = nullptr;
  size_t sol_bytes = 0;
  double* d_red = nullptr;              // reduction partials
  size_t red_bytes = 0;
  double* h_red = nullptr;              // pinned host mirror
  // tensor-core receive and aggregation (FP32 product, one right-hand side)
  bool tc_enable = true, tc_ready = false;
  int tc_nK = 0, tc_ntile = 0;
  int tc_nsplit = 1;                      // splits of the receive's K chunks
  float* d_tc_part = nullptr;             // [tc_nsplit][p][4 n_psi] partial rows (null for one split)
  size_t tc_part_bytes = 0;
  float* d_tc_rec = nullptr;              // [S][nK][hi | lo][128][32] swizzled coefficient images
  int* d_tc_perm = nullptr;
  int* d_tc_shape = nullptr;
  int* d_tc_start = nullptr;
  int* d_tc_count = nullptr;
  int* d_tc_err = nullptr;                // set when a pipeline wait runs out
  uint32_t tc_spin = 1u << 24;            // polling limit of the pipeline waits (smr_set_wait_limit)
  bool tc_agg_ready = false;
  int tc_nMT = 0, tc_nKc = 0;
  int tc_nmsplit = 1;                     // CTAs along a tile's M tiles
  float* d_tc_agg = nullptr;              // [S][M tiles][K chunks][hi | lo][128][32] aggregation images
  // tensor cores for aggregation / receive chosen by smr_autotune (-1: not tuned)
  int tune_tc_agg = -1, tune_tc_rec = -1, tune_tc_near = -1;
  // near product on the tensor cores: block images, and per lattice offset
  // (phase; self blocks first) tiles of up to 128 pairs sharing a block
  bool tcn_ready = false;
  int tcn_nK = 0;
  std::vector<int> tcn_phase;             // [n phases + 1] tile ranges
  std::vector<double> tcn_bytes, tcn_flops;   // algorithmic bytes and flops per phase
  float* d_tcn_img = nullptr;             // [nblk][nK][hi | lo][128][32] swizzled block images
  int* d_tcn_blk = nullptr;               // per tile: block
  int* d_tcn_start = nullptr;
  int* d_tcn_count = nullptr;
  int* d_tcn_nu = nullptr;                // per pair: source particle (x row)
  int* d_tcn_mu = nullptr;                // per pair: partial row, phase * p + target particle
  unsigned short* d_tcn_mask = nullptr;   // per particle: phases in which it has a pair
  float* d_tcn_part = nullptr;            // [phase][p][4 n_psi] FP32 partial products
  float2* d_x32 = nullptr;                // x in FP32 for the gathers
  const double2* x32_of = nullptr;        // which x d_x32 holds (set by prep_x32)
  // column buffers of split products ([R][N] in, [R][N] out)
  bool split_cols = true;
  double2* d_split = nullptr;
  size_t split_elems = 0;
  size_t tcn_part_bytes = 0;
  // Column lanes of split products: the columns are dealt round-robin to
  // n_lanes lanes, each with its own FP32 work buffers and stream, so that
  // the small upper-level launches of several columns overlap.  Lane 0 is
  // the context's own buffers and the caller's stream (copied, not owned);
  // lanes 1.. own theirs.
  struct Lane {
    std::vector<void*> out, in;           // per level FP32 spectra
    float2* x32 = nullptr;
    float* tcn_part = nullptr;
    float* tc_part = nullptr;
    cudaStream_t s = nullptr;
    cudaEvent_t ev = nullptr;             // end of the lane's columns
  };
  std::vector<Lane> lanes;
  // Overlapped product (smr_set_overlap): per lane a side stream for the
  // translations, one for the near product, and the events that order them
  struct Side {
    cudaStream_t tr = nullptr, nr = nullptr;
    cudaEvent_t ex = nullptr, enear = nullptr, efork = nullptr;
    std::vector<cudaEvent_t> eout, etr;   // per level: outgoing spectra ready, translation done
  };
  std::vector<Side> side;
  bool overlap = true;
  int cur_side = 0;                       // the side set far_impl uses
  cudaEvent_t near_ev = nullptr;          // the receive waits for it when set
  int n_lanes = 4;                        // columns in flight (smr_set_column_lanes, smr_autotune)
  cudaEvent_t lane_fork = nullptr;
  // cluster block-Jacobi preconditioner (k_cluster.cu): members [ncl][4]
  // (-1 for an absent one), inverses [ncl][4m][4m] transposed, m = 2 n_psi
  bool cl_ready = false;
  int ncl = 0;
  int* d_cl_mem = nullptr;
  double2* d_cl_inv64 = nullptr;
  float2* d_cl_inv32 = nullptr;
  // polynomial preconditioner (smr_solve_opts.poly_degree): roots in Leja
  // order for the running solve, four [N] work vectors, products it made
  std::vector<std::complex<double>> poly_roots;
  bool poly_busy = false;
  int poly_mv = 0;
  double2* d_polyw = nullptr;
  size_t polyw_elems = 0;
  // near-field sweeps preconditioner: three [N][R] work vectors, sweep count
  double2* d_pcw = nullptr;
  size_t pcw_elems = 0;
  int pc_sweeps = 1;
  // learned local-coupling preconditioner: diagonal D [N] (one right-hand side)
  double2* d_lpc = nullptr;
  bool lpc_ready = false;
};

// ------------------------------------------------------------------ helpers
#define SMR_CUDA(ctx, call)                                                        \
  do {                                                                             \
    cudaError_t e_ = (call);                                                       \
    if (e_ != cudaSuccess) {                                                       \
      (ctx)->err = std::string(#call) + ": " + cudaGetErrorString(e_);             \
      return SMR_E_CUDA;                                                           \
    }                                                                              \
  } while (0)

#define SMR_LAUNCH(ctx)                                                            \
  do {                                                                             \
    cudaError_t e_ = cudaGetLastError();                                           \
    if (e_ != cudaSuccess) {                                                       \
      (ctx)->err = std::string("kernel launch: ") + cudaGetErrorString(e_);        \
      return SMR_E_CUDA;                                                           \
    }                                                                              \
  } while (0)

template <typename T>
int upload(Ctx* c, T** dst, const std::vector<T>& src) {
  if (*dst) cudaFree(*dst);
  *dst = nullptr;
  if (src.empty()) return SMR_OK;
  SMR_CUDA(c, cudaMalloc((void**)dst, src.size() * sizeof(T)));
  SMR_CUDA(c, cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice));
  return SMR_OK;
}

inline void pbeg(Ctx* c, cudaStream_t st, const char* name, int level, double bytes, double flops) {
  if (!c->prof) return;
  ProfRec r{name, level, bytes, flops, nullptr, nullptr};
  cudaEventCreate(&r.a);
  cudaEventCreate(&r.b);
  cudaEventRecord(r.a, st);
  c->prof->push_back(r);
}
inline void pend(Ctx* c, cudaStream_t st) {
  if (c->prof) cudaEventRecord(c->prof->back().b, st);
}

// ------------------------------------------------------------------ setup (k_setup.cu)
int build_modes(Ctx* c);          // d_modes, d_rq (host evaluation, upload)
int build_patterns(Ctx* c);       // d_P64, d_Pd* and d_Pm* on the GPU (FP64)
int build_translations(Ctx* c);   // per level d_T64 / d_T32 on the GPU (FP64)
int build_near(Ctx* c);           // d_Bs*, d_Bc* on the GPU (FP64) + self blocks
// Entry (row i, column j) of near block b from its stored form: an exterior block
// is [z T, K; -K, T / z], stored as T -+ j K
__host__ __device__ inline double2 near_entry(const double2* self, const double2* circ, int S, int n, double z, int b,
                                              int i, int j) {
  const int n2 = 2 * n;
  if (b < S) return self[((size_t)b * n2 + j) * n2 + i];
  const double2* q = circ + ((size_t)(b - S) * n + j % n) * n2 + i % n;
  const double2 p = q[0], m = q[n];
  if (i / n == j / n) {
    const double f = i < n ? 0.5 * z : 0.5 / z;
    return make_double2(f * (p.x + m.x), f * (p.y + m.y));
  }
  const double f = i < n ? 0.5 : -0.5;             // K = j (B+ - B-) / 2
  return make_double2(-f * (p.y - m.y), f * (p.x - m.x));
}
int launch_rhs(Ctx* c, int R, const double* d_khat, const double2* d_pol, double2* b,
               cudaStream_t st);
// R = 1 right-hand side with incidence number arr[mu] for particle mu
// (host khat/pol hold one plane wave per array)
int launch_rhs_arrays(Ctx* c, const double* d_khat, const double2* d_pol, double2* b, cudaStream_t st);
int launch_rhs_scratch(Ctx* c, int R, const double* d_khat, const double2* d_pol, double2* Sv,
                       double2* b, cudaStream_t st);

int copy_fields(Ctx* c, int level, int kind, double* out);   // k_mlfma.cu

// ------------------------------------------------------------------ fields (k_fields.cu)
int launch_far_field(Ctx* c, int R, const double2* x, int nd, const double* d_dirs,
                     double2* F, cudaStream_t st);
int launch_cross_sections(Ctx* c, int R, const double2* x, int n_sca, const double* d_dirs,
                          const double* d_w, const double2* d_pol, double* d_cs, cudaStream_t st);
int launch_near_field(Ctx* c, int R, const double2* x, int npt, const double* d_pts,
                      double2* EH, cudaStream_t st);

// ------------------------------------------------------------------ learned initial guess (k_learned.cu)
int nn_init(Ctx* c, int width, unsigned long long seed);
void nn_free(Ctx* c);
int nn_features(Ctx* c, const double* d_khat, const double* d_pol, float* feat, cudaStream_t st);
int nn_targets(Ctx* c, const double* d_khat, const double2* x, double scale, float* tgt, cudaStream_t st);
int nn_forward_backward(Ctx* c, int n, const float* feat, const int* idx, const float* tgt, bool backward,
                        double* loss_host, cudaStream_t st);
int nn_adam(Ctx* c, float lr, cudaStream_t st);
int nn_predict(Ctx* c, const double* d_khat, const double* d_pol, double scale, double2* x0, cudaStream_t st);
int nn_precond(Ctx* c, const double* d_khat, const double* d_pol, double scale, const double2* b, cudaStream_t st);
int lpc_apply(Ctx* c, double2* z, cudaStream_t st);

// ------------------------------------------------------------------ hot path (k_mlfma.cu)
int ensure_spectra(Ctx* c, int R, int prec);
int run_near(Ctx* c, int R, int prec, const double2* x, double2* y, cudaStream_t st);
int run_far(Ctx* c, int R, int prec, const double2* x, double2* y, bool accumulate,
            cudaStream_t st);
int run_precond(Ctx* c, int R, int prec, const double2* r, double2* z, cudaStream_t st);
// y = Z x through a CUDA graph captured on first use for (x, y, R, prec)
int run_matvec_graph(Ctx* c, int R, int prec, const double2* x, double2* y, cudaStream_t st);
// y = Z x (near + far); FP32 with R > 1 runs column by column (split products)
int run_product(Ctx* c, int R, int prec, const double2* x, double2* y, cudaStream_t st);
void free_graphs(Ctx* c);
// meshed shapes (mesh.cu)
int mesh_static_modes(Ctx* c, int nv, const double* verts, int nt, const int* tris, int n_perp, int n_par,
                      MeshModes& out);
int mesh_self_block(Ctx* c, const Shape& sh, std::vector<cd>& Z);
// cluster block-Jacobi preconditioner (k_cluster.cu)
bool cluster_ok(const Ctx* c);
int build_clusters(Ctx* c);
int run_cluster(Ctx* c, int R, int prec, const double2* r, double2* z, cudaStream_t st);
void free_clusters(Ctx* c);
// column lanes of split FP32 products (buffers allocated outside graph capture)
int ensure_lanes(Ctx* c, int nl);
void free_lanes(Ctx* c);
int ensure_side(Ctx* c, int n);
void free_side(Ctx* c);
// tensor-core receive and aggregation (k_tc.cu)
int build_tc(Ctx* c);
bool tc_receive_ok(const Ctx* c, int R);
int run_receive_tc(Ctx* c, const float2* in0, double2* y, bool accumulate, cudaEvent_t ready, cudaStream_t st);
bool tc_aggregate_ok(const Ctx* c, int R);
int build_near_tc(Ctx* c);
bool tc_near_ok(const Ctx* c, int R);
int run_near_tc(Ctx* c, double2* y, cudaStream_t st);
int prep_x32(Ctx* c, int R, int prec, const double2* x, cudaStream_t st);
int run_aggregate_tc(Ctx* c, const double2* x, const float2* x32, float2* out0, cudaStream_t st);
int tc_check(Ctx* c);
// FP32 translation of one right-hand side (k_translate.cu)
int build_translate_tiles(Ctx* c, Level& L, const std::vector<int>& tiles, const std::vector<int>& boxmap);
int run_translate_tiles(Ctx* c, int s, cudaStream_t st);
// interpolation s -> s + 1 and anterpolation s + 1 -> s (k_march.cu)
int run_interp(Ctx* c, int s, int R, int prec, cudaStream_t st);
int run_anterp(Ctx* c, int s, int R, int prec, cudaStream_t st);

// ------------------------------------------------------------------ linear algebra (k_linalg.cu)
// h[j*R + r] = sum_i conj(V_j[i][r]) w[i][r] for j < J (V_j = V + j*ldv), FP64.
int multidot(Ctx* c, int J, long long n, int R, const double2* V, long long ldv,
             const double2* w, double2* h_host, cudaStream_t st);
// w[i][r] -= sum_j V_j[i][r] h[j][r]   (h on the device, [J][R])
int multi_axpy(Ctx* c, int J, long long n, int R, const double2* V, long long ldv,
               const double2* d_h, double2* w, double sign, cudaStream_t st);
// norms[r] = ||v[:, r]||_2
int col_norms(Ctx* c, long long n, int R, const double2* v, double* norms_host, cudaStream_t st);
// y[i][r] = a[r] * x[i][r] + b[r] * y[i][r]  (a, b complex per column, device)
int col_axpby(long long n, int R, const double2* d_a, const double2* x, const double2* d_b,
              double2* y, cudaStream_t st);

int solve(Ctx* c, int R, const double2* b, double2* x, const smr_solve_opts* o,
          smr_solve_stats* stats, cudaStream_t st);

}  // namespace smr

// The C ABI wrapper around a context (defined in api.cu).
struct smr_ctx {
  smr::Ctx c;
};

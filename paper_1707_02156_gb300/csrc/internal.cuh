// Internal declarations shared by the CUDA translation units of the library.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "../../include/bie.h"

namespace bie {

void set_error(const std::string& msg);
void count_launch(int n = 1);  // kernel launches issued by the library (all threads)
int ctx_device(const bie_ctx* ctx);  // CUDA device ordinal of a context

#define BIE_CUDA_TRY(expr)                                                                     \
  do {                                                                                         \
    cudaError_t e_ = (expr);                                                                   \
    if (e_ != cudaSuccess) {                                                                   \
      ::bie::set_error(std::string(#expr) + ": " + cudaGetErrorString(e_));                    \
      return BIE_ECUDA;                                                                        \
    }                                                                                          \
  } while (0)

#define BIE_TRY(expr)              \
  do {                             \
    int s_ = (expr);               \
    if (s_ != BIE_OK) return s_;   \
  } while (0)

// Dynamic shared memory of a launch above the default 48 KB.  The attribute belongs to the kernel on its device and all
// threads of the process share it, so every launch sets the same value: with a value per launch, a thread
// with a smaller degree could lower it between another thread's setting and its launch, which then failed.
constexpr size_t kMaxSmem = 226 * 1024;  // a block's 227 KB less a kernel's own arrays
template <typename K>
cudaError_t allow_smem(K kern, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
}

__host__ __device__ inline long long leg_row(int p, int m, int n, int nj) {
  long long before = (long long)m * (p + 1) - (long long)m * (m - 1) / 2;
  return (before + (n - m)) * nj;
}

// ---- transforms (transforms.cu) ----
// Weighted source densities, fields [drop][3]: w_s f_c(s) on the degree-P grid to out[c * ld + off[drop] + s],
// the weights in row 6 of the records rec ([7][N] at 7 off[drop]).
struct SynthSources {
  const double* rec;
  const long long* off;
  long long ld;
};
// A synthesis of nfield fields of degree p on the grid of degree P: the s-th kind asked for of field f goes to
// out + s * kind_stride + f * field_stride (or to the sources' place).  Coefficients of field f start at
// field_off ? field_off[f] : f * coef_stride.  T1, T2 may be null when no kind needs them.
template <typename R>
struct SynGroup {
  long long nfield;
  const long long* field_off;
  long long coef_stride;
  int p, P;
  const R *T0, *T1, *T2, *cs;
  R* out;
  long long kind_stride, field_stride;
  SynthSources src;
  long long begin;  // first block and latitude pairs per block: set by the launcher
  int jb;
};
constexpr int kMaxSynGroups = 8;
template <typename R>
struct SynGroups {
  int n;
  SynGroup<R> g[kMaxSynGroups];
};
// Several of them in one launch, with the derivative kinds of the mask `kinds` (bit 0 f, 1 t, 2 p, 3 tt, 4 tp,
// 5 pp; the masks 1, 6, 7, 62, 63).
int launch_synth(int kinds, const double* coef, std::vector<SynGroup<double>> groups, int sms, cudaStream_t s);
template <typename R>
int launch_synth_sources(const double* coef, std::vector<SynGroup<R>> groups, int sms, cudaStream_t s);
inline int launch_synth(int kinds, const double* coef, const long long* field_off, long long coef_stride,
                        long long nfield, int p, int P, const double* T0, const double* T1, const double* T2,
                        const double* cs, double* out, long long kind_stride, long long field_stride, int sms,
                        cudaStream_t s) {
  return launch_synth(kinds, coef, {{nfield, field_off, coef_stride, p, P, T0, T1, T2, cs, out, kind_stride, field_stride, {}, 0, 0}},
                      sms, s);
}
// analysis: grids (degree P) -> coefficients (degree p <= P), FP64, for several degree groups in one launch.
// Offsets per field, or null and a stride; begin is set by the launcher.
struct AnaGroup {
  long long begin, nfield;
  const long long* grid_off;
  const long long* coef_off;
  long long grid_base, grid_stride, coef_base, coef_stride;  // grid f at base + (off[f] or f stride)
  const double* cs;
  const double* At;  // weighted Legendre table, rows (m, j) with the degree n = m..p fastest
  int P, p;
};
constexpr int kMaxAnaGroups = 8;
struct AnaGroups {
  int n, cl, orders;  // groups; blocks per field, or (orders) one block per field and order
  AnaGroup g[kMaxAnaGroups];
};
// early: the launch need not wait until the kernel before it on the stream has been flushed (that one must be a
// kernel launched in full stream order).
int launch_analyze(std::vector<AnaGroup> groups, const double* grid, double* coef, int sms, cudaStream_t s,
                   bool early = false);
// rotation (App. B): out[ld][a*nb+b][c] = blocks(a) applied to e^{i m alpha_b} coef[ld][c]
template <typename CT, typename R>
int launch_rotate(const CT* coef, const long long* field_off, int ncomp, long long ndrop, int p, const R* blocks,
                  long long blk_stride, int na, int nb, const R* ph, R* out, long long out_drop_stride,
                  cudaStream_t s);
// multiply coefficients by e^{i m gamma} (in place), ncomp fields per drop
int launch_phase(double* coef, long long nfield, int p, double gamma, cudaStream_t s);

// ---- pair sums and geometry (pairs.cu) ----
// Surface quantities from x, x_theta, x_phi grids [f=drop*3+c][j][k]: writes SoA source records
// [7][N] = (x, n, wgt*J) of drop d at rec + 7 * off[d], with wgt the regular weight (pi/(P+1)) w_j,
// J = W/sin(theta_j).
int launch_surface(const double* X, const double* Xt, const double* Xp, long long ndrop, int P,
                   const double* wsin /*[j] = w_j pi/(P+1)/sin theta_j*/, double* rec, const long long* off,
                   cudaStream_t s);
// Rotated-grid cache for nt targets, from target tl0 on, of each of ndrop drops (ng targets): cache[t][7][nq] = (x0 - x', w n', w), w =
// w^s_j W'/sin theta_j, on the degree-pq grid; x0 of drop ld's targets read from the standard-grid
// records at rec_std + rec_off[ld] ([7][ng] per drop; the drops need not be adjacent there).
template <typename R>
int launch_rotgeo(const double* X, const double* Xt, const double* Xp, long long ndrop, int nt, int tl0, int ng, int pq,
                  const double* rec_std, const long long* rec_off, const double* wsq, R* cache, cudaStream_t s);
// The same cache from the shape coefficients in one kernel (rotgeo.cu), for the degrees whose block fits shared
// memory.  Fixed-point tables (fixed.cuh) of the degree-pq grid: LT0, LT1[j][diag(n - m) + m] = P~_n^m(t_j) 2^56
// and its theta derivative times 2^(56 - t1[n]) for the latitudes j <= pq/2, diag(d) the entries with a
// smaller n - m; CM, CP[m][k] = cos, sin (m phi_k) times 2^56 and times m 2^(55 - floor(log2 m)) for the
// longitudes k <= (pq+1)/2; wblk the Wigner blocks times 2^56.
struct RotGeo {
  int p, pq, nt, tl0;        // nt targets, from tl0 on, of each drop
  const double* coef;
  const long long* foff3;    // [drop][3]
  const double* ph;          // phases of the degree-p grid
  const int2* wblk;
  long long wstride;
  const int2 *LT0, *LT1;
  const int* t1;
  const int4 *CM, *CP;
  const double* rec_std;
  const long long* rec_off;
  const double* wsq;
};
bool rotgeo_fix_fits(int p, int pq);
int launch_rotgeo_fix(const RotGeo& A, long long ndrop, double* cache, cudaStream_t s);
// Singular self interaction (Thm 1, Sec. 2.2), one block per target of ndrop drops of degree p:
// direct form against the rotated-geometry cache.
template <typename R>
int launch_self_direct(int kind, const double* dens, const long long* foff3, long long ndrop, int p, int pq,
                       const R* wblk, long long wstride, const R* ph, const R* T0, const R* cs, const R* cache,
                       const double* wts, const long long* val_off, double* vals, size_t smem_budget,
                       cudaStream_t s);
// Projected kernel factors Q[t][12][tri(n,m)] of ntarget targets (see self.cu), from the FP64
// rotated-geometry cache, with fixed-point tables (fixed.cuh): CT[k][m] = cos, sin (m phi_k) 2^55 for the
// longitudes k <= (pq+1)/2, PT[j][tri(n, m)] = P~_n^m(t_j) 2^55 for the latitudes j <= pq/2.
// The stresslet (kind 1) first: it leaves its factors in the cache's row 3, the Stokeslet its own in rows 3 and 6.
// self_dense_fits: whether the dense form serves the degrees.
bool self_dense_fits(int p, int pq);
int launch_kernel_proj(int kind, double* cache, long long ntarget, int p, int pq, const int4* CT, const int2* PT,
                       double* Q64, cudaStream_t s);
// Entries per plane of the dense self form: (p+1)^2 rounded up to whole 16-byte loads in every precision.
__host__ __device__ inline int self_row(int p) { return ((p + 1) * (p + 1) + 3) & ~3; }
// Dense factors S[target][6][self_row(p)] of the latitude rows row0 .. row0 + nrow - 1 (row = drop * (p+1) + a)
// from their projected factors Q (Q64 starts at row0), written at the rows' places in S64 and S32; wblk: the
// Wigner blocks times 2^56 in fixed point.
int launch_unrotate(const double* Q64, long long row0, long long nrow, int p, const int2* wblk, long long wstride,
                    const double* ph, double* S64, float* S32, cudaStream_t s);
// One degree group of the dense-form apply (device pointers; begin is set by the launcher).
template <typename R>
struct SelfGroup {
  long long begin;          // first block of the group
  long long ndrop;          // drops of the group
  const long long* foff3;   // [drop][3] offsets of the density coefficients
  const R* S;               // dense factors
  const double* wts;        // per-drop weight
  const long long* val_off; // per-drop offset into vals
  int p;
};
constexpr int kMaxSelfGroups = 8;
template <typename R>
struct SelfGroups {
  int n;
  SelfGroup<R> g[kMaxSelfGroups];
};
// out[i] = double-float split of in[i] (dff: dfloat.cuh)
struct dff;
int launch_split_dff(const double* in, dff* out, long long n, cudaStream_t s);
// All dense-form groups in one launch (eight groups per launch at most).
template <typename R, typename CT>
int launch_self_dense(std::vector<SelfGroup<R>> groups, const CT* dens, double* vals, int sms, cudaStream_t s);
// interfacial force at the N grid points of nd drops from x derivatives [5][nd][3][N] (t, p, tt, tp, pp) and
// Gamma and its derivatives [3][nd][N] (f, t, p): f [nd][3][N]
int launch_force(const double* X, const double* Gm, long long nd, long long N, double es, double xs, double* f,
                 cudaStream_t s);
// out[i] = (float) in[i]
int launch_to_float(const double* in, float* out, long long n, cudaStream_t s);

// ---- surfactant transport (surfactant.cu) ----
// f_E and (fi non-null) inv_pe * lap Gamma at the N grid points of nd drops: X [6][nd*3][N] (x and
// its derivatives f, t, p, tt, tp, pp), U [3][nd*3][N] (u: f, t, p), Gm [6][nd][N]; fe, fi [nd][N]
int launch_surf_rates(const double* X, const double* U, const double* Gm, long long nd, long long N, double inv_pe,
                      double* fe, double* fi, cudaStream_t s);
// coefficients of the surface Laplacian L[5][nd][N] (s_tt, s_tp, s_pp, s_t, s_p) from X [6][nd*3][N]
int launch_lap_coef(const double* X, long long nd, long long N, double* L, long long ld, cudaStream_t s);
// out[nd][N] = lap s from L and the fields S [6][nd][N] of s (kinds t..pp used)
int launch_lap_apply(const double* L, const double* S, long long nd, long long N, double* out, cudaStream_t s);
// per-drop integral on the grid of degree P (mode 0: volume from X kinds f, t, p; mode 1: mass of
// Gm [nd][N] from X kinds t, p), wsin[j] = (pi/(P+1)) w_j / sin(theta_j); out[nd] on the device
int launch_drop_integral(const double* X, const double* Gm, long long nd, int P, const double* wsin, int mode,
                         double* out, cudaStream_t s);
// out[d] = max |F| over the nper fields of drop d, F [nd*nper][N]
int launch_drop_absmax(const double* F, long long nd, int nper, long long N, double* out, cudaStream_t s);
// w = (y - a c) * inv_diag
int launch_implicit_combine(const double* y, const double* c, double a, const double* inv_diag, long long n,
                            double* w, cudaStream_t s);
// y = x * sc (elementwise)
int launch_mul(const double* x, const double* sc, long long n, double* y, cudaStream_t s);

// ---- angle reparametrisation (reparam.cu) ----
// zero-padded copies [d][c][(P+1)^2] of degree-p coefficients at src + off[d] + c (p+1)^2
int launch_pad_coef(const double* src, const long long* off, int p, int P, long long nd, int ncomp, double* dst,
                    cudaStream_t s);
// values (and, with derivs, theta and phi derivatives) of nf (1 or 3) expansions of degree P per drop at the
// N points (th, ph)[d][N]: out[d][f][kind][N]; ab = recursion coefficients (a, b) per (m, n), rows of order m
int launch_eval_points(const double* coef, int nf, int P, long long nd, long long N, const double* th,
                       const double* ph, const double* ab, int derivs, double* out, cudaStream_t s);
// norms[d][n][2] = (sum_m |x_n^m|, sum_m |x_n^m|^2), m = -n..n, of [d][3][(P+1)^2]
int launch_mode_norms(const double* coef, int P, long long nd, double* norms, cudaStream_t s);
// out = scale * a[d][n] * in, per drop and degree
int launch_scale_degrees(const double* in, const double* a, int P, long long nd, int ncomp, double scale, double* out,
                         cudaStream_t s);
// g = tangential part of gradE at the points (E = x0 and its derivatives there), gmax[d] = max |g|
int launch_rep_gradient(const double* E, const double* gradE, long long N, long long nd, double* g, double* gmax,
                        cudaStream_t s);
// forward Euler step of the angles of the active drops with the pseudo-velocity -g
int launch_rep_step(const double* E, const double* g, long long N, long long nd, const int* active, double dtau,
                    double* th, double* ph, cudaStream_t s);
// the degree-P grid's parameter points for nd drops, from the Gauss nodes t_j
int launch_grid_points(const double* nodes, int P, long long nd, double* th, double* ph, cudaStream_t s);

}  // namespace bie

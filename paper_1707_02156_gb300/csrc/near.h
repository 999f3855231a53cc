// Near-singular (Omega_2) step of Sec. 2.3: records and launchers.
#pragma once
#include <cuda_runtime.h>

namespace bie {

// One (target, source drop) pair of the nearest region, with its closest point.
struct NearPair {
  long long target;  // global target index
  int src_drop;
  int pad;
  double d0;         // |x0 - x*|
  double theta_v;    // parameters of x* in the source drop's own parametrisation
  double phi_v;
};

int launch_near_seed(const NearPair* pairs, int npair, const double* rec_std, const long long* toff, const int* ngd,
                     const long long* tgt_loc, const int* tdrop, int* seed, cudaStream_t s);
// shape coefficients of each pair's source drop with the phases e^{i m alpha} of its seed longitude alpha =
// pi lon[pair] / (p+1) applied, to out + dst_off[pair] as [3][(p+1)^2]
int launch_near_phase_shift(const NearPair* pairs, int npair, const double* coef, const long long* coef_off,
                            const int* pdeg, const int* lon, const long long* dst_off, double* out,
                            cudaStream_t s);
// the Legendre recursion's coefficients for degrees up to P (near_rec_table_doubles(P) doubles), which
// the closest-point Newton iteration reads
int near_rec_table_doubles(int P);
int launch_near_rec_table(int P, double* tab, cudaStream_t s);
int launch_near_newton(const NearPair* pairs, int npair, const double* xr, const int* pdeg, const long long* xr_off,
                       const double* x0, const double* tab, int tabP, double* result, cudaStream_t s);
// d0 and the own-frame parameters of x* into the pairs, and the check points [pair][L][3], from the Newton results
int launch_near_checkpoints(NearPair* pairs, int npair, int L, const double* res, const double* x0, const int* lon,
                            const double* beta, const int* pdeg, const double* hdrop, double* pts, cudaStream_t s);
int launch_near_checkgrid(const NearPair* pairs, int npair, int L, const double* pts, const double* centre,
                          const double* bound, const double* h, double a_tilde, const double* rec_up,
                          const long long* up_off, const long long* up_n, int* grid, cudaStream_t s);
template <typename R>
int launch_near_checks(int kind, const NearPair* pairs, int npair, int L, const double* pts, const int* grid,
                       const double* centre, const long long* toff, const int* ngd, const long long* up_off,
                       const long long* up_n, const R* Xs, const R* Ns, const R* Qs, long long nstd, const R* Xu,
                       const R* Nu, const R* Qu, long long nup, const double* wts, double* cv, cudaStream_t s);
// Sources of one grid, [3][ld] each: positions relative to the drop centres, normals, weighted densities of the
// single (F) and the double layer (U).
struct NearSources {
  const double *X, *N, *F, *U;
  long long ld;
};
// cv[pair][l] = wS S[f] + wD D[u] of the pair's source drop at its check points
int launch_near_checks_both(const NearPair* pairs, int npair, int L, const double* pts, const int* grid,
                            const double* centre, const long long* toff, const int* ngd, const long long* up_off,
                            const long long* up_n, const NearSources& std_, const NearSources& up, const double* wS,
                            const double* wD, double* cv, cudaStream_t s);
int launch_near_interp(const NearPair* pairs, const int* tbeg, int ntgt, int L, int kind, const double* selfcoef,
                       const double* dens, const long long* coef_off, const int* pdeg, const double* hdrop,
                       const double* wts, const double* cv, const int* tdrop, const long long* tgt_loc,
                       const long long* val_off, const int* ngd, double* vals, cudaStream_t s);

// One grid (standard or upsampled) of the drops of one degree p, as the rows read it.
struct NearRowsSrc {
  int P;
  const double* T0;  // Legendre table of (p, P)
  const double* cs;  // its phases
  const double* X;   // sources relative to their drop's centre, normals: [3][ld]
  const double* N;
  long long ld;
  const double* rec;     // records, weights in row 6
  const long long* off;  // first source, by drop
};
// The near-singular rule of the n pairs list[] (source drops of degree p) as rows of the operator (near.cu):
// 7 planes of self_row(p) doubles at rows + row_off[pair].  near_rows_smem: the block's shared memory, with P
// the larger of the two grids' degrees.
size_t near_rows_smem(int p, int P);
int launch_near_rows(int kind, const NearPair* pairs, const int* list, int n, int p, int L, const double* pts,
                     const int* grid, const double* centre, const double* hdrop, const NearRowsSrc& std_,
                     const NearRowsSrc& up, const long long* row_off, double* rows, cudaStream_t s);
// vals += the near values of the ntgt targets from their pairs' rows
int launch_near_rows_apply(const NearPair* pairs, const int* tbeg, int ntgt, const double* rows, const long long* row_off,
                           const double* selfcoef, const double* dens, const long long* coef_off, const int* pdeg,
                           const double* wts, const int* tdrop, const long long* tgt_loc, const long long* val_off,
                           const int* ngd, double* vals, cudaStream_t s);

}  // namespace bie

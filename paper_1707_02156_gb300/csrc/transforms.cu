// SH transforms and Wigner rotation kernels (Sec. 1.1, Sec. 2.1, App. A, App. B).
//
// Synthesis (k_synth) and analysis (k_analyze) each run their Legendre and phi steps in one kernel, with
// the intermediate per-order values in shared memory.  Both steps use the symmetries of the grid:
//   theta -> pi - theta:  P~_n^m(-t) = (-1)^(n+m) P~_n^m(t) (the theta derivative with the opposite
//     sign), so the sums over even and odd n - m serve two latitudes;
//   phi_k, pi - phi_k, pi + phi_k, 2 pi - phi_k share |cos m phi| and |sin m phi|, so the sums over
//     even and odd m of the cosine and the sine parts serve four longitudes.
// In FP64, whose rate is 1/76 of FP32's here, the operation count is the bound of every large batch; the
// symmetries and the plain multiply-adds leave a quarter of the direct sums' operations.  Measured against
// the direct sums in two kernels: the rotated grids of 64 drops of degree 24 (80000 targets x 3 fields x 3
// kinds) 103.5 -> 62.7 ms with their rotation (by now a kernel of their own, rotgeo.cu), the projection of 192
// drops of degree 24 0.52 -> 0.076 ms, the surfactant's rates and implicit stage of 48 drops 10.4 -> 6.2 ms.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "internal.cuh"

namespace bie {

namespace {

namespace cg = cooperative_groups;

constexpr int kThreads = 256;

inline unsigned blocks_for(long long n, int t = kThreads) { return (unsigned)((n + t - 1) / t); }

// Derivative kinds of a synthesis, in output order: f, t, p, tt, tp, pp.  Bit k of a mask asks for kind k.
__host__ __device__ constexpr int kind_slot(int kinds, int k) {
  int s = 0;
  for (int i = 0; i < k; ++i) s += (kinds >> i) & 1;
  return s;
}

constexpr int kSynThreads = 128;
constexpr int kSynStageP = BIE_MAX_P;  // coefficients are staged in shared memory up to this degree

// One block per (field, jb latitude pairs j and P - j).  Phase 1, thread per (Legendre table, orders m and p - m,
// pair): the sums over even and odd n - m for both latitudes, and from them the complex value per order of
// each kind that the table serves (factors i m and -m^2, and the 2 of m > 0) in shared memory
// h[kind][row][m].  Phase 2, thread per (kind, row, longitude quadruple).  The two orders make every
// thread's sums p + 2 long, and the tables and kinds go to threads of their own: a block of one latitude
// pair (a few fields spread over the SMs) otherwise ran two warps, the second with one lane, each as long
// as its lowest order: 16 fields of degree 32 with five kinds on the degree-65 grid 50 -> 42 us (cold cache),
// the rotated grids of 64 drops of degree 24 56.8 -> 50.3 ms.  Where the block has a thread for every order
// anyway, each takes one.  With SRC (values only) field 3 d + c is
// component c of drop d's density, and the weighted source w_s f(s) goes to the sources' place instead of
// the value to a grid.  Several syntheses (degree groups; the standard and the upsampled grid) share a launch:
// a small one is as long as its chain of dependent loads, whatever its size, and they have nothing to wait for
// from one another: an apply's sources on both grids of two drops of degree 32 26 -> 19 us, the five
// derivatives of 16 fields each of degree 16, 24 and 32 115 -> 88 us.
template <typename R, int KINDS, bool SRC>
__global__ void __launch_bounds__(kSynThreads) k_synth(const double* __restrict__ coef, SynGroups<R> G) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int NK = kind_slot(KINDS, 6);
  SynGroup<R> A = G.g[0];
#pragma unroll
  for (int i = 1; i < kMaxSynGroups; ++i)
    if (i < G.n && (long long)blockIdx.x >= G.g[i].begin) A = G.g[i];
  const int p = A.p, P = A.P, jb = A.jb;
  const R* __restrict__ cs = A.cs;
  const int nj = P + 1, nk = 2 * P + 2, half = P + 1, np = (nj + 1) / 2, k4n = half / 2 + 1;
  const int njb = (np + jb - 1) / jb;
  const unsigned bl = blockIdx.x - (unsigned)A.begin;
  const long long f = bl / njb;
  const int q0 = (int)(bl % njb) * jb, jbn = min(jb, np - q0);
  R* h = reinterpret_cast<R*>(smem_raw);  // [NK][2 jb][p+1][2]
  const long long hk = 2LL * jb * (p + 1) * 2;
  const double* __restrict__ cg = coef + (A.field_off ? A.field_off[f] : f * A.coef_stride);
  const bool staged = p <= kSynStageP;
  R* c = h + NK * hk;
  if (staged) {
    for (int i = threadIdx.x; i < (p + 1) * (p + 1); i += kSynThreads) c[i] = (R)cg[i];
    __syncthreads();
  }
  constexpr int TABS = ((KINDS & 37) != 0) | ((KINDS & 18) != 0) << 1 | ((KINDS & 8) != 0) << 2;  // {f, p, pp}, {t, tp}, {tt}
  constexpr int NT = (TABS & 1) + (TABS >> 1 & 1) + (TABS >> 2);
  const bool both = NT * (p + 1) * jbn > kSynThreads;
  const int mh = both ? p / 2 + 1 : p + 1;  // orders a and p - a, or a alone
  for (int i = threadIdx.x; i < NT * mh * jbn; i += kSynThreads) {
    const int q = i % jbn, a = i / jbn % mh, j = q0 + q;
    int t = i / (jbn * mh);  // the t-th table in use
    if (!(TABS & 1)) ++t;
    if (t > 0 && !(TABS & 2)) ++t;
    const R* __restrict__ T = t == 0 ? A.T0 : t == 1 ? A.T1 : A.T2;
    for (int half_m = 0; half_m < 2; ++half_m) {
      const int m = half_m ? p - a : a;
      if (half_m && (!both || m == a)) break;
      R er = 0, ei = 0, odr = 0, odi = 0;  // sums over even and odd n - m
      const R* Tm = T + leg_row(p, m, m, nj) + j;
      int n = m;
#pragma unroll 2
      for (; n + 1 <= p; n += 2) {
        const int at = n * (n + 1), bt = at + 2 * n + 2;
        const R v = Tm[(long long)(n - m) * nj], w = Tm[(long long)(n + 1 - m) * nj];
        const R r0 = staged ? c[at + m] : (R)cg[at + m], r1 = staged ? c[bt + m] : (R)cg[bt + m];
        er += r0 * v;
        odr += r1 * w;
        if (m > 0) {
          const R i0 = staged ? c[at - m] : (R)cg[at - m], i1 = staged ? c[bt - m] : (R)cg[bt - m];
          ei += i0 * v;
          odi += i1 * w;
        }
      }
      if (n <= p) {
        const int at = n * (n + 1);
        const R v = Tm[(long long)(n - m) * nj];
        er += (staged ? c[at + m] : (R)cg[at + m]) * v;
        if (m > 0) ei += (staged ? c[at - m] : (R)cg[at - m]) * v;
      }
      const R fac = m == 0 ? 1 : 2;
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const R re = fac * (side == 0 ? er + odr : t == 1 ? odr - er : er - odr);
        const R im = fac * (side == 0 ? ei + odi : t == 1 ? odi - ei : ei - odi);
        R* d = h + ((2 * q + side) * (p + 1) + m) * 2;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          if (!((KINDS >> k) & 1) || t != (k == 3 ? 2 : (k == 1 || k == 4) ? 1 : 0)) continue;
          R* e = d + kind_slot(KINDS, k) * hk;
          e[0] = k == 2 || k == 4 ? -(R)m * im : k == 5 ? -(R)(m * m) * re : re;  // times 1, i m or -m^2
          e[1] = k == 2 || k == 4 ? (R)m * re : k == 5 ? -(R)(m * m) * im : im;
        }
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < NK * 2 * jbn * k4n; i += kSynThreads) {
    const int s = i / (2 * jbn * k4n), rk = i - s * 2 * jbn * k4n, row = rk / k4n, k = rk - row * k4n;
    const int j = row & 1 ? P - (q0 + row / 2) : q0 + row / 2;
    if ((row & 1) && 2 * j == P) continue;  // the middle latitude is its own mirror
    const R* hr = h + s * hk + (long long)row * (p + 1) * 2;
    R ce = hr[0], co = 0, se = 0, so = 0;
    int m = 1;
#pragma unroll 2
    for (; m + 1 <= p; m += 2) {
      const R c1 = cs[((long long)m * nk + k) * 2], s1 = cs[((long long)m * nk + k) * 2 + 1];
      const R c2 = cs[((long long)(m + 1) * nk + k) * 2], s2 = cs[((long long)(m + 1) * nk + k) * 2 + 1];
      const R* a = hr + 2 * m;
      co += a[0] * c1;
      so += a[1] * s1;
      ce += a[2] * c2;
      se += a[3] * s2;
    }
    if (m <= p) {
      co += hr[2 * m] * cs[((long long)m * nk + k) * 2];
      so += hr[2 * m + 1] * cs[((long long)m * nk + k) * 2 + 1];
    }
    const bool rot = k > 0, mir = 2 * k < half;  // k = 0 and the middle k have two longitudes, not four
    R* d0;
    R w[4] = {1, 1, 1, 1};  // the weights at k, half + k, 2 half - k, half - k
    if constexpr (SRC) {
      const long long o = A.src.off[f / 3], N = (long long)nj * nk;
      const double* __restrict__ wj = A.src.rec + 7 * o + 6 * N + (long long)j * nk;
      d0 = A.out + (f % 3) * A.src.ld + o + (long long)j * nk;
      w[0] = (R)wj[k];
      if (mir) w[1] = (R)wj[half + k];
      if (rot) w[2] = (R)wj[2 * half - k];
      if (rot && mir) w[3] = (R)wj[half - k];
    } else {
      d0 = A.out + f * A.field_stride + (long long)j * nk;
    }
    R* d = d0 + s * A.kind_stride;
    const R cp = ce + co, cm = ce - co, sp = se + so, sm = se - so;
    d[k] = w[0] * (cp - sp);
    if (mir) d[half + k] = w[1] * (cm - sm);
    if (rot) d[2 * half - k] = w[2] * (cp + sp);
    if (rot && mir) d[half - k] = w[3] * (cm + sm);
  }
}

// One cluster of cl blocks per field (cl = 1, 2, 4 or 8).  Block r of the cluster takes every cl-th part of the
// field's rows: they pass through shared memory kr at a time, folded over the four longitudes of each
// quadruple into what the even and odd orders' cosine and sine sums need, and F(m, row) of all orders stays
// in the block's shared memory.  Then block r takes the orders m = r, r + cl, ...: it folds F(m, .) over the
// latitude pairs (rows of the other blocks through distributed shared memory) and forms the products with
// the weighted Legendre table (stored with the degree fastest, so that neighbouring threads read
// neighbouring entries).  A large batch has one block per field; fewer fields spread over cl blocks each, so
// that every row is folded once however many blocks share a field (blocks of some orders, each folding the
// whole field, spend four fifths of their additions on that: 16 fields of degree 32 on the degree-65
// grid 27 us, 22 by clusters).  Only when every order of every field can have a block of its own on the SMs
// (one drop) do the blocks take one order each and fold the whole field: no block then waits for another
// (one drop of degree 32: 12 us, 16 by clusters).  Several degree groups share a launch: block ranges per
// group, arguments by value.  Behind the kernels of an apply it is launched with programmatic dependence: its
// blocks are set up as those of the kernel before end, and wait here for its results (an apply of one drop 20.6
// -> 18.6 us at degree 16 in FP64, 31.9 -> 29.8 us at degree 32).  The kernel before does not trigger the launch
// itself: with an early trigger the waiting blocks take room from its own (33.9 us).
constexpr int kAnaThreads = 256;

__host__ __device__ inline int ana_rows(int P, int cl) {  // rows per pass: at most 40 KB folded
  const int own = (P + cl) / cl, fit = (40 << 10) / (32 * ((P + 1) / 2 + 1));
  return own < fit ? own : fit < 1 ? 1 : fit;
}

__global__ void __launch_bounds__(kAnaThreads) k_analyze(AnaGroups G, const double* __restrict__ grid,
                                                         double* __restrict__ coef) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  cg::cluster_group cluster = cg::this_cluster();
  AnaGroup A = G.g[0];
#pragma unroll
  for (int i = 1; i < kMaxAnaGroups; ++i)
    if (i < G.n && (long long)blockIdx.x >= G.g[i].begin) A = G.g[i];
  // one order per block (G.orders): the block's only row part is the whole field, its only order m_own
  const int P = A.P, p = A.p, cl = G.cl, rank = (int)cluster.block_rank();
  const int per_f = G.orders ? p + 1 : cl;
  const int nj = P + 1, nk = 2 * P + 2, half = P + 1, np = (nj + 1) / 2, k4n = half / 2 + 1, kr = ana_rows(P, cl);
  const long long f = ((long long)blockIdx.x - A.begin) / per_f;
  const int m_own = G.orders ? (int)((long long)blockIdx.x - A.begin - f * per_f) : 0, nm = G.orders ? 1 : p + 1;
  const int own = (nj + cl - 1) / cl;  // rows per block: rank * own ..
  const int r0 = rank * own, r1 = min(nj, r0 + own);
  double* F = reinterpret_cast<double*>(smem_raw);      // [own][nm][2]
  double* fold = F + 2LL * own * nm;               // [cos even, cos odd, sin even, sin odd][k4n][kr]
  double* E = fold;                                     // later: [nj][2] per order of a pass
  const double* src = grid + A.grid_base + (A.grid_off ? A.grid_off[f] : f * A.grid_stride);
  for (int j0 = r0; j0 < r1; j0 += kr) {
    const int rn = min(kr, r1 - j0);
    for (int i = threadIdx.x; i < rn * k4n; i += kAnaThreads) {
      const int r = i / k4n, k = i - r * k4n;
      const double* g = src + (long long)(j0 + r) * nk;
      const bool rot = k > 0, mir = 2 * k < half;
      const double a = g[k], b = rot ? g[2 * half - k] : 0.0, c = mir ? g[half + k] : 0.0,
                   d = rot && mir ? g[half - k] : 0.0;
      const double ab = a + b, cd = c + d, amb = a - b, cmd = c - d;
      double* o = fold + k * kr + r;
      o[0] = ab + cd;
      o[k4n * kr] = ab - cd;
      o[2 * k4n * kr] = amb + cmd;
      o[3 * k4n * kr] = amb - cmd;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nm * rn; i += kAnaThreads) {
      const int mi = i / rn, r = i - mi * rn, m = m_own + mi, odd = m & 1;
      const double* c = A.cs + (long long)m * nk * 2;
      const double* fc = fold + (long long)odd * k4n * kr + r;
      const double* fs = fold + (long long)(2 + odd) * k4n * kr + r;
      double re = 0, im = 0;
#pragma unroll 4
      for (int k = 0; k < k4n; ++k) {
        re += fc[k * kr] * c[2 * k];
        im -= fs[k * kr] * c[2 * k + 1];
      }
      double* o = F + 2 * ((long long)(j0 - r0 + r) * nm + mi);
      o[0] = re;
      o[1] = im;
    }
    __syncthreads();
  }
  cluster.sync();
  double* out = coef + A.coef_base + (A.coef_off ? A.coef_off[f] : f * A.coef_stride);
  const int mp = max(1, 2 * k4n * kr / nj);  // orders per pass: E in the space of the folded rows
  for (int a0 = m_own + rank; a0 < m_own + nm; a0 += cl * mp) {
    const int mn = min(mp, (m_own + nm - 1 - a0) / cl + 1);  // orders a0, a0 + cl, ...
    // latitude pairs: F(j) + F(P-j) at j for even n - m, F(j) - F(P-j) at P-j for odd
    for (int i = threadIdx.x; i < mn * np; i += kAnaThreads) {
      const int mm = i / np, j = i - mm * np, m = a0 + mm * cl, jm = P - j;
      const double* lo = cluster.map_shared_rank(F, j / own) + 2 * ((long long)(j % own) * nm + m - m_own);
      const double* hi = cluster.map_shared_rank(F, jm / own) + 2 * ((long long)(jm % own) * nm + m - m_own);
      const double ar = lo[0], ai = lo[1], br = hi[0], bi = hi[1];
      double* e = E + 2 * (long long)mm * nj;
      if (j == jm) {  // the middle latitude is its own mirror
        e[2 * j] = ar;
        e[2 * j + 1] = ai;
      } else {
        e[2 * j] = ar + br;
        e[2 * j + 1] = ai + bi;
        e[2 * jm] = ar - br;
        e[2 * jm + 1] = ai - bi;
      }
    }
    __syncthreads();
    const int per = p + 1 - a0;  // degrees of the pass's lowest order
    // a pass of few sums splits each over four neighbouring threads (a quarter of the serial loads), a pass of
    // many does not (the partial sums would cost half as many additions again)
    const int split = mn * per <= kAnaThreads / 4 ? 4 : 1;
    for (int i0 = 0; i0 < mn * per * split; i0 += kAnaThreads) {
      const int i = (i0 + (int)threadIdx.x) / split, part = threadIdx.x % split;
      const int mm = i / per, d = i - mm * per, m = a0 + mm * cl, n = m + d;
      const bool valid = i < mn * per && n <= p;
      double re = 0, im = 0;
      if (valid) {
        const bool odd = d & 1;
        const double* a = A.At + leg_row(p, m, m, nj) + d;
        const double* Em = E + 2 * (long long)mm * nj;
#pragma unroll 4
        for (int j = part; j < (odd ? nj / 2 : np); j += split) {
          const double v = a[(long long)j * (p + 1 - m)];
          const int jj = odd ? P - j : j;
          re += v * Em[2 * jj];
          im += v * Em[2 * jj + 1];
        }
      }
      if (split > 1)
        for (int o = 2; o > 0; o >>= 1) {
          re += __shfl_xor_sync(0xffffffffu, re, o);
          im += __shfl_xor_sync(0xffffffffu, im, o);
        }
      if (!valid || part) continue;
      out[n * (n + 1) + m] = re;
      if (m > 0) out[n * (n + 1) - m] = im;
    }
    __syncthreads();
  }
  cluster.sync();  // a block's F stays until the others have read it
}

constexpr int kRotB = 16;  // targets (longitudes) per rotation block

// One block per (drop, latitude a, degree n, chunk of kRotB longitudes b).
// Stage: real blocks C (n+1)^2 and S n^2 of the latitude, and g = e^{i m alpha_b} f_n^m for the
// chunk; then Re g'_{m'} = sum_m C[m'][m] Re g_m,  Im g'_{m'} = sum_m S[m'-1][m-1] Im g_m.
template <typename CT, typename R>
__global__ void k_rotate(const CT* __restrict__ coef, const long long* __restrict__ field_off, int ncomp,
                         int p, const R* __restrict__ blocks, long long blk_stride, int na, int nb,
                         const R* __restrict__ ph, R* __restrict__ out, long long out_drop_stride) {
  extern __shared__ unsigned char smem_raw[];
  R* sm = reinterpret_cast<R*>(smem_raw);
  const int nbch = (nb + kRotB - 1) / kRotB;
  long long item = blockIdx.x;
  const int bc = (int)(item % nbch);
  item /= nbch;
  const int n = (int)(item % (p + 1));
  item /= (p + 1);
  const int a = (int)(item % na);
  const long long ld = item / na;
  const int b0 = bc * kRotB;
  const int nbh = min(kRotB, nb - b0);
  const int w = 2 * n + 1;
  const int nC = (n + 1) * (n + 1), nS = n * n;
  R* sC = sm;
  R* sS = sC + nC;
  R* sG = sS + nS;  // [bb][c][w]: entries 0..n = Re g_m, n+1..2n = Im g_m (m = 1..n)
  const R* blk = blocks + (long long)a * blk_stride;
  long long boff = 0;
  for (int k = 0; k < n; ++k) boff += (long long)(k + 1) * (k + 1) + (long long)k * k;
  for (int i = threadIdx.x; i < nC + nS; i += blockDim.x) sC[i] = blk[boff + i];
  const int ng = nbh * ncomp;
  for (int i = threadIdx.x; i < ng * (n + 1); i += blockDim.x) {
    int m = i % (n + 1);
    int g = i / (n + 1);
    int c = g % ncomp;
    int bb = g / ncomp;
    const CT* cf = coef + field_off[ld * ncomp + c];
    R fr = (R)cf[n * (n + 1) + m];
    R fi = m > 0 ? (R)cf[n * (n + 1) - m] : (R)0;
    R cr = 1, ci = 0;
    if (ph) {
      cr = ph[((long long)m * nb + (b0 + bb)) * 2];
      ci = ph[((long long)m * nb + (b0 + bb)) * 2 + 1];
    }
    sG[g * w + m] = fr * cr - fi * ci;
    if (m > 0) sG[g * w + n + m] = fr * ci + fi * cr;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ng * w; i += blockDim.x) {
    int o = i % w;
    int g = i / w;
    int c = g % ncomp;
    int bb = g / ncomp;
    const R* G = sG + g * w;
    R acc = 0;
    int dst;
    if (o <= n) {  // Re g'_{o}
      for (int m = 0; m <= n; ++m) acc += sC[m * (n + 1) + o] * G[m];
      dst = n * (n + 1) + o;
    } else {  // Im g'_{mp}, mp = o - n
      int mp = o - n;
      for (int m = 1; m <= n; ++m) acc += sS[(m - 1) * n + (mp - 1)] * G[n + m];
      dst = n * (n + 1) - mp;
    }
    long long t = (long long)a * nb + b0 + bb;
    out[ld * out_drop_stride + (t * ncomp + c) * (long long)((p + 1) * (p + 1)) + dst] = acc;
  }
}

__global__ void k_phase(double* __restrict__ coef, long long nfield, int p, double gamma) {
  long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  long long per = (long long)(p + 1) * (p + 1);
  if (idx >= nfield * per) return;
  long long f = idx / per;
  int r = (int)(idx - f * per);
  int n = 0;
  while ((n + 1) * (n + 1) <= r) ++n;
  int m = r - n * (n + 1);
  if (m <= 0) return;  // the thread owning Re f_n^m (m > 0) rotates the pair
  double* c = coef + f * per;
  double re = c[n * (n + 1) + m], im = c[n * (n + 1) - m];
  double s, co;
  sincos(m * gamma, &s, &co);
  c[n * (n + 1) + m] = re * co - im * s;
  c[n * (n + 1) - m] = re * s + im * co;
}

}  // namespace

template <typename R, int KINDS, bool SRC = false>
static int synth_launch(const double* coef, std::vector<SynGroup<R>> groups, int sms, cudaStream_t s) {
  std::sort(groups.begin(), groups.end(), [](const SynGroup<R>& x, const SynGroup<R>& y) { return x.P > y.P; });
  long long work = 0;  // latitude pairs of all fields
  for (const auto& g : groups) work += g.nfield * ((g.P + 2) / 2);
  if (work == 0) return BIE_OK;
  // latitude pairs per block: all of them when there are fields for four blocks per SM (the coefficients
  // are staged once), fewer when not, so that small batches spread over the SMs; at most 64 KB a block
  const long long want = std::max(1LL, work / (4LL * sms));
  auto kern = k_synth<R, KINDS, SRC>;
  for (size_t g0 = 0; g0 < groups.size(); g0 += kMaxSynGroups) {
    SynGroups<R> G{};
    G.n = (int)std::min<size_t>(kMaxSynGroups, groups.size() - g0);
    size_t smem = 0;
    long long nblk = 0;
    for (int i = 0; i < G.n; ++i) {
      SynGroup<R>& g = G.g[i] = groups[g0 + i];
      const int np = (g.P + 2) / 2;
      const size_t stage = g.p <= kSynStageP ? sizeof(R) * (size_t)(g.p + 1) * (g.p + 1) : 0;
      const size_t pair = sizeof(R) * kind_slot(KINDS, 6) * 4 * (size_t)(g.p + 1);
      const long long fit = std::max<long long>(1, ((64 << 10) - (long long)stage) / (long long)pair);
      g.jb = (int)std::min<long long>(np, std::min(want, fit));
      g.begin = nblk;
      nblk += g.nfield * ((np + g.jb - 1) / g.jb);
      smem = std::max(smem, stage + pair * g.jb);
    }
    if (nblk == 0) continue;
    if (nblk > 0x7fffffffLL) return BIE_EINVAL;
    BIE_CUDA_TRY(allow_smem(kern, smem));
    kern<<<(unsigned)nblk, kSynThreads, smem, s>>>(coef, G);
    count_launch();
    BIE_CUDA_TRY(cudaGetLastError());
  }
  return BIE_OK;
}

int launch_synth(int kinds, const double* coef, std::vector<SynGroup<double>> groups, int sms, cudaStream_t s) {
#define BIE_SYNTH(K) \
  if (kinds == K) return synth_launch<double, K>(coef, std::move(groups), sms, s)
  BIE_SYNTH(1);
  BIE_SYNTH(6);
  BIE_SYNTH(7);
  BIE_SYNTH(62);
  BIE_SYNTH(63);
#undef BIE_SYNTH
  return BIE_EINVAL;
}

template <typename R>
int launch_synth_sources(const double* coef, std::vector<SynGroup<R>> groups, int sms, cudaStream_t s) {
  return synth_launch<R, 1, true>(coef, std::move(groups), sms, s);
}

int launch_analyze(std::vector<AnaGroup> groups, const double* grid, double* coef, int sms, cudaStream_t s, bool early) {
  std::sort(groups.begin(), groups.end(), [](const AnaGroup& x, const AnaGroup& y) { return x.P > y.P; });
  long long fields = 0;
  for (const auto& g : groups) fields += g.nfield;
  if (fields == 0) return BIE_OK;
  for (size_t g0 = 0; g0 < groups.size(); g0 += kMaxAnaGroups) {
    AnaGroups G{};
    G.n = (int)std::min<size_t>(kMaxAnaGroups, groups.size() - g0);
    for (int i = 0; i < G.n; ++i) G.g[i] = groups[g0 + i];
    long long orders = 0;
    for (int i = 0; i < G.n; ++i) orders += G.g[i].nfield * (G.g[i].p + 1);
    G.orders = orders <= sms;
    auto bytes = [&](int cl) {
      size_t v = 0;
      for (int i = 0; i < G.n; ++i) {
        const int P = G.g[i].P;
        v = std::max(v, sizeof(double) * (2 * (size_t)((P + cl) / cl) * (G.orders ? 1 : G.g[i].p + 1) +
                                          std::max(4 * (size_t)((P + 1) / 2 + 1) * ana_rows(P, cl), 2 * (size_t)(P + 1))));
      }
      return v;
    };
    // blocks per field: as few as give two blocks per SM, and as many as the largest group's F needs
    G.cl = 1;
    while (!G.orders && G.cl < 8 && (fields * G.cl < 2LL * sms || bytes(G.cl) > 96 * 1024)) G.cl *= 2;
    const size_t smem = bytes(G.cl);
    if (smem > kMaxSmem) return BIE_EINVAL;
    long long nblk = 0;
    for (int i = 0; i < G.n; ++i) {
      G.g[i].begin = nblk;
      nblk += G.g[i].nfield * (G.orders ? G.g[i].p + 1 : G.cl);
    }
    if (nblk == 0) continue;
    if (nblk > 0x7fffffffLL) return BIE_EINVAL;
    BIE_CUDA_TRY(allow_smem(k_analyze, smem));
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[2]{};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)G.cl;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)nblk);
    cfg.blockDim = dim3(kAnaThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = early && g0 == 0 ? 2 : 1;  // a second launch follows one that is early itself
    BIE_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_analyze, G, grid, coef));
    count_launch();
    BIE_CUDA_TRY(cudaGetLastError());
  }
  return BIE_OK;
}

template <typename CT, typename R>
int launch_rotate(const CT* coef, const long long* field_off, int ncomp, long long ndrop, int p, const R* blocks,
                  long long blk_stride, int na, int nb, const R* ph, R* out, long long out_drop_stride,
                  cudaStream_t s) {
  const int nbch = (nb + kRotB - 1) / kRotB;
  long long nblk = ndrop * na * (long long)(p + 1) * nbch;
  if (nblk == 0) return BIE_OK;
  size_t smem = sizeof(R) * ((size_t)(p + 1) * (p + 1) + (size_t)p * p + (size_t)kRotB * ncomp * (2 * p + 1));
  BIE_CUDA_TRY(allow_smem(k_rotate<CT, R>, smem));
  if (nblk > 0x7fffffffLL) return BIE_EINVAL;
  k_rotate<CT, R><<<(unsigned)nblk, 128, smem, s>>>(coef, field_off, ncomp, p, blocks, blk_stride, na, nb, ph, out,
                                                    out_drop_stride);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_phase(double* coef, long long nfield, int p, double gamma, cudaStream_t s) {
  long long n = nfield * (long long)(p + 1) * (p + 1);
  if (n == 0 || gamma == 0.0) return BIE_OK;
  k_phase<<<blocks_for(n), kThreads, 0, s>>>(coef, nfield, p, gamma);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

// explicit instantiations
template int launch_synth_sources<double>(const double*, std::vector<SynGroup<double>>, int, cudaStream_t);
template int launch_synth_sources<float>(const double*, std::vector<SynGroup<float>>, int, cudaStream_t);
template int launch_rotate<double, double>(const double*, const long long*, int, long long, int, const double*,
                                           long long, int, int, const double*, double*, long long, cudaStream_t);
template int launch_rotate<double, float>(const double*, const long long*, int, long long, int, const float*,
                                          long long, int, int, const float*, float*, long long, cudaStream_t);

}  // namespace bie

// Singular self interaction of every drop (Thm 1, Sec. 2.2, App. B): one block per target.
//
// Both forms rotate the density so that the target sits at the pole (App. B, real blocks of the
// latitude's Wigner matrices applied to e^{i m phi_b} rho_n^m).
//
//  * direct form: the Legendre step of the synthesis on the degree-pq grid,
//    h_m(theta_j) = sum_n rho'_n^m P~_n^m(cos theta_j), runs in shared memory; the phi step rho'(theta_j, phi_k) = h_0 + 2 Re sum_m h_m e^{i m phi_k} is evaluated
//    for the longitude pair (k, k + pq + 1) from the even and odd orders, and the Stokeslet or
//    stresslet pair sum of Thm 1 is accumulated against the cached rotated geometry;
//  * dense form (the default): the same double sum reassociated exactly,
//        sum_{j,k} M_jk rho'_jk = sum_j sum_m c_m Re[ Mhat_jm h_m(theta_j) ]
//                               = sum_{n, m >= 0} Re[ Q_nm rho'_n^m ],   Q_nm = c_m sum_j Mhat_jm P~_n^m(cos theta_j),
//    with c_0 = 1, c_m = 2, M_jk the 3x3 kernel weight of the quadrature point
//    (w^s_j K(x0 - x') W'/sin theta_j, geometry only) and Mhat_jm = sum_k M_jk e^{i m phi_k} its phi
//    transform; and since rho' = R rho with the target's rotation R (App. B), the sum is
//    sum_r (R^T Q)_r rho_r: the rotation is applied to the factors once per geometry, not to the
//    density on every apply.  S = R^T Q (six symmetric 3x3 entries per coefficient and target) is what
//    an apply reads, once.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "dfloat.cuh"
#include "device.cuh"
#include "fixed.cuh"
#include "internal.cuh"

namespace bie {
namespace {

// Stages 0-1: g = e^{i m phi_b} rho_n^m (three components) then the rotation, rc = rotated
// coefficients (real-packed, [3][(p+1)^2]).  g and rc are shared-memory arrays.
template <typename R>
__device__ void rotate_target(const double* __restrict__ dens, const long long* __restrict__ foff3, long long ld,
                              int p, int a, int b, const R* __restrict__ wblk, long long wstride,
                              const R* __restrict__ ph, R* rc, R* g) {
  const int nc = (p + 1) * (p + 1);
  const int nb = 2 * p + 2;
  for (int i = threadIdx.x; i < 3 * nc; i += blockDim.x) {
    const int c = i / nc, r = i - c * nc;
    const int n = degree_of(r);
    const int m = r - n * (n + 1);
    if (m < 0) continue;  // the owner of Re rho_n^m writes both parts
    const double* f = dens + foff3[ld * 3 + c];
    const R fr = (R)f[n * (n + 1) + m];
    const R fi = m > 0 ? (R)f[n * (n + 1) - m] : (R)0;
    const R co = ph[((long long)m * nb + b) * 2], si = ph[((long long)m * nb + b) * 2 + 1];
    g[c * nc + n * (n + 1) + m] = fr * co - fi * si;
    if (m > 0) g[c * nc + n * (n + 1) - m] = fr * si + fi * co;
  }
  __syncthreads();
  const R* blk = wblk + (long long)a * wstride;
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    const int n = degree_of(i);
    const int o = i - n * n;  // 0..2n
    // blocks of degree n start after sum_{k<n} (k+1)^2 + k^2 entries
    const long long boff = (long long)n * (n + 1) * (2 * n + 1) / 6 + (long long)(n - 1) * n * (2 * n - 1) / 6;
    const R* g0 = g + n * (n + 1);
    R a0 = 0, a1 = 0, a2 = 0;
    int dst;
    if (o <= n) {
      const R* Cc = blk + boff + o;  // column-major: entry (o, m) at m (n+1) + o
      for (int m = 0; m <= n; ++m) {
        const R cv = Cc[(long long)m * (n + 1)];
        a0 += cv * g0[m];
        a1 += cv * g0[nc + m];
        a2 += cv * g0[2 * nc + m];
      }
      dst = n * (n + 1) + o;
    } else {
      const int mp = o - n;
      const R* Sc = blk + boff + (long long)(n + 1) * (n + 1) + (mp - 1);
      for (int m = 1; m <= n; ++m) {
        const R sv = Sc[(long long)(m - 1) * n];
        a0 += sv * g0[-m];
        a1 += sv * g0[nc - m];
        a2 += sv * g0[2 * nc - m];
      }
      dst = n * (n + 1) - mp;
    }
    rc[dst] = a0;
    rc[nc + dst] = a1;
    rc[2 * nc + dst] = a2;
  }
  __syncthreads();
}

// Stage 2: h[c][jj][m] (complex) = sum_n rc[c](n, m) T0[m][n][j0 + jj] for jj < jn.
template <typename R>
__device__ void legendre_chunk(const R* rc, int p, int nq_j, int j0, int jn, const R* __restrict__ T0, R* h) {
  const int nc = (p + 1) * (p + 1);
  const long long cstride = (long long)jn * (p + 1) * 2;
  for (int i = threadIdx.x; i < (p + 1) * jn; i += blockDim.x) {
    const int m = i / jn, jj = i - m * jn;
    const R* Tm = T0 + leg_row(p, m, m, nq_j) + j0 + jj;
    R r0 = 0, r1 = 0, r2 = 0, i0 = 0, i1 = 0, i2 = 0;
    for (int n = m; n <= p; ++n) {
      const R tv = Tm[(long long)(n - m) * nq_j];
      const int re = n * (n + 1) + m;
      r0 += rc[re] * tv;
      r1 += rc[nc + re] * tv;
      r2 += rc[2 * nc + re] * tv;
      if (m > 0) {
        const int im = n * (n + 1) - m;
        i0 += rc[im] * tv;
        i1 += rc[nc + im] * tv;
        i2 += rc[2 * nc + im] * tv;
      }
    }
    R* hh = h + ((long long)jj * (p + 1) + m) * 2;
    hh[0] = r0;
    hh[1] = i0;
    hh[cstride] = r1;
    hh[cstride + 1] = i1;
    hh[2 * cstride] = r2;
    hh[2 * cstride + 1] = i2;
  }
  __syncthreads();
}

template <typename R>
__device__ inline void write_target(R s0, R s1, R s2, const double* __restrict__ wts,
                                    const long long* __restrict__ val_off, double* __restrict__ vals, long long ld,
                                    int tl, int ng) {
  __shared__ R red[3 * 32];
  block_sum3<R>(s0, s1, s2, red);
  if (threadIdx.x == 0) {
    const double wt = wts[ld];
    double* v = vals + val_off[ld] + tl;
    v[0] = wt * (double)s0;
    v[ng] = wt * (double)s1;
    v[2 * (long long)ng] = wt * (double)s2;
  }
}

// ---- direct form ----
template <typename R, int KIND>
__global__ void __launch_bounds__(256) k_self_direct(
    const double* __restrict__ dens, const long long* __restrict__ foff3, int p, int pq, const R* __restrict__ wblk,
    long long wstride, const R* __restrict__ ph, const R* __restrict__ T0, const R* __restrict__ cs,
    const R* __restrict__ cache, int ng, const double* __restrict__ wts, const long long* __restrict__ val_off,
    double* __restrict__ vals, int jc) {
  extern __shared__ unsigned char smem_raw[];
  R* rc = reinterpret_cast<R*>(smem_raw);
  const int nc = (p + 1) * (p + 1);
  R* un = rc + 3 * nc;
  const long long t = blockIdx.x;
  const long long ld = t / ng;
  const int tl = (int)(t - ld * ng);
  const int a = tl / (2 * p + 2), b = tl - a * (2 * p + 2);
  const int nq_j = pq + 1, nk = 2 * pq + 2, half = pq + 1;
  const long long nq = (long long)nq_j * nk;
  rotate_target<R>(dens, foff3, ld, p, a, b, wblk, wstride, ph, rc, un);
  const R* geo = cache + t * 7 * nq;
  R s0 = 0, s1 = 0, s2 = 0;
  for (int j0 = 0; j0 < nq_j; j0 += jc) {
    const int jn = min(jc, nq_j - j0);
    legendre_chunk<R>(rc, p, nq_j, j0, jn, T0, un);
    const long long cstride = (long long)jn * (p + 1) * 2;
    for (int i = threadIdx.x; i < jn * half; i += blockDim.x) {
      const int jj = i / half, k = i - jj * half;
      const R* hh = un + (long long)jj * (p + 1) * 2;
      R e0 = hh[0], e1 = hh[cstride], e2 = hh[2 * cstride];
      R o0 = 0, o1 = 0, o2 = 0;
      for (int m = 1; m <= p; ++m) {
        const R co = cs[((long long)m * nk + k) * 2], si = cs[((long long)m * nk + k) * 2 + 1];
        const R* hm = hh + 2 * m;
        const R v0 = 2 * (hm[0] * co - hm[1] * si);
        const R v1 = 2 * (hm[cstride] * co - hm[cstride + 1] * si);
        const R v2 = 2 * (hm[2 * cstride] * co - hm[2 * cstride + 1] * si);
        if (m & 1) {
          o0 += v0;
          o1 += v1;
          o2 += v2;
        } else {
          e0 += v0;
          e1 += v1;
          e2 += v2;
        }
      }
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const long long q = (long long)(j0 + jj) * nk + k + side * half;
        const R r0 = side ? e0 - o0 : e0 + o0;
        const R r1 = side ? e1 - o1 : e1 + o1;
        const R r2 = side ? e2 - o2 : e2 + o2;
        const R x0 = geo[q], x1 = geo[nq + q], x2 = geo[2 * nq + q];
        const R ri = rsqrt_<R>(x0 * x0 + x1 * x1 + x2 * x2);
        const R xr = x0 * r0 + x1 * r1 + x2 * r2;
        if (KIND == 0) {
          const R wi = geo[6 * nq + q] * ri;
          const R c = wi * xr * ri * ri;
          s0 += wi * r0 + c * x0;
          s1 += wi * r1 + c * x1;
          s2 += wi * r2 + c * x2;
        } else {
          const R xn = x0 * geo[3 * nq + q] + x1 * geo[4 * nq + q] + x2 * geo[5 * nq + q];  // with the weight
          const R ri2 = ri * ri;
          const R c = (R)(-6) * xr * xn * ri2 * ri2 * ri;
          s0 += c * x0;
          s1 += c * x1;
          s2 += c * x2;
        }
      }
    }
    __syncthreads();
  }
  write_target<R>(s0, s1, s2, wts, val_off, vals, ld, tl, ng);
}

// ---- dense form: set-up of the projected factors Q (FP64) ----
// For each target, Q[t][e][ri][tri(n,m)] = c_m sum_j Mhat_{e,jm} P~_n^m(cos theta_j), with
// Mhat_{e,jm} = sum_k M_{e,jk} e^{i m phi_k} the phi transform of entry e of the 3x3 kernel weight
// over (xx, yy, zz, xy, xz, yz), ri = real / imaginary part, c_0 = 1 and c_m = 2.  Latitudes are
// processed NP pairs (q, pq - q) at a time: kernel weights; their sums over the longitude
// quadruples that share |cos m phi| and |sin m phi|, in place; the phi transform of both rows, whose sum
// and difference serve even and odd n - m; and the Legendre projection, accumulated in shared memory.
// The phi transform and the projection (0.15M multiply-adds per target and kind at p = pq = 24) run in
// fixed point on the integer pipe (fixed.cuh), on one scale per target and entry from a first pass over the
// kernel weights, which leaves their factors c and d in the cache for the second; the FP64 pipe, which bounded
// the kernel before, keeps the weights themselves.  64 drops of degree 24, both kinds: 127 ms by the direct sums,
// 62 by the symmetries in FP64, now 31.
// Two pairs a pass where they fit a block's shared memory (fewer barriers: 43.8 ms with the rotation below; three or
// four 46.9 and 45.1), one at the largest degrees.

__device__ inline int tri_index_degree(int it) {
  int n = (int)((sqrtf(8.0f * it + 1.0f) - 1.0f) * 0.5f);
  while ((n + 1) * (n + 2) / 2 <= it) ++n;
  while (n * (n + 1) / 2 > it) --n;
  return n;
}

// Bounds on the exponents of a target's six entries, each on a scale of its own (a drop that is thin along an axis has
// entries of very different size): with d = w/r the Stokeslet's diagonal part and b_i = c x_i^2 (c = w/r^3 or -6 x.a /
// r^5), |entry ij| = |c x_i x_j| < 2^((E(b_i) + E(b_j))/2), E the exponent of the largest over the points (em their
// magnitudes); the Stokeslet's diagonal entries are below 2 d.
template <int KIND>
__device__ __forceinline__ int entry_exponent(const int* em, int entry) {
  const int i = entry < 3 ? entry : entry == 5 ? 1 : 0, j = entry < 3 ? entry : entry == 3 ? 1 : 2;
  const int ei = fix_exponent(em[KIND == 0 && entry < 3 ? 3 : i]), ej = fix_exponent(em[KIND == 0 && entry < 3 ? 3 : j]);
  return ei == fix_none || ej == fix_none ? 0 : (ei + ej + 1) >> 1;
}

template <int KIND, int NP>
__global__ void __launch_bounds__(256) k_kernel_proj(double* cache, int pq, int p,
                                                     const int4* __restrict__ CT, const int2* __restrict__ PT,
                                                     double* __restrict__ Q64) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int em[4], es[6];
  const long long t = blockIdx.x;
  const int nq_j = pq + 1, nk = 2 * pq + 2, half = pq + 1, np = (nq_j + 1) / 2, k4n = half / 2 + 1;
  const int ntri = (p + 1) * (p + 2) / 2;
  const int mid = half % 2 == 0 ? half / 2 : -1;
  double* sk = reinterpret_cast<double*>(smem_raw);                                  // [pair][row][6][nk]
  int2* si = reinterpret_cast<int2*>(sk);                                            // the folded sums, in place
  int2* sd = reinterpret_cast<int2*>(sk + NP * 12 * nk);                     // [pair][even, odd][12][p+1]
  long long* sq = reinterpret_cast<long long*>(sd + NP * 24 * (p + 1));      // [12][ntri]
  const long long nq = (long long)nq_j * nk;
  double* geo = cache + t * 7 * nq;
  for (int i = threadIdx.x; i < 12 * ntri; i += blockDim.x) sq[i] = 0;
  if (threadIdx.x < 4) em[threadIdx.x] = 0;
  __syncthreads();
  {
    int e[4] = {0, 0, 0, 0};
#pragma unroll 2
    for (int o = threadIdx.x; o < nq; o += blockDim.x) {
      const double x0 = geo[o], x1 = geo[nq + o], x2 = geo[2 * nq + o];
      const double y0 = x0 * x0, y1 = x1 * x1, y2 = x2 * x2;
      const double r2 = y0 + y1 + y2;
      double c;
      if (KIND == 0) {
        const double ri = rsqrt_<double>(r2), d = geo[6 * nq + o] * ri;
        c = d * (ri * ri);
        geo[6 * nq + o] = d;  // for the second pass
        e[3] = max(e[3], fix_magnitude(d));
      } else {
        c = (-6.0 * (x0 * geo[3 * nq + o] + x1 * geo[4 * nq + o] + x2 * geo[5 * nq + o])) * rsqrt5_<double>(r2);
      }
      geo[3 * nq + o] = c;
      e[0] = max(e[0], fix_magnitude(c * y0));
      e[1] = max(e[1], fix_magnitude(c * y1));
      e[2] = max(e[2], fix_magnitude(c * y2));
    }
#pragma unroll
    for (int k = 0; k < (KIND == 0 ? 4 : 3); ++k) {
      e[k] = __reduce_max_sync(0xffffffffu, e[k]);
      // with a margin of 1e-4 for their rounding (in the magnitude's mantissa); the Stokeslet's diagonal entries are below 2 d
      if ((threadIdx.x & 31) == 0 && e[k]) atomicMax(&em[k], e[k] + (KIND == 0 && k == 3 ? (1 << 20) + 128 : 128));
    }
  }
  __syncthreads();
  const bool bad = fix_exponent(max(max(em[0], em[1]), max(em[2], em[3]))) == fix_bad;
  if (threadIdx.x < 6) es[threadIdx.x] = entry_exponent<KIND>(em, threadIdx.x);  // read after the next barriers
  // units (e the entry's exponent, lk the bits of k4n): entries 2^(e - 61 + lk), folded sums of four below 2^(63 - lk),
  // which leaves the phi transform (tables 2^-55) room for its k4n products, and below 2^60 (by the bounds' margin of
  // 1e-4), so that their high parts are 32-bit; the transforms 2^(e - 57 + lk), the sum of two rows' below 2^60 (the
  // projection adds NP products of it, and no more); the projections (tables 2^-55) 2^(e - 54 + lk + sf) (np <= 64:
  // larger grids take the direct form)
  const int lk = max(3, ceil_log2(k4n)), sf = max(0, ceil_log2(np) - 3);
  const long long rnd = sf > 0 ? 1LL << (sf - 1) : 0, xrnd = sf > 0 ? 0 : 1LL << (kFixPart - 1);  // unbiased
  for (int q0 = 0; q0 < np && !bad; q0 += NP) {
    const int qn = min(NP, np - q0);
    for (int i = threadIdx.x; i < qn * 2 * nk; i += blockDim.x) {
      const int row = i / nk, k = i - row * nk;
      const int q = q0 + row / 2, j = row & 1 ? pq - q : q;
      double* v = sk + row * 6 * nk + k;
      if ((row & 1) && 2 * q == pq) {  // the middle latitude has no mirror
#pragma unroll
        for (int c = 0; c < 6; ++c) v[c * nk] = 0.0;
        continue;
      }
      const long long o = (long long)j * nk + k;
      const double x0 = geo[o], x1 = geo[nq + o], x2 = geo[2 * nq + o], c = geo[3 * nq + o];
      const double d = KIND == 0 ? geo[6 * nq + o] : 0.0;
      const double a0 = c * x0, a1 = c * x1;
      v[0] = d + a0 * x0;
      v[nk] = d + a1 * x1;
      v[2 * nk] = d + (c * x2) * x2;
      v[3 * nk] = a0 * x1;
      v[4 * nk] = a0 * x2;
      v[5 * nk] = a1 * x2;
    }
    __syncthreads();
    // cosine sums of the even and odd orders at k and half + k, sine sums at 2 half - k and half - k (a middle
    // k has two longitudes: one cosine sum at k, one sine sum at half + k)
    for (int i = threadIdx.x; i < qn * 12 * k4n; i += blockDim.x) {
      const int k = i % k4n, e = es[i / k4n % 6] - 4 + lk;  // 57 - e: 61 - lk bits below the entry's scale
      double* v = sk + (i / k4n) * nk;
      int2* w = si + (i / k4n) * nk;
      const long long a = fix_encode(v[k], e), c = fix_encode(v[half + k], e);
      if (k == 0 || k == mid) {
        w[k] = fix_split(a + c);
        w[half + k] = fix_split(a - c);
      } else {
        const long long b = fix_encode(v[2 * half - k], e), d = fix_encode(v[half - k], e);
        w[k] = fix_split((a + b) + (c + d));
        w[half + k] = fix_split((a + b) - (c + d));
        w[2 * half - k] = fix_split((a - b) + (c - d));
        w[half - k] = fix_split((a - b) - (c - d));
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < qn * 6 * (p + 1); i += blockDim.x) {
      const int m = i % (p + 1);
      const int r = i / (p + 1);
      const int c = r % 6, pair = r / 6;
      const int2* v0 = si + (pair * 12 + c) * nk;  // row q; row pq - q is 6 nk further
      const int2* vc = v0 + ((m & 1) ? half : 0);
      const int2* vs = v0 + ((m & 1) ? half : 2 * half);
      long long h[4] = {0, 0, 0, 0}, x[4] = {0, 0, 0, 0};  // cosine and sine sums of the two rows
      const int4 c0 = CT[m];
      fix_mad(h[0], x[0], vc[0], make_int2(c0.x, c0.y));
      fix_mad(h[1], x[1], vc[6 * nk], make_int2(c0.x, c0.y));
#pragma unroll 2
      for (int k = 1; 2 * k < half; ++k) {
        const int4 cs = CT[k * (p + 1) + m];
        const int2 co = make_int2(cs.x, cs.y), sn = make_int2(cs.z, cs.w);
        fix_mad(h[0], x[0], vc[k], co);
        fix_mad(h[1], x[1], vc[6 * nk + k], co);
        fix_mad(h[2], x[2], vs[-k], sn);
        fix_mad(h[3], x[3], vs[6 * nk - k], sn);
      }
      if (mid > 0) {
        const int4 cs = CT[mid * (p + 1) + m];
        if (m & 1) {
          fix_mad(h[2], x[2], v0[half + mid], make_int2(cs.z, cs.w));
          fix_mad(h[3], x[3], v0[6 * nk + half + mid], make_int2(cs.z, cs.w));
        } else {
          fix_mad(h[0], x[0], v0[mid], make_int2(cs.x, cs.y));
          fix_mad(h[1], x[1], v0[6 * nk + mid], make_int2(cs.x, cs.y));
        }
      }
      const long long re0 = fix_half(h[0], x[0]), re1 = fix_half(h[1], x[1]), im0 = fix_half(h[2], x[2]),
                      im1 = fix_half(h[3], x[3]);
      int2* d = sd + (pair * 24 + 2 * c) * (p + 1) + m;
      d[0] = fix_split(re0 + re1);
      d[p + 1] = fix_split(im0 + im1);
      d[12 * (p + 1)] = fix_split(re0 - re1);
      d[13 * (p + 1)] = fix_split(im0 - im1);
    }
    __syncthreads();
    for (int it = threadIdx.x; it < ntri; it += blockDim.x) {
      const int n = tri_index_degree(it);
      const int m = it - n * (n + 1) / 2;
      int2 P[NP];
#pragma unroll
      for (int pair = 0; pair < NP; ++pair)
        P[pair] = pair < qn ? PT[(long long)(q0 + pair) * ntri + it] : make_int2(0, 0);
      const int2* d = sd + (((n - m) & 1) ? 12 : 0) * (p + 1) + m;
#pragma unroll
      for (int c = 0; c < 12; ++c) {
        long long h = 0, x = 0;
#pragma unroll
        for (int pair = 0; pair < NP; ++pair)
          if (pair < qn) fix_mad(h, x, d[(pair * 24 + c) * (p + 1)], P[pair]);
        sq[c * ntri + it] += (h + ((x + xrnd) >> kFixPart) + rnd) >> sf;
      }
    }
    __syncthreads();
  }
  double* o64 = Q64 + t * 12 * ntri;
  for (int i = threadIdx.x; i < 12 * ntri; i += blockDim.x) {
    const int it = i % ntri;
    const int n = tri_index_degree(it);
    const double v = bad ? __longlong_as_double(0x7ff8000000000000LL) : fix_decode(sq[i], es[i / ntri / 2] - 54 + lk + sf);
    o64[i] = (it == n * (n + 1) / 2 ? 1.0 : 2.0) * v;  // c_m
  }
}

// ---- dense form: set-up, S = R^T Q ----
// One block per (latitude row, degree n, chunk of kUnB longitudes).  With q_m = Q_re(n, m) for the real
// and -Q_im(n, m) for the imaginary parts of rho'_n^m, and rho' = (C Re g, S Im g), g = e^{i m phi_b} rho,
// the transposed rotation is s_re = C^T q_re, s_im = S^T q_im and the transposed phase
// (s_re cos + s_im sin, s_im cos - s_re sin).  The 2n+1 products per entry and coefficient run in fixed point
// on the integer pipe (fixed.cuh), on one scale per longitude and entry; two entries at a time share the reads of the
// Wigner block, and the leading dimensions of the staged blocks are odd, so that the strided reads of the
// transposed products hit every bank.  64 drops of p = 24, both kinds: 20 ms in FP64, now 11.
constexpr int kUnB = 8;

__global__ void __launch_bounds__(128) k_unrotate(const double* __restrict__ Q64, long long row0, int p,
                                                  const int2* __restrict__ wblk, long long wstride,
                                                  const double* __restrict__ ph, int ncp, double* __restrict__ S64,
                                                  float* __restrict__ S32) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int es[kUnB * 6];
  const int nb = 2 * p + 2, nbch = (nb + kUnB - 1) / kUnB;
  const int b0 = (int)(blockIdx.x % nbch) * kUnB;
  const long long row = row0 + blockIdx.x / nbch;  // latitude row of the group: drop * (p+1) + a
  const int a = (int)(row % (p + 1));
  const int n = p - (int)blockIdx.y;  // the longest blocks first
  const int nbh = min(kUnB, nb - b0);
  const int ntri = (p + 1) * (p + 2) / 2, t0 = n * (n + 1) / 2;
  const int ldC = (n + 1) | 1, ldS = n | 1;
  int2* sC = reinterpret_cast<int2*>(smem_raw);  // [m][m']
  int2* sS = sC + (n + 1) * ldC;
  int2* sq = sS + n * ldS;                        // [bb][e][re 0..n, im 1..n]
  const int2* blk = wblk + (long long)a * wstride + (long long)n * (n + 1) * (2 * n + 1) / 6 +
                    (long long)(n - 1) * n * (2 * n - 1) / 6;
  for (int i = threadIdx.x; i < (n + 1) * (n + 1); i += blockDim.x) sC[(i / (n + 1)) * ldC + i % (n + 1)] = blk[i];
  for (int i = threadIdx.x; i < n * n; i += blockDim.x) sS[(i / n) * ldS + i % n] = blk[(n + 1) * (n + 1) + i];
  const int w = 2 * n + 1;
  const double* Qr = Q64 + (row - row0) * nb * 12 * ntri + (long long)b0 * 12 * ntri + t0;
  // the 2 (n + 1) factors of a longitude and entry (at most 4 per lane, see self_dense_fits) and their scale, by a warp,
  // or by a half or a quarter of one where they are no more than that; three at a time, so that their loads overlap
  constexpr int kFly = 3;
  const int width = n < 4 ? 8 : n < 8 ? 16 : 32, lane = threadIdx.x & (width - 1), ngr = nbh * 6, step = 128 / width;
  for (int g0 = threadIdx.x / width; g0 - (int)(threadIdx.x / width) < ngr; g0 += step * kFly) {  // all lanes of a warp
    double v[kFly][4];
#pragma unroll
    for (int r = 0; r < kFly; ++r)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        v[r][u] = 0.0;
        if (32 * u >= 2 * (n + 1)) continue;
        const int g = g0 + step * r, k = lane + 32 * u, im = k > n, m = im ? k - (n + 1) : k;
        if (g < ngr && k < 2 * (n + 1)) v[r][u] = Qr[(2 * g + im) * ntri + m];
      }
#pragma unroll
    for (int r = 0; r < kFly; ++r) {
      const int g = g0 + step * r;
      int e = 0;
#pragma unroll
      for (int u = 0; u < 4; ++u) e = max(e, fix_magnitude(v[r][u]));
      if (width == 32) {
        e = __reduce_max_sync(0xffffffffu, e);
      } else {
        for (int o = width / 2; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
      }
      if (g >= ngr) continue;
      e = fix_exponent(e);
      if (lane == 0) es[g] = e;
      const bool bad = e == fix_bad;
      if (e == fix_none) e = 0;
      int2* q = sq + g * w;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (32 * u >= 2 * (n + 1)) break;
        const int k = lane + 32 * u;
        if (k <= n)
          q[k] = bad ? make_int2(0, 0) : fix_split(fix_encode(v[r][u], e));
        else if (k > n + 1 && k < 2 * (n + 1))  // the imaginary parts m = k - (n + 1) > 0, at n + m
          q[k - 1] = bad ? make_int2(0, 0) : fix_split(-fix_encode(v[r][u], e));
      }
    }
  }
  __syncthreads();
  // units: factors 2^(e-57), blocks 2^-56 (up to 2), sums 2^(e-55) with xb more bits: (n+1) 2^56 2^xb <= 2^62
  const int xb = 6 - ceil_log2(n + 1);
  for (int i = threadIdx.x; i < nbh * 3 * (n + 1); i += blockDim.x) {
    const int m = i % (n + 1), g = i / (n + 1) * 2;  // entries g and g + 1 of [bb][e]
    const int2* q = sq + g * w;
    const int2* c = sC + m * ldC;
    long long h[4] = {0, 0, 0, 0}, x[4] = {0, 0, 0, 0};  // real parts of the two entries, then imaginary
#pragma unroll 2
    for (int k = 0; k <= n; ++k) {
      const int2 cv = c[k];
      fix_mad(h[0], x[0], cv, q[k]);
      fix_mad(h[1], x[1], cv, q[w + k]);
    }
    if (m > 0) {
      const int2* sn = sS + (m - 1) * ldS - 1;
#pragma unroll 2
      for (int k = 1; k <= n; ++k) {
        const int2 sv = sn[k];
        fix_mad(h[2], x[2], sv, q[n + k]);
        fix_mad(h[3], x[3], sv, q[w + n + k]);
      }
    }
    const int bb = g / 6, en = g - bb * 6;
    const double co = ph[((long long)m * nb + b0 + bb) * 2], si = ph[((long long)m * nb + b0 + bb) * 2 + 1];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const double nan = __longlong_as_double(0x7ff8000000000000LL);
      const bool bad = es[g + u] == fix_bad;
      const int e = es[g + u] == fix_none ? 0 : es[g + u];
      const double re = bad ? nan : fix_decode(fix_sum(h[u], x[u], xb), e - 55 - xb);
      const double im = bad ? nan : fix_decode(fix_sum(h[2 + u], x[2 + u], xb), e - 55 - xb);
      const long long o = ((row * nb + b0 + bb) * 6 + en + u) * ncp + n * (n + 1);
      const double vr = m > 0 ? re * co + im * si : re;
      S64[o + m] = vr;
      S32[o + m] = (float)vr;
      if (m > 0) {
        const double vi = im * co - re * si;
        S64[o - m] = vi;
        S32[o - m] = (float)vi;
      } else if (n == p) {  // the padding of the row
        for (int r = p + 1; r < ncp - p * (p + 1); ++r) {
          S64[o + r] = 0.0;
          S32[o + r] = 0.0f;
        }
      }
    }
  }
}

// ---- dense form: apply ----
// vals[t] = sum_r S[t][r] rho[r] (symmetric 3x3 times 3-vector), one warp per target, the density of the
// drop in shared memory.  Every factor is read once, with 128-bit loads: bound by memory in FP32 and
// double-float (9 multiply-adds per 6 words), by the FP64 pipe in FP64.  Eight targets per block and
// warp for large batches (the density is staged once per block), one when the batch is small, so that
// every SM gets work.  Measured against rotating the density in every apply (36k flops per target, bound by
// the latency of the Wigner loads): FP32, p = 32 41 -> 17 us with the launch (57 MB), 192 drops of p = 24
// 1.93 -> 0.56 ms (6.5 TB/s); FP64, p = 16 41 -> 18 us, 16 drops of p = 16 and 24 0.67 -> 0.16 ms;
// double-float, 80 drops of p = 24 2.42 -> 0.59 ms.
constexpr int kSelfThreads = 256;

// acc += S v for the symmetric 3x3 matrix S with entries (xx, yy, zz, xy, xz, yz) in q
template <typename R>
__device__ inline void sym_mul_add(const R* q, const R* v, R* acc) {
  acc[0] = fmad(q[4], v[2], fmad(q[3], v[1], fmad(q[0], v[0], acc[0])));
  acc[1] = fmad(q[5], v[2], fmad(q[1], v[1], fmad(q[3], v[0], acc[1])));
  acc[2] = fmad(q[2], v[2], fmad(q[5], v[1], fmad(q[4], v[0], acc[2])));
}

// value v of 16 loaded bytes
template <typename R>
__device__ __forceinline__ R lane_of(const uint4& u, int v);
template <>
__device__ __forceinline__ float lane_of<float>(const uint4& u, int v) {
  return __uint_as_float(v == 0 ? u.x : v == 1 ? u.y : v == 2 ? u.z : u.w);
}
template <>
__device__ __forceinline__ double lane_of<double>(const uint4& u, int v) {
  return v == 0 ? __hiloint2double((int)u.y, (int)u.x) : __hiloint2double((int)u.w, (int)u.z);
}
template <>
__device__ __forceinline__ dff lane_of<dff>(const uint4& u, int v) {
  return v == 0 ? dff(__uint_as_float(u.x), __uint_as_float(u.y)) : dff(__uint_as_float(u.z), __uint_as_float(u.w));
}

// 16 bytes of a factor plane, read once: no L1 allocation
__device__ __forceinline__ uint4 load_factor(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// One launch covers every degree group (a batch over drops of uneven degree): the groups' arguments
// travel by value.
template <typename R, typename CT>
__global__ void __launch_bounds__(kSelfThreads, 2) k_self_dense(SelfGroups<R> G, int per_warp,
                                                                const CT* __restrict__ dens,
                                                                double* __restrict__ vals) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int V = 16 / sizeof(R);
  SelfGroup<R> A = G.g[0];
#pragma unroll
  for (int i = 1; i < kMaxSelfGroups; ++i)
    if (i < G.n && (long long)blockIdx.x >= G.g[i].begin) A = G.g[i];
  const int p = A.p;
  const int nc = (p + 1) * (p + 1), ncp = self_row(p), ng = 2 * nc;
  R* rho = reinterpret_cast<R*>(smem_raw);  // [3][ncp]
  const int tb = per_warp * (kSelfThreads / 32), tiles = (ng + tb - 1) / tb;
  const long long bid = (long long)blockIdx.x - A.begin;
  const long long ld = bid / tiles;
  const int t0 = (int)(bid - ld * tiles) * tb;
  for (int i = threadIdx.x; i < 3 * ncp; i += kSelfThreads) {
    const int c = i / ncp, r = i - c * ncp;
    rho[i] = r < nc ? R(dens[A.foff3[ld * 3 + c] + r]) : R(0);
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nv = ncp / V;
  for (int k = 0; k < per_warp; ++k) {
    const int t = t0 + k * (kSelfThreads / 32) + warp;
    if (t >= ng) break;
    const uint4* S = reinterpret_cast<const uint4*>(A.S + (ld * ng + t) * 6 * (long long)ncp);
    R acc[3] = {R(0), R(0), R(0)}, odd[3] = {R(0), R(0), R(0)};  // FP64: the sums of even and odd entries
#pragma unroll 2
    for (int i = lane; i < nv; i += 32) {
      uint4 s[6], f[3];
#pragma unroll
      for (int e = 0; e < 6; ++e) s[e] = load_factor(S + e * nv + i);
#pragma unroll
      for (int c = 0; c < 3; ++c) f[c] = reinterpret_cast<const uint4*>(rho + c * ncp)[i];
      R sum[3] = {R(0), R(0), R(0)};  // FP32: the 12 products first, then 9 such sums; as one sum of 108 it errs 1.5e-7, now 7.4e-8
#pragma unroll
      for (int v = 0; v < V; ++v) {
        R q[6], x[3];
#pragma unroll
        for (int e = 0; e < 6; ++e) q[e] = lane_of<R>(s[e], v);
#pragma unroll
        for (int c = 0; c < 3; ++c) x[c] = lane_of<R>(f[c], v);
        sym_mul_add<R>(q, x, sizeof(R) == 4 ? sum : (v & 1) && std::is_same<R, double>::value ? odd : acc);
      }
      if (sizeof(R) == 4)
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[c] = acc[c] + sum[c];
    }
    if (std::is_same<R, double>::value)
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[c] = acc[c] + odd[c];
    // the three sums over the lanes in six additions (fifteen one by one, 2 us of an FP64 apply of one drop of degree 16):
    // the halves of the warp exchange components first, so that lanes 0, 8 and 16 end up with one each
    const bool up = lane & 16, mid = lane & 8;
    const R a0 = (up ? acc[2] : acc[0]) + shfl_xor(up ? acc[0] : acc[2], 16);
    const R a1 = (up ? R(0) : acc[1]) + shfl_xor(up ? acc[1] : R(0), 16);
    R a = (mid ? a1 : a0) + shfl_xor(mid ? a0 : a1, 8);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) a = a + shfl_xor(a, off);
    if (lane % 8 == 0 && lane < 24) vals[A.val_off[ld] + t + (lane / 8) * (long long)ng] = A.wts[ld] * (double)a;
  }
}

// Latitudes per chunk of the direct kernel within a shared-memory budget.
template <typename R>
int pick_jc(int p, int pq, size_t budget, size_t* smem) {
  const size_t nc = (size_t)(p + 1) * (p + 1);
  const size_t fixed = sizeof(R) * 3 * nc;
  int jc = (int)((budget > 2 * fixed ? budget - fixed : 0) / (sizeof(R) * 6 * (p + 1)));
  jc = std::max(1, std::min(jc, pq + 1));
  *smem = fixed + sizeof(R) * std::max(3 * nc, (size_t)6 * (p + 1) * jc);
  return jc;
}

// out[i] = the double-float split of in[i]
__global__ void k_split_dff(const double* __restrict__ in, dff* __restrict__ out, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = dff(in[i]);
}

}  // namespace

int launch_split_dff(const double* in, dff* out, long long n, cudaStream_t s) {
  if (n == 0) return BIE_OK;
  k_split_dff<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(in, out, n);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

template <typename R>
int launch_self_direct(int kind, const double* dens, const long long* foff3, long long ndrop, int p, int pq,
                       const R* wblk, long long wstride, const R* ph, const R* T0, const R* cs, const R* cache,
                       const double* wts, const long long* val_off, double* vals, size_t smem_budget,
                       cudaStream_t s) {
  const int ng = (p + 1) * (2 * p + 2);
  const long long nt = ndrop * ng;
  if (nt == 0) return BIE_OK;
  if (nt > 0x7fffffffLL) return BIE_EINVAL;
  size_t smem;
  const int jc = pick_jc<R>(p, pq, smem_budget, &smem);
  auto kern = kind == 0 ? k_self_direct<R, 0> : k_self_direct<R, 1>;
  BIE_CUDA_TRY(allow_smem(kern, smem));
  kern<<<(unsigned)nt, 256, smem, s>>>(dens, foff3, p, pq, wblk, wstride, ph, T0, cs, cache, ng, wts, val_off, vals,
                                       jc);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

// dynamic shared memory of k_kernel_proj with np latitude pairs a pass
static size_t kernel_proj_smem(int p, int pq, int np) {
  return sizeof(double) * (24 * (size_t)np * (pq + p + 2) + 6 * (size_t)(p + 1) * (p + 2));
}

// Degrees up to 62 at pq = p and 59 at pq = 2p + 1.  Above, neither the coefficients of one target (rotgeo.cu) nor twice
// its projected factors fit a block, and the direct form serves as it always has.
bool self_dense_fits(int p, int pq) { return 8 * (36 * (size_t)(pq + p + 2) + 6 * (size_t)(p + 1) * (p + 2)) <= 227 * 1024; }

int launch_kernel_proj(int kind, double* cache, long long ntarget, int p, int pq, const int4* CT, const int2* PT,
                       double* Q64, cudaStream_t s) {
  if (ntarget == 0) return BIE_OK;
  if (ntarget > 0x7fffffffLL) return BIE_EINVAL;
  const bool two = kernel_proj_smem(p, pq, 2) <= kMaxSmem;
  const size_t smem = kernel_proj_smem(p, pq, two ? 2 : 1);
  if (smem > kMaxSmem) {
    set_error("degree too large for the dense self form (shared memory)");
    return BIE_ENOTSUP;
  }
  auto kern = kind == 0 ? (two ? k_kernel_proj<0, 2> : k_kernel_proj<0, 1>) : (two ? k_kernel_proj<1, 2> : k_kernel_proj<1, 1>);
  BIE_CUDA_TRY(allow_smem(kern, smem));
  kern<<<(unsigned)ntarget, 256, smem, s>>>(cache, pq, p, CT, PT, Q64);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_unrotate(const double* Q64, long long row0, long long nrow, int p, const int2* wblk, long long wstride,
                    const double* ph, double* S64, float* S32, cudaStream_t s) {
  if (nrow == 0) return BIE_OK;
  const int nbch = (2 * p + 2 + kUnB - 1) / kUnB;
  if (nrow * nbch > 0x7fffffffLL) return BIE_EINVAL;
  const size_t smem = sizeof(double) * ((size_t)(p + 1) * (p + 2) + (size_t)p * (p + 1) + (size_t)kUnB * 6 * (2 * p + 1));
  BIE_CUDA_TRY(allow_smem(k_unrotate, smem));
  k_unrotate<<<dim3((unsigned)(nrow * nbch), p + 1), 128, smem, s>>>(Q64, row0, p, wblk, wstride, ph, self_row(p), S64,
                                                                     S32);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

template <typename R, typename CT>
int launch_self_dense(std::vector<SelfGroup<R>> groups, const CT* dens, double* vals, int sms, cudaStream_t s) {
  std::sort(groups.begin(), groups.end(), [](const SelfGroup<R>& x, const SelfGroup<R>& y) { return x.p > y.p; });
  long long targets = 0;
  for (const auto& g : groups) targets += g.ndrop * 2 * (long long)(g.p + 1) * (g.p + 1);
  // one target per warp until every SM has about eight blocks, then up to eight
  const int nw = kSelfThreads / 32;
  const int per_warp = (int)std::max(1LL, std::min<long long>(8, targets / (8LL * nw * sms)));
  for (size_t g0 = 0; g0 < groups.size(); g0 += kMaxSelfGroups) {
    SelfGroups<R> G{};
    G.n = (int)std::min<size_t>(kMaxSelfGroups, groups.size() - g0);
    long long nblk = 0;
    size_t smem = 0;
    for (int i = 0; i < G.n; ++i) {
      G.g[i] = groups[g0 + i];
      const int p = G.g[i].p, ng = 2 * (p + 1) * (p + 1);
      G.g[i].begin = nblk;
      nblk += G.g[i].ndrop * ((ng + per_warp * nw - 1) / (per_warp * nw));
      smem = std::max(smem, sizeof(R) * 3 * (size_t)self_row(p));
      if (G.g[i].ndrop * (long long)ng > 0x7fffffffLL) return BIE_EINVAL;
    }
    if (nblk == 0) continue;
    if (nblk > 0x7fffffffLL) return BIE_EINVAL;
    auto kern = k_self_dense<R, CT>;
    BIE_CUDA_TRY(allow_smem(kern, smem));
    kern<<<(unsigned)nblk, kSelfThreads, smem, s>>>(G, per_warp, dens, vals);
    count_launch();
    BIE_CUDA_TRY(cudaGetLastError());
  }
  return BIE_OK;
}

template int launch_self_direct<double>(int, const double*, const long long*, long long, int, int, const double*,
                                        long long, const double*, const double*, const double*, const double*,
                                        const double*, const long long*, double*, size_t, cudaStream_t);
template int launch_self_direct<float>(int, const double*, const long long*, long long, int, int, const float*,
                                       long long, const float*, const float*, const float*, const float*,
                                       const double*, const long long*, double*, size_t, cudaStream_t);
template int launch_self_dense<double, double>(std::vector<SelfGroup<double>>, const double*, double*, int, cudaStream_t);
template int launch_self_dense<float, double>(std::vector<SelfGroup<float>>, const double*, double*, int, cudaStream_t);
template int launch_self_dense<dff, double>(std::vector<SelfGroup<dff>>, const double*, double*, int, cudaStream_t);

}  // namespace bie

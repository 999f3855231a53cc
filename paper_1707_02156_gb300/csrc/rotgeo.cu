// Rotated-grid cache of the singular self rule (Sec. 2.2, App. B) in one kernel, one block per target: the shape
// coefficients rotated so that the target sits at the pole, x' and its parameter derivatives on the rotated
// grid, and from them (x0 - x', w n', w).
//
// Bound before by the FP64 pipe (0.28M operations per target at p = pq = 24: rotation, Legendre sums, phi
// sums), through 0.2 MB of temporaries per target in three kernels.  The sums run in fixed point on the integer
// pipe here (fixed.cuh), each stage on a scale taken from its largest operand, and nothing but the cache
// leaves the block; the FP64 pipe keeps the phases and the pointwise geometry.
//   * The three components have scales of their own throughout: a drop that is thin along an axis keeps the
//     precision of its thin component.
//   * A rotation mixes the coefficients of one degree only, so each degree has its own scale there: the small
//     high degrees of a smooth drop keep relative precision until the Legendre sums bring all to one scale.
//   * The degree-0 coefficient, the drop's position, is left out of the sums and taken off the target instead:
//     only x0 - x' is needed, and the scale is then the drop's own size.
//   * theta derivatives grow like n and phi derivatives like m; the tables of the theta derivative carry a
//     power of two per degree and those of the phi derivative one per order, moved to the coefficients, so
//     that the low orders keep their bits.
//   * Rotated coefficients are stored by (n - m, m), so that neighbouring threads, on neighbouring orders, read
//     neighbouring entries of them and of the Legendre tables; a thread takes the orders a and p - a, which
//     makes all sums equally long.
// 64 drops of degree 24: 59 ms, 50 of them in the synthesis; now 24.  Neither pipe is full any more (FP64 28 %,
// issue slots 47 % busy): the phases of a pass wait for one another, with three blocks per SM.  Blocks of as
// many threads as the phases have items (320, 480) are slower (26, 28 ms).
#include <cuda_runtime.h>

#include <algorithm>

#include "device.cuh"
#include "fixed.cuh"
#include "internal.cuh"

namespace bie {
namespace {

constexpr int kGeoThreads = 256, kMaxDeg = 64;

__device__ __forceinline__ int bit_length(long long v) { return 64 - __clzll(v < 0 ? -v : v); }
// v 2^s, rounded, for s <= 57
__device__ __forceinline__ long long shifted(long long v, int s) {
  if (s >= 0) return v << s;
  return s < -62 ? 0 : (v + (1LL << (-s - 1))) >> -s;
}
constexpr int kHeadBits = 30;
// (v + f 2^-30) 2^s, for s <= 57
__device__ __forceinline__ long long shifted(long long v, unsigned f, int s) {
  if (s <= 0) return shifted(v, s);
  return (v << s) + (s <= kHeadBits ? (long long)((f >> (kHeadBits - s))) : (long long)f << (s - kHeadBits));
}
// first entry of the coefficients with n - m = d
__host__ __device__ inline int diag_row(int p, int d) { return d * (p + 1) - d * (d - 1) / 2; }

__device__ __forceinline__ void block_max(int v, int* out) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) atomicMax(out, v);
}

template <int JP>
__global__ void __launch_bounds__(kGeoThreads, 3) k_rotgeo_fix(RotGeo A, double* __restrict__ cache) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // exponents per component: of the largest coefficient, per table, and per kind in a pass; en: by degree
  __shared__ int emax, bits[2][3], kbits[3][3], en[3][kMaxDeg + 1];
  const int p = A.p, pq = A.pq, nc = (p + 1) * (p + 1), ntri = (p + 1) * (p + 2) / 2;
  const int nj = pq + 1, nk = 2 * pq + 2, half = pq + 1, np = (nj + 1) / 2, k4n = half / 2 + 1, nb = 2 * p + 2;
  const long long nq = (long long)nj * nk, ng = (long long)(p + 1) * nb;
  const long long t = blockIdx.x, ld = t / A.nt, tl = A.tl0 + (t - ld * A.nt);
  const int a = (int)(tl / nb), b = (int)(tl - (long long)a * nb);
  long long* rc = reinterpret_cast<long long*>(smem_raw);  // [comp][re, im][tri]: rotated coefficients, then split (T0)
  int2* r0 = reinterpret_cast<int2*>(rc);
  double* g = reinterpret_cast<double*>(rc + 6 * ntri);    // [comp][(p+1)^2]: phase-shifted coefficients, in doubles,
  int2* gi = reinterpret_cast<int2*>(g);                   // then split; then the rotated ones split for T1 in its place
  int2* r1 = gi;
  long long* h = reinterpret_cast<long long*>(rc + 12 * ntri);  // [kind][comp][row][m][2], then split
  int2* hi = reinterpret_cast<int2*>(h);
  double* X = reinterpret_cast<double*>(h + 9 * 2 * JP * (p + 1) * 2);  // [kind][comp][row][nk]
  unsigned* hf = reinterpret_cast<unsigned*>(X);                        // before: the next 30 bits of h
  if (threadIdx.x == 0) emax = 0;
  if (threadIdx.x < 6) (&bits[0][0])[threadIdx.x] = fix_none;
  for (int i = threadIdx.x; i < 3 * (kMaxDeg + 1); i += kGeoThreads) (&en[0][0])[i] = 0;
  __syncthreads();
  {  // g = e^{i m phi_b} x_n^m, n >= 1
    int e = 0;
    for (int i = threadIdx.x; i < 3 * nc; i += kGeoThreads) {
      const int c = i / nc, r = i - c * nc, n = degree_of(r), m = r - n * (n + 1);
      if (m < 0) continue;  // the owner of Re writes both parts
      const double* f = A.coef + A.foff3[ld * 3 + c];
      double gr = 0.0, gm = 0.0;
      if (n > 0) {
        const double fr = f[n * (n + 1) + m], fi = m > 0 ? f[n * (n + 1) - m] : 0.0;
        const double co = A.ph[((long long)m * nb + b) * 2], si = A.ph[((long long)m * nb + b) * 2 + 1];
        gr = fr * co - fi * si;
        gm = fr * si + fi * co;
      }
      g[c * nc + n * (n + 1) + m] = gr;
      if (m > 0) g[c * nc + n * (n + 1) - m] = gm;
      const int el = max(fix_magnitude(gr), fix_magnitude(gm));
      if (el) atomicMax(&en[c][n], el);
      e = max(e, el);
    }
    block_max(e, &emax);
  }
  __syncthreads();
  double* out = cache + t * 7 * nq;
  if (fix_exponent(emax) == fix_bad) {  // a NaN or an infinity among the coefficients
    for (long long i = threadIdx.x; i < 7 * nq; i += kGeoThreads) out[i] = __longlong_as_double(0x7ff8000000000000LL);
    return;
  }
  for (int i = threadIdx.x; i < 3 * (kMaxDeg + 1); i += kGeoThreads) (&en[0][0])[i] = fix_exponent((&en[0][0])[i]);
  __syncthreads();
  for (int i = threadIdx.x; i < 3 * nc; i += kGeoThreads)
    gi[i] = fix_split(fix_encode(g[i], en[i / nc][degree_of(i % nc)]));
  __syncthreads();
  // rotation: sums of at most p + 1 <= 64 products of 2^57 and 2^57, in units of 2^(en - 55 - xb)
  const int xb = 6 - ceil_log2(p + 1);
  {
    const int2* blk = A.wblk + (long long)a * A.wstride;
    int m0[3] = {fix_none, fix_none, fix_none}, m1[3] = {fix_none, fix_none, fix_none};
    for (int r = threadIdx.x; r < nc; r += kGeoThreads) {
      const int n = degree_of(r), o = r - n * n;
      if (n == 0) {
        for (int c = 0; c < 3; ++c) rc[2 * c * ntri] = 0;
        continue;
      }
      const bool re = o <= n;
      const int mo = re ? o : o - n, len = re ? n + 1 : n;
      const int2* C = blk + (long long)n * (n + 1) * (2 * n + 1) / 6 + (long long)(n - 1) * n * (2 * n - 1) / 6 +
                      (re ? o : (n + 1) * (n + 1) + mo - 1);
      const int2* gc = gi + n * (n + 1);
      long long hs[3] = {0, 0, 0}, xs[3] = {0, 0, 0};
#pragma unroll 2
      for (int k = 0; k < len; ++k) {
        const int2 cv = C[(long long)k * len];
        const int at = re ? k : -(k + 1);
        fix_mad(hs[0], xs[0], cv, gc[at]);
        fix_mad(hs[1], xs[1], cv, gc[nc + at]);
        fix_mad(hs[2], xs[2], cv, gc[2 * nc + at]);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const long long v = fix_sum(hs[c], xs[c], xb);
        rc[(2 * c + (re ? 0 : 1)) * ntri + diag_row(p, n - mo) + mo] = v;
        if (v != 0) {
          const int bl = bit_length(v) + en[c][n];
          m0[c] = max(m0[c], bl);
          m1[c] = max(m1[c], bl + A.t1[n]);
        }
      }
    }
    for (int i = threadIdx.x; i < 3 * (p + 1); i += kGeoThreads)  // imaginary parts of order 0
      rc[(2 * (i / (p + 1)) + 1) * ntri + diag_row(p, i % (p + 1))] = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      block_max(m0[c], &bits[0][c]);
      block_max(m1[c], &bits[1][c]);
    }
  }
  __syncthreads();
  auto bits_of = [&](int table, int c) { return bits[table][c] == fix_none ? 0 : bits[table][c]; };
  for (int i = threadIdx.x; i < 6 * ntri; i += kGeoThreads) {
    // (n - m, m) of the entry: the diagonal rows are p + 1 - d long
    int q = i % ntri, d = (int)((2 * p + 3 - sqrtf((float)((2 * p + 3) * (2 * p + 3) - 8 * q))) * 0.5f);
    while (d > 0 && diag_row(p, d) > q) --d;
    while (diag_row(p, d + 1) <= q && d < p) ++d;
    const int n = d + (q - diag_row(p, d)), c = i / (2 * ntri);
    const long long v = rc[i];
    r1[i] = fix_split(shifted(v, 57 - bits_of(1, c) + en[c][n] + A.t1[n]));
    r0[i] = fix_split(shifted(v, 57 - bits_of(0, c) + en[c][n]));
  }
  const double* x0p = A.rec_std + A.rec_off[ld] + tl;
  double x0[3];
#pragma unroll
  for (int c = 0; c < 3; ++c)
    x0[c] = x0p[c * ng] - A.coef[A.foff3[ld * 3 + c]] * 0.28209479177387814347;  // less x_0^0 Y_0^0 = the centre
  const int mh = p / 2 + 1, ext = 5 - ceil_log2(mh);  // at most mh products of one parity
  for (int q0 = 0; q0 < np; q0 += JP) {
    const int qn = min(JP, np - q0);
    if (threadIdx.x < 9) (&kbits[0][0])[threadIdx.x] = fix_none;
    __syncthreads();
    {  // Legendre sums over even and odd n - m, the orders a and p - a, both latitudes (tables 2^-56; at most 32
       // products of 2^57 and 2^58), in units of 2^59 of their products, so that a sum of both parities stays below 2^63;
       // most are far below that bound, so the 30 bits that follow are kept until the common scale is known
      for (int i = threadIdx.x; i < 6 * qn * mh; i += kGeoThreads) {
        const int am = i % mh, s = i / mh, c = s % 3, tab = s / 3 % 2, q = s / 6;
        const int2* R = (tab ? r1 : r0) + 2 * c * ntri;
        const int2* T = (tab ? A.LT1 : A.LT0) + (long long)(q0 + q) * ntri;
        int bk = fix_none, bp = fix_none;  // bits of the values, and of the phi derivative's
        for (int half_m = 0; half_m < 2; ++half_m) {
          const int m = half_m ? p - am : am;
          if (half_m && m == am) break;
          long long hs[4] = {0, 0, 0, 0}, xs[4] = {0, 0, 0, 0};  // even re, im, odd re, im
          int d = 0, at = m;
          for (; d + 1 <= p - m; d += 2) {
            const int bt = at + p + 1 - d;
            const int2 v = T[at], w = T[bt];
            fix_mad(hs[0], xs[0], R[at], v);
            fix_mad(hs[1], xs[1], R[ntri + at], v);
            fix_mad(hs[2], xs[2], R[bt], w);
            fix_mad(hs[3], xs[3], R[ntri + bt], w);
            at = bt + p - d;
          }
          if (d <= p - m) {
            const int2 v = T[at];
            fix_mad(hs[0], xs[0], R[at], v);
            fix_mad(hs[1], xs[1], R[ntri + at], v);
          }
          __int128 S[4];  // twice for m > 0, in units of 2^29 of the products
#pragma unroll
          for (int k = 0; k < 4; ++k) S[k] = (((__int128)hs[k] << kFixPart) + xs[k]) << (m > 0);
          const int tm = 31 - __clz(max(m, 1));  // 2^tm <= m
#pragma unroll
          for (int side = 0; side < 2; ++side) {
            const __int128 vr = side == 0 ? S[0] + S[2] : tab ? S[2] - S[0] : S[0] - S[2];
            const __int128 vi = side == 0 ? S[1] + S[3] : tab ? S[3] - S[1] : S[1] - S[3];
            const long long re = (long long)(vr >> kHeadBits), im = (long long)(vi >> kHeadBits);
            const int at2 = (((tab * 3 + c) * 2 * JP + 2 * q + side) * (p + 1) + m) * 2;
            h[at2] = re;
            h[at2 + 1] = im;
            hf[at2] = (unsigned)vr & ((1u << kHeadBits) - 1);
            hf[at2 + 1] = (unsigned)vi & ((1u << kHeadBits) - 1);
            const int bl = max(re != 0 ? bit_length(re) : fix_none, im != 0 ? bit_length(im) : fix_none);
            bk = max(bk, bl);
            if (m > 0) bp = max(bp, bl + tm);
          }
        }
        atomicMax(&kbits[tab][c], bk);  // one item a thread or fewer
        if (!tab) atomicMax(&kbits[2][c], bp);
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 6 * JP * (p + 1); i += kGeoThreads) {  // split in place; kind 2 is i m times kind 0
      const int m = i % (p + 1), c = i / (2 * JP * (p + 1));
      const int tm = 31 - __clz(max(m, 1)), kb0 = max(kbits[0][c], 0), kb1 = max(kbits[1][c], 0), kb2 = max(kbits[2][c], 0);
      long long *o0 = h + 2LL * i, *o1 = h + 2LL * (6 * JP * (p + 1) + i);
      const long long re = o0[0], im = o0[1], re1 = o1[0], im1 = o1[1];
      const unsigned fr = hf[2 * i], fi = hf[2 * i + 1];
      const unsigned fr1 = hf[2 * (6 * JP * (p + 1) + i)], fi1 = hf[2 * (6 * JP * (p + 1) + i) + 1];
      int2 *w0 = hi + 2LL * i, *w1 = hi + 2LL * (6 * JP * (p + 1) + i), *w2 = hi + 2LL * (12 * JP * (p + 1) + i);
      w0[0] = fix_split(shifted(re, fr, 57 - kb0));
      w0[1] = fix_split(shifted(im, fi, 57 - kb0));
      w1[0] = fix_split(shifted(re1, fr1, 57 - kb1));
      w1[1] = fix_split(shifted(im1, fi1, 57 - kb1));
      w2[0] = m > 0 ? fix_split(-shifted(im, fi, 57 - kb2 + tm)) : make_int2(0, 0);
      w2[1] = m > 0 ? fix_split(shifted(re, fr, 57 - kb2 + tm)) : make_int2(0, 0);
    }
    __syncthreads();
    // phi sums over even and odd orders' cosine and sine parts for a longitude quadruple of both latitudes
    for (int i = threadIdx.x; i < 9 * qn * k4n; i += kGeoThreads) {
      const int k = i % k4n, s = i / k4n, f = s % 9, q = s / 9, kind = f / 3;  // f = kind * 3 + comp
      const int4* E = kind == 2 ? A.CP : A.CM;  // [m][k]
      const int4* v0 = reinterpret_cast<const int4*>(hi + 2LL * ((long long)f * 2 * JP + 2 * q) * (p + 1));
      const int4* v1 = v0 + (p + 1);
      long long hs[8] = {0, 0, 0, 0, 0, 0, 0, 0}, xs[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // per row: ce, co, se, so
      auto add = [&](int m, int odd) {
        const int4 cs = E[m * k4n + k], a0 = v0[m], a1 = v1[m];
        const int2 co = make_int2(cs.x, cs.y), sn = make_int2(cs.z, cs.w);
        fix_mad(hs[odd], xs[odd], make_int2(a0.x, a0.y), co);
        fix_mad(hs[2 + odd], xs[2 + odd], make_int2(a0.z, a0.w), sn);
        fix_mad(hs[4 + odd], xs[4 + odd], make_int2(a1.x, a1.y), co);
        fix_mad(hs[6 + odd], xs[6 + odd], make_int2(a1.z, a1.w), sn);
      };
      int m = 0;
      for (; m + 1 <= p; m += 2) {
        add(m, 0);
        add(m + 1, 1);
      }
      if (m <= p) add(m, 0);
      // units: rotated coefficients 2^(-55 - xb), split 2^(bits - 57) of that, Legendre sums 2^(59 - 56) of that, split
      // 2^(kbits - 57), tables 2^-56 (2^-55 for kind 2), sums 2^(58 - ext) of their products, which leaves room for four
      // of them
      const int unit = bits_of(kind == 1, f % 3) - 55 - xb - 57 + 3 + max(kbits[kind][f % 3], 0) - 57 -
                       (kind == 2 ? 55 : 56) + 58 - ext;
      const bool rot = k > 0, mir = 2 * k < half;
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const long long ce = fix_sum(hs[4 * side], xs[4 * side], ext), co = fix_sum(hs[4 * side + 1], xs[4 * side + 1], ext),
                        se = fix_sum(hs[4 * side + 2], xs[4 * side + 2], ext),
                        so = fix_sum(hs[4 * side + 3], xs[4 * side + 3], ext);
        double* d = X + ((long long)f * 2 * JP + 2 * q + side) * nk;
        d[k] = fix_decode(ce + co - se - so, unit);
        if (mir) d[half + k] = fix_decode(ce - co - se + so, unit);
        if (rot) d[2 * half - k] = fix_decode(ce + co + se + so, unit);
        if (rot && mir) d[half - k] = fix_decode(ce - co + se - so, unit);
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * qn * nk; i += kGeoThreads) {
      const int row = i / nk, k = i - row * nk, q = q0 + row / 2;
      if ((row & 1) && 2 * q == pq) continue;  // the middle latitude has no mirror
      const int j = row & 1 ? pq - q : q;
      const long long fs = 2LL * JP * nk;  // from one field to the next
      const double* v = X + (long long)row * nk + k;
      const double t0 = v[3 * fs], t1 = v[4 * fs], t2 = v[5 * fs], p0 = v[6 * fs], p1 = v[7 * fs], p2 = v[8 * fs];
      const double c0 = t1 * p2 - t2 * p1, c1 = t2 * p0 - t0 * p2, c2 = t0 * p1 - t1 * p0;
      const double W2 = c0 * c0 + c1 * c1 + c2 * c2, ws = A.wsq[j];
      double* o = out + (long long)j * nk + k;
      o[0] = x0[0] - v[0];
      o[nq] = x0[1] - v[fs];
      o[2 * nq] = x0[2] - v[2 * fs];
      o[3 * nq] = ws * c0;
      o[4 * nq] = ws * c1;
      o[5 * nq] = ws * c2;
      o[6 * nq] = ws * (W2 * rsqrt_<double>(W2));
    }
    __syncthreads();
  }
}

size_t rotgeo_smem(int p, int pq, int jp) {
  return 8 * (12 * (size_t)(p + 1) * (p + 2) / 2 + 9 * 2 * (size_t)jp * (2 * (p + 1) + 2 * pq + 2));
}

}  // namespace

// Above degree 62 at pq = p the split coefficients don't fit a block's shared memory; the three kernels through memory
// that such a set-up then takes are the form it replaced (twice its time at degree 24).
bool rotgeo_fix_fits(int p, int pq) { return rotgeo_smem(p, pq, 1) <= 225 * 1024; }

int launch_rotgeo_fix(const RotGeo& A, long long ndrop, double* cache, cudaStream_t s) {
  const long long n = ndrop * A.nt;
  if (n == 0) return BIE_OK;
  if (n > 0x7fffffffLL) return BIE_EINVAL;
  // two latitude pairs per pass where two blocks still fit an SM
  const bool two = rotgeo_smem(A.p, A.pq, 2) <= 110 * 1024;
  const size_t smem = rotgeo_smem(A.p, A.pq, two ? 2 : 1);
  auto kern = two ? k_rotgeo_fix<2> : k_rotgeo_fix<1>;
  BIE_CUDA_TRY(allow_smem(kern, smem));
  kern<<<(unsigned)n, kGeoThreads, smem, s>>>(A, cache);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

}  // namespace bie

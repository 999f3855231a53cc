// Near-singular (Omega_2) step of Sec. 2.3: closest point on the source surface by damped Newton
// (Eqs. f_phi, f_theta, newton_ite and the Levenberg-Marquardt footnote), check points along the
// line through the closest point and the target, their regular-rule values, the on-surface value
// from the SH expansion of the source drop's self-interaction values, and 1-D Lagrange interpolation
// in the distance.
#include <cuda_runtime.h>

#include "device.cuh"
#include "internal.cuh"
#include "near.h"

namespace bie {
namespace {

constexpr double kPiD = 3.14159265358979323846;

// Coefficients of the normalised Legendre recursion of App. A at (n, m):
// P_n^m = rec_a (cos(theta) P_{n-1}^m - rec_b P_{n-2}^m) for n >= m + 2, and the factor rec_c of the
// derivative identity dP_n^m = rec_c P_n^{m+1} + m cot(theta) P_n^m.
__device__ __forceinline__ double rec_a(int n, int m) {
  return sqrt((4.0 * n * n - 1.0) / ((double)n * n - (double)m * m));
}
__device__ __forceinline__ double rec_b(int n, int m) {
  return sqrt(((n - 1.0) * (n - 1.0) - (double)m * m) / (4.0 * (n - 1.0) * (n - 1.0) - 1.0));
}
__device__ __forceinline__ double rec_c(int n, int m) { return sqrt((double)(n - m) * (n + m + 1.0)); }
__device__ __forceinline__ long long tri(int n, int m) { return (long long)n * (n + 1) / 2 + m; }

// tab[3 tri(n, m) + k] = rec_a, rec_b (0 for n < m + 2), rec_c, for 0 <= m <= n <= P; then the P + 2
// constants of P~_m^m(theta) = C_m sin^m(theta), C_0 = sqrt(1/4pi), C_(m+1) = -sqrt(1 + 1/(2m+2)) C_m
__global__ void k_rec_table(int P, double* __restrict__ tab) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t == 0) {
    double c = sqrt(1.0 / (4.0 * kPiD));
    for (int m = 0; m <= P + 1; ++m) {
      tab[3 * tri(P + 1, 0) + m] = c;
      c *= -sqrt(1.0 + 1.0 / (2.0 * (m + 1)));
    }
  }
  if (t >= tri(P + 1, 0)) return;
  int n = (int)((sqrt(8.0 * t + 1.0) - 1.0) / 2.0);
  while (tri(n + 1, 0) <= t) ++n;
  while (tri(n, 0) > t) --n;
  const int m = (int)(t - tri(n, 0));
  tab[3 * t] = n >= m + 2 ? rec_a(n, m) : 0.0;
  tab[3 * t + 1] = n >= m + 2 ? rec_b(n, m) : 0.0;
  tab[3 * t + 2] = rec_c(n, m);
}

// Value and first/second parameter derivatives of three real SH series (coefficients c[3][(p+1)^2])
// at (theta, phi), with the Legendre recursion of App. A and the derivative identities
// dP = alpha P^{m+1} + m cot(theta) P^m and the Legendre equation (theta away from the poles).
// One warp per point: lane l runs the recursions of the orders l, l + 32, ..., so a point takes p + 1
// serial steps, not (p+1)(p+2)/2; the xor sums leave the same values in every lane.  Closest points of 2051
// points off drops of degree 24, with their rotations: 27.0 -> 3.8 ms.
// tab: k_rec_table's for degrees up to tabP.  out[k][c], k: 0 f, 1 f_t, 2 f_p, 3 f_tt, 4 f_tp, 5 f_pp; without
// FULL only the value, by the same operations.
template <bool FULL>
__device__ void sh_eval_d2(const double* __restrict__ c, long long cstride, int p, double th, double ph,
                           const double* __restrict__ tab, int tabP, double (*out)[3]) {
  constexpr int NK = FULL ? 6 : 1;
  for (int k = 0; k < NK; ++k)
    for (int q = 0; q < 3; ++q) out[k][q] = 0;
  double st, ct;
  sincos(th, &st, &ct);
  const double cot = ct / st, s2 = st * st;
  const double* diag = tab + 3 * tri(tabP + 1, 0);
  for (int m = threadIdx.x & 31; m <= p; m += 32) {
    double pw = 1.0;
    for (int k = 0; k < m; ++k) pw *= st;
    const double dm = diag[m] * pw;  // P~_m^m
    const double dm1 = m + 1 <= p ? diag[m + 1] * (pw * st) : 0.0;
    double pm2 = 0, pm1 = 0, qm2 = 0, qm1 = 0;
    double h0r[3] = {0, 0, 0}, h0i[3] = {0, 0, 0}, h1r[3] = {0, 0, 0}, h1i[3] = {0, 0, 0}, h2r[3] = {0, 0, 0},
           h2i[3] = {0, 0, 0};
    const double f1 = sqrt(2.0 * m + 3.0), f2 = sqrt(2.0 * m + 5.0);
    const int m1 = m + 1;
    for (int n = m; n <= p; ++n) {
      double P;
      if (n == m)
        P = dm;
      else if (n == m1)
        P = f1 * ct * dm;
      else
        P = tab[3 * tri(n, m)] * (ct * pm1 - tab[3 * tri(n, m) + 1] * pm2);
      if (!FULL) {
        pm2 = pm1;
        pm1 = P;
        for (int q = 0; q < 3; ++q) {
          const double re = c[q * cstride + n * (n + 1) + m];
          const double im = m > 0 ? c[q * cstride + n * (n + 1) - m] : 0.0;
          h0r[q] += re * P;
          h0i[q] += im * P;
        }
        continue;
      }
      double Q = 0;  // P~_n^{m+1}
      if (n == m1)
        Q = dm1;
      else if (n == m1 + 1)
        Q = f2 * ct * dm1;
      else if (n > m1 + 1)
        Q = tab[3 * tri(n, m1)] * (ct * qm1 - tab[3 * tri(n, m1) + 1] * qm2);
      pm2 = pm1;
      pm1 = P;
      if (n >= m1) {
        qm2 = qm1;
        qm1 = Q;
      }
      const double dP = tab[3 * tri(n, m) + 2] * Q + m * cot * P;
      const double d2P = -cot * dP + ((double)m * m / s2 - n * (n + 1.0)) * P;
      for (int q = 0; q < 3; ++q) {
        const double re = c[q * cstride + n * (n + 1) + m];
        const double im = m > 0 ? c[q * cstride + n * (n + 1) - m] : 0.0;
        h0r[q] += re * P;
        h0i[q] += im * P;
        h1r[q] += re * dP;
        h1i[q] += im * dP;
        h2r[q] += re * d2P;
        h2i[q] += im * d2P;
      }
    }
    double sm, cm;
    sincos(m * ph, &sm, &cm);
    const double fac = m == 0 ? 1.0 : 2.0;
    for (int q = 0; q < 3; ++q) {
      const double v0 = h0r[q] * cm - h0i[q] * sm, w0 = h0r[q] * sm + h0i[q] * cm;  // Re, Im of h0 e^{i m phi}
      const double v1 = h1r[q] * cm - h1i[q] * sm, w1 = h1r[q] * sm + h1i[q] * cm;
      const double v2 = h2r[q] * cm - h2i[q] * sm;
      out[0][q] += fac * v0;
      if (!FULL) continue;
      out[1][q] += fac * v1;
      out[3][q] += fac * v2;
      out[2][q] += fac * (-m * w0);  // Re(i m h e^{i m phi})
      out[4][q] += fac * (-m * w1);
      out[5][q] += fac * (-(double)m * m * v0);
    }
  }
  for (int k = 0; k < NK; ++k)
    for (int q = 0; q < 3; ++q)
      for (int o = 16; o > 0; o >>= 1) out[k][q] += __shfl_xor_sync(0xffffffffu, out[k][q], o);
}

// Value of three real SH series at (theta, phi) (any theta, poles included), by one warp: lane l runs the
// orders l, l + 32, ...; every lane returns the value.
__device__ void sh_eval3(const double* __restrict__ c, long long cstride, int p, double th, double ph, double* out) {
  out[0] = out[1] = out[2] = 0;
  double st, ct;
  sincos(th, &st, &ct);
  for (int m = threadIdx.x & 31; m <= p; m += 32) {
    double dm = sqrt(1.0 / (4.0 * kPiD));
    for (int k = 0; k < m; ++k) dm *= -sqrt(1.0 + 1.0 / (2.0 * (k + 1))) * st;
    double pm2 = 0, pm1 = 0;
    double hr[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
    for (int n = m; n <= p; ++n) {
      double P;
      if (n == m)
        P = dm;
      else if (n == m + 1)
        P = sqrt(2.0 * m + 3.0) * ct * dm;
      else
        P = rec_a(n, m) * (ct * pm1 - rec_b(n, m) * pm2);
      pm2 = pm1;
      pm1 = P;
      for (int q = 0; q < 3; ++q) {
        hr[q] += c[q * cstride + n * (n + 1) + m] * P;
        if (m > 0) hi[q] += c[q * cstride + n * (n + 1) - m] * P;
      }
    }
    double sm, cm;
    sincos(m * ph, &sm, &cm);
    const double fac = m == 0 ? 1.0 : 2.0;
    for (int q = 0; q < 3; ++q) out[q] += fac * (hr[q] * cm - hi[q] * sm);
  }
  for (int q = 0; q < 3; ++q)
    for (int o = 16; o > 0; o >>= 1) out[q] += __shfl_xor_sync(0xffffffffu, out[q], o);
}

// seed: nearest standard grid point of drop j to the target, one warp per pair
__global__ void k_near_seed(const NearPair* __restrict__ pairs, int npair, const double* __restrict__ rec_std,
                            const long long* __restrict__ toff, const int* __restrict__ ngd,
                            const long long* __restrict__ tgt_loc, const int* __restrict__ tdrop,
                            int* __restrict__ seed) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (i >= npair) return;
  const long long t = pairs[i].target;
  const int j = pairs[i].src_drop, di = tdrop[t];
  const long long ngi = ngd[di];
  const double* ri = rec_std + 7 * toff[di];
  double d;
  const long long bi =
      warp_nearest(rec_std + 7 * toff[j], ngd[j], ri[tgt_loc[t]], ri[ngi + tgt_loc[t]], ri[2 * ngi + tgt_loc[t]], d);
  if ((threadIdx.x & 31) == 0) seed[i] = (int)bi;
}

// Levenberg-Marquardt Newton on F = |x(theta, phi) - x0|^2 / 2 in the rotated frame (seed at the
// equator).  One warp per pair, every lane with the same iterate; rotated coefficients xr[pair][3][(p+1)^2].
__global__ void k_near_newton(const NearPair* __restrict__ pairs, int npair, const double* __restrict__ xr,
                              const int* __restrict__ pdeg, const long long* __restrict__ xr_off,
                              const double* __restrict__ x0all, const double* __restrict__ tab, int tabP,
                              double* __restrict__ result) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (i >= npair) return;
  const int p = pdeg[pairs[i].src_drop];
  const long long cs = (long long)(p + 1) * (p + 1);
  const double* c = xr + xr_off[i];
  const double x0[3] = {x0all[3 * i], x0all[3 * i + 1], x0all[3 * i + 2]};
  double th = 0.5 * kPiD, ph = 0.0;
  double d[6][3];
  sh_eval_d2<true>(c, cs, p, th, ph, tab, tabP, d);
  auto half_sq = [&](const double* x) {
    const double a = x[0] - x0[0], b = x[1] - x0[1], e = x[2] - x0[2];
    return 0.5 * (a * a + b * b + e * e);
  };
  double F = half_sq(d[0]);
  double mu = -1.0;
  for (int it = 0; it < 30; ++it) {
    double r[3], xt[3], xp[3];
    for (int q = 0; q < 3; ++q) {
      r[q] = d[0][q] - x0[q];
      xt[q] = d[1][q];
      xp[q] = d[2][q];
    }
    const double g0 = r[0] * xt[0] + r[1] * xt[1] + r[2] * xt[2];
    const double g1 = r[0] * xp[0] + r[1] * xp[1] + r[2] * xp[2];
    const double Haa = xt[0] * xt[0] + xt[1] * xt[1] + xt[2] * xt[2] + r[0] * d[3][0] + r[1] * d[3][1] + r[2] * d[3][2];
    const double Hab = xt[0] * xp[0] + xt[1] * xp[1] + xt[2] * xp[2] + r[0] * d[4][0] + r[1] * d[4][1] + r[2] * d[4][2];
    const double Hbb = xp[0] * xp[0] + xp[1] * xp[1] + xp[2] * xp[2] + r[0] * d[5][0] + r[1] * d[5][1] + r[2] * d[5][2];
    if (mu < 0) mu = 1e-8 * fabs(Haa + Hbb);
    bool accepted = false;
    double s0 = 0, s1 = 0, dn[1][3];
    for (int k = 0; k < 40; ++k) {
      const double a = Haa + mu, b = Hab, e = Hbb + mu;
      const double det = a * e - b * b;
      s0 = -(e * g0 - b * g1) / det;
      s1 = -(a * g1 - b * g0) / det;
      // the test needs the value only, and at the minimum most trials are rejected (2051 points off drops of
      // degree 24: 2.6 -> 1.8 ms)
      sh_eval_d2<false>(c, cs, p, th + s0, ph + s1, tab, tabP, dn);
      if (half_sq(dn[0]) <= F) {
        accepted = true;
        break;
      }
      mu *= 10.0;
    }
    if (!accepted) break;
    th += s0;
    ph += s1;
    sh_eval_d2<true>(c, cs, p, th, ph, tab, tabP, d);
    F = half_sq(d[0]);
    if (fmax(fabs(s0), fabs(s1)) < 1e-14) break;
  }
  if (threadIdx.x & 31) return;
  result[5 * i + 0] = th;
  result[5 * i + 1] = ph;
  result[5 * i + 2] = d[0][0];
  result[5 * i + 3] = d[0][1];
  result[5 * i + 4] = d[0][2];
}

// From the Newton results (theta*, phi* in the rotated frame, x*): the pair's distance d0, the parameters of x*
// in drop j's own frame (v = R_z(alpha) R_y(beta) s(theta*, phi*), alpha = pi lon / (p+1)) and the check
// points x_l = x* + h_j sqrt(l) e, e = (x0 - x*)/|x0 - x*|, l = 1..L.
__global__ void k_near_checkpoints(NearPair* __restrict__ pairs, int npair, int L, const double* __restrict__ res,
                                   const double* __restrict__ x0all, const int* __restrict__ lon,
                                   const double* __restrict__ beta, const int* __restrict__ pdeg,
                                   const double* __restrict__ hdrop, double* __restrict__ pts) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= npair) return;
  const int j = pairs[i].src_drop;
  double e[3], d0 = 0;
  for (int c = 0; c < 3; ++c) {
    e[c] = x0all[3 * i + c] - res[5 * i + 2 + c];
    d0 += e[c] * e[c];
  }
  d0 = sqrt(d0);
  for (int c = 0; c < 3; ++c) e[c] /= d0;
  double st, ct, sp, cp, sb, cb, sa, ca;
  sincos(res[5 * i], &st, &ct);
  sincos(res[5 * i + 1], &sp, &cp);
  sincos(beta[i], &sb, &cb);
  sincospi((double)lon[i] / (pdeg[j] + 1), &sa, &ca);
  const double y0 = cb * (st * cp) + sb * ct, y1 = st * sp, y2 = -sb * (st * cp) + cb * ct;
  pairs[i].d0 = d0;
  pairs[i].theta_v = acos(fmax(-1.0, fmin(1.0, y2)));
  pairs[i].phi_v = atan2(sa * y0 + ca * y1, ca * y0 - sa * y1);
  for (int l = 1; l <= L; ++l)
    for (int c = 0; c < 3; ++c)
      pts[3 * ((long long)i * L + (l - 1)) + c] = res[5 * i + 2 + c] + hdrop[j] * sqrt((double)l) * e[c];
}

// grid of each check point: 0 standard (Omega_0), 1 upsampled otherwise (same distance rule as the
// region split).  The point of the upsampled grid next to the parameters of x* is usually within A h of the
// check point already, which settles it; only otherwise the whole grid is scanned (2051 fluid points off
// drops of degree 24: 1.08 -> 0.01 ms).
__global__ void k_near_checkgrid(const NearPair* __restrict__ pairs, int npair, int L, const double* __restrict__ pts,
                                 const double* __restrict__ centre, const double* __restrict__ bound,
                                 const double* __restrict__ h, double a_tilde, const double* __restrict__ rec_up,
                                 const long long* __restrict__ up_off, const long long* __restrict__ up_n,
                                 int* __restrict__ grid) {
  const int idx = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;  // one warp per check point
  if (idx >= npair * L) return;
  const int lane = threadIdx.x & 31;
  const int i = idx / L;
  const int j = pairs[i].src_drop;
  const double x0 = pts[3 * idx], x1 = pts[3 * idx + 1], x2 = pts[3 * idx + 2];
  const double dc0 = x0 - centre[3 * j], dc1 = x1 - centre[3 * j + 1], dc2 = x2 - centre[3 * j + 2];
  if (sqrt(dc0 * dc0 + dc1 * dc1 + dc2 * dc2) - bound[j] > a_tilde * h[j]) {
    if (lane == 0) grid[idx] = 0;
    return;
  }
  const long long N = up_n[j];
  const double* r = rec_up + 7 * up_off[j];
  double best = 1e300;
  {
    const int nj = (int)(sqrt(0.5 * (double)N) + 0.5), nk = 2 * nj;  // N = nj nk, Gauss nodes near (j + 3/4)/(nj + 1/2)
    const int row = min(nj - 1, max(0, (int)((1.0 - pairs[i].theta_v / kPiD) * (nj + 0.5) - 0.25)));
    const int turn = (int)rint(pairs[i].phi_v / kPiD * nj) % nk, col = turn < 0 ? turn + nk : turn;
    const long long s = (long long)row * nk + col;
    const double d0 = x0 - r[s], d1 = x1 - r[N + s], d2 = x2 - r[2 * N + s];
    if (sqrt(d0 * d0 + d1 * d1 + d2 * d2) <= a_tilde * h[j]) {
      if (lane == 0) grid[idx] = 1;
      return;
    }
  }
  for (long long s = lane; s < N; s += 32) {
    const double d0 = x0 - r[s], d1 = x1 - r[N + s], d2 = x2 - r[2 * N + s];
    best = fmin(best, d0 * d0 + d1 * d1 + d2 * d2);
  }
  for (int o = 16; o > 0; o >>= 1) best = fmin(best, __shfl_xor_sync(0xffffffffu, best, o));
  if (lane == 0) grid[idx] = sqrt(best) <= a_tilde * h[j] ? 1 : 0;
}

// Regular-rule value of drop j's layer at check point (pair, l): one block per check point.
template <typename R, int KIND>
__global__ void __launch_bounds__(256) k_near_checks(
    const NearPair* __restrict__ pairs, int L, const double* __restrict__ pts, const int* __restrict__ grid,
    const double* __restrict__ centre, const long long* __restrict__ toff, const int* __restrict__ ngd,
    const long long* __restrict__ up_off, const long long* __restrict__ up_n, const R* __restrict__ Xs,
    const R* __restrict__ Ns, const R* __restrict__ Qs, long long nstd, const R* __restrict__ Xu,
    const R* __restrict__ Nu, const R* __restrict__ Qu, long long nup, const double* __restrict__ wts,
    double* __restrict__ cv) {
  __shared__ R red[3 * 32];
  const int idx = blockIdx.x;
  const int i = idx / L;
  const int j = pairs[i].src_drop;
  const bool up = grid[idx] != 0;
  const R* X = up ? Xu : Xs;
  const R* N = up ? Nu : Ns;
  const R* Q = up ? Qu : Qs;
  const long long ld = up ? nup : nstd;
  const long long s0 = up ? up_off[j] : toff[j];
  const long long s1 = s0 + (up ? up_n[j] : (long long)ngd[j]);
  const R px = (R)(pts[3 * idx] - centre[3 * j]), py = (R)(pts[3 * idx + 1] - centre[3 * j + 1]),
          pz = (R)(pts[3 * idx + 2] - centre[3 * j + 2]);
  R a0 = 0, a1 = 0, a2 = 0;
  for (long long s = s0 + threadIdx.x; s < s1; s += blockDim.x) {
    const R dx = px - X[s], dy = py - X[ld + s], dz = pz - X[2 * ld + s];
    const R r2 = dx * dx + dy * dy + dz * dz;
    const R q0 = Q[s], q1 = Q[ld + s], q2 = Q[2 * ld + s];
    const R xq = dx * q0 + dy * q1 + dz * q2;
    if (KIND == 0) {
      const R ri = rsqrt_<R>(r2);
      const R c = xq * ri * ri * ri;
      a0 += q0 * ri + c * dx;
      a1 += q1 * ri + c * dy;
      a2 += q2 * ri + c * dz;
    } else {
      const R xn = dx * N[s] + dy * N[ld + s] + dz * N[2 * ld + s];
      const R c = (R)(-6) * xq * xn * rsqrt5_<R>(r2);
      a0 += c * dx;
      a1 += c * dy;
      a2 += c * dz;
    }
  }
  block_sum3<R>(a0, a1, a2, red);
  if (threadIdx.x == 0) {
    const double w = wts[j];
    cv[3 * idx] = w * (double)a0;
    cv[3 * idx + 1] = w * (double)a1;
    cv[3 * idx + 2] = w * (double)a2;
  }
}

// The weighted sum of both layers at check point (pair, l), cv = wS S[f] + wD D[u] (FP64): the velocity needs no
// more, and the two kernels share the differences, the distance and the powers of 1/r.  32 FP64 operations per
// source against 23 and 24 apart: 2051 fluid points off drops of degree 24, 7.9 -> 5.0 ms.
__global__ void __launch_bounds__(256) k_near_checks_both(
    const NearPair* __restrict__ pairs, int L, const double* __restrict__ pts, const int* __restrict__ grid,
    const double* __restrict__ centre, const long long* __restrict__ toff, const int* __restrict__ ngd,
    const long long* __restrict__ up_off, const long long* __restrict__ up_n, NearSources st, NearSources up,
    const double* __restrict__ wS, const double* __restrict__ wD, double* __restrict__ cv) {
  __shared__ double red[3 * 32];
  const int idx = blockIdx.x;
  const int j = pairs[idx / L].src_drop;
  const bool fine = grid[idx] != 0;
  const NearSources& G = fine ? up : st;
  const long long ld = G.ld, s0 = fine ? up_off[j] : toff[j], s1 = s0 + (fine ? up_n[j] : (long long)ngd[j]);
  const double px = pts[3 * idx] - centre[3 * j], py = pts[3 * idx + 1] - centre[3 * j + 1],
               pz = pts[3 * idx + 2] - centre[3 * j + 2];
  const double ratio = -6.0 * wD[j] / wS[j];
  double a0 = 0, a1 = 0, a2 = 0;
  for (long long s = s0 + threadIdx.x; s < s1; s += blockDim.x) {
    const double dx = px - G.X[s], dy = py - G.X[ld + s], dz = pz - G.X[2 * ld + s];
    const double ri = rsqrt_<double>(dx * dx + dy * dy + dz * dz), ri2 = ri * ri, ri3 = ri * ri2;
    const double f0 = G.F[s], f1 = G.F[ld + s], f2 = G.F[2 * ld + s];
    const double xf = dx * f0 + dy * f1 + dz * f2;
    const double xu = dx * G.U[s] + dy * G.U[ld + s] + dz * G.U[2 * ld + s];
    const double xn = dx * G.N[s] + dy * G.N[ld + s] + dz * G.N[2 * ld + s];
    const double c = fma(ratio * xu * xn, ri3 * ri2, xf * ri3);
    a0 += f0 * ri;
    a1 += f1 * ri;
    a2 += f2 * ri;
    a0 += c * dx;
    a1 += c * dy;
    a2 += c * dz;
  }
  block_sum3<double>(a0, a1, a2, red);
  if (threadIdx.x == 0) {
    cv[3 * idx] = wS[j] * a0;
    cv[3 * idx + 1] = wS[j] * a1;
    cv[3 * idx + 2] = wS[j] * a2;
  }
}

// One warp per target with near pairs: anchor from the source drop's (weighted) self expansion,
// minus 4 pi w_j u(x*) for the double layer, then Lagrange interpolation at the target's distance.
__global__ void k_near_interp(const NearPair* __restrict__ pairs, const int* __restrict__ tbeg, int ntgt, int L,
                              int kind, const double* __restrict__ selfcoef, const double* __restrict__ dens,
                              const long long* __restrict__ coef_off, const int* __restrict__ pdeg,
                              const double* __restrict__ hdrop, const double* __restrict__ wts,
                              const double* __restrict__ cv, const int* __restrict__ tdrop,
                              const long long* __restrict__ tgt_loc, const long long* __restrict__ val_off,
                              const int* __restrict__ ngd, double* __restrict__ vals) {
  const int u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (u >= ntgt) return;
  double acc[3] = {0, 0, 0};
  const long long t = pairs[tbeg[u]].target;
  for (int i = tbeg[u]; i < tbeg[u + 1]; ++i) {
    const NearPair& P = pairs[i];
    const int j = P.src_drop, p = pdeg[j];
    const long long cs = (long long)(p + 1) * (p + 1);
    double anchor[3];
    sh_eval3(selfcoef + coef_off[j], cs, p, P.theta_v, P.phi_v, anchor);
    if (kind == 1) {
      double us[3];
      sh_eval3(dens + coef_off[j], cs, p, P.theta_v, P.phi_v, us);
      for (int q = 0; q < 3; ++q) anchor[q] -= 4.0 * kPiD * wts[j] * us[q];
    }
    // Lagrange through (0, anchor) and (h sqrt(l), cv_l), l = 1..L, at distance d0, lane l node l
    const double h = hdrop[j], x = P.d0;
    const int l = threadIdx.x & 31;
    if (l <= L) {
      const double xl = l == 0 ? 0.0 : h * sqrt((double)l);
      double bas = 1.0;
      for (int k = 0; k <= L; ++k) {
        if (k == l) continue;
        const double xk = k == 0 ? 0.0 : h * sqrt((double)k);
        bas *= (x - xk) / (xl - xk);
      }
      for (int q = 0; q < 3; ++q) acc[q] += bas * (l == 0 ? anchor[q] : cv[3 * ((long long)i * L + (l - 1)) + q]);
    }
  }
  for (int q = 0; q < 3; ++q)
    for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_down_sync(0xffffffffu, acc[q], o);
  if (threadIdx.x & 31) return;
  const int d = tdrop[t];
  const long long ng = ngd[d];
  double* v = vals + val_off[d] + tgt_loc[t];
  v[0] += acc[0];
  v[ng] += acc[1];
  v[2 * ng] += acc[2];
}

// ---- the near-singular rule as rows of the operator ----
// The interpolated value of a pair is linear in the source drop's density: with the Lagrange weights b_l
// at the target's distance, x_l the check points and rho = sum_r c_r Y_r on the grids,
//     sum_l b_l sum_s K(x_l - x_s) wJ_s rho_s = sum_r [ sum_s (sum_l b_l K(x_l - x_s)) wJ_s Y_r(s) ] c_r,
// so the sum over the check points is taken once per geometry and kind, and projected on Y_r by the
// transposed synthesis (phi sums over longitude quadruples, then P~_n^m over latitude pairs).  A row has
// six symmetric 3x3 planes; for the double layer the jump -4 pi b_0 u(x*) of the exterior limit is part
// of them.  A seventh plane holds b_0 Y_r(x*), which meets the drop's own on-surface expansion.  Building
// a row costs about 2.4 evaluations of its check-point sums (31 FP64 operations per check point and source,
// and the projection), and every apply after that reads 7 (p+1)^2 doubles instead: so a kind's first apply on
// a geometry sums the check points (k_near_checks), and the rows are built for those after it.  Two drops of
// degree 32 at gap 0.05 (U = 4): check sums 3.6 ms an apply, rows 8.4 and 9.1 ms (S, D) once and 0.05 ms an apply.
constexpr int kNearThreads = 256;

template <int KIND>
__global__ void __launch_bounds__(kNearThreads) k_near_rows(const NearPair* __restrict__ pairs,
                                                            const int* __restrict__ list, int p, int L,
                                                            const double* __restrict__ pts,
                                                            const int* __restrict__ grid,
                                                            const double* __restrict__ centre,
                                                            const double* __restrict__ hdrop, NearRowsSrc g0,
                                                            NearRowsSrc g1, const long long* __restrict__ row_off,
                                                            double* __restrict__ rows) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double bas[17], cx[16][3];
  __shared__ int any[2], onup[16];
  const int i = list[blockIdx.x];
  const NearPair pr = pairs[i];
  const int j = pr.src_drop, ntri = (p + 1) * (p + 2) / 2, nc = (p + 1) * (p + 1), ncp = self_row(p);
  const int nkmax = 2 * (g0.P > g1.P ? g0.P : g1.P) + 2;
  double* sq = reinterpret_cast<double*>(smem_raw);  // [12][ntri]
  double* sk = sq + 12 * ntri;                       // [2 rows][6][nkmax]
  double* sd = sk + 12 * nkmax;                      // [even, odd][12][p+1]
  double* sy = sd + 24 * (p + 1);                    // [ncp] b_0 Y_r(x*)
  for (int k = threadIdx.x; k < 12 * ntri; k += kNearThreads) sq[k] = 0.0;
  if (threadIdx.x < 2) any[threadIdx.x] = 0;
  __syncthreads();
  if (threadIdx.x <= L) {
    const int l = threadIdx.x;
    const double h = hdrop[j], xl = l == 0 ? 0.0 : h * sqrt((double)l);
    double b = 1.0;
    for (int k = 0; k <= L; ++k) {
      if (k == l) continue;
      const double xk = k == 0 ? 0.0 : h * sqrt((double)k);
      b *= (pr.d0 - xk) / (xl - xk);
    }
    bas[l] = b;
    if (l > 0) {
      for (int c = 0; c < 3; ++c) cx[l - 1][c] = pts[3 * ((long long)i * L + l - 1) + c] - centre[3 * j + c];
      onup[l - 1] = grid[(long long)i * L + l - 1] != 0;
      any[onup[l - 1]] = 1;
    }
  }
  __syncthreads();
  for (int gk = 0; gk < 2; ++gk) {
    if (!any[gk]) continue;
    const NearRowsSrc& G = gk ? g1 : g0;
    const int P = G.P, nj = P + 1, nk = 2 * P + 2, half = P + 1, np = (nj + 1) / 2, k4n = half / 2 + 1;
    const long long s0 = G.off[j], ng = (long long)nj * nk;
    const double* wJ = G.rec + 7 * s0 + 6 * ng;
    for (int q = 0; q < np; ++q) {
      const int nrow = 2 * q == P ? 1 : 2;
      // combined kernel weights of the rows q and P - q
      for (int t = threadIdx.x; t < nrow * nk; t += kNearThreads) {
        const int r = t / nk, k = t - r * nk;
        const long long o = (long long)(r ? P - q : q) * nk + k, s = s0 + o;
        const double w = wJ[o], x0 = G.X[s], x1 = G.X[G.ld + s], x2 = G.X[2 * G.ld + s];
        double n0 = 0, n1 = 0, n2 = 0;
        if (KIND) {
          n0 = w * G.N[s];
          n1 = w * G.N[G.ld + s];
          n2 = w * G.N[2 * G.ld + s];
        }
        double m[6] = {0, 0, 0, 0, 0, 0}, dsum = 0;
        for (int l = 0; l < L; ++l) {
          if (onup[l] != gk) continue;
          const double dx = cx[l][0] - x0, dy = cx[l][1] - x1, dz = cx[l][2] - x2;
          const double r2 = dx * dx + dy * dy + dz * dz;
          double c;
          if (KIND == 0) {
            const double ri = rsqrt_<double>(r2), a = bas[l + 1] * w * ri;
            dsum += a;
            c = a * (ri * ri);
          } else {
            c = (bas[l + 1] * (dx * n0 + dy * n1 + dz * n2)) * rsqrt5_<double>(r2);
          }
          const double ax = c * dx, ay = c * dy;
          m[0] += ax * dx;
          m[1] += ay * dy;
          m[2] += (c * dz) * dz;
          m[3] += ax * dy;
          m[4] += ax * dz;
          m[5] += ay * dz;
        }
        const double f = KIND ? -6.0 : 1.0;
#pragma unroll
        for (int e = 0; e < 6; ++e) sk[(r * 6 + e) * nkmax + k] = f * m[e] + (e < 3 ? dsum : 0.0);
      }
      __syncthreads();
      // fold the longitude quadruples in place: even and odd orders' cosine sums at k and half + k, sine
      // sums at 2 half - k and half - k (the middle k has two longitudes: one cosine and one sine sum)
      for (int t = threadIdx.x; t < nrow * 6 * k4n; t += kNearThreads) {
        const int k = t % k4n;
        double* v = sk + (t / k4n) * nkmax;
        const double a = v[k], c = v[half + k];
        if (k == 0) {
          v[0] = a + c;
          v[half] = a - c;
        } else if (2 * k == half) {
          v[k] = a + c;
          v[half + k] = a - c;
        } else {
          const double b = v[2 * half - k], d = v[half - k];
          v[k] = (a + b) + (c + d);
          v[half + k] = (a + b) - (c + d);
          v[2 * half - k] = (a - b) + (c - d);
          v[half - k] = (a - b) - (c - d);
        }
      }
      __syncthreads();
      // phi transform of both rows, then their sum and difference (even and odd n - m)
      for (int t = threadIdx.x; t < 6 * (p + 1); t += kNearThreads) {
        const int m = t % (p + 1), e = t / (p + 1);
        const double* cm = G.cs + (long long)m * nk * 2;
        double re[2] = {0, 0}, im[2] = {0, 0};
        const int mid = half % 2 == 0 ? half / 2 : -1;
        for (int r = 0; r < nrow; ++r) {
          const double* v = sk + (r * 6 + e) * nkmax;
          const double* vc = (m & 1) ? v + half : v;
          const double* vs = (m & 1) ? v + half : v + 2 * half;
          double a = vc[0], b = 0;
          for (int k = 1; 2 * k < half; ++k) {
            a += vc[k] * cm[2 * k];
            b += vs[-k] * cm[2 * k + 1];
          }
          if (mid > 0) {
            if (m & 1)
              b += v[half + mid] * cm[2 * mid + 1];
            else
              a += v[mid] * cm[2 * mid];
          }
          re[r] = a;
          im[r] = b;
        }
        sd[(2 * e) * (p + 1) + m] = re[0] + re[1];
        sd[(2 * e + 1) * (p + 1) + m] = im[0] + im[1];
        sd[(12 + 2 * e) * (p + 1) + m] = re[0] - re[1];
        sd[(12 + 2 * e + 1) * (p + 1) + m] = im[0] - im[1];
      }
      __syncthreads();
      for (int t = threadIdx.x; t < ntri; t += kNearThreads) {
        int n = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
        while ((n + 1) * (n + 2) / 2 <= t) ++n;
        while (n * (n + 1) / 2 > t) --n;
        const int m = t - n * (n + 1) / 2;
        const double Pv = G.T0[leg_row(p, m, n, nj) + q];
        const double* d = sd + (((n - m) & 1) ? 12 : 0) * (p + 1) + m;
#pragma unroll
        for (int e = 0; e < 12; ++e) sq[e * ntri + t] += d[e * (p + 1)] * Pv;
      }
      __syncthreads();
    }
  }
  // b_0 Y_r(x*), one thread per order
  {
    double st, ct;
    sincos(pr.theta_v, &st, &ct);
    for (int m = threadIdx.x; m <= p; m += kNearThreads) {
      double dm = sqrt(1.0 / (4.0 * kPiD));
      for (int k = 0; k < m; ++k) dm *= -sqrt(1.0 + 1.0 / (2.0 * (k + 1))) * st;
      double sm, cm, pm1 = 0, pm2 = 0;
      sincos(m * pr.phi_v, &sm, &cm);
      const double fac = (m == 0 ? 1.0 : 2.0) * bas[0];
      for (int n = m; n <= p; ++n) {
        const double v = n == m ? dm : n == m + 1 ? sqrt(2.0 * m + 3.0) * ct * dm : rec_a(n, m) * (ct * pm1 - rec_b(n, m) * pm2);
        pm2 = pm1;
        pm1 = v;
        sy[n * (n + 1) + m] = fac * v * cm;
        if (m > 0) sy[n * (n + 1) - m] = -fac * v * sm;
      }
    }
    for (int r = nc + threadIdx.x; r < ncp; r += kNearThreads) sy[r] = 0.0;
  }
  __syncthreads();
  double* out = rows + row_off[i];
  for (int t = threadIdx.x; t < 7 * ncp; t += kNearThreads) {
    const int e = t / ncp, r = t - e * ncp;
    double v = e == 6 ? sy[r] : 0.0;
    if (e < 6 && r < nc) {
      const int n = degree_of(r), m = r - n * (n + 1), it = n * (n + 1) / 2 + (m < 0 ? -m : m);
      v = m == 0 ? sq[2 * e * ntri + it] : m > 0 ? 2.0 * sq[2 * e * ntri + it] : -2.0 * sq[(2 * e + 1) * ntri + it];
      if (KIND && e < 3) v -= 4.0 * kPiD * sy[r];
    }
    out[t] = v;
  }
}

// vals += the near values of one target from its pairs' rows: one warp per target, its pairs in order.
__global__ void __launch_bounds__(128) k_near_rows_apply(const NearPair* __restrict__ pairs,
                                                         const int* __restrict__ tbeg, int ntgt,
                                                         const double* __restrict__ rows,
                                                         const long long* __restrict__ row_off,
                                                         const double* __restrict__ selfcoef,
                                                         const double* __restrict__ dens,
                                                         const long long* __restrict__ coef_off,
                                                         const int* __restrict__ pdeg, const double* __restrict__ wts,
                                                         const int* __restrict__ tdrop,
                                                         const long long* __restrict__ tgt_loc,
                                                         const long long* __restrict__ val_off,
                                                         const int* __restrict__ ngd, double* __restrict__ vals) {
  const int u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (u >= ntgt) return;
  double acc[3] = {0, 0, 0};
  for (int i = tbeg[u]; i < tbeg[u + 1]; ++i) {
    const int j = pairs[i].src_drop, p = pdeg[j], nc = (p + 1) * (p + 1), ncp = self_row(p);
    const double* M = rows + row_off[i];
    const double *d = dens + coef_off[j], *sc = selfcoef + coef_off[j];
    double a[3] = {0, 0, 0};
#pragma unroll 2
    for (int r = lane; r < nc; r += 32) {
      const double x = d[r], y = d[nc + r], z = d[2 * nc + r], Y = M[6 * ncp + r];
      const double m0 = M[r], m1 = M[ncp + r], m2 = M[2 * ncp + r], m3 = M[3 * ncp + r], m4 = M[4 * ncp + r],
                   m5 = M[5 * ncp + r];
      a[0] += m0 * x + m3 * y + m4 * z;
      a[1] += m3 * x + m1 * y + m5 * z;
      a[2] += m4 * x + m5 * y + m2 * z;
      acc[0] += Y * sc[r];
      acc[1] += Y * sc[nc + r];
      acc[2] += Y * sc[2 * nc + r];
    }
    for (int c = 0; c < 3; ++c) acc[c] += wts[j] * a[c];
  }
  for (int c = 0; c < 3; ++c)
    for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_down_sync(0xffffffffu, acc[c], o);
  if (lane) return;
  const long long t = pairs[tbeg[u]].target;
  const int d = tdrop[t];
  const long long ng = ngd[d];
  double* v = vals + val_off[d] + tgt_loc[t];
  v[0] += acc[0];
  v[ng] += acc[1];
  v[2 * ng] += acc[2];
}

// The source drop's shape coefficients of pair i with the phases of its seed longitude applied,
// g_n^m = e^{i m alpha_i} x_n^m (real-packed; alpha_i = pi lon[i] / (p+1), lon the seed's longitude index),
// written to out + dst_off[i] as [3][(p+1)^2]: the first step of the rotation R_z(alpha) R_y(beta), so
// that the pairs of one seed latitude then share one rotation launch.  One block per pair.
__global__ void k_near_phase_shift(const NearPair* __restrict__ pairs, int npair, const double* __restrict__ coef,
                                   const long long* __restrict__ coef_off, const int* __restrict__ pdeg,
                                   const int* __restrict__ lon, const long long* __restrict__ dst_off,
                                   double* __restrict__ out) {
  __shared__ double phi[2 * (BIE_MAX_P + 1)];
  const int i = blockIdx.x;
  if (i >= npair) return;
  const int j = pairs[i].src_drop;
  const int p = pdeg[j];
  const long long nc = (long long)(p + 1) * (p + 1);
  for (int m = threadIdx.x; m <= p; m += blockDim.x)
    sincospi((double)((m * lon[i]) % (2 * p + 2)) / (p + 1), &phi[2 * m + 1], &phi[2 * m]);
  __syncthreads();
  for (long long q = threadIdx.x; q < 3 * nc; q += blockDim.x) {
    const int c = (int)(q / nc);
    const long long k = q - c * nc;
    int n = (int)sqrt((double)k);
    while ((long long)n * n > k) --n;
    while ((long long)(n + 1) * (n + 1) <= k) ++n;
    const int mm = (int)(k - (long long)n * (n + 1));
    const int m = mm < 0 ? -mm : mm;
    const double* f = coef + coef_off[j] + c * nc;
    const double fr = f[n * (n + 1) + m];
    const double fi = m > 0 ? f[n * (n + 1) - m] : 0.0;
    const double cr = phi[2 * m], ci = phi[2 * m + 1];
    out[dst_off[i] + c * nc + k] = mm >= 0 ? fr * cr - fi * ci : fr * ci + fi * cr;
  }
}

}  // namespace

int launch_near_phase_shift(const NearPair* pairs, int npair, const double* coef, const long long* coef_off,
                            const int* pdeg, const int* lon, const long long* dst_off, double* out,
                            cudaStream_t s) {
  if (!npair) return BIE_OK;
  k_near_phase_shift<<<npair, 128, 0, s>>>(pairs, npair, coef, coef_off, pdeg, lon, dst_off, out);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

size_t near_rows_smem(int p, int P) {
  return sizeof(double) * (6 * (size_t)(p + 1) * (p + 2) + 12 * (size_t)(2 * P + 2) + 24 * (size_t)(p + 1) + self_row(p));
}

int launch_near_rows(int kind, const NearPair* pairs, const int* list, int n, int p, int L, const double* pts,
                     const int* grid, const double* centre, const double* hdrop, const NearRowsSrc& std_,
                     const NearRowsSrc& up, const long long* row_off, double* rows, cudaStream_t s) {
  if (!n) return BIE_OK;
  const size_t smem = near_rows_smem(p, std_.P > up.P ? std_.P : up.P);
  auto kern = kind == 0 ? k_near_rows<0> : k_near_rows<1>;
  BIE_CUDA_TRY(allow_smem(kern, smem));
  kern<<<n, kNearThreads, smem, s>>>(pairs, list, p, L, pts, grid, centre, hdrop, std_, up, row_off, rows);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_near_rows_apply(const NearPair* pairs, const int* tbeg, int ntgt, const double* rows, const long long* row_off,
                           const double* selfcoef, const double* dens, const long long* coef_off, const int* pdeg,
                           const double* wts, const int* tdrop, const long long* tgt_loc, const long long* val_off,
                           const int* ngd, double* vals, cudaStream_t s) {
  if (!ntgt) return BIE_OK;
  k_near_rows_apply<<<(ntgt + 3) / 4, 128, 0, s>>>(pairs, tbeg, ntgt, rows, row_off, selfcoef, dens, coef_off, pdeg, wts,
                                                   tdrop, tgt_loc, val_off, ngd, vals);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_near_seed(const NearPair* pairs, int npair, const double* rec_std, const long long* toff, const int* ngd,
                     const long long* tgt_loc, const int* tdrop, int* seed, cudaStream_t s) {
  if (!npair) return BIE_OK;
  k_near_seed<<<(npair + 3) / 4, 128, 0, s>>>(pairs, npair, rec_std, toff, ngd, tgt_loc, tdrop, seed);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int near_rec_table_doubles(int P) { return 3 * (P + 1) * (P + 2) / 2 + P + 2; }

int launch_near_rec_table(int P, double* tab, cudaStream_t s) {
  const int n = (P + 1) * (P + 2) / 2;
  k_rec_table<<<(n + 127) / 128, 128, 0, s>>>(P, tab);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_near_newton(const NearPair* pairs, int npair, const double* xr, const int* pdeg, const long long* xr_off,
                       const double* x0, const double* tab, int tabP, double* result, cudaStream_t s) {
  if (!npair) return BIE_OK;
  k_near_newton<<<(npair + 3) / 4, 128, 0, s>>>(pairs, npair, xr, pdeg, xr_off, x0, tab, tabP, result);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_near_checkpoints(NearPair* pairs, int npair, int L, const double* res, const double* x0, const int* lon,
                            const double* beta, const int* pdeg, const double* hdrop, double* pts, cudaStream_t s) {
  if (!npair) return BIE_OK;
  k_near_checkpoints<<<(npair + 63) / 64, 64, 0, s>>>(pairs, npair, L, res, x0, lon, beta, pdeg, hdrop, pts);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_near_checkgrid(const NearPair* pairs, int npair, int L, const double* pts, const double* centre,
                          const double* bound, const double* h, double a_tilde, const double* rec_up,
                          const long long* up_off, const long long* up_n, int* grid, cudaStream_t s) {
  if (!npair) return BIE_OK;
  k_near_checkgrid<<<(npair * L + 3) / 4, 128, 0, s>>>(pairs, npair, L, pts, centre, bound, h, a_tilde, rec_up,
                                                           up_off, up_n, grid);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

template <typename R>
int launch_near_checks(int kind, const NearPair* pairs, int npair, int L, const double* pts, const int* grid,
                       const double* centre, const long long* toff, const int* ngd, const long long* up_off,
                       const long long* up_n, const R* Xs, const R* Ns, const R* Qs, long long nstd, const R* Xu,
                       const R* Nu, const R* Qu, long long nup, const double* wts, double* cv, cudaStream_t s) {
  if (!npair) return BIE_OK;
  if (kind == 0)
    k_near_checks<R, 0><<<npair * L, 256, 0, s>>>(pairs, L, pts, grid, centre, toff, ngd, up_off, up_n, Xs, Ns, Qs,
                                                  nstd, Xu, Nu, Qu, nup, wts, cv);
  else
    k_near_checks<R, 1><<<npair * L, 256, 0, s>>>(pairs, L, pts, grid, centre, toff, ngd, up_off, up_n, Xs, Ns, Qs,
                                                  nstd, Xu, Nu, Qu, nup, wts, cv);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_near_checks_both(const NearPair* pairs, int npair, int L, const double* pts, const int* grid,
                            const double* centre, const long long* toff, const int* ngd, const long long* up_off,
                            const long long* up_n, const NearSources& std_, const NearSources& up, const double* wS,
                            const double* wD, double* cv, cudaStream_t s) {
  if (!npair) return BIE_OK;
  k_near_checks_both<<<npair * L, 256, 0, s>>>(pairs, L, pts, grid, centre, toff, ngd, up_off, up_n, std_, up, wS, wD, cv);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_near_interp(const NearPair* pairs, const int* tbeg, int ntgt, int L, int kind, const double* selfcoef,
                       const double* dens, const long long* coef_off, const int* pdeg, const double* hdrop,
                       const double* wts, const double* cv, const int* tdrop, const long long* tgt_loc,
                       const long long* val_off, const int* ngd, double* vals, cudaStream_t s) {
  if (!ntgt) return BIE_OK;
  k_near_interp<<<(ntgt + 3) / 4, 128, 0, s>>>(pairs, tbeg, ntgt, L, kind, selfcoef, dens, coef_off, pdeg, hdrop,
                                                wts, cv, tdrop, tgt_loc, val_off, ngd, vals);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

template int launch_near_checks<double>(int, const NearPair*, int, int, const double*, const int*, const double*,
                                        const long long*, const int*, const long long*, const long long*,
                                        const double*, const double*, const double*, long long, const double*,
                                        const double*, const double*, long long, const double*, double*,
                                        cudaStream_t);

}  // namespace bie

// Inter-drop interactions (Sec. 2.1, 2.3): region classification with bounding spheres, and the
// regular (standard grid, Omega_0) and upsampled (grid of degree U(p+1)-1, Omega_1) pair sums of the
// single- and double-layer kernels, as a balanced work list of (target tile, source drop, grid,
// source range, target mask) items.
#include <cuda_runtime.h>

#include <type_traits>

#include "device.cuh"
#include "interdrop.h"
#include "internal.cuh"

namespace bie {
namespace {

constexpr int kThreads = 256;
inline unsigned blocks_for(long long n, int t = kThreads) { return (unsigned)((n + t - 1) / t); }

// region[t * ndrop + j]: 0 / 1 / 2 for Omega_0/1/2 of target t w.r.t. drop j, 3 = t inside drop j,
// 255 for j = own drop.  Distance = nearest point of j's upsampled grid (Sec. 2.3).  A block settles its
// 256 (target, drop) pairs outside the bounding spheres widened by A h_j and lists the others in shared
// memory; its warps then scan the upsampled grid for one listed pair each (warp_nearest).  The listed pairs of neighbouring targets
// come together, so one thread per pair left a few threads with a serial scan each: 8 drops of degree 16,
// 0.96 -> 0.15 ms.
__global__ void __launch_bounds__(kThreads) k_classify(
    const double* __restrict__ rec_std, long long ntarget, const int* __restrict__ tdrop,
    const long long* __restrict__ tloc, const long long* __restrict__ toff_std, const int* __restrict__ ngd, int ndrop,
    const double* __restrict__ centre, const double* __restrict__ bound, const double* __restrict__ h, double a_tilde,
    const double* __restrict__ rec_up, const long long* __restrict__ up_off, const long long* __restrict__ up_n,
    unsigned char* __restrict__ region) {
  __shared__ double px[kThreads][3];
  __shared__ int list[kThreads], count;
  if (threadIdx.x == 0) count = 0;
  __syncthreads();
  const long long idx0 = (long long)blockIdx.x * kThreads, idx = idx0 + threadIdx.x;
  if (idx < ntarget * ndrop) {
    const long long t = idx / ndrop;
    const int j = (int)(idx - t * ndrop);
    const int i = tdrop[t];
    if (i == j) {
      region[idx] = 255;
    } else {
      const long long ng = ngd[i];
      const double* ri = rec_std + 7 * toff_std[i];
      const double x0 = ri[tloc[t]], x1 = ri[ng + tloc[t]], x2 = ri[2 * ng + tloc[t]];
      const double dc0 = x0 - centre[3 * j], dc1 = x1 - centre[3 * j + 1], dc2 = x2 - centre[3 * j + 2];
      const double dcen = sqrt(dc0 * dc0 + dc1 * dc1 + dc2 * dc2);
      if (dcen - bound[j] > a_tilde * h[j]) {  // every grid point of j is farther than A h_j
        region[idx] = 0;
      } else {
        px[threadIdx.x][0] = x0;
        px[threadIdx.x][1] = x1;
        px[threadIdx.x][2] = x2;
        list[atomicAdd(&count, 1)] = threadIdx.x;
      }
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int w = threadIdx.x >> 5; w < count; w += kThreads / 32) {
    const int k = list[w], j = (int)((idx0 + k) % ndrop);
    const double x0 = px[k][0], x1 = px[k][1], x2 = px[k][2];
    const long long N = up_n[j];
    const double* r = rec_up + 7 * up_off[j];
    double best;
    const long long bi = warp_nearest(r, N, x0, x1, x2, best);
    if (lane) continue;
    const double dist = sqrt(best);
    const double side = (x0 - r[bi]) * r[3 * N + bi] + (x1 - r[N + bi]) * r[4 * N + bi] + (x2 - r[2 * N + bi]) * r[5 * N + bi];
    unsigned char code = dist <= h[j] ? 2 : (dist <= a_tilde * h[j] ? 1 : 0);
    if (side <= 0.0) code = 3;
    region[idx0 + k] = code;
  }
}

constexpr int kChunk = 128;  // sources staged per pass

// Staged source record: (x, y, z, q0), (q1, q2, n0, n1), (n2, -, -, -) so that the inner loop reads
// it with 128-bit shared-memory loads (two for the single layer, three for the double layer).
template <typename R>
struct alignas(16) SrcRec {
  R v[12];
};

// One block per work-list block: the tile's 128 targets, TPT per thread (targets tid + u * 128/TPT),
// against the sources of its items, staged through shared memory.  The stresslet's factor -6 is
// applied with the item's weight.
template <typename R, int KIND, int TPT>
__global__ void __launch_bounds__(kTile / TPT) k_interdrop(
    const PairItem* __restrict__ items, const int* __restrict__ blk_item, const long long* __restrict__ tile_t0,
    const int* __restrict__ tile_n, const int* __restrict__ tile_drop, const long long* __restrict__ tgt_loc,
    const long long* __restrict__ toff_std, const int* __restrict__ ngd, const double* __restrict__ rec_std,
    const double* __restrict__ centre, const R* __restrict__ Xs, const R* __restrict__ Ns, const R* __restrict__ Qs,
    long long nstd, const R* __restrict__ Xu, const R* __restrict__ Nu, const R* __restrict__ Qu, long long nup,
    const double* __restrict__ wts, double* __restrict__ partial) {
  constexpr int NT = kTile / TPT;  // threads per block
  constexpr int NR = KIND ? 9 : 6;  // values used per source
  __shared__ SrcRec<R> src[kChunk];
  const int b = blockIdx.x;
  const int it0 = blk_item[b], it1 = blk_item[b + 1];
  const int tile = items[it0].tile;
  const int tid = threadIdx.x;
  const int nt = tile_n[tile];
  const int di = tile_drop[tile];
  double tx[TPT], ty[TPT], tz[TPT], acc[TPT][3];
#pragma unroll
  for (int u = 0; u < TPT; ++u) {
    const int k = tid + u * NT;
    tx[u] = ty[u] = tz[u] = 0;
    acc[u][0] = acc[u][1] = acc[u][2] = 0;
    if (k < nt) {
      const long long t = tile_t0[tile] + k;
      const long long ng = ngd[di];
      const double* ri = rec_std + 7 * toff_std[di];
      const long long l = tgt_loc[t];
      tx[u] = ri[l];
      ty[u] = ri[ng + l];
      tz[u] = ri[2 * ng + l];
    }
  }
  for (int it = it0; it < it1; ++it) {
    const PairItem item = items[it];
    const int j = item.src_drop;
    bool act[TPT], any = false;
    R px[TPT], py[TPT], pz[TPT];
#pragma unroll
    for (int u = 0; u < TPT; ++u) {
      const int k = tid + u * NT;
      act[u] = k < nt && ((item.mask[k >> 5] >> (k & 31)) & 1u);
      any = any || act[u];
      px[u] = (R)(tx[u] - centre[3 * j]);
      py[u] = (R)(ty[u] - centre[3 * j + 1]);
      pz[u] = (R)(tz[u] - centre[3 * j + 2]);
    }
    const R* X = item.grid ? Xu : Xs;
    const R* N = item.grid ? Nu : Ns;
    const R* Q = item.grid ? Qu : Qs;
    const long long ld = item.grid ? nup : nstd;
    R s[TPT][3];
#pragma unroll
    for (int u = 0; u < TPT; ++u) s[u][0] = s[u][1] = s[u][2] = 0;
    for (long long c0 = item.s0; c0 < item.s1; c0 += kChunk) {
      const int cn = (int)min((long long)kChunk, item.s1 - c0);
      for (int k = tid; k < cn; k += NT) {
        const long long sidx = c0 + k;
        SrcRec<R> r;
        r.v[0] = X[sidx];
        r.v[1] = X[ld + sidx];
        r.v[2] = X[2 * ld + sidx];
        r.v[3] = Q[sidx];
        r.v[4] = Q[ld + sidx];
        r.v[5] = Q[2 * ld + sidx];
        if (KIND) {
          r.v[6] = N[sidx];
          r.v[7] = N[ld + sidx];
          r.v[8] = N[2 * ld + sidx];
        } else {
          r.v[6] = r.v[7] = r.v[8] = 0;
        }
        r.v[9] = r.v[10] = r.v[11] = 0;
        src[k] = r;
      }
      __syncthreads();
      if (any) {
        for (int k = 0; k < cn; ++k) {
          R v[12];
          // 128-bit shared-memory loads of the record (the double-layer record needs all three)
          typedef typename std::conditional<sizeof(R) == 4, float4, double2>::type V;
          constexpr int per = 16 / sizeof(R);
          constexpr int nv = (NR + per - 1) / per;
#pragma unroll
          for (int q = 0; q < nv; ++q) *reinterpret_cast<V*>(v + q * per) = reinterpret_cast<const V*>(&src[k])[q];
          const R xs_ = v[0], ys_ = v[1], zs_ = v[2], q0 = v[3], q1 = v[4], q2 = v[5];
#pragma unroll
          for (int u = 0; u < TPT; ++u) {
            const R dx = px[u] - xs_, dy = py[u] - ys_, dz = pz[u] - zs_;
            const R r2 = dx * dx + dy * dy + dz * dz;
            const R xq = dx * q0 + dy * q1 + dz * q2;
            if (KIND == 0) {  // Stokeslet
              const R ri = rsqrt_<R>(r2);
              const R c = xq * ri * ri * ri;
              s[u][0] += q0 * ri + c * dx;
              s[u][1] += q1 * ri + c * dy;
              s[u][2] += q2 * ri + c * dz;
            } else {  // stresslet, without its factor -6
              const R xn = dx * v[6] + dy * v[7] + dz * v[8];
              const R c = xq * xn * rsqrt5_<R>(r2);
              s[u][0] += c * dx;
              s[u][1] += c * dy;
              s[u][2] += c * dz;
            }
          }
        }
      }
      __syncthreads();
    }
    const double wj = KIND ? -6.0 * wts[j] : wts[j];
#pragma unroll
    for (int u = 0; u < TPT; ++u) {
      const double w = act[u] ? wj : 0.0;
      acc[u][0] += w * (double)s[u][0];
      acc[u][1] += w * (double)s[u][1];
      acc[u][2] += w * (double)s[u][2];
    }
  }
  double* pp = partial + (long long)b * 3 * kTile;
#pragma unroll
  for (int u = 0; u < TPT; ++u) {
    const int k = tid + u * NT;
    pp[k] = acc[u][0];
    pp[kTile + k] = acc[u][1];
    pp[2 * kTile + k] = acc[u][2];
  }
}

// ---- FP32 pair sums on packed lane pairs ----
// Two targets share one 64-bit register pair and every FP32 operation of their two pairs issues as
// one fma/mul/sub.rn.f32x2 instruction: half the issue slots of the scalar kernel for the same
// FP32-pipe work, which leaves room for the shared-memory loads and the two MUFU rsqrt of each
// source without starving the FMA pipe.  Rounding is that of the scalar operations (each lane is
// an IEEE round-to-nearest FP32 operation).
typedef unsigned long long fx2;  // lanes (lo, hi) = two FP32 values

__device__ __forceinline__ fx2 x2_pack(float lo, float hi) {
  fx2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void x2_unpack(fx2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ fx2 x2_add(fx2 a, fx2 b) {
  fx2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ fx2 x2_sub(fx2 a, fx2 b) {
  fx2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ fx2 x2_mul(fx2 a, fx2 b) {
  fx2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ fx2 x2_fma(fx2 a, fx2 b, fx2 c) {
  fx2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ fx2 x2_rsqrt(fx2 v) {
  float lo, hi;
  x2_unpack(v, lo, hi);
  return x2_pack(rsqrt_est(lo), rsqrt_est(hi));
}

constexpr int kChunkX2 = 64;  // sources staged per pass of the packed kernel
// Sources per FP32 sum.  One sum per item (up to 4096 terms) was less accurate than the scalar kernel's, since the packed
// form adds the two parts of a Stokeslet to it one by one: velocity at points among 64 drops of degree 24 3.4e-8
// (scalar, the tuned variant there once) and 3.7e-8, now 2.7e-8 at the same time (256 sources: 2.5e-8, 0.3 % slower).
constexpr int kFlushX2 = 512;

// Staged source of the packed kernel: each value duplicated into both lanes, in the order
// x, y, z, q0, q1, q2, n0, n1, n2 (and one pad), read with 128-bit shared-memory loads (three for
// the single layer, five for the double layer).
struct alignas(16) SrcRecX2 {
  fx2 v[10];
};

// Same work list, layout and result as k_interdrop<float, KIND, TPT>; TPT even, the thread's
// targets tid + u * (128/TPT) taken two by two (u = 2w, 2w + 1 share lane pair w).  The tile's target
// coordinates and the FP64 accumulators live in shared memory, not in registers, so that more warps fit per SM; the
// source loop takes two sources per iteration (2 x TPT/2 independent chains per thread).  PF = 1 software-pipelines the staging: the next chunk's sources are loaded
// into registers while the current chunk is summed, so the global-memory latency of the staging
// overlaps the arithmetic.
template <int KIND, int TPT, int PF, int CH = kChunkX2>
__global__ void __launch_bounds__(kTile / TPT) k_interdrop_x2(
    const PairItem* __restrict__ items, const int* __restrict__ blk_item, const long long* __restrict__ tile_t0,
    const int* __restrict__ tile_n, const int* __restrict__ tile_drop, const long long* __restrict__ tgt_loc,
    const long long* __restrict__ toff_std, const int* __restrict__ ngd, const double* __restrict__ rec_std,
    const double* __restrict__ centre, const float* __restrict__ Xs, const float* __restrict__ Ns,
    const float* __restrict__ Qs, long long nstd, const float* __restrict__ Xu, const float* __restrict__ Nu,
    const float* __restrict__ Qu, long long nup, const double* __restrict__ wts, double* __restrict__ partial) {
  static_assert(TPT % 2 == 0, "targets are taken in lane pairs");
  constexpr int NT = kTile / TPT;
  constexpr int NW = TPT / 2;  // lane pairs per thread
  constexpr int NV = KIND ? 9 : 6;
  constexpr int nv = (NV + 1) / 2;  // 128-bit loads per staged source
  static_assert(CH % NT == 0 && CH >= NT, "a chunk is a whole number of sources per thread");
  constexpr int RPT = CH / NT;  // staged sources per thread and chunk
  __shared__ SrcRecX2 src[CH];
  __shared__ double tgt[3][kTile];  // the tile's targets
  __shared__ double acc[3][kTile];  // per-target sums over the block's items
  const int b = blockIdx.x;
  const int it0 = blk_item[b], it1 = blk_item[b + 1];
  const int tile = items[it0].tile;
  const int tid = threadIdx.x;
  const int nt = tile_n[tile];
  const int di = tile_drop[tile];
  {
    const long long ng = ngd[di];
    const double* ri = rec_std + 7 * toff_std[di];
    for (int k = tid; k < kTile; k += NT) {
      const long long l = tgt_loc[tile_t0[tile] + (k < nt ? k : 0)];
      for (int c = 0; c < 3; ++c) {
        tgt[c][k] = ri[c * ng + l];
        acc[c][k] = 0.0;
      }
    }
  }
  // the block's shared arrays are written before any thread reads them (the first staging barrier
  // below comes after the target loads; each thread reads only its own targets' entries)
  __syncthreads();
  // sources c0 + tid + r NT of a chunk, r < RPT (zero past the item's end: zero weight)
  auto load_chunk = [&](float (&v)[RPT][NV], const float* X, const float* N, const float* Q, long long ld,
                        long long c0, long long s1) {
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
      const long long sidx = c0 + tid + r * NT;
#pragma unroll
      for (int q = 0; q < NV; ++q) v[r][q] = 0.f;
      if (sidx < s1) {
        v[r][0] = X[sidx];
        v[r][1] = X[ld + sidx];
        v[r][2] = X[2 * ld + sidx];
        v[r][3] = Q[sidx];
        v[r][4] = Q[ld + sidx];
        v[r][5] = Q[2 * ld + sidx];
        if (KIND) {
          v[r][6] = N[sidx];
          v[r][7] = N[ld + sidx];
          v[r][8] = N[2 * ld + sidx];
        }
      }
    }
  };
  auto store_chunk = [&](const float (&v)[RPT][NV]) {
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
      SrcRecX2 rec;
#pragma unroll
      for (int q = 0; q < NV; ++q) rec.v[q] = x2_pack(v[r][q], v[r][q]);
#pragma unroll
      for (int q = NV; q < 10; ++q) rec.v[q] = 0ull;
      src[tid + r * NT] = rec;
    }
  };
  for (int it = it0; it < it1; ++it) {
    const int j = items[it].src_drop;
    unsigned act = 0u;  // bit u: target tid + u * NT is in this item
#pragma unroll
    for (int u = 0; u < TPT; ++u) {
      const int k = tid + u * NT;
      if (k < nt && ((items[it].mask[k >> 5] >> (k & 31)) & 1u)) act |= 1u << u;
    }
    // targets relative to the source drop's centre, rounded to FP32 once
    const double cx = centre[3 * j], cy = centre[3 * j + 1], cz = centre[3 * j + 2];
    fx2 px[NW], py[NW], pz[NW], s[NW][3];
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const int k0 = tid + 2 * w * NT, k1 = k0 + NT;
      px[w] = x2_pack((float)(tgt[0][k0] - cx), (float)(tgt[0][k1] - cx));
      py[w] = x2_pack((float)(tgt[1][k0] - cy), (float)(tgt[1][k1] - cy));
      pz[w] = x2_pack((float)(tgt[2][k0] - cz), (float)(tgt[2][k1] - cz));
      s[w][0] = s[w][1] = s[w][2] = 0ull;  // +0.0f in both lanes
    }
    const int grid = items[it].grid;
    const float* X = grid ? Xu : Xs;
    const float* N = grid ? Nu : Ns;
    const float* Q = grid ? Qu : Qs;
    const long long ld = grid ? nup : nstd;
    const long long s0 = items[it].s0, s1 = items[it].s1;
    // the FP32 sums go to the FP64 ones of the block after every kFlushX2 sources
    const double wj = KIND ? -6.0 * wts[j] : wts[j];
    auto flush = [&]() {
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const int k0 = tid + 2 * w * NT, k1 = k0 + NT;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float lo, hi;
          x2_unpack(s[w][c], lo, hi);
          if (act & (1u << (2 * w))) acc[c][k0] += wj * (double)lo;
          if (act & (1u << (2 * w + 1))) acc[c][k1] += wj * (double)hi;
          s[w][c] = 0ull;
        }
      }
    };
    float pre[RPT][NV];
    if (PF) load_chunk(pre, X, N, Q, ld, s0, s1);
    for (long long c0 = s0; c0 < s1; c0 += CH) {
      const int cn = (int)min((long long)CH, s1 - c0);
      if (!PF) load_chunk(pre, X, N, Q, ld, c0, s1);
      store_chunk(pre);
      __syncthreads();
      if (PF && c0 + CH < s1) load_chunk(pre, X, N, Q, ld, c0 + CH, s1);  // next chunk, in flight
      if (act) {
        const int cn2 = (cn + 1) & ~1;
        for (int k = 0; k < cn2; k += 2) {
          fx2 va[10], vb[10];
#pragma unroll
          for (int q = 0; q < nv; ++q) {
            *reinterpret_cast<ulonglong2*>(va + 2 * q) = reinterpret_cast<const ulonglong2*>(&src[k])[q];
            *reinterpret_cast<ulonglong2*>(vb + 2 * q) = reinterpret_cast<const ulonglong2*>(&src[k + 1])[q];
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const fx2* v = h ? vb : va;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
              const fx2 dx = x2_sub(px[w], v[0]), dy = x2_sub(py[w], v[1]), dz = x2_sub(pz[w], v[2]);
              const fx2 r2 = x2_fma(dz, dz, x2_fma(dy, dy, x2_mul(dx, dx)));
              const fx2 ri = x2_rsqrt(r2);
              const fx2 xq = x2_fma(dz, v[5], x2_fma(dy, v[4], x2_mul(dx, v[3])));
              const fx2 ri2 = x2_mul(ri, ri);
              if (KIND == 0) {  // Stokeslet: q/r + (xh.q) xh/r^3
                const fx2 c = x2_mul(x2_mul(xq, ri2), ri);
                s[w][0] = x2_fma(c, dx, x2_fma(v[3], ri, s[w][0]));
                s[w][1] = x2_fma(c, dy, x2_fma(v[4], ri, s[w][1]));
                s[w][2] = x2_fma(c, dz, x2_fma(v[5], ri, s[w][2]));
              } else {  // stresslet without its factor -6: (xh.q)(xh.n) xh/r^5
                const fx2 xn = x2_fma(dz, v[8], x2_fma(dy, v[7], x2_mul(dx, v[6])));
                const fx2 c = x2_mul(x2_mul(x2_mul(x2_mul(xq, xn), ri2), ri2), ri);
                s[w][0] = x2_fma(c, dx, s[w][0]);
                s[w][1] = x2_fma(c, dy, s[w][1]);
                s[w][2] = x2_fma(c, dz, s[w][2]);
              }
            }
          }
        }
        if ((c0 - s0) % kFlushX2 == kFlushX2 - CH) flush();
      }
      __syncthreads();
    }
    flush();
  }
  double* pp = partial + (long long)b * 3 * kTile;
#pragma unroll
  for (int u = 0; u < TPT; ++u) {
    const int k = tid + u * NT;
    pp[k] = acc[0][k];
    pp[kTile + k] = acc[1][k];
    pp[2 * kTile + k] = acc[2][k];
  }
}

// ---- double-float pair sums ----
// A double-float value is an unevaluated sum h + l of two FP32 numbers (about 44 significant bits).
// Every operation runs on the FP32 pipe, packed for two targets at a time (fma/mul/add/sub.rn.f32x2): the
// kernel is bound by that pipe's operations, and the packed form leaves half of the issue slots for the
// shared-memory loads and the rest.  Sums use Knuth's TwoSum, products the FMA-based TwoProduct; results are
// left unnormalised (l may exceed ulp(h)/2 by a few units, which costs no accuracy in the short chains of
// one pair) and the per-target sums are renormalised after every staged chunk.  1/r^3 and 1/r^5 come from
// the estimate y of 1/r directly: with e = 1 - r^2 y^2 (about 2^-22),
// r^-k = y^k (1 - e)^(-k/2) = y^k (1 + (k/2) e + (k/2)(k/2 + 1)/2 e^2 + O(e^3)).
// About 170 operations per pair; scalar, the kernel reached 67% of the pipe at 75% of the issue slots.  80
// drops of degree 24 (1.0e10 pairs): 90.4 -> 68.7 ms.  Rounding the high parts of positions to a common grid,
// so that their difference is exact in one operation, saved another tenth but lost accuracy where the points of
// a tile lie at very different distances (3.9e-11 of the field at some fluid points, over the 1e-11 that
// double-float sums are to keep), and was left out.
struct d2 {
  fx2 h, l;
};
struct df2 {
  float h, l;
};

__device__ __forceinline__ fx2 x2_neg(fx2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ fx2 x2_both(float v) { return x2_pack(v, v); }
__device__ inline df2 df_from(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ d2 d2_add(d2 a, d2 b) {
  const fx2 s = x2_add(a.h, b.h), v = x2_sub(s, a.h);
  return {s, x2_add(x2_add(x2_add(x2_sub(a.h, x2_sub(s, v)), x2_sub(b.h, v)), a.l), b.l)};
}
__device__ __forceinline__ d2 d2_sub(d2 a, d2 b) {
  const fx2 s = x2_sub(a.h, b.h), v = x2_sub(s, a.h);
  return {s, x2_sub(x2_add(x2_sub(x2_sub(a.h, x2_sub(s, v)), x2_add(b.h, v)), a.l), b.l)};
}
__device__ __forceinline__ d2 d2_renorm(d2 a) {
  const fx2 s = x2_add(a.h, a.l), v = x2_sub(s, a.h);
  return {s, x2_add(x2_sub(a.h, x2_sub(s, v)), x2_sub(a.l, v))};
}
__device__ __forceinline__ d2 d2_mul(d2 a, d2 b) {
  const fx2 p = x2_mul(a.h, b.h);
  return {p, x2_fma(a.l, b.h, x2_fma(a.h, b.l, x2_fma(a.h, b.h, x2_neg(p))))};
}
__device__ __forceinline__ d2 d2_sqr(d2 a) {
  const fx2 p = x2_mul(a.h, a.h);
  return {p, x2_fma(x2_add(a.h, a.h), a.l, x2_fma(a.h, a.h, x2_neg(p)))};
}
// a b for b without a low part
__device__ __forceinline__ d2 d2_mul1(d2 a, fx2 b) {
  const fx2 p = x2_mul(a.h, b);
  return {p, x2_fma(a.l, b, x2_fma(a.h, b, x2_neg(p)))};
}

// Same work list and result as k_interdrop; the sources are read in FP64 and split as they are staged, each
// part duplicated in both lanes; the thread's targets tid and tid + 64 share the lanes.
template <int KIND>
__global__ void __launch_bounds__(kTile / 2) k_interdrop_df(
    const PairItem* __restrict__ items, const int* __restrict__ blk_item, const long long* __restrict__ tile_t0,
    const int* __restrict__ tile_n, const int* __restrict__ tile_drop, const long long* __restrict__ tgt_loc,
    const long long* __restrict__ toff_std, const int* __restrict__ ngd, const double* __restrict__ rec_std,
    const double* __restrict__ centre, const double* __restrict__ Xs, const double* __restrict__ Ns,
    const double* __restrict__ Qs, long long nstd, const double* __restrict__ Xu, const double* __restrict__ Nu,
    const double* __restrict__ Qu, long long nup, const double* __restrict__ wts, double* __restrict__ partial) {
  constexpr int NT = kTile / 2;
  constexpr int NV = KIND ? 9 : 6;  // staged values per source: x, q (and n)
  __shared__ __align__(16) d2 sv[NV][kChunk];
  const int b = blockIdx.x;
  const int it0 = blk_item[b], it1 = blk_item[b + 1];
  const int tile = items[it0].tile;
  const int tid = threadIdx.x;
  const int nt = tile_n[tile];
  const int di = tile_drop[tile];
  double tx[2][3], acc[2][3];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int k = tid + u * NT;
    const long long ng = ngd[di];
    const double* ri = rec_std + 7 * toff_std[di] + tgt_loc[tile_t0[tile] + (k < nt ? k : 0)];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      tx[u][c] = ri[c * ng];
      acc[u][c] = 0;
    }
  }
  for (int it = it0; it < it1; ++it) {
    const PairItem item = items[it];
    const int j = item.src_drop;
    bool act[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int k = tid + u * NT;
      act[u] = k < nt && ((item.mask[k >> 5] >> (k & 31)) & 1u);
    }
    d2 px[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const df2 a = df_from(tx[0][c] - centre[3 * j + c]), e = df_from(tx[1][c] - centre[3 * j + c]);
      px[c] = {x2_pack(a.h, e.h), x2_pack(a.l, e.l)};
    }
    const double* X = item.grid ? Xu : Xs;
    const double* N = item.grid ? Nu : Ns;
    const double* Q = item.grid ? Qu : Qs;
    const long long ld = item.grid ? nup : nstd;
    d2 s[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) s[c] = {0ull, 0ull};
    for (long long c0 = item.s0; c0 < item.s1; c0 += kChunk) {
      const int cn = (int)min((long long)kChunk, item.s1 - c0);
      for (int k = tid; k < cn; k += NT) {
        const long long sidx = c0 + k;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const df2 x = df_from(X[c * ld + sidx]), q = df_from(Q[c * ld + sidx]);
          sv[c][k] = {x2_both(x.h), x2_both(x.l)};
          sv[3 + c][k] = {x2_both(q.h), x2_both(q.l)};
          if (KIND) {
            const df2 n = df_from(N[c * ld + sidx]);
            sv[6 + c][k] = {x2_both(n.h), x2_both(n.l)};
          }
        }
      }
      __syncthreads();
      if (act[0] || act[1]) {
        for (int k = 0; k < cn; ++k) {
          d2 dx[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) dx[c] = d2_sub(px[c], sv[c][k]);
          const d2 r2 = d2_add(d2_add(d2_sqr(dx[0]), d2_sqr(dx[1])), d2_sqr(dx[2]));
          const fx2 y = x2_rsqrt(r2.h);
          const fx2 yy = x2_mul(y, y);
          const d2 y2 = {yy, x2_fma(y, y, x2_neg(yy))};
          const d2 ay2 = d2_mul(r2, y2);
          const fx2 e = x2_sub(x2_sub(x2_both(1.0f), ay2.h), ay2.l);
          const d2 q0 = sv[3][k], q1 = sv[4][k], q2 = sv[5][k];
          const d2 xq = d2_add(d2_add(d2_mul(dx[0], q0), d2_mul(dx[1], q1)), d2_mul(dx[2], q2));
          if (KIND == 0) {  // Stokeslet: q/r + (xh.q) xh/r^3
            const fx2 t1 = x2_mul(e, x2_fma(x2_both(0.375f), e, x2_both(0.5f)));
            const fx2 t3 = x2_mul(e, x2_fma(x2_both(1.875f), e, x2_both(1.5f)));
            const d2 ri = {y, x2_mul(y, t1)};
            d2 c3 = d2_mul1(y2, y);
            c3.l = x2_fma(c3.h, t3, c3.l);
            const d2 c = d2_mul(xq, c3);
            s[0] = d2_add(s[0], d2_add(d2_mul(q0, ri), d2_mul(c, dx[0])));
            s[1] = d2_add(s[1], d2_add(d2_mul(q1, ri), d2_mul(c, dx[1])));
            s[2] = d2_add(s[2], d2_add(d2_mul(q2, ri), d2_mul(c, dx[2])));
          } else {  // stresslet without its factor -6: (xh.q)(xh.n) xh/r^5
            const fx2 t5 = x2_mul(e, x2_fma(x2_both(4.375f), e, x2_both(2.5f)));
            d2 c5 = d2_mul1(d2_sqr(y2), y);
            c5.l = x2_fma(c5.h, t5, c5.l);
            const d2 xn = d2_add(d2_add(d2_mul(dx[0], sv[6][k]), d2_mul(dx[1], sv[7][k])), d2_mul(dx[2], sv[8][k]));
            const d2 c = d2_mul(d2_mul(xq, xn), c5);
#pragma unroll
            for (int a = 0; a < 3; ++a) s[a] = d2_add(s[a], d2_mul(c, dx[a]));
          }
        }
      }
      __syncthreads();
#pragma unroll
      for (int c = 0; c < 3; ++c) s[c] = d2_renorm(s[c]);
    }
    const double wj = KIND ? -6.0 * wts[j] : wts[j];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float h0, h1, l0, l1;
      x2_unpack(s[c].h, h0, h1);
      x2_unpack(s[c].l, l0, l1);
      if (act[0]) acc[0][c] += wj * ((double)h0 + (double)l0);
      if (act[1]) acc[1][c] += wj * ((double)h1 + (double)l1);
    }
  }
  double* pp = partial + (long long)b * 3 * kTile;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int c = 0; c < 3; ++c) pp[c * kTile + tid + u * NT] = acc[u][c];
}

// Per (tile, source drop j): the tile's targets in Omega_0, Omega_1 and Omega_2 of drop j as 128-bit
// masks, and whether any target lies inside drop j.  Consecutive threads take consecutive j, so the
// region reads of one target are coalesced.
__global__ void k_tile_masks(const unsigned char* __restrict__ region, int nd, const long long* __restrict__ tile_t0,
                             const int* __restrict__ tile_n, long long ntile, TileMask* __restrict__ out) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= ntile * nd) return;
  const long long ti = idx / nd;
  const int j = (int)(idx - ti * nd);
  TileMask m{};
  const long long t0 = tile_t0[ti];
  const int n = tile_n[ti];
  for (int k = 0; k < n; ++k) {
    const unsigned char r = region[(t0 + k) * nd + j];
    if (r < 3) m.m[r][k >> 5] |= 1u << (k & 31);
    else if (r == 3) m.inside = 1;
  }
  out[idx] = m;
}

// vals += sum of the partials of the tile's blocks; PARTS threads per (tile, component, target), each on every
// PARTS-th block.  With one thread a small batch, whose tiles are split over a hundred blocks each, waits for
// fifteen dependent groups of loads: 8 drops of degree 16 11.4 -> 8.1 us.
constexpr int kRedThreads = 256, kRedParts = 8;

template <int PARTS>
__global__ void __launch_bounds__(kRedThreads) k_reduce_tiles(
    const double* __restrict__ partial, const int* __restrict__ tile_blk, const long long* __restrict__ tile_t0,
    const int* __restrict__ tile_n, const int* __restrict__ tile_drop, const long long* __restrict__ tgt_loc,
    const long long* __restrict__ val_off, const int* __restrict__ ngd, int ntile, double* __restrict__ vals) {
  constexpr int OUT = kRedThreads / PARTS;  // a divisor of kTile: the block's outputs lie in one tile
  __shared__ double part[PARTS][OUT];
  const int o = threadIdx.x % OUT, k = threadIdx.x / OUT;
  const long long idx = (long long)blockIdx.x * OUT + o;
  const int tile = (int)(idx / (3 * kTile)), r = (int)(idx - 3LL * tile * kTile), c = r / kTile, tid = r - c * kTile;
  const bool in = tile < ntile && tid < tile_n[tile];
  const int b0 = in ? tile_blk[tile] : 0, b1 = in ? tile_blk[tile + 1] : 0;
  double a = 0;
#pragma unroll 8
  for (int b = b0 + k; b < b1; b += PARTS) a += partial[3LL * kTile * b + r];
  if (PARTS > 1) {
    part[k][o] = a;
    __syncthreads();
    if (k > 0) return;
    for (int i = 1; i < PARTS; ++i) a += part[i][o];
  }
  if (b0 == b1) return;
  const int d = tile_drop[tile];
  vals[val_off[d] + (long long)c * ngd[d] + tgt_loc[tile_t0[tile] + tid]] += a;
}

// Per drop of a degree group (blockIdx.y; records of N points at rec + 7 off[i]): sum_s x.n wJ (for the
// volume) and max_s |x - c| over each of 64 blocks, out[i][block][2].
__global__ void k_drop_stats(const double* __restrict__ rec, const long long* __restrict__ off,
                             const int* __restrict__ ids, const double* __restrict__ centre, long long N,
                             double* __restrict__ out) {
  __shared__ double sv[kThreads], sm[kThreads];
  rec += 7 * off[blockIdx.y];
  out += (long long)blockIdx.y * 2 * gridDim.x;
  const double *c = centre + 3 * ids[blockIdx.y], cx = c[0], cy = c[1], cz = c[2];
  double v = 0, mx = 0;
  for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < N; s += (long long)gridDim.x * blockDim.x) {
    const double x = rec[s], y = rec[N + s], z = rec[2 * N + s];
    v += (x * rec[3 * N + s] + y * rec[4 * N + s] + z * rec[5 * N + s]) * rec[6 * N + s];
    const double dx = x - cx, dy = y - cy, dz = z - cz;
    mx = fmax(mx, sqrt(dx * dx + dy * dy + dz * dz));
  }
  sv[threadIdx.x] = v;
  sm[threadIdx.x] = mx;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sv[threadIdx.x] += sv[threadIdx.x + o];
      sm[threadIdx.x] = fmax(sm[threadIdx.x], sm[threadIdx.x + o]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[2 * blockIdx.x] = sv[0];
    out[2 * blockIdx.x + 1] = sm[0];
  }
}

// SoA source positions relative to the drop centres and normals in both precisions, for the nd drops of a
// degree group (records of N points at rec + 7 off[i], sources at off[i])
__global__ void k_source_geometry(const double* __restrict__ rec, const long long* __restrict__ off,
                                  const int* __restrict__ ids, const double* __restrict__ centre, long long nd,
                                  long long N, double* __restrict__ X64, double* __restrict__ N64,
                                  float* __restrict__ X32, float* __restrict__ N32, long long ld) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= nd * N) return;
  const long long d = idx / N, s = idx - d * N, o = off[d] + s;
  const double* r = rec + 7 * off[d] + s;
  for (int c = 0; c < 3; ++c) {
    const double x = r[c * N] - centre[3 * ids[d] + c], n = r[(3 + c) * N];
    X64[c * ld + o] = x;
    N64[c * ld + o] = n;
    X32[c * ld + o] = (float)x;
    N32[c * ld + o] = (float)n;
  }
}

}  // namespace

int launch_classify(const double* rec_std, long long ntarget, const int* tdrop, const long long* tloc,
                    const long long* toff_std, const int* ngd, int ndrop, const double* centre, const double* bound,
                    const double* h, double a_tilde, const double* rec_up, const long long* up_off,
                    const long long* up_n, unsigned char* region, cudaStream_t s) {
  long long n = ntarget * ndrop;
  if (n == 0) return BIE_OK;
  k_classify<<<blocks_for(n), kThreads, 0, s>>>(rec_std, ntarget, tdrop, tloc, toff_std, ngd, ndrop, centre, bound, h,
                                                a_tilde, rec_up, up_off, up_n, region);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

template <typename R, int TPT, int PF = 0, int CH = kChunkX2>
static void interdrop_kernel(int kind, int nblk, const PairItem* items, const int* blk_item, const long long* tile_t0,
                             const int* tile_n, const int* tile_drop, const long long* tgt_loc,
                             const long long* toff_std, const int* ngd, const double* rec_std, const double* centre,
                             const R* Xs, const R* Ns, const R* Qs, long long nstd, const R* Xu, const R* Nu,
                             const R* Qu, long long nup, const double* wts, double* partial, cudaStream_t s) {
  if constexpr (std::is_same<R, float>::value && TPT % 2 == 0) {
    // FP32 with two or more targets per thread: packed lane pairs
    if (kind == 0)
      k_interdrop_x2<0, TPT, PF, CH><<<nblk, kTile / TPT, 0, s>>>(items, blk_item, tile_t0, tile_n, tile_drop, tgt_loc,
                                                              toff_std, ngd, rec_std, centre, Xs, Ns, Qs, nstd, Xu,
                                                              Nu, Qu, nup, wts, partial);
    else
      k_interdrop_x2<1, TPT, PF, CH><<<nblk, kTile / TPT, 0, s>>>(items, blk_item, tile_t0, tile_n, tile_drop, tgt_loc,
                                                              toff_std, ngd, rec_std, centre, Xs, Ns, Qs, nstd, Xu,
                                                              Nu, Qu, nup, wts, partial);
    return;
  }
  if (kind == 0)
    k_interdrop<R, 0, TPT><<<nblk, kTile / TPT, 0, s>>>(items, blk_item, tile_t0, tile_n, tile_drop, tgt_loc,
                                                        toff_std, ngd, rec_std, centre, Xs, Ns, Qs, nstd, Xu, Nu, Qu,
                                                        nup, wts, partial);
  else
    k_interdrop<R, 1, TPT><<<nblk, kTile / TPT, 0, s>>>(items, blk_item, tile_t0, tile_n, tile_drop, tgt_loc,
                                                        toff_std, ngd, rec_std, centre, Xs, Ns, Qs, nstd, Xu, Nu, Qu,
                                                        nup, wts, partial);
}

template <typename R>
int launch_interdrop(int kind, int tpt, int nblk, const PairItem* items, const int* blk_item, const long long* tile_t0,
                     const int* tile_n, const int* tile_drop, const long long* tgt_loc, const long long* toff_std,
                     const int* ngd, const double* rec_std, const double* centre, const R* Xs, const R* Ns,
                     const R* Qs, long long nstd, const R* Xu, const R* Nu, const R* Qu, long long nup,
                     const double* wts, double* partial, cudaStream_t s) {
  if (nblk == 0) return BIE_OK;
  if (std::is_same<R, float>::value && (tpt == 12 || tpt == 14 || tpt == 24 || tpt == 34)) {
    // packed FP32: 12, 14 = 2 or 4 targets per thread with pipelined staging; 24, 34 = 4 targets per
    // thread with 32-source chunks, without and with pipelined staging
    if (tpt == 12)
      interdrop_kernel<R, 2, 1>(kind, nblk, items, blk_item, tile_t0, tile_n, tile_drop, tgt_loc, toff_std, ngd,
                                rec_std, centre, Xs, Ns, Qs, nstd, Xu, Nu, Qu, nup, wts, partial, s);
    else if (tpt == 14)
      interdrop_kernel<R, 4, 1>(kind, nblk, items, blk_item, tile_t0, tile_n, tile_drop, tgt_loc, toff_std, ngd,
                                rec_std, centre, Xs, Ns, Qs, nstd, Xu, Nu, Qu, nup, wts, partial, s);
    else if (tpt == 24)
      interdrop_kernel<R, 4, 0, 32>(kind, nblk, items, blk_item, tile_t0, tile_n, tile_drop, tgt_loc, toff_std, ngd,
                                    rec_std, centre, Xs, Ns, Qs, nstd, Xu, Nu, Qu, nup, wts, partial, s);
    else
      interdrop_kernel<R, 4, 1, 32>(kind, nblk, items, blk_item, tile_t0, tile_n, tile_drop, tgt_loc, toff_std, ngd,
                                    rec_std, centre, Xs, Ns, Qs, nstd, Xu, Nu, Qu, nup, wts, partial, s);
    count_launch();
    BIE_CUDA_TRY(cudaGetLastError());
    return BIE_OK;
  }
  if (tpt == 1)
    interdrop_kernel<R, 1>(kind, nblk, items, blk_item, tile_t0, tile_n, tile_drop, tgt_loc, toff_std, ngd, rec_std,
                           centre, Xs, Ns, Qs, nstd, Xu, Nu, Qu, nup, wts, partial, s);
  else if (tpt == 4)
    interdrop_kernel<R, 4>(kind, nblk, items, blk_item, tile_t0, tile_n, tile_drop, tgt_loc, toff_std, ngd, rec_std,
                           centre, Xs, Ns, Qs, nstd, Xu, Nu, Qu, nup, wts, partial, s);
  else
    interdrop_kernel<R, 2>(kind, nblk, items, blk_item, tile_t0, tile_n, tile_drop, tgt_loc, toff_std, ngd, rec_std,
                           centre, Xs, Ns, Qs, nstd, Xu, Nu, Qu, nup, wts, partial, s);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_interdrop_df(int kind, int nblk, const PairItem* items, const int* blk_item, const long long* tile_t0,
                        const int* tile_n, const int* tile_drop, const long long* tgt_loc, const long long* toff_std,
                        const int* ngd, const double* rec_std, const double* centre, const double* Xs,
                        const double* Ns, const double* Qs, long long nstd, const double* Xu, const double* Nu,
                        const double* Qu, long long nup, const double* wts, double* partial, cudaStream_t s) {
  if (nblk == 0) return BIE_OK;
  auto kern = kind == 0 ? k_interdrop_df<0> : k_interdrop_df<1>;
  kern<<<nblk, kTile / 2, 0, s>>>(items, blk_item, tile_t0, tile_n, tile_drop, tgt_loc, toff_std, ngd, rec_std,
                                    centre, Xs, Ns, Qs, nstd, Xu, Nu, Qu, nup, wts, partial);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_tile_masks(const unsigned char* region, int nd, const long long* tile_t0, const int* tile_n,
                      long long ntile, TileMask* out, cudaStream_t s) {
  const long long n = ntile * nd;
  if (n == 0) return BIE_OK;
  k_tile_masks<<<blocks_for(n), kThreads, 0, s>>>(region, nd, tile_t0, tile_n, ntile, out);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_reduce_tiles(const double* partial, const int* tile_blk, const long long* tile_t0, const int* tile_n,
                        const int* tile_drop, const long long* tgt_loc, const long long* val_off, const int* ngd,
                        int ntile, long long nblk, double* vals, cudaStream_t s) {
  if (ntile == 0) return BIE_OK;
  // a long list of blocks per tile is split; short lists (2.6 blocks per tile at 192 drops of degree 24) leave
  // nothing to split and eight times the threads
  const bool split = nblk >= 2LL * kRedParts * ntile;
  const long long out = kRedThreads / (split ? kRedParts : 1), n = (3LL * ntile * kTile + out - 1) / out;
  if (n > 0x7fffffffLL) return BIE_EINVAL;
  auto kern = split ? k_reduce_tiles<kRedParts> : k_reduce_tiles<1>;
  kern<<<(unsigned)n, kRedThreads, 0, s>>>(partial, tile_blk, tile_t0, tile_n, tile_drop, tgt_loc, val_off, ngd, ntile,
                                           vals);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int launch_drop_stats(const double* rec, const long long* off, const int* ids, const double* centre, long long nd,
                      long long N, double* out, cudaStream_t s) {
  for (long long i = 0; i < nd; i += 65535) {
    k_drop_stats<<<dim3(64, (unsigned)(nd - i < 65535 ? nd - i : 65535)), kThreads, 0, s>>>(rec, off + i, ids + i, centre,
                                                                                           N, out + 128 * i);
    count_launch();
    BIE_CUDA_TRY(cudaGetLastError());
  }
  return BIE_OK;
}

int launch_source_geometry(const double* rec, const long long* off, const int* ids, const double* centre, long long nd,
                           long long N, double* X64, double* N64, float* X32, float* N32, long long ld,
                           cudaStream_t s) {
  if (nd * N == 0) return BIE_OK;
  k_source_geometry<<<blocks_for(nd * N), kThreads, 0, s>>>(rec, off, ids, centre, nd, N, X64, N64, X32, N32, ld);
  count_launch();
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

template int launch_interdrop<double>(int, int, int, const PairItem*, const int*, const long long*, const int*,
                                      const int*, const long long*, const long long*, const int*, const double*,
                                      const double*, const double*, const double*, const double*, long long,
                                      const double*, const double*, const double*, long long, const double*, double*,
                                      cudaStream_t);
template int launch_interdrop<float>(int, int, int, const PairItem*, const int*, const long long*, const int*, const int*,
                                     const long long*, const long long*, const int*, const double*, const double*,
                                     const float*, const float*, const float*, long long, const float*, const float*,
                                     const float*, long long, const double*, double*, cudaStream_t);
}  // namespace bie

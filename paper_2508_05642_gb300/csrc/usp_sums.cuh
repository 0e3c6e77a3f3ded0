// usp_sums.cuh -- the FP64 particle sums behind the moments of Sec. 2.A in one
// pass over the particles: sums of d = c - w about a reference velocity w near
// the cell mean, from which the central moments follow exactly.
#pragma once

#include <cuda_runtime.h>

#include "usp_device.cuh"

namespace usp {

// S_k = sum d_k | Q = sum d_i d_j (xx yy zz xy xz yz) | T_k = sum |d|^2 d_k |
// E_k = sum d_k eps | L_k = sum d_k I | sum eps | sum I
enum { kRS = 0, kRQ = 3, kRT = 9, kRE = 12, kRL = 15, kRe = 18, kRI = 19, kRawN = 20 };

// One particle: 19 FP64 operations, 4 more for an excited level (the level
// sum stays an integer).  Two passes (means, then central sums) take 34 and
// read the state twice.
__device__ __forceinline__ void raw_add(double* a, long long& aI, double d0, double d1, double d2,
                                        double e, int l) {
  a[kRS] += d0; a[kRS + 1] += d1; a[kRS + 2] += d2;
  a[kRQ] = fma(d0, d0, a[kRQ]); a[kRQ + 1] = fma(d1, d1, a[kRQ + 1]);
  a[kRQ + 2] = fma(d2, d2, a[kRQ + 2]); a[kRQ + 3] = fma(d0, d1, a[kRQ + 3]);
  a[kRQ + 4] = fma(d0, d2, a[kRQ + 4]); a[kRQ + 5] = fma(d1, d2, a[kRQ + 5]);
  const double q = fma(d0, d0, fma(d1, d1, d2 * d2));
  a[kRT] = fma(q, d0, a[kRT]); a[kRT + 1] = fma(q, d1, a[kRT + 1]);
  a[kRT + 2] = fma(q, d2, a[kRT + 2]);
  a[kRE] = fma(d0, e, a[kRE]); a[kRE + 1] = fma(d1, e, a[kRE + 1]);
  a[kRE + 2] = fma(d2, e, a[kRE + 2]);
  a[kRe] += e;
  if (l != 0) {
    const double li = (double)l;
    a[kRL] = fma(d0, li, a[kRL]); a[kRL + 1] = fma(d1, li, a[kRL + 1]);
    a[kRL + 2] = fma(d2, li, a[kRL + 2]);
    aI += l;
  }
}

// The reference velocity of a cell of n particles: the FP32 mean of 32 of them
// taken at equal distances (every caller of a cell gets the same one), 0 where
// that is not finite.  It is within about 0.2 thermal speeds of the mean, so
// the shifted sums lose no digit, and exact in FP64 whatever its value.
struct RawRef {
  double w[3];
};
template <typename Load>
__device__ __forceinline__ double raw_mean32(long long n, Load load) {
  const int lane = threadIdx.x & 31;
  const int m = n < 32 ? (int)n : 32;
  float v = lane < m ? (float)load((long long)lane * n / m) : 0.0f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  v = __fdiv_rn(v, (float)m);
  return fabsf(v) < 3.0e38f ? (double)v : 0.0;
}

__device__ __forceinline__ RawRef raw_reference(long long b, long long n,
                                                const double* __restrict__ cx,
                                                const double* __restrict__ cy,
                                                const double* __restrict__ cz) {
  return RawRef{{raw_mean32(n, [&](long long k) { return cx[b + k]; }),
                 raw_mean32(n, [&](long long k) { return cy[b + k]; }),
                 raw_mean32(n, [&](long long k) { return cz[b + k]; })}};
}

// Central moments of a cell from its raw sums and reference velocity: mean
// velocity U, C_ij, |C|^2 C_k / 2, C_k eps, C_k I (each a mean), eps, I.
struct RawMoments {
  double U[3], P[6], qt[3], qr[3], ql[3], eps, lev;
};
__device__ __forceinline__ RawMoments raw_moments(const double* a, double n, const double* w) {
  RawMoments r;
  const double inv = 1.0 / n;
  double m[3];
  for (int i = 0; i < 3; ++i) {
    m[i] = a[kRS + i] * inv;
    r.U[i] = w[i] + m[i];
  }
  const double Q[6] = {a[kRQ] * inv, a[kRQ + 1] * inv, a[kRQ + 2] * inv,
                       a[kRQ + 3] * inv, a[kRQ + 4] * inv, a[kRQ + 5] * inv};
  r.P[0] = Q[0] - m[0] * m[0]; r.P[1] = Q[1] - m[1] * m[1]; r.P[2] = Q[2] - m[2] * m[2];
  r.P[3] = Q[3] - m[0] * m[1]; r.P[4] = Q[4] - m[0] * m[2]; r.P[5] = Q[5] - m[1] * m[2];
  const double q2 = Q[0] + Q[1] + Q[2], m2 = m[0] * m[0] + m[1] * m[1] + m[2] * m[2];
  r.eps = a[kRe] * inv;
  r.lev = a[kRI] * inv;
  const int ix[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};
  for (int k = 0; k < 3; ++k) {
    const double mq = m[0] * Q[ix[k][0]] + m[1] * Q[ix[k][1]] + m[2] * Q[ix[k][2]];
    r.qt[k] = 0.5 * (a[kRT + k] * inv - m[k] * q2) - mq + m2 * m[k];
    r.qr[k] = a[kRE + k] * inv - m[k] * r.eps;
    r.ql[k] = a[kRL + k] * inv - m[k] * r.lev;
  }
  // a single particle has no spread and no variance is negative: what the
  // differences above leave of either is rounding
  for (int i = 0; i < 6; ++i)
    if (n == 1.0 || (i < 3 && r.P[i] < 0.0)) r.P[i] = 0.0;
  if (n == 1.0)
    for (int k = 0; k < 3; ++k) r.qt[k] = r.qr[k] = r.ql[k] = 0.0;
  return r;
}

// The raw sums of one cell (n particles from element b on; ref() gives its
// reference velocity to a whole warp, which one thread stores at
// wout[0], wout[ws], wout[2 ws]) added to acc[20] by
// the gridDim.x blocks of 256 threads that share it.  The particles are cut into
// chunks of at least chunk_min, dealt to the blocks first and then to their
// warps, so that one cell of a few thousand particles spreads over the SMs'
// FP64 pipes while a small cell costs one warp one reduction; a block adds
// its warps' totals with one atomic per sum.
constexpr int kRawBlock = 256;
template <typename Ref>
__device__ __forceinline__ void raw_cell(long long b, long long n, int chunk_min, Ref ref,
                                         const double* __restrict__ cx,
                                         const double* __restrict__ cy,
                                         const double* __restrict__ cz,
                                         const double* __restrict__ er,
                                         const int* __restrict__ lev, double* __restrict__ acc,
                                         double* __restrict__ wout, long long ws) {
  __shared__ double red[kRawBlock / 32][kRawN];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long long warps = (long long)gridDim.x * (kRawBlock / 32);
  long long chunk = (n + warps - 1) / warps;
  chunk = chunk < chunk_min ? chunk_min : (chunk + 31) & ~31ll;
  if ((long long)blockIdx.x * chunk >= n) return;             // uniform over the block
  const long long k0 = ((long long)wid * gridDim.x + blockIdx.x) * chunk;
  const long long k1 = k0 + chunk < n ? k0 + chunk : n;
  double mine = 0.0;
  int index = -1;
  if (k0 < k1) {                                              // uniform over the warp
    const RawRef w = ref();
    if (blockIdx.x == 0 && threadIdx.x == 0)
      for (int i = 0; i < 3; ++i) wout[i * ws] = w.w[i];
    double a[kRawN];
    long long aI = 0;
#pragma unroll
    for (int i = 0; i < kRawN; ++i) a[i] = 0.0;
#pragma unroll 2
    for (long long k = b + k0 + lane; k < b + k1; k += 32)
      raw_add(a, aI, cx[k] - w.w[0], cy[k] - w.w[1], cz[k] - w.w[2], er[k], lev[k]);
    a[kRI] = (double)aI;
    // 21 additions per lane instead of the 100 of twenty butterfly sums: the
    // FP64 pipe issues one warp instruction per 16 cycles, and a warp here
    // holds few particles
    index = halve_totals<kRawN>(a);
    mine = a[0];
  }
  __syncthreads();                                            // the previous cell's readers
  if (lane < kRawN) red[wid][lane] = 0.0;
  __syncwarp();
  if (index >= 0) red[wid][index] = mine;
  __syncthreads();
  if (threadIdx.x < kRawN) {
    double s = 0.0;
    for (int w = 0; w < kRawBlock / 32; ++w) s += red[w][threadIdx.x];
    atomicAdd(&acc[threadIdx.x], s);
  }
}
// blocks per cell and the smallest chunk for a launch over ncell cells: many
// cells fill the chip by themselves; a few are cut finely
inline int raw_blocks(int ncell) { return ncell >= 304 ? 2 : (608 + ncell - 1) / ncell; }
inline int raw_chunk(int ncell) { return ncell >= 1024 ? 512 : ncell >= 256 ? 128 : 64; }

}  // namespace usp

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

// The reference velocity of a cell of n particles: the FP32 mean of all of them, or of
// 2,048 (4,096 by a block) in runs of 8 (two sectors) at equal distances, 0 where that
// is not finite.  It is within 1 / 45 (1 / 64) of a thermal speed of the mean, so that a
// sum's size, and with it its rounding, stays near that of n random numbers: about the
// mean of 32, a fifth of a thermal speed, the mean velocities of cells of 10,000 to
// 40,000 at rest were off by 5.1e-15 of themselves, now by less than 1.5e-15.  Its
// 24 bits leave c - w exact: about the FP64 mean all c of a binade are rounded to the
// same side, which moves the mean of n of them by up to sqrt(n) 6e-17 of itself.
struct RawRef {
  double w[3];
};
// x rounded towards zero, by its bits: a conversion takes the FP64 pipe as long as a
// multiply-add (0 for what FP32 has no normal number for)
__device__ __forceinline__ float narrow(float x) { return x; }
__device__ __forceinline__ float narrow(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t a = hi & 0x7fffffffu;
  if (a - 0x38100000u >= 0x0fe00000u) return 0.0f;
  return __uint_as_float((hi & 0x80000000u) | ((a - 0x38000000u) << 3) | (lo >> 29));
}
__device__ __forceinline__ double ref_mean(float sum, float m) {
  const float v = __fdiv_rn(sum, m);
  return fabsf(v) < 3.0e38f ? (double)v : 0.0;
}
// by the G threads of a warp (32) or block (256), stored at wout[0], wout[ws], wout[2 ws]
constexpr int kRawBlock = 256;
template <int G>
__device__ __forceinline__ void raw_reference(long long b, long long n,
                                              const double* __restrict__ cx,
                                              const double* __restrict__ cy,
                                              const double* __restrict__ cz,
                                              double* __restrict__ wout, long long ws) {
  static_assert(G == 32 || G == kRawBlock, "a warp or a block");
  constexpr int kBits = G == 32 ? 11 : 12, kMost = 1 << kBits;
  const int t = threadIdx.x % G, m = n < kMost ? (int)n : kMost;
  float v[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll 8
  for (int i = t; i < m; i += G) {
    const long long k = b + (n <= kMost ? i : (((i >> 3) * n) >> (kBits - 3)) + (i & 7));
    v[0] += narrow(cx[k]); v[1] += narrow(cy[k]); v[2] += narrow(cz[k]);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i)
    for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
  if constexpr (G > 32) {
    __shared__ float part[G / 32][3];
    __syncthreads();                                          // the previous cell's readers
    if ((t & 31) == 0)
      for (int i = 0; i < 3; ++i) part[t >> 5][i] = v[i];
    __syncthreads();
    for (int i = 0; i < 3; ++i) {
      v[i] = part[0][i];
      for (int w = 1; w < G / 32; ++w) v[i] += part[w][i];
    }
  }
  if (t == 0)
    for (int i = 0; i < 3; ++i) wout[i * ws] = n > 0 ? ref_mean(v[i], (float)m) : 0.0;
}
// a warp per cell where they fill the chip: 15.5 million particles in 4,096 cells,
// references and sums, 0.93 ms (0.90 about the mean of 32; 0.98 with 4,096 of them
// taken one by one)
inline bool ref_by_warp(int ncell) { return ncell >= 608; }

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

// The raw sums of one cell (n particles from element b on, about ref()) added to acc[20]
// by the gridDim.x blocks of 256 threads that share it.  The particles are cut into
// chunks of at least chunk_min, dealt to the blocks first and then to their
// warps, so that one cell of a few thousand particles spreads over the SMs'
// FP64 pipes while a small cell costs one warp one reduction; a block adds
// its warps' totals with one atomic per sum.
template <typename Ref>
__device__ __forceinline__ void raw_cell(long long b, long long n, int chunk_min, Ref ref,
                                         const double* __restrict__ cx,
                                         const double* __restrict__ cy,
                                         const double* __restrict__ cz,
                                         const double* __restrict__ er,
                                         const int* __restrict__ lev,
                                         double* __restrict__ acc) {
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

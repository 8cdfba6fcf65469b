// FP64 products on the tensor path (mma.sync m8n8k4 .f64, "DMMA") in small
// output tiles, operands straight from global memory.
//
// A DMMA occupies its sub-partition's FP64 pipe for about 512 cycles on this
// GPU, so operand traffic is negligible (an 8 x 8 tile reads 512 bytes per
// DMMA, 1.2 TB/s over all SMs from the caches) and what counts is that every
// sub-partition has DMMAs to do.  A CTA's warps (four, one per sub-partition, or
// more when there are few tiles) share one output tile and take the K steps in
// turn; their sums are added in shared memory in a fixed order.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace {

__device__ __forceinline__ void fp64_dmma(double (&d)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};\n"
               : "+d"(d[0]), "+d"(d[1])
               : "d"(a), "d"(b));
}

template <class T>
struct Fp64Acc;
template <>
struct Fp64Acc<double> {
  double v[2];
  __device__ __forceinline__ void zero() { v[0] = v[1] = 0.0; }
  __device__ __forceinline__ void mma(double a, double b) { fp64_dmma(v, a, b); }
  __device__ __forceinline__ double get(int q) const { return v[q]; }
  __device__ __forceinline__ void set(int q, double x) { v[q] = x; }
};
template <>
struct Fp64Acc<cplx> {
  double re[2], im[2];
  __device__ __forceinline__ void zero() { re[0] = re[1] = im[0] = im[1] = 0.0; }
  __device__ __forceinline__ void mma(cplx a, cplx b) {
    fp64_dmma(re, a.re, b.re);
    fp64_dmma(im, a.re, b.im);
    fp64_dmma(re, -a.im, b.im);
    fp64_dmma(im, a.im, b.re);
  }
  __device__ __forceinline__ cplx get(int q) const { return cplx{re[q], im[q]}; }
  __device__ __forceinline__ void set(int q, cplx x) {
    re[q] = x.re;
    im[q] = x.im;
  }
};

// Rows m0 .. m0 + 8 WM - 1 and columns n0 .. n0 + 8 WN - 1 of A B over
// k < K (A: M x K column-major, B: K x N column-major; entries outside read as
// zero).  All NW warps of the CTA take part; the tile is left in red[0]
// (column-major, 8 WM rows) after a CTA barrier.
//
// tri: A is lower triangular.  The warps share k < m0 only; the tile's own
// diagonal block (k >= m0) is added on top of their sum, by one warp for each 8 x 8
// part.  The product with the diagonal is usually the largest term by far: as one
// of many partial sums it made every later addition of a partial round at the
// size of the result (512 x 64 FP64: 1.31e-16 from the exact solution, 8.2e-17
// with one sum in order of k).
template <class T, int WM, int WN, int NW>
__device__ __forceinline__ void fp64_tile(const T *__restrict__ A, int64_t lda, const T *__restrict__ B, int64_t ldb,
                                          int M, int N, int K, int tri, int m0, int n0, T (*red)[8 * WM * 8 * WN]) {
  using E = Elem<T>;
  constexpr int U = WM * WN >= 16 ? 2 : 4;  // K steps per load group; one group is in flight while another is multiplied
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int kend = tri ? min(K, m0) : K;
  auto load_a = [&](int r, int k, int ke) { return (k < ke && r < M) ? E::ld(A + r + (int64_t)k * lda) : E::zero(); };
  auto load_b = [&](int k, int c, int ke) { return (k < ke && c < N) ? E::ld(B + k + (int64_t)c * ldb) : E::zero(); };
  // this warp's operands in the diagonal block of a small tile, loaded with the first group
  constexpr int kDiag = 2 * WM;  // K steps of a diagonal block
  constexpr bool kEarly = WM * WN <= NW && kDiag <= 4;
  constexpr bool kFour = E::kComplex && WM * WN == 1;  // one warp for each of the complex product's four
  T da[kEarly ? kDiag : 1], db[kEarly ? kDiag : 1];
  const int di = warp % WM, dj = kFour ? 0 : warp / WM;  // (kEarly) this warp's part
  if constexpr (kEarly) {
    if (tri && warp < (kFour ? 4 : WM * WN)) {
#pragma unroll
      for (int u = 0; u < kDiag; ++u) {
        da[u] = load_a(m0 + 8 * di + g, m0 + 4 * u + t, K);
        db[u] = load_b(m0 + 4 * u + t, n0 + 8 * dj + g, K);
      }
    }
  }
  Fp64Acc<T> acc[WM][WN];
#pragma unroll
  for (int i = 0; i < WM; ++i)
#pragma unroll
    for (int j = 0; j < WN; ++j) acc[i][j].zero();
  T a[2][U][WM], b[2][U][WN];
  auto load = [&](int k0, int s) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = k0 + 4 * NW * u + t;
#pragma unroll
      for (int i = 0; i < WM; ++i) a[s][u][i] = load_a(m0 + 8 * i + g, k, kend);
#pragma unroll
      for (int j = 0; j < WN; ++j) b[s][u][j] = load_b(k, n0 + 8 * j + g, kend);
    }
  };
  auto mul = [&](int k0, int s) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (k0 + 4 * NW * u >= kend) break;  // warp-uniform
#pragma unroll
      for (int i = 0; i < WM; ++i)
#pragma unroll
        for (int j = 0; j < WN; ++j) acc[i][j].mma(a[s][u][i], b[s][u][j]);
    }
  };
  constexpr int kGroup = 4 * NW * U;
  int k0 = 4 * warp;
  load(k0, 0);
  while (k0 < kend) {
    load(k0 + kGroup, 1);
    mul(k0, 0);
    k0 += kGroup;
    if (k0 >= kend) break;
    load(k0 + kGroup, 0);
    mul(k0, 1);
    k0 += kGroup;
  }
  auto at = [&](int i, int j, int q) { return (8 * i + g) + (8 * j + 2 * t + q) * 8 * WM; };
#pragma unroll
  for (int i = 0; i < WM; ++i)
#pragma unroll
    for (int j = 0; j < WN; ++j)
#pragma unroll
      for (int q = 0; q < 2; ++q) red[warp][at(i, j, q)] = acc[i][j].get(q);
  __syncthreads();
  for (int e = threadIdx.x; e < 8 * WM * 8 * WN; e += 32 * NW) {
    T v = red[0][e];
#pragma unroll
    for (int w = 1; w < NW; ++w) v = E::add(v, red[w][e]);
    red[0][e] = v;
  }
  __syncthreads();
  if (!tri) return;  // CTA-uniform
  if constexpr (kFour) {
    if (warp < 4) {
      const bool im = (warp & 2) != 0, second = (warp & 1) != 0;
      double d[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) d[q] = second ? 0.0 : im ? red[0][at(0, 0, q)].im : red[0][at(0, 0, q)].re;
#pragma unroll
      for (int u = 0; u < kDiag; ++u)
        fp64_dmma(d, second ? (im ? da[u].im : -da[u].im) : da[u].re, im != second ? db[u].im : db[u].re);
#pragma unroll
      for (int q = 0; q < 2; ++q) (im ? red[second][at(0, 0, q)].im : red[second][at(0, 0, q)].re) = d[q];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 64; e += 32 * NW) red[0][e] = E::add(red[0][e], red[1][e]);
    __syncthreads();
    return;
  }
  for (int p = warp; p < WM * WN; p += NW) {
    const int i = p % WM, j = p / WM;
    Fp64Acc<T> d;
#pragma unroll
    for (int q = 0; q < 2; ++q) d.set(q, red[0][at(i, j, q)]);
    if constexpr (kEarly) {
#pragma unroll
      for (int u = 0; u < kDiag; ++u)
        if (u < 2 * (i + 1)) d.mma(da[u], db[u]);
    } else {
      for (int k = m0; k < min(K, m0 + 8 * (i + 1)); k += 4)
        d.mma(load_a(m0 + 8 * i + g, k + t, K), load_b(k + t, n0 + 8 * j + g, K));
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) red[0][at(i, j, q)] = d.get(q);
  }
  __syncthreads();
}

}  // namespace

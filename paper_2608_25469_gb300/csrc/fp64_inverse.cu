// FP64 inverses of the N_B x N_B diagonal blocks (phase 1 of the blocked
// algorithm, Section 4.3) by doubling.
//
// Inverting an N_B-row block by substitution (Algorithm 2) is a chain of N_B
// dependent steps, 0.3 ms at N_B = 256 and 1 ms at N_B = 512 on this GPU
// whatever the number of blocks.  Here substitution inverts 32 x 32 blocks only,
// one column per warp and lane-per-row, and each level joins adjacent h x h
// inverses into a 2h x 2h one: for
//   T = [A 0; C D],   T^-1 = [A^-1 0; -D^-1 C A^-1  D^-1],
// W = C A^-1 and then -D^-1 W, for every pair of the level in one launch each,
// with the known zeros of the triangular inverses left out.  The products are
// small tiles on the FP64 tensor path; the tile size is the largest that still
// gives every SM's sub-partitions work.
#include <cuda_runtime.h>

#include <algorithm>

#include "blocked.h"
#include "common.cuh"
#include "fp64_tile.cuh"
#include "trace.h"
#include "workspace.h"

namespace {

constexpr int kBase = 32;      // blocks inverted by substitution
constexpr int kBaseWarps = 4;  // columns per CTA of the base kernel
constexpr int kFp64Warps = 4;  // warps per CTA of the products

// Columns 4 y .. 4 y + 3 of the inverse of base block b (rows 32 b .. of the
// matrix), one per warp: lane r holds row r of the block, scaled by 1/a_rr, in
// registers, and step k takes entry k of the column from its lane.  A step is
// one warp-wide multiply-add behind a shuffle (about 100 cycles, 400 complex);
// several columns per warp would add their pipe time to every step.
template <class T>
__global__ void __launch_bounds__(32 * kBaseWarps) inv_base_kernel(const T *__restrict__ A, int64_t lda, int64_t m,
                                                                   int nb, int unit, T *Dinv) {
  using E = Elem<T>;
  const int lane = threadIdx.x & 31, j = blockIdx.y * kBaseWarps + (threadIdx.x >> 5);
  const int64_t r0 = (int64_t)blockIdx.x * kBase;
  const int s = (int)min((int64_t)kBase, m - r0);
  const T *D = A + r0 + r0 * lda;
  T rv = E::zero();
  if (lane < s) rv = unit ? E::one() : E::recip(E::ld(D + lane + (int64_t)lane * lda));
  T row[kBase];
#pragma unroll
  for (int k = 0; k < kBase; ++k) row[k] = (k >= j && lane > k && lane < s) ? E::ld(D + lane + (int64_t)k * lda) : E::zero();
  T x = lane == j ? rv : E::zero();
#pragma unroll
  for (int k = 0; k < kBase - 1; ++k) {
    if (k >= j) {  // warp-uniform
      const T y = E::fms(E::mul(rv, row[k]), E::shfl(x, k), x);
      if (lane > k) x = y;
    }
  }
  T *Y = Dinv + (r0 / nb) * (int64_t)nb * nb;
  const int l = (int)(r0 % nb);
  if (j < s && lane < s && lane >= j) Y[(l + lane) + (int64_t)(l + j) * nb] = x;
}

// Level h.  blockIdx.y = pair (rows 2 h y .. of the matrix), blockIdx.x = output
// tile.  Pass 0: W = C A^-1 (ld h per pair); pass 1: the lower-left block of the
// 2h inverse, -D^-1 W.  A partial last pair has a shorter D; a pair without a D
// block does nothing.
template <class T, int WT, int PASS>
__global__ void __launch_bounds__(32 * kFp64Warps) inv_level_kernel(const T *__restrict__ A, int64_t lda, int64_t m,
                                                                    int nb, int h, T *Dinv, T *W) {
  constexpr int TS = 8 * WT;
  __shared__ T red[kFp64Warps][TS * TS];
  const int64_t i0 = (int64_t)blockIdx.y * 2 * h;
  const int sd = (int)min((int64_t)h, m - i0 - h);
  const int tiles = h / TS;
  const int m0 = (blockIdx.x % tiles) * TS, n0 = (blockIdx.x / tiles) * TS;
  if (m0 >= sd) return;
  T *Y = Dinv + (i0 / nb) * (int64_t)nb * nb;
  const int l0 = (int)(i0 % nb);
  T *Wp = W + (int64_t)blockIdx.y * h * h;
  if (PASS == 0) {  // column tile n0 of A^-1 starts at row n0
    fp64_tile<T, WT, WT, kFp64Warps>(A + (i0 + h) + i0 * lda, lda, Y + l0 + (int64_t)l0 * nb, nb, sd, h, n0, h, m0, n0, red);
  } else {  // row tile m0 of D^-1 ends at its diagonal
    fp64_tile<T, WT, WT, kFp64Warps>(Y + (l0 + h) + (int64_t)(l0 + h) * nb, nb, Wp, h, sd, h, 0, min(sd, m0 + TS), m0, n0, red);
  }
  T *out = PASS == 0 ? Wp : Y + (l0 + h) + (int64_t)l0 * nb;
  const int64_t ldo = PASS == 0 ? h : nb;
  for (int e = threadIdx.x; e < TS * TS; e += 32 * kFp64Warps) {
    const int i = m0 + e % TS, jc = n0 + e / TS;
    if (i < sd) {
      const T v = red[0][e];
      out[i + (int64_t)jc * ldo] = PASS == 0 ? v : fp64_neg(v);
    }
  }
}

template <class T, int WT>
void launch_level(const T *A, int64_t lda, int64_t m, int nb, int h, unsigned pairs, T *Dinv, T *W, cudaStream_t st) {
  const unsigned tiles = (unsigned)(h / (8 * WT));
  const dim3 grid(tiles * tiles, pairs);
  inv_level_kernel<T, WT, 0><<<grid, 32 * kFp64Warps, 0, st>>>(A, lda, m, nb, h, Dinv, W);
  inv_level_kernel<T, WT, 1><<<grid, 32 * kFp64Warps, 0, st>>>(A, lda, m, nb, h, Dinv, W);
}

}  // namespace

size_t hsma_fp64_inverse_scratch(int nb, int64_t m, size_t esize) {
  // the pairs of the last level, the largest: (N_B / 2)^2 per outer block
  return nb > kBase ? esize * (size_t)((m + nb - 1) / nb) * (nb / 2) * (nb / 2) : 0;
}

template <class T>
hsma_status_t hsma_fp64_diag_inverse(int nb, const T *A, int64_t lda, int64_t m, int unit, T *Dinv, T *W,
                                     cudaStream_t st) {
  if (nb < kBase || nb > 512 || (nb & (nb - 1)) != 0) return HSMA_ERR_UNSUPPORTED;
  const int64_t nblk = (m + nb - 1) / nb, nbase = (m + kBase - 1) / kBase;
  int levels = 0;
  for (int h = kBase; h < nb; h *= 2) ++levels;
  HsmaTraceScope ts("diag_inverse", st, 1 + 2 * levels);
  // zeros above the diagonals and outside a partial block
  HSMA_CUDA_TRY(cudaMemsetAsync(Dinv, 0, sizeof(T) * (size_t)nblk * nb * nb, st));
  inv_base_kernel<T><<<dim3((unsigned)nbase, kBase / kBaseWarps), 32 * kBaseWarps, 0, st>>>(A, lda, m, nb, unit,
                                                                                           Dinv);
  for (int h = kBase; h < nb; h *= 2) {
    const int64_t pairs = (m + 2 * h - 1) / (2 * h);
    if (pairs > 65535) return HSMA_ERR_UNSUPPORTED;
    const int64_t want = 4 * (int64_t)hsma_sm_count();  // CTAs for the SMs to share evenly
    const int64_t t32 = pairs * (h / 32) * (h / 32);
    bool done = false;
    if constexpr (sizeof(T) == sizeof(double)) {  // complex: too many registers
      if ((done = t32 >= want)) launch_level<T, 4>(A, lda, m, nb, h, (unsigned)pairs, Dinv, W, st);
    }
    if (done) continue;
    if (4 * t32 >= want)
      launch_level<T, 2>(A, lda, m, nb, h, (unsigned)pairs, Dinv, W, st);
    else
      launch_level<T, 1>(A, lda, m, nb, h, (unsigned)pairs, Dinv, W, st);
  }
  return hsma_from_cuda(cudaGetLastError());
}

template hsma_status_t hsma_fp64_diag_inverse<double>(int, const double *, int64_t, int64_t, int, double *, double *,
                                                      cudaStream_t);
template hsma_status_t hsma_fp64_diag_inverse<cplx>(int, const cplx *, int64_t, int64_t, int, cplx *, cplx *,
                                                    cudaStream_t);

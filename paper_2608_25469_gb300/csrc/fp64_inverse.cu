// FP64 inverses of the N_B x N_B diagonal blocks (phase 1 of the blocked
// algorithm, Section 4.3): forward substitution against the identity
// (Section 4.3.1) in blocks of 32 rows.
//
// Substitution row by row (Algorithm 2) is a chain of N_B dependent steps, 0.3 ms at
// N_B = 256 and 1 ms at N_B = 512 on this GPU whatever the number of blocks.
// Here it inverts 32 x 32 base blocks only; below them a CTA carries one column
// x of the inverse down the block rows,
//   x_i = -D_ii^-1 (sum_{k < i} D_ik x_k),
// with the column in shared memory and a lane per row: the sum is a run of
// independent loads and multiply-adds, and what depends on the row before is
// one 32-step product.  The CTAs need nothing from each other.
//
// Only inverses of 32-row blocks are multiplied, so D X - I stays at the level of
// row-by-row substitution.  Joining inverses by doubling, -D22^-1 (D21 D11^-1),
// costs the same multiply-adds but leaves the condition of the half-size blocks in
// it: on LU factors of random matrices the residual of the solve was 1.3 (N_B =
// 128) to 2.7 times (512) that of substitution, this form 1.0 to 1.1 times.
#include <cuda_runtime.h>

#include <algorithm>

#include "blocked.h"
#include "common.cuh"
#include "trace.h"

namespace {

constexpr int kBase = 32;    // blocks inverted row by row
constexpr int kInvWarps = 4;  // one per SM sub-partition
constexpr int kMaxNb = 512;

// Columns 4 y .. 4 y + 3 of the inverse of base block b (rows 32 b .. of the
// matrix), one per warp: lane r holds row r of the block, scaled by 1/a_rr, in
// registers, and step k takes entry k of the column from its lane.  A step is
// one warp-wide multiply-add behind a shuffle (about 100 cycles, 400 complex);
// several columns per warp would add their pipe time to every step.
template <class T>
__global__ void __launch_bounds__(32 * kInvWarps) inv_base_kernel(const T *__restrict__ A, int64_t lda, int64_t m,
                                                                  int nb, int unit, T *Dinv) {
  using E = Elem<T>;
  const int lane = threadIdx.x & 31, j = blockIdx.y * kInvWarps + (threadIdx.x >> 5);
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
  Y[(l + lane) + (int64_t)(l + j) * nb] = j < s && lane < s && lane >= j ? x : E::zero();
}

// One column of the inverse of an outer block whose base blocks are in place; zeros
// above the base block and past the matrix included.  The four warps take turns in
// both products, kDepth columns of D at a time (the next kDepth in flight), and add
// their parts through shared memory.  The FP64 pipe (64 cycles per warp-wide
// multiply-add) bounds the longest column or, with many columns, the launch; a
// block's longest columns start first.  A column per warp and one per two warps
// leave the longest column's chain exposed: solves of 512 x 32 FP64 84 / 76 / 73 us
// with 1 / 2 / 4 warps per column, emulated 512 x 128 (N_B = 512) 326 / 230 / 190 us
// (joined by doubling 83 and 186 us; 8192 x 4096 emulated 7.53 -> 7.39 ms).
template <class T>
__global__ void __launch_bounds__(32 * kInvWarps) inv_columns_kernel(const T *__restrict__ A, int64_t lda, int64_t m,
                                                                     int nb, T *Dinv) {
  using E = Elem<T>;
  constexpr int kDepth = 4, kPart = kBase / kInvWarps;
  static_assert(2 * kDepth * kInvWarps == kBase && kPart == 2 * kDepth, "a block row is one turn of every warp");
  __shared__ T sX[kInvWarps][kMaxNb];      // the column, a copy per warp
  __shared__ T sSum[2][kInvWarps][kBase];  // the warps' parts of a sum and of a block row
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // block by block: CTAs that go to different SMs hold columns of nearly the same length
  const int j = blockIdx.x % nb, blk = blockIdx.x / nb;
  const int64_t r0 = (int64_t)blk * nb;
  const int s = (int)min((int64_t)nb, m - r0);
  const T *D = A + r0 + r0 * lda;
  T *Y = Dinv + (int64_t)blk * nb * nb;
  T *out = Y + (int64_t)j * nb, *x = sX[warp];
  const int j0 = j & ~(kBase - 1);
  for (int r = threadIdx.x; r < nb; r += 32 * kInvWarps)
    if (r < j0 || j >= s || (r >= s && r >= j0 + kBase)) out[r] = E::zero();
  if (j >= s) return;
  auto sum_warps = [&](T v, int h) {  // in the same order in every warp
    sSum[h][warp][lane] = v;
    __syncthreads();
    v = sSum[h][0][lane];
#pragma unroll
    for (int w = 1; w < kInvWarps; ++w) v = E::add(v, sSum[h][w][lane]);
    return v;
  };
  x[j0 + lane] = out[j0 + lane];
  __syncwarp();
  for (int i0 = j0 + kBase; i0 < s; i0 += kBase) {
    const T *d = D + min(i0 + lane, s - 1);  // lanes past the matrix repeat its last row
    const T *inv = Y + (i0 + lane) + (int64_t)(i0 + kPart * warp) * nb;
    T a[2][kDepth];
    auto load = [&](int k0, int h) {  // columns before j meet zeros of x: not read
#pragma unroll
      for (int u = 0; u < kDepth; ++u) a[h][u] = k0 + u >= j ? E::ld(d + (int64_t)(k0 + u) * lda) : E::zero();
    };
    auto load_inv = [&](int k0, int h) {
#pragma unroll
      for (int u = 0; u < kDepth; ++u) a[h][u] = E::ld(inv + (int64_t)(k0 + u) * nb);
    };
    T acc = E::zero();
    int k0 = j0 + kPart * warp;
    load(k0, 0);
    for (; k0 < i0; k0 += kBase) {
      load(k0 + kDepth, 1);
#pragma unroll
      for (int u = 0; u < kDepth; ++u) acc = E::fms(a[0][u], x[k0 + u], acc);
      if (k0 + kBase < i0)
        load(k0 + kBase, 0);
      else
        load_inv(0, 0);
#pragma unroll
      for (int u = 0; u < kDepth; ++u) acc = E::fms(a[1][u], x[k0 + kDepth + u], acc);
    }
    x[i0 + lane] = E::neg(sum_warps(acc, 0));
    __syncwarp();
    load_inv(kDepth, 1);
    T y = E::zero();
#pragma unroll
    for (int u = 0; u < kPart; ++u) {
      const int k = kPart * warp + u;
      const T t = E::fms(a[u / kDepth][u % kDepth], x[i0 + k], y);
      if (k <= lane) y = t;  // nothing above the diagonal is multiplied
    }
    y = sum_warps(y, 1);
    __syncwarp();
    x[i0 + lane] = y;
    __syncwarp();
    if (warp == 0 && i0 + lane < s) out[i0 + lane] = y;
  }
}

}  // namespace

template <class T>
hsma_status_t hsma_fp64_diag_inverse(int nb, const T *A, int64_t lda, int64_t m, int unit, T *Dinv, cudaStream_t st) {
  if (nb < kBase || nb > kMaxNb || (nb & (nb - 1)) != 0) return HSMA_ERR_UNSUPPORTED;
  const int64_t nblk = (m + nb - 1) / nb, nbase = (m + kBase - 1) / kBase;
  HsmaTraceScope ts("diag_inverse", st, nb > kBase ? 2 : 1);
  inv_base_kernel<T><<<dim3((unsigned)nbase, kBase / kInvWarps), 32 * kInvWarps, 0, st>>>(A, lda, m, nb, unit, Dinv);
  if (nb > kBase) inv_columns_kernel<T><<<(unsigned)(nblk * nb), 32 * kInvWarps, 0, st>>>(A, lda, m, nb, Dinv);
  return hsma_from_cuda(cudaGetLastError());
}

template hsma_status_t hsma_fp64_diag_inverse<double>(int, const double *, int64_t, int64_t, int, double *,
                                                      cudaStream_t);
template hsma_status_t hsma_fp64_diag_inverse<cplx>(int, const cplx *, int64_t, int64_t, int, cplx *, cudaStream_t);

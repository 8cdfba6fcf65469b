// Varlen batch of small solves (m <= 64) in FP32 (float and float complex):
// triangular solves, and LU- and Cholesky-factor solves fused per instance.
//
// FP32 arithmetic is cheap here; what bounds this work is instruction fetch,
// load latency and shared-memory reads.  The fully unrolled substitution of the
// FP64 kernels (X in registers, one variant per row-group count) spends most of
// its issue slots waiting for instructions when the arithmetic is this fast
// (10.5 of 18 stall cycles per instruction, 362 us for 8192 complex64 solves
// with m, n ~ U{8..64}).  Here the substitution runs in 8-row blocks with
// rolled loops (about 600 instructions in all):
//
//  * one CTA of four warps per instance, in any order (the hardware deals
//    instances to SMs as they free up; there is no schedule pass);
//  * the triangle (8 x 8 blocks) and the right-hand sides are copied to shared
//    memory asynchronously, all of an instance's loads in flight at once;
//  * a warp owns 16 columns, two lanes per column with four rows of each block;
//    block row J gathers
//        acc = alpha B_J - sum_{I < J} L_JI X_I
//    from shared memory before its own eight steps, X overwrites B there, and
//    the warp writes its columns back row-contiguously.
//
// Measured on 8192 complex64 solves: 362 us unrolled, 233 us in this form with
// B read and X written from the lanes' own columns, 172 us as it stands.
//
// The per-instance arithmetic does not depend on the batch it sits in.
#include <cuda_runtime.h>

#include "common.cuh"
#include "small.h"
#include "trace.h"

namespace {

constexpr int kWarps = 4;
constexpr int kCols = 16;  // columns per warp
constexpr int kBlk = 8;    // rows per block
constexpr int kMaxBlocks = 64 / kBlk;
constexpr int kLdX = kCols + 1;  // row pitch of the right-hand sides: column reads and row writes miss bank conflicts

// Index map from the solved lower-triangular form onto the operand: with rev,
// row r of the form is row m-1-r of the operand and of B; with tr, A is read
// transposed; with cj, conjugated.
struct Map {
  int rev, tr, cj;
};

// block (J, I), I <= J, of the staged triangle: 8 columns of 8 rows
__device__ __forceinline__ int blk_at(int J, int I) { return (J * (J + 1) / 2 + I) * kBlk * kBlk; }

template <class T>
constexpr size_t smem_bytes() {
  return sizeof(T) * (kMaxBlocks * (kMaxBlocks + 1) / 2 * kBlk * kBlk + 64 + kWarps * 64 * kLdX);
}

// four consecutive elements (16-byte aligned)
__device__ __forceinline__ void ld4(float (&v)[4], const float *p) {
  const float4 q = *reinterpret_cast<const float4 *>(p);
  v[0] = q.x;
  v[1] = q.y;
  v[2] = q.z;
  v[3] = q.w;
}
__device__ __forceinline__ void ld4(cplxf (&v)[4], const cplxf *p) {
  const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 2);
  v[0] = cplxf{a.x, a.y};
  v[1] = cplxf{a.z, a.w};
  v[2] = cplxf{b.x, b.y};
  v[3] = cplxf{b.z, b.w};
}

// 1 / a with three divisions (Elem's complex form saves one and loses an ulp;
// here every solved row is multiplied by it)
__device__ __forceinline__ float recip(float a) { return 1.0f / a; }
__device__ __forceinline__ cplxf recip(cplxf a) {
  const bool big = fabsf(a.re) >= fabsf(a.im);
  const float p = big ? a.re : a.im, q = big ? a.im : a.re;
  const float t = q / p, d = fmaf(q, t, p);
  const float u = 1.0f / d, v = t / d;
  return big ? cplxf{u, -v} : cplxf{v, -u};
}

template <class T>
__device__ __forceinline__ void copy_async(T *dst, const T *src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(T) == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Start copying the lower-triangular form: a warp per stored column (row with
// tr), lanes along it.  Rows past m and entries above the diagonal are not
// written: they only reach values that are never used.  The diagonal is part of
// its block.
template <class T>
__device__ __forceinline__ void stage_a(T *sL, const T *__restrict__ A, int64_t lda, int m, bool unit, Map mp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = warp; o < m; o += kWarps) {
    const T *line = A + (int64_t)(mp.rev ? m - 1 - o : o) * lda;
    for (int i = lane + (mp.tr ? 0 : o & ~31); i < (mp.tr ? o + 1 : m); i += 32) {
      const int r = mp.tr ? o : i, c = mp.tr ? i : o;
      if (r < c || (unit && r == c)) continue;
      copy_async(sL + blk_at(r / kBlk, c / kBlk) + (c % kBlk) * kBlk + r % kBlk, line + (mp.rev ? m - 1 - i : i));
    }
  }
}

// Start copying this warp's columns j0 .. j0 + 15 of B (rows reversed with rev).
template <class T>
__device__ __forceinline__ void stage_b(T *X, const T *B, int64_t ldb, int m, int n, int j0, int rev) {
  const int lane = threadIdx.x & 31;
  for (int j = 0; j < min(kCols, n - j0); ++j) {
    const T *col = B + (int64_t)(j0 + j) * ldb;
    for (int r = lane; r < m; r += 32) copy_async(X + r * kLdX + j, col + (rev ? m - 1 - r : r));
  }
}

// X = alpha L^-1 B for the staged columns of this warp, in shared memory; cj:
// with conj(L), by solving for conj(X).
template <class T>
__device__ __forceinline__ void solve_tile(const T *sL, const T *sR, T *X0, int m, T alpha, int cj) {
  using E = Elem<T>;
  const int lane = threadIdx.x & 31;
  const int c = lane % kCols, h = lane / kCols;  // this lane's column of the tile and half of each block
  T *X = X0 + c;
  const int nblk = (m + kBlk - 1) / kBlk;
#pragma unroll 1
  for (int J = 0; J < nblk; ++J) {
    T acc[4];
    T *xJ = X + J * kBlk * kLdX;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      acc[q] = E::mul(alpha, xJ[(4 * h + q) * kLdX]);
      if constexpr (E::kComplex) {
        if (cj) acc[q].im = -acc[q].im;
      }
    }
    const T *L = sL + blk_at(J, 0) + 4 * h;
    const T *x = X;
#pragma unroll 1
    for (int I = 0; I < J; ++I, L += kBlk * kBlk, x += kBlk * kLdX) {
#pragma unroll
      for (int k = 0; k < kBlk; ++k) {
        const T xk = x[k * kLdX];
        T l[4];
        ld4(l, L + k * kBlk);
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = E::fms(l[q], xk, acc[q]);
      }
    }
    // the block's own rows: row k is final after k steps; later updates of rows
    // at or above k touch values that are no longer used
    T out[4];
#pragma unroll
    for (int k = 0; k < kBlk; ++k) {
      const T mine = E::mul(acc[k % 4], sR[J * kBlk + k]);
      if (k < 4 || h == 1) out[k % 4] = mine;  // rows 0 .. 3 are the first half's: kept below
      if (k + 1 < kBlk) {
        const T xk = E::shfl(mine, (k / 4) * kCols + c);
        T l[4];
        ld4(l, L + k * kBlk);
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = E::fms(l[q], xk, acc[q]);
      }
    }
    __syncwarp();  // both lanes of a column have read this block's B
#pragma unroll
    for (int q = 0; q < 4; ++q) xJ[(4 * h + q) * kLdX] = out[q];
    __syncwarp();
  }
}

template <class T>
__device__ __forceinline__ void write_x(const T *X, T *B, int64_t ldb, int m, int n, int j0, int rev, int cj) {
  using E = Elem<T>;
  const int lane = threadIdx.x & 31;
#pragma unroll 4
  for (int j = 0; j < min(kCols, n - j0); ++j) {
    T *col = B + (int64_t)(j0 + j) * ldb;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = lane + 32 * h;
      if (r >= m) continue;
      T v = X[r * kLdX + j];
      if constexpr (E::kComplex) {
        if (cj) v.im = -v.im;
      }
      E::st(col + (rev ? m - 1 - r : r), v);
    }
  }
}

// One triangular solve of an instance in place on B, all threads of the CTA.
template <class T>
__device__ __forceinline__ void solve(T *sL, T *sR, T *sX, const T *__restrict__ A, int64_t lda, T *B, int64_t ldb,
                                      int m, int n, T alpha, bool unit, Map mp) {
  using E = Elem<T>;
  const int warp = threadIdx.x >> 5;
  T *X = sX + warp * 64 * kLdX;
  stage_a<T>(sL, A, lda, m, unit, mp);
  if (warp * kCols < n) stage_b<T>(X, B, ldb, m, n, warp * kCols, mp.rev);
  copies_wait();
  __syncthreads();
  if (threadIdx.x < 64) {
    const int r = threadIdx.x;
    if (r < m) sR[r] = unit ? E::one() : recip(sL[blk_at(r / kBlk, r / kBlk) + (r % kBlk) * (kBlk + 1)]);
  }
  __syncthreads();
  for (int j0 = warp * kCols; j0 < n; j0 += kWarps * kCols) {
    if (j0 >= kWarps * kCols) {
      stage_b<T>(X, B, ldb, m, n, j0, mp.rev);
      copies_wait();
      __syncwarp();
    }
    solve_tile<T>(sL, sR, X, m, alpha, mp.cj);
    write_x<T>(X, B, ldb, m, n, j0, mp.rev, mp.cj);
    __syncwarp();  // before the next columns' copies
  }
}

template <class T>
__device__ __forceinline__ void zero(T *B, int64_t ldb, int m, int n) {
  for (int j = threadIdx.x >> 5; j < n; j += kWarps)
    for (int r = threadIdx.x & 31; r < m; r += 32) B[r + (int64_t)j * ldb] = Elem<T>::zero();
}

// LAPACK's interchanges as one gather per column (row r takes the old row
// perm[r]).  False, with B untouched, when a pivot lies outside [k, m).
template <class T>
__device__ __forceinline__ bool permute(T *B, int64_t ldb, int m, int n, const int32_t *__restrict__ ipiv, int *sPiv,
                                        int *sPerm) {
  using E = Elem<T>;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  bool bad = false;
  for (int k = tid; k < m; k += 32 * kWarps) {
    sPiv[k] = ipiv[k] - 1;
    sPerm[k] = k;
    bad |= sPiv[k] < k || sPiv[k] >= m;
  }
  if (__syncthreads_or(bad)) return false;
  if (tid == 0) {
    for (int k = 0; k < m; ++k) {
      const int p = sPiv[k], t = sPerm[k];
      sPerm[k] = sPerm[p];
      sPerm[p] = t;
    }
  }
  __syncthreads();
  const int p0 = lane < m ? sPerm[lane] : 0, p1 = lane + 32 < m ? sPerm[lane + 32] : 0;
  for (int j = warp; j < n; j += kWarps) {  // warp-uniform: every lane shuffles
    T *col = B + (int64_t)j * ldb;
    const T v0 = lane < m ? col[lane] : E::zero(), v1 = lane + 32 < m ? col[lane + 32] : E::zero();
    const T a0 = E::shfl(v0, p0 & 31), b0 = E::shfl(v1, p0 & 31);
    const T a1 = E::shfl(v0, p1 & 31), b1 = E::shfl(v1, p1 & 31);
    if (lane < m) col[lane] = p0 < 32 ? a0 : b0;
    if (lane + 32 < m) col[lane + 32] = p1 < 32 ? a1 : b1;
  }
  __syncthreads();
  return true;
}

enum { KIND_TRSM = 0, KIND_LU = 1, KIND_CHOL = 2 };

template <class T>
__global__ void __launch_bounds__(32 * kWarps) batch_f32_kernel(const int32_t *__restrict__ dm,
                                                                const int32_t *__restrict__ dn,
                                                                const int32_t *__restrict__ dlda,
                                                                const int32_t *__restrict__ dldb,
                                                                const void *const *__restrict__ dA,
                                                                const int32_t *const *__restrict__ dipiv,
                                                                void *const *__restrict__ dB, T alpha, int unit,
                                                                uint32_t *status, Map mp, int kind, int skip_large) {
  using E = Elem<T>;
  extern __shared__ __align__(16) unsigned char smem[];
  T *sL = reinterpret_cast<T *>(smem);
  T *sR = sL + kMaxBlocks * (kMaxBlocks + 1) / 2 * kBlk * kBlk;
  T *sX = sR + 64;
  const int b = blockIdx.x;
  const int m = dm[b], n = dn[b], lda = dlda[b], ldb = dldb[b];
  const T *A = static_cast<const T *>(dA[b]);
  T *B = static_cast<T *>(dB[b]);
  const int lo = m > 1 ? m : 1;
  if (skip_large && m > 64) return;  // solved by the caller on the blocked path
  uint32_t err = 0;
  if (m < 0 || n < 0 || m > 64 || lda < lo || ldb < lo)
    err = HSMA_DEVERR_BAD_SIZE;
  else if (m == 0 || n == 0)
    return;
  else if (A == nullptr || B == nullptr)
    err = HSMA_DEVERR_NULL_PTR;
  if (err == 0 && kind == KIND_LU && dipiv != nullptr && dipiv[b] != nullptr) {
    int *sPiv = reinterpret_cast<int *>(sX);
    if (!permute<T>(B, ldb, m, n, dipiv[b], sPiv, sPiv + 64)) err = HSMA_DEVERR_BAD_PIVOT;
  }
  if (err != 0) {
    if (threadIdx.x == 0 && status != nullptr) atomicOr(status, err);
    return;
  }
  if (E::is_zero(alpha)) {
    zero<T>(B, ldb, m, n);
    return;
  }
  // factor solves: L (unit for LU), then U, or L^H through the reversed,
  // transposed, conjugated map
#pragma unroll 1
  for (int pass = 0; pass < (kind == KIND_TRSM ? 1 : 2); ++pass) {
    const Map pm = kind == KIND_TRSM ? mp : pass == 0 ? Map{0, 0, 0} : Map{1, kind == KIND_CHOL, kind == KIND_CHOL};
    const bool un = kind == KIND_TRSM ? unit != 0 : pass == 0 && kind == KIND_LU;
    if (pass != 0) __syncthreads();  // the first solve has read the staged triangle and written B
    solve<T>(sL, sR, sX, A, lda, B, ldb, m, n, pass == 0 ? alpha : E::one(), un, pm);
  }
}

template <class T>
hsma_status_t launch(int32_t batch, const int32_t *dm, const int32_t *dn, const double *alpha, const void *const *dA,
                     const int32_t *dlda, const int32_t *const *dipiv, void *const *dB, const int32_t *dldb, int unit,
                     uint32_t *status, cudaStream_t st, Map mp, int kind, int skip_large) {
  static DeviceFlags attr_done;
  if (!attr_done.test()) {
    HSMA_CUDA_TRY(cudaFuncSetAttribute(batch_f32_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem_bytes<T>()));
    attr_done.set();
  }
  HsmaTraceScope ts(kind == KIND_TRSM ? "vbatched_solve" : "vbatched_lu", st);
  batch_f32_kernel<T><<<batch, 32 * kWarps, smem_bytes<T>(), st>>>(dm, dn, dlda, dldb, dA, dipiv, dB,
                                                                   hsma_alpha_as<T>(alpha), unit, status, mp, kind,
                                                                   skip_large);
  return hsma_from_cuda(cudaGetLastError());
}

}  // namespace

hsma_status_t hsma_f32_vbatched(int dtype, int32_t batch, const int32_t *dm, const int32_t *dn, const double *alpha,
                                const void *const *dA, const int32_t *dlda, void *const *dB, const int32_t *dldb,
                                int unit, uint32_t *status, cudaStream_t st, int uplo, int trans, int skip_large) {
  const bool op_lower = (uplo == HSMA_LOWER) != (trans != HSMA_NO_TRANS);
  const Map mp{op_lower ? 0 : 1, trans != HSMA_NO_TRANS ? 1 : 0, trans == HSMA_CONJ_TRANS ? 1 : 0};
  if (dtype == HSMA_R32)
    return launch<float>(batch, dm, dn, alpha, dA, dlda, nullptr, dB, dldb, unit, status, st, mp, KIND_TRSM,
                         skip_large);
  return launch<cplxf>(batch, dm, dn, alpha, dA, dlda, nullptr, dB, dldb, unit, status, st, mp, KIND_TRSM,
                       skip_large);
}

hsma_status_t hsma_f32_factor_vbatched(int dtype, int32_t batch, const int32_t *dm, const int32_t *dn,
                                       const double *alpha, const void *const *dA, const int32_t *dlda,
                                       const int32_t *const *dipiv, void *const *dB, const int32_t *dldb,
                                       uint32_t *status, cudaStream_t st, int chol, int skip_large) {
  const int kind = chol ? KIND_CHOL : KIND_LU;
  if (dtype == HSMA_R32)
    return launch<float>(batch, dm, dn, alpha, dA, dlda, dipiv, dB, dldb, 0, status, st, Map{0, 0, 0}, kind,
                         skip_large);
  return launch<cplxf>(batch, dm, dn, alpha, dA, dlda, dipiv, dB, dldb, 0, status, st, Map{0, 0, 0}, kind,
                       skip_large);
}

// Varlen batch of small solves (m <= 64) in double, float and float complex:
// triangular solves, and LU- and Cholesky-factor solves fused per instance.
// (Double complex has the column-packed kernels, packed.cu.)
//
// The fully unrolled substitution (X in registers, one variant per row-group
// count) left the arithmetic waiting: in FP32 for instructions (10.5 of 18 stall
// cycles, 362 us for 8192 complex64 solves with m, n ~ U{8..64}), in FP64 for
// staging and for shared-memory operands with 12 warps per SM (FP64 pipe 69%
// busy, 717 us for 4097 double LU solves).  Here the substitution runs in
// blocks of rows with rolled loops (some 600 instructions, 50 to 60 registers):
//
//  * one CTA of four warps per instance; the hardware deals them to the SMs as
//    these free up (double, whose large instances take long: largest first within
//    groups of 256 instances, by a pass of a few microseconds);
//  * the triangle (square blocks) and the right-hand sides are copied to shared
//    memory asynchronously, all of an instance's loads in flight at once;
//  * a warp owns 16 columns, two lanes per column with half the rows of each
//    block (a last tile of at most 8 columns: four lanes with a quarter each, half
//    the instructions); block row J gathers
//        acc = B_J - sum_{I < J} L_JI X_I
//    from shared memory before its own steps, X overwrites B there, and the warp
//    writes its columns back row-contiguously;
//  * as in the single solve, row r of the triangle is first scaled by 1/a_rr and
//    B's row by alpha/a_rr, so that a solved value needs no further arithmetic;
//    the operations and their order are the single solve's, bit for bit.
//
// Blocks of 8 rows in FP32 (fewer loads per multiply-add); of 4 in FP64, where
// only the multiply-adds count and a block's own steps are the half-idle ones.
// Measured: 8192 complex64 solves 180 us, 4097 double LU solves 565 us (pipe 84% busy).
//
// The per-instance arithmetic does not depend on the batch it sits in.
#include <cuda_runtime.h>

#include "common.cuh"
#include "small.h"
#include "trace.h"

namespace {

constexpr int kWarps = 4;
constexpr int kCols = 16;  // columns per warp
constexpr int kLdX = kCols + 1;  // row pitch of the right-hand sides: column reads and row writes miss bank conflicts

// Index map from the solved lower-triangular form onto the operand: with rev,
// row r of the form is row m-1-r of the operand and of B; with tr, A is read
// transposed; with cj, conjugated.
struct Map {
  int rev, tr, cj;
};

// Rows per block and per lane, elements of the staged triangle.
template <class T>
struct Blk {
  static constexpr int kRows = sizeof(T) == sizeof(double) && !Elem<T>::kComplex ? 4 : 8;
  static constexpr int kNum = 64 / kRows;
  static constexpr int kTri = kNum * (kNum + 1) / 2 * kRows * kRows;
  // block (J, I), I <= J: kRows columns of kRows rows
  __device__ __forceinline__ static int at(int J, int I) { return (J * (J + 1) / 2 + I) * kRows * kRows; }
};

template <class T>
constexpr size_t smem_bytes() {
  return sizeof(T) * (Blk<T>::kTri + 128 + kWarps * 64 * kLdX);
}

// the rows of one lane in a column of a block (aligned to their size)
__device__ __forceinline__ void ldv(double (&v)[1], const double *p) { v[0] = *p; }
__device__ __forceinline__ void ldv(float (&v)[2], const float *p) {
  const float2 q = *reinterpret_cast<const float2 *>(p);
  v[0] = q.x;
  v[1] = q.y;
}
__device__ __forceinline__ void ldv(cplxf (&v)[2], const cplxf *p) {
  const float4 q = *reinterpret_cast<const float4 *>(p);
  v[0] = cplxf{q.x, q.y};
  v[1] = cplxf{q.z, q.w};
}
__device__ __forceinline__ void ldv(double (&v)[2], const double *p) {
  const double2 q = *reinterpret_cast<const double2 *>(p);
  v[0] = q.x;
  v[1] = q.y;
}
__device__ __forceinline__ void ldv(float (&v)[4], const float *p) {
  const float4 q = *reinterpret_cast<const float4 *>(p);
  v[0] = q.x;
  v[1] = q.y;
  v[2] = q.z;
  v[3] = q.w;
}
__device__ __forceinline__ void ldv(cplxf (&v)[4], const cplxf *p) {
  const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 2);
  v[0] = cplxf{a.x, a.y};
  v[1] = cplxf{a.z, a.w};
  v[2] = cplxf{b.x, b.y};
  v[3] = cplxf{b.z, b.w};
}

__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Start copying the lower-triangular form: a warp per stored column (row with
// tr), lanes along it.  Rows past m and entries above the diagonal are not
// written: they only reach values that are never used.  The diagonal is part of
// its block.
template <class T>
__device__ __forceinline__ void stage_a(T *sL, const T *__restrict__ A, int64_t lda, int m, bool unit, Map mp) {
  constexpr int kBlk = Blk<T>::kRows;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = warp; o < m; o += kWarps) {
    const T *line = A + (int64_t)(mp.rev ? m - 1 - o : o) * lda;
    for (int i = lane + (mp.tr ? 0 : o & ~31); i < (mp.tr ? o + 1 : m); i += 32) {
      const int r = mp.tr ? o : i, c = mp.tr ? i : o;
      if (r < c || (unit && r == c)) continue;
      copy_async(sL + Blk<T>::at(r / kBlk, c / kBlk) + (c % kBlk) * kBlk + r % kBlk, line + (mp.rev ? m - 1 - i : i));
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

// The staged columns of this warp (32 / LPC of them, LPC lanes each) solved in
// shared memory (sC: alpha / a_rr); cj: with conj(L), by solving for conj(X).
template <class T, int LPC>
__device__ __forceinline__ void solve_tile(const T *sL, const T *sC, T *X0, int m, int cj) {
  using E = Elem<T>;
  constexpr int kBlk = Blk<T>::kRows, kMine = kBlk / LPC, kTile = 32 / LPC;
  const int lane = threadIdx.x & 31;
  const int c = lane % kTile, h = lane / kTile;  // this lane's column of the tile and part of each block
  T *X = X0 + c;
  const int nblk = (m + kBlk - 1) / kBlk;
#pragma unroll 1
  for (int J = 0; J < nblk; ++J) {
    T acc[kMine];
    T *xJ = X + J * kBlk * kLdX;
#pragma unroll
    for (int q = 0; q < kMine; ++q) {
      T b = xJ[(kMine * h + q) * kLdX];
      if constexpr (E::kComplex) {
        if (cj) b.im = -b.im;
      }
      acc[q] = E::mul(sC[J * kBlk + kMine * h + q], b);
    }
    const T *L = sL + Blk<T>::at(J, 0) + kMine * h;
    const T *x = X;
#pragma unroll 1
    for (int I = 0; I < J; ++I, L += kBlk * kBlk, x += kBlk * kLdX) {
#pragma unroll
      for (int k = 0; k < kBlk; ++k) {
        const T xk = x[k * kLdX];
        T l[kMine];
        ldv(l, L + k * kBlk);
#pragma unroll
        for (int q = 0; q < kMine; ++q) acc[q] = E::fms(l[q], xk, acc[q]);
      }
    }
    // the block's own rows: row k is final after k steps; later updates of rows
    // at or above k touch values that are no longer used
    T out[kMine];
#pragma unroll
    for (int k = 0; k < kBlk; ++k) {
      if (h >= k / kMine) out[k % kMine] = acc[k % kMine];  // kept by the lane whose row it is
      if (k + 1 < kBlk) {
        const T xk = E::shfl(acc[k % kMine], (k / kMine) * kTile + c);
        T l[kMine];
        ldv(l, L + k * kBlk);
#pragma unroll
        for (int q = 0; q < kMine; ++q)
          if ((LPC - 1) * kMine + q > k) acc[q] = E::fms(l[q], xk, acc[q]);  // else: final in every part
      }
    }
    __syncwarp();  // every lane of a column has read this block's B
#pragma unroll
    for (int q = 0; q < kMine; ++q) xJ[(kMine * h + q) * kLdX] = out[q];
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
__device__ __forceinline__ void solve(T *sL, T *sR, T *sC, T *sX, const T *__restrict__ A, int64_t lda, T *B, int64_t ldb,
                                      int m, int n, T alpha, bool unit, Map mp) {
  using E = Elem<T>;
  constexpr int kBlk = Blk<T>::kRows;
  const int warp = threadIdx.x >> 5;
  T *X = sX + warp * 64 * kLdX;
  stage_a<T>(sL, A, lda, m, unit, mp);
  if (warp * kCols < n) stage_b<T>(X, B, ldb, m, n, warp * kCols, mp.rev);
  copies_wait();
  __syncthreads();
  if (threadIdx.x < m) {
    const int r = threadIdx.x;
    const T rv = unit ? E::one() : E::recip(sL[Blk<T>::at(r / kBlk, r / kBlk) + (r % kBlk) * (kBlk + 1)]);
    if constexpr (E::kComplex) {
      if (mp.cj) alpha.im = -alpha.im;
    }
    sR[r] = rv;
    sC[r] = E::mul(alpha, rv);
  }
  __syncthreads();
  if (!unit) {  // row r times 1/a_rr: a warp per row of blocks, two rows of a column per lane
    const int lane = threadIdx.x & 31;
    for (int J = warp; J * kBlk < m; J += kWarps) {
      T *L = sL + Blk<T>::at(J, 0);
      const T *r = sR + J * kBlk + 2 * lane % kBlk;
      for (int e = 2 * lane; e < (J + 1) * kBlk * kBlk; e += 64) {
        L[e] = E::mul(r[0], L[e]);
        L[e + 1] = E::mul(r[1], L[e + 1]);
      }
    }
    __syncthreads();
  }
  for (int j0 = warp * kCols; j0 < n; j0 += kWarps * kCols) {
    if (j0 >= kWarps * kCols) {
      stage_b<T>(X, B, ldb, m, n, j0, mp.rev);
      copies_wait();
      __syncwarp();
    }
    if (n - j0 <= kCols / 2)
      solve_tile<T, 4>(sL, sC, X, m, mp.cj);
    else
      solve_tile<T, 2>(sL, sC, X, m, mp.cj);
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

// An order of the instances: each group of 256 consecutive ones by decreasing
// work (m^2 times column tiles, eight classes per octave), the groups
// interleaved rank by rank.  Started in this order the last CTAs are short ones.
constexpr int kOrderGroup = 256;

__global__ void __launch_bounds__(kOrderGroup) batch_order_kernel(int batch, const int32_t *__restrict__ dm,
                                                                  const int32_t *__restrict__ dn, int32_t *order) {
  __shared__ int hist[256], first[256];
  const int t = threadIdx.x, g = blockIdx.x, b = g * kOrderGroup + t;
  hist[t] = 0;
  __syncthreads();
  int cls = 255, at = 0;
  if (b < batch) {
    const int m = dm[b], n = dn[b];
    if (m > 0 && m <= 64 && n > 0) {
      const uint64_t w = 8ull * m * m * (uint64_t)((n + kCols - 1) / kCols);
      const int lead = 63 - __clzll((long long)w);
      cls = 254 - min(254, 8 * lead + (int)((w >> (lead - 3)) & 7));
    }
    at = atomicAdd(&hist[cls], 1);
  }
  __syncthreads();
  // exclusive sums of the 256 classes, 32 at a time
  int v = hist[t];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, v, o);
    if ((t & 31) >= o) v += y;
  }
  first[t] = v;
  __syncthreads();
  int base = 0;
  for (int w = 0; w < (cls >> 5); ++w) base += first[32 * w + 31];
  if (b >= batch) return;
  const int rank = base + first[cls] - hist[cls] + at;
  const int full = batch / kOrderGroup, rest = batch % kOrderGroup;  // whole groups, and a last one of `rest`
  const int groups = full + (rest != 0);
  order[rank < rest || rest == 0 ? (int64_t)rank * groups + g
                                 : (int64_t)rest * groups + (int64_t)(rank - rest) * full + g] = b;
}

template <class T>
__global__ void __launch_bounds__(32 * kWarps) batch_kernel(const int32_t *__restrict__ dm,
                                                                const int32_t *__restrict__ dn,
                                                                const int32_t *__restrict__ dlda,
                                                                const int32_t *__restrict__ dldb,
                                                                const void *const *__restrict__ dA,
                                                                const int32_t *const *__restrict__ dipiv,
                                                                void *const *__restrict__ dB, T alpha, int unit,
                                                                const int32_t *__restrict__ order, uint32_t *status, Map mp, int kind,
                                                                int skip_large) {
  using E = Elem<T>;
  extern __shared__ __align__(16) unsigned char smem[];
  T *sL = reinterpret_cast<T *>(smem);
  T *sR = sL + Blk<T>::kTri;
  T *sC = sR + 64;
  T *sX = sC + 64;
  const int b = order != nullptr ? order[blockIdx.x] : blockIdx.x;
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
    solve<T>(sL, sR, sC, sX, A, lda, B, ldb, m, n, pass == 0 ? alpha : E::one(), un, pm);
  }
}

template <class T>
hsma_status_t launch(int32_t batch, const int32_t *dm, const int32_t *dn, const double *alpha, const void *const *dA,
                     const int32_t *dlda, const int32_t *const *dipiv, void *const *dB, const int32_t *dldb, int unit,
                     uint32_t *status, int32_t *order, cudaStream_t st, Map mp, int kind, int skip_large) {
  static DeviceFlags attr_done;
  if (!attr_done.test()) {
    HSMA_CUDA_TRY(cudaFuncSetAttribute(batch_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem_bytes<T>()));
    attr_done.set();
  }
  if constexpr (sizeof(T) == sizeof(double) && !Elem<T>::kComplex) {
    HsmaTraceScope ts("vbatched_schedule", st);
    batch_order_kernel<<<(batch + kOrderGroup - 1) / kOrderGroup, kOrderGroup, 0, st>>>(batch, dm, dn, order);
    HSMA_CUDA_TRY(cudaGetLastError());
  } else {
    order = nullptr;
  }
  HsmaTraceScope ts(kind == KIND_TRSM ? "vbatched_solve" : "vbatched_lu", st);
  batch_kernel<T><<<batch, 32 * kWarps, smem_bytes<T>(), st>>>(dm, dn, dlda, dldb, dA, dipiv, dB,
                                                                   hsma_alpha_as<T>(alpha), unit, order, status, mp, kind,
                                                                   skip_large);
  return hsma_from_cuda(cudaGetLastError());
}

}  // namespace

hsma_status_t hsma_blk_vbatched(int dtype, int32_t batch, const int32_t *dm, const int32_t *dn, const double *alpha,
                                const void *const *dA, const int32_t *dlda, void *const *dB, const int32_t *dldb,
                                int unit, uint32_t *status, int32_t *scratch, cudaStream_t st, int uplo, int trans,
                                int skip_large) {
  const bool op_lower = (uplo == HSMA_LOWER) != (trans != HSMA_NO_TRANS);
  const Map mp{op_lower ? 0 : 1, trans != HSMA_NO_TRANS ? 1 : 0, trans == HSMA_CONJ_TRANS ? 1 : 0};
  auto *f = dtype == HSMA_R32 ? launch<float> : dtype == HSMA_C64 ? launch<cplxf> : launch<double>;
  return f(batch, dm, dn, alpha, dA, dlda, nullptr, dB, dldb, unit, status, scratch, st, mp, KIND_TRSM, skip_large);
}

hsma_status_t hsma_blk_factor_vbatched(int dtype, int32_t batch, const int32_t *dm, const int32_t *dn,
                                       const double *alpha, const void *const *dA, const int32_t *dlda,
                                       const int32_t *const *dipiv, void *const *dB, const int32_t *dldb,
                                       uint32_t *status, int32_t *scratch, cudaStream_t st, int chol,
                                       int skip_large) {
  auto *f = dtype == HSMA_R32 ? launch<float> : dtype == HSMA_C64 ? launch<cplxf> : launch<double>;
  return f(batch, dm, dn, alpha, dA, dlda, dipiv, dB, dldb, 0, status, scratch, st, Map{0, 0, 0}, chol ? KIND_CHOL : KIND_LU,
           skip_large);
}

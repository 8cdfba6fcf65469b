// Persistent, warp-specialised tcgen05 product (BF16 x BF16 -> FP32 in tensor
// memory) behind the FP32-result mode and the emulated FP64 products; used by
// mixed.cu only.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include "blocked.h"
#include "common.cuh"
#include "oz_tables.cuh"
#include "tma.cuh"
#include "trace.h"

namespace {

// ---------------------------------------------------------------------------
// tcgen05 BF16 x BF16 -> FP32 update:  C (M x N, column-major fp32) =
// beta*C - A' B'^T with A' (M x K) and B' (N x K) row-major BF16 (K-major).
// ---------------------------------------------------------------------------
constexpr int TC_BM = 128;             // rows of a tile per CTA
constexpr int TC_PM = 2 * TC_BM;       // rows of a tile (a pair of CTAs)
constexpr int TC_BK = 64;              // K-block of a pipeline stage: 128-byte rows, 128-byte swizzle
constexpr int TC_A_BYTES = TC_BM * TC_BK * 2;
constexpr uint32_t TC_TMEM_COLS = 512;  // all of the SM's tensor memory (one CTA per SM)

// A pair of CTAs (a cluster on two SMs) forms 256 x BN results with one
// cta_group::2 MMA stream: each CTA stages its 128 rows of A and half of B's
// rows, and holds its 128 rows of the accumulators.  With one CTA per tile
// (128 x 256) every K-block moved 48 KB into an SM's shared memory and 48 KB out
// of it to the tensor core, 768 cycles at 128 bytes per cycle against the 512
// its products take (712 measured); a pair moves 32 KB each way.
// BN = 256 does the most products per operand byte, BN = 128 gives twice the
// tiles when a launch has too few for the SMs.
template <int BN>
struct TcTile {
  static constexpr int B_ROWS = BN / 2;  // rows of B staged per CTA
  static constexpr int BLOCK_BYTES = TC_A_BYTES + B_ROWS * TC_BK * 2;  // one K-block of A and B
  // K-blocks per stage: a narrow tile's products of one block (256 cycles) do not
  // cover the issue loop's round, a wide tile's do and prefer more stages
  static constexpr int SUB = BN == 256 ? 1 : 2;
  static constexpr int STAGE_BYTES = SUB * BLOCK_BYTES;
  static constexpr int STAGES = BN == 256 ? 6 : 4;
  static constexpr int SMEM = STAGES * STAGE_BYTES + 1024;
  static constexpr int ACCS = TC_TMEM_COLS / BN;  // accumulators in tensor memory
  // instruction descriptor: FP32 accumulator, BF16 A and B, both K-major, M x N
  static constexpr uint32_t IDESC =
      (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(TC_PM >> 4) << 24);
  static_assert(SMEM <= 227 * 1024 - 512, "stages fit the shared memory of one CTA");
  static_assert(STAGE_BYTES % 1024 == 0, "every stage starts on a swizzle-pattern boundary");
};

// Shared-memory matrix descriptor: K-major operand, rows of 128 bytes in groups
// of 8 (1024 bytes apart), 128-byte swizzle.
__device__ __forceinline__ uint64_t sw_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1u << 16;            // leading-dimension offset (unused when swizzled)
  d |= (uint64_t)(1024u >> 4) << 32;  // stride between 8-row groups
  d |= (uint64_t)1u << 46;            // descriptor version
  d |= (uint64_t)2u << 61;            // swizzle mode
  return d;
}

// Address, in the cluster's shared memory, of the same variable in CTA `rank`.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// true in one lane of a converged warp (the same one every time)
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

// every thread of both CTAs
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Arrive on an mbarrier of either CTA of the pair (address from cluster_addr) to
// hand back an accumulator.  Relaxed: what it orders are this warp's tensor-memory
// loads, complete at their tcgen05.wait::ld; a release at cluster scope would wait
// for the epilogue's global stores to be acknowledged as well.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}

// arrive on the mbarrier at this offset in both CTAs once the pair's MMAs issued so far are done
__device__ __forceinline__ void tc_commit_pair(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}

// TMA load into this CTA's shared memory, completing on an mbarrier of the pair
__device__ __forceinline__ void tma_load_3d_pair(void *dst, const CUtensorMap *map, uint32_t bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, "
      "%5}], [%2];" ::"r"(smem_u32(dst)),
      "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Epilogues of the tensor-core product:
//   TC_F32: C32 = beta*C32 - acc                    (the FP32-result update)
//   TC_OZ:  C64 -/+= 2^(rexp[i] + cexp[j]) * S      (an emulated FP64 product:
//           S, an integer, from its residues modulo the kOzP moduli of oz_tables.cuh)
enum { TC_F32 = 0, TC_OZ = 1 };

constexpr int kTcMaxPairs = 8;

struct TcArgs {
  float *C32;
  double *C64;
  int64_t ldc;
  float beta;      // TC_F32
  int beta0;       // TC_OZ: 0 = the product overwrites C64 (old values not read)
  int negate;      // TC_OZ: add the product instead of subtracting it
  const int *rexp;  // TC_OZ: row exponents of A
  const int *cexp;  // TC_OZ: column exponents of B
  uint32_t *scratch;  // TC_OZ: 2 kOzTileWords words per CTA (residue bytes of a tile being written and one being converted)
  int M, N, K;
  int tri;          // row tile i0 needs k < i0 + TC_PM only
  int row0;         // TC_OZ, tri: row 0 and column 0 are this row and column of the operand
  int npairs;       // TC_F32: slice pairs summed in the accumulator
  int band;         // tile rows per band of the tile order (set by the launcher)
  uint8_t pa[kTcMaxPairs], pb[kTcMaxPairs];  // TC_F32: slice of A and of B for each pair
  const int *skip;  // device flag: when set, the launch does nothing
  unsigned int *err;
  uint64_t limit_ns;
  // TC_F32 side outputs: BF16 splits of the stored values, the right operands
  // of the next products (null: none)
  __nv_bfloat16 *xs2;  // rows < rows2: [col][ld2] hi at k = row; terms2 = 3 adds lo at nb2 + row, hi at 2 nb2 + row
  int ld2, nb2, terms2, rows2;
  __nv_bfloat16 *xs3;  // rows r3 .. r3 + rows3 - 1: three exact slices [s][col][ld3] at k = row - r3, slice stride per3
  int64_t per3;
  int ld3, r3, rows3;
};

// x = hi + lo with hi, lo in BF16 (the split of the FP32-result products)
__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16 &hi, __nv_bfloat16 &lo) {
  hi = __float2bfloat16_rn(x);
  lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

// x = a + b + c exactly (24 bits in three BF16 slices)
__device__ __forceinline__ void split3_bf16(float x, __nv_bfloat16 &a, __nv_bfloat16 &b, __nv_bfloat16 &c) {
  a = __float2bfloat16_rn(x);
  float r = x - __bfloat162float(a);
  b = __float2bfloat16_rn(r);
  r -= __bfloat162float(b);
  c = __float2bfloat16_rn(r);
}

// 32 lanes x 16 consecutive 32-bit tensor-memory columns into registers
// (completion awaited separately with tcgen05.wait::ld).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t *v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}

// Conversion of ncols columns (a multiple of 4) from column c_beg on of a 128 x BN
// tile at (m0, n0), rows 32 quarter + lane, from the residues in half h of the
// CTA's scratch: four columns at a time, the next four's loads in flight.
template <int BN>
__device__ __forceinline__ void oz_convert(const TcArgs &p, int cid, int h, int m0, int n0, int quarter, int c_beg,
                                           int ncols) {
  const int rl = quarter * 32 + (threadIdx.x & 31), row = m0 + rl;
  const int cols = min(ncols, p.N - n0 - c_beg);
  if (row >= p.M || cols <= 0) return;
  const uint32_t *mine = p.scratch + oz_scratch_at(cid, h, c_beg) + rl;
  const int rx = p.rexp[row] - 2 * kOzFrac;
  const int *cx = p.cexp + n0 + c_beg;
  double *crow = p.C64 + row + (int64_t)(n0 + c_beg) * p.ldc;
  uint32_t nw[kOzP];
  double nold[4];
  auto load4 = [&](int c0) {
#pragma unroll
    for (int l = 0; l < kOzP; ++l) nw[l] = mine[l * kOzPlaneWords + c0 / 4 * TC_BM];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      nold[j] = (p.beta0 != 0 && c0 + j < cols) ? crow[(int64_t)(c0 + j) * p.ldc] : 0.0;
  };
  load4(0);
#pragma unroll 1
  for (int c0 = 0; c0 < cols; c0 += 4) {
    uint32_t w[kOzP];
    double old[4];
    int e[4];
    uint64_t y[4];
    bool normal = true;
#pragma unroll
    for (int l = 0; l < kOzP; ++l) w[l] = nw[l] ^ 0x80808080u;
#pragma unroll
    for (int j = 0; j < 4; ++j) old[j] = nold[j];
    if (c0 + 4 < cols) load4(c0 + 4);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      y[j] = oz_crt(w, j, e[j]);
      e[j] += rx + __ldg(cx + min(c0 + j, cols - 1));
      normal &= (y[j] == 0 && e[j] < kOzExpFlag) || oz_scales(e[j]);
    }
    double x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = oz_scaled(y[j], e[j]);
    if (!normal) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = __ldg(cx + min(c0 + j, cols - 1));
        bool bad = rx >= kOzExpFlag;
        if (c >= kOzExpFlag) {
          bad |= p.tri == 0 || row + p.row0 >= (c >> 16) - 1;
          e[j] += (int)(int16_t)(c & 0xffff) - c;
        }
        x[j] = bad ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(__longlong_as_double((long long)y[j]), e[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (c0 + j < cols) crow[(int64_t)(c0 + j) * p.ldc] = p.negate ? old[j] + x[j] : old[j] - x[j];
  }
}

// Persistent, warp-specialised product: warp 0 loads operand stages by TMA,
// warp 1 issues the MMAs, warps 2..9 drain accumulators, and (TC_OZ) warps
// 10..17 turn a finished tile's residues into FP64.  A tile is a sequence of
// accumulation units: one for TC_F32 (every slice pair over the whole K range),
// and for TC_OZ one per modulus and K chunk of kOzChunk (the longest whose FP32
// sums of residue products stay exact).  The accumulators (512 tensor-memory
// columns) rotate between units, so one unit's epilogue runs while the next
// units' products accumulate.  Tiles are dealt round-robin to the pairs of CTAs
// (one CTA per SM).  Operands are 3-D: (K, rows, slice).
//
// In a pair, both producers fill their own stage and signal the first CTA's
// `full`; its MMA thread issues for both; its commits release the stage and hand
// over the accumulator in both CTAs; both CTAs' epilogue warps return the
// accumulator to the first CTA's acc_empty.  Everything else is per CTA.
constexpr int TC_WARPS = 10;
constexpr int TC_EPI_WARPS = 8;
constexpr int TC_CRT_WARPS = 8;

template <int MODE>
constexpr int tc_threads() {
  return 32 * (TC_WARPS + (MODE == TC_OZ ? TC_CRT_WARPS : 0));
}

template <int MODE, int BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(tc_threads<MODE>(), 1) tc_gemm_kernel(const __grid_constant__ CUtensorMap mapA,
                                                                        const __grid_constant__ CUtensorMap mapB,
                                                                        const __grid_constant__ TcArgs p) {
  using TL = TcTile<BN>;
  constexpr int TC_BN = BN, TC_STAGES = TL::STAGES, TC_STAGE_BYTES = TL::STAGE_BYTES, NACC = TL::ACCS;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[TC_STAGES];
  __shared__ __align__(8) uint64_t empty[TC_STAGES];
  __shared__ __align__(8) uint64_t acc_full[NACC];
  __shared__ __align__(8) uint64_t acc_empty[NACC];
  __shared__ __align__(8) uint64_t res_full[2];   // TC_OZ: residues of a tile complete in scratch half
  __shared__ __align__(8) uint64_t res_empty[2];  // ... and converted
  __shared__ __align__(8) uint64_t drained;
  __shared__ uint32_t tmem_base;
  if (p.skip != nullptr && *(volatile const int *)p.skip != 0) return;
  unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int M = p.M, N = p.N;
  const int nslices = MODE == TC_OZ ? kOzP : p.npairs;  // passes over the K range per tile
  const uint32_t rank = cluster_rank();
  const int cid = blockIdx.x >> 1, ncl = gridDim.x >> 1;  // the pair and the number of pairs
  const int tiles_m = (M + TC_PM - 1) / TC_PM, tiles_n = (N + TC_BN - 1) / TC_BN;
  const int ntiles = tiles_m * tiles_n;
  // TC_OZ with no more than one tile per pair: the conversion warps have nothing
  // to convert until the end, so they drain accumulators too
  const bool single = MODE == TC_OZ && ntiles <= ncl;
  // Tiles run in bands of p.band tile rows, column by column inside a band.
  // With 8 tile rows the tiles in flight at once (one per pair of SMs) cover
  // about 8 row tiles x 10 column tiles, the fewest operand rows; long TC_F32 products
  // take one band over all rows (column-major order), so the right operand is
  // shared by every row tile in flight.
  const int G = max(1, p.band);
  auto tile_k = [&](int t, int &m0, int &n0) {  // tile -> its origin and K-block count
    const int band = t / (G * tiles_n);
    const int gb = min(G, tiles_m - band * G);
    const int idx = t - band * G * tiles_n;
    int pm = band * G + idx % gb;
    if (p.tri) pm = tiles_m - 1 - pm;  // the longest K ranges first: the tail is short tiles
    m0 = pm * TC_PM + (int)rank * TC_BM;  // this CTA's rows
    n0 = (idx / gb) * TC_BN;
    const int kall = p.tri ? min(p.K, (pm + 1) * TC_PM) : p.K;
    return (kall + TC_BK - 1) / TC_BK;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < TC_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < NACC; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 2 * (TC_EPI_WARPS + (single ? TC_CRT_WARPS : 0)));
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&res_full[b], TC_EPI_WARPS);
      mbar_init(&res_empty[b], TC_CRT_WARPS);
    }
    mbar_init(&drained, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(TC_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers are initialised and tensor memory allocated
  tc_fence_after();
  const uint32_t tmem = tmem_base;

  if (warp == 0) {
    // producer: TMA loads into a ring of stages, across tiles.  The whole warp
    // runs the loop and one elected lane issues (here and below): as a branch of
    // a single lane the MMA loop took 800 cycles per K block whatever the tile,
    // this form 540 (BN = 128) to 560 (BN = 256, 512 of them products).
    const uint32_t bar0 = cluster_addr(&full[0], 0);
    int s = 0;
    uint32_t phase = 1;  // the first round finds every stage empty
    uint32_t fills = 0;  // stages filled so far
    bool ok = true;
    for (int t = cid; t < ntiles && ok; t += ncl) {
      int m0, n0;
      const int nk = tile_k(t, m0, n0);
      for (int q = 0; q < nslices && ok; ++q) {
        const int sa = MODE == TC_OZ ? q : p.pa[q], sb = MODE == TC_OZ ? q : p.pb[q];
        for (int kb = 0; kb < nk; kb += TL::SUB) {
          if (!mbar_wait_bounded(&empty[s], phase, p.limit_ns, p.err)) {
            ok = false;
            break;
          }
          if (elect_one()) {
            unsigned char *st = smem + s * TC_STAGE_BYTES;
            const uint32_t bar = bar0 + (uint32_t)s * 8u;
            const int nsub = min(TL::SUB, nk - kb);  // a slice's last stage may hold fewer blocks
            if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * nsub * TL::BLOCK_BYTES);
#pragma unroll
            for (int u = 0; u < TL::SUB; ++u, st += TL::BLOCK_BYTES) {
              if (u > 0 && u >= nsub) break;
              tma_load_3d_pair(st, &mapA, bar, (kb + u) * TC_BK, m0, sa);
              tma_load_3d_pair(st + TC_A_BYTES, &mapB, bar, (kb + u) * TC_BK, n0 + (int)rank * TL::B_ROWS, sb);
            }
          }
          __syncwarp();
          ++fills;
          if (++s == TC_STAGES) {
            s = 0;
            phase ^= 1;
          }
        }
      }
    }
    // A CTA leaves with nothing outstanding: every stage has been released (so its
    // loads have landed and the releases have arrived), and in the second CTA, where
    // nobody else waits for them, the last commits have.
    for (int k = 0; k < TC_STAGES && ok; ++k) {
      ok = mbar_wait_bounded(&empty[s], phase, p.limit_ns, p.err);
      if (++s == TC_STAGES) {
        s = 0;
        phase ^= 1;
      }
    }
    // after a wait that gave up: the loads of the last fill of every stage
    if (!ok && rank == 0)
      for (uint32_t f = fills > TC_STAGES ? fills - TC_STAGES : 0; f < fills; ++f)
        mbar_wait_bounded(&full[f % TC_STAGES], (f / TC_STAGES) & 1, p.limit_ns, p.err);
    if (rank != 0) mbar_wait_bounded(&drained, 0, p.limit_ns, p.err);
  } else if (warp == 1) {
    if (rank == 0) {
      // MMA issuer (first CTA of the pair): per unit, wait for a drained
      // accumulator, then four K = 16 steps per stage; each stage is released by
      // a commit, the unit by another
      const uint64_t desc0 = sw_desc(smem_u32(smem));
      int s = 0, b = 0;
      uint32_t phase = 0, acc_phase = 1;  // the first round finds every accumulator drained
      bool ok = true;
      for (int t = cid; t < ntiles && ok; t += ncl) {
        int m0, n0;
        const int nk = tile_k(t, m0, n0);
        const int total = nslices * nk;  // K blocks of the tile, slice by slice
        for (int g0 = 0; g0 < total && ok;) {
          // the unit's K blocks: all of them, or (TC_OZ) the next chunk of this modulus
          const int glen = MODE == TC_OZ ? min(kOzChunk / TC_BK, nk - g0 % nk) : total;
          if (!mbar_wait_bounded(&acc_empty[b], acc_phase, p.limit_ns, p.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t acc_cols = tmem + (uint32_t)(b * BN);
          for (int kb = 0, nsub; kb < glen; kb += nsub) {
            // blocks in this stage (TC_F32's unit spans slices, each with its own last stage)
            nsub = TL::SUB == 1 ? 1 : min(TL::SUB, MODE == TC_OZ ? glen - kb : nk - kb % nk);
            if (!mbar_wait_bounded(&full[s], phase, p.limit_ns, p.err)) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (elect_one()) {
              const uint64_t d0 = desc0 + (uint64_t)(s * (TC_STAGE_BYTES >> 4));
#pragma unroll
              for (int u = 0; u < TL::SUB; ++u) {
                if (u > 0 && u >= nsub) break;
                const uint64_t da = d0 + (uint64_t)(u * (TL::BLOCK_BYTES >> 4)), db = da + (TC_A_BYTES >> 4);
#pragma unroll
                for (int kk = 0; kk < TC_BK / 16; ++kk)
                  asm volatile(
                      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(acc_cols),
                      "l"(da + 2ull * kk), "l"(db + 2ull * kk), "r"(TL::IDESC), "r"(kb + u + kk)
                      : "memory");
              }
              tc_commit_pair(&empty[s]);
              if (kb + nsub == glen) tc_commit_pair(&acc_full[b]);
            }
            __syncwarp();
            if (++s == TC_STAGES) {
              s = 0;
              phase ^= 1;
            }
          }
          g0 += glen;
          if (++b == NACC) {
            b = 0;
            acc_phase ^= 1;
          }
        }
      }
      // every issued product has finished before tensor memory is released, also
      // when a wait above gave up (the second CTA's producer waits there)
      if (elect_one()) tc_commit_pair(&drained);
      __syncwarp();
      mbar_wait_bounded(&drained, 0, p.limit_ns, p.err);
    }
  } else if (warp < TC_WARPS || single) {
    // epilogue warps: thread = one row of the 128-row tile (its tensor-memory
    // lane); two warps (or four) per lane quarter split the columns.
    const int ew = warp - 2;
    const int width = single ? TC_BN / 4 : TC_BN / 2;  // columns per warp
    const int quarter = warp & 3, cbeg = (ew >> 2) * width;
    constexpr int CW = 16;  // columns per chunk: keeps ten warps within the register file
    int i = 0;
    bool ok = true;
    for (int t = cid; t < ntiles && ok; t += ncl) {
      int m0, n0;
      const int nk = tile_k(t, m0, n0);
      const int row = m0 + quarter * 32 + lane;
      if constexpr (MODE == TC_OZ) {
        // Every unit: residues of the exact FP32 sums, four columns to a word of
        // this half of the CTA's scratch (chunks of one modulus after the first
        // add to the byte that the same thread wrote).
        const int ti = (t - cid) / ncl, h = ti & 1;
        if (ti >= 2) {
          ok = __all_sync(0xffffffffu, mbar_wait_bounded(&res_empty[h], ((ti >> 1) - 1) & 1, p.limit_ns, p.err));
          if (!ok) break;
        }
        uint32_t *mine = p.scratch + oz_scratch_at(blockIdx.x, h, cbeg) + quarter * 32 + lane;
        const int cols = min(width, N - n0 - cbeg);  // this warp's columns inside the matrix
        for (int l = 0; l < kOzP && ok; ++l) {
          const float mod = c_oz.modf[l], inv = c_oz.inv[l];
          for (int g0 = 0; g0 < nk; g0 += kOzChunk / TC_BK, ++i) {
            const int b = i % NACC;
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(&acc_full[b], (i / NACC) & 1, p.limit_ns, p.err));
            if (!ok) break;
            tc_fence_after();
            uint32_t *dst = mine + l * kOzPlaneWords;
#pragma unroll 2
            for (int c0 = 0; c0 < cols; c0 += CW, dst += CW / 4 * TC_BM) {
              uint32_t v[CW];
              tmem_ld16(tmem + (uint32_t)(b * BN) + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(cbeg + c0), v);
              asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
              for (int w = 0; w < CW / 4; ++w) {
                float r[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) r[j] = oz_residue(__uint_as_float(v[4 * w + j]), mod, inv);
                if (g0 != 0) oz_add_bytes(r, dst[w * TC_BM], mod, inv);
                dst[w * TC_BM] = oz_pack_bytes(r);
              }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(cluster_addr(&acc_empty[b], 0));  // this warp is done with accumulator b
          }
        }
        if (!ok) break;
        if (single) {  // each thread converts what it wrote
          oz_convert<BN>(p, blockIdx.x, h, m0, n0, quarter, cbeg, width);
          continue;
        }
        if (lane == 0) mbar_arrive(&res_full[h]);  // (after the last unit's __syncwarp)
        if (t + ncl >= ntiles) oz_convert<BN>(p, blockIdx.x, h, m0, n0, quarter, cbeg + TC_BN / 4, TC_BN / 4);
      } else {
        // the old values of the next 16-column chunk are loaded before this chunk's stores
        const int b = i % NACC;
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(&acc_full[b], (i / NACC) & 1, p.limit_ns, p.err));
        if (!ok) break;
        ++i;
        tc_fence_after();
        float old[CW], nxt[CW];
        auto load_chunk = [&](int c0, float *dst) {
#pragma unroll
          for (int j = 0; j < CW; ++j) {
            const int col = n0 + c0 + j;
            dst[j] = (p.beta != 0.0f && row < M && col < N) ? __ldcs(p.C32 + row + (int64_t)col * p.ldc) : 0.0f;
          }
        };
        load_chunk(cbeg, nxt);
#pragma unroll 1
        for (int c0 = cbeg; c0 < cbeg + TC_BN / 2; c0 += CW) {
#pragma unroll
          for (int j = 0; j < CW; ++j) old[j] = nxt[j];
          if (c0 + CW < cbeg + TC_BN / 2) load_chunk(c0 + CW, nxt);
          uint32_t v[CW];
          tmem_ld16(tmem + (uint32_t)(b * BN) + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0, v);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (row < M && nk > 0) {
#pragma unroll
            for (int j = 0; j < CW; ++j) {
              const int col = n0 + c0 + j;
              if (col < N) {
                const float a = __uint_as_float(v[j]);
                const float y = (p.beta == 1.0f) ? (old[j] - a) : fmaf(p.beta, old[j], -a);
                __stcs(p.C32 + row + (int64_t)col * p.ldc, y);
                if (p.xs2 != nullptr && row < p.rows2) {
                  __nv_bfloat16 hi, lo;
                  split_bf16(y, hi, lo);
                  __nv_bfloat16 *o = p.xs2 + (int64_t)col * p.ld2 + row;
                  o[0] = hi;
                  if (p.terms2 == 3) {
                    o[p.nb2] = lo;
                    o[2 * p.nb2] = hi;
                  }
                }
                if (p.xs3 != nullptr && row >= p.r3 && row < p.r3 + p.rows3) {
                  __nv_bfloat16 x0, x1, x2;
                  split3_bf16(y, x0, x1, x2);
                  __nv_bfloat16 *o = p.xs3 + (int64_t)col * p.ld3 + (row - p.r3);
                  o[0] = x0;
                  o[p.per3] = x1;
                  o[2 * p.per3] = x2;
                }
              }
            }
          }
        }
        // this warp is done with accumulator b
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(cluster_addr(&acc_empty[b], 0));
      }
    }
  } else if constexpr (MODE == TC_OZ) {
    // Conversion warps (the rows and columns of the epilogue warps): a tile's
    // integers from their residues, one addition to C each.  Run by the epilogue
    // warps between units this held the accumulators for 110 us per 128 x 256
    // tile, longer than the products of K = 1024 take.
    const int cw = warp - TC_WARPS;
    for (int t = cid, ti = 0; t < ntiles; t += ncl, ++ti) {
      int m0, n0;
      tile_k(t, m0, n0);
      const int h = ti & 1;
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&res_full[h], (ti >> 1) & 1, p.limit_ns, p.err))) break;
      // the CTA's last tile is shared with the epilogue warps, which are done
      oz_convert<BN>(p, blockIdx.x, h, m0, n0, cw & 3, (cw >> 2) * (TC_BN / 2), t + ncl >= ntiles ? TC_BN / 4 : TC_BN / 2);
      __syncwarp();
      if (lane == 0) mbar_arrive(&res_empty[h]);
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // no arrival or product of the other CTA is outstanding
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS)
                 : "memory");
  }
}

// 3-D tensor map over BF16 operand slices (K contiguous, rows, slice), one
// box = TC_BK K-values x box_rows rows of one slice, swizzled over its row
// width as the shared-memory descriptor expects.
bool make_slice_map(CUtensorMap *map, const void *base, uint64_t K, uint64_t rows, uint64_t slices,
                    uint32_t box_rows, uint64_t ld, uint64_t sst) {
  PFN_encodeTiled enc = hsma_encode_fn();
  if (enc == nullptr || (uintptr_t)base % 16 != 0 || (ld * 2) % 16 != 0 || (sst * 2) % 16 != 0 || K > ld) return false;
  const cuuint64_t dims[3] = {K, rows, slices};
  const cuuint64_t strides[2] = {ld * 2, sst * 2};
  const cuuint32_t box[3] = {(cuuint32_t)TC_BK, box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Layout of an operand's slice stack in memory: rows, K extent addressable
// from the base (0: the product's K), row stride and slice stride in elements
// (0: dense, ld = K extent, sst = rows * ld).  A view into a larger stack (a
// row and K offset) keeps the stack's strides.
struct SliceLayout {
  int64_t rows = 0, kext = 0, ld = 0, sst = 0;
};

// Launch the persistent product.  A: sa slices of M x K (row-major), B: sb
// slices of N x K.  TC_F32: a0 names the slice pairs (one pair of slice 0 unless
// given); TC_OZ: slice l of both holds residues modulo modulus l.  One CTA per SM.
template <int MODE, int BN>
hsma_status_t tc_gemm_tiled(const __nv_bfloat16 *Ap, int sa, const __nv_bfloat16 *Bp, int sb, const TcArgs &a0,
                      const char *phase, cudaStream_t st, SliceLayout la, SliceLayout lb) {
  if (a0.M <= 0 || a0.N <= 0) return HSMA_OK;
  if (a0.K % TC_BK != 0 || a0.K <= 0) return HSMA_ERR_INVALID_ARG;
  static DeviceFlags attr;
  if (!attr.test()) {
    HSMA_CUDA_TRY(
        cudaFuncSetAttribute(tc_gemm_kernel<MODE, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, TcTile<BN>::SMEM));
    attr.set();
  }
  const int tiles_m = (a0.M + TC_PM - 1) / TC_PM, tiles_n = (a0.N + BN - 1) / BN;
  CUtensorMap ma, mb;
  auto dense = [&](SliceLayout l, int64_t rows) {
    if (l.rows == 0) l.rows = rows;
    if (l.kext == 0) l.kext = a0.K;
    if (l.ld == 0) l.ld = l.kext;
    if (l.sst == 0) l.sst = l.rows * l.ld;
    return l;
  };
  la = dense(la, a0.M);
  lb = dense(lb, a0.N);
  if (la.kext < a0.K || lb.kext < a0.K) return HSMA_ERR_INVALID_ARG;
  if (!make_slice_map(&ma, Ap, (uint64_t)la.kext, (uint64_t)la.rows, (uint64_t)sa, TC_BM, (uint64_t)la.ld,
                      (uint64_t)la.sst) ||
      !make_slice_map(&mb, Bp, (uint64_t)lb.kext, (uint64_t)lb.rows, (uint64_t)sb, TcTile<BN>::B_ROWS, (uint64_t)lb.ld,
                      (uint64_t)lb.sst))
    return HSMA_ERR_CUDA;
  TcArgs a = a0;
  if constexpr (MODE == TC_OZ) {
    if (sa != kOzP || sb != kOzP || a.K > kOzMaxK || a.scratch == nullptr) return HSMA_ERR_INVALID_ARG;
  } else {
    if (a.npairs == 0) {
      a.npairs = 1;
      a.pa[0] = a.pb[0] = 0;
    }
    if (a.npairs > kTcMaxPairs) return HSMA_ERR_INVALID_ARG;
    for (int q = 0; q < a.npairs; ++q)
      if (a.pa[q] >= sa || a.pb[q] >= sb) return HSMA_ERR_INVALID_ARG;
  }
  a.err = hsma_dev_error_ptr();
  if (a.err == nullptr) return HSMA_ERR_CUDA;
  if (a.limit_ns == 0) a.limit_ns = 4000000000ull;
  const int ntiles = tiles_m * tiles_n;
  a.band = MODE == TC_OZ || a.K <= 2048 ? 8 : tiles_m;
  const int grid = 2 * std::max(1, std::min(ntiles, hsma_sm_count() / 2));
  HsmaTraceScope ts(phase, st);
  tc_gemm_kernel<MODE, BN><<<grid, tc_threads<MODE>(), TcTile<BN>::SMEM, st>>>(ma, mb, a);
  HSMA_CUDA_TRY(cudaGetLastError());
  return HSMA_OK;
}

// Tile width: the one whose busiest pair of CTAs has the least to do, a tile of
// BN columns counting BN + 96 (a 256 x 128 tile takes about 0.64 of the time of
// a 256 x 256 one).
template <int MODE>
hsma_status_t tc_gemm(const __nv_bfloat16 *Ap, int sa, const __nv_bfloat16 *Bp, int sb, const TcArgs &a0,
                      const char *phase, cudaStream_t st, SliceLayout la = {}, SliceLayout lb = {}) {
  const int64_t tm = (a0.M + TC_PM - 1) / TC_PM, pairs = hsma_sm_count() / 2;
  auto cost = [&](int bn) { return (tm * ((a0.N + bn - 1) / bn) + pairs - 1) / pairs * (bn + 96); };
  if (cost(128) < cost(256)) return tc_gemm_tiled<MODE, 128>(Ap, sa, Bp, sb, a0, phase, st, la, lb);
  return tc_gemm_tiled<MODE, 256>(Ap, sa, Bp, sb, a0, phase, st, la, lb);
}

}  // namespace

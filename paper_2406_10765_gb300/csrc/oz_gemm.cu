// FP64-accurate complex GEMM on the FP16 tensor cores (an Ozaki-type split
// of each operand into short integer slices), for the dense products of the
// Rayleigh-Ritz step -- the Cholesky and triangular-inverse updates, the
// Householder panel updates and the back-transformation of the small
// eigensolve (Syevd, Sec. III-D) -- which the FP64 pipe of this part runs at
// only ~1.2 TFLOP/s.
//
// Arithmetic (C = op(A) op(B), complex, K = inner dimension):
//   * Real form: row i of op(A) becomes one real row over K' = 2K,
//     (re_k, im_k) interleaved; column j of op(B) becomes two real rows,
//     (re, -im) and (im, re), so D[i][2j] = Re C_ij and D[i][2j+1] = Im C_ij.
//   * Each real row r is scaled by a power of two 2^e_r so that its largest
//     entry lies in [1/2, 1), and the scaled entry x is written exactly (to
//     2^-56) as x = sum_{p=1..S} d_p 2^(-BETA p) with integer digits,
//     |d_1| <= 2^BETA, |d_p| <= 2^(BETA-1), stored as FP16 (S = 8, BETA = 7).
//   * The slice products d_p(a) d_q(b) with p + q = g are summed in one FP32
//     tensor-memory accumulator per group g (g = 2..S+1; the pairs with
//     p + q > S + 1 are below 2^-55 of the largest product and dropped).  Over
//     a chunk of 96 real K every partial sum is an integer below 2^22 (two
//     pairs of at most 2^13 and six of at most 2^12 per K: 2.5 2^14 96), so
//     the FP32 accumulation is exact whatever its rounding.
//   * After each chunk the epilogue adds every group, shifted to a common
//     binary point 2^-L, into a 64-bit integer per output (exact except for
//     a rounding of the lowest groups below 2^-L), and at the end converts
//     to FP64 and removes the row and column scales.
// The error is at most 5.5 K' 2^-55 max|a_i| max|b_j| per entry (the row and
// column maxima; each real term is off by at most 1.375 2^-55 in scaled
// units -- the 2^-57 roundings of both digit expansions and the dropped
// pairs -- and the scales add a factor of at most 4), plus the final
// rounding to FP64: inside the usual FP64 bound K' u |a||b| for rows
// without large internal dynamic range.
//
// Kernel: tile of 128 complex rows x 32 complex columns (128 x 64 real) per
// CTA; warp 0 = TMA producer, warp 1 = MMA issuer (one thread), warps 2..9 =
// epilogue.  Two shared-memory stages of 32 real K, each holding all S slices
// of the A and B tiles (64-byte swizzle); eight 64-column FP32 accumulators
// fill the 512 tensor-memory columns.
//
// The slices of B lie one after the other in a stage, behind three slices of
// zeros, and the accumulators of the groups one after the other in tensor
// memory.  So slice p of A times four consecutive slices of B is ONE MMA of
// 256 columns onto four consecutive groups, the pairs that do not exist
// (q < 1) multiplying zeros: 12 MMAs of one shape per 16 K, 8 onto the upper
// four groups and 4 onto the lower four, instead of 36 of 64 columns.  A is
// read from shared memory 12 times instead of 36 (94 B/clock at the tensor
// peak instead of 192; 128 are available), and the issuing thread no longer
// limits the rate.  The two halves of the groups are emptied half a chunk
// apart, so that the MMAs of one run while the epilogue reads the other.
// Measured, 3,456 x 1,152 x 3,456: 6.15 ms with one MMA per slice pair, 3.35 ms
// so (33 TFLOP/s FP64-equivalent).  What it issues, zeros included, is 1.58
// PFLOP/s, 0.82 of the measured cuBLAS burst rate, with the tensor pipe active
// 74% of the time: that pipe bounds it, a quarter of its work for zeros, and the
// last of 6.4 waves (81% without it).  Operand reads are not at their limit.
// Every mbarrier wait is bounded; on timeout the CTA records an error word,
// frees its tensor memory and returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>
#include <mutex>

#include "oz_gemm.cuh"
#include "pw_internal.cuh"
#include "umma.cuh"

namespace {

using namespace pw_umma;

constexpr int BM = 128, BN = 64, BK = 32;   // real rows, real columns, real K per stage
constexpr int A_T = BM * BK * 2;      // 8 KB per slice
constexpr int B_T = BN * BK * 2;      // 4 KB per slice
constexpr int HG = S / 2;             // groups emptied together (a half of them)
constexpr int ZB_T = (HG - 1) * B_T;  // zero slices in front of B's
constexpr int OFF_Z = S * A_T, OFF_B = OFF_Z + ZB_T;
constexpr int STAGE = OFF_B + S * B_T;   // 108 KB
constexpr int STAGE_LOAD = S * (A_T + B_T);   // of which TMA writes 96 KB
constexpr int NSTAGE = 2;
constexpr int NG = S;                 // accumulator groups g = 2..S+1
// K blocks per exact accumulation chunk: 96 real K, or in a fixed order of
// operations (pw_oz_ws::fixed) 64, after which every group is rounded to the
// sum's binary point
constexpr int CHUNK_KB = 3, CHUNK_KB_FIXED = 2;
constexpr int PERSIST_KB = 16;        // K blocks up to which a CTA takes several tiles
constexpr int STEPS_KB = BK / 16;     // MMA steps (16 real K) per K block
constexpr int NH = 2;
constexpr int SMEM_BYTES = NSTAGE * STAGE + 1024 + 512;
static_assert(SMEM_BYTES <= 232448, "shared memory per CTA");
constexpr int TMEM_COLS = 512;
constexpr int EPI_WARPS = 8;
constexpr int NTHREADS = 64 + 32 * EPI_WARPS;

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
// shared-memory matrix descriptor: K-major, 64-byte swizzle (rows of 32
// FP16), 8-row groups 512 B apart
__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t addr) { return smem_desc(addr, 16, 512, 4); }

// whether half h (0: groups 2..5, 1: groups 6..9) is emptied after MMA step t
// of nsteps: every chunk (CKB blocks), the halves half a chunk apart, and at the
// end
template <int CKB>
__device__ __forceinline__ bool oz_flush(int h, int t, int nsteps) {
  constexpr int CHUNK = CKB * STEPS_KB;
  return (t + 1 + (h == 0 ? CHUNK / 2 : 0)) % CHUNK == 0 || t == nsteps - 1;
}

// The slice products of half H for one step: slice p of A times the slices
// q0..q0 + 3 of B, q0 = 4 H + 2 - p, onto the groups p + q = 4 H + 2.. (q < 1:
// zeros).  Every MMA has the same shape and accumulators, which is what
// orders them.  `first`: the step opens the half's chunk, and its first MMA
// overwrites the accumulators.  db: the stage's first zero slice.
template <int H>
__device__ __forceinline__ void oz_mmas(uint32_t tmem, uint64_t da, uint64_t db, bool first) {
#pragma unroll
  for (int p = 1; p <= (H + 1) * HG; ++p) {
    const int q0 = H * HG + 2 - p;
    mma_f16(tmem + (uint32_t)(H * HG * BN), da + (uint64_t)((p - 1) * (A_T >> 4)),
            db + (uint64_t)((q0 + HG - 2) * (B_T >> 4)), idesc_f16(BM, HG * BN, false), !(first && p == 1));
  }
}

// bits of the FP32 accumulator value v + 1.5 2^23 (an integer |v| < 2^22): kBias + v
constexpr uint32_t kBias = 0x4B400000u;
__device__ __forceinline__ uint32_t biased(uint32_t v) {
  return __float_as_uint(__uint_as_float(v) + 12582912.0f);
}

// The tiles of a product in the order of their rows, each row's range of column
// tiles [lo, hi) without those that hold nothing wanted of a Hermitian output
// (herm 1: strictly below the diagonal, mirrored later; herm 2: no element with
// j/64 <= i/64; ioff, joff: the block's place in the whole product).
struct OzTiles {
  int mtiles, ntiles, bj, herm, ioff, joff;
  __host__ __device__ void range(int mt, int &lo, int &hi) const {
    lo = 0;
    hi = ntiles;
    const int gm0 = ioff + mt * BM;
    if (herm == 1) {
      const int d = gm0 - joff - (BN / 2 - 1);   // wanted: (BN / 2) nt >= d
      lo = d <= 0 ? 0 : (d + BN / 2 - 1) / (BN / 2);
      if (lo > ntiles) lo = ntiles;
    }
    if (herm == 2) {
      const int e = (((gm0 + BM - 1) >> 6) + 1) * 64 - joff;   // wanted: (BN / 2) nt < e
      hi = e <= 0 ? 0 : (e + BN / 2 - 1) / (BN / 2);
      if (hi > ntiles) hi = ntiles;
    }
  }
};
// item's tile, or false past the last one
__device__ __forceinline__ bool oz_tile(const OzTiles &g, int item, int &m0, int &j0) {
  if (g.herm != 1 && g.herm != 2) {
    const int mt = item / g.ntiles;
    m0 = mt * BM;
    j0 = (item - mt * g.ntiles) * g.bj;
    return mt < g.mtiles;
  }
  for (int mt = 0; mt < g.mtiles; ++mt) {
    int lo, hi;
    g.range(mt, lo, hi);
    if (item < hi - lo) {
      m0 = mt * BM;
      j0 = (lo + item) * g.bj;
      return true;
    }
    item -= max(0, hi - lo);
  }
  return false;
}
// the K range of a tile (real K blocks; triangular operands are zero outside),
// of its part z: an equal share, in whole chunks
template <int CKB>
__device__ __forceinline__ void oz_krange(const OzTiles &g, int m0, int j0, int kblocks, int &kb_beg, int &nkb) {
  const int gm0 = g.ioff + m0, gj0 = g.joff + j0;
  int kb_lo = 0, kb_hi = kblocks;
  if (g.herm == 3) kb_lo = min(kblocks, (2 * gm0) / BK);
  if (g.herm == 4) kb_lo = min(kblocks, (2 * gj0) / BK);
  if (g.herm == 5) kb_hi = min(kblocks, (2 * (gm0 + BM) + BK - 1) / BK);
  const int ntot = max(0, kb_hi - kb_lo);
  const int nch = (ntot + CKB - 1) / CKB;
  const int per = (nch + (int)gridDim.y - 1) / (int)gridDim.y;
  const int c0 = min(nch, (int)blockIdx.y * per), c1 = min(nch, c0 + per);
  kb_beg = kb_lo + c0 * CKB;
  nkb = max(0, min(kb_hi, kb_lo + c1 * CKB) - kb_beg);
}

// PERSIST: a CTA takes every gridDim.x-th tile, so that the copies and MMAs
// of its next tile run while the sums of this one are converted and written.  A
// K of one chunk is mostly that: the rank-64 update of order 3,400 takes 218 us
// so and 236 us with one CTA per tile (84 us of it MMAs).
template <int CKB, bool PERSIST>
__global__ void __launch_bounds__(NTHREADS, 1)
    k_oz_gemm(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
              int a_slice_rows, int b_slice_rows, int m, int n, int kblocks, int mtiles, int ntiles,
              const int *__restrict__ ea, const int *__restrict__ eb, double2 alpha, double2 beta,
              double2 *__restrict__ C, int ldc, int herm, int ioff, int joff, double2 *__restrict__ part,
              int *__restrict__ err, int real_out) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t *full = (uint64_t *)(smem + NSTAGE * STAGE);
  uint64_t *empty = full + NSTAGE;
  uint64_t *accf = empty + NSTAGE;     // [NH] a half's accumulators ready
  uint64_t *acce = accf + NH;          // [NH] a half's accumulators drained
  uint32_t *tmem_slot = (uint32_t *)(acce + NH);

  // a tile is 128 complex rows and 32 complex columns, or with real_out (real
  // operands: one slice row per real column of B, output real, ld ldc in
  // doubles) 64 real columns
  const OzTiles g{mtiles, ntiles, real_out ? BN : BN / 2, herm, ioff, joff};
  int m0, j0;
  if (!oz_tile(g, blockIdx.x, m0, j0)) return;
  // every tile of the CTA has the K range of the first (one with its own, of a
  // triangular operand, is alone)
  int kb_beg, nkb;
  oz_krange<CKB>(g, m0, j0, kblocks, kb_beg, nkb);
  const int nsteps = nkb * STEPS_KB;
  // binary point of the fixed-point sum: |sum| <= K' (scaled entries < 1)
  int lg = 0;
  while ((1 << lg) < max(1, nkb * BK)) ++lg;
  const int Lfix = min(56, 62 - lg);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < NSTAGE; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int h = 0; h < NH; ++h) { mbar_init(&accf[h], 1); mbar_init(&acce[h], EPI_WARPS); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the zero slices, for the tensor core's reads (the async proxy)
  for (int s = 0; s < NSTAGE; ++s)
    for (int w = threadIdx.x; w < ZB_T / 16; w += NTHREADS)
      *(uint4 *)(smem + s * STAGE + OFF_Z + w * 16) = make_uint4(0u, 0u, 0u, 0u);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer: all S slices of the A and B tiles per stage
      int kc = 0;
      bool ok = true;
      for (int item = blockIdx.x;;) {
        for (int i = 0; i < nkb; ++i, ++kc) {
          const int s = kc % NSTAGE;
          const uint32_t u = kc / NSTAGE;
          if (!mbar_wait(&empty[s], (u & 1) ^ 1)) { atomicOr(err, 1); ok = false; break; }
          unsigned char *st = smem + s * STAGE;
          mbar_expect_tx(&full[s], STAGE_LOAD);
          const int x = (kb_beg + i) * BK;
#pragma unroll
          for (int p = 0; p < S; ++p) {
            tma_load_2d(st + p * A_T, &mapA, &full[s], x, p * a_slice_rows + m0);
            tma_load_2d(st + OFF_B + p * B_T, &mapB, &full[s], x, p * b_slice_rows + (real_out ? j0 : 2 * j0));
          }
        }
        if (!PERSIST || !ok || !oz_tile(g, item += gridDim.x, m0, j0)) break;
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------- MMA issuer.  The descriptors are formed once; slices,
      // K steps and stages only move their start address (16-byte units in the
      // low 14 bits, which cover all of shared memory, so nothing carries out)
      const uint64_t da0 = smem_desc_sw64(smem_u32(smem)), db0 = smem_desc_sw64(smem_u32(smem + OFF_Z));
      uint32_t nfl0 = 0, nfl1 = 0;          // times each half was handed to the epilogue
      int kc = 0;
      bool ok = true;
      for (int item = blockIdx.x;;) {
        bool first0 = true, first1 = true;  // the next step opens the half's chunk
        for (int i = 0; i < nkb; ++i, ++kc) {
          const int s = kc % NSTAGE;
          const uint32_t u = kc / NSTAGE;
          if (!mbar_wait(&full[s], u & 1)) { atomicOr(err, 2); ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
          for (int kk = 0; kk < STEPS_KB; ++kk) {
            const int t = i * STEPS_KB + kk;
            const uint64_t off = (uint64_t)(s * (STAGE >> 4) + 2 * kk);
            if (first1) {
              // the epilogue has read the half's previous chunk
              if (!mbar_wait(&acce[1], (nfl1 & 1) ^ 1)) { atomicOr(err, 8); ok = false; break; }
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            }
            oz_mmas<1>(tmem, da0 + off, db0 + off, first1);
            first1 = oz_flush<CKB>(1, t, nsteps);
            if (first1) { mma_commit(&accf[1]); ++nfl1; }
            if (first0) {
              if (!mbar_wait(&acce[0], (nfl0 & 1) ^ 1)) { atomicOr(err, 8); ok = false; break; }
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            }
            oz_mmas<0>(tmem, da0 + off, db0 + off, first0);
            first0 = oz_flush<CKB>(0, t, nsteps);
            if (first0) { mma_commit(&accf[0]); ++nfl0; }
          }
          if (!ok) break;
          mma_commit(&empty[s]);
        }
        if (!PERSIST || !ok || !oz_tile(g, item += gridDim.x, m0, j0)) break;
      }
    }
  } else {
    // ---------------- epilogue: warps 2..9; lane quarter q, column half h
    const int q = warp & 3, h = (warp - 2) >> 2;
    const uint32_t lanes = (uint32_t)(q * 32) << 16;
    bool ok = true;
    uint32_t nfl[NH] = {0, 0};
    for (int item = blockIdx.x;;) {
    // 64-bit fixed-point sums modulo 2^64; groups with a left shift add
    // kBias + v, and the biases are taken off at the end
    unsigned long long acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0;
    // CARRY: the two lowest groups, weights 2^-56 and 2^-63, are added in units of
    // 2^-63, and what lies below the sum's binary point stays in rem until the
    // end: one rounding instead of two per chunk
    constexpr bool CARRY = CKB == CHUNK_KB;
    uint32_t rem[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) rem[i] = 0;
    const int slow = BETA * (S + 1) - Lfix;      // 7..
    const uint32_t mlow = (1u << slow) - 1u;
    unsigned long long bias = 0;
    for (int t = 0; t < nsteps && ok; ++t) {
#pragma unroll
      for (int hh = NH - 1; hh >= 0; --hh) {
        if (!ok || !oz_flush<CKB>(hh, t, nsteps)) continue;
        if (!mbar_wait(&accf[hh], nfl[hh] & 1)) { atomicOr(err, 4); ok = false; continue; }
        ++nfl[hh];
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int gend = CARRY && hh == NH - 1 ? NG - 2 : (hh + 1) * HG;
#pragma unroll 1
        for (int gr = hh * HG; gr < gend; ++gr) {
          uint32_t v[32];
          tmem_ld32(tmem + lanes + (uint32_t)(gr * BN + h * 32), v);
          if (gr == HG - 1 || (!CARRY && gr == NG - 1)) {
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&acce[hh]);
          }
          const int sh = Lfix - BETA * (gr + 2);
          if (sh >= 32) {
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] += (unsigned long long)(biased(v[i]) << (sh - 32)) << 32;
          } else if (sh >= 0) {
            const uint32_t f = 1u << sh;
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] += (unsigned long long)biased(v[i]) * f;
          } else {
            // rounded to nearest (with CARRY the third lowest group of very long sums)
            const int half = 1 << (-sh - 1);
#pragma unroll
            for (int i = 0; i < 32; ++i)
              acc[i] += (unsigned long long)(long long)(((int)(biased(v[i]) - kBias) + half) >> -sh);
          }
          if (sh >= 0) bias += (unsigned long long)kBias << sh;
        }
        if (CARRY && hh == NH - 1) {
          const uint32_t tv = tmem + lanes + (uint32_t)((NG - 2) * BN + h * 32), tu = tv + BN;
#pragma unroll
          for (int c = 0; c < 32; c += 16) {
            uint32_t v[16], u[16];
            tmem_ld16x2(tv + c, tu + c, v, u);
            if (c == 16) {
              asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
              __syncwarp();
              if (lane == 0) mbar_arrive(&acce[NH - 1]);
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              // |v| 2^7 + |u| + rem < 2^29 + 2^22 + 2^30: a signed 32-bit sum
              const uint32_t w = (biased(v[i]) << BETA) + biased(u[i]) + (rem[c + i] - ((kBias << BETA) + kBias));
              acc[c + i] += (unsigned long long)(long long)((int)w >> slow);
              rem[c + i] = w & mlow;
            }
          }
        }
      }
    }
    if (CARRY) {
#pragma unroll
      for (int i = 0; i < 32; ++i) acc[i] += (rem[i] + (1u << (slow - 1))) >> slow;
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] -= bias;
    if (PERSIST) {
      // the tile's place again rather than in registers over its sums, which fill them
      asm volatile("" : "+r"(item));
      oz_tile(g, item, m0, j0);
    }
    // alpha = +-1, beta = 0 or 1 (all products of the eigensolver): no products,
    // which would take the FP64 pipe eight instructions per element besides the
    // two conversions and two additions, and the old values all requested first.
    // The same results: the general form multiplies by 1 and adds zeros.
    const bool unit = alpha.y == 0.0 && fabs(alpha.x) == 1.0 && beta.y == 0.0 && (beta.x == 0.0 || beta.x == 1.0);
    const int i = m0 + q * 32 + lane;              // complex output row
    if (ok && i < m && real_out) {
      double *Cr = (double *)C;
      const int ka = -Lfix - ea[i];
#pragma unroll
      for (int t = 0; t < 32; ++t) {
        const int j = j0 + h * 32 + t;
        if (j >= n) continue;
        double r = alpha.x * scale_pow2((double)(long long)acc[t], ka - eb[j]);
        if (beta.x != 0.0) r += beta.x * Cr[i + (long)j * ldc];
        Cr[i + (long)j * ldc] = r;
      }
    } else if (ok && i < m) {
      const int jb = j0 + h * 16;                  // first complex column of this thread
      const int ka = -Lfix - ea[i];
      if (unit && !part) {
#pragma unroll
        for (int t0 = 0; t0 < 16; t0 += 4) {
          double2 c[4];
          bool on[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const int j = jb + t0 + t;
            on[t] = j < n && !(herm == 2 && ((joff + j) >> 6) > ((ioff + i) >> 6));
            if (on[t] && beta.x != 0.0) c[t] = C[i + (long)j * ldc];
          }
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            if (!on[t]) continue;
            const int j = jb + t0 + t, k = ka - eb[j];
            long long ar = (long long)acc[2 * (t0 + t)], ai = (long long)acc[2 * (t0 + t) + 1];
            if (alpha.x < 0.0) {
              ar = -ar;
              ai = -ai;
            }
            double2 r = make_double2(scale_pow2((double)ar, k), scale_pow2((double)ai, k));
            if (beta.x != 0.0) {
              r.x += c[t].x;
              r.y += c[t].y;
            }
            C[i + (long)j * ldc] = r;
          }
        }
      } else
#pragma unroll
      for (int t = 0; t < 16; ++t) {
        const int j = jb + t;
        if (j >= n) continue;
        if (herm == 2 && ((joff + j) >> 6) > ((ioff + i) >> 6)) continue;
        const int k = ka - eb[j];
        const double re = scale_pow2((double)(long long)acc[2 * t], k);
        const double im = scale_pow2((double)(long long)acc[2 * t + 1], k);
        if (part) {
          part[(long)blockIdx.y * m * n + i + (long)j * m] = make_double2(re, im);
        } else {
          double2 r = make_double2(alpha.x * re - alpha.y * im, alpha.x * im + alpha.y * re);
          if (beta.x != 0.0 || beta.y != 0.0) {
            const double2 c = C[i + (long)j * ldc];
            r.x += beta.x * c.x - beta.y * c.y;
            r.y += beta.x * c.y + beta.y * c.x;
          }
          C[i + (long)j * ldc] = r;
        }
      }
    }
    if (!PERSIST || !ok || !oz_tile(g, item += gridDim.x, m0, j0)) break;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
  }
}

// sum of the K-split parts (in part order), then alpha, beta; same element
// selection as the single-part epilogue
__global__ void k_oz_reduce(const double2 *__restrict__ part, int splits, int m, int n, double2 alpha,
                            double2 beta, double2 *__restrict__ C, int ldc, int herm, int ioff, int joff) {
  const long idx = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (idx >= (long)m * n) return;
  const int i = (int)(idx % m), j = (int)(idx / m);
  if (herm == 1 && ioff + i > joff + j) return;     // mirrored later; tiles below the diagonal have no parts
  double2 s = make_double2(0.0, 0.0);
  for (int z = 0; z < splits; ++z) {
    const double2 v = part[(long)z * m * n + idx];
    s.x += v.x;
    s.y += v.y;
  }
  double2 r = make_double2(alpha.x * s.x - alpha.y * s.y, alpha.x * s.y + alpha.y * s.x);
  if (beta.x != 0.0 || beta.y != 0.0) {
    const double2 c = C[i + (long)j * ldc];
    r.x += beta.x * c.x - beta.y * c.y;
    r.y += beta.x * c.y + beta.y * c.x;
  }
  C[i + (long)j * ldc] = r;
}

// lower triangle <- conj(upper) (n x n, ld)
__global__ void k_oz_mirror(double2 *C, int ldc, int n) {
  const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 32 + threadIdx.y;
  if (i >= n || j >= n || i <= j) return;
  const double2 u = C[j + (long)i * ldc];
  C[i + (long)j * ldc] = make_double2(u.x, -u.y);
}

// ------------------------------------------------------------- slicing ----
// Slices of the real rows of an operand.  The complex "row" r over k is
//   contiguous:  v_kappa = X[kappa + r ld]      (a column of X)
//   strided:     v_kappa = X[r + kappa ld]      (a row of X)
// conjugated if conj.  bside = 0: one real row r = (re, im) over K' = 2k;
// bside = 1: two real rows 2r = (re, -im), 2r + 1 = (im, re).
// out: [S][rows_total][kpad] FP16, e: row exponents (one per complex row).
// Bound: memory (48 or 80 bytes per element); S^H S and S^H (H S) of the
// 216-atom cell's FP64 step were at a fifth of it while each digit was peeled
// and converted on its own.
__device__ __forceinline__ void store_slices(double re, double im, int ex, int bside, int r, int t, int kpad,
                                             long slice, __half *__restrict__ out) {
  uint32_t d[S];
  digit_pairs(re, im, ex, d);
  if (!bside) {
    __half *o = out + (long)r * kpad + 2 * t;
#pragma unroll
    for (int p = 0; p < S; ++p) *(uint32_t *)(o + p * slice) = d[p];
  } else {
    __half *o0 = out + (long)(2 * r) * kpad + 2 * t, *o1 = o0 + kpad;
#pragma unroll
    for (int p = 0; p < S; ++p) {
      *(uint32_t *)(o0 + p * slice) = d[p] ^ 0x80000000u;            // (re, -im)
      *(uint32_t *)(o1 + p * slice) = __byte_perm(d[p], 0, 0x1032);  // (im, re)
    }
  }
}
__global__ void __launch_bounds__(256) k_oz_slice_contig(const double2 *__restrict__ X, int ld, int k, int conj,
                                                         int bside, int kpad, int rows_total,
                                                         __half *__restrict__ out, int *__restrict__ e) {
  __shared__ unsigned long long shm[8];
  const int r = blockIdx.x;
  const double2 *x = X + (long)r * ld;
  unsigned long long mb = 0;
  for (int t = threadIdx.x; t < k; t += blockDim.x) {
    const double2 v = x[t];
    const unsigned long long a = abs_bits(v.x), c = abs_bits(v.y);
    mb = max(mb, max(a, c));
  }
  for (int o = 16; o > 0; o >>= 1) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
  if ((threadIdx.x & 31) == 0) shm[threadIdx.x >> 5] = mb;
  __syncthreads();
  mb = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mb = max(mb, shm[w]);
  const int ex = row_exp(mb);
  if (threadIdx.x == 0) e[r] = ex;
  const long slice = (long)rows_total * kpad;
  for (int t = threadIdx.x; t < kpad / 2; t += blockDim.x) {
    double re = 0.0, im = 0.0;
    if (t < k) {
      const double2 v = x[t];
      re = v.x;
      im = conj ? -v.y : v.y;
    }
    store_slices(re, im, ex, bside, r, t, kpad, slice, out);
  }
}

// row maxima of the strided rows as ordered bits: block (32 rows, 8 warps)
// over a 256-long K range, lane = row (reads coalesced across rows), the
// warps' maxima combined in shared memory, then one atomicMax per row into mx
// (cleared before)
constexpr int RX_K = 256;
__global__ void __launch_bounds__(256) k_oz_rowmax(const double2 *__restrict__ X, int ld, int nrows, int k,
                                                   unsigned long long *__restrict__ mx) {
  __shared__ unsigned long long sh[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int r = blockIdx.x * 32 + lane;
  const int t0 = blockIdx.y * RX_K, t1 = min(k, t0 + RX_K);
  unsigned long long m = 0;
  if (r < nrows)
    for (int t = t0 + w; t < t1; t += 8) {
      const double2 v = X[r + (long)t * ld];
      m = max(m, max(abs_bits(v.x), abs_bits(v.y)));
    }
  sh[w][lane] = m;
  __syncthreads();
  if (w == 0 && r < nrows) {
#pragma unroll
    for (int q = 1; q < 8; ++q) m = max(m, sh[q][lane]);
    atomicMax(&mx[r], m);
  }
}

// strided rows: 32 rows x 64 K tile through shared memory (reads along r,
// writes along K)
__global__ void __launch_bounds__(256) k_oz_slice_strided(const double2 *__restrict__ X, int ld, int nrows, int k,
                                                          int conj, int bside, int kpad, int rows_total,
                                                          const unsigned long long *__restrict__ mx,
                                                          int *__restrict__ e, __half *__restrict__ out) {
  __shared__ double2 tileS[64][33];
  const int r0 = blockIdx.x * 32, t0 = blockIdx.y * 64;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 32 x 8
  for (int tt = ty; tt < 64; tt += 8) {
    const int r = r0 + tx, t = t0 + tt;
    double2 v = make_double2(0.0, 0.0);
    if (r < nrows && t < k) v = X[r + (long)t * ld];
    if (conj) v.y = -v.y;
    tileS[tt][tx] = v;
  }
  __syncthreads();
  const long slice = (long)rows_total * kpad;
  for (int rr = ty; rr < 32; rr += 8) {
    const int r = r0 + rr;
    if (r >= nrows) continue;
    const int ex = row_exp(mx[r]);
    if (blockIdx.y == 0 && tx == 0) e[r] = ex;
    for (int tt = tx; tt < 64; tt += 32) {
      const int t = t0 + tt;
      if (2 * t >= kpad) continue;
      const double2 v = tileS[tt][rr];
      store_slices(v.x, v.y, ex, bside, r, t, kpad, slice, out);
    }
  }
}

// Slices of real rows (the real mode, C = A B with real A, B): row r of A
// is strided (A[r + t lda]), row j of the B side is column j of B,
// contiguous (B[t + j ldb]); out: [S][rows_total][kpad] FP16, e: row
// exponents.  Row maxima of the strided rows come from k_ozr_rowmax (mx,
// cleared before).
__global__ void __launch_bounds__(256) k_ozr_slice_contig(const double *__restrict__ X, int ld, int k, int kpad,
                                                          int rows_total, __half *__restrict__ out,
                                                          int *__restrict__ e) {
  __shared__ unsigned long long shm[8];
  const int r = blockIdx.x;
  const double *x = X + (long)r * ld;
  unsigned long long mb = 0;
  for (int t = threadIdx.x; t < k; t += blockDim.x) mb = max(mb, abs_bits(x[t]));
  for (int o = 16; o > 0; o >>= 1) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
  if ((threadIdx.x & 31) == 0) shm[threadIdx.x >> 5] = mb;
  __syncthreads();
  mb = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mb = max(mb, shm[w]);
  const int ex = row_exp(mb);
  if (threadIdx.x == 0) e[r] = ex;
  const long slice = (long)rows_total * kpad;
  for (int t2 = threadIdx.x; t2 < kpad / 2; t2 += blockDim.x) {
    const int t = 2 * t2;
    uint32_t d[S];
    digit_pairs(t < k ? x[t] : 0.0, t + 1 < k ? x[t + 1] : 0.0, ex, d);
    __half *o = out + (long)r * kpad + t;
#pragma unroll
    for (int p = 0; p < S; ++p) *(uint32_t *)(o + p * slice) = d[p];
  }
}
__global__ void __launch_bounds__(256) k_ozr_rowmax(const double *__restrict__ X, int ld, int nrows, int k,
                                                    unsigned long long *__restrict__ mx) {
  __shared__ unsigned long long sh[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int r = blockIdx.x * 32 + lane;
  const int t0 = blockIdx.y * RX_K, t1 = min(k, t0 + RX_K);
  unsigned long long m = 0;
  if (r < nrows)
    for (int t = t0 + w; t < t1; t += 8) m = max(m, abs_bits(X[r + (long)t * ld]));
  sh[w][lane] = m;
  __syncthreads();
  if (w == 0 && r < nrows) {
#pragma unroll
    for (int q = 1; q < 8; ++q) m = max(m, sh[q][lane]);
    atomicMax(&mx[r], m);
  }
}
__global__ void __launch_bounds__(256) k_ozr_slice_strided(const double *__restrict__ X, int ld, int nrows, int k,
                                                           int kpad, int rows_total,
                                                           const unsigned long long *__restrict__ mx,
                                                           int *__restrict__ e, __half *__restrict__ out) {
  __shared__ double tileS[64][33];
  const int r0 = blockIdx.x * 32, t0 = blockIdx.y * 64;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 32 x 8
  for (int tt = ty; tt < 64; tt += 8) {
    const int r = r0 + tx, t = t0 + tt;
    tileS[tt][tx] = (r < nrows && t < k) ? X[r + (long)t * ld] : 0.0;
  }
  __syncthreads();
  const long slice = (long)rows_total * kpad;
  for (int rr = ty; rr < 32; rr += 8) {
    const int r = r0 + rr;
    if (r >= nrows) continue;
    const int ex = row_exp(mx[r]);
    if (blockIdx.y == 0 && tx == 0) e[r] = ex;
    const int t = t0 + 2 * tx;
    if (t >= kpad) continue;
    uint32_t d[S];
    digit_pairs(tileS[2 * tx][rr], tileS[2 * tx + 1][rr], ex, d);
    __half *o = out + (long)r * kpad + t;
#pragma unroll
    for (int p = 0; p < S; ++p) *(uint32_t *)(o + p * slice) = d[p];
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  });
  return fn;
}

bool make_map(CUtensorMap *map, const void *base, int kpad, long rows, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)kpad, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)kpad * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void *>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// slices of op(X)'s rows (bside 0) or of op(X)'s columns (bside 1):
//   A side: op = 'N': rows of X (m x k) -> strided; op = 'C': columns of X (k x m) -> contiguous, conj
//   B side: op = 'N': columns of X (k x n) -> contiguous; op = 'C': rows of X (n x k) -> strided, conj
pw_status slice_operand(char op, int bside, const double2 *X, int ld, int nrows, int k, int kpad,
                        int rows_total, __half *out, int *e, unsigned long long *mx, cudaStream_t st) {
  const bool contig = bside ? op == 'N' : op == 'C';
  const int conj = op == 'C';
  if (contig) {
    pw_count_launch();
    k_oz_slice_contig<<<nrows, 256, 0, st>>>(X, ld, k, conj, bside, kpad, rows_total, out, e);
  } else {
    PW_CUDA(cudaMemsetAsync(mx, 0, (size_t)nrows * sizeof(unsigned long long), st));
    pw_count_launch();
    k_oz_rowmax<<<dim3((nrows + 31) / 32, (k + RX_K - 1) / RX_K), 256, 0, st>>>(X, ld, nrows, k, mx);
    pw_count_launch();
    k_oz_slice_strided<<<dim3((nrows + 31) / 32, (kpad / 2 + 63) / 64), 256, 0, st>>>(
        X, ld, nrows, k, conj, bside, kpad, rows_total, mx, e, out);
  }
  return pw_check_launch("oz slice");
}

using OzKernel = decltype(&k_oz_gemm<CHUNK_KB, false>);
OzKernel oz_kernel(bool fixed, bool persist) {
  if (fixed) return persist ? k_oz_gemm<CHUNK_KB_FIXED, true> : k_oz_gemm<CHUNK_KB_FIXED, false>;
  return persist ? k_oz_gemm<CHUNK_KB, true> : k_oz_gemm<CHUNK_KB, false>;
}
// One CTA per SM over its share of the tiles for a short K, where the next tile's
// start hides the sums' conversion (order-1,458 eigensolve 35.2 -> 34.7 ms, 3,456
// 125.9 -> 124.9 ms); else one per tile: the loop over tiles takes registers that
// the sums need (K = 3,456: 3.72 ms with it, 3.49 without), except in the fixed
// order, which carries no remainders (Si-512 mixed step 379 -> 374-378 ms).  One
// per tile also for triangular operands, whose tiles differ in K.
bool oz_persist(bool fixed, int kblocks, int herm) { return herm < 3 && (fixed || kblocks <= PERSIST_KB); }

int g_max_parts = 16;

// the kernel's shared-memory opt-in, once per device (outside any later
// stream capture: the first product on a device runs uncaptured)
pw_status allow_smem() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  PW_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return PW_ERR_ARG;
  std::lock_guard<std::mutex> g(mu);
  if (!done[dev]) {
    for (auto kern : {oz_kernel(false, false), oz_kernel(false, true), oz_kernel(true, false), oz_kernel(true, true)})
      PW_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
    done[dev] = true;
  }
  return PW_OK;
}

}  // namespace

size_t pw_oz_ws_bytes(int m, int n, int k) {
  const size_t kpad = ((size_t)2 * k + BK - 1) / BK * BK;
  const size_t arows = ((size_t)m + BM - 1) / BM * BM, brows = (2 * (size_t)n + BN - 1) / BN * BN;
  return (size_t)S * (arows + brows) * kpad * 2 + (arows + brows) * 4 + std::max(arows, brows) * 8 + 4096;
}

void pw_oz_free(pw_oz_ws *w) {
  const pw_mem m = w->mem;
  pw_mem_free(m, w->buf);
  pw_mem_free(m, w->part);
  pw_mem_free(m, w->err);
  *w = pw_oz_ws();
  w->mem = m;
}

pw_status pw_oz_check(pw_oz_ws *w, cudaStream_t st) {
  if (!w->err) return PW_OK;
  int e = 0;
  PW_CUDA(cudaMemcpyAsync(&e, w->err, 4, cudaMemcpyDeviceToHost, st));
  PW_CUDA(cudaStreamSynchronize(st));
  return e ? PW_ERR_TIMEOUT : PW_OK;
}

namespace {
// One block of the product: rows [i0, i0 + mb) of op(A), columns [j0, j0 + nb)
// of op(B), the whole K (given operand pointers already offset); herm
// predicates use the global offsets.
pw_status oz_block(pw_oz_ws *w, char opA, char opB, int mb, int nb, int k, double2 alpha, const double2 *A,
                   int lda, const double2 *B, int ldb, double2 beta, double2 *C, int ldc, cudaStream_t st,
                   int herm, int ioff, int joff) {
  const int kpad = (2 * k + BK - 1) / BK * BK;
  const int kblocks = kpad / BK;
  // slice storage: rows padded to the tile (the tensor map of the last slice
  // then never reads another slice's rows)
  const int arows = (mb + BM - 1) / BM * BM, brows = (2 * nb + BN - 1) / BN * BN;
  const size_t abytes = (size_t)S * arows * kpad * 2, bbytes = (size_t)S * brows * kpad * 2;
  const size_t mxrows = (size_t)std::max(arows, brows);
  const size_t need = abytes + bbytes + ((size_t)arows + brows) * 4 + 256 + mxrows * 8 + 1024;
  if (need > w->bytes) {
    pw_mem_free(w->mem, w->buf);
    w->buf = nullptr;
    w->bytes = 0;
    ++w->gen;
    if (pw_mem_alloc(w->mem, &w->buf, need) != cudaSuccess) return PW_ERR_OOM;
    w->bytes = need;
  }
  if (!w->err) {
    if (pw_mem_alloc(w->mem, (void **)&w->err, 16) != cudaSuccess) return PW_ERR_OOM;
    PW_CUDA(cudaMemsetAsync(w->err, 0, 16, st));
    ++w->gen;
  }
  unsigned char *p = (unsigned char *)w->buf;
  __half *sa = (__half *)p, *sb = (__half *)(p + abytes);
  int *ea = (int *)(p + abytes + bbytes), *eb = ea + arows;
  unsigned long long *mx =
      (unsigned long long *)(((uintptr_t)(eb + brows) + 255) & ~(uintptr_t)255);   // strided row maxima
  PW_TRY(slice_operand(opA, 0, A, lda, mb, k, kpad, arows, sa, ea, mx, st));
  PW_TRY(slice_operand(opB, 1, B, ldb, nb, k, kpad, brows, sb, eb, mx, st));
  CUtensorMap ma, mbm;
  if (!make_map(&ma, sa, kpad, (long)S * arows, BM) || !make_map(&mbm, sb, kpad, (long)S * brows, BN))
    return PW_ERR_CUDA;
  PW_TRY(allow_smem());
  const int mtiles = arows / BM, ntiles = brows / BN, tiles = mtiles * ntiles;
  // K split when the tiles alone leave SMs idle (herm 1: about half of them
  // are skipped).  A part is at least two chunks, 12 steps of ~0.8 us, which is
  // what its start and its share of the reduction cost; a tile alone on its SM
  // takes ~1.1 us a step (S^H S of the 8-atom cell, 72 x 72 x 1,647: 227 us in
  // one part, 28 us split).
  const int ckb = w->fixed ? CHUNK_KB_FIXED : CHUNK_KB;
  const int nch = (kblocks + ckb - 1) / ckb;
  const int act = herm == 1 && !w->fixed ? (tiles + 1) / 2 : tiles;
  int parts = 1;
  if (herm <= (w->fixed ? 0 : 1) && act < 152) {
    // (a fixed order of operations keeps parts of eight chunks)
    parts = std::min({(2 * 152 + act - 1) / act, std::max(1, nch / (w->fixed ? 8 : 2)), g_max_parts});
    const size_t pbytes = (size_t)parts * mb * nb * 16;
    if (parts > 1 && pbytes > w->part_bytes) {
      pw_mem_free(w->mem, w->part);
      w->part = nullptr;
      w->part_bytes = 0;
      ++w->gen;
      if (pw_mem_alloc(w->mem, (void **)&w->part, pbytes) != cudaSuccess) parts = 1;
      else w->part_bytes = pbytes;
    }
  }
  pw_count_launch();
  const bool persist = parts == 1 && oz_persist(w->fixed, kblocks, herm);
  oz_kernel(w->fixed, persist)<<<dim3(persist ? std::min(tiles, 152) : tiles, parts), NTHREADS, SMEM_BYTES, st>>>(ma, mbm, arows, brows, mb, nb, kblocks, mtiles,
                                                               ntiles, ea, eb, alpha, beta, C, ldc, herm, ioff,
                                                               joff, parts > 1 ? w->part : nullptr, w->err, 0);
  PW_TRY(pw_check_launch("oz gemm"));
  if (parts > 1) {
    pw_count_launch();
    k_oz_reduce<<<(unsigned)(((long)mb * nb + 255) / 256), 256, 0, st>>>(w->part, parts, mb, nb, alpha, beta, C,
                                                                          ldc, herm, ioff, joff);
    PW_TRY(pw_check_launch("oz reduce"));
  }
  return PW_OK;
}

// operand pointer of op(X) at (row r, K index t): op 'N' -> X[r + t ld],
// op 'C' -> X[t + r ld]
const double2 *at(const double2 *X, char op, int ld, long r, long t) {
  return op == 'N' ? X + r + t * (long)ld : X + t + r * (long)ld;
}
}  // namespace

pw_status pw_dgemm_oz(pw_oz_ws *w, int m, int n, int k, const double *A, int lda, const double *B, int ldb,
                      double *C, int ldc, cudaStream_t st) {
  if (m <= 0 || n <= 0 || k <= 0 || lda < m || ldb < k || ldc < m) return PW_ERR_ARG;
  const int kpad = (k + BK - 1) / BK * BK;
  const int kblocks = kpad / BK;
  const int arows = (m + BM - 1) / BM * BM, brows = (n + BN - 1) / BN * BN;
  const size_t abytes = (size_t)S * arows * kpad * 2, bbytes = (size_t)S * brows * kpad * 2;
  const size_t need = abytes + bbytes + ((size_t)arows + brows) * 4 + 256 + (size_t)arows * 8 + 1024;
  if (need > w->bytes) {
    pw_mem_free(w->mem, w->buf);
    w->buf = nullptr;
    w->bytes = 0;
    ++w->gen;
    if (pw_mem_alloc(w->mem, &w->buf, need) != cudaSuccess) return PW_ERR_OOM;
    w->bytes = need;
  }
  if (!w->err) {
    if (pw_mem_alloc(w->mem, (void **)&w->err, 16) != cudaSuccess) return PW_ERR_OOM;
    PW_CUDA(cudaMemsetAsync(w->err, 0, 16, st));
    ++w->gen;
  }
  unsigned char *p = (unsigned char *)w->buf;
  __half *sa = (__half *)p, *sb = (__half *)(p + abytes);
  int *ea = (int *)(p + abytes + bbytes), *eb = ea + arows;
  unsigned long long *mx = (unsigned long long *)(((uintptr_t)(eb + brows) + 255) & ~(uintptr_t)255);
  // A: strided rows (row maxima first); B: its columns, contiguous.  Slice
  // rows past m and n are never written: they only feed output rows and
  // columns that are not stored
  PW_CUDA(cudaMemsetAsync(mx, 0, (size_t)m * 8, st));
  pw_count_launch();
  k_ozr_rowmax<<<dim3((m + 31) / 32, (k + RX_K - 1) / RX_K), 256, 0, st>>>(A, lda, m, k, mx);
  pw_count_launch();
  k_ozr_slice_strided<<<dim3((m + 31) / 32, (kpad + 63) / 64), 256, 0, st>>>(A, lda, m, k, kpad, arows, mx, ea, sa);
  pw_count_launch();
  k_ozr_slice_contig<<<n, 256, 0, st>>>(B, ldb, k, kpad, brows, sb, eb);
  PW_TRY(pw_check_launch("oz real slices"));
  CUtensorMap ma, mbm;
  if (!make_map(&ma, sa, kpad, (long)S * arows, BM) || !make_map(&mbm, sb, kpad, (long)S * brows, BN))
    return PW_ERR_CUDA;
  PW_TRY(allow_smem());
  const int mtiles = arows / BM, ntiles = brows / BN;
  pw_count_launch();
  const bool persist = oz_persist(w->fixed, kblocks, 0);
  oz_kernel(w->fixed, persist)<<<dim3(persist ? std::min(mtiles * ntiles, 152) : mtiles * ntiles, 1), NTHREADS, SMEM_BYTES, st>>>(
      ma, mbm, arows, brows, m, n, kblocks, mtiles, ntiles, ea, eb, make_double2(1.0, 0.0), make_double2(0.0, 0.0),
      (double2 *)C, ldc, 0, 0, 0, nullptr, w->err, 1);
  return pw_check_launch("oz gemm (real)");
}

pw_status pw_zgemm_oz(pw_oz_ws *w, char opA, char opB, int m, int n, int k, double2 alpha, const double2 *A,
                      int lda, const double2 *B, int ldb, double2 beta, double2 *C, int ldc, cudaStream_t st,
                      int herm) {
  if ((opA != 'N' && opA != 'C') || (opB != 'N' && opB != 'C') || herm < 0 || herm > 5) return PW_ERR_ARG;
  if (m <= 0 || n <= 0) return PW_OK;
  if (k <= 0) return PW_ERR_ARG;
  if (herm == 1 && m != n) return PW_ERR_ARG;
  // Blocks of rows, columns and (for the modes whose predicates do not
  // depend on K) K, so that the slices of one block stay under the cap; K
  // blocks after the first accumulate into C (beta = 1).
  const size_t cap = std::max(w->bytes, (size_t)PW_OZ_SLICE_CAP);
  const double per_k = (double)S * 2 * 2;     // slice bytes per real row per complex K index
  int kc = k, mc = m, nc = n;
  auto bytes = [&]() { return per_k * ((double)mc + 2.0 * nc) * kc; };
  auto shrink_k = [&]() {
    if (herm <= 2)
      while (kc > 512 && bytes() > (double)cap) kc = (kc + 1) / 2;
  };
  // K longest (Gram-type products): K blocks first; otherwise rows and
  // columns first (K blocks cost a pass over C each)
  if ((double)k > (double)m + 2.0 * n) shrink_k();
  while (bytes() > (double)cap && (mc > BM || nc > BN / 2)) {
    if ((double)mc >= 2.0 * nc && mc > BM) mc = ((mc + 1) / 2 + BM - 1) / BM * BM;
    else if (nc > BN / 2) nc = ((nc + 1) / 2 + BN / 2 - 1) / (BN / 2) * (BN / 2);
    else mc = ((mc + 1) / 2 + BM - 1) / BM * BM;
  }
  shrink_k();
  const double2 one = make_double2(1.0, 0.0);
  for (int k0 = 0; k0 < k; k0 += kc) {
    const int kb = std::min(kc, k - k0);
    const double2 bt = k0 == 0 ? beta : one;
    for (int i0 = 0; i0 < m; i0 += mc) {
      const int mb = std::min(mc, m - i0);
      for (int j0 = 0; j0 < n; j0 += nc) {
        const int nb = std::min(nc, n - j0);
        // skip blocks the Hermitian modes leave alone
        if (herm == 1 && i0 > j0 + nb - 1) continue;
        if (herm == 2 && (j0 >> 6) > ((i0 + mb - 1) >> 6)) continue;
        PW_TRY(oz_block(w, opA, opB, mb, nb, kb, alpha, at(A, opA, lda, i0, k0), lda,
                        at(B, opB == 'N' ? 'C' : 'N', ldb, j0, k0), ldb, bt, C + i0 + (long)j0 * ldc, ldc, st,
                        herm, i0, j0));
      }
    }
  }
  if (herm == 1) {
    pw_count_launch();
    k_oz_mirror<<<dim3((m + 31) / 32, (m + 31) / 32), dim3(32, 32), 0, st>>>(C, ldc, m);
    PW_TRY(pw_check_launch("oz mirror"));
  }
  return PW_OK;
}

namespace {
std::atomic<int> g_f64_products{1};
// complex multiply-adds below which the FP64 pipe beats slicing the operands
constexpr double kOzMinMacs = 8.0 * (1 << 20);
}  // namespace

int pw_f64_products_mode() { return g_f64_products.load(); }

extern "C" pw_status pw_dense_products(int mode) {
  if (mode != 0 && mode != 1) return PW_ERR_ARG;
  g_f64_products.store(mode);
  return PW_OK;
}

bool pw_use_oz(int m, int n, int k) {
  return k > 0 && g_f64_products.load() == 1 && (double)m * n * k >= kOzMinMacs;
}

pw_status pw_gemm64(pw_oz_ws *w, char opA, char opB, int m, int n, int k, double2 alpha, const double2 *A,
                    int lda, const double2 *B, int ldb, double2 beta, double2 *C, int ldc, double2 *ws,
                    size_t ws_elems, cudaStream_t st, int herm) {
  if (m <= 0 || n <= 0) return PW_OK;
  if (w && pw_use_oz(m, n, k))
    return pw_zgemm_oz(w, opA, opB, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, st, herm);
  return pw_zgemm_ex(opA, opB, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, ws, ws_elems, st, herm);
}

namespace {
pw_status zgemm_f64tc(char opA, char opB, int m, int n, int k, const double *alpha, const void *A, int lda,
                      const void *B, int ldb, const double *beta, void *C, int ldc, bool fixed, void *stream) {
  if (!alpha || !beta || m < 0 || n < 0 || k < 1 || !A || !B || !C) return PW_ERR_ARG;
  if (ldc < m || lda < (opA == 'N' ? m : k) || ldb < (opB == 'N' ? k : n)) return PW_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  pw_oz_ws w;
  w.mem = pw_mem{true, st};
  w.fixed = fixed;
  const pw_status r = pw_zgemm_oz(&w, opA, opB, m, n, k, make_double2(alpha[0], alpha[1]), (const double2 *)A, lda,
                                  (const double2 *)B, ldb, make_double2(beta[0], beta[1]), (double2 *)C, ldc, st, 0);
  return pw_finish(r, w.err, st, [&] { pw_oz_free(&w); });
}
}  // namespace

extern "C" pw_status pw_zgemm_f64tc(char opA, char opB, int m, int n, int k, const double *alpha,
                                    const void *A, int lda, const void *B, int ldb, const double *beta, void *C,
                                    int ldc, void *stream) {
  return zgemm_f64tc(opA, opB, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, false, stream);
}
extern "C" pw_status pw_zgemm_f64tc_fixed(char opA, char opB, int m, int n, int k, const double *alpha,
                                          const void *A, int lda, const void *B, int ldb, const double *beta,
                                          void *C, int ldc, void *stream) {
  return zgemm_f64tc(opA, opB, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, true, stream);
}

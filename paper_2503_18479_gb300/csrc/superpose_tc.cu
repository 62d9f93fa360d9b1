// superpose_tc.cu -- (c) B = H I (paper Eq. 7) on the 5th-generation tensor cores.
//
// Real GEMM per structure: rows = field points p (A operand: H, bf16 pieces), columns =
// (configuration, frequency, re/im) (B operand: I, bf16 pieces), K = ports. With
// x = x0 + x1 + x2 (bf16 pieces, exact for FP32 data) the product keeps the six piece
// pairs of order >= 2^-16 (x0y0, x0y1, x1y0, x0y2, x1y1, x2y0) accumulated in FP32 in
// tensor memory: relative error ~2^-24 per product (MTS_MIXED). MTS_BF16 uses x0 y0 only.
// When K spans more than kSumMaxPlain 64-wide chunks (MTS_MIXED, more than 256 ports), each
// group of kSumChunks chunks goes to a fresh accumulator and the epilogue adds the group
// partials into a running double-float sum (hi + lo, Knuth's TwoSum) held in two more TMEM
// regions: the FP32 accumulator then grows only to the magnitude of one group's partial sum
// instead of the running sum over the whole K range (measured on the 1024-port array:
// 2.4e-6 relative error with one accumulator, 2e-7 with one per chunk).
//
// Persistent kernel, one CTA per SM, 192 threads:
//   warp 0      producer: cp.async.bulk copies of the pre-swizzled 16 KB operand tiles
//               (global images already in the 128-byte-swizzled K-major layout) into a
//               ring of shared-memory stages, completion via mbarrier transaction counts
//   warp 1      allocates 256 TMEM columns (two 128x128 FP32 accumulators); lane 0
//               issues tcgen05.mma (M=128, N=128, K=16, kind::f16 with bf16 inputs) and
//               tcgen05.commit to release stages and hand accumulators to the epilogue
//   warps 2..5  epilogue: tcgen05.ld of the accumulator (warp w reads lanes 32*(w%4)..),
//               release of the accumulator, then streaming complex64 stores: lane = point,
//               so each warp store writes 32 consecutive points (256 contiguous bytes)
// Every mbarrier wait is bounded; on timeout the kernel records an error word, stops
// issuing work, waits (bounded) for its own copies, frees TMEM and returns.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"
#include "tc_common.cuh"

namespace mts {

namespace tc {

constexpr int kThreads = 192;
constexpr uint32_t kTileBytes = kTileP * kChunkK * 2;  // 16 KB (also kTileN x 64 x 2)
constexpr uint32_t kTmemCols = 512;  // two 128-column accumulators + running sum hi, lo
constexpr uint32_t kHiCol = 256, kLoCol = 384;
constexpr int kSumChunks = 2;    // K chunks per accumulator when the running sum is used
constexpr int kSumMaxPlain = 4;  // up to this many K chunks, one FP32 accumulator (at most
                                 // 4 x 4 K-steps x 6 piece pairs = 96 FP32 roundings)

struct Unit {
  int s, N, F, nkc;
  int64_t P, pt, nt, nptile, nntile;
};

__device__ inline Unit unit_info(const SuperposeArgs& a, int64_t u) {
  Unit x;
  if (a.uni.on) {  // one structure: geometry from the arguments, no table loads
    x.s = 0;
    x.N = a.uni.N;
    x.F = a.uni.F;
    x.P = a.uni.P;
    x.nkc = a.uni.nkc;
    x.nptile = a.uni.nptile;
    x.nntile = a.uni.nntile;
    x.pt = u % x.nptile;
    x.nt = u / x.nptile;
    return x;
  }
  x.s = find_struct_i64(a.unit_off, a.n_struct, u);
  x.N = a.port_off[x.s + 1] - a.port_off[x.s];
  x.F = a.freq_off[x.s + 1] - a.freq_off[x.s];
  x.P = a.point_off[x.s + 1] - a.point_off[x.s];
  x.nkc = (x.N + kChunkK - 1) / kChunkK;
  x.nptile = (x.P + kTileP - 1) / kTileP;
  x.nntile = (2 * a.n_cfg * x.F + kTileN - 1) / kTileN;
  int64_t lu = u - a.unit_off[x.s];
  x.pt = lu % x.nptile;
  x.nt = lu / x.nptile;
  return x;
}

// Rows of B_out that the systems of a column tile write, in order: system (b, f) of a
// structure starts at b sumFP + fp_off + f P. Both cases are one addition per row: the rows
// are evenly spaced when the structure is alone (sumFP = F P, so stride P runs on across
// configurations) or has one frequency (stride sumFP); otherwise the stride is P with a jump
// after the last frequency. Recomputing the 64-bit products per row instead made the epilogue
// the bound of every batch with several frequencies: 3477 us against 1121 us for the same
// 6.76 GB (8 ports, 1024 configurations x 201 frequencies x 4104 points).
struct RowWalk {
  float2* dst;
  int64_t stride, jump;
  int f, F;
  bool even;
  __device__ RowWalk(const SuperposeArgs& a, const Unit& x, int64_t sys, int64_t fpo, int64_t p) {
    const int64_t b = a.uni.on ? 0 : sys / x.F;
    F = x.F;
    f = a.uni.on ? 0 : (int)(sys - b * x.F);
    even = a.uni.on || x.F == 1;
    stride = a.uni.on || x.F > 1 ? x.P : a.sumFP;
    jump = a.sumFP - (int64_t)x.F * x.P;
    dst = static_cast<float2*>(a.B_out) + (a.uni.on ? sys * x.P : b * a.sumFP + (int64_t)f * x.P) +
          fpo + p;
  }
  __device__ void next() {
    dst += stride;
    if (!even && ++f == F) {
      f = 0;
      dst += jump;
    }
  }
};

// One point's 128 accumulator columns (64 systems, re and im) to the field
__device__ __forceinline__ void store_tile(const SuperposeArgs& a, const Unit& x, int64_t sys0, int64_t fpo,
                                           int64_t nsys, int64_t p, const float* v) {
  if (p >= x.P) return;
  RowWalk w(a, x, sys0, fpo, p);
  if (w.even && sys0 + kTileN / 2 <= nsys) {
    float2* dst = w.dst;
    const int64_t stride = w.stride;
#pragma unroll
    for (int i = 0; i < kTileN / 2; ++i) {
      st_cs_f2(dst, v[2 * i], v[2 * i + 1]);
      dst += stride;
    }
  } else {
    const int n = (int)min((int64_t)kTileN / 2, nsys - sys0);
#pragma unroll
    for (int i = 0; i < kTileN / 2; ++i) {
      if (i < n) st_cs_f2(w.dst, v[2 * i], v[2 * i + 1]);
      w.next();
    }
  }
}

template <int NPIECE>
__global__ void __launch_bounds__(kThreads, 1) superpose_tc_kernel(SuperposeArgs a, int32_t* err) {
  constexpr int NSTAGE = NPIECE == 3 ? 2 : 4;
  constexpr uint32_t kStageBytes = 2u * NPIECE * kTileBytes;
  constexpr int NPAIR = NPIECE == 3 ? 6 : 1;
  // piece pairs (A piece, B piece), smallest products first
  constexpr int pa[6] = {2, 1, 0, 1, 0, 0};
  constexpr int pb[6] = {0, 1, 2, 0, 1, 0};

  extern __shared__ __align__(1024) unsigned char smem_dyn[];
  // 1024-byte aligned operand area
  uintptr_t sbase = (reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023);
  unsigned char* stages = reinterpret_cast<unsigned char*>(sbase);
  uint64_t* bars = reinterpret_cast<uint64_t*>(stages + NSTAGE * kStageBytes);
  uint64_t* full = bars;                 // [NSTAGE]
  uint64_t* empty = bars + NSTAGE;       // [NSTAGE]
  uint64_t* tfull = bars + 2 * NSTAGE;   // [2]
  uint64_t* tempty = tfull + 2;          // [2]
  uint64_t* mdone = tempty + 2;          // [1] all issued MMAs complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mdone + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t G = gridDim.x;
  const int64_t u_begin = a.total_units * blockIdx.x / G;
  const int64_t u_end = a.total_units * (blockIdx.x + 1) / G;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NSTAGE; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 128);
    }
    mbar_init(mdone, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ---------------- producer ----------------
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      uint32_t last_phase[NSTAGE];
      bool used[NSTAGE];
      // the B-operand tile (structure, column tile, K chunk) each stage holds: consecutive
      // units of a CTA usually share it (units advance along the point tiles first), and a
      // stage whose B image is already the one needed only refills its A pieces
      uint64_t bkey[NSTAGE];
      for (int i = 0; i < NSTAGE; ++i) {
        used[i] = false;
        last_phase[i] = 0;
        bkey[i] = ~0ull;
      }
      for (int64_t u = u_begin; u < u_end && ok; ++u) {
        Unit x = unit_info(a, u);
        const unsigned char* Ab =
            reinterpret_cast<const unsigned char*>(a.Aop + (a.uni.on ? 0 : a.t.aop_off[x.s]));
        const unsigned char* Bb =
            reinterpret_cast<const unsigned char*>(a.Bop + (a.uni.on ? 0 : a.bop_off[x.s]));
        for (int kc = 0; kc < x.nkc && ok; ++kc) {
          if (!mbar_wait(&empty[stage], phase ^ 1u, err, 1)) {
            ok = false;
            break;
          }
          unsigned char* sA = stages + stage * kStageBytes;
          unsigned char* sB = sA + NPIECE * kTileBytes;
          const uint64_t key = ((uint64_t)x.s << 44) | ((uint64_t)x.nt << 12) | (uint64_t)kc;
          const bool needB = bkey[stage] != key;
          mbar_arrive_expect_tx(&full[stage], needB ? kStageBytes : NPIECE * kTileBytes);
          for (int q = 0; q < NPIECE; ++q) {
            const unsigned char* ga =
                Ab + ((size_t)(q * x.nptile + x.pt) * x.nkc + kc) * kTileBytes;
            bulk_g2s(sA + q * kTileBytes, ga, kTileBytes, &full[stage]);
            if (needB) {
              const unsigned char* gb =
                  Bb + ((size_t)(q * x.nntile + x.nt) * x.nkc + kc) * kTileBytes;
              bulk_g2s(sB + q * kTileBytes, gb, kTileBytes, &full[stage]);
            }
          }
          bkey[stage] = key;
          used[stage] = true;
          last_phase[stage] = phase;
          if (++stage == NSTAGE) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      // no copy may still be in flight when the CTA exits
      for (int i = 0; i < NSTAGE; ++i)
        if (used[i]) mbar_wait(&full[i], last_phase[i], err, 5);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t aphase = 0;
      bool ok = true;
      for (int64_t u = u_begin; u < u_end && ok; ++u) {
        Unit x = unit_info(a, u);
        // K chunks per accumulator hand-off: all of them, or kSumChunks with the running sum
        const int group = (NPIECE == 3 && x.nkc > kSumMaxPlain) ? kSumChunks : x.nkc;
        for (int k0 = 0; k0 < x.nkc && ok; k0 += group) {
          if (!mbar_wait(&tempty[acc], aphase ^ 1u, err, 2)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + (uint32_t)acc * 128u;
          const int k1 = min(k0 + group, x.nkc);
          for (int kc = k0; kc < k1; ++kc) {
            if (!mbar_wait(&full[stage], phase, err, 3)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t sA = smem_u32(stages + stage * kStageBytes);
            const uint32_t sB = sA + NPIECE * kTileBytes;
            // K-steps of 16 that hold data (the tail of the last chunk is zero in both
            // operands: its all-zero steps are not issued)
            const int ksteps = min(kChunkK / 16, (x.N - kc * kChunkK + 15) / 16);
#pragma unroll
            for (int pp = 0; pp < NPAIR; ++pp) {
              const int qa = NPIECE == 3 ? pa[pp] : 0, qb = NPIECE == 3 ? pb[pp] : 0;
              const uint64_t da = make_desc(sA + qa * kTileBytes);
              const uint64_t db = make_desc(sB + qb * kTileBytes);
#pragma unroll
              for (int kk = 0; kk < kChunkK / 16; ++kk) {
                // advance 16 elements (32 bytes) along K inside the swizzle atom
                if (kk < ksteps)
                  mma_bf16(d_tmem, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2),
                           (kc > k0 || pp > 0 || kk > 0) ? 1u : 0u);
              }
            }
            mma_commit(&empty[stage]);
            if (++stage == NSTAGE) {
              stage = 0;
              phase ^= 1u;
            }
          }
          if (!ok) break;
          mma_commit(&tfull[acc]);
          if (++acc == 2) {
            acc = 0;
            aphase ^= 1u;
          }
        }
      }
      // every MMA issued by this thread has finished before TMEM is released
      mma_commit(mdone);
      mbar_wait(mdone, 0, err, 6);
    }
  } else {
    // ---------------- epilogue (warps 2..5) ----------------
    const int quarter = warp & 3;  // TMEM lanes 32*quarter .. +31
    int acc = 0;
    uint32_t aphase = 0;
    bool alive = true;
    for (int64_t u = u_begin; u < u_end && alive; ++u) {
      Unit x = unit_info(a, u);
      const int64_t p = x.pt * kTileP + quarter * 32 + lane;
      const int64_t nsys = a.n_cfg * x.F;
      const int64_t sys0 = x.nt * (kTileN / 2);
      const int64_t fpo = a.uni.on ? 0 : a.t.fp_off[x.s];
      if (NPIECE == 3 && x.nkc > kSumMaxPlain) {
        // one partial per group of kSumChunks K chunks, added into the running sum (hi, lo)
        const uint32_t lrow = (uint32_t)(quarter * 32) << 16;
        for (int kc = 0; kc < x.nkc; kc += kSumChunks) {
          int ok = (lane == 0) ? (int)mbar_wait(&tfull[acc], aphase, err, 4) : 1;
          ok = __shfl_sync(0xffffffffu, ok, 0);
          if (!ok) {
            alive = false;
            break;
          }
          mbar_wait(&tfull[acc], aphase, err, 4);
          tc_fence_after();
          const bool last = kc + kSumChunks >= x.nkc;
#pragma unroll 1
          for (int c = 0; c < 4; ++c) {
            float pv[32], hi[32], lo[32];
            tmem_ld32(tmem_base + lrow + (uint32_t)acc * 128u + c * 32, pv);
            if (kc > 0) {
              tmem_ld32(tmem_base + lrow + kHiCol + c * 32, hi);
              tmem_ld32(tmem_base + lrow + kLoCol + c * 32, lo);
            }
            tmem_wait_ld();
            if (kc == 0) {
#pragma unroll
              for (int i = 0; i < 32; ++i) {
                hi[i] = pv[i];
                lo[i] = 0.0f;
              }
            } else {
#pragma unroll
              for (int i = 0; i < 32; ++i) two_sum_acc(hi[i], lo[i], pv[i]);
            }
            if (!last) {
              tmem_st32(tmem_base + lrow + kHiCol + c * 32, hi);
              tmem_st32(tmem_base + lrow + kLoCol + c * 32, lo);
            } else if (p < x.P) {
              // columns 32c .. 32c + 31: systems sys0 + 16c .. + 15
              RowWalk w(a, x, sys0 + 16 * c, fpo, p);
              const int n = (int)min((int64_t)16, nsys - sys0 - 16 * c);
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                if (i < n)
                  st_cs_f2(w.dst, __fadd_rn(hi[2 * i], lo[2 * i]), __fadd_rn(hi[2 * i + 1], lo[2 * i + 1]));
                w.next();
              }
            }
          }
          tmem_wait_st();
          tc_fence_before();
          mbar_arrive(&tempty[acc]);
          if (++acc == 2) {
            acc = 0;
            aphase ^= 1u;
          }
        }
        continue;
      }
      // lane 0 does the bounded wait; the outcome is made warp-uniform before the
      // warp-collective tcgen05.ld
      int ok = (lane == 0) ? (int)mbar_wait(&tfull[acc], aphase, err, 4) : 1;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      mbar_wait(&tfull[acc], aphase, err, 4);  // already complete: acquire for every lane
      tc_fence_after();
      float v[128];
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)acc * 128u;
#pragma unroll
      for (int c = 0; c < 4; ++c) tmem_ld32(taddr + c * 32, v + c * 32);
      tmem_wait_ld();
      tc_fence_before();
      mbar_arrive(&tempty[acc]);
      if (++acc == 2) {
        acc = 0;
        aphase ^= 1u;
      }
      store_tile(a, x, sys0, fpo, nsys, p, v);
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(kTmemCols)
                 : "memory");
  }
}

// One structure whose column tile (NPIECE pieces of every K chunk) fits in shared memory beside a
// ring for the point tiles: the column tile stays while the point tiles pass, piece by piece. With
// both operands through stages of a chunk, a unit of more than one chunk read both tiles again
// each time (65,600 points, 8192 columns, K = 130: 288 KB a unit, 970 us; resident 913 us), and a
// last chunk of at most 16 columns took three tiles for six MMAs; as one tile with its pieces side
// by side (tail_packed): 783 us. With one chunk the stages keep their column tile anyway and
// hold more of the point tiles (64 ports: 381 us in both forms), so that form stays there.
// Barriers: full/empty per ring slot, bfull/bempty per chunk of a column tile; bempty is
// committed by the last unit that reads it.
constexpr int kSlots = 14;       // 16 KB each: the column tile first, the ring behind it
constexpr int kResidentMax = 9;  // of them at most for the column tile

// An MMA of M = 128 takes much the same time for N = 128 and N = 256, so the products of an A
// piece with the first two B pieces go out as one MMA of N = 256: the pieces' tiles follow each
// other in shared memory as the rows of one operand, and the second one's products have an
// accumulator of their own, which the epilogue adds (65,600 points below: 783 -> 726 us).
//
// MMAs are only sure to run in order on one accumulator in one shape. So a unit's products of
// N = 256 (every A piece with B pieces 0 and 1) go out first, and when they are done those of
// N = 128: piece 0 with the third B piece, and the packed last chunk. The A tiles come as pieces 1
// and 2 of every full chunk, then their pieces 0, whose slots are held until both shapes have
// read them (at most three of five slots or more), then the last chunk. The products of N = 128 go
// to the second accumulator, which is small: added to the first one, behind the largest products,
// they put B of 80 ports 2.6e-7 off instead of 1.7e-7.
// The wait itself costs nothing (the bound is the latency of the point tiles, 16 KB each, over the
// ring's slots), the held slots do: 651 us in the order of arrival against 726 us, 282 against
// 321 us for half the columns at K = 104. A tile of zeros beside the third pieces, which makes their
// products N = 256 too, takes a slot for good: 734 and 305 us, 534 against 511 us at K = 192.
constexpr uint32_t kIdesc256 = (kIdesc & ~(0x3fu << 17)) | ((256u >> 3) << 17);

// 16 KB tiles that one side of a unit takes
__host__ __device__ inline int unit_tiles(int N, int nkc, int npieces) {
  return tail_packed(N, npieces) ? (nkc - 1) * npieces + 1 : nkc * npieces;
}

template <int NPIECE>
__global__ void __launch_bounds__(kThreads, 1) superpose_tc_resident_kernel(SuperposeArgs a, int32_t* err) {
  constexpr uint32_t kAcc = NPIECE == 3 ? 256 : 128;  // TMEM columns of an accumulator
  extern __shared__ __align__(1024) unsigned char smem_dyn[];
  const uintptr_t sbase = (reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023);
  unsigned char* sB = reinterpret_cast<unsigned char*>(sbase);
  uint64_t* full = reinterpret_cast<uint64_t*>(sB + kSlots * kTileBytes);  // [kSlots]
  uint64_t* empty = full + kSlots;                                         // [kSlots]
  uint64_t* bfull = empty + kSlots;                                        // [kResidentMax]
  uint64_t* bempty = bfull + kResidentMax;                                 // [kResidentMax]
  uint64_t* tfull = bempty + kResidentMax;                                 // [2]
  uint64_t* tempty = tfull + 2;                                            // [2]
  uint64_t* mdone = tempty + 2;
  uint64_t* wide = mdone + 1;  // a unit's products of N = 256 done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(wide + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkc = a.uni.nkc, N = a.uni.N;
  const bool packed = tail_packed(N, NPIECE);
  const int nfull = packed ? nkc - 1 : nkc;  // chunks with a tile per piece
  const int nB = unit_tiles(N, nkc, NPIECE), ring = kSlots - nB;
  unsigned char* sA = sB + nB * kTileBytes;
  const int64_t nptile = a.uni.nptile, nntile = a.uni.nntile;
  const int64_t u_begin = a.total_units * blockIdx.x / gridDim.x;
  const int64_t u_end = a.total_units * (blockIdx.x + 1) / gridDim.x;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2 * (kSlots + kResidentMax); ++i) mbar_init(&full[i], 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 128);
    }
    mbar_init(mdone, 1);
    mbar_init(wide, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(2 * kAcc)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ---------------- producer ----------------
    if (lane == 0) {
      const unsigned char* Ab = reinterpret_cast<const unsigned char*>(a.Aop);
      const unsigned char* Bb = reinterpret_cast<const unsigned char*>(a.Bop);
      int slot = 0, nb = 0;  // ring slot, column tiles begun
      uint32_t phase = 0;
      int64_t copies = 0, held = -1;
      int b_chunks = 0;  // chunks of the current column tile asked for
      bool ok = true;
      for (int64_t u = u_begin; u < u_end && ok; ++u) {
        const int64_t nt = u / nptile, pt = u - nt * nptile;
        const bool fresh = nt != held;
        if (fresh) {
          held = nt;
          ++nb;
          b_chunks = 0;
        }
        auto tile = [&](int q, int kc) {  // piece q of chunk kc of the point tile
          ok = mbar_wait(&empty[slot], phase ^ 1u, err, 1);
          if (!ok) return;
          mbar_arrive_expect_tx(&full[slot], kTileBytes);
          bulk_g2s(sA + slot * kTileBytes, Ab + ((size_t)(q * nptile + pt) * nkc + kc) * kTileBytes,
                   kTileBytes, &full[slot]);
          ++copies;
          if (++slot == ring) {
            slot = 0;
            phase ^= 1u;
          }
        };
        for (int kc = 0; kc < nkc && ok; ++kc) {
          const int np = kc == nfull ? 1 : NPIECE;
          if (fresh) {
            ok = mbar_wait(&bempty[kc], (uint32_t)nb & 1u, err, 1);
            if (!ok) break;
            mbar_arrive_expect_tx(&bfull[kc], np * kTileBytes);
            for (int q = 0; q < np; ++q)
              bulk_g2s(sB + (kc * NPIECE + q) * kTileBytes,
                       Bb + ((size_t)(q * nntile + nt) * nkc + kc) * kTileBytes, kTileBytes, &bfull[kc]);
            b_chunks = kc + 1;
          }
          for (int q = NPIECE == 1 ? 0 : 1; q < np && ok; ++q) tile(q, kc);
        }
        if constexpr (NPIECE == 3)
          for (int kc = 0; kc < nkc && ok; ++kc) tile(0, kc);
      }
      // no copy may still be in flight when the CTA exits: the last use of every slot and chunk
      for (int i = 0; i < ring && i < copies; ++i)
        mbar_wait(&full[i], (uint32_t)(((copies - 1 - i) / ring) & 1), err, 5);
      for (int kc = 0; kc < nkc; ++kc) {
        const int uses = kc < b_chunks ? nb : nb - 1;
        if (uses > 0) mbar_wait(&bfull[kc], (uint32_t)(uses - 1) & 1u, err, 5);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      int slot = 0, nb = 0, acc = 0;
      uint32_t phase = 0, aphase = 0, wphase = 0;
      int64_t held_nt = -1;
      bool ok = true;
      for (int64_t u = u_begin; u < u_end && ok; ++u) {
        const int64_t nt = u / nptile;
        const bool fresh = nt != held_nt, last = u + 1 == u_end || (u + 1) / nptile != nt;
        if (fresh) {
          held_nt = nt;
          ++nb;
        }
        ok = mbar_wait(&tempty[acc], aphase ^ 1u, err, 2);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)acc * kAcc;
        // K steps of the A tile in a slot with piece qb of chunk kc, to the accumulator d
        auto steps = [&](uint32_t d, int s, int kc, int qb, uint32_t idesc, bool first) {
          const int ksteps = min(kChunkK / 16, (N - kc * kChunkK + 15) / 16);
          const uint64_t da = make_desc(smem_u32(sA) + (uint32_t)s * kTileBytes);
          const uint64_t db = make_desc(smem_u32(sB) + (uint32_t)(kc * NPIECE + qb) * kTileBytes);
#pragma unroll
          for (int kk = 0; kk < kChunkK / 16; ++kk)
            if (kk < ksteps)
              mma_bf16(d, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), (!first || kk > 0) ? 1u : 0u, idesc);
        };
        auto arrived = [&]() {
          ok = mbar_wait(&full[slot], phase, err, 3);
          if (ok) tc_fence_after();
          return ok;
        };
        auto advance = [&]() {
          if (++slot == ring) {
            slot = 0;
            phase ^= 1u;
          }
        };
        if constexpr (NPIECE == 3) {  // piece pairs of order >= 2^-16, and (2, 1)
          for (int kc = 0; kc < nfull && ok; ++kc) {
            if (fresh) ok = mbar_wait(&bfull[kc], (uint32_t)(nb - 1) & 1u, err, 3);
            for (int q = 1; q < 3 && ok; ++q) {
              if (!arrived()) break;
              steps(d_tmem, slot, kc, 0, kIdesc256, kc == 0 && q == 1);
              mma_commit(&empty[slot]);
              advance();
            }
          }
          int held = slot;  // of the first piece 0
          for (int kc = 0; kc < nfull && ok; ++kc) {
            if (!arrived()) break;
            steps(d_tmem, slot, kc, 0, kIdesc256, false);
            advance();
          }
          if (!ok) break;
          mma_commit(wide);
          ok = mbar_wait(wide, wphase, err, 8);
          if (!ok) break;
          wphase ^= 1u;
          tc_fence_after();
          const uint32_t d_low = d_tmem + kTileN;  // the small products' accumulator
          for (int kc = 0; kc < nfull; ++kc) {
            steps(d_low, held, kc, 2, kIdesc, false);
            mma_commit(&empty[held]);
            if (last) mma_commit(&bempty[kc]);
            if (++held == ring) held = 0;
          }
          if (packed) {  // piece q is K step q of the one tile
            if (fresh) ok = mbar_wait(&bfull[nfull], (uint32_t)(nb - 1) & 1u, err, 3);
            if (!ok || !arrived()) break;
            const uint64_t da = make_desc(smem_u32(sA) + (uint32_t)slot * kTileBytes);
            const uint64_t db = make_desc(smem_u32(sB) + (uint32_t)(nfull * NPIECE) * kTileBytes);
#pragma unroll
            for (int qa = 2; qa >= 0; --qa)
#pragma unroll
              for (int qb = 2 - qa; qb >= 0; --qb)
                mma_bf16(d_low, da + (uint64_t)(qa * 2), db + (uint64_t)(qb * 2), 1u);
            mma_commit(&empty[slot]);
            if (last) mma_commit(&bempty[nfull]);
            advance();
          }
        } else {
          for (int kc = 0; kc < nkc && ok; ++kc) {
            if (fresh) ok = mbar_wait(&bfull[kc], (uint32_t)(nb - 1) & 1u, err, 3);
            if (!ok || !arrived()) break;
            steps(d_tmem, slot, kc, 0, kIdesc, kc == 0);
            mma_commit(&empty[slot]);
            advance();
            if (last) mma_commit(&bempty[kc]);
          }
        }
        if (!ok) break;
        mma_commit(&tfull[acc]);
        if (++acc == 2) {
          acc = 0;
          aphase ^= 1u;
        }
      }
      // every MMA issued by this thread has finished before TMEM is released
      mma_commit(mdone);
      mbar_wait(mdone, 0, err, 6);
    }
  } else {
    // ---------------- epilogue (warps 2..5) ----------------
    const int quarter = warp & 3;  // TMEM lanes 32*quarter .. +31
    int acc = 0;
    uint32_t aphase = 0;
    for (int64_t u = u_begin; u < u_end; ++u) {
      const Unit x = unit_info(a, u);
      int ok = (lane == 0) ? (int)mbar_wait(&tfull[acc], aphase, err, 4) : 1;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      mbar_wait(&tfull[acc], aphase, err, 4);  // already complete: acquire for every lane
      tc_fence_after();
      float v[128];
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)acc * kAcc;
#pragma unroll
      for (int c = 0; c < 4; ++c) tmem_ld32(taddr + c * 32, v + c * 32);
      tmem_wait_ld();
      if constexpr (NPIECE == 3) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float y[32];
          tmem_ld32(taddr + 128 + c * 32, y);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) v[32 * c + i] += y[i];
        }
      }
      tc_fence_before();
      mbar_arrive(&tempty[acc]);
      if (++acc == 2) {
        acc = 0;
        aphase ^= 1u;
      }
      store_tile(a, x, x.nt * (kTileN / 2), 0, a.n_cfg * x.F, x.pt * kTileP + quarter * 32 + lane, v);
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(2 * kAcc)
                 : "memory");
  }
}

template <int NPIECE>
size_t smem_bytes() {
  constexpr int NSTAGE = NPIECE == 3 ? 2 : 4;
  return 1024 + (size_t)NSTAGE * 2 * NPIECE * kTileBytes + 8 * (2 * NSTAGE + 5) + 16;
}

constexpr size_t kResidentSmem = 1024 + (size_t)kSlots * kTileBytes + 8 * (2 * (kSlots + kResidentMax) + 6) + 16;

template <int NPIECE>
cudaError_t launch(const SuperposeArgs& a, int64_t grid, int32_t* err, cudaStream_t st) {
  const bool resident = a.uni.on && a.uni.nkc > 1 && unit_tiles(a.uni.N, a.uni.nkc, NPIECE) <= kResidentMax;
  const auto kernel = resident ? superpose_tc_resident_kernel<NPIECE> : superpose_tc_kernel<NPIECE>;
  const size_t sm = resident ? kResidentSmem : smem_bytes<NPIECE>();
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  kernel<<<(unsigned)grid, kThreads, sm, st>>>(a, err);
  return cudaSuccess;
}

}  // namespace tc

static int g_num_sms = 0;

cudaError_t launch_superpose_tc(const SuperposeArgs& a, mts_precision prec, cudaStream_t st) {
  if (g_num_sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_num_sms <= 0) g_num_sms = 1;
  }
  int64_t grid = a.total_units < g_num_sms ? a.total_units : g_num_sms;
  int32_t* err = a.err;
  if (err == nullptr) return cudaErrorInvalidValue;
  const cudaError_t e = prec == MTS_MIXED ? tc::launch<3>(a, grid, err, st) : tc::launch<1>(a, grid, err, st);
  if (e != cudaSuccess) return e;
  note_launch();
  return cudaGetLastError();
}

}  // namespace mts

// superpose_fp64_tc.cu -- (c) B = H I in FP64 on the tensor cores (MTS_FP64, one structure):
// both operands are cut into eight signed 8-bit digits on a common exponent per row, the digit
// products are summed exactly, and the sum is rounded to FP64 once (Ozaki's error-free split of a
// matrix product).
//
// This part's FP64 pipe does 1/76 of the FP32 rate, so the SIMT kernel ran at 1.05 TFLOP/s, its
// peak: 4005 us for 1024 configurations x 16,448 points x 64 ports, where this form takes 280.
// (8 ports, 8192 systems x 4104 points: 989 -> 476 us; 132 ports, 200 x 4160: 652 -> 83 us.) The tensor cores have no FP64
// rate to speak of either, but their bf16 products of 8-bit integers are exact, and so are FP32
// sums of integers below 2^24.
//
// Split. With E the largest exponent of a row over 64 ports, every element is x = X 2^(E - 61), X
// an integer below 2^62 (exact for elements within 2^9 of the largest, rounded at 2^-63 of it
// otherwise). Adding 0x80 to every byte of X makes its bytes the digits plus 128: X = sum_s d_s
// 256^(7-s), d_s in [-128, 127] and |d_0| <= 64. Products d_i e_j with i + j = g share the weight
// 256^(14-g); the groups g = 0..7 (36 pairs) are kept, each summed in its own FP32 accumulator:
// at most 64 x (6 2^14 + 2 2^13) = 7 2^20 in magnitude, an exact integer after every MMA. What
// is dropped (g >= 8) is 2^-61 of the row maxima's product, below the rounding of one FP64
// product. The eight integers of an output combine to a 75-bit one, rounded to FP64 once.
//
// Tile: 128 points x 64 columns (32 systems, re and im), so that its eight accumulators fill the
// 512 columns of tensor memory. 512 threads, one CTA per SM, units contiguous
// along the column tiles (the digits of H stay in shared memory while the point tile lasts):
//   digits of the next column tile from registers into the 128-byte-swizzled K-major image (a
//   warp per row: lane = two ports, the row's exponent by one redux), epilogue of the previous
//   tile, MMAs (thread 0), then the next tile's currents loaded while they run.
// The digits are made on the fly because the stored form would triple the basis (16 bytes a
// value) and grow the tape. More than 64 ports: 64 at a time, the later chunks added
// to the field by the thread that wrote it.
// Rows or columns with infinities or NaN, and results outside the FP64 exponent range, are
// computed by a plain FP64 sum.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"
#include "tc_common.cuh"

namespace mts {
namespace oz {

using namespace tc;

constexpr int kThreads = 512;
constexpr int kDigits = 8;
constexpr int kCols = 64;                             // columns of a tile: kSys systems, re and im
constexpr int kSys = kCols / 2;
constexpr uint32_t kABytes = kTileP * kChunkK * 2;    // one digit of the point tile: 16 KB
constexpr uint32_t kBBytes = kCols * kChunkK * 2;     // one digit of the column tile: 8 KB
constexpr int kWin = 4;                               // groups of a window: N = 256
constexpr int kRows = kTileP / (kThreads / 32);       // rows of H per warp
constexpr int kSysWarp = kSys / (kThreads / 32);      // systems per warp

// kind::f16, A = B = bf16, D = f32, both K-major, M = 128, N = kWin kCols
constexpr uint32_t kIdescWin = (kIdesc & ~(0x3fu << 17)) | ((uint32_t)(kWin * kCols >> 3) << 17);

__device__ inline void tmem_ld4(uint32_t taddr, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

__device__ inline unsigned warp_max(unsigned v) {
  unsigned m;
  asm volatile("redux.sync.max.u32 %0, %1, 0xffffffff;" : "=r"(m) : "r"(v));
  return m;
}

__device__ inline unsigned exponent_of(double v) {
  return ((unsigned)__double2hiint(v) >> 20) & 0x7ffu;
}

// the biased digits (bytes, most significant first at the top) of v on the row exponent E
__device__ inline unsigned long long digits(double v, int E) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int e = (int)(b >> 52) & 0x7ff;
  unsigned long long m = b & 0xfffffffffffffull;
  if (e) m |= 1ull << 52;
  const int sh = 9 - (E - (e ? e : 1));  // E >= e
  unsigned long long x;
  if (sh >= 0) x = m << sh;
  else x = sh < -53 ? 0ull : ((m >> (-sh - 1)) + 1) >> 1;  // round half up in magnitude
  if ((long long)b < 0) x = 0ull - x;
  return x + 0x8080808080808080ull;
}

// digit s of two values as two bf16 (exact): byte - 128 through the FP32 integer range
template <int S>
__device__ inline uint32_t digit_pair(unsigned long long a, unsigned long long b) {
  constexpr int byte = 7 - S;
  const uint32_t wa = byte >= 4 ? (uint32_t)(a >> 32) : (uint32_t)a;
  const uint32_t wb = byte >= 4 ? (uint32_t)(b >> 32) : (uint32_t)b;
  const float fa = __uint_as_float(__byte_perm(wa, 0x4b000000u, 0x7440 | (byte & 3))) - 8388736.0f;
  const float fb = __uint_as_float(__byte_perm(wb, 0x4b000000u, 0x7440 | (byte & 3))) - 8388736.0f;
  return __byte_perm(__float_as_uint(fa), __float_as_uint(fb), 0x7632);
}

// all digits of elements (k, k + 1) of a row into the eight images, `off` their place in one
__device__ inline void put_digits(unsigned char* img, uint32_t stride, uint32_t off,
                                  unsigned long long a, unsigned long long b) {
  auto put = [&](int s, uint32_t v) { *reinterpret_cast<uint32_t*>(img + s * stride + off) = v; };
  put(0, digit_pair<0>(a, b));
  put(1, digit_pair<1>(a, b));
  put(2, digit_pair<2>(a, b));
  put(3, digit_pair<3>(a, b));
  put(4, digit_pair<4>(a, b));
  put(5, digit_pair<5>(a, b));
  put(6, digit_pair<6>(a, b));
  put(7, digit_pair<7>(a, b));
}

// sum_g acc_g 256^(7-g) 2^sc rounded to FP64; *ok = false where the exponent leaves its range
__device__ inline double combine(const float* acc, int sc, bool* ok) {
  int i[kDigits];
#pragma unroll
  for (int g = 0; g < kDigits; ++g) i[g] = __float2int_rn(acc[g]);
  // pairs stay below 2^31: |i0| <= 2^18, |i2| <= 2^21, |i4| <= 2^22, |i6| <= 6 2^20
  const long long hi = (long long)(i[0] * 256 + i[1]) * 65536 + (i[2] * 256 + i[3]);
  const long long lo = (long long)(i[4] * 256 + i[5]) * 65536 + (i[6] * 256 + i[7]);
  long long t = hi + (lo >> 32);
  uint32_t r = (uint32_t)lo;  // the value is t 2^32 + r
  const bool neg = t < 0;
  if (neg) {
    t = ~t + (r == 0);
    r = 0u - r;
  }
  if (t == 0) {
    if (r == 0) return 0.0;
    t = r;
    r = 0;
    sc -= 32;
  }
  const int s = __clzll(t);
  unsigned long long x = (unsigned long long)t << s;
  x |= s >= 32 ? (unsigned long long)r << (s - 32) : (unsigned long long)(r >> (32 - s));
  const unsigned long long m = (x >> 11) + ((x >> 10) & 1);
  const int e = 1023 + 95 - s + sc;
  if (e < 1 || e > 2045) *ok = false;
  const unsigned long long bits = ((unsigned long long)(unsigned)(e - 1) << 52) + m;
  return __longlong_as_double((long long)(bits | ((unsigned long long)neg << 63)));
}

__global__ void __launch_bounds__(kThreads, 1) superpose_fp64_tc_kernel(SuperposeArgs a, int64_t units,
                                                                        int32_t* err) {
  extern __shared__ __align__(1024) unsigned char smem_dyn[];
  const uintptr_t sbase = (reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023);
  unsigned char* sA = reinterpret_cast<unsigned char*>(sbase);
  unsigned char* sZ = sA + kDigits * kABytes;  // images of zeros before those of the columns
  unsigned char* sB = sZ + (kWin - 1) * kBBytes;
  uint64_t* bar = reinterpret_cast<uint64_t*>(sB + kDigits * kBBytes);  // MMAs of a turn done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar + 1);
  int* eA = reinterpret_cast<int*>(tmem_slot + 2);  // [2][128] row exponents, two point tiles in turn
  int* eB = eA + 2 * kTileP;                         // [2][64] column exponents by turn parity

  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int N = a.uni.N;
  const int64_t P = a.uni.P, nsys = a.n_cfg * a.uni.F, nntile = (nsys + kSys - 1) / kSys;
  const int nkc = a.uni.nkc;
  const double* __restrict__ H = static_cast<const double*>(a.H);
  const double* __restrict__ I = a.I;
  const bool vec = (N & 1) == 0;  // rows of H on 16-byte boundaries
  const int64_t u_begin = units * blockIdx.x / gridDim.x, u_end = units * (blockIdx.x + 1) / gridDim.x;

  for (uint32_t o = 16 * t; o < (kWin - 1) * kBBytes; o += 16 * kThreads)
    *reinterpret_cast<uint4*>(sZ + o) = make_uint4(0u, 0u, 0u, 0u);
  if (t == 0) {
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // digits of the rows warp * kRows .. of a point tile: ports (2 lane, 2 lane + 1) of chunk kc
  auto put_rows = [&](int64_t pt, int kc, int par) {
    const int k = kc * kChunkK + 2 * lane;
    double2 hv[kRows];
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int64_t p = pt * kTileP + warp * kRows + i;
      double2 v = make_double2(0.0, 0.0);
      if (p < P) {
        if (vec) {
          if (k < N) v = *reinterpret_cast<const double2*>(H + p * N + k);
        } else {
          if (k < N) v.x = H[p * N + k];
          if (k + 1 < N) v.y = H[p * N + k + 1];
        }
      }
      hv[i] = v;
    }
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int r = warp * kRows + i;
      const int E = (int)warp_max(max(exponent_of(hv[i].x), exponent_of(hv[i].y)));
      if (lane == 0) eA[par * kTileP + r] = E;
      put_digits(sA, kABytes, swz128(r, 2 * lane), digits(hv[i].x, E), digits(hv[i].y, E));
    }
  };
  // currents of the warp's systems of a column tile, same ports, loaded a turn ahead
  double2 iv[kSysWarp][2];
  auto load_currents = [&](int64_t nt, int kc) {
    const int k = kc * kChunkK + 2 * lane;
#pragma unroll
    for (int i = 0; i < kSysWarp; ++i) {
      const int64_t s = nt * kSys + warp * kSysWarp + i;
      iv[i][0] = iv[i][1] = make_double2(0.0, 0.0);
      if (s < nsys) {
        const double2* row = reinterpret_cast<const double2*>(I + 2 * s * N);
        if (k < N) iv[i][0] = row[k];
        if (k + 1 < N) iv[i][1] = row[k + 1];
      }
    }
  };
  auto put_currents = [&](int par) {
#pragma unroll
    for (int i = 0; i < kSysWarp; ++i) {
      const int q = warp * kSysWarp + i;
      const double2 c0 = iv[i][0], c1 = iv[i][1];
      const int Ex = (int)warp_max(max(exponent_of(c0.x), exponent_of(c1.x)));
      const int Ey = (int)warp_max(max(exponent_of(c0.y), exponent_of(c1.y)));
      if (lane == 0) {
        eB[par * kCols + 2 * q] = Ex;
        eB[par * kCols + 2 * q + 1] = Ey;
      }
      put_digits(sB, kBBytes, swz128(2 * q, 2 * lane), digits(c0.x, Ex), digits(c1.x, Ex));
      put_digits(sB, kBBytes, swz128(2 * q + 1, 2 * lane), digits(c0.y, Ey), digits(c1.y, Ey));
    }
  };
  // field of the tile in tensor memory: lane = point, this warp's 16 columns
  auto epilogue = [&](int64_t pt, int64_t nt, int kc, int par, int parA) {
    const int quarter = warp & 3, c0 = (warp >> 2) * 16;
    const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16);
    const int row = quarter * 32 + lane;
    const int64_t p = pt * kTileP + row;
    const int Er = eA[parA * kTileP + row];
    double2* out = static_cast<double2*>(a.B_out);
#pragma unroll 1
    for (int c = c0; c < c0 + 16; c += 4) {
      float v[kDigits][4];
#pragma unroll
      for (int g = 0; g < kDigits; ++g)
        tmem_ld4(acc + (uint32_t)(g * kCols + c), v[g]);
      tmem_wait_ld();
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int64_t s = nt * kSys + c / 2 + q;
        const int Ex = eB[par * kCols + c + 2 * q], Ey = eB[par * kCols + c + 2 * q + 1];
        float ax[kDigits], ay[kDigits];
#pragma unroll
        for (int g = 0; g < kDigits; ++g) {
          ax[g] = v[g][2 * q];
          ay[g] = v[g][2 * q + 1];
        }
        bool ok = Er != 0x7ff && Ex != 0x7ff && Ey != 0x7ff;
        // x = X 2^(E - 61) each, 256^7 per digit product: E + E' - 2 1023 - 122 + 56
        double2 b = make_double2(combine(ax, Er + Ex - 2112, &ok), combine(ay, Er + Ey - 2112, &ok));
        if (p < P && s < nsys) {
          if (!ok) {
            b = make_double2(0.0, 0.0);
            const int k1 = min(N, (kc + 1) * kChunkK);
            for (int k = kc * kChunkK; k < k1; ++k) {
              const double h = H[p * N + k];
              b.x = fma(h, I[2 * (s * N + k)], b.x);
              b.y = fma(h, I[2 * (s * N + k) + 1], b.y);
            }
          }
          double2* dst = out + s * P + p;
          if (kc > 0) {
            const double2 o = *dst;
            b.x += o.x;
            b.y += o.y;
          }
          *dst = b;
        }
      }
    }
  };

  // A turn is one K chunk of one unit. (Two half tiles of 32 columns, whose MMAs ran under each
  // other's epilogues, took 297 us where this form takes 280: the turns' fixed parts count more
  // than the MMAs.)
  int turn = 0, parA = 0, prev_kc = 0;
  int64_t last_pt = -1, prev_pt = 0, prev_nt = 0;
  bool alive = true;
  if (u_begin < u_end) load_currents(u_begin % nntile, 0);
  for (int64_t u = u_begin; u < u_end && alive; ++u) {
    const int64_t pt = u / nntile, nt = u - pt * nntile;
    for (int kc = 0; kc < nkc; ++kc, ++turn) {
      const int prev_parA = parA;
      put_currents(turn & 1);
      if (nkc > 1 || pt != last_pt) {
        parA ^= 1;  // the epilogue below still needs the previous rows' exponents
        put_rows(pt, kc, parA);
        last_pt = pt;
      }
      if (turn > 0) epilogue(prev_pt, prev_nt, prev_kc, (turn - 1) & 1, prev_parA);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncthreads();
      if (t == 0) {
        tc_fence_after();
        const int ksteps = min(kChunkK / 16, (N - kc * kChunkK + 15) / 16);
        const uint32_t aA = smem_u32(sA), aB = smem_u32(sB);
        // Digit i of the points with four digits of the columns, those of the groups g .. g + 3, as
        // one N = 256 MMA: the digits' images follow each other in shared memory as rows of
        // one operand, and so do the groups' accumulators in tensor memory (12 MMAs a K step
        // instead of 36 of N = 64, which take as long each). The images before digit 0 are
        // zeros. MMAs are only sure to run in order on one accumulator and in one shape, so the
        // two windows are fixed: with N = 64 to 256 at every group's base the same 12 took the
        // same time.
        for (int kk = 0; kk < ksteps; ++kk)
          for (int g = 0; g < kDigits; g += kWin)
            for (int i = 0; i < g + kWin; ++i)
              mma_bf16(tmem + g * kCols, make_desc(aA + i * kABytes) + (uint64_t)(kk * 2),
                       make_desc(aB + g * kBBytes - i * kBBytes) + (uint64_t)(kk * 2),
                       (i > 0 || kk > 0) ? 1u : 0u, kIdescWin);
        mma_commit(bar);
      }
      prev_pt = pt;
      prev_nt = nt;
      prev_kc = kc;
      // the next turn's currents while the MMAs run
      if (kc + 1 < nkc) load_currents(nt, kc + 1);
      else if (u + 1 < u_end) load_currents((u + 1) % nntile, 0);
      if (!mbar_wait(bar, (uint32_t)turn & 1u, err, 7)) alive = false;
      alive = __syncthreads_and(alive) != 0;
      tc_fence_after();
      if (!alive) break;
    }
  }
  if (turn > 0 && alive) epilogue(prev_pt, prev_nt, prev_kc, (turn - 1) & 1, parA);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

constexpr size_t kSmem = 1024 + kDigits * (size_t)kABytes + (kDigits + kWin - 1) * (size_t)kBBytes + 16 + 8 +
                         4 * 2 * (kTileP + kCols);
static_assert(kSmem <= 232448, "227 KB a CTA");

}  // namespace oz

// Units of the FP64 tensor-core superposition, or 0 where the SIMT kernel is the faster one.
// Measured cycles of the busiest SM: a tile of 128 x 32 (point, system) pairs takes kTile + kPort
// per port of the chunk, whatever part of it exists, and kChunk for every full chunk before (its
// rows are cut anew each time); the SIMT kernel takes 1 + 1.1 N per pair.
int64_t superpose_fp64_tc_units(int64_t N, int64_t P, int64_t nsys, int sms) {
  constexpr double kTile = 17100.0, kPort = 56.0, kChunk = 28000.0;
  const int64_t nkc = (N + kChunkK - 1) / kChunkK;
  const int64_t units = ((P + kTileP - 1) / kTileP) * ((nsys + oz::kSys - 1) / oz::kSys);
  const double tile = kTile + kPort * (double)(N - (nkc - 1) * kChunkK) + kChunk * (double)(nkc - 1);
  const double tc = (double)((units + sms - 1) / sms) * tile;
  const double simt = (1.0 + 1.1 * (double)N) * (double)P * (double)nsys / (double)sms;
  return tc < simt ? units : 0;
}

cudaError_t launch_superpose_fp64_tc(const SuperposeArgs& a, int64_t units, int sms, cudaStream_t st) {
  if (a.err == nullptr) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(oz::superpose_fp64_tc_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)oz::kSmem);
  if (e != cudaSuccess) return e;
  const int64_t grid = units < sms ? units : sms;
  oz::superpose_fp64_tc_kernel<<<(unsigned)grid, oz::kThreads, oz::kSmem, st>>>(a, units, a.err);
  note_launch();
  return cudaGetLastError();
}

}  // namespace mts

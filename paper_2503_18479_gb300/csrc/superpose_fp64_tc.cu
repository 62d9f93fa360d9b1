// superpose_fp64_tc.cu -- (c) B = H I in FP64 on the tensor cores (MTS_FP64, one structure):
// both operands are cut into nine signed 8-bit digits on a common exponent per row, the digit
// products are summed exactly, and the sum is rounded to FP64 once (Ozaki's error-free split of a
// matrix product).
//
// This part's FP64 pipe does 1/76 of the FP32 rate, so the SIMT kernel ran at 1.05 TFLOP/s, its
// peak: 4005 us for 1024 configurations x 16,448 points x 64 ports, where this form takes 374 to
// 468, by how many values are left to plain sums (8 ports, 8192 systems x 4104 points: 989 ->
// 609 us; 132 ports, 200 x 4160: 652 -> 92 us). The tensor cores have no FP64 rate to speak of
// either, but their bf16 products of 8-bit integers are exact, and so are FP32 sums of integers
// below 2^24.
//
// Split. With E the largest exponent of a row over 64 ports, every element is x = X 2^(E - 69), X
// an integer below 2^70 (exact for elements within 2^17 of the largest, rounded to nearest
// otherwise). Adding 0x80 to every byte of X makes its bytes the digits plus 128: X = sum_s d_s
// 256^(8-s), d_s in [-128, 127] and |d_0| <= 64. Products d_i e_j with i + j = g share the weight
// 256^(16-g); the groups g = 0..8 (45 pairs) are kept, each summed in its own FP32 accumulator:
// at most 64 x (7 2^14 + 2 2^13) = 2^23 in magnitude, an exact integer after every MMA. The nine
// integers of an output combine to an 84-bit one, rounded to FP64 once.
//
// Error. The groups that are dropped and the rounding of X come to at most 2^73.2 a port in
// units of the product X Y, where a plain FP64 sum of N products loses up to N 2^-53 sum |X Y|.
// So the form is as accurate wherever sum |X Y| >= 2^126: where one port has its two factors
// within 2^-3 and 2^-9 of their rows' largest (64-bit masks of such ports are kept beside the
// exponents), or where the result itself is that large. The remaining outputs, those of data
// graded so that large factors only meet small ones, are summed in plain FP64, eight lanes an
// output, while the next tile's MMAs run. They are a few in a thousand for arrays at 3 to 40 mm
// (currents spread over 2^7 and fields over 2^10 of their largest; with eight digits, 277 us, half
// of the outputs were below the line that corresponds), a tenth with a third of the ports nearly
// open and one port driven. So are rows or columns with infinities or NaN, and results outside the
// FP64 exponent range.
//
// A turn of 64 ports takes about 19,500 cycles: digits of the currents 2900, epilogue 8600 (its
// integer work), MMAs 6100.
//
// Tile: 128 points x 48 columns (24 systems, re and im), so that its nine accumulators fit in
// the 512 columns of tensor memory and nine digits of both in shared memory. 512 threads, one CTA
// per SM, units contiguous along the column tiles (the digits of H stay in shared memory while
// the point tile lasts):
//   digits of the next column tile from registers into the 128-byte-swizzled K-major image (a
//   warp per row: lane = two ports, the row's exponent by one redux), epilogue of the previous
//   tile, MMAs (thread 0), then the next tile's currents loaded and the plain sums made while
//   they run.
// The digits are made on the fly because the stored form would triple the basis (18 bytes a
// value) and grow the tape. More than 64 ports: 64 at a time, the later chunks added
// to the field by the warp that wrote it.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"
#include "tc_common.cuh"

namespace mts {
namespace oz {

using namespace tc;

constexpr int kThreads = 512;
constexpr int kDigits = 9;
constexpr int kCols = 48;                             // columns of a tile: kSys systems, re and im
constexpr int kSys = kCols / 2;
constexpr uint32_t kABytes = kTileP * kChunkK * 2;    // one digit of the point tile: 16 KB
constexpr uint32_t kBBytes = kCols * kChunkK * 2;     // one digit of the column tile: 6 KB
constexpr int kWin = 5;                               // groups of the first window
constexpr int kRows = kTileP / (kThreads / 32);       // rows of H per warp
constexpr int kColsWarp = kCols / (kThreads / 32);    // columns per warp

// kind::f16, A = B = bf16, D = f32, both K-major, M = 128, N = kCols for each of the groups
__host__ __device__ constexpr uint32_t idesc_groups(int groups) {
  return (kIdesc & ~(0x3fu << 17)) | ((uint32_t)(groups * kCols >> 3) << 17);
}

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

// the biased digits of a value on the row exponent E: digit 0 in the low byte of hi, then the
// bytes of lo, most significant first
struct Digits {
  unsigned long long lo;
  unsigned hi;
};
__device__ inline Digits digits(double v, int E) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int e = (int)(b >> 52) & 0x7ff;
  unsigned long long m = b & 0xfffffffffffffull;
  if (e) m |= 1ull << 52;
  const int sh = 17 - (E - (e ? e : 1));  // E >= e; 18 at most
  Digits x;
  if (sh >= 0) {
    x.lo = m << sh;
    x.hi = sh > 11 ? (unsigned)(m >> (64 - sh)) : 0u;
  } else {
    x.lo = sh < -53 ? 0ull : ((m >> (-sh - 1)) + 1) >> 1;  // round half up in magnitude
    x.hi = 0u;
  }
  if ((long long)b < 0) {
    x.hi = ~x.hi + (x.lo == 0ull);
    x.lo = 0ull - x.lo;
  }
  const unsigned long long biased = x.lo + 0x8080808080808080ull;
  x.hi += 0x80u + (biased < x.lo);
  x.lo = biased;
  return x;
}

// digit S of two values as two bf16 (exact): byte - 128 through the FP32 integer range
template <int S>
__device__ inline uint32_t digit_pair(const Digits& a, const Digits& b) {
  constexpr int byte = S == 0 ? 0 : 8 - S;
  const uint32_t wa = S == 0 ? a.hi : (byte >= 4 ? (uint32_t)(a.lo >> 32) : (uint32_t)a.lo);
  const uint32_t wb = S == 0 ? b.hi : (byte >= 4 ? (uint32_t)(b.lo >> 32) : (uint32_t)b.lo);
  const float fa = __uint_as_float(__byte_perm(wa, 0x4b000000u, 0x7440 | (byte & 3))) - 8388736.0f;
  const float fb = __uint_as_float(__byte_perm(wb, 0x4b000000u, 0x7440 | (byte & 3))) - 8388736.0f;
  return __byte_perm(__float_as_uint(fa), __float_as_uint(fb), 0x7632);
}

// all digits of elements (k, k + 1) of a row into the images, `off` their place in one
__device__ inline void put_digits(unsigned char* img, uint32_t stride, uint32_t off, const Digits& a,
                                  const Digits& b) {
  auto put = [&](int s, uint32_t v) { *reinterpret_cast<uint32_t*>(img + s * stride + off) = v; };
  put(0, digit_pair<0>(a, b));
  put(1, digit_pair<1>(a, b));
  put(2, digit_pair<2>(a, b));
  put(3, digit_pair<3>(a, b));
  put(4, digit_pair<4>(a, b));
  put(5, digit_pair<5>(a, b));
  put(6, digit_pair<6>(a, b));
  put(7, digit_pair<7>(a, b));
  put(8, digit_pair<8>(a, b));
}

// Ports of a row (two per lane) within 2^-3 and within 2^-9 of its largest, by exponent: bit l of
// the low word port 2 l, of the high word port 2 l + 1. Every port where the row is all zeros.
struct Masks {
  unsigned long long near, wide;
};
__device__ inline Masks port_masks(double v0, double v1, int E) {
  const int e0 = (int)exponent_of(v0), e1 = (int)exponent_of(v1);
  auto ports = [&](int j) {
    const int least = max(E - j, 1);
    return (unsigned long long)__ballot_sync(0xffffffffu, e0 >= least) |
           (unsigned long long)__ballot_sync(0xffffffffu, e1 >= least) << 32;
  };
  Masks m = {ports(3), ports(9)};
  if (E == 0 && !__any_sync(0xffffffffu, v0 != 0.0 || v1 != 0.0)) m = {~0ull, ~0ull};
  return m;
}

// sum_g acc_g 256^(8-g) 2^sc rounded to FP64; *ok = false where it is below the size that it is
// accurate at and not known to be (sure), or where the exponent leaves its range
__device__ inline double combine(const float* acc, int sc, bool sure, bool* ok) {
  int i[kDigits];
#pragma unroll
  for (int g = 0; g < kDigits; ++g)  // through the FP32 integer range where |acc| <= 2^22
    i[g] = g <= 4 ? __float_as_int(acc[g] + 12582912.0f) - 0x4b400000 : __float2int_rn(acc[g]);
  // pairs stay below 2^31: |i0| <= 2^18, |i2| <= 2^21, |i4| <= 2^22, |i6| <= 6 2^20
  const long long hi = (long long)(i[0] * 256 + i[1]) * 65536 + (i[2] * 256 + i[3]);
  const long long lo = (long long)(i[4] * 256 + i[5]) * 65536 + (i[6] * 256 + i[7]);
  const long long low = (long long)(unsigned)lo * 256 + i[8];
  constexpr unsigned long long kMask = (1ull << 40) - 1;
  long long t = hi + (lo >> 32) + (low >> 40);
  unsigned long long r = (unsigned long long)low & kMask;  // the value is t 2^40 + r
  const bool neg = t < 0;
  if (neg) {
    t = ~t + (r == 0);
    r = (0ull - r) & kMask;
  }
  if (!sure && t < (1ll << 22)) *ok = false;  // |sum| < 2^62: sum |X Y| may be below 2^126
  if (t == 0) {
    if (r == 0) return 0.0;
    t = (long long)r;
    r = 0;
    sc -= 40;
  }
  const int s = __clzll(t);
  unsigned long long x = (unsigned long long)t << s;
  x |= s >= 40 ? r << (s - 40) : r >> (40 - s);
  const unsigned long long m = (x >> 11) + ((x >> 10) & 1);
  const int e = 1023 + 103 - s + sc;
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
  Masks* mA = reinterpret_cast<Masks*>(tmem_slot + 2);  // [128] of the rows
  Masks* mB = mA + kTileP;                               // [2][48] of the columns, by turn parity
  int16_t* eA = reinterpret_cast<int16_t*>(mB + 2 * kCols);  // [128] row exponents
  int16_t* eB = eA + kTileP;                                 // [2][48] column exponents

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
  auto put_rows = [&](int64_t pt, int kc) {
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
      const Masks m = port_masks(hv[i].x, hv[i].y, E);
      if (lane == 0) {
        eA[r] = (int16_t)E;
        mA[r] = m;
      }
      put_digits(sA, kABytes, swz128(r, 2 * lane), digits(hv[i].x, E), digits(hv[i].y, E));
    }
  };
  // currents of the warp's columns (re or im of a system) of a column tile, same ports, loaded a
  // turn ahead
  double iv[kColsWarp][2];
  auto load_currents = [&](int64_t nt, int kc) {
    const int k = kc * kChunkK + 2 * lane;
#pragma unroll
    for (int i = 0; i < kColsWarp; ++i) {
      const int c = warp * kColsWarp + i;
      const int64_t s = nt * kSys + c / 2;
      iv[i][0] = iv[i][1] = 0.0;
      if (s < nsys) {
        const double* row = I + 2 * s * N + c % 2;
        if (k < N) iv[i][0] = row[2 * k];
        if (k + 1 < N) iv[i][1] = row[2 * k + 2];
      }
    }
  };
  auto put_currents = [&](int par) {
#pragma unroll
    for (int i = 0; i < kColsWarp; ++i) {
      const int c = warp * kColsWarp + i;
      const double v0 = iv[i][0], v1 = iv[i][1];
      const int E = (int)warp_max(max(exponent_of(v0), exponent_of(v1)));
      const Masks m = port_masks(v0, v1, E);
      if (lane == 0) {
        eB[par * kCols + c] = (int16_t)E;
        mB[par * kCols + c] = m;
      }
      put_digits(sB, kBBytes, swz128(c, 2 * lane), digits(v0, E), digits(v1, E));
    }
  };
  // field of the tile in tensor memory: lane = point, this warp's 12 columns; returns the systems
  // (bits) whose value is left to plain_sums
  constexpr int kWarpCols = kCols / 4;
  const int quarter = warp & 3, wc0 = (warp >> 2) * kWarpCols;
  double2* __restrict__ const out = static_cast<double2*>(a.B_out);
  auto epilogue = [&](int64_t pt, int64_t nt, int kc, int par) -> unsigned {
    const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16);
    const int row = quarter * 32 + lane;
    const int64_t p = pt * kTileP + row;
    const int Er = eA[row];
    const Masks mr = mA[row];
    unsigned left = 0;
#pragma unroll 1
    for (int c = wc0; c < wc0 + kWarpCols; c += 4) {
      float v[kDigits][4];
#pragma unroll
      for (int g = 0; g < kDigits; ++g)
        tmem_ld4(acc + (uint32_t)(g * kCols + c), v[g]);
      tmem_wait_ld();
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int64_t s = nt * kSys + c / 2 + q;
        bool ok = Er != 0x7ff;
        double b[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int col = par * kCols + c + 2 * q + h;
          const int Ec = eB[col];
          const Masks mc = mB[col];
          float y[kDigits];
#pragma unroll
          for (int g = 0; g < kDigits; ++g) y[g] = v[g][2 * q + h];
          if (Ec == 0x7ff) ok = false;
          // x = X 2^(E - 69) each, 256^8 per digit product: E + E' - 2 1023 - 138 + 64
          b[h] = combine(y, Er + Ec - 2120, ((mr.near & mc.wide) | (mr.wide & mc.near)) != 0ull, &ok);
        }
        if (p < P && s < nsys) {
          if (ok) {
            double2* dst = out + s * P + p;
            if (kc > 0) {
              const double2 o = *dst;
              b[0] += o.x;
              b[1] += o.y;
            }
            *dst = make_double2(b[0], b[1]);
          } else {
            left |= 1u << ((c - wc0) / 2 + q);
          }
        }
      }
    }
    return left;
  };
  // the values that epilogue left, in FP64: eight lanes an output
  auto plain_sums = [&](int64_t pt, int64_t nt, int kc, unsigned left) {
    if (!__any_sync(0xffffffffu, left != 0u)) return;
    const int k0 = kc * kChunkK, kn = min(N - k0, kChunkK), sub = lane & 7;
    int j = 0;  // system, and the rows left of it
    unsigned rows = __ballot_sync(0xffffffffu, left & 1u);
    while (true) {
      int row = -1, sys = 0;  // of this group: the (lane / 8)-th of the next four
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        while (rows == 0u && j + 1 < kWarpCols / 2) rows = __ballot_sync(0xffffffffu, (left >> ++j) & 1u);
        if (rows != 0u && q == (lane >> 3)) {
          row = __ffs(rows) - 1;
          sys = j;
        }
        rows &= rows - 1u;
      }
      if (!__any_sync(0xffffffffu, row >= 0)) break;
      const int64_t p = pt * kTileP + quarter * 32 + row, s = nt * kSys + wc0 / 2 + sys;
      const double* h = H + p * N + k0;
      const double2* in = reinterpret_cast<const double2*>(I) + s * N + k0;
      double hk[kChunkK / 8];
      double2 ik[kChunkK / 8];
#pragma unroll
      for (int k = 0; k < kChunkK / 8; ++k) {  // all loads in flight
        const bool in_row = row >= 0 && 8 * k + sub < kn;
        hk[k] = in_row ? h[8 * k + sub] : 0.0;
        ik[k] = in_row ? in[8 * k + sub] : make_double2(0.0, 0.0);
      }
      double2 b = make_double2(0.0, 0.0);
#pragma unroll
      for (int k = 0; k < kChunkK / 8; ++k) {
        b.x = fma(hk[k], ik[k].x, b.x);
        b.y = fma(hk[k], ik[k].y, b.y);
      }
      __syncwarp();
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        b.x += __shfl_xor_sync(0xffffffffu, b.x, o);
        b.y += __shfl_xor_sync(0xffffffffu, b.y, o);
      }
      if (row >= 0 && sub == 0) {
        double2* dst = out + s * P + p;
        if (kc > 0) {
          const double2 o = *dst;
          b.x += o.x;
          b.y += o.y;
        }
        *dst = b;
      }
    }
    __syncwarp();  // another lane adds the next chunk to these values
  };

  // A turn is one K chunk of one unit.
  int turn = 0, prev_kc = 0;
  int64_t last_pt = -1, prev_pt = 0, prev_nt = 0;
  bool alive = true;
  if (u_begin < u_end) load_currents(u_begin % nntile, 0);
  for (int64_t u = u_begin; u < u_end && alive; ++u) {
    const int64_t pt = u / nntile, nt = u - pt * nntile;
    for (int kc = 0; kc < nkc; ++kc, ++turn) {
      put_currents(turn & 1);
      unsigned left = 0;
      if (turn > 0) left = epilogue(prev_pt, prev_nt, prev_kc, (turn - 1) & 1);
      if (nkc > 1 || pt != last_pt) {
        __syncthreads();  // the epilogue has read the previous rows' exponents and masks
        put_rows(pt, kc);
        last_pt = pt;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncthreads();
      if (t == 0) {
        tc_fence_after();
        const int ksteps = min(kChunkK / 16, (N - kc * kChunkK + 15) / 16);
        const uint32_t aA = smem_u32(sA), aB = smem_u32(sB);
        // Digit i of the points with the digits of the columns that belong to the groups 0 .. 4 or
        // 5 .. 8, as one MMA of N = 240 or 192: the digits' images follow each other in shared
        // memory as rows of one operand, and so do the groups' accumulators in tensor memory
        // (14 MMAs a K step instead of 45 of N = 48). The images before digit 0 are zeros. MMAs
        // are only sure to run in order on one accumulator and in one shape, so the two windows
        // are fixed.
        for (int kk = 0; kk < ksteps; ++kk)
          for (int g = 0; g < kDigits; g += kWin) {
            const int n = min(kWin, kDigits - g);
            for (int i = 0; i < g + n; ++i)
              mma_bf16(tmem + g * kCols, make_desc(aA + i * kABytes) + (uint64_t)(kk * 2),
                       make_desc(aB + g * kBBytes - i * kBBytes) + (uint64_t)(kk * 2),
                       (i > 0 || kk > 0) ? 1u : 0u, idesc_groups(n));
          }
        mma_commit(bar);
      }
      // while the MMAs run: the next turn's currents, the plain sums of the previous tile
      if (kc + 1 < nkc) load_currents(nt, kc + 1);
      else if (u + 1 < u_end) load_currents((u + 1) % nntile, 0);
      plain_sums(prev_pt, prev_nt, prev_kc, left);
      prev_pt = pt;
      prev_nt = nt;
      prev_kc = kc;
      if (!mbar_wait(bar, (uint32_t)turn & 1u, err, 7)) alive = false;
      alive = __syncthreads_and(alive) != 0;
      tc_fence_after();
      if (!alive) break;
    }
  }
  if (turn > 0 && alive) plain_sums(prev_pt, prev_nt, prev_kc, epilogue(prev_pt, prev_nt, prev_kc, (turn - 1) & 1));
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

constexpr size_t kSmem = 1024 + kDigits * (size_t)kABytes + (kDigits + kWin - 1) * (size_t)kBBytes + 16 +
                         (sizeof(Masks) + sizeof(int16_t)) * (kTileP + 2 * kCols);
static_assert(kSmem <= 232448, "227 KB a CTA");

}  // namespace oz

// Units of the FP64 tensor-core superposition, or 0 where the SIMT kernel is the faster one.
// Measured cycles of the busiest SM: a tile of 128 x 24 (point, system) pairs takes kTile + kPort
// per port of the chunk, whatever part of it exists (15,300 at 8 ports, 16,900 at 32 and 19,800 at
// 64, and up to a tenth more where values are left to plain sums), and kChunk for every full chunk
// before (its rows are cut anew each time: 90,000 for three chunks of 64); the SIMT kernel takes
// 1 + 1.1 N per pair (N = 4: 14,100 for as many pairs).
int64_t superpose_fp64_tc_units(int64_t N, int64_t P, int64_t nsys, int sms) {
  constexpr double kTile = 16200.0, kPort = 80.0, kChunk = 34000.0;
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

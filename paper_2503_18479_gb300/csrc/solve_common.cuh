// solve_common.cuh -- device helpers shared by the FP64 and mixed-precision solve kernels.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"

namespace mts {


// ---------------------------------------------------------------------------------------
// small helpers
// ---------------------------------------------------------------------------------------
struct cd {
  double x, y;
};
__device__ inline cd cmul(cd a, cd b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
__device__ inline double cabs2(cd a) { return a.x * a.x + a.y * a.y; }

// Objective term of one loss point and its cotangent G = de/dRe b + j de/dIm b.
__device__ inline double point_loss(int mode, cd b, const double* t, cd* G) {
  if (mode == 0) {
    double a = sqrt(b.x * b.x + b.y * b.y);
    double r = a - t[0];
    if (a > 0.0) {
      G->x = 2.0 * r * b.x / a;
      G->y = 2.0 * r * b.y / a;
    } else {
      G->x = 0.0;
      G->y = 0.0;
    }
    return r * r;
  }
  cd e = {b.x - t[0], b.y - t[1]};
  G->x = 2.0 * e.x;
  G->y = 2.0 * e.y;
  return e.x * e.x + e.y * e.y;
}

// arg-max of (key, idx) over aligned groups of `width` lanes (width a power of 2 <= 32);
// ties go to the smaller index.
__device__ inline void argmax_shfl(float& key, int& idx, int width) {
  for (int off = width >> 1; off > 0; off >>= 1) {
    float k2 = __shfl_xor_sync(0xffffffffu, key, off, width);
    int i2 = __shfl_xor_sync(0xffffffffu, idx, off, width);
    if (k2 > key || (k2 == key && i2 < idx)) {
      key = k2;
      idx = i2;
    }
  }
}
__device__ inline void argmax_shfl_d(double& key, int& idx, int width) {
  for (int off = width >> 1; off > 0; off >>= 1) {
    double k2 = __shfl_xor_sync(0xffffffffu, key, off, width);
    int i2 = __shfl_xor_sync(0xffffffffu, idx, off, width);
    if (k2 > key || (k2 == key && i2 < idx)) {
      key = k2;
      idx = i2;
    }
  }
}

// ---------------------------------------------------------------------------------------
// Double-float values (h + l, |l| <= ulp(h) / 2 after df_norm; about 2^-46 relative) on the FP32
// and integer pipes. An FP64 instruction of a warp, conversions included, holds the FP64 pipe
// for 16 cycles here, the issue slots of 64 FP32 instructions.
// ---------------------------------------------------------------------------------------
struct df {
  float h, l;
};
__device__ __forceinline__ df df_norm(float h, float l) {  // |h| >= |l| or h = 0
  const float s = __fadd_rn(h, l);
  return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
// a += b (+ bl), unnormalised low part
__device__ __forceinline__ void df_acc(df& a, float b, float bl) {
  const float s = __fadd_rn(a.h, b), z = __fsub_rn(s, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, z)), __fsub_rn(b, z));
  a.h = s;
  a.l = __fadd_rn(a.l, __fadd_rn(e, bl));
}
__device__ __forceinline__ df df_mul(df a, df b) {
  const float p = __fmul_rn(a.h, b.h);
  return {p, fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p)))};
}
__device__ __forceinline__ df df_mulf(df a, float b) {
  const float p = __fmul_rn(a.h, b);
  return {p, fmaf(a.l, b, fmaf(a.h, b, -p))};
}
// the mantissa of a normal FP64 value as a pair in [1, 2) with the value's sign, and its
// exponent; (0, 0) for zero and subnormal values, the value itself for infinities and NaN
__device__ __forceinline__ df df_mantissa(double v, int* exponent) {
  const int hi = __double2hiint(v);
  const unsigned lo = (unsigned)__double2loint(v);
  const int e = (hi >> 20) & 0x7ff;
  if (e == 0) {
    *exponent = 0;
    return {0.0f, 0.0f};
  }
  if (e == 0x7ff) {
    *exponent = 0;
    return {(float)v, 0.0f};
  }
  *exponent = e - 1023;
  const float h = __int_as_float((hi & 0x80000000) | 0x3f800000 | ((hi & 0xfffff) << 3) | (int)(lo >> 29));
  const float l = __uint2float_rn(lo & 0x1fffffffu) * 0x1p-52f;
  return df_norm(h, hi < 0 ? -l : l);
}
__device__ __forceinline__ df df_from(double v) {
  const int hi = __double2hiint(v);
  const unsigned lo = (unsigned)__double2loint(v);
  const int e = (hi >> 20) & 0x7ff;
  if ((unsigned)(e - 897) > 253u) {  // zero, or outside the normal FP32 range
    if (((unsigned)(hi << 1) | lo) == 0u) return {0.0f, 0.0f};
    const float h = (float)v;
    return {h, isfinite(h) ? (float)(v - (double)h) : 0.0f};
  }
  const float h = __int_as_float((hi & 0x80000000) | ((e - 896) << 23) | ((hi & 0xfffff) << 3) | (int)(lo >> 29));
  // the low 29 bits times 2^(e - 1075), by the exponent field (0 where that underflows)
  const int b = __float_as_int(__uint2float_rn(lo & 0x1fffffffu));
  const float l = (b >> 23) + e - 1075 > 0 ? __int_as_float(b + (e - 1075) * (1 << 23)) : 0.0f;
  return df_norm(h, hi < 0 ? -l : l);
}
// the pair as FP64 (round to nearest of the pair's own bits), from its bits where h is an
// ordinary FP32 value
__device__ __forceinline__ double df_double(df a) {
  if (!isfinite(a.h)) return (double)a.h;
  a = df_norm(a.h, a.l);
  const int hb = __float_as_int(a.h), lb = __float_as_int(a.l);
  const int e = (hb >> 23) & 255;
  if (e == 0 || e == 255) return (double)a.h + (double)a.l;
  // l in units of the last FP64 bit of h's binade: at most 2^28
  const int el = ((lb >> 23) & 255) + 179 - e;
  int li = el > 0 && (lb & 0x7f800000) != 0 ? __float2int_rn(__int_as_float(lb + (179 - e) * (1 << 23))) : 0;
  if (hb < 0) li = -li;
  long long m = ((long long)((hb & 0x7fffff) | 0x800000) << 29) + li;
  const int down = m < (1ll << 52);  // h a power of two and l of the other sign
  m <<= down;
  const unsigned long long bits = ((unsigned long long)(unsigned)(hb & 0x80000000) << 32) |
                                  ((unsigned long long)(e + 896 - down) << 52) |
                                  ((unsigned long long)m & 0xfffffffffffffull);
  return __longlong_as_double((long long)bits);
}
// y = 1 / (w c)
__device__ __forceinline__ df df_recip_product(double w, double c) {
  int ew, ec;
  const df m = df_mul(df_mantissa(w, &ew), df_mantissa(c, &ec));
  float q;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(m.h));
  // one Newton step on the exact remainder: q (1 + r), r = 1 - q m of about 2^-23
  const float r = q == 0.0f ? 0.0f : fmaf(-q, m.l, fmaf(-q, m.h, 1.0f));  // w c infinite: 0
  const df y = df_norm(q, fmaf(q, r, q * r * r));
  const int e = -(ew + ec);  // |e| <= 2046: two factors cover the FP32 range and saturate
  const int e1 = min(max(e, -126), 127), e2 = min(max(e - e1, -126), 127);
  const float s1 = __int_as_float((e1 + 127) << 23), s2 = __int_as_float((e2 + 127) << 23);
  return {y.h * s1 * s2, y.l * s1 * s2};
}

// n / d of non-negative n and positive d, in 32 bits where both fit (the 64-bit division is a
// sequence of about a hundred instructions)
__device__ __forceinline__ int64_t div_i64(int64_t n, int64_t d) {
  if (((n | d) >> 32) == 0) return (int64_t)((uint32_t)n / (uint32_t)d);
  return n / d;
}

// System of launch index li: li itself, or configuration li / gcount at the frequency
// glist[li % gcount] of the launch's port class.
__device__ inline int64_t launch_sys(const SolveArgs& a, int64_t li) {
  if (a.glist == nullptr) return li;
  const int64_t b = div_i64(li, a.gcount);
  return b * a.n_freq + a.glist[li - b * a.gcount];
}

// Locate system `sys` (= b * n_freq + g).
struct SysInfo {
  int64_t b;
  int g, s, f, N, k0;
  double w;
};
__device__ inline SysInfo sys_info(const SolveArgs& a, int64_t sys) {
  SysInfo si;
  si.b = div_i64(sys, a.n_freq);
  si.g = (int)(sys - si.b * a.n_freq);
  si.s = a.t.freq_struct[si.g];
  si.f = si.g - a.freq_off[si.s];
  si.k0 = a.port_off[si.s];
  si.N = a.port_off[si.s + 1] - si.k0;
  si.w = a.omega[si.g];
  return si;
}

}  // namespace mts

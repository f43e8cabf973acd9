// Accumulators and loads of the batched GEMVs (step_gemv.cu) and of the truncated apply (step_band.cu).
#pragma once
#include <cuda_runtime.h>

#include "ff_convert.h"

namespace lem {

static __device__ __forceinline__ void two_sum_d(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// A propagator's place in L2: of ordinary priority, so that it outlives what passes through and is there
// in the next step, or passing through. (A priority above the ordinary would outlast the steps.)
static __device__ __forceinline__ unsigned long long l2_policy(bool keep) {
  unsigned long long policy;
  if (keep) asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(policy));
  else asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  return policy;
}
static __device__ __forceinline__ int4 load_policy(const int4* p, unsigned long long policy) {
  int4 v;
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.s32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p), "l"(policy));
  return v;
}

// Two FP32 values in one register pair: Blackwell's packed FP32 arithmetic issues one instruction for
// both, and the float-float sums below are bound by issue slots, not by the FP32 lanes.
typedef unsigned long long f32x2;
static __device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
static __device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
static __device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
static __device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
static __device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
static __device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// a + b = s + e exactly, in both halves
static __device__ __forceinline__ void two_sum2(f32x2 a, f32x2 b, f32x2& s, f32x2& e) {
  s = add2(a, b);
  const f32x2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// Per-lane accumulators of one 16-byte chunk of a row after another. FP64 rows: fused multiply-add.
// FP32 rows: each product split exactly (FMA) and accumulated in float-float, even and odd elements
// in one packed pair of sums.
struct AccD {
  double s = 0.0;
  __device__ __forceinline__ void add(double a, double b) { s = fma(a, b, s); }
  __device__ __forceinline__ void chunk(const double* p, const double* w) {
    add(p[0], w[0]);
    add(p[1], w[1]);
  }
};
struct AccF {
  f32x2 hi = 0, lo = 0;
  __device__ __forceinline__ void add2p(f32x2 a, f32x2 b) {
    const f32x2 p = mul2(a, b), pe = fma2(a, b, p ^ 0x8000000080000000ull);
    f32x2 s, e;
    two_sum2(hi, p, s, e);
    hi = s;
    lo = add2(lo, add2(e, pe));
  }
  __device__ __forceinline__ void add(float a, float b) { add2p(pack2(a, 0.0f), pack2(b, 0.0f)); }
  __device__ __forceinline__ void chunk(const float* p, const float* w) {
    add2p(pack2(p[0], p[1]), pack2(w[0], w[1]));
    add2p(pack2(p[2], p[3]), pack2(w[2], w[3]));
  }
};
// Zeros in place of what a row's last chunk holds past its end (left: values of the row from the chunk on).
static __device__ __forceinline__ void row_end(int4& q, const float*, int left) {
  if (left < 4) {
    q.w = 0;
    if (left < 3) q.z = 0;
    if (left < 2) q.y = 0;
  }
}
static __device__ __forceinline__ void row_end(int4& q, const double*, int left) {
  if (left < 2) q.z = q.w = 0;
}

// Reduction over the 8 lanes of a row group (lanes 8g .. 8g + 7).
static __device__ __forceinline__ double group_reduce(AccD& a) {
  for (int o = 4; o > 0; o >>= 1) a.s += __shfl_xor_sync(0xffffffffu, a.s, o);
  return a.s;
}
static __device__ __forceinline__ double group_reduce(AccF& a) {
  float h0, h1, l0, l1, hi, e;
  unpack2(a.hi, h0, h1);
  unpack2(a.lo, l0, l1);
  two_sum_d(h0, h1, hi, e);
  float lo = __fadd_rn(__fadd_rn(l0, l1), e);
  for (int o = 4; o > 0; o >>= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, hi, o);
    const float ol = __shfl_xor_sync(0xffffffffu, lo, o);
    float s;
    two_sum_d(hi, oh, s, e);
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(ol, e));
  }
  return f32_to_f64(hi) + f32_to_f64(lo);
}
// Complex rows: the sums of the real and the imaginary part. FP32: one packed pair of float-float sums.
struct AccCD {
  double re = 0.0, im = 0.0;
  __device__ __forceinline__ void add(double pa, double pb, double wr, double wi) {
    re = fma(pa, wr, re);
    re = fma(-pb, wi, re);
    im = fma(pb, wr, im);
    im = fma(pa, wi, im);
  }
  // one 16-byte chunk of a row pair (pa: real parts, pb: imaginary parts) against the window's parts
  __device__ __forceinline__ void chunk(const double* pa, const double* pb, const double* wr, const double* wi) {
    add(pa[0], pb[0], wr[0], wi[0]);
    add(pa[1], pb[1], wr[1], wi[1]);
  }
};
struct AccCF {
  f32x2 hi = 0, lo = 0;  // (real, imaginary)
  __device__ __forceinline__ void add_exact(f32x2 a, f32x2 b) {
    const f32x2 p = mul2(a, b), pe = fma2(a, b, p ^ 0x8000000080000000ull);
    f32x2 s, e;
    two_sum2(hi, p, s, e);
    hi = s;
    lo = add2(lo, add2(e, pe));
  }
  __device__ __forceinline__ void add(float pa, float pb, float wr, float wi) {
    add_exact(pack2(pa, pb), pack2(wr, wr));
    add_exact(pack2(-pb, pa), pack2(wi, wi));
  }
  // the chunk's eight products per part are summed by FMA in FP32 and the chunk sum enters the
  // float-float accumulator (an exact product split for each of the four products an element takes
  // part in would make the launch ALU-bound)
  __device__ __forceinline__ void chunk(const float* pa, const float* pb, const float* wr, const float* wi) {
    float sr = 0.0f, si = 0.0f;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      sr = fmaf(pa[h], wr[h], sr);
      sr = fmaf(-pb[h], wi[h], sr);
      si = fmaf(pb[h], wr[h], si);
      si = fmaf(pa[h], wi[h], si);
    }
    f32x2 s, e;
    two_sum2(hi, pack2(sr, si), s, e);
    hi = s;
    lo = add2(lo, e);
  }
};
static __device__ __forceinline__ void group_reduce(AccCD& a, double& re, double& im) {
  for (int o = 4; o > 0; o >>= 1) {
    a.re += __shfl_xor_sync(0xffffffffu, a.re, o);
    a.im += __shfl_xor_sync(0xffffffffu, a.im, o);
  }
  re = a.re;
  im = a.im;
}
static __device__ __forceinline__ void group_reduce(AccCF& a, double& re, double& im) {
  for (int o = 4; o > 0; o >>= 1) {
    const f32x2 oh = __shfl_xor_sync(0xffffffffu, a.hi, o), ol = __shfl_xor_sync(0xffffffffu, a.lo, o);
    f32x2 s, e;
    two_sum2(a.hi, oh, s, e);
    a.hi = s;
    a.lo = add2(a.lo, add2(ol, e));
  }
  float hr, hi, lr, li;
  unpack2(a.hi, hr, hi);
  unpack2(a.lo, lr, li);
  re = f32_to_f64(hr) + f32_to_f64(lr);
  im = f32_to_f64(hi) + f32_to_f64(li);
}

// a double rounded to the propagator's precision; to FP32 with integer operations (GB300 converts on
// the FP64 pipe, 2 a clock and SM, and warps that stage windows of their own repeat the work)
static __device__ __forceinline__ void to_prec(double v, double& w) { w = v; }
static __device__ __forceinline__ void to_prec(double v, float& w) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v));
  const unsigned mag_hi = static_cast<unsigned>(b >> 32) & 0x7FFFFFFFu, lo = static_cast<unsigned>(b);
  const int e = static_cast<int>(mag_hi >> 20) - 1023 + 127;
  const unsigned m = (mag_hi << 3) | (lo >> 29);  // its low 23 bits: the float's mantissa, cut
  const unsigned rest = lo & 0x1FFFFFFFu;
  const unsigned up = rest > 0x10000000u || (rest == 0x10000000u && (m & 1u)) ? 1u : 0u;
  const unsigned f = (static_cast<unsigned>(e) << 23) | (m & 0x7FFFFFu);
  const bool fast = e >= 1 && e <= 253;
  w = fast ? __uint_as_float((f + up) | (static_cast<unsigned>(b >> 32) & 0x80000000u)) : static_cast<float>(v);
}

}  // namespace lem

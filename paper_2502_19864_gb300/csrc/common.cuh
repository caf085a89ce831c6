// common.cuh -- device helpers shared by the libringada kernels (sm_103a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ra {

typedef __nv_bfloat16 bf16;

// ---- element conversions --------------------------------------------------------------
__device__ __forceinline__ float to_f(float x) { return x; }
__device__ __forceinline__ float to_f(bf16 x) { return __bfloat162float(x); }
template <typename T> __device__ __forceinline__ T from_f(float x);
template <> __device__ __forceinline__ float from_f<float>(float x) { return x; }
template <> __device__ __forceinline__ bf16 from_f<bf16>(float x) { return __float2bfloat16_rn(x); }

// ---- reductions ------------------------------------------------------------------------
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// ---- GELU (sigma of Eq. 1, exact erf form) --------------------------------------------
// erf by Abramowitz & Stegun, Handbook of Mathematical Functions, formula 7.1.28:
//   erf(x) = 1 - (1 + a1 x + ... + a6 x^6)^-16 for x >= 0, odd extension, |error| <= 3e-7.
// Evaluated without cancellation: with e = p - 1 carried exactly through the four squarings
// (p^2k - 1 = e (2 + e)), erf = e16 / (1 + e16); x is clamped at 5, where erf is 1 in fp32.
// Branch-free with one reciprocal.  Evaluated by the adapters and the fp32 kernels.
__device__ __forceinline__ float erf_as7128(float x) {
  const float t = fminf(fabsf(x), 5.0f);
  float p = fmaf(t, 4.30638e-5f, 2.765672e-4f);
  p = fmaf(t, p, 1.520143e-4f);
  p = fmaf(t, p, 9.2705272e-3f);
  p = fmaf(t, p, 4.22820123e-2f);
  float e = __fmul_rn(t, fmaf(t, p, 7.05230784e-2f));  // p - 1
  e = __fmul_rn(e, __fadd_rn(e, 2.0f));  // p^2 - 1
  e = __fmul_rn(e, __fadd_rn(e, 2.0f));  // p^4 - 1
  e = __fmul_rn(e, __fadd_rn(e, 2.0f));  // p^8 - 1
  e = __fmul_rn(e, __fadd_rn(e, 2.0f));  // p^16 - 1
  return copysignf(__fdividef(e, __fadd_rn(e, 1.0f)), x);
}
// GELU(x) = x Phi(x) = h + h erf(x / sqrt 2) with h = x / 2
__device__ __forceinline__ float gelu_f(float x) {
  const float h = __fmul_rn(x, 0.5f);
  return __fmaf_rn(h, erf_as7128(__fmul_rn(x, 0.70710678118654752f)), h);
}
// d/dx GELU = Phi(x) + x phi(x)
__device__ __forceinline__ float gelu_grad_f(float x) {
  const float Phi = __fmaf_rn(erf_as7128(__fmul_rn(x, 0.70710678118654752f)), 0.5f, 0.5f);
  const float q = __fmul_rn(__fmul_rn(x, -0.5f), x);
  return __fadd_rn(Phi, __fmul_rn(__fmul_rn(x, __expf(q)), 0.39894228040143268f));
}

// ---- packed forms: two values per instruction with the sm_100 fp32x2 arithmetic --------
__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }
// 2^x on the special function unit (ex2.approx): about 2 ulp, results below 2^-126 flushed to
// zero -- the softmax probabilities it serves are rounded to bf16, and one below 2^-126
// contributes nothing
__device__ __forceinline__ float ex2_fast(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// the same with results below 2^-126 (a scaling on either side of the exponential)
__device__ __forceinline__ float ex2_subnormal(float x) {
  float y;
  asm("ex2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// GELU and GELU' of the GEMM epilogues, which evaluate them for every element of a large tile and
// are paced by it.  Phi(-|x|) in the form of Abramowitz & Stegun 7.1.26,
//   Phi(-|x|) = (b1 r + ... + b5 r^5) exp(-x^2 / 2), r = 1 / (1 + c |x|):
// one reciprocal and one exponential per element (which GELU' needs anyway) and 14 multiply-adds, where
// 7.1.28 and its four squarings took 25.  c and b are fitted for the least largest error, 5.9e-8; the published
// ones give 7.5e-8, and as they are larger and of both signs they lose more to rounding near 0.  Largest (rms)
// error against 64 bits over [-12, 12]: GELU 3.8e-7 (0.7e-7), by 7.1.28 8.8e-7 (1.7e-7); GELU' 2.3e-7
// (0.3e-7), by 7.1.28 2.8e-7 (0.6e-7).  Both leave the epilogue in bf16.
__device__ __forceinline__ float rcp_fast(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Phi(x) up to its sign (1 - Phi(-x) for x >= 0, -Phi(x) below), and e = exp(-x^2 / 2)
__device__ __forceinline__ float2 normal_cdf2(float2 x, float2& e) {
  const float2 r = make_float2(rcp_fast(__fmaf_rn(fabsf(x.x), 0.3308f, 1.0f)), rcp_fast(__fmaf_rn(fabsf(x.y), 0.3308f, 1.0f)));
  float2 p = __ffma2_rn(r, f2(0.110379077f), f2(-0.375332892f));
  p = __ffma2_rn(r, p, f2(0.0914756581f));
  p = __ffma2_rn(r, p, f2(-0.204449788f));
  p = __ffma2_rn(r, p, f2(-0.122071989f));
  p = __fmul2_rn(p, r);  // minus the polynomial
  const float2 z = __fmul2_rn(__fmul2_rn(x, f2(-0.72134752044448170f)), x);  // -x^2 / 2 in powers of two
  e = make_float2(ex2_fast(z.x), ex2_fast(z.y));
  return __ffma2_rn(p, e, make_float2(x.x < 0.f ? 0.f : 1.f, x.y < 0.f ? 0.f : 1.f));
}
__device__ __forceinline__ float2 gelu2(float2 x) {
  float2 e;
  const float2 Phi = normal_cdf2(x, e);
  return make_float2(__fmul_rn(x.x, fabsf(Phi.x)), __fmul_rn(x.y, fabsf(Phi.y)));
}
// GELU(x) and GELU'(x) = Phi(x) + x phi(x) together
__device__ __forceinline__ void gelu_both2(float2 x, float2& y, float2& dy) {
  float2 e;
  const float2 Phi = normal_cdf2(x, e), d = __fmul2_rn(__fmul2_rn(x, f2(0.39894228040143268f)), e);
  y = make_float2(__fmul_rn(x.x, fabsf(Phi.x)), __fmul_rn(x.y, fabsf(Phi.y)));
  dy = make_float2(__fadd_rn(d.x, fabsf(Phi.x)), __fadd_rn(d.y, fabsf(Phi.y)));
}
// SiLU and its derivative with the special-function exponential and the fast division (a few
// ulp; they run per element in the SwiGLU epilogues).  For x below about -88 the denominator
// overflows and the sigmoid is 0, its limit.
__device__ __forceinline__ float silu_f(float x) { return __fdividef(x, 1.0f + __expf(-x)); }
__device__ __forceinline__ float silu_grad_f(float x) {
  const float s = __fdividef(1.0f, 1.0f + __expf(-x));
  return s * (1.0f + x * (1.0f - s));
}

// ---- RoPE ---------------------------------------------------------------------------------
// inverse frequency of rotate-half pair i of a head of dh dims: theta^(-2 i / dh); the angle
// at position s is s times this (every RoPE kernel evaluates it this way)
__device__ __forceinline__ float rope_freq(int i, int dh, float theta) {
  return expf(-logf(theta) * (2.0f * (float)i / (float)dh));
}

// ---- programmatic dependent launch ----------------------------------------------------
// A kernel started with launch_pdl may begin while the kernel before it in the stream is
// still finishing.  pdl_wait() blocks until that kernel has completed and its writes are
// visible; it precedes every access to memory that earlier kernels write or read.
// pdl_trigger() lets the next kernel of the stream be scheduled (its CTAs then wait in their
// own pdl_wait).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- error word written by kernels whose bounded waits ran out -------------------------
// Bit 0: a wait timed out.  The host reads and clears it in ra_sync_status.
enum : unsigned { RA_DEVERR_TIMEOUT = 1u, RA_DEVERR_BOUNDS = 2u };

__device__ __forceinline__ void set_dev_error(unsigned* flag, unsigned bits) {
  if (flag) atomicOr(flag, bits);
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Upper bound for any single in-kernel wait: far above the longest legitimate wait
// (one tile's main loop, microseconds), short enough that a broken pipeline ends.
constexpr uint64_t kWaitLimitNs = 2000000000ull;

}  // namespace ra

// simt.cuh -- operand copies shared by the CUDA-core kernels (fp32 arithmetic).
#pragma once

#include "common.cuh"

namespace ra {

// four consecutive elements in shared memory or global memory (16- or 8-byte aligned) as floats
__device__ __forceinline__ float4 ld4s(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4s(const bf16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}

// A warp's operand ring: blocks of a few k are copied ahead into shared memory, by cp.async where the
// rows allow 16-byte copies, by plain loads and stores else; the reader waits for the group (cp_wait)
// and for the other lanes (__syncwarp).
__device__ __forceinline__ void cp16(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
// nr x nc block of a row-major matrix (row stride ld, nc a multiple of 4) at src into dst (row stride
// ldd): entry (r, c) is taken where r < vr and c < vc and zero elsewhere.  All lanes of a warp.
template <typename T>
__device__ __forceinline__ void copy_block(T* dst, int ldd, const T* src, size_t ld, int nr, int nc, int vr, int vc,
                                           bool vec, int lane) {
  constexpr int E = 16 / sizeof(T);
  if (vec) {
    const int per = nc / E;
    for (int e = lane; e < nr * per; e += 32) {
      const int r = e / per, c = (e % per) * E;
      const bool ok = r < vr && c < vc;
      cp16(dst + r * ldd + c, src + (ok ? r * ld + c : 0), ok);
    }
  } else {
    for (int e = lane; e < nr * nc; e += 32) {
      const int r = e / nc, c = e % nc;
      dst[r * ldd + c] = r < vr && c < vc ? src[r * ld + c] : from_f<T>(0.f);
    }
  }
}

}  // namespace ra

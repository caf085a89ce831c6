// k_gemm_simt.cu -- CUDA-core GEMM with the step's fused epilogues.
//
// C[M, N] = A[M, K] B[N, K]^T, fp32 accumulation.  This is the path of the fp32 model
// (tcgen05 has no fp32-in/fp32-accurate mode: tf32 keeps 10 mantissa bits, which cannot
// meet a 1e-4 relative bar) and of shapes the tensor-core kernel does not take.
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "simt.cuh"
#include "tcgen05.cuh"

namespace ra {
namespace {

// 32 x 32 output tiles; the 8 warps of a CTA split K
constexpr int BT = 32, NW = 8, NT = NW * 32, KC = 8, NS = 3, LDP = BT + 8;

template <typename T>
__device__ __forceinline__ float ld(const void* p, int64_t i) {
  return to_f(reinterpret_cast<const T*>(p)[i]);
}
__device__ __forceinline__ float ld_dt(const void* p, int dt, int64_t i) {
  return dt == DT_BF16 ? ld<bf16>(p, i) : ld<float>(p, i);
}
__device__ __forceinline__ void st_dt(void* p, int dt, int64_t i, float v) {
  if (dt == DT_BF16) reinterpret_cast<bf16*>(p)[i] = __float2bfloat16_rn(v);
  else reinterpret_cast<float*>(p)[i] = v;
}

// packed gate/up layout: 64-column blocks alternate gate, up
__device__ __forceinline__ int64_t gate_col(int j) { return (int64_t)(j >> 6) * 128 + (j & 63); }

__device__ __forceinline__ void epilogue(const GemmArgs& g, int m, int n, float acc) {
  switch (g.epi) {
    case EPI_STORE:
    case EPI_SWIGLU: {
      if (g.bias) acc += g.bias[n];
      st_dt(g.C, g.c_dtype, (int64_t)m * g.ldc + n, acc);
    } break;
    case EPI_BIAS_GELU: {
      float u = acc + (g.bias ? g.bias[n] : 0.f);
      if (g.C) st_dt(g.C, g.c_dtype, (int64_t)m * g.ldc + n, u);
      st_dt(g.C2, g.c2_dtype, (int64_t)m * g.ldc2 + n, gelu_f(u));
    } break;
    case EPI_BIAS_GELU_G: {
      float u = acc + (g.bias ? g.bias[n] : 0.f);
      if (g.C) st_dt(g.C, g.c_dtype, (int64_t)m * g.ldc + n, gelu_grad_f(u));
      st_dt(g.C2, g.c2_dtype, (int64_t)m * g.ldc2 + n, gelu_f(u));
    } break;
    case EPI_MUL: {
      float f = ld_dt(g.aux, g.aux_dtype, (int64_t)m * g.ldaux + n);
      st_dt(g.C, g.c_dtype, (int64_t)m * g.ldc + n, acc * f);
    } break;
    case EPI_RESID: {
      float r = ld_dt(g.aux, g.aux_dtype, (int64_t)m * g.ldaux + n);
      st_dt(g.C, g.c_dtype, (int64_t)m * g.ldc + n, acc + r);
    } break;
    case EPI_DSWIGLU: {
      int64_t gc = gate_col(n), uc = gc + 64;
      float gt = ld_dt(g.aux, g.aux_dtype, (int64_t)m * g.ldaux + gc);
      float up = ld_dt(g.aux, g.aux_dtype, (int64_t)m * g.ldaux + uc);
      st_dt(g.C, g.c_dtype, (int64_t)m * g.ldc + gc, acc * up * silu_grad_f(gt));
      st_dt(g.C, g.c_dtype, (int64_t)m * g.ldc + uc, acc * silu_f(gt));
    } break;
  }
}

// four consecutive values of a row (n a multiple of 4, `vec`: 16-byte (f32) or 8-byte (bf16) accesses)
__device__ __forceinline__ float4 ld4_dt(const void* p, int dt, int64_t i, bool vec) {
  if (!vec) return make_float4(ld_dt(p, dt, i), ld_dt(p, dt, i + 1), ld_dt(p, dt, i + 2), ld_dt(p, dt, i + 3));
  if (dt == DT_F32) return *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(p) + i);
  return ld4s(reinterpret_cast<const bf16*>(p) + i);
}
__device__ __forceinline__ void st4_dt(void* p, int dt, int64_t i, bool vec, float4 v) {
  if (!vec) {
    st_dt(p, dt, i, v.x); st_dt(p, dt, i + 1, v.y); st_dt(p, dt, i + 2, v.z); st_dt(p, dt, i + 3, v.w);
  } else if (dt == DT_F32) {
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(p) + i) = v;
  } else {
    __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2*>(reinterpret_cast<bf16*>(p) + i) = make_uint2(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b));
  }
}
// the epilogue of columns n .. n + 3, all below N
__device__ __forceinline__ void epilogue4(const GemmArgs& g, int m, int n, float4 u, bool vec) {
  const int64_t c = (int64_t)m * g.ldc + n;
  if (g.bias && g.epi != EPI_MUL && g.epi != EPI_RESID && g.epi != EPI_DSWIGLU) {
    u.x += g.bias[n]; u.y += g.bias[n + 1]; u.z += g.bias[n + 2]; u.w += g.bias[n + 3];
  }
  if (g.epi == EPI_BIAS_GELU || g.epi == EPI_BIAS_GELU_G) {
    if (g.C)
      st4_dt(g.C, g.c_dtype, c, vec,
             g.epi == EPI_BIAS_GELU ? u : make_float4(gelu_grad_f(u.x), gelu_grad_f(u.y), gelu_grad_f(u.z), gelu_grad_f(u.w)));
    st4_dt(g.C2, g.c2_dtype, (int64_t)m * g.ldc2 + n, vec, make_float4(gelu_f(u.x), gelu_f(u.y), gelu_f(u.z), gelu_f(u.w)));
    return;
  }
  if (g.epi == EPI_DSWIGLU) {
    const int64_t gc = gate_col(n), ax = (int64_t)m * g.ldaux + gc, cc = (int64_t)m * g.ldc + gc;
    const float4 gt = ld4_dt(g.aux, g.aux_dtype, ax, vec), up = ld4_dt(g.aux, g.aux_dtype, ax + 64, vec);
    st4_dt(g.C, g.c_dtype, cc, vec, make_float4(u.x * up.x * silu_grad_f(gt.x), u.y * up.y * silu_grad_f(gt.y),
                                                u.z * up.z * silu_grad_f(gt.z), u.w * up.w * silu_grad_f(gt.w)));
    st4_dt(g.C, g.c_dtype, cc + 64, vec, make_float4(u.x * silu_f(gt.x), u.y * silu_f(gt.y), u.z * silu_f(gt.z), u.w * silu_f(gt.w)));
    return;
  }
  if (g.epi == EPI_MUL || g.epi == EPI_RESID) {
    const float4 f = ld4_dt(g.aux, g.aux_dtype, (int64_t)m * g.ldaux + n, vec);
    u = g.epi == EPI_MUL ? make_float4(u.x * f.x, u.y * f.y, u.z * f.z, u.w * f.w)
                         : make_float4(u.x + f.x, u.y + f.y, u.z + f.z, u.w + f.w);
  }
  st4_dt(g.C, g.c_dtype, c, vec, u);
}

// The warps' tiles of a CTA (those with a share of K) take the place of their rings, are summed in warp
// order and go through the epilogue.  SPLIT = 2: the two CTAs of a cluster have a half of K each; each
// sends the other its sums of 16 rows and finishes the other 16.
template <bool KN, int SPLIT>
__device__ __forceinline__ void finish(const GemmArgs& g, int ks, bool vc, bool have, const float2 (&acc)[8][4],
                                       uint8_t* smb, int m0, int n0) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lr = lane >> 3, lc = lane & 7;
  __syncthreads();  // every ring is read
  float* part = reinterpret_cast<float*>(smb);
  if (have) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      float* row = part + (warp * BT + lr + 4 * q) * LDP;
      if (KN) {
        *reinterpret_cast<float4*>(row + 4 * lc) = make_float4(acc[q][0].x, acc[q][0].y, acc[q][1].x, acc[q][1].y);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) row[lc + 8 * j] = acc[q][j].x + acc[q][j].y;
      }
    }
  }
  __syncthreads();
  const int rank = SPLIT > 1 ? (int)blockIdx.z : 0;
  const int nk = min(NW, (g.K + ks - 1) / ks - rank * NW), r = threadIdx.x >> 3, c = (threadIdx.x & 7) * 4;
  const int m = m0 + r, col = n0 + c;
  if (SPLIT == 1 && (m >= g.M || col >= g.N)) return;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (SPLIT == 1 || nk > 0) s = *reinterpret_cast<const float4*>(part + r * LDP + c);
  for (int w = 1; w < nk; ++w) {
    const float4 t = *reinterpret_cast<const float4*>(part + (w * BT + r) * LDP + c);
    s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
  }
  if (SPLIT > 1) {
    __shared__ __align__(16) float other[BT / 2][LDP];
    tc::cluster_wait();  // the other CTA runs: its shared memory may be written
    const bool mine = (r >> 4) == rank;
    if (!mine) {
      const float v[4] = {s.x, s.y, s.z, s.w};
      tc::st_cluster4(tc::peer_addr(tc::smem_u32(&other[r & 15][c]), (uint32_t)(1 - rank)), v);
    }
    tc::cluster_arrive();
    tc::cluster_wait();
    if (!mine || m >= g.M || col >= g.N) return;
    const float4 t = *reinterpret_cast<const float4*>(&other[r & 15][c]);
    s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
  }
  if (col + 3 < g.N) {
    epilogue4(g, m, col, s, vc);
  } else {
    const float v[4] = {s.x, s.y, s.z, s.w};
    for (int i = 0; i < 4 && col + i < g.N; ++i) epilogue(g, m, col + i, v[i]);
  }
}

// The fp32 models' GEMMs have a few hundred rows at most (128 to 512 tokens), so time goes to the chain
// over K on the few SMs that have a tile: the tile is small (32 x 32) and the CTA's 8 warps split K.  A
// lane holds 8 x 4 sums; each warp copies its own operands through a ring of three 8-deep chunks
// (cp.async; the accumulation never waits for a whole load) and the warps' tiles are summed in warp
// order.  Packed FMAs: two k at a time with B [N, K] (both operands come as pairs), two columns with
// B [K, N].  A launch alone (64 x 64 tiles, one chain over K, scalar loads before): 128 x 128, K = 512 41 ->
// 8.8 us, K = 128 14 -> 4.4; 385 x 192, K = 768 49 -> 11.5, K = 192 19 -> 5.3; 385 x 768, K = 192 22.7 -> 10.3.
// The form for rows that TMA does not take; the one below serves the rest.
template <typename TI, bool KN>
__global__ void __launch_bounds__(NT, 2) gemm_simt_kernel(GemmArgs g, int ks, bool va, bool vb, bool vc) {
  constexpr int LDA = sizeof(TI) == 4 ? KC + 4 : KC;  // elements
  constexpr int LDB = KN ? BT : LDA;
  constexpr int ASZ = BT * LDA, STAGE = ASZ + (KN ? KC : BT) * LDB;
  extern __shared__ __align__(16) uint8_t smb[];
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lr = lane >> 3, lc = lane & 7;
  const int m0 = blockIdx.y * BT, n0 = blockIdx.x * BT;
  const TI* A = reinterpret_cast<const TI*>(g.A);
  const TI* B = reinterpret_cast<const TI*>(g.B);
  const int k0 = warp * ks, k1 = min(g.K, k0 + ks), n = k0 < k1 ? (k1 - k0 + KC - 1) / KC : 0;
  TI* ring = reinterpret_cast<TI*>(smb) + warp * NS * STAGE;
  auto issue = [&](int i) {
    if (i < n) {
      TI* st = ring + (i % NS) * STAGE;
      const int k = k0 + i * KC;
      copy_block(st, LDA, A + (size_t)m0 * g.lda + k, (size_t)g.lda, BT, KC, g.M - m0, k1 - k, va, lane);
      if (KN) copy_block(st + ASZ, LDB, B + (size_t)k * g.ldb + n0, (size_t)g.ldb, KC, BT, k1 - k, g.N - n0, vb, lane);
      else copy_block(st + ASZ, LDB, B + (size_t)n0 * g.ldb + k, (size_t)g.ldb, BT, KC, g.N - n0, k1 - k, vb, lane);
    }
    cp_commit();
  };
  // KN: acc[i][j] = columns 4 lc + 2 j, + 1 (j < 2); else the even and odd k of column lc + 8 j
  float2 acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = make_float2(0.f, 0.f);
  for (int i = 0; i < NS - 1; ++i) issue(i);
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    cp_wait<NS - 2>();
    __syncwarp();
    issue(i + NS - 1);  // (its stage was read before this __syncwarp)
    const TI* as = ring + (i % NS) * STAGE;
    const TI* bs = as + ASZ;
#pragma unroll
    for (int kq = 0; kq < KC; kq += 4) {
      float4 b[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = KN ? ld4s(bs + (kq + j) * LDB + 4 * lc) : ld4s(bs + (lc + 8 * j) * LDB + kq);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float4 x = ld4s(as + (lr + 4 * q) * LDA + kq);
        if (KN) {
          const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            acc[q][0] = __ffma2_rn(f2(xv[kk]), make_float2(b[kk].x, b[kk].y), acc[q][0]);
            acc[q][1] = __ffma2_rn(f2(xv[kk]), make_float2(b[kk].z, b[kk].w), acc[q][1]);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            acc[q][j] = __ffma2_rn(make_float2(x.x, x.y), make_float2(b[j].x, b[j].y), acc[q][j]);
            acc[q][j] = __ffma2_rn(make_float2(x.z, x.w), make_float2(b[j].z, b[j].w), acc[q][j]);
          }
        }
      }
    }
  }
  cp_wait<0>();
  finish<KN, 1>(g, ks, vc, n > 0, acc, smb, m0, n0);
}

// The same product where both operands' rows allow TMA (16-byte aligned, strides multiples of four
// floats), in 16-deep chunks of one box per operand: 32 rows x 16 k (64-byte rows under the 64-byte
// swizzle), with B [K, N] 16 k x 32 columns (128-byte rows).  One lane asks for a warp's next chunk; all
// of a warp's chunks are in flight at once where shared memory holds them.  By cp.async each instruction
// touched 16 lines for 32 bytes of each, and starting the first two chunks took 1800 cycles (500 here).
// What is left is the loop's shared-memory reads: a lane loads 12 floats per 32 multiply-adds, about 950
// cycles for 8 k on one CTA an SM (385 x 192, K = 768 on 78 CTAs: the shared-memory path is busy for 54 % of
// the cycles of an SM that has one); so, where half the SMs have no tile and K is at least 512, a cluster
// of two CTAs takes a half of K each.  Against the form above, a launch alone: 128 x 128, K = 512 8.8 -> 6.9 us;
// 385 x 192, K = 768 11.5 -> 10.8; at K below 256 0.4 us more alone, but in the stream the steps gain: the
// fp32 tiny step 113 -> 105 us, the 385-token fp32 step 405 -> 387.
constexpr int KT = 16, TSTAGE = BT * KT * 4 * 2, MAX_NS = 6;

__device__ __forceinline__ void tma_box(const CUtensorMap* tm, uint32_t dst, uint64_t* bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(tc::smem_u32(bar))
      : "memory");
}

template <bool KN, int SPLIT>
__global__ void __launch_bounds__(NT, 2)
    gemm_simt_tma_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, GemmArgs g,
                         int ks, int ns, bool vc) {
  extern __shared__ __align__(16) uint8_t smb[];
  // (the swizzles' periods are 512 and 1024 bytes)
  uint8_t* smt = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smb) + 1023) & ~static_cast<uintptr_t>(1023));
  __shared__ __align__(8) uint64_t bars[NW][MAX_NS];
  __shared__ volatile int abort_sh;
  const int warp = tc::warp_index(), lane = threadIdx.x & 31, lr = lane >> 3, lc = lane & 7;
  const int m0 = blockIdx.y * BT, n0 = blockIdx.x * BT;
  const int rank = SPLIT > 1 ? (int)blockIdx.z : 0;
  const int k0 = (rank * NW + warp) * ks, k1 = min(g.K, k0 + ks), n = k0 < k1 ? (k1 - k0 + KT - 1) / KT : 0;
  uint8_t* ring = smt + warp * ns * TSTAGE;
  if (threadIdx.x == 0) abort_sh = 0;
  if (lane < ns) tc::mbar_init(&bars[warp][lane], 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (SPLIT > 1) tc::cluster_arrive();  // (waited for before the first store to the other CTA)
  pdl_wait();
  pdl_trigger();
  auto issue = [&](int i, int stage) {  // chunk i of this warp's share
    if (tc::elect_one()) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // (the stage was read by every lane)
      uint64_t* bar = &bars[warp][stage];
      const uint32_t st = tc::smem_u32(ring + stage * TSTAGE);
      const int k = k0 + i * KT;
      tc::mbar_expect_tx(bar, TSTAGE);
      tma_box(&tmA, st, bar, k, m0);
      if (KN) tma_box(&tmB, st + TSTAGE / 2, bar, n0, k);
      else tma_box(&tmB, st + TSTAGE / 2, bar, k, n0);
    }
    __syncwarp();
  };
  // KN: acc[i][j] = columns 4 lc + 2 j, + 1 (j < 2); else the even and odd k of column lc + 8 j
  float2 acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = make_float2(0.f, 0.f);
  for (int i = 0; i < min(n, ns); ++i) issue(i, i);
  int stage = 0;
  uint32_t phase = 0;
  bool ok = true;
  int i = 0;
#pragma unroll 1
  for (; i < n; ++i) {
    if (!tc::mbar_wait_warp(&bars[warp][stage], phase, &abort_sh, g.err)) { ok = false; break; }
    const uint8_t* as = ring + stage * TSTAGE;
    const uint8_t* bs = as + TSTAGE / 2;
    // 16-byte piece c of row r of a box: 64-byte rows at c ^ ((r >> 1) & 3), 128-byte rows at c ^ (r & 7)
    // (rows of A are lr + 4 q and of B lc + 8 j, which differ from lr and lc by multiples that the
    // swizzle folds into q and drops for j)
#pragma unroll
    for (int kq = 0; kq < KT; kq += 4) {
      float4 b[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = KN ? kq + j : lc + 8 * j;
        b[j] = *reinterpret_cast<const float4*>(KN ? bs + r * 128 + ((lc ^ (r & 7)) << 4)
                                                   : bs + r * 64 + (((kq >> 2) ^ ((r >> 1) & 3)) << 4));
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int r = lr + 4 * q;
        const float4 x = *reinterpret_cast<const float4*>(as + r * 64 + (((kq >> 2) ^ ((r >> 1) & 3)) << 4));
        if (KN) {
          const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            acc[q][0] = __ffma2_rn(f2(xv[kk]), make_float2(b[kk].x, b[kk].y), acc[q][0]);
            acc[q][1] = __ffma2_rn(f2(xv[kk]), make_float2(b[kk].z, b[kk].w), acc[q][1]);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            acc[q][j] = __ffma2_rn(make_float2(x.x, x.y), make_float2(b[j].x, b[j].y), acc[q][j]);
            acc[q][j] = __ffma2_rn(make_float2(x.z, x.w), make_float2(b[j].z, b[j].w), acc[q][j]);
          }
        }
      }
    }
    __syncwarp();  // the stage is read
    if (i + ns < n) issue(i + ns, stage);
    if (++stage == ns) { stage = 0; phase ^= 1u; }
  }
  if (!ok) {  // given up: this warp's copies land before the CTA goes away
    volatile int no_abort = 0;
    for (int d = 0; d < min(ns, n - i); ++d)
      tc::mbar_wait(&bars[warp][(stage + d) % ns], stage + d < ns ? phase : phase ^ 1u, &no_abort, nullptr);
    __syncwarp();
  }
  finish<KN, SPLIT>(g, ks, vc, n > 0, acc, smt, m0, n0);
}

template <typename TI, bool KN>
cudaError_t launch_simt(const GemmArgs& g, cudaStream_t st) {
  constexpr int LDA = sizeof(TI) == 4 ? KC + 4 : KC, E = 16 / (int)sizeof(TI);
  constexpr size_t ring = (size_t)NW * NS * (BT * LDA + (KN ? KC * BT : BT * LDA)) * sizeof(TI), part = (size_t)NW * BT * LDP * 4;
  constexpr size_t smem = ring > part ? ring : part;
  auto k = gemm_simt_kernel<TI, KN>;
  cudaError_t e = allow_smem(k, (int)smem);
  if (e != cudaSuccess) return e;
  const int ks = ((g.K + NW - 1) / NW + KC - 1) / KC * KC;
  auto al = [](const void* p, int ld) { return ((uintptr_t)p & 15) == 0 && ld % 4 == 0; };
  const bool va = g.K % E == 0 && g.lda % E == 0 && ((uintptr_t)g.A & 15) == 0;
  const bool vb = (KN ? g.N : g.K) % E == 0 && g.ldb % E == 0 && ((uintptr_t)g.B & 15) == 0;
  const bool vc = al(g.C, g.ldc) && al(g.C2, g.ldc2) && al(g.aux, g.ldaux);
  if constexpr (sizeof(TI) == 4) {
    CUtensorMap ma, mb;
    if (va && vb && tc_available() && tma_map_f32(&ma, g.A, g.M, g.K, g.lda, KT, BT) &&
        (KN ? tma_map_f32(&mb, g.B, g.K, g.N, g.ldb, BT, KT) : tma_map_f32(&mb, g.B, g.N, g.K, g.ldb, KT, BT))) {
      const int tiles = ((g.N + BT - 1) / BT) * ((g.M + BT - 1) / BT);
      // two CTAs to a tile where that still is one CTA an SM and halves a long chain
      const int split = 2 * tiles <= device_sm_count() && g.K >= 512 ? 2 : 1, shares = NW * split;
      const int kt = ((g.K + shares - 1) / shares + KT - 1) / KT * KT;
      // two CTAs an SM where there are more tiles than SMs
      const int ns = std::min(kt / KT, tiles > device_sm_count() ? 3 : MAX_NS);
      const size_t sm = std::max((size_t)NW * ns * TSTAGE, part) + 1024;
      auto kern = split == 2 ? gemm_simt_tma_kernel<KN, 2> : gemm_simt_tma_kernel<KN, 1>;
      cudaError_t e = allow_smem(kern, (int)std::max((size_t)NW * MAX_NS * TSTAGE, part) + 1024);
      if (e != cudaSuccess) return e;
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute attr[2];
      attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[0].val.programmaticStreamSerializationAllowed = 1;
      attr[1].id = cudaLaunchAttributeClusterDimension;
      attr[1].val.clusterDim.x = attr[1].val.clusterDim.y = 1;
      attr[1].val.clusterDim.z = split;
      cfg.gridDim = dim3((g.N + BT - 1) / BT, (g.M + BT - 1) / BT, split);
      cfg.blockDim = dim3(NT);
      cfg.dynamicSmemBytes = sm;
      cfg.stream = st;
      cfg.attrs = attr;
      cfg.numAttrs = split == 2 ? 2 : 1;
      e = cudaLaunchKernelEx(&cfg, kern, ma, mb, g, kt, ns, vc);
      note_launch(1);
      return e != cudaSuccess ? e : cudaGetLastError();
    }
  }
  e = launch_pdl(k, dim3((g.N + BT - 1) / BT, (g.M + BT - 1) / BT), dim3(NT), smem, st, g, ks, va, vb, vc);
  note_launch(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// h[m, j] = silu(gate) * up from the packed [gate|up] matrix
__global__ void swiglu_kernel(const void* gu, int ld_gu, int gu_dtype, void* h, int ld_h,
                              int h_dtype, int M, int F) {
  int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)M * F) return;
  int m = (int)(idx / F), j = (int)(idx % F);
  int64_t gc = gate_col(j);
  float gt = ld_dt(gu, gu_dtype, (int64_t)m * ld_gu + gc);
  float up = ld_dt(gu, gu_dtype, (int64_t)m * ld_gu + gc + 64);
  st_dt(h, h_dtype, (int64_t)m * ld_h + j, silu_f(gt) * up);
}

}  // namespace

cudaError_t gemm_simt(const GemmArgs& g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  // a grid's y dimension holds 65535 row tiles; the rows past them are a product of their own
  constexpr int ROWS = 65535 * BT;
  if (g.M > ROWS) {
    auto down = [](const void* p, int64_t ld, int dt) {
      return p ? const_cast<char*>(static_cast<const char*>(p)) + ROWS * ld * (int64_t)dtype_size(dt) : nullptr;
    };
    GemmArgs head = g, rest = g;
    head.M = ROWS;
    rest.M = g.M - ROWS;
    rest.A = down(g.A, g.lda, g.in_dtype);
    rest.C = down(g.C, g.ldc, g.c_dtype);
    rest.C2 = down(g.C2, g.ldc2, g.c2_dtype);
    rest.aux = down(g.aux, g.ldaux, g.aux_dtype);
    const cudaError_t e = gemm_simt(head, st);
    return e != cudaSuccess ? e : gemm_simt(rest, st);
  }
  cudaError_t e = g.in_dtype == DT_BF16 ? (g.b_kn ? launch_simt<bf16, true>(g, st) : launch_simt<bf16, false>(g, st))
                                        : (g.b_kn ? launch_simt<float, true>(g, st) : launch_simt<float, false>(g, st));
  if (e != cudaSuccess || g.epi != EPI_SWIGLU) return e;
  int F = g.N / 2;
  int64_t n = (int64_t)g.M * F;
  swiglu_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(g.C, g.ldc, g.c_dtype, g.C2,
                                                             g.ldc2, g.c2_dtype, g.M, F);
  note_launch(1);
  return cudaGetLastError();
}

cudaError_t gemm(const GemmArgs& g, cudaStream_t st) {
  if (g.in_dtype == DT_BF16 && tc_available()) {
    cudaError_t e = gemm_tc(g, st);
    if (e != cudaErrorNotSupported) return e;
  }
  return gemm_simt(g, st);
}

}  // namespace ra

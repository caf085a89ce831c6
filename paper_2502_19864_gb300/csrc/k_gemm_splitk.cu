// k_gemm_splitk.cu -- tcgen05 GEMM for products of few output tiles: K split over a cluster.
//
// The persistent kernel gives a tile to one CTA, so a product of few rows runs on few SMs, each
// walking all of K: 128 x 768 with K = 3072 was 6 CTAs and 48 k-blocks one after the other.
// Here a cluster of S CTAs (2, 4 or 8) shares a 128 x BN tile: each multiplies its share of
// the k-blocks into TMEM, sends the rows of its fp32 partial to the CTAs that own them (128 / S
// rows each) through distributed shared memory, and each CTA adds the S partials of its rows in
// cluster order (fixed: deterministic) and runs the epilogue on them.  What bounds it is the
// chain: set-up, the copies' latency (all stages are in flight at once), one exchange.
// 128 x 768 x 3072: 12.1 us there, 5.9 here; 128 x 768 x 768: 5.8 and 5.0 (a launch of K = 64 takes
// about 4).
//   warp 0      TMA producer, warp 1 TMEM allocation and tcgen05.mma issue, as in the persistent
//               kernel; then all eight warps take the accumulator out (two per TMEM lane
//               quadrant, half of the columns each) and share the epilogue.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "tcgen05.cuh"

namespace ra {
namespace {

using namespace tc;

constexpr int BM = 128, BK = 64, THREADS = 256;

template <int BN>
struct Cfg {
  static constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2, STAGE = A_BYTES + B_BYTES;
  static constexpr int STAGES = BN == 64 ? 7 : 4;
  // received partials: S x (128 / S) rows of BN floats, 16 bytes of padding a row
  static constexpr int LDR = BN + 4;
  static constexpr int RECV = BM * LDR * 4;
  static constexpr int SMEM = STAGES * STAGE + RECV + 1024;  // + alignment slack
};

struct Params {
  int M, N, k_blocks, b_kn, b_frozen, epi, split, m_tiles;
  void* C; int ldc; int c_dtype;
  const float* bias;
  void* C2; int ldc2; int c2_dtype;
  const void* aux; int ldaux; int aux_dtype;
  unsigned* err;
};

__device__ __forceinline__ void tma_load_2d(const CUtensorMap* tm, uint32_t dst, uint64_t* bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
      : "memory");
}
// four consecutive values at element offset `at` of a bf16 or fp32 matrix
__device__ __forceinline__ float4 load4(const void* p, int dt, size_t at) {
  if (dt == DT_F32) return *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(p) + at);
  const uint2 u = *reinterpret_cast<const uint2*>(reinterpret_cast<const bf16*>(p) + at);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void store4(void* p, int dt, size_t at, float4 v) {
  if (dt == DT_F32) {
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(p) + at) = v;
    return;
  }
  uint2 u;
  *reinterpret_cast<__nv_bfloat162*>(&u.x) = __floats2bfloat162_rn(v.x, v.y);
  *reinterpret_cast<__nv_bfloat162*>(&u.y) = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(reinterpret_cast<bf16*>(p) + at) = u;
}

template <int BN>
__global__ void __launch_bounds__(THREADS, 1)
    gemm_splitk_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const Params p) {
  using C = Cfg<BN>;
  constexpr int STAGES = C::STAGES;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES], done_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ volatile int abort_sh;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const uint32_t smem_base = smem_u32(smem);
  float* recv = reinterpret_cast<float*>(smem + STAGES * C::STAGE);
  const int warp = warp_index(), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    mbar_init(&done_bar, 1);
    abort_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                 "r"((uint32_t)BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_sh;
  cluster_arrive();  // (waited for before the first store to a peer: every CTA has then started)
  const int S = p.split, rank = (int)cluster_rank();
  const int tile = blockIdx.x / S;
  const int m0 = (tile % p.m_tiles) * BM, n0 = (tile / p.m_tiles) * BN;
  const int kb0 = rank * p.k_blocks / S, kb1 = (rank + 1) * p.k_blocks / S;

  // The set-up above overlaps the previous kernel's tail; a frozen B's first stages do too (at one
  // sequence its weights come from DRAM, and the CTAs are mostly on idle SMs by then)
  auto load_b = [&](int stage, int kb) {
    const uint32_t sb = smem_base + stage * C::STAGE + C::A_BYTES;
    if (p.b_kn) {
#pragma unroll
      for (int a = 0; a < BN / 64; ++a) tma_load_2d(&tmB, sb + a * 8192, &full_bar[stage], n0 + 64 * a, kb * BK);
    } else {
      tma_load_2d(&tmB, sb, &full_bar[stage], kb * BK, n0);
    }
  };
  const int early = p.b_frozen ? min(STAGES, kb1 - kb0) : 0;
  if (warp == 0 && elect_one())
    for (int i = 0; i < early; ++i) {
      mbar_expect_tx(&full_bar[i], C::STAGE);
      load_b(i, kb0 + i);
    }
  __syncwarp();
  pdl_wait();
  pdl_trigger();
  if (warp == 0) {
    if (elect_one()) {
      int stage = 0, kb = kb0;
      uint32_t phase = 0;
      for (; kb < kb1; ++kb) {
        const bool b_here = kb - kb0 < early;
        if (!b_here) {
          if (!mbar_wait(&empty_bar[stage], phase ^ 1u, &abort_sh, p.err)) break;
          mbar_expect_tx(&full_bar[stage], C::STAGE);
          load_b(stage, kb);
        }
        tma_load_2d(&tmA, smem_base + stage * C::STAGE, &full_bar[stage], kb * BK, m0);
        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
      }
      if (kb < kb1) {  // given up: every copy that was started lands before the CTA goes away
        volatile int no_abort = 0;
        for (int i = max(kb0, kb - STAGES); i < kb; ++i)
          mbar_wait(&full_bar[(i - kb0) % STAGES], (uint32_t)((i - kb0) / STAGES) & 1u, &no_abort, nullptr);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (elect_one()) {
      const uint64_t ring = sdesc_sw128(smem_base), ring_kn = sdesc_mn_sw128_lbo(smem_base, 8192);
      auto issue = [&](auto kn) {  // KN: B as stored [K, N]
        constexpr bool KN = decltype(kn)::value;
        constexpr uint32_t idesc = KN ? idesc_bf16_bmn(BM, BN) : idesc_bf16(BM, BN);
        // K-major B: 16 elements = 32 bytes a step; [K, N] B (MN-major): 16 rows = 2048 bytes
        constexpr uint64_t bstep = KN ? 128u : 2u;
        int stage = 0;
        uint32_t phase = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(&full_bar[stage], phase, &abort_sh, p.err)) return;
          tc_fence_after();
          const uint64_t off = (uint64_t)(stage * (C::STAGE / 16));
          const uint64_t adesc = ring + off, bdesc = (KN ? ring_kn : ring) + off + (uint64_t)(C::A_BYTES / 16);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            umma_bf16(tmem_base, adesc + (uint64_t)(2 * k), bdesc + bstep * (uint64_t)k, idesc, (kb != kb0 || k != 0) ? 1u : 0u);
          umma_commit(&empty_bar[stage]);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
      };
      if (p.b_kn) issue(std::true_type());
      else issue(std::false_type());
      // every product issued above is complete before TMEM and shared memory are released
      umma_commit(&done_bar);
      volatile int no_abort = 0;
      mbar_wait(&done_bar, 0, &no_abort, nullptr);
    }
    __syncwarp();
  }

  const bool ok = mbar_wait_warp(&done_bar, 0, &abort_sh, p.err);
  tc_fence_after();
  cluster_wait();  // every CTA of the cluster runs: its shared memory may be written
  const int rows = BM / S;
  {
    const int quad = warp & 3, half = warp >> 2;
    const int row = quad * 32 + lane, owner = row / rows;
    uint32_t dst = peer_addr(smem_u32(recv + (size_t)(rank * rows + row % rows) * C::LDR + half * (BN / 2)), (uint32_t)owner);
#pragma unroll
    for (int c = 0; c < BN / 2; c += 32) {
      float v[32];
      tmem_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * (BN / 2) + c), v);
#pragma unroll
      for (int q = 0; q < 8; ++q) st_cluster4(dst + (c + 4 * q) * 4, v + 4 * q);
    }
  }
  tc_fence_before();
  cluster_arrive();
  cluster_wait();  // the partials of this CTA's rows are here, and no peer writes any more
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)BN) : "memory");
  }
  if (!ok) return;

  auto sum4 = [&](int r, int c) {
    float4 s = *reinterpret_cast<const float4*>(recv + (size_t)r * C::LDR + c);
    for (int q = 1; q < S; ++q) {
      const float4 x = *reinterpret_cast<const float4*>(recv + (size_t)(q * rows + r) * C::LDR + c);
      s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
    }
    return s;
  };
  // SwiGLU: per 128 columns, 64 of the gate and the matching 64 of the up projection
  const int cols = p.epi == EPI_SWIGLU ? 64 : BN;
  for (int e = threadIdx.x; e < rows * (cols / 4); e += THREADS) {
    const int r = e / (cols / 4), c = (e % (cols / 4)) * 4;
    const int m = m0 + rank * rows + r, n = n0 + c;
    if (m >= p.M || n >= p.N) continue;
    float4 v = sum4(r, c);
    if (p.epi == EPI_SWIGLU) {
      if (BN < 128) continue;  // (not launched: the gate|up blocks are 128 wide)
      const float4 u = sum4(r, BN < 128 ? 0 : c + 64);
      if (p.C) {
        store4(p.C, p.c_dtype, (size_t)m * p.ldc + n, v);
        store4(p.C, p.c_dtype, (size_t)m * p.ldc + n + 64, u);
      }
      store4(p.C2, p.c2_dtype, (size_t)m * p.ldc2 + n0 / 2 + c,
             make_float4(silu_f(v.x) * u.x, silu_f(v.y) * u.y, silu_f(v.z) * u.z, silu_f(v.w) * u.w));
    } else if (p.epi == EPI_DSWIGLU) {
      // d(h) -> d(gate), d(up) in the packed layout
      const size_t gc = (size_t)(n >> 6) * 128 + (n & 63);
      const float4 g = load4(p.aux, DT_BF16, (size_t)m * p.ldaux + gc), u = load4(p.aux, DT_BF16, (size_t)m * p.ldaux + gc + 64);
      store4(p.C, p.c_dtype, (size_t)m * p.ldc + gc,
             make_float4(v.x * u.x * silu_grad_f(g.x), v.y * u.y * silu_grad_f(g.y), v.z * u.z * silu_grad_f(g.z),
                         v.w * u.w * silu_grad_f(g.w)));
      store4(p.C, p.c_dtype, (size_t)m * p.ldc + gc + 64,
             make_float4(v.x * silu_f(g.x), v.y * silu_f(g.y), v.z * silu_f(g.z), v.w * silu_f(g.w)));
    } else if (p.epi == EPI_MUL || p.epi == EPI_RESID) {
      const float4 x = load4(p.aux, p.aux_dtype, (size_t)m * p.ldaux + n);
      v = p.epi == EPI_MUL ? make_float4(v.x * x.x, v.y * x.y, v.z * x.z, v.w * x.w)
                           : make_float4(v.x + x.x, v.y + x.y, v.z + x.z, v.w + x.w);
      store4(p.C, p.c_dtype, (size_t)m * p.ldc + n, v);
    } else {
      if (p.bias) {
        const float4 b = __ldg(reinterpret_cast<const float4*>(p.bias + n));
        v.x += b.x; v.y += b.y; v.z += b.z; v.w += b.w;
      }
      if (p.epi == EPI_STORE || (p.epi == EPI_BIAS_GELU && p.C)) store4(p.C, p.c_dtype, (size_t)m * p.ldc + n, v);
      if (p.epi == EPI_BIAS_GELU) {
        const float2 y0 = gelu2(make_float2(v.x, v.y)), y1 = gelu2(make_float2(v.z, v.w));
        store4(p.C2, p.c2_dtype, (size_t)m * p.ldc2 + n, make_float4(y0.x, y0.y, y1.x, y1.y));
      } else if (p.epi == EPI_BIAS_GELU_G) {
        float2 y0, d0, y1, d1;
        gelu_both2(make_float2(v.x, v.y), y0, d0);
        gelu_both2(make_float2(v.z, v.w), y1, d1);
        if (p.C) store4(p.C, p.c_dtype, (size_t)m * p.ldc + n, make_float4(d0.x, d0.y, d1.x, d1.y));
        store4(p.C2, p.c2_dtype, (size_t)m * p.ldc2 + n, make_float4(y0.x, y0.y, y1.x, y1.y));
      }
    }
  }
}

template <int BN>
cudaLaunchConfig_t config(cudaLaunchAttribute* attr, int grid, int split, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = split;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = Cfg<BN>::SMEM;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

template <int BN>
bool prepare() {
  static const bool ok =
      cudaFuncSetAttribute(gemm_splitk_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<BN>::SMEM) == cudaSuccess;
  return ok;
}

// Clusters of 2^i CTAs that the device holds at once (at one CTA an SM: fewer than SMs / 2^i, since
// a cluster stays within one group of SMs)
template <int BN>
int resident_clusters(int i) {
  struct Counts {
    int n[4];
    Counts() {
      for (int i = 0; i < 4; ++i) {
        cudaLaunchAttribute attr[2];
        const cudaLaunchConfig_t cfg = config<BN>(attr, device_sm_count() >> i << i, 1 << i, nullptr);
        n[i] = 0;
        if (!prepare<BN>() || cudaOccupancyMaxActiveClusters(&n[i], gemm_splitk_kernel<BN>, &cfg) != cudaSuccess) {
          n[i] = 0;
          cudaGetLastError();  // (not the caller's)
        }
      }
    }
  };
  static const Counts c;
  return c.n[i];
}

template <int BN>
cudaError_t launch(const CUtensorMap& a, const CUtensorMap& b, const Params& p, int grid, cudaStream_t st) {
  if (!prepare<BN>()) return cudaErrorNotSupported;
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = config<BN>(attr, grid, p.split, st);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, gemm_splitk_kernel<BN>, a, b, p);
  note_launch(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// CTAs to a tile (0: the persistent kernel): the most that leave each two k-blocks and run in one
// wave.  Measured, back to back with cold weights: the persistent kernel takes 3.7 us + 0.175 us a
// k-block, this one 4.9 + 0.155 a k-block of its share (tiles 64 wide), so the split has to save
// the fixed 1.2 us: from 8 k-blocks at 8 CTAs a tile (128 x 768, K = 3072: 12.1 -> 5.9 us), 9 at 4
// (128 x 2304, K = 768: 6.1 -> 5.5), 13 at 2 (512 x 1024, K = 1024: 6.8 -> 6.2; K = 256: 4.7, not
// 5.2).  The GELU epilogues cost the persistent kernel 1.4 us more than here (eight rows of a tile
// a warp instead of 32): any split wins (128 x 3072, K = 768: 8.0 -> 6.6).  The SwiGLU epilogue
// needs 128-wide tiles, whose exchange costs 1.7 us more.
int choose_split(const GemmArgs& g, int bn) {
  const int kb = (g.K + BK - 1) / BK;
  const int tiles = ((g.M + BM - 1) / BM) * ((g.N + bn - 1) / bn);
  const bool gelu = g.epi == EPI_BIAS_GELU || g.epi == EPI_BIAS_GELU_G;
  const int least[4] = {0, gelu ? 4 : bn == 64 ? 13 : 33, gelu ? 8 : bn == 64 ? 9 : 20, gelu || bn == 64 ? 16 : 17};
  for (int i = 3; i > 0; --i)
    if (kb >= 2 << i && kb >= least[i] && tiles <= (bn == 64 ? resident_clusters<64>(i) : resident_clusters<128>(i)))
      return 1 << i;
  return 0;
}

}  // namespace

// Called with arguments that gemm_tc has checked
cudaError_t gemm_splitk(const GemmArgs& g, cudaStream_t st) {
  const int bn = g.epi == EPI_SWIGLU ? 128 : 64;
  const int split = choose_split(g, bn);
  if (split == 0) return cudaErrorNotSupported;
  const bool aux = g.epi == EPI_MUL || g.epi == EPI_RESID || g.epi == EPI_DSWIGLU;
  if ((aux && !g.aux) || (g.epi == EPI_DSWIGLU && g.aux_dtype != DT_BF16)) return cudaErrorNotSupported;
  CUtensorMap ma, mb;
  if (!tma_map_bf16(&ma, g.A, g.M, g.K, g.lda, BK, BM)) return cudaErrorNotSupported;
  if (g.b_kn ? !tma_map_bf16(&mb, g.B, g.K, g.N, g.ldb, 64, BK) : !tma_map_bf16(&mb, g.B, g.N, g.K, g.ldb, BK, bn))
    return cudaErrorNotSupported;
  Params p;
  p.M = g.M; p.N = g.N; p.k_blocks = (g.K + BK - 1) / BK; p.b_kn = g.b_kn; p.b_frozen = g.b_frozen; p.epi = g.epi; p.split = split;
  p.m_tiles = (g.M + BM - 1) / BM;
  p.C = g.C; p.ldc = g.ldc; p.c_dtype = g.c_dtype; p.bias = g.bias;
  p.C2 = g.C2; p.ldc2 = g.ldc2; p.c2_dtype = g.c2_dtype;
  p.aux = g.aux; p.ldaux = g.ldaux; p.aux_dtype = g.aux_dtype; p.err = g.err;
  const int grid = p.m_tiles * ((g.N + bn - 1) / bn) * split;
  return bn == 64 ? launch<64>(ma, mb, p, grid, st) : launch<128>(ma, mb, p, grid, st);
}

}  // namespace ra

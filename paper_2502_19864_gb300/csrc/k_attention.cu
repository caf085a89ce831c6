// k_attention.cu -- fused attention forward and backward in fp32 arithmetic on the CUDA cores: the
// fp32 models, and bf16 head dims the tensor-core kernels do not take (32, 96).
//
// softmax(q k^T * scale [+ causal mask]) v per (batch, head), with the online softmax so
// the S x S score matrix never reaches memory.  The forward saves the row log-sum-exp;
// the backward recomputes P from q, k and that statistic (no P is stored).  RoPE
// (rotate-half, pairs (i, i + dh/2)) is applied to q and k as they are loaded, and its
// transpose to dq and dk as they are stored, so the saved q|k|v are the raw projections.
// The backward is deterministic: one role holds queries and streams keys (dQ), the other holds
// keys and streams queries (dK, dV).
//
// A CTA of 4 warps holds 16 rows (4 a warp) and streams blocks of 64: these models have 32 to a few
// hundred positions, so the row tile is small to give many CTAs, and each step is a small product in
// registers: a lane takes 2 columns x 4 rows of the scores (16-byte shared loads along the head dim,
// packed FMAs), writes P or dS to shared memory and then takes dims lane + 32 c of 4 rows.  Measured
// (64 queries a CTA, one query at a time, scalar loads, before): S 32, 8 heads: forward 56 -> 7.7 us; S 77,
// 15 heads: forward 111 -> 13.7 us, backward 160 -> 17.7 us.
#include "common.cuh"
#include "kernels.h"
#include "simt.cuh"

namespace ra {
namespace {

constexpr int RB = 16;    // rows a CTA holds
constexpr int CB = 64;    // rows of a streamed block
constexpr int AT = 128;   // threads
constexpr int LP = CB + 4;
constexpr int MAXD = 128;

__device__ __forceinline__ void st4s(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

// Rows [r0, r0 + n) of one head's dh columns (src: position 0's first column; row stride ld) into
// shared memory as float [n][dh + 4], rotated by RoPE if asked.  Rows at or beyond S are zero.
template <typename T>
__device__ __forceinline__ void load_rows(float* dst, const T* src, size_t ld, int S, int r0, int n, int dh, bool rope,
                                          float theta) {
  const int half = dh / 2, per = dh / 8, lds = dh + 4;
  for (int e = threadIdx.x; e < n * per; e += AT) {
    const int r = e / per, i = (e % per) * 4, s = r0 + r;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
    if (s < S) {
      a = ld4s(src + (size_t)s * ld + i);
      b = ld4s(src + (size_t)s * ld + i + half);
      if (rope) {
        float* x = &a.x;
        float* y = &b.x;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float sn, cs;
          sincosf((float)s * rope_freq(i + q, dh, theta), &sn, &cs);
          const float u = x[q] * cs - y[q] * sn, v = y[q] * cs + x[q] * sn;
          x[q] = u;
          y[q] = v;
        }
      }
    }
    st4s(dst + r * lds + i, a);
    st4s(dst + r * lds + i + half, b);
  }
}

// s[r][c] = X[4 w + r] . Y[lane + 32 c] for this warp's 4 rows of X and two rows of Y
__device__ __forceinline__ void scores(const float* X, const float* Y, int dh, int lane, float (&s)[4][2]) {
  const int lds = dh + 4;
  float2 a[4][2];
#pragma unroll
  for (int r = 0; r < 4; ++r) a[r][0] = a[r][1] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int d = 0; d < dh; d += 4) {
    const float4 y0 = ld4s(Y + lane * lds + d), y1 = ld4s(Y + (lane + 32) * lds + d);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 x = ld4s(X + r * lds + d);
      a[r][0] = __ffma2_rn(make_float2(x.x, x.y), make_float2(y0.x, y0.y), a[r][0]);
      a[r][0] = __ffma2_rn(make_float2(x.z, x.w), make_float2(y0.z, y0.w), a[r][0]);
      a[r][1] = __ffma2_rn(make_float2(x.x, x.y), make_float2(y1.x, y1.y), a[r][1]);
      a[r][1] = __ffma2_rn(make_float2(x.z, x.w), make_float2(y1.z, y1.w), a[r][1]);
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    s[r][0] = a[r][0].x + a[r][0].y;
    s[r][1] = a[r][1].x + a[r][1].y;
  }
}

// o[r][c] += sum_j P[r][j] Y[j][lane + 32 c] over a block (P: this warp's 4 rows)
__device__ __forceinline__ void accumulate(const float* P, const float* Y, int dh, int lane, float (&o)[4][MAXD / 32]) {
  const int lds = dh + 4, nd = dh / 32;
#pragma unroll 4
  for (int j = 0; j < CB; j += 4) {
    float4 p[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) p[r] = ld4s(P + r * LP + j);
#pragma unroll
    for (int c = 0; c < MAXD / 32; ++c) {
      if (c < nd) {
        const float* y = Y + j * lds + lane + 32 * c;
        const float y0 = y[0], y1 = y[lds], y2 = y[2 * lds], y3 = y[3 * lds];
#pragma unroll
        for (int r = 0; r < 4; ++r)
          o[r][c] = fmaf(p[r].w, y3, fmaf(p[r].z, y2, fmaf(p[r].y, y1, fmaf(p[r].x, y0, o[r][c]))));
      }
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(AT) attn_fwd_kernel(AttnArgs a) {
  extern __shared__ __align__(16) float sm[];
  pdl_wait();
  pdl_trigger();
  const int dh = a.head_dim, lds = dh + 4, S = a.S;
  float* Qs = sm;               // [RB][lds]
  float* Ks = Qs + RB * lds;    // [CB][lds]
  float* Vs = Ks + CB * lds;    // [CB][lds]
  const int bh = blockIdx.y, b = bh / a.n_heads, hh = bh % a.n_heads;
  const int H = a.n_heads * dh, q0 = blockIdx.x * RB;
  const T* qkv = reinterpret_cast<const T*>(a.qkv) + (size_t)b * S * 3 * H + hh * dh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* P = Vs + CB * lds + warp * 4 * LP;  // [4][LP] of this warp

  load_rows<T>(Qs, qkv, 3 * H, S, q0, RB, dh, a.rope, a.rope_theta);
  float o[4][MAXD / 32], m[4], l[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    m[r] = -INFINITY;
    l[r] = 0.f;
#pragma unroll
    for (int c = 0; c < MAXD / 32; ++c) o[r][c] = 0.f;
  }
  const int kend = a.causal ? min(S, q0 + RB) : S;
  for (int k0 = 0; k0 < kend; k0 += CB) {
    __syncthreads();
    load_rows<T>(Ks, qkv + H, 3 * H, S, k0, CB, dh, a.rope, a.rope_theta);
    load_rows<T>(Vs, qkv + 2 * H, 3 * H, S, k0, CB, dh, false, 0.f);
    __syncthreads();
    float s[4][2];
    scores(Qs + warp * 4 * lds, Ks, dh, lane, s);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int q = q0 + warp * 4 + r;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int key = k0 + lane + 32 * c;
        s[r][c] = key < S && (!a.causal || key <= q) ? s[r][c] * a.scale : -INFINITY;
      }
      const float mn = fmaxf(m[r], warp_max(fmaxf(s[r][0], s[r][1])));
      float p0 = 0.f, p1 = 0.f, alpha = 1.f;
      if (mn > -INFINITY) {  // some key of the row is live by now
        alpha = expf(m[r] - mn);
        p0 = expf(s[r][0] - mn);
        p1 = expf(s[r][1] - mn);
        m[r] = mn;
      }
      l[r] = l[r] * alpha + warp_sum(p0 + p1);
      P[r * LP + lane] = p0;
      P[r * LP + lane + 32] = p1;
#pragma unroll
      for (int c = 0; c < MAXD / 32; ++c) o[r][c] *= alpha;
    }
    __syncwarp();
    accumulate(P, Vs, dh, lane, o);
  }
  T* O = reinterpret_cast<T*>(a.O);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int q = q0 + warp * 4 + r;
    if (q >= S) break;
    const float inv = 1.f / l[r];
    const int64_t row = (int64_t)(b * S + q) * H + hh * dh;
#pragma unroll
    for (int c = 0; c < MAXD / 32; ++c)
      if (32 * c < dh) O[row + lane + 32 * c] = from_f<T>(o[r][c] * inv);
    if (a.lse && lane == 0) a.lse[(int64_t)bh * S + q] = m[r] + logf(l[r]);
  }
}

// D[b, h, s] = sum_d dO * O  (one warp per (token, head))
template <typename T>
__global__ void attn_bwd_pre_kernel(AttnArgs a) {
  pdl_wait();
  pdl_trigger();
  int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  int T_ = a.B * a.S;
  if (gw >= T_ * a.n_heads) return;
  int t = gw / a.n_heads, hh = gw % a.n_heads;
  int b = t / a.S, s = t % a.S;
  int dh = a.head_dim, H = a.n_heads * dh;
  const T* O = reinterpret_cast<const T*>(a.O);
  const T* dO = reinterpret_cast<const T*>(a.dO);
  float acc = 0.f;
  for (int d = lane; d < dh; d += 32) {
    int64_t i = (int64_t)t * H + hh * dh + d;
    acc += to_f(O[i]) * to_f(dO[i]);
  }
  acc = warp_sum(acc);
  if (lane == 0) a.Dscratch[((int64_t)b * a.n_heads + hh) * a.S + s] = acc;
}

// bf16, head_dim 64 or 128: G = head_dim / 8 threads per (token, head), 16-byte loads
template <int G>
__global__ void __launch_bounds__(256) attn_bwd_pre_vec_kernel(AttnArgs a) {
  pdl_wait();
  pdl_trigger();
  const int64_t gi = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
  const int r = threadIdx.x % G;
  const int T_ = a.B * a.S;
  // groups past the end stay for the shuffles below (full warps) but touch no memory
  const bool live = gi < (int64_t)T_ * a.n_heads;
  const int t = live ? (int)(gi / a.n_heads) : 0, hh = live ? (int)(gi % a.n_heads) : 0;
  const int b = t / a.S, s = t % a.S;
  const int dh = 8 * G, H = a.n_heads * dh;
  const int64_t i = (int64_t)t * H + hh * dh + 8 * r;
  uint4 o = make_uint4(0, 0, 0, 0), g = o;
  if (live) {
    o = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const bf16*>(a.O) + i));
    g = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const bf16*>(a.dO) + i));
  }
  const __nv_bfloat162* o2 = reinterpret_cast<const __nv_bfloat162*>(&o);
  const __nv_bfloat162* g2 = reinterpret_cast<const __nv_bfloat162*>(&g);
  float acc = 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 x = __bfloat1622float2(o2[k]), y = __bfloat1622float2(g2[k]);
    acc += x.x * y.x + x.y * y.y;
  }
#pragma unroll
  for (int off = G / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (live && r == 0) a.Dscratch[((int64_t)b * a.n_heads + hh) * a.S + s] = acc;
}

// f * acc of this warp's rows -> dst (position 0's first column; row stride ld), un-rotated if asked
// (the rotation's transpose; a lane's dims lane + 32 c have their partners i + dh/2 in other lanes when
// dh/2 is not a multiple of 32, so rotated rows go through shared memory).
template <typename T>
__device__ __forceinline__ void store_rows(T* dst, size_t ld, const float (&acc)[4][MAXD / 32], float* tmp, int row0,
                                           int S, int dh, int lane, bool rope, float theta) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int s = row0 + r;
    if (s >= S) break;
    T* out = dst + (size_t)s * ld;
    if (!rope) {
#pragma unroll
      for (int c = 0; c < MAXD / 32; ++c)
        if (32 * c < dh) out[lane + 32 * c] = from_f<T>(acc[r][c]);
      continue;
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < MAXD / 32; ++c)
      if (32 * c < dh) tmp[lane + 32 * c] = acc[r][c];
    __syncwarp();
    const int half = dh / 2;
    for (int i = lane; i < half; i += 32) {
      float sn, cs;
      sincosf((float)s * rope_freq(i, dh, theta), &sn, &cs);
      const float d1 = tmp[i], d2 = tmp[i + half];
      out[i] = from_f<T>(d1 * cs + d2 * sn);
      out[i + half] = from_f<T>(d2 * cs - d1 * sn);
    }
  }
}

// blockIdx.z = 0: rows are keys, blocks are queries -> dK, dV; 1: rows are queries, blocks keys -> dQ
template <typename T>
__global__ void __launch_bounds__(AT) attn_bwd_kernel(AttnArgs a) {
  extern __shared__ __align__(16) float sm[];
  pdl_wait();
  pdl_trigger();
  const int dh = a.head_dim, lds = dh + 4, S = a.S;
  float* X1 = sm;               // [RB][lds] k (or q) of the CTA's rows
  float* X2 = X1 + RB * lds;    // [RB][lds] v (or dO)
  float* Y1 = X2 + RB * lds;    // [CB][lds] q (or k) of the block
  float* Y2 = Y1 + CB * lds;    // [CB][lds] dO (or v)
  const bool keys = blockIdx.z == 0;
  const int bh = blockIdx.y, b = bh / a.n_heads, hh = bh % a.n_heads;
  const int H = a.n_heads * dh, r0 = blockIdx.x * RB;
  const T* q = reinterpret_cast<const T*>(a.qkv) + (size_t)b * S * 3 * H + hh * dh;
  const T* dO = reinterpret_cast<const T*>(a.dO) + (size_t)b * S * H + hh * dh;
  T* dq = reinterpret_cast<T*>(a.dqkv) + (size_t)b * S * 3 * H + hh * dh;
  const float* lse = a.lse + (size_t)bh * S;
  const float* D = a.Dscratch + (size_t)bh * S;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* P = Y2 + CB * lds + warp * 8 * LP;  // [4][LP] P and [4][LP] dS of this warp
  float* dS = P + 4 * LP;

  load_rows<T>(X1, keys ? q + H : q, 3 * H, S, r0, RB, dh, a.rope, a.rope_theta);
  if (keys) load_rows<T>(X2, q + 2 * H, 3 * H, S, r0, RB, dh, false, 0.f);
  else load_rows<T>(X2, dO, H, S, r0, RB, dh, false, 0.f);
  float o1[4][MAXD / 32], o2[4][MAXD / 32], rl[4], rd[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int row = r0 + warp * 4 + r;
    rl[r] = !keys && row < S ? lse[row] : 0.f;
    rd[r] = !keys && row < S ? D[row] : 0.f;
#pragma unroll
    for (int c = 0; c < MAXD / 32; ++c) o1[r][c] = o2[r][c] = 0.f;
  }
  const int begin = keys && a.causal ? r0 / CB * CB : 0;
  const int end = !keys && a.causal ? min(S, r0 + RB) : S;
  for (int c0 = begin; c0 < end; c0 += CB) {
    __syncthreads();
    load_rows<T>(Y1, keys ? q : q + H, 3 * H, S, c0, CB, dh, a.rope, a.rope_theta);
    if (keys) load_rows<T>(Y2, dO, H, S, c0, CB, dh, false, 0.f);
    else load_rows<T>(Y2, q + 2 * H, 3 * H, S, c0, CB, dh, false, 0.f);
    float cl[2], cd[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int col = c0 + lane + 32 * c;
      cl[c] = keys && col < S ? lse[col] : 0.f;
      cd[c] = keys && col < S ? D[col] : 0.f;
    }
    __syncthreads();
    float s[4][2], dp[4][2];
    scores(X1 + warp * 4 * lds, Y1, dh, lane, s);
    scores(X2 + warp * 4 * lds, Y2, dh, lane, dp);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int row = r0 + warp * 4 + r;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int col = c0 + lane + 32 * c;
        // key <= query
        const bool live = row < S && col < S && (!a.causal || (keys ? row <= col : col <= row));
        const float p = live ? expf(s[r][c] * a.scale - (keys ? cl[c] : rl[r])) : 0.f;
        P[r * LP + lane + 32 * c] = p;
        dS[r * LP + lane + 32 * c] = p * (dp[r][c] - (keys ? cd[c] : rd[r])) * a.scale;
      }
    }
    __syncwarp();
    accumulate(dS, Y1, dh, lane, o1);
    if (keys) accumulate(P, Y2, dh, lane, o2);
  }
  __syncwarp();
  store_rows<T>(keys ? dq + H : dq, 3 * H, o1, P, r0 + warp * 4, S, dh, lane, a.rope, a.rope_theta);
  if (keys) store_rows<T>(dq + 2 * H, 3 * H, o2, P, r0 + warp * 4, S, dh, lane, false, 0.f);
}

template <typename T>
cudaError_t fwd_impl(const AttnArgs& a, cudaStream_t st) {
  auto bytes = [](int dh) { return ((size_t)(RB + 2 * CB) * (dh + 4) + RB * LP) * sizeof(float); };
  const size_t smem = bytes(a.head_dim);
  cudaError_t e = allow_smem(attn_fwd_kernel<T>, (int)bytes(MAXD));
  if (e != cudaSuccess) return e;
  e = launch_pdl(attn_fwd_kernel<T>, dim3((a.S + RB - 1) / RB, a.B * a.n_heads), dim3(AT), smem, st, a);
  note_launch(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T>
cudaError_t bwd_impl(const AttnArgs& a, cudaStream_t st) {
  int T_ = a.B * a.S;
  int64_t warps = (int64_t)T_ * a.n_heads;
  cudaError_t le;
  if (a.dtype == DT_BF16 && (a.head_dim == 64 || a.head_dim == 128)) {
    const int G = a.head_dim / 8;
    const unsigned blocks = (unsigned)((warps * G + 255) / 256);
    le = G == 8 ? launch_pdl(attn_bwd_pre_vec_kernel<8>, dim3(blocks), dim3(256), (size_t)0, st, a)
                : launch_pdl(attn_bwd_pre_vec_kernel<16>, dim3(blocks), dim3(256), (size_t)0, st, a);
  } else {
    le = launch_pdl(attn_bwd_pre_kernel<T>, dim3((unsigned)((warps * 32 + 255) / 256)), dim3(256),
                    (size_t)0, st, a);
  }
  note_launch(1);
  if (le != cudaSuccess) return le;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (attention_mma_ok(a)) return attention_bwd_mma(a, st);
  auto bytes = [](int dh) { return ((size_t)2 * (RB + CB) * (dh + 4) + 2 * RB * LP) * sizeof(float); };
  const size_t smem = bytes(a.head_dim);
  e = allow_smem(attn_bwd_kernel<T>, (int)bytes(MAXD));
  if (e != cudaSuccess) return e;
  e = launch_pdl(attn_bwd_kernel<T>, dim3((a.S + RB - 1) / RB, a.B * a.n_heads, 2), dim3(AT), smem, st, a);
  note_launch(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t attention_fwd(const AttnArgs& a, cudaStream_t st) {
  if (a.head_dim > MAXD || a.head_dim % 32 != 0) return cudaErrorInvalidValue;
  if (attention_mma_ok(a)) return attention_fwd_mma(a, st);
  return a.dtype == DT_BF16 ? fwd_impl<bf16>(a, st) : fwd_impl<float>(a, st);
}

cudaError_t attention_bwd(const AttnArgs& a, cudaStream_t st) {
  if (a.head_dim > MAXD || a.head_dim % 32 != 0) return cudaErrorInvalidValue;
  return a.dtype == DT_BF16 ? bwd_impl<bf16>(a, st) : bwd_impl<float>(a, st);
}

}  // namespace ra

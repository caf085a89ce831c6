// k_adapter_simt.cu -- the adapter (Eq. 1) in fp32 arithmetic on the CUDA cores: the fp32 models,
// the stand-alone adapter backward, and the bf16 models whose bottleneck or width the
// tensor-core kernels do not take (their weights and GELU(z) stay fp32 here).
//
//   forward   z = a W_down; v = resid + a + GELU(z) W_up; LayerNorm / RMSNorm / nothing
//   backward  dz = (g W_up^T) GELU'(z); dh = g + dz W_down^T
//   dW        per row-chunk partials of dW_up = GELU(z)^T g and dW_down^T = dz^T h
//
// Both row kernels are two skinny products per row tile, 4 T H m flops against 12 to 16 T H bytes.  No unit is at
// its limit (4096 x 768, m = 64, backward rows: FFMA pipe 33 % and shared-memory path 30 % busy, an instruction
// issued in 46 % of the cycles): the chain of copy, product and reduction of 16 warps an SM sets the time.
// One CTA of 16 warps takes R = 4 TR rows:
//   phase 1  [R, m] = X[R, H] W[H, m]: the warps split H; a lane holds TR x TC sums (4 lane rows
//            x 8 lane columns, packed fp32x2 FMAs, which leave issue slots for the shared loads);
//            the 16 partial tiles are summed in warp order;
//   phase 2  [R, H] = S[R, m] W'[m, H]: the warps split H in 32-column tiles.
// Each warp copies its own operands through a ring of 8-deep chunks (2 to 4 in flight): loads straight
// to registers left the warps waiting for L2 (7.2 of 8.4 stall cycles an instruction, 58 us below).
// TR is the largest that still gives three quarters of the SMs a CTA, so a small batch is spread
// over many SMs by rows and the weights are read from L2 by fewer CTAs when it is large.
// Measured (one row per warp pair and scalar loads before): 4608 x 768, m = 48, bf16 rows,
// forward 485 -> 45 us, backward rows 240 -> 29 us; fp32 4096 x 768, m = 64, backward rows
// 200 -> 33 us; fp32 128 x 128, m = 16, forward 31 -> 5.4 us.
#include "common.cuh"
#include "kernels.h"
#include "simt.cuh"

namespace ra {
namespace {

constexpr int NW = 16, NT = NW * 32;

template <typename T>
__device__ __forceinline__ float4 ld4v(const T* p);
template <>
__device__ __forceinline__ float4 ld4v<float>(const float* p) {
  return __ldg(reinterpret_cast<const float4*>(p));
}
template <>
__device__ __forceinline__ float4 ld4v<bf16>(const bf16* p) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st4v(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void st4v(bf16* p, float4 v) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b));
}
// elements [c, c + 4) of a row of n elements: one access where `vec` (n and the base a multiple of 4
// elements, so c < n has all four), else one by one; zero beyond n
template <typename T>
__device__ __forceinline__ float4 ld4(const T* row, int c, int n, bool vec) {
  if (vec) return c < n ? ld4v(row + c) : make_float4(0.f, 0.f, 0.f, 0.f);
  float4 v;
  v.x = c < n ? to_f(row[c]) : 0.f;
  v.y = c + 1 < n ? to_f(row[c + 1]) : 0.f;
  v.z = c + 2 < n ? to_f(row[c + 2]) : 0.f;
  v.w = c + 3 < n ? to_f(row[c + 3]) : 0.f;
  return v;
}
template <typename T>
__device__ __forceinline__ void st4(T* row, int c, int n, bool vec, float4 v) {
  if (vec) {
    if (c < n) st4v(row + c, v);
    return;
  }
  if (c < n) row[c] = from_f<T>(v.x);
  if (c + 1 < n) row[c + 1] = from_f<T>(v.y);
  if (c + 2 < n) row[c + 2] = from_f<T>(v.z);
  if (c + 3 < n) row[c + 3] = from_f<T>(v.w);
}

// Shared memory (bytes): [0, s) first the warps' copy rings, then the phase 1 partials [NW][R][MP], then
// the rows v [R][ldv] (forward with a norm) -- and the phase 2 rings behind them; [s, total) GELU(z) or
// dz [R][MP + 4].  Rows 4 floats (mod 32) apart put the four lane rows' 16-byte reads into distinct banks.
template <typename TX, int TR, int TC>
struct Plan {
  static constexpr int R = 4 * TR, MP = 8 * TC, KC = 8;
  static constexpr int LDX = sizeof(TX) == 4 ? KC + 4 : KC;        // elements
  static constexpr int XB = R * LDX * (int)sizeof(TX), STAGE = XB + KC * MP * 4;
  static constexpr int NS = MP > 64 ? 2 : 3, RING = NW * NS * STAGE;
  static constexpr int NS2 = 4, STAGE2 = KC * 32 * 4, RING2 = NW * NS2 * STAGE2;
  static constexpr int PART = NW * R * MP * 4, LDS = MP + 4;
  int ldv, v, s, total;
  __host__ __device__ Plan(int H, bool keep_v) {
    ldv = (H + 31) / 32 * 32 + 4;
    v = keep_v ? R * ldv * 4 : 0;
    s = RING > PART ? RING : PART;
    if (v + RING2 > s) s = v + RING2;
    total = s + R * LDS * 4;
  }
};

struct RowsArgs {
  int T, H, m, ks;        // ks: columns of H per warp in phase 1 (a multiple of 4)
  bool vx, vm, vh;        // 4-element accesses: rows of X; rows of m floats; rows of H floats
  const void* X;          // [T, H]: the adapter input a (type TX), or g (f32)
  const float* W1;        // [H, m]: W_down, or W_up^T
  const float* W2;        // [m, H]: W_up, or W_down^T
  AdapterFwdArgs f;       // forward operands
  const float* z;         // backward: [T, m]
  float* dz;              // backward: [T, m]
  void* dh;               // backward: [T, H] or null
};

// TX: type of X; TO: type of the outputs (forward: y and xhat; backward: dh)
template <typename TX, typename TO, bool FWD, int TR, int TC>
__global__ void __launch_bounds__(NT, 1) adapter_rows_simt_kernel(RowsArgs p) {
  using Pl = Plan<TX, TR, TC>;
  constexpr int R = Pl::R, MP = Pl::MP, LDS = Pl::LDS, KC = Pl::KC;
  extern __shared__ __align__(16) uint8_t smb[];
  pdl_wait();
  pdl_trigger();
  const int H = p.H, m = p.m;
  const bool norm = FWD && !p.f.no_norm;
  const Pl L(H, norm);
  float* part = reinterpret_cast<float*>(smb);
  float* V = part;
  float* S = reinterpret_cast<float*>(smb + L.s);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int lr = lane >> 3, lc = lane & 7;  // lane row (rows lr + 4 i) and lane column (columns 4 lc + 32 g)
  const int t0 = blockIdx.x * R;
  const TX* X = reinterpret_cast<const TX*>(p.X);

  // ---- phase 1: this warp's columns [k0, k1) of H
  const int k0 = warp * p.ks, k1 = min(H, k0 + p.ks), n1 = k0 < k1 ? (k1 - k0 + KC - 1) / KC : 0;
  float2 acc[TR][TC / 2];
#pragma unroll
  for (int i = 0; i < TR; ++i)
#pragma unroll
    for (int c = 0; c < TC / 2; ++c) acc[i][c] = make_float2(0.f, 0.f);
  {
    uint8_t* ring = smb + warp * Pl::NS * Pl::STAGE;
    auto issue = [&](int n) {
      if (n < n1) {
        uint8_t* st = ring + (n % Pl::NS) * Pl::STAGE;
        const int k = k0 + n * KC;
        copy_block(reinterpret_cast<TX*>(st), Pl::LDX, X + (size_t)t0 * H + k, (size_t)H, R, KC, p.T - t0, k1 - k, p.vx, lane);
        copy_block(reinterpret_cast<float*>(st + Pl::XB), MP, p.W1 + (size_t)k * m, (size_t)m, KC, MP, k1 - k, m, p.vm, lane);
      }
      cp_commit();
    };
    for (int n = 0; n < Pl::NS - 1; ++n) issue(n);
#pragma unroll 1
    for (int n = 0; n < n1; ++n) {
      cp_wait<Pl::NS - 2>();
      __syncwarp();
      issue(n + Pl::NS - 1);  // (its stage was read before the last __syncwarp)
      const uint8_t* st = ring + (n % Pl::NS) * Pl::STAGE;
      const TX* xs = reinterpret_cast<const TX*>(st);
      const float* ws = reinterpret_cast<const float*>(st + Pl::XB);
#pragma unroll
      for (int kq = 0; kq < KC; kq += 4) {
        float4 x[TR];
#pragma unroll
        for (int i = 0; i < TR; ++i) x[i] = ld4s(xs + (lr + 4 * i) * Pl::LDX + kq);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int g = 0; g < TC / 4; ++g) {
            const float4 b = *reinterpret_cast<const float4*>(ws + (kq + kk) * MP + 4 * lc + 32 * g);
#pragma unroll
            for (int i = 0; i < TR; ++i) {
              const float2 a = f2(kk == 0 ? x[i].x : kk == 1 ? x[i].y : kk == 2 ? x[i].z : x[i].w);
              acc[i][2 * g] = __ffma2_rn(a, make_float2(b.x, b.y), acc[i][2 * g]);
              acc[i][2 * g + 1] = __ffma2_rn(a, make_float2(b.z, b.w), acc[i][2 * g + 1]);
            }
          }
      }
    }
    cp_wait<0>();
  }
  __syncthreads();  // every ring is read: the partials take their place
  if (n1 > 0) {
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
      for (int g = 0; g < TC / 4; ++g)
        *reinterpret_cast<float4*>(part + (warp * R + lr + 4 * i) * MP + 4 * lc + 32 * g) =
            make_float4(acc[i][2 * g].x, acc[i][2 * g].y, acc[i][2 * g + 1].x, acc[i][2 * g + 1].y);
  }
  __syncthreads();
  const int nk = (H + p.ks - 1) / p.ks;  // warps that took part
  for (int e = threadIdx.x; e < R * MP; e += NT) {
    const int r = e / MP, j = e % MP, t = t0 + r;
    float s = 0.f;
    if (j < m) {
      for (int w = 0; w < nk; ++w) s += part[(w * R + r) * MP + j];
      if (FWD) {
        if (p.f.z && t < p.T) p.f.z[(size_t)t * m + j] = s;
        s = gelu_f(s);
      } else if (t < p.T) {
        s *= gelu_grad_f(p.z[(size_t)t * m + j]);
        p.dz[(size_t)t * m + j] = s;
      }
    }
    S[r * LDS + j] = s;
  }
  if (!FWD && !p.dh) return;
  __syncthreads();

  // ---- phase 2: 32-column tiles of H, warp by warp, one stream of chunks over all of them
  const int nj = (m + KC - 1) / KC, n_tiles = (H + 31) / 32;
  const int n2 = warp < n_tiles ? (n_tiles - warp + NW - 1) / NW * nj : 0;
  uint8_t* ring = smb + L.v + warp * Pl::NS2 * Pl::STAGE2;
  int it = 0, ij = 0, iw = 0;  // the next chunk to copy: tile, chunk of the tile, stage
  auto issue = [&]() {
    if (it * NW + warp < n_tiles) {
      const int c = (it * NW + warp) * 32, j = ij * KC;
      copy_block(reinterpret_cast<float*>(ring + iw * Pl::STAGE2), 32, p.W2 + (size_t)j * H + c, (size_t)H, KC, 32, m - j, H - c, p.vh, lane);
      if (++ij == nj) { ij = 0; ++it; }
    }
    cp_commit();
    iw = (iw + 1) % Pl::NS2;
  };
  for (int n = 0; n < Pl::NS2 - 1; ++n) issue();
  int n = 0;
  for (int c0 = warp * 32; n < n2; c0 += NW * 32) {
    const int c = c0 + 4 * lc;
    float2 o[TR][2];
#pragma unroll
    for (int i = 0; i < TR; ++i) o[i][0] = o[i][1] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int q = 0; q < nj; ++q, ++n) {
      cp_wait<Pl::NS2 - 2>();
      __syncwarp();
      issue();
      const float* ws = reinterpret_cast<const float*>(ring + (n % Pl::NS2) * Pl::STAGE2) + 4 * lc;
#pragma unroll
      for (int jq = 0; jq < KC; jq += 4) {
        float4 b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) b[u] = *reinterpret_cast<const float4*>(ws + (jq + u) * 32);
#pragma unroll
        for (int i = 0; i < TR; ++i) {
          const float4 s = *reinterpret_cast<const float4*>(S + (lr + 4 * i) * LDS + q * KC + jq);  // zero from m on
          const float sv[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            o[i][0] = __ffma2_rn(f2(sv[u]), make_float2(b[u].x, b[u].y), o[i][0]);
            o[i][1] = __ffma2_rn(f2(sv[u]), make_float2(b[u].z, b[u].w), o[i][1]);
          }
        }
      }
    }
    const float (*acc)[4] = reinterpret_cast<const float (*)[4]>(o);
#pragma unroll
    for (int i = 0; i < TR; ++i) {
      const int r = lr + 4 * i, t = t0 + r;
      if (t >= p.T) continue;
      const size_t row = (size_t)t * H;
      const float4 x = ld4(X + row, c, H, p.vx);
      float4 v = make_float4(x.x + acc[i][0], x.y + acc[i][1], x.z + acc[i][2], x.w + acc[i][3]);
      if (FWD && p.f.resid) {
        const float4 q = p.f.decoder ? ld4(reinterpret_cast<const float*>(p.f.resid) + row, c, H, p.vh)
                                     : ld4(reinterpret_cast<const TX*>(p.f.resid) + row, c, H, p.vx);
        v = make_float4(q.x + x.x + acc[i][0], q.y + x.y + acc[i][1], q.z + x.z + acc[i][2], q.w + x.w + acc[i][3]);
      }
      if (norm) *reinterpret_cast<float4*>(V + r * L.ldv + c) = v;  // (columns past H: padding of the row)
      else st4(reinterpret_cast<TO*>(FWD ? p.f.y : p.dh) + row, c, H, p.vx && p.vh, v);
    }
  }
  if (!norm) return;
  __syncthreads();

  // ---- the norm of each row, a warp per row
  const AdapterFwdArgs& f = p.f;
  for (int r = warp; r < R; r += NW) {
    const int t = t0 + r;
    if (t >= p.T) break;
    const float* v = V + r * L.ldv;
    const size_t row = (size_t)t * H;
    TO* y = reinterpret_cast<TO*>(f.y) + row;
    const bool vo = p.vx && p.vh;
    if (!f.decoder) {
      float s = 0.f;
      for (int i = lane; i < H; i += 32) s += v[i];
      const float mu = warp_sum(s) / H;
      float q = 0.f;
      for (int i = lane; i < H; i += 32) { const float d = v[i] - mu; q += d * d; }
      const float rstd = rsqrtf(warp_sum(q) / H + f.eps);
      TO* xh = f.xhat ? reinterpret_cast<TO*>(f.xhat) + row : nullptr;
      for (int c = 4 * lane; c < H; c += 128) {
        const float4 x = *reinterpret_cast<const float4*>(v + c);
        const float4 h = make_float4((x.x - mu) * rstd, (x.y - mu) * rstd, (x.z - mu) * rstd, (x.w - mu) * rstd);
        const float4 gm = ld4(f.gamma, c, H, p.vh), bt = ld4(f.beta, c, H, p.vh);
        st4(y, c, H, vo, make_float4(h.x * gm.x + bt.x, h.y * gm.y + bt.y, h.z * gm.z + bt.z, h.w * gm.w + bt.w));
        if (xh) st4(xh, c, H, vo, h);
      }
      if (f.rstd && lane == 0) f.rstd[t] = rstd;
    } else {
      float q = 0.f;
      for (int i = lane; i < H; i += 32) q += v[i] * v[i];
      const float rstd = rsqrtf(warp_sum(q) / H + f.eps);
      for (int c = 4 * lane; c < H; c += 128) {
        const float4 x = *reinterpret_cast<const float4*>(v + c);
        const float4 gm = ld4(f.gamma, c, H, p.vh);
        st4(f.x_out + row, c, H, p.vh, x);
        st4(y, c, H, vo, make_float4(x.x * rstd * gm.x, x.y * rstd * gm.y, x.z * rstd * gm.z, x.w * rstd * gm.w));
      }
      if (f.rstd && lane == 0) f.rstd[t] = rstd;
    }
  }
}

bool al(const void* p, size_t n) { return (reinterpret_cast<uintptr_t>(p) & (n - 1)) == 0; }

template <typename TX, typename TO, bool FWD, int TR, int TC>
cudaError_t launch_rows(RowsArgs& p, cudaStream_t st) {
  auto k = adapter_rows_simt_kernel<TX, TO, FWD, TR, TC>;
  const size_t smem = (size_t)Plan<TX, TR, TC>(p.H, FWD && !p.f.no_norm).total;
  cudaError_t e = allow_smem(k, MAX_DYNAMIC_SMEM);
  if (e != cudaSuccess) return e;
  e = launch_pdl(k, dim3((p.T + 4 * TR - 1) / (4 * TR)), dim3(NT), smem, st, p);
  note_launch(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename TX, typename TO, bool FWD>
cudaError_t rows_dispatch(RowsArgs& p, cudaStream_t st) {
  p.ks = ((p.H + NW - 1) / NW + 7) / 8 * 8;  // H split evenly over the warps, whole chunks each
  const bool keep_v = FWD && !p.f.no_norm;
  auto fits = [&](int tr, int tc) {
    const int smem = tc == 4   ? (tr == 8 ? Plan<TX, 8, 4>(p.H, keep_v).total : tr == 4 ? Plan<TX, 4, 4>(p.H, keep_v).total
                                                                                        : Plan<TX, 2, 4>(p.H, keep_v).total)
                     : tc == 8 ? (tr == 8 ? Plan<TX, 8, 8>(p.H, keep_v).total : tr == 4 ? Plan<TX, 4, 8>(p.H, keep_v).total
                                                                                        : Plan<TX, 2, 8>(p.H, keep_v).total)
                               : (tr == 4 ? Plan<TX, 4, 16>(p.H, keep_v).total : Plan<TX, 2, 16>(p.H, keep_v).total);
    return smem <= MAX_DYNAMIC_SMEM;
  };
  const int tc = p.m <= 32 ? 4 : p.m <= 64 ? 8 : 16, sms = device_sm_count();
  int tr = tc == 16 ? 4 : 8;
  while (tr > 1 && ((p.T + 4 * tr - 1) / (4 * tr) * 4 < 3 * sms || !fits(tr, tc))) tr >>= 1;
#define RA_ROWS(TR, TC) return launch_rows<TX, TO, FWD, TR, TC>(p, st)
  if (tc == 4) {
    switch (tr) { case 8: RA_ROWS(8, 4); case 4: RA_ROWS(4, 4); case 2: RA_ROWS(2, 4); default: RA_ROWS(1, 4); }
  } else if (tc == 8) {
    switch (tr) { case 8: RA_ROWS(8, 8); case 4: RA_ROWS(4, 8); case 2: RA_ROWS(2, 8); default: RA_ROWS(1, 8); }
  } else {
    switch (tr) { case 4: RA_ROWS(4, 16); case 2: RA_ROWS(2, 16); default: RA_ROWS(1, 16); }
  }
#undef RA_ROWS
}

// ---------------------------------------------------------------------------------------
// Weight-gradient partials over a chunk of rows, one product per CTA (blockIdx.z = 0: GELU(z)^T g ->
// pWu [m][H]; 1: dz^T h -> pWdT [m][H]): 64 bottleneck columns x 64 columns of H, 128 threads, a
// thread holds 8 x 4 sums (packed FMAs); 16 rows at a time staged in shared memory, the next 16 in
// registers meanwhile.  Per row a thread does 32 FMAs for three 16-byte shared loads (the kernel this
// replaces: 32 for 33 scalar loads, and always for 128 columns).  4096 x 768, m = 64: 180 -> 23 us.  8 x 8
// sums a thread on 64 x 128 tiles, with one or two groups of threads, took 29 to 38 us: too few warps.
// The sums run over a chunk's rows in order.
constexpr int DWJ = 64, DWI = 64, DWT = 16, DWN = 128;
template <typename T>
__global__ void __launch_bounds__(DWN) adapter_dw_simt_kernel(AdapterBwdArgs a, int chunk, bool vm, bool vh) {
  __shared__ __align__(16) float Xs[DWT][DWJ], Ys[DWT][DWI];
  pdl_wait();
  pdl_trigger();
  const int H = a.H, m = a.m, which = blockIdx.z;
  const int njt = (m + DWJ - 1) / DWJ;
  const int j0 = (blockIdx.x % njt) * DWJ, i0 = (blockIdx.x / njt) * DWI, c = blockIdx.y;
  const int tb = c * chunk, te = min(a.T, tb + chunk);
  const int tj = threadIdx.x >> 4, ti = threadIdx.x & 15;  // 8 columns j = 8 tj.., 4 columns i = 4 ti..
  const float* X = which ? a.dz : a.z;
  const T* h = reinterpret_cast<const T*>(a.h);
  constexpr int NL = DWT * DWJ / 4 / DWN;  // 16-byte groups per thread and tile
  float4 xr[NL], yr[NL];
  auto fetch = [&](int t0) {
#pragma unroll
    for (int q = 0; q < NL; ++q) {
      const int e = threadIdx.x + q * DWN, r = e >> 4, col = (e & 15) * 4, t = t0 + r;
      xr[q] = yr[q] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (t < te) {
        xr[q] = ld4(X + (size_t)t * m, j0 + col, m, vm);
        yr[q] = which ? ld4(h + (size_t)t * H, i0 + col, H, vh) : ld4(a.g + (size_t)t * H, i0 + col, H, vh);
      }
    }
  };
  float2 acc[8][2];
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
  if (tb < te) fetch(tb);
  for (int t0 = tb; t0 < te; t0 += DWT) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NL; ++q) {
      const int e = threadIdx.x + q * DWN, r = e >> 4, col = (e & 15) * 4;
      float4 x = xr[q];
      // (rows past the chunk hold zeros, and GELU(0) = 0)
      if (!which) x = make_float4(gelu_f(x.x), gelu_f(x.y), gelu_f(x.z), gelu_f(x.w));
      *reinterpret_cast<float4*>(&Xs[r][col]) = x;
      *reinterpret_cast<float4*>(&Ys[r][col]) = yr[q];
    }
    __syncthreads();
    if (t0 + DWT < te) fetch(t0 + DWT);
#pragma unroll
    for (int r = 0; r < DWT; ++r) {
      const float4 x0 = *reinterpret_cast<const float4*>(&Xs[r][8 * tj]), x1 = *reinterpret_cast<const float4*>(&Xs[r][8 * tj + 4]);
      const float4 y = *reinterpret_cast<const float4*>(&Ys[r][4 * ti]);
      const float xv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        acc[j][0] = __ffma2_rn(f2(xv[j]), make_float2(y.x, y.y), acc[j][0]);
        acc[j][1] = __ffma2_rn(f2(xv[j]), make_float2(y.z, y.w), acc[j][1]);
      }
    }
  }
  float* out = a.partials + (size_t)c * 2 * H * m + (which ? (size_t)H * m : 0);
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (j0 + 8 * tj + j < m)
      st4(out + (size_t)(j0 + 8 * tj + j) * H, i0 + 4 * ti, H, vh,
          make_float4(acc[j][0].x, acc[j][0].y, acc[j][1].x, acc[j][1].y));
}

}  // namespace

cudaError_t adapter_fwd_simt(const AdapterFwdArgs& a, cudaStream_t st) {
  RowsArgs p{};
  p.T = a.T; p.H = a.H; p.m = a.m;
  p.X = a.a; p.W1 = a.Wd; p.W2 = a.Wu; p.f = a;
  const size_t es = dtype_size(a.dtype);
  p.vm = a.m % 4 == 0 && al(a.Wd, 16);
  p.vh = a.H % 4 == 0 && al(a.Wu, 16) && al(a.gamma, 16) && al(a.beta, 16) && al(a.x_out, 16) &&
         (!a.decoder || al(a.resid, 16));
  p.vx = a.H % (16 / es) == 0 && al(a.a, 16) && al(a.y, 4 * es) && al(a.xhat, 4 * es) &&
         (a.decoder || al(a.resid, 4 * es));
  return a.dtype == DT_BF16 ? rows_dispatch<bf16, bf16, true>(p, st) : rows_dispatch<float, float, true>(p, st);
}

cudaError_t adapter_bwd_simt(const AdapterBwdArgs& a, cudaStream_t st) {
  RowsArgs p{};
  p.T = a.T; p.H = a.H; p.m = a.m;
  p.X = a.g; p.W1 = a.WuT; p.W2 = a.WdT; p.z = a.z; p.dz = a.dz; p.dh = a.dh;
  p.vm = a.m % 4 == 0 && al(a.WuT, 16);
  p.vh = a.H % 4 == 0 && al(a.WdT, 16);
  p.vx = a.H % 4 == 0 && al(a.g, 16) && al(a.dh, 4 * dtype_size(a.dh_dtype));
  cudaError_t e = a.dh_dtype == DT_BF16 ? rows_dispatch<float, bf16, false>(p, st)
                                        : rows_dispatch<float, float, false>(p, st);
  if (e != cudaSuccess) return e;
  // four CTAs an SM in one wave (two products; with a fifth CTA on some SMs the launch takes a quarter longer)
  const int tiles = (a.H + DWI - 1) / DWI * ((a.m + DWJ - 1) / DWJ);
  const int nchunk = adapter_dw_chunks(a.T, a.H, tiles);
  const bool vm = a.m % 4 == 0 && al(a.z, 16) && al(a.dz, 16);
  const bool vh = a.H % 4 == 0 && al(a.g, 16) && al(a.h, 4 * dtype_size(a.dtype)) && al(a.partials, 16);
  const dim3 grid(tiles, nchunk, 2);
  const int chunk = (a.T + nchunk - 1) / nchunk;
  e = a.dtype == DT_BF16 ? launch_pdl(adapter_dw_simt_kernel<bf16>, grid, dim3(DWN), (size_t)0, st, a, chunk, vm, vh)
                         : launch_pdl(adapter_dw_simt_kernel<float>, grid, dim3(DWN), (size_t)0, st, a, chunk, vm, vh);
  note_launch(1);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return adapter_dw_reduce(a.partials, nchunk, a.H, a.m, a.dWd, a.dWu, st);
}

}  // namespace ra

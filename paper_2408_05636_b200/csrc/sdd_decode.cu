// Forward of a few token rows (plain decoding, the autoregressive drafter's evaluations, verification): weight-streaming
// kernels that start on their weights before the kernel ahead of them has finished.
//
// The products of such a forward are bound by the weights' way from HBM, 61 MB a block of the XL target, and by the chain of
// dependent launches in front of each of them.  A CTA here owns 16 to 48 output features (and, for the additive products, a
// share of K); its weight rows are one cp.async.bulk per row into shared memory, issued before the dependency wait, so the
// next kernels' weights stream while this one's activations are being produced.  For that to happen two or three CTAs have
// to fit an SM and a launch has to be one wave: with one 200 KB CTA an SM every launch waits for its own weights (one row of
// the XL target: 31 us a block instead of 23).  After the wait a kernel only fetches the activation rows, multiplies and stores.
// For one or two rows LayerNorm is part of the product that consumes it (every CTA normalises the rows it needs anyway: 6 KB a
// row), which makes five launches a block instead of seven; for more the rows take too much of the shared memory and of
// every CTA's time.
//
// The multiplication is mma.sync m16n8k16: 16 features x 8 columns x 16 of K.  tcgen05 has nothing to offer here -- a tile
// of 128 features would be fed at one SM's rate, and CTAs of few features are what spreads 4800 of them over 148 SMs -- and the
// tensor work is hidden under the weight stream.  The order of K inside a slice of 32 is permuted so that a lane's operands
// are 16 consecutive bytes of a weight row and of an activation row: lane t of a group of four takes elements 8t .. 8t+7, two
// MMAs use the first and the last four of them, for both operands alike.
// Normalised rows of the MLP and its hidden layer enter as hi/lo bf16 pairs, 16 significant bits.
#include <mutex>

#include "sdd_kernels.h"
#include "sdd_tc.cuh"

namespace sdd {
namespace dec {

using tc::mbar_expect_tx;
using tc::mbar_init;
using tc::mbar_try;
using tc::smem_u32;

constexpr int TOK = 8;                   // token rows = MMA N
constexpr int SMS = 148;

// weight rows in shared memory start 64 bytes (mod 128) apart: a quarter-warp of the operand loads covers two rows and all banks
__host__ __device__ constexpr int row_pitch(int k_elems) { return (k_elems * 2) % 128 == 0 ? k_elems * 2 + 64 : k_elems * 2; }

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void st_cluster(uint32_t cluster_addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_addr), "f"(v) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack(float a, float b) {
  __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&t);
}
// Weight rows f0 .. f0 + nr - 1, columns [k0, k0 + kn), to shared memory, the rows dealt out to the warps; before the dependency
// wait; all threads call it.  bar: completes once with the rows and `extra` bytes more.
template <int NW>
__device__ __forceinline__ void fetch_weights(uint32_t sw, uint32_t bar, const __nv_bfloat16* __restrict__ W, int f0, int nr, int K,
                                              int k0, int kn, uint32_t extra = 0) {
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(bar, (uint32_t)(nr * kn * 2) + extra);
  }
  __syncthreads();
  if (tc::elect_one()) {
    const int pitch = row_pitch(kn);
    for (int r = (int)(threadIdx.x >> 5); r < nr; r += NW) bulk_load(sw + r * pitch, W + (long long)(f0 + r) * K + k0, (uint32_t)(kn * 2), bar);
  }
  __syncwarp();
}
__device__ __forceinline__ bool wait_weights(uint32_t bar, int* status) {
  const long long t0 = clock64();
  while (!mbar_try(bar, 0u)) {
    if (clock64() - t0 > tc::WAIT_LIMIT_CYCLES) {
      if (status != nullptr) atomicCAS(status, DEV_OK, DEV_TIMEOUT);
      return false;
    }
  }
  return true;
}
// Element (row r, token c) of the CTA's tile, summed over the warps' partial tiles [NW][rows][cols]
template <int NW>
__device__ __forceinline__ float warp_tiles_sum(const float* red, int tile, int at) {
  float s = 0.f;
#pragma unroll
  for (int w = 0; w < NW; ++w) s += red[w * tile + at];
  return s;
}
// GELU as a hi/lo pair of bf16, or a fused QKV element: Q to out, K and V^T to the caches (verification positions)
__device__ __forceinline__ void store_gelu(__nv_bfloat16* out, __nv_bfloat16* out_lo, long long o, float v) {
  const float y = gelu_tanh(v);
  const __nv_bfloat16 yh = __float2bfloat16_rn(y);
  out[o] = yh;
  out_lo[o] = __float2bfloat16_rn(y - __bfloat162float(yh));
}
__device__ __forceinline__ void store_qkv(__nv_bfloat16* out, const QkvDst& qd, int N, int f, int c, float v) {
  const __nv_bfloat16 y = __float2bfloat16_rn(v);
  if (f < qd.d) {
    out[(long long)c * N + f] = y;
    return;
  }
  const int sb = c / qd.rows_per_seq, pos = qd.ctx_len[sb] - 1 + c - sb * qd.rows_per_seq;
  if (f < 2 * qd.d) {
    if (pos < qd.k_seq_rows) qd.k_dst[((long long)sb * qd.k_seq_rows + pos) * qd.d + f - qd.d] = y;
  } else if (pos < qd.vt_ld) {
    qd.vt_dst[((long long)sb * qd.d + f - 2 * qd.d) * qd.vt_ld + pos] = y;
  }
}

// ---------------------------------------------------------------------------------------------
// out = epilogue(LayerNorm(h) W^T + bias) for one or two rows of width K <= 2048; a CTA owns 16 features.
// qd.vt_dst != null: fused QKV; else GELU.  The rows are normalised by the whole CTA, WARPS / M warps to a row, and meet the
// MMAs as hi/lo pairs in shared memory, hi rows in columns 0 .. M - 1 and lo rows in columns M .. 2M - 1 of one MMA.  (In the
// lanes' own operand layout only the four lanes of a live token have work to do; the conversions of the whole warp took 2.3 us.)
// ---------------------------------------------------------------------------------------------
constexpr int WARPS = 8, THREADS = 32 * WARPS;

// partial tiles red[warp][16 features][8 columns] of W (16 rows in shared memory) times `ROWS` activation rows behind each other
template <int ROWS>
__device__ __forceinline__ void multiply_rows(bool ok, const uint8_t* w_s, const uint8_t* x_s, int pitch, int n_sl, float* red, int warp, int g,
                                              int t) {
  // two accumulators: a single chain would be bound by the latency of dependent MMAs
  float acc[4] = {0.f, 0.f, 0.f, 0.f}, acc2[4] = {0.f, 0.f, 0.f, 0.f};
  if (ok) {
    const bool live = g < ROWS;
    const uint8_t *wl = w_s + g * pitch + t * 16, *xl = x_s + (live ? g : 0) * pitch + t * 16;
#pragma unroll 2
    for (int s = warp; s < n_sl; s += WARPS) {
      const uint4 w0 = *reinterpret_cast<const uint4*>(wl + s * 64), w1 = *reinterpret_cast<const uint4*>(wl + 8 * pitch + s * 64);
      uint4 y = *reinterpret_cast<const uint4*>(xl + s * 64);
      if (!live) y = make_uint4(0, 0, 0, 0);
      mma16816(acc, w0.x, w1.x, w0.y, w1.y, y.x, y.y);
      mma16816(acc2, w0.z, w1.z, w0.w, w1.w, y.z, y.w);
    }
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) red[(warp * 16 + g + 8 * (e >> 1)) * TOK + 2 * t + (e & 1)] = acc[e] + acc2[e];
  __syncthreads();
}

template <int M>
__global__ void __launch_bounds__(THREADS, 3)
gemv_ln_kernel(const float* h, const float* __restrict__ ln_g, const float* __restrict__ ln_b,
               const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias, int K, int N,
               __nv_bfloat16* out, __nv_bfloat16* out_lo, const QkvDst qd, int* status) {
  constexpr int WPT = WARPS / M, NV = 16 / WPT;         // groups of four elements per lane: 128 * WPT * NV = 2048
  extern __shared__ __align__(128) uint8_t dyn[];
  __shared__ __align__(8) unsigned long long bar_s;
  __shared__ float red[WARPS * 16 * TOK];
  __shared__ float st_s[2][WARPS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int f0 = blockIdx.x * 16;
  const uint32_t bar = smem_u32(&bar_s), sw = smem_u32(dyn);
  const int pitch = row_pitch(K), w_bytes = 16 * pitch;
  const float* gain = reinterpret_cast<const float*>(dyn + w_bytes);          // [K] gain, [K] bias of the LayerNorm
  uint8_t* xs = dyn + w_bytes + 8 * K;                                        // [hi | lo][M] rows
  fetch_weights<WARPS>(sw, bar, W, f0, 16, K, 0, K, (uint32_t)(8 * K));
  if (threadIdx.x == 0) {
    bulk_load(sw + w_bytes, ln_g, (uint32_t)(4 * K), bar);
    bulk_load(sw + w_bytes + 4 * K, ln_b, (uint32_t)(4 * K), bar);
  }
  float bv = 0.f;
  if (threadIdx.x < 16 * TOK) bv = bias[f0 + (threadIdx.x >> 3)];
  pdl_launch_dependents();
  pdl_wait();

  const int tok = warp / WPT, part = warp % WPT;
  float4 x[NV];
  float sum = 0.f;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int e = ((i * WPT + part) * 32 + lane) * 4;
    x[i] = e < K ? *reinterpret_cast<const float4*>(h + (long long)tok * K + e) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll
  for (int i = 0; i < NV; ++i) sum += (x[i].x + x[i].y) + (x[i].z + x[i].w);
  auto row_sum = [&](float v, int which) {              // over the WPT warps of the row
    v = warp_sum(v);
    if (lane == 0) st_s[which][warp] = v;
    __syncthreads();
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < WPT; ++w) s += st_s[which][tok * WPT + w];
    return s;
  };
  const float mu = row_sum(sum, 0) / (float)K;
  float var = 0.f;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int e = ((i * WPT + part) * 32 + lane) * 4;
    if (e < K) {
      const float a = x[i].x - mu, b = x[i].y - mu, c = x[i].z - mu, dd = x[i].w - mu;
      var += (a * a + b * b) + (c * c + dd * dd);
    }
  }
  const float rstd = rsqrtf(row_sum(var, 1) / (float)K + 1e-5f);
  const bool ok = wait_weights(bar, status);            // gains and weights
  {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int e = ((i * WPT + part) * 32 + lane) * 4;
      if (e < K) {
        const float4 gg = *reinterpret_cast<const float4*>(gain + e), bb = *reinterpret_cast<const float4*>(gain + K + e);
        const float y0 = (x[i].x - mu) * rstd * gg.x + bb.x, y1 = (x[i].y - mu) * rstd * gg.y + bb.y;
        const float y2 = (x[i].z - mu) * rstd * gg.z + bb.z, y3 = (x[i].w - mu) * rstd * gg.w + bb.w;
        const uint32_t h0 = pack(y0, y1), h1 = pack(y2, y3);
        *reinterpret_cast<uint2*>(xs + tok * pitch + e * 2) = make_uint2(h0, h1);
        *reinterpret_cast<uint2*>(xs + (M + tok) * pitch + e * 2) =
            make_uint2(pack(y0 - __uint_as_float(h0 << 16), y1 - __uint_as_float(h0 & 0xffff0000u)),
                       pack(y2 - __uint_as_float(h1 << 16), y3 - __uint_as_float(h1 & 0xffff0000u)));
      }
    }
  }
  __syncthreads();

  multiply_rows<2 * M>(ok, dyn, xs, pitch, K / 32, red, warp, g, t);
  const int r = threadIdx.x >> 3, c = threadIdx.x & 7;
  if (r >= 16 || c >= M) return;
  const float v = warp_tiles_sum<WARPS>(red, 16 * TOK, r * TOK + c) + warp_tiles_sum<WARPS>(red, 16 * TOK, r * TOK + c + M) + bv;
  if (qd.vt_dst == nullptr) store_gelu(out, out_lo, (long long)c * N + f0 + r, v);
  else store_qkv(out, qd, N, f0 + r, c, v);
}

// ---------------------------------------------------------------------------------------------
// h += x W^T + bias for one or two rows of bf16, row stride K (LO: hi/lo pairs); a CTA owns 16 features and a share of K
// (grid.y).  The activations pass through shared memory, 16 bytes a thread, as columns of one MMA: one round trip to L2.
// Every share adds its part to h with one reduction per element, share 0 brings the bias.
// ---------------------------------------------------------------------------------------------
template <int M, bool LO>
__global__ void __launch_bounds__(THREADS, 3)
gemv_add_kernel(const __nv_bfloat16* xin, const __nv_bfloat16* xin_lo, const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias,
                int K, int N, float* h, int* status) {
  constexpr int ROWS = LO ? 2 * M : M;
  extern __shared__ __align__(128) uint8_t dyn[];
  __shared__ __align__(8) unsigned long long bar_s;
  __shared__ float red[WARPS * 16 * TOK];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int f0 = blockIdx.x * 16;
  const int all = K / 32, per = (all + (int)gridDim.y - 1) / (int)gridDim.y;
  const int s0 = (int)blockIdx.y * per, n_sl = min(per, all - s0);          // host: >= 1
  const uint32_t bar = smem_u32(&bar_s), sw = smem_u32(dyn);
  fetch_weights<WARPS>(sw, bar, W, f0, 16, K, s0 * 32, n_sl * 32);
  float bv = 0.f;
  if (threadIdx.x < 16 * TOK && blockIdx.y == 0) bv = bias[f0 + (threadIdx.x >> 3)];
  pdl_launch_dependents();
  pdl_wait();

  const int pitch = row_pitch(n_sl * 32);
  uint8_t* xs = dyn + 16 * pitch;
  for (int u = threadIdx.x; u < ROWS * n_sl * 4; u += THREADS) {
    const int row = u / (n_sl * 4), c16 = u - row * (n_sl * 4);
    const __nv_bfloat16* src = (LO && row >= M ? xin_lo + (long long)(row - M) * K : xin + (long long)row * K) + s0 * 32 + c16 * 8;
    *reinterpret_cast<uint4*>(xs + row * pitch + c16 * 16) = *reinterpret_cast<const uint4*>(src);
  }
  const bool ok = wait_weights(bar, status);
  __syncthreads();
  multiply_rows<ROWS>(ok, dyn, xs, pitch, n_sl, red, warp, g, t);
  const int r = threadIdx.x >> 3, c = threadIdx.x & 7;
  if (r >= 16 || c >= M) return;
  float v = warp_tiles_sum<WARPS>(red, 16 * TOK, r * TOK + c) + bv;
  if (LO) v += warp_tiles_sum<WARPS>(red, 16 * TOK, r * TOK + c + M);
  float* o = h + (long long)c * N + f0 + r;
  if (gridDim.y == 1) *o += v;
  else atomicAdd(o, v);
}

// ---------------------------------------------------------------------------------------------
// out = epilogue(x W^T + bias) for M <= 8 CG rows of bf16 (LO: hi/lo pairs), row stride K; a CTA owns 16 MT features and, in
// the additive form, a share of K (grid.y).  Activations go from L2 into the lanes' registers in operand layout, each once
// per CTA; a warp takes every WARPS-th slice of K, and the warps' partial tiles meet in the weights' shared memory.
// ---------------------------------------------------------------------------------------------
enum StreamOut : int { SO_ADD = 0, SO_GELU = 1, SO_QKV = 2 };

template <int MT, int CG, bool LO>
__global__ void __launch_bounds__(THREADS, MT == 1 && CG <= 2 ? 3 : MT <= 2 && CG <= 5 ? 2 : 1)
stream_kernel(const __nv_bfloat16* x, const __nv_bfloat16* x_lo, const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias, int M,
              int K, int N, int kind, void* out, __nv_bfloat16* out_lo, const QkvDst qd, int* status) {
  constexpr int R = 16 * MT, C = 8 * CG, TILE = R * C;
  extern __shared__ __align__(128) uint8_t dyn[];
  __shared__ __align__(8) unsigned long long bar_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int f0 = blockIdx.x * R, nr = min(R, N - f0);
  const int all = K / 32, per = (all + (int)gridDim.y - 1) / (int)gridDim.y;
  const int s0 = (int)blockIdx.y * per, n_sl = min(per, all - s0);          // host: >= 1
  const uint32_t bar = smem_u32(&bar_s), sw = smem_u32(dyn);
  const int pitch = row_pitch(n_sl * 32);
  fetch_weights<WARPS>(sw, bar, W, f0, nr, K, s0 * 32, n_sl * 32);
  pdl_launch_dependents();
  pdl_wait();

  float acc[MT][CG][4] = {};
  const uint8_t *wl[MT], *wh[MT];                       // rows past the last one repeat it
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    wl[i] = dyn + min(i * 16 + g, nr - 1) * pitch + t * 16;
    wh[i] = dyn + min(i * 16 + g + 8, nr - 1) * pitch + t * 16;
  }
  const long long xo = (long long)s0 * 32 + t * 8;
  auto load_x = [&](int s, uint4 (&hi)[CG], uint4 (&lo)[LO ? CG : 1]) {
#pragma unroll
    for (int j = 0; j < CG; ++j) {
      const int row = min(j * 8 + g, M - 1);            // columns past the last token repeat it; they are not stored
      const long long o = (long long)row * K + xo + s * 32;
      hi[j] = *reinterpret_cast<const uint4*>(x + o);
      if (LO) lo[LO ? j : 0] = *reinterpret_cast<const uint4*>(x_lo + o);
    }
  };
  // slices whose activations are in flight together (more of them spill: 8 at one column group cost 0.1 ms of a 1.2 ms step)
  constexpr int NB = MT == 3 ? (CG <= 4 ? 3 : CG <= 6 ? 2 : 1) : CG == 1 ? 4 : CG == 2 ? (LO ? 2 : 4) : CG == 5 && LO ? 1 : 2;
  bool ok = true, waited = false;
  for (int i0 = warp; i0 < n_sl; i0 += WARPS * NB) {
    uint4 hi[NB][CG], lo[LO ? NB : 1][LO ? CG : 1];
#pragma unroll
    for (int n = 0; n < NB; ++n)
      if (i0 + n * WARPS < n_sl) load_x(i0 + n * WARPS, hi[n], lo[LO ? n : 0]);
    if (!waited) { ok = wait_weights(bar, status); waited = true; }
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      const int s = i0 + n * WARPS;
      if (s < n_sl && ok) {
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          const uint4 w0 = *reinterpret_cast<const uint4*>(wl[i] + s * 64), w1 = *reinterpret_cast<const uint4*>(wh[i] + s * 64);
#pragma unroll
          for (int j = 0; j < CG; ++j) {
            mma16816(acc[i][j], w0.x, w1.x, w0.y, w1.y, hi[n][j].x, hi[n][j].y);
            mma16816(acc[i][j], w0.z, w1.z, w0.w, w1.w, hi[n][j].z, hi[n][j].w);
            if (LO) {
              const uint4& y = lo[LO ? n : 0][LO ? j : 0];
              mma16816(acc[i][j], w0.x, w1.x, w0.y, w1.y, y.x, y.y);
              mma16816(acc[i][j], w0.z, w1.z, w0.w, w1.w, y.z, y.w);
            }
          }
        }
      }
    }
  }
  if (!waited) wait_weights(bar, status);               // the copies land before the shared memory is used again
  __syncthreads();                                      // every warp is done with the weights: their memory takes the partial tiles
  // [warp][token][feature], a token's features consecutive
  float* red = reinterpret_cast<float*>(dyn);
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < CG; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) red[warp * TILE + (j * 8 + 2 * t + (e & 1)) * R + i * 16 + g + 8 * (e >> 1)] = acc[i][j][e];
  __syncthreads();
  for (int u = threadIdx.x; u < M * R; u += THREADS) {
    const int c = u / R, r = u - c * R, f = f0 + r;
    if (r >= nr) continue;
    float v = warp_tiles_sum<WARPS>(red, TILE, u);
    if (bias != nullptr && blockIdx.y == 0) v += bias[f];
    if (kind == SO_ADD) {
      float* o = reinterpret_cast<float*>(out) + (long long)c * N + f;
      if (gridDim.y == 1) *o += v;
      else atomicAdd(o, v);
    } else if (kind == SO_GELU) {
      store_gelu(reinterpret_cast<__nv_bfloat16*>(out), out_lo, (long long)c * N + f, v);
    } else {
      store_qkv(reinterpret_cast<__nv_bfloat16*>(out), qd, N, f, c, v);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// attention of R new rows of a sequence (positions ctx_len - 1 + r) over its KV cache, eight rows to a CTA; what further groups
// of rows read of the cache comes from L2 (33 rows of 25 heads, 512 keys: XL verification 2.99 -> 2.94 ms against one 128-row
// tcgen05 CTA a head that walks all keys; 9 rows 1.99 -> 1.86).  The keys of a head are dealt
// out in slices of 32 to a cluster of one, two or four CTAs (slice s to CTA s % S): what bounds the kernel is how fast an SM
// takes in its part of the cache (one CTA per head: 4.5 us at 512 keys), so the heads are spread over the chip.
// Scores are K (16 keys x 64) times Q^T (64 x 8 rows), the output V^T (16 features x keys) times P^T: both operands of both
// products come straight from the caches in 16-byte pieces (same permutation of the contracted index as above); scores
// and probabilities pass through shared memory.  Soft-max in fp32, probabilities in bf16 like the tcgen05 kernel's.
// ---------------------------------------------------------------------------------------------
constexpr int AT_WARPS = 8;

struct FewParams {
  const __nv_bfloat16* q;
  const __nv_bfloat16 *kc, *vt;
  __nv_bfloat16* out;
  const int* ctx_len;
  int q_ld, R, n_ctx, d, s_ld, splits, groups;
};

template <int R_MAX>
__global__ void __launch_bounds__(32 * AT_WARPS, 2)
attn_few_kernel(const FewParams p) {
  extern __shared__ __align__(128) uint8_t dyn[];
  const int n_ctx = p.n_ctx, d = p.d, S = p.splits;
  const int b = blockIdx.y / p.groups, r0 = (blockIdx.y - b * p.groups) * TOK, R = min(p.R - r0, R_MAX);     // rows r0 .. r0 + R - 1
  float* s_s = reinterpret_cast<float*>(dyn);                                 // [R][s_ld] scores of this CTA's keys
  __nv_bfloat16* s_p = reinterpret_cast<__nv_bfloat16*>(s_s + R * p.s_ld);    // [R][s_ld + 8] probabilities
  __shared__ float o_s[2][64][TOK];
  __shared__ float recv_o[4][64][R_MAX], recv_m[4][R_MAX], recv_l[4][R_MAX];  // partial states of the cluster's CTAs
  __shared__ float m_s[AT_WARPS], sum_s[AT_WARPS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int hd = blockIdx.x / S, rank = blockIdx.x % S;
  const __nv_bfloat16* kb = p.kc + (long long)b * n_ctx * d + hd * 64;
  const __nv_bfloat16* vh = p.vt + ((long long)b * d + hd * 64) * n_ctx;
  {
    // the cache of this layer has left L2 since the last step: ask for it while the kernel ahead is still at work (the length
    // may be out of date; only hints follow from it)
    const int seen = min(max(*reinterpret_cast<const volatile int*>(p.ctx_len + b), 0), n_ctx);
    for (int k = threadIdx.x; k < seen; k += 32 * AT_WARPS)
      if ((k >> 5) % S == rank) prefetch_l2(kb + (long long)k * d);
    for (int u = rank * 32 * AT_WARPS + threadIdx.x; u < 64 * ((seen + 63) / 64); u += S * 32 * AT_WARPS)
      prefetch_l2(vh + (long long)(u & 63) * n_ctx + (u >> 6) * 64);
  }
  pdl_launch_dependents();
  pdl_wait();
  const int c = p.ctx_len[b] + r0;                      // the first row's keys
  const int n_keys = min(c - 1 + R, n_ctx);
  const long long row0 = (long long)b * p.R + r0;
  uint4 qf[2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
    qf[i] = g < R ? *reinterpret_cast<const uint4*>(p.q + (row0 + g) * p.q_ld + hd * 64 + i * 32 + t * 8) : make_uint4(0, 0, 0, 0);
  const float scale = 0.125f * 1.4426950408889634f;                           // 1 / sqrt(64) * log2(e)
  // j: the CTA's 16-key tiles, two to a slice; slice i of the CTA is slice rank + S i of the sequence
  auto key_of = [&](int j) { return ((rank + S * (j >> 1)) * 2 + (j & 1)) * 16; };
  auto load_k = [&](int j, uint4 (&a)[4]) {             // positions past the last key: any row of the cache (masked below)
    const int k0 = key_of(j) + g;
    const __nv_bfloat16* r0 = kb + (long long)min(k0, n_ctx - 1) * d + t * 8;
    const __nv_bfloat16* r1 = kb + (long long)min(k0 + 8, n_ctx - 1) * d + t * 8;
    a[0] = *reinterpret_cast<const uint4*>(r0); a[1] = *reinterpret_cast<const uint4*>(r1);
    a[2] = *reinterpret_cast<const uint4*>(r0 + 32); a[3] = *reinterpret_cast<const uint4*>(r1 + 32);
  };
  auto scores = [&](int j, const uint4 (&a)[4]) {
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    mma16816(s, a[0].x, a[1].x, a[0].y, a[1].y, qf[0].x, qf[0].y);
    mma16816(s, a[0].z, a[1].z, a[0].w, a[1].w, qf[0].z, qf[0].w);
    mma16816(s, a[2].x, a[3].x, a[2].y, a[3].y, qf[1].x, qf[1].y);
    mma16816(s, a[2].z, a[3].z, a[2].w, a[3].w, qf[1].z, qf[1].w);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int row = 2 * t + (e & 1), kl = g + (e >> 1) * 8, kk = key_of(j) + kl;
      if (row < R) s_s[row * p.s_ld + j * 16 + kl] = kk <= c - 1 + row && kk < n_keys ? s[e] * scale : -INFINITY;
    }
  };
  // the first tiles of K and V are fetched before the length is known, together with it and Q: one round trip for all
  uint4 ka[2][4];
  load_k(warp, ka[0]);
  load_k(warp + AT_WARPS, ka[1]);
  // V^T tiles: warp = (feature tile of 16, half of the slices)
  const int mt = warp & 3, kq = warp >> 2;
  const __nv_bfloat16* vb = vh + (long long)(mt * 16 + g) * n_ctx + t * 8;
  auto load_v = [&](int i, uint4& v0, uint4& v1) {
    const int k0 = (rank + S * i) * 32;
    v0 = v1 = make_uint4(0, 0, 0, 0);
    if (k0 + t * 8 + 8 <= n_ctx) {
      v0 = *reinterpret_cast<const uint4*>(vb + k0);
      v1 = *reinterpret_cast<const uint4*>(vb + 8ll * n_ctx + k0);
    }
  };
  constexpr int PRE = 3;
  uint4 v0[PRE], v1[PRE];
#pragma unroll
  for (int i = 0; i < PRE; ++i) load_v(kq + 2 * i, v0[i], v1[i]);
  const int all = (n_keys + 31) / 32, n_sl = rank < all ? (all - rank + S - 1) / S : 0, n_t = 2 * n_sl;
  if (warp < n_t) scores(warp, ka[0]);
  if (warp + AT_WARPS < n_t) scores(warp + AT_WARPS, ka[1]);
  for (int j = warp + 2 * AT_WARPS; j < n_t; j += 2 * AT_WARPS) {
    load_k(j, ka[0]);
    load_k(j + AT_WARPS, ka[1]);
    scores(j, ka[0]);
    if (j + AT_WARPS < n_t) scores(j + AT_WARPS, ka[1]);
  }
  __syncthreads();
  // soft-max over the CTA's keys: AT_WARPS / R_MAX warps per row, merged through shared memory
  constexpr int WPR = AT_WARPS / R_MAX;
  const int row = warp / WPR, part = warp % WPR;
  const bool mine = row < R;
  const int n_loc = n_sl * 32;
  float mx = -INFINITY;
  if (mine)
    for (int k = part * 32 + lane; k < n_loc; k += WPR * 32) mx = fmaxf(mx, s_s[row * p.s_ld + k]);
  mx = warp_max(mx);
  if (WPR > 1) {
    if (lane == 0) m_s[warp] = mx;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < WPR; ++w) mx = fmaxf(mx, m_s[row * WPR + w]);
  }
  const float m_use = mx == -INFINITY ? 0.f : mx;       // no visible key among the CTA's
  float sum = 0.f;
  if (mine)
    for (int k = part * 32 + lane; k < n_loc; k += WPR * 32) {
      const float e = exp2f(s_s[row * p.s_ld + k] - m_use);
      sum += e;
      s_p[row * (p.s_ld + 8) + k] = __float2bfloat16_rn(e);
    }
  sum = warp_sum(sum);
  if (lane == 0) { m_s[warp] = mx; sum_s[warp] = sum; }
  __syncthreads();
  float o[2][4] = {};
  const __nv_bfloat16* pr = s_p + g * (p.s_ld + 8) + t * 8;
  auto pv = [&](int i, const uint4& a, const uint4& e) {
    if (i >= n_sl) return;
    const uint4 w = g < R ? *reinterpret_cast<const uint4*>(pr + i * 32) : make_uint4(0, 0, 0, 0);
    mma16816(o[0], a.x, e.x, a.y, e.y, w.x, w.y);
    mma16816(o[1], a.z, e.z, a.w, e.w, w.z, w.w);
  };
#pragma unroll
  for (int i = 0; i < PRE; ++i) pv(kq + 2 * i, v0[i], v1[i]);
  for (int i = kq + 2 * PRE; i < n_sl; i += 4) {
    load_v(i, v0[0], v1[0]);
    load_v(i + 2, v0[1], v1[1]);
    pv(i, v0[0], v1[0]);
    pv(i + 2, v0[1], v1[1]);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) o_s[kq][mt * 16 + g + 8 * (e >> 1)][2 * t + (e & 1)] = o[0][e] + o[1][e];
  __syncthreads();
  // every CTA hands its state to CTA 0 of the cluster, which adds them up
  for (int u = threadIdx.x; u < R * 64; u += 32 * AT_WARPS) {
    const int r = u >> 6, f = u & 63;
    const float x = o_s[0][f][r] + o_s[1][f][r];
    if (S == 1) recv_o[0][f][r] = x;
    else st_cluster(tc::map_to_cta(smem_u32(&recv_o[rank][f][r]), 0u), x);
    if (f == 0) {
      float l = 0.f;
      for (int w = 0; w < WPR; ++w) l += sum_s[r * WPR + w];
      float m = m_s[r * WPR];
      for (int w = 1; w < WPR; ++w) m = fmaxf(m, m_s[r * WPR + w]);
      if (S == 1) {
        recv_m[0][r] = m;
        recv_l[0][r] = l;
      } else {
        st_cluster(tc::map_to_cta(smem_u32(&recv_m[rank][r]), 0u), m);
        st_cluster(tc::map_to_cta(smem_u32(&recv_l[rank][r]), 0u), l);
      }
    }
  }
  if (S == 1) __syncthreads();
  else tc::cluster_sync_all();
  if (rank != 0) return;
  for (int u = threadIdx.x; u < R * 64; u += 32 * AT_WARPS) {
    const int r = u >> 6, f = u & 63;
    float m = -INFINITY, l = 0.f, x = 0.f;
    for (int w = 0; w < S; ++w) m = fmaxf(m, recv_m[w][r]);
    for (int w = 0; w < S; ++w) {
      const float e = exp2f(recv_m[w][r] - m);          // CTA without a visible key: exp2(-inf) = 0
      l = fmaf(recv_l[w][r], e, l);
      x = fmaf(recv_o[w][f][r], e, x);
    }
    p.out[(row0 + r) * d + hd * 64 + f] = __float2bfloat16_rn(x / l);
  }
}

constexpr int SMEM_MAX = 220 * 1024;
static int ln_smem(int M, int K) { return (16 + 2 * M) * row_pitch(K) + 8 * K; }
// (the last share of K may be shorter and its row pitch longer by the padding)
static int stream_smem(int R, int C, int per) {
  const int pitch = row_pitch(per * 32) > row_pitch(per * 32 - 32) ? row_pitch(per * 32) : row_pitch(per * 32 - 32);
  const int tiles = WARPS * R * C * 4;
  return R * pitch > tiles ? R * pitch : tiles;
}
static int scores_ld(int n_ctx, int S) { return ((n_ctx + 31) / 32 + S - 1) / S * 32 + 8; }   // keys of a CTA
static size_t attn_smem(int R, int n_ctx, int S) { return (size_t)R * (scores_ld(n_ctx, S) * 4 + (scores_ld(n_ctx, S) + 8) * 2); }
constexpr size_t ATTN_SMEM_MAX = 100 * 1024;            // two CTAs an SM

}  // namespace dec

cudaError_t prepare_decode() {
  using namespace dec;
  static std::once_flag once;
  static cudaError_t prep = cudaSuccess;
  std::call_once(once, [] {
    auto set = [](auto k, size_t bytes) {
      if (prep == cudaSuccess) prep = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    set(gemv_ln_kernel<1>, SMEM_MAX);
    set(gemv_ln_kernel<2>, SMEM_MAX);
    set(gemv_add_kernel<1, false>, SMEM_MAX); set(gemv_add_kernel<1, true>, SMEM_MAX);
    set(gemv_add_kernel<2, false>, SMEM_MAX); set(gemv_add_kernel<2, true>, SMEM_MAX);
    auto set2 = [&](auto k1, auto k2) { set(k1, SMEM_MAX); set(k2, SMEM_MAX); };
    set2(stream_kernel<1, 1, false>, stream_kernel<1, 1, true>);
    set2(stream_kernel<1, 2, false>, stream_kernel<1, 2, true>);
    set2(stream_kernel<2, 3, false>, stream_kernel<2, 3, true>);
    set2(stream_kernel<2, 4, false>, stream_kernel<2, 4, true>);
    set2(stream_kernel<2, 5, false>, stream_kernel<2, 5, true>);
    set2(stream_kernel<2, 6, false>, stream_kernel<2, 6, true>);
    set2(stream_kernel<2, 8, false>, stream_kernel<2, 8, true>);
    set2(stream_kernel<3, 3, false>, stream_kernel<3, 3, true>);
    set2(stream_kernel<3, 4, false>, stream_kernel<3, 4, true>);
    set2(stream_kernel<3, 5, false>, stream_kernel<3, 5, true>);
    set2(stream_kernel<3, 6, false>, stream_kernel<3, 6, true>);
    set(attn_few_kernel<1>, ATTN_SMEM_MAX);
    set(attn_few_kernel<2>, ATTN_SMEM_MAX);
    set(attn_few_kernel<8>, ATTN_SMEM_MAX);
  });
  return prep;
}

// Up to 64 rows while FC1 is one wave of 32-feature CTAs (width 1184), up to 48 beyond: there every CTA's own copy of the
// activations outweighs the weights' head start.  Against the tcgen05 kernels, 512 keys: 12 layers of width 768, 33 rows
// 0.70 -> 0.52 ms, 64 rows 0.89 -> 0.65; 24 of 1024, 64 rows 1.73 -> 1.36; 48 of 1600, 33 rows 3.22 -> 2.94, 48 rows
// 3.55 -> 3.40, but 49 rows 3.56 -> 3.86.
bool few_rows_fit(int M, int d, int d_head) {
  const bool one_wave = (4 * d + 31) / 32 <= dec::SMS;
  return M <= (one_wave ? 64 : 48) && d_head == 64 && d <= 2048;
}
// CTAs that share a head's keys: `key_splits` (by the context's length) while that is no more than one CTA an SM
int attn_few_splits(int batch, int R, int n_head, int key_splits) {
  const int groups = (R + dec::TOK - 1) / dec::TOK;
  while (key_splits > 1 && n_head * batch * groups * key_splits > dec::SMS) key_splits >>= 1;
  return key_splits;
}
bool attn_few_fits(int R, int n_ctx) { return (n_ctx & 7) == 0 && dec::attn_smem(R < dec::TOK ? R : dec::TOK, n_ctx, 1) <= dec::ATTN_SMEM_MAX; }

cudaError_t launch_gemv_ln(const float* h, const float* ln_g, const float* ln_b, const __nv_bfloat16* W, const float* bias, int M, int K,
                           int N, __nv_bfloat16* out, __nv_bfloat16* out_lo, const QkvDst* qkv, int* status, cudaStream_t st) {
  using namespace dec;
  if (M < 1 || M > 2 || (K % 32) != 0 || K > 2048 || (N % 16) != 0) return cudaErrorInvalidValue;
  cudaError_t e = prepare_decode();
  if (e != cudaSuccess) return e;
  QkvDst qd = {};
  if (qkv != nullptr) qd = *qkv;
  return launch_k(M == 1 ? gemv_ln_kernel<1> : gemv_ln_kernel<2>, dim3(N / 16), dim3(THREADS), (size_t)ln_smem(M, K), st, h, ln_g, ln_b, W,
                  bias, K, N, out, out_lo, qd, status);
}

cudaError_t launch_stream_gemm(const __nv_bfloat16* x, const __nv_bfloat16* x_lo, const __nv_bfloat16* W, const float* bias, int M, int K, int N,
                               int epi, void* out, __nv_bfloat16* out_lo, const QkvDst* qkv, int* status, cudaStream_t st) {
  using namespace dec;
  if (M < 1 || M > 64 || (K % 32) != 0 || N < 1 || (epi != EPI_RESIDUAL && epi != EPI_GELU && epi != EPI_QKV)) return cudaErrorInvalidValue;
  if ((epi == EPI_GELU && out_lo == nullptr) || (epi == EPI_QKV && qkv == nullptr)) return cudaErrorInvalidValue;
  cudaError_t e = prepare_decode();
  if (e != cudaSuccess) return e;
  QkvDst qd = {};
  if (qkv != nullptr) qd = *qkv;
  const int kind = epi == EPI_RESIDUAL ? SO_ADD : epi == EPI_GELU ? SO_GELU : SO_QKV;
  // up to 16 rows: 16 features a CTA; beyond, every CTA's own copy of the activations (2 M K or 4 M K bytes from L2) asks for 32
  const int cg = M <= 8 ? 1 : M <= 16 ? 2 : M <= 24 ? 3 : M <= 32 ? 4 : M <= 40 ? 5 : M <= 48 ? 6 : 8;
  // and for 48 where 32 would make more CTAs than SMs (XL verification of 33 rows: 3.03 -> 2.94 ms; where 32 features fill one
  // wave, 48 only idle SMs: 12 layers of width 768, 33 rows 0.54 -> 0.58 ms).  Additive products have K shares to fill the chip.
  const bool mt3 = cg >= 3 && cg <= 6 && kind != SO_ADD && (N + 31) / 32 > SMS;
  const int R = cg <= 2 ? 16 : mt3 ? 48 : 32, tiles = (N + R - 1) / R, all = K / 32;
  int ks = 1;
  if (kind == SO_ADD) {
    // K shares: about two CTAs an SM, at least 8 slices of 32 (one a warp) each, and three CTAs an SM in shared memory
    auto full = [&](int k) { return ((all + k - 1) / k) * (k - 1) < all; };        // no empty share
    ks = (2 * SMS + tiles - 1) / tiles;
    if (ks > all / 8) ks = all / 8;
    if (ks < 1) ks = 1;
    while (ks > 1 && !full(ks)) --ks;
    while (ks < all && (!full(ks) || stream_smem(R, 8 * cg, (all + ks - 1) / ks) > 72 * 1024)) ++ks;
  }
  if (M <= 2 && kind == SO_ADD && (N % 16) == 0) {
    const size_t sm = stream_smem(16 + (x_lo != nullptr ? 2 * M : M), 1, (all + ks - 1) / ks);
    if (sm <= SMEM_MAX) {
      auto add = M == 1 ? (x_lo != nullptr ? gemv_add_kernel<1, true> : gemv_add_kernel<1, false>)
                        : (x_lo != nullptr ? gemv_add_kernel<2, true> : gemv_add_kernel<2, false>);
      return launch_k(add, dim3(tiles, ks), dim3(THREADS), sm, st, x, x_lo, W, bias, K, N, reinterpret_cast<float*>(out), status);
    }
  }
  const size_t smem = stream_smem(R, 8 * cg, (all + ks - 1) / ks);
  if (smem > SMEM_MAX) return cudaErrorInvalidValue;
  auto go = [&](auto plain, auto pair) {
    return launch_k(x_lo != nullptr ? pair : plain, dim3(tiles, ks), dim3(THREADS), smem, st, x, x_lo, W, bias, M, K, N, kind, out, out_lo, qd,
                    status);
  };
  switch (cg) {
    case 1: return go(stream_kernel<1, 1, false>, stream_kernel<1, 1, true>);
    case 2: return go(stream_kernel<1, 2, false>, stream_kernel<1, 2, true>);
    case 3: return mt3 ? go(stream_kernel<3, 3, false>, stream_kernel<3, 3, true>) : go(stream_kernel<2, 3, false>, stream_kernel<2, 3, true>);
    case 4: return mt3 ? go(stream_kernel<3, 4, false>, stream_kernel<3, 4, true>) : go(stream_kernel<2, 4, false>, stream_kernel<2, 4, true>);
    case 5: return mt3 ? go(stream_kernel<3, 5, false>, stream_kernel<3, 5, true>) : go(stream_kernel<2, 5, false>, stream_kernel<2, 5, true>);
    case 6: return mt3 ? go(stream_kernel<3, 6, false>, stream_kernel<3, 6, true>) : go(stream_kernel<2, 6, false>, stream_kernel<2, 6, true>);
    default: return go(stream_kernel<2, 8, false>, stream_kernel<2, 8, true>);
  }
}

cudaError_t launch_attn_few(const __nv_bfloat16* q, int q_ld, const __nv_bfloat16* kc, const __nv_bfloat16* vt, __nv_bfloat16* out,
                            const int* ctx_len, int batch, int R, int n_ctx, int n_head, int key_splits, cudaStream_t st) {
  using namespace dec;
  cudaError_t e = prepare_decode();
  if (e != cudaSuccess) return e;
  FewParams p;
  p.q = q; p.q_ld = q_ld; p.kc = kc; p.vt = vt; p.out = out; p.ctx_len = ctx_len; p.R = R; p.n_ctx = n_ctx; p.d = n_head * 64;
  p.groups = (R + TOK - 1) / TOK;
  p.splits = attn_few_splits(batch, R, n_head, key_splits);
  p.s_ld = scores_ld(n_ctx, p.splits);
  const dim3 grid(n_head * p.splits, batch * p.groups), block(32 * AT_WARPS);
  const size_t smem = attn_smem(R < TOK ? R : TOK, n_ctx, p.splits);
  auto go = [&](auto kernel) {
    if (p.splits > 1) return launch_k_cluster(kernel, grid, block, smem, st, (unsigned)p.splits, p);
    return launch_k(kernel, grid, block, smem, st, p);
  };
  if (R == 1) return go(attn_few_kernel<1>);
  if (R == 2) return go(attn_few_kernel<2>);
  return go(attn_few_kernel<8>);
}

}  // namespace sdd

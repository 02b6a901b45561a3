// Forward of at most eight token rows (plain decoding, the autoregressive drafter's evaluations, short verifications):
// weight-streaming kernels that start on their weights before the kernel ahead of them has finished.
//
// The products of such a forward are bound by the weights' way from HBM, 61 MB a block of the XL target, and by the chain of
// dependent launches in front of each of them.  A CTA here owns 16 output features (and, for the additive products, a
// share of K), small enough for two or three CTAs an SM: its weight rows are one cp.async.bulk per row into shared
// memory, issued before the dependency wait, so the next kernels' weights stream while this one's activations are being
// produced.  After the wait a kernel only fetches the few activation rows, multiplies and stores.  LayerNorm is part of
// the product that consumes it (every CTA normalises the rows it needs anyway: 6 KB a row), which makes five launches a
// block instead of seven and leaves the normalised rows unrounded.
//
// The multiplication is mma.sync m16n8k16: 16 features x 8 token columns x 16 of K.  tcgen05 has nothing to offer here -- a
// tile of 128 x 8 would be fed at one SM's rate, and 16-feature CTAs are what spreads 4800 features over 148 SMs -- and
// the tensor work is hidden under the weight stream either way.  The order of K inside a slice of 32 is permuted so that a
// lane's operands are 16 consecutive bytes of a weight row and 8 consecutive activations: lane t of a group of four takes
// elements 8t .. 8t+7, two MMAs use the first and the last four of them, for both operands alike.
// fp32 activations (normalised rows, the MLP's hidden layer) enter as hi/lo bf16 pairs, 16 significant bits.
#include <mutex>

#include "sdd_kernels.h"
#include "sdd_tc.cuh"

namespace sdd {
namespace dec {

using tc::mbar_expect_tx;
using tc::mbar_init;
using tc::mbar_try;
using tc::smem_u32;

constexpr int ROWS = 16;                 // output features per CTA = MMA M
constexpr int TOK = 8;                   // token columns = MMA N
constexpr int WARPS = 8, THREADS = 32 * WARPS;

// weight rows in shared memory start 64 bytes (mod 128) apart: a quarter-warp of the operand loads covers two rows and all banks
__host__ __device__ constexpr int row_pitch(int k_elems) { return (k_elems * 2) % 128 == 0 ? k_elems * 2 + 64 : k_elems * 2; }
constexpr int weight_smem(int k_elems) { return ROWS * row_pitch(k_elems); }

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
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
// eight activations as packed hi and lo halves
__device__ __forceinline__ void split8(const float (&x)[8], uint32_t (&hi)[4], uint32_t (&lo)[4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    hi[e] = pack(x[2 * e], x[2 * e + 1]);
    lo[e] = pack(x[2 * e] - __uint_as_float(hi[e] << 16), x[2 * e + 1] - __uint_as_float(hi[e] & 0xffff0000u));
  }
}
__device__ __forceinline__ void load8(const float* p, float (&x)[8]) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}

// The CTA's 16 weight rows, columns [k0, k0 + kn), to shared memory; lanes 0..15 of warp 0, before the dependency wait.
// bar: one arrival + the bytes.
__device__ __forceinline__ void fetch_weights(uint32_t sw, uint32_t bar, const __nv_bfloat16* __restrict__ W, int f0, int K, int k0,
                                              int kn, int lane) {
  if (lane == 0) mbar_expect_tx(bar, (uint32_t)(ROWS * kn * 2));
  __syncwarp();
  if (lane < ROWS) bulk_load(sw + lane * row_pitch(kn), W + (long long)(f0 + lane) * K + k0, (uint32_t)(kn * 2), bar);
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
// acc += W[16 features, 32 of K] x[8 tokens, 32 of K]; sw_lane: row g of the slice at the lane's 16 bytes
template <bool LO>
__device__ __forceinline__ void slice_mma(float (&acc)[4], const uint8_t* sw_lane, int pitch, const uint32_t (&hi)[4], const uint32_t (&lo)[4]) {
  const uint4 w0 = *reinterpret_cast<const uint4*>(sw_lane), w1 = *reinterpret_cast<const uint4*>(sw_lane + 8 * pitch);
  mma16816(acc, w0.x, w1.x, w0.y, w1.y, hi[0], hi[1]);
  mma16816(acc, w0.z, w1.z, w0.w, w1.w, hi[2], hi[3]);
  if (LO) {
    mma16816(acc, w0.x, w1.x, w0.y, w1.y, lo[0], lo[1]);
    mma16816(acc, w0.z, w1.z, w0.w, w1.w, lo[2], lo[3]);
  }
}
// sum of the warps' 16 x 8 partial tiles; thread (feature f = tid >> 3, token = tid & 7) of the first 128 gets its element
__device__ __forceinline__ float reduce_tiles(const float (&acc)[4], float* red, int warp, int g, int t) {
  float* mine = red + warp * ROWS * TOK;
  mine[g * TOK + 2 * t] = acc[0];
  mine[g * TOK + 2 * t + 1] = acc[1];
  mine[(g + 8) * TOK + 2 * t] = acc[2];
  mine[(g + 8) * TOK + 2 * t + 1] = acc[3];
  __syncthreads();
  float s = 0.f;
  if (threadIdx.x < ROWS * TOK) {
#pragma unroll
    for (int w = 0; w < WARPS; ++w) s += red[w * ROWS * TOK + threadIdx.x];
  }
  return s;
}

// out = epilogue(LayerNorm(h) W^T + bias) for M <= 8 rows of width K <= 256 * NS.
// qd.vt_dst != null: fused QKV (Q to out_q, K and V^T to the caches); else GELU to out_f (fp32).
template <int NS>
__global__ void __launch_bounds__(THREADS, NS <= 4 ? 3 : 2)
gemv_ln_kernel(const float* h, const float* __restrict__ ln_g, const float* __restrict__ ln_b,
               const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias, int M, int K, int N,
               __nv_bfloat16* out_q, float* out_f, const QkvDst qd, int* status) {
  extern __shared__ __align__(128) uint8_t dyn[];
  __shared__ __align__(8) unsigned long long bar_s;
  __shared__ float red[WARPS * ROWS * TOK];
  __shared__ float st_s[2][WARPS][TOK];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int f0 = blockIdx.x * ROWS;
  const uint32_t bar = smem_u32(&bar_s), sw = smem_u32(dyn);
  if (warp == 0) {
    if (lane == 0) {
      mbar_init(bar, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    fetch_weights(sw, bar, W, f0, K, 0, K, lane);
  }
  const int n_sl = K / 32;                              // slices of 32 of K; slice s belongs to warp s % WARPS
  float bv = 0.f;
  if (threadIdx.x < ROWS * TOK) bv = bias[f0 + (threadIdx.x >> 3)];
  __syncthreads();
  pdl_launch_dependents();
  pdl_wait();

  float x[NS][8];
  float sum = 0.f;
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const int s = warp + i * WARPS;
#pragma unroll
    for (int e = 0; e < 8; ++e) x[i][e] = 0.f;
    if (s < n_sl && g < M) load8(h + (long long)g * K + s * 32 + t * 8, x[i]);
  }
#pragma unroll
  for (int i = 0; i < NS; ++i)
#pragma unroll
    for (int e = 0; e < 8; ++e) sum += x[i][e];
  sum += __shfl_xor_sync(0xffffffffu, sum, 1);
  sum += __shfl_xor_sync(0xffffffffu, sum, 2);
  if (t == 0) st_s[0][warp][g] = sum;
  __syncthreads();
  float mu = 0.f;
#pragma unroll
  for (int w = 0; w < WARPS; ++w) mu += st_s[0][w][g];
  mu /= (float)K;
  float var = 0.f;
#pragma unroll
  for (int i = 0; i < NS; ++i)
    if (warp + i * WARPS < n_sl) {
#pragma unroll
      for (int e = 0; e < 8; ++e) { const float c = x[i][e] - mu; var += c * c; }
    }
  var += __shfl_xor_sync(0xffffffffu, var, 1);
  var += __shfl_xor_sync(0xffffffffu, var, 2);
  if (t == 0) st_s[1][warp][g] = var;
  __syncthreads();
  var = 0.f;
#pragma unroll
  for (int w = 0; w < WARPS; ++w) var += st_s[1][w][g];
  const float rstd = rsqrtf(var / (float)K + 1e-5f);
  const bool live = g < M;

  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  const bool ok = wait_weights(bar, status);
  const int pitch = row_pitch(K);
  const uint8_t* wl = dyn + g * pitch + t * 16;
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const int s = warp + i * WARPS;
    if (s < n_sl && ok) {
      float gg[8], bb[8];
      load8(ln_g + s * 32 + t * 8, gg);
      load8(ln_b + s * 32 + t * 8, bb);
#pragma unroll
      for (int e = 0; e < 8; ++e) x[i][e] = live ? (x[i][e] - mu) * rstd * gg[e] + bb[e] : 0.f;
      uint32_t hi[4], lo[4];
      split8(x[i], hi, lo);
      slice_mma<true>(acc, wl + s * 64, pitch, hi, lo);
    }
  }
  const float v = reduce_tiles(acc, red, warp, g, t) + bv;
  const int f = f0 + (int)(threadIdx.x >> 3), c = threadIdx.x & 7;
  if (threadIdx.x >= ROWS * TOK || c >= M) return;
  if (qd.vt_dst == nullptr) {
    out_f[(long long)c * N + f] = gelu_tanh(v);
    return;
  }
  const __nv_bfloat16 y = __float2bfloat16_rn(v);
  if (f < qd.d) {
    out_q[(long long)c * N + f] = y;
    return;
  }
  const int sb = c / qd.rows_per_seq, pos = qd.ctx_len[sb] - 1 + c - sb * qd.rows_per_seq;
  if (f < 2 * qd.d) {
    if (pos < qd.k_seq_rows) qd.k_dst[((long long)sb * qd.k_seq_rows + pos) * qd.d + f - qd.d] = y;
  } else if (pos < qd.vt_ld) {
    qd.vt_dst[((long long)sb * qd.d + f - 2 * qd.d) * qd.vt_ld + pos] = y;
  }
}

// h += x W^T + bias for M <= 8 rows; x bf16 (attention output) or fp32 (hidden layer), row stride K.  grid = (N / 16, K
// shares): every share adds its part to h with one reduction per element, share 0 brings the bias.
template <bool F32>
__global__ void __launch_bounds__(THREADS, 3)
gemv_add_kernel(const void* xin, const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias, int M, int K, int N, float* h,
                int* status) {
  extern __shared__ __align__(128) uint8_t dyn[];
  __shared__ __align__(8) unsigned long long bar_s;
  __shared__ float red[WARPS * ROWS * TOK];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int f0 = blockIdx.x * ROWS;
  const int all = K / 32, per = (all + (int)gridDim.y - 1) / (int)gridDim.y;
  const int s0 = (int)blockIdx.y * per, n_sl = min(per, all - s0);          // host: >= 1
  const uint32_t bar = smem_u32(&bar_s), sw = smem_u32(dyn);
  if (warp == 0) {
    if (lane == 0) {
      mbar_init(bar, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    fetch_weights(sw, bar, W, f0, K, s0 * 32, n_sl * 32, lane);
  }
  float bv = 0.f;
  if (threadIdx.x < ROWS * TOK && blockIdx.y == 0) bv = bias[f0 + (threadIdx.x >> 3)];
  __syncthreads();
  pdl_launch_dependents();
  pdl_wait();

  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  const int pitch = row_pitch(n_sl * 32);
  const uint8_t* wl = dyn + g * pitch + t * 16;
  bool ok = true, waited = false;
  constexpr int UNR = 4;                                // slices whose activations are in flight together
  for (int i0 = warp; i0 < n_sl; i0 += WARPS * UNR) {
    uint32_t hi[UNR][4], lo[UNR][4];
#pragma unroll
    for (int u = 0; u < UNR; ++u) {
      const int s = i0 + u * WARPS;
      const bool in = s < n_sl && g < M;
      if (F32) {
        float x[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (in) load8(reinterpret_cast<const float*>(xin) + (long long)g * K + (s0 + s) * 32 + t * 8, x);
        split8(x, hi[u], lo[u]);
      } else {
        uint4 v = make_uint4(0, 0, 0, 0);
        if (in) v = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(xin) + (long long)g * K + (s0 + s) * 32 + t * 8);
        hi[u][0] = v.x; hi[u][1] = v.y; hi[u][2] = v.z; hi[u][3] = v.w;
        lo[u][0] = lo[u][1] = lo[u][2] = lo[u][3] = 0u;
      }
    }
    if (!waited) { ok = wait_weights(bar, status); waited = true; }
#pragma unroll
    for (int u = 0; u < UNR; ++u) {
      const int s = i0 + u * WARPS;
      if (s < n_sl && ok) slice_mma<F32>(acc, wl + s * 64, pitch, hi[u], lo[u]);
    }
  }
  if (!waited) wait_weights(bar, status);               // the copies have landed before the shared memory is given back
  const float v = reduce_tiles(acc, red, warp, g, t) + bv;
  const int f = f0 + (int)(threadIdx.x >> 3), c = threadIdx.x & 7;
  if (threadIdx.x >= ROWS * TOK || c >= M) return;
  float* o = h + (long long)c * N + f;
  if (gridDim.y == 1) *o += v;
  else atomicAdd(o, v);
}

// ---------------------------------------------------------------------------------------------
// attention of R <= 8 new rows of a sequence (positions ctx_len - 1 + r) over its KV cache; one CTA per head and sequence.
// Scores are K (16 keys x 64) times Q^T (64 x 8 rows), the output V^T (16 features x keys) times P^T: both operands of both
// products come straight from the caches in 16-byte pieces (same permutation of the contracted index as above); scores
// and probabilities pass through shared memory.  Soft-max in fp32, probabilities in bf16 like the tcgen05 kernel's.
// ---------------------------------------------------------------------------------------------
constexpr int AT_WARPS = 16;

template <int R_MAX>
__global__ void __launch_bounds__(32 * AT_WARPS, 2)
attn_few_kernel(const __nv_bfloat16* q, int q_ld, const __nv_bfloat16* kc, const __nv_bfloat16* vt, __nv_bfloat16* out,
                const int* ctx_len, int R, int n_ctx, int d, int s_ld) {
  extern __shared__ __align__(128) uint8_t dyn[];
  float* s_s = reinterpret_cast<float*>(dyn);                                 // [R][s_ld] scores
  __nv_bfloat16* s_p = reinterpret_cast<__nv_bfloat16*>(s_s + R * s_ld);      // [R][s_ld + 8] probabilities
  __shared__ float o_s[4][64][TOK];
  __shared__ float l_s[TOK];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int hd = blockIdx.x, b = blockIdx.y;
  pdl_launch_dependents();
  pdl_wait();
  const int c = ctx_len[b];
  const int n_keys = min(c - 1 + R, n_ctx);
  const __nv_bfloat16* kb = kc + (long long)b * n_ctx * d + hd * 64 + t * 8;
  uint4 qf[2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
    qf[i] = g < R ? *reinterpret_cast<const uint4*>(q + ((long long)b * R + g) * q_ld + hd * 64 + i * 32 + t * 8) : make_uint4(0, 0, 0, 0);
  const int n_kb = (n_keys + 15) / 16;
  const float scale = 0.125f * 1.4426950408889634f;                           // 1 / sqrt(64) * log2(e)
#pragma unroll 2
  for (int k16 = warp; k16 < n_kb; k16 += AT_WARPS) {
    const int key = k16 * 16 + g;
    const __nv_bfloat16* r0 = kb + (long long)min(key, n_keys - 1) * d;
    const __nv_bfloat16* r1 = kb + (long long)min(key + 8, n_keys - 1) * d;
    const uint4 a0 = *reinterpret_cast<const uint4*>(r0), a1 = *reinterpret_cast<const uint4*>(r1);
    const uint4 a2 = *reinterpret_cast<const uint4*>(r0 + 32), a3 = *reinterpret_cast<const uint4*>(r1 + 32);
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    mma16816(s, a0.x, a1.x, a0.y, a1.y, qf[0].x, qf[0].y);
    mma16816(s, a0.z, a1.z, a0.w, a1.w, qf[0].z, qf[0].w);
    mma16816(s, a2.x, a3.x, a2.y, a3.y, qf[1].x, qf[1].y);
    mma16816(s, a2.z, a3.z, a2.w, a3.w, qf[1].z, qf[1].w);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int row = 2 * t + (e & 1), kk = key + (e >> 1) * 8;
      if (row < R) s_s[row * s_ld + kk] = kk <= c - 1 + row && kk < n_keys ? s[e] * scale : -INFINITY;
    }
  }
  // V^T tiles: warp = (feature tile of 16, key quarter); the first slices are fetched while the soft-max runs
  const int mt = warp & 3, kq = warp >> 2;
  const __nv_bfloat16* vb = vt + ((long long)b * d + hd * 64 + mt * 16 + g) * n_ctx + t * 8;
  const int n_sl = (n_keys + 31) / 32;
  auto load_v = [&](int sl, uint4& v0, uint4& v1) {
    v0 = v1 = make_uint4(0, 0, 0, 0);
    if (sl < n_sl && sl * 32 + t * 8 + 8 <= n_ctx) {
      v0 = *reinterpret_cast<const uint4*>(vb + sl * 32);
      v1 = *reinterpret_cast<const uint4*>(vb + 8ll * n_ctx + sl * 32);
    }
  };
  constexpr int PRE = 4;
  uint4 v0[PRE], v1[PRE];
#pragma unroll
  for (int i = 0; i < PRE; ++i) load_v(kq + 4 * i, v0[i], v1[i]);
  __syncthreads();
  // soft-max: 16 / R_MAX warps per row (R_MAX = 1: all sixteen), merged through shared memory
  constexpr int WPR = AT_WARPS / R_MAX;
  __shared__ float m_s[AT_WARPS], sum_s[AT_WARPS];
  const int row = warp / WPR, part = warp % WPR;
  const bool mine = row < R;
  const int pad = n_sl * 32;
  float mx = -INFINITY;
  if (mine)
    for (int k = part * 32 + lane; k < n_keys; k += WPR * 32) mx = fmaxf(mx, s_s[row * s_ld + k]);
  mx = warp_max(mx);
  if (lane == 0) m_s[warp] = mx;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < WPR; ++w) mx = fmaxf(mx, m_s[row * WPR + w]);
  float sum = 0.f;
  if (mine)
    for (int k = part * 32 + lane; k < pad; k += WPR * 32) {
      const float p = k < n_keys ? exp2f(s_s[row * s_ld + k] - mx) : 0.f;
      sum += p;
      s_p[row * (s_ld + 8) + k] = __float2bfloat16_rn(p);
    }
  sum = warp_sum(sum);
  if (lane == 0) sum_s[warp] = sum;
  __syncthreads();
  if (threadIdx.x < R) {
    float l = 0.f;
#pragma unroll
    for (int w = 0; w < WPR; ++w) l += sum_s[threadIdx.x * WPR + w];
    l_s[threadIdx.x] = l;
  }
  float o[4] = {0.f, 0.f, 0.f, 0.f};
  const __nv_bfloat16* pr = s_p + g * (s_ld + 8) + t * 8;
  auto pv = [&](int sl, const uint4& a, const uint4& e) {
    if (sl >= n_sl) return;
    const uint4 p = g < R ? *reinterpret_cast<const uint4*>(pr + sl * 32) : make_uint4(0, 0, 0, 0);
    mma16816(o, a.x, e.x, a.y, e.y, p.x, p.y);
    mma16816(o, a.z, e.z, a.w, e.w, p.z, p.w);
  };
#pragma unroll
  for (int i = 0; i < PRE; ++i) pv(kq + 4 * i, v0[i], v1[i]);
  for (int sl = kq + 4 * PRE; sl < n_sl; sl += 8) {
    uint4 a[2], e[2];
    load_v(sl, a[0], e[0]);
    load_v(sl + 4, a[1], e[1]);
    pv(sl, a[0], e[0]);
    pv(sl + 4, a[1], e[1]);
  }
  o_s[kq][mt * 16 + g][2 * t] = o[0];
  o_s[kq][mt * 16 + g][2 * t + 1] = o[1];
  o_s[kq][mt * 16 + g + 8][2 * t] = o[2];
  o_s[kq][mt * 16 + g + 8][2 * t + 1] = o[3];
  __syncthreads();
  const int r = threadIdx.x >> 6, f = threadIdx.x & 63;
  if (r < R)
    out[((long long)b * R + r) * d + hd * 64 + f] = __float2bfloat16_rn((o_s[0][f][r] + o_s[1][f][r] + o_s[2][f][r] + o_s[3][f][r]) / l_s[r]);
}

static int scores_ld(int n_ctx) { return (n_ctx + 31) / 32 * 32 + 8; }
static size_t attn_smem(int R, int n_ctx) { return (size_t)R * (scores_ld(n_ctx) * 4 + (scores_ld(n_ctx) + 8) * 2); }
constexpr size_t ATTN_SMEM_MAX = 112 * 1024;            // two CTAs an SM

}  // namespace dec

cudaError_t prepare_decode() {
  using namespace dec;
  static std::once_flag once;
  static cudaError_t prep = cudaSuccess;
  std::call_once(once, [] {
    auto set = [](auto k, size_t bytes) {
      if (prep == cudaSuccess) prep = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    set(gemv_ln_kernel<4>, weight_smem(1024));
    set(gemv_ln_kernel<8>, weight_smem(2048));
    set(gemv_add_kernel<false>, weight_smem(2048));
    set(gemv_add_kernel<true>, weight_smem(2048));
    set(attn_few_kernel<1>, ATTN_SMEM_MAX);
    set(attn_few_kernel<2>, ATTN_SMEM_MAX);
    set(attn_few_kernel<8>, ATTN_SMEM_MAX);
  });
  return prep;
}

bool decode_fits(int batch, int rows_per_seq, int d, int d_head, int n_ctx) {
  return batch * rows_per_seq <= dec::TOK && d_head == 64 && d <= 2048 && (n_ctx & 7) == 0 &&
         dec::attn_smem(rows_per_seq, n_ctx) <= dec::ATTN_SMEM_MAX;
}

cudaError_t launch_gemv_ln(const float* h, const float* ln_g, const float* ln_b, const __nv_bfloat16* W, const float* bias, int M, int K,
                           int N, __nv_bfloat16* out_q, float* out_f, const QkvDst* qkv, int* status, cudaStream_t st) {
  using namespace dec;
  if (M < 1 || M > TOK || (K % 32) != 0 || K > 2048 || (N % ROWS) != 0) return cudaErrorInvalidValue;
  cudaError_t e = prepare_decode();
  if (e != cudaSuccess) return e;
  QkvDst qd = {};
  if (qkv != nullptr) qd = *qkv;
  if (K <= 1024)
    return launch_k(gemv_ln_kernel<4>, dim3(N / ROWS), dim3(THREADS), weight_smem(K), st, h, ln_g, ln_b, W, bias, M, K, N, out_q, out_f, qd, status);
  return launch_k(gemv_ln_kernel<8>, dim3(N / ROWS), dim3(THREADS), weight_smem(K), st, h, ln_g, ln_b, W, bias, M, K, N, out_q, out_f, qd, status);
}

cudaError_t launch_gemv_add(const void* x, bool x_f32, const __nv_bfloat16* W, const float* bias, int M, int K, int N, float* h,
                            int* status, cudaStream_t st) {
  using namespace dec;
  if (M < 1 || M > TOK || (K % 32) != 0 || (N % ROWS) != 0) return cudaErrorInvalidValue;
  cudaError_t e = prepare_decode();
  if (e != cudaSuccess) return e;
  // K shares: about two CTAs an SM, at least 8 slices of 32 (one a warp) each, at most 2048 of K in shared memory
  const int all = K / 32, tiles = N / ROWS;
  int ks = (2 * 148 + tiles - 1) / tiles;
  if (ks > all / 8) ks = all / 8;
  if (ks < (K + 2047) / 2048) ks = (K + 2047) / 2048;
  if (ks < 1) ks = 1;
  while (ks > 1 && ((all + ks - 1) / ks) * (ks - 1) >= all) --ks;           // no empty share
  const int per = (all + ks - 1) / ks;
  if (per * 32 > 2048) return cudaErrorInvalidValue;
  const size_t smem = weight_smem(per * 32) > weight_smem(per * 32 - 32) ? weight_smem(per * 32) : weight_smem(per * 32 - 32);
  if (x_f32)
    return launch_k(gemv_add_kernel<true>, dim3(tiles, ks), dim3(THREADS), smem, st, x, W, bias, M, K, N, h, status);
  return launch_k(gemv_add_kernel<false>, dim3(tiles, ks), dim3(THREADS), smem, st, x, W, bias, M, K, N, h, status);
}

cudaError_t launch_attn_few(const __nv_bfloat16* q, int q_ld, const __nv_bfloat16* kc, const __nv_bfloat16* vt, __nv_bfloat16* out,
                            const int* ctx_len, int batch, int R, int n_ctx, int n_head, cudaStream_t st) {
  using namespace dec;
  cudaError_t e = prepare_decode();
  if (e != cudaSuccess) return e;
  const dim3 grid(n_head, batch), block(32 * AT_WARPS);
  const size_t smem = attn_smem(R, n_ctx);
  const int ld = scores_ld(n_ctx), d = n_head * 64;
  if (R == 1) return launch_k(attn_few_kernel<1>, grid, block, smem, st, q, q_ld, kc, vt, out, ctx_len, R, n_ctx, d, ld);
  if (R == 2) return launch_k(attn_few_kernel<2>, grid, block, smem, st, q, q_ld, kc, vt, out, ctx_len, R, n_ctx, d, ld);
  return launch_k(attn_few_kernel<8>, grid, block, smem, st, q, q_ld, kc, vt, out, ctx_len, R, n_ctx, d, ld);
}

}  // namespace sdd

// Attention of the configurations without a tensor-core attention kernel (fp32; bf16 with d_head 32):
//   bidirectional (drafter): softmax(Q K^T / sqrt(d_head)) V over all rows of the sequence, no mask
//   cached causal (target) : row at position p attends to KV-cache positions 0..p
//
// One CTA owns 32 query rows of one head; K and V tiles of 128 keys are double-buffered in shared memory (cp.async) and
// shared out over eight warps, 16 keys each.  A warp is an online soft-max of its own over its keys -- a lane holds 4 rows x
// 4 keys of the scores and 4 rows x d_head / 4 columns of the output in registers, probabilities move between the four
// lanes of a row by shuffles -- and the eight states are merged once at the end.  Bound by FMA issue: 2048 FMAs to 190
// shared-memory reads a warp and tile, about 2.5 us a tile.  (One warp per query row, every key row read from L2 by every
// row: 564 us a layer at 12 heads x 315 rows; this kernel: 23.)
#include <mutex>

#include "sdd_kernels.h"

namespace sdd {

constexpr int FA_Q = 32, FA_K = 128, FA_WARPS = 8, FA_THREADS = 32 * FA_WARPS;
constexpr int FA_KW = FA_K / FA_WARPS;                       // keys of a tile per warp

template <typename T> struct FaPad;                          // row padding: rows start 16 bytes (mod 128) apart
template <> struct FaPad<float> { static constexpr int v = 4; };
template <> struct FaPad<__nv_bfloat16> { static constexpr int v = 8; };
template <typename T, int DH> constexpr int fa_row() { return DH + FaPad<T>::v; }
template <typename T, int DH> constexpr int fa_smem() {
  constexpr int tiles = 2 * 2 * FA_K * fa_row<T, DH>() * (int)sizeof(T);
  constexpr int merge = FA_WARPS * FA_Q * (DH + 4) * 4;      // the warps' states, over the tiles
  return (tiles > merge ? tiles : merge) + FA_Q * fa_row<float, DH>() * 4 + 2 * FA_WARPS * FA_Q * 4;
}

template <typename T> __device__ __forceinline__ float4 load4(const T* p);
template <> __device__ __forceinline__ float4 load4<float>(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <> __device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// q: row 0 of the CTA's query rows (row stride q_ld), head's columns; k / v: key 0 (row stride kv_ld); rows past n_q are
// not stored; query row i sees keys 0 .. min(n_keys, limit0 + i * limit_step) - 1
template <typename T, int DH>
__device__ __forceinline__ void attn_rows(const T* q, long long q_ld, const T* k, const T* v,
                                          long long kv_ld, int n_q, int n_keys, int limit0, int limit_step, T* __restrict__ out,
                                          int out_ld) {
  constexpr int ROW = fa_row<T, DH>(), QROW = fa_row<float, DH>(), PER16 = 16 / (int)sizeof(T), COLS = DH / 4;
  extern __shared__ __align__(16) uint8_t fa_raw[];
  T* tiles = reinterpret_cast<T*>(fa_raw);                   // [2 buffers][K | V][FA_K][ROW]
  float* qs = reinterpret_cast<float*>(fa_raw + fa_smem<T, DH>() - 2 * FA_WARPS * FA_Q * 4 - FA_Q * QROW * 4);
  float* s_m = qs + FA_Q * QROW;                             // [FA_WARPS][FA_Q]
  float* s_l = s_m + FA_WARPS * FA_Q;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int qi = lane >> 2, ki = lane & 3;                   // rows qi + 8 a; keys ki + 4 j; output columns 16 c + 4 ki
  auto fetch = [&](int t) {
    T* dst = tiles + (t & 1) * 2 * FA_K * ROW;
    for (int u = tid; u < 2 * FA_K * (DH / PER16); u += FA_THREADS) {
      const int row = u / (DH / PER16), c = (u % (DH / PER16)) * PER16;
      const int key = min(t * FA_K + (row & (FA_K - 1)), n_keys - 1);     // past the last key: any valid row (masked)
      cp_async16(dst + row * ROW + c, (row < FA_K ? k : v) + (long long)key * kv_ld + c);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(0);
  const float scale = rsqrtf((float)DH);
  for (int u = tid; u < FA_Q * (DH / 4); u += FA_THREADS) {
    const int row = u / (DH / 4), c = (u % (DH / 4)) * 4;
    float4 x = load4<T>(q + (long long)min(row, n_q - 1) * q_ld + c);
    x.x *= scale; x.y *= scale; x.z *= scale; x.w *= scale;
    *reinterpret_cast<float4*>(qs + row * QROW + c) = x;
  }
  float m[4], l[4], o[4][COLS];
  int lim[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    m[a] = -INFINITY;
    l[a] = 0.f;
    lim[a] = min(n_keys, limit0 + (qi + 8 * a) * limit_step);
#pragma unroll
    for (int c = 0; c < COLS; ++c) o[a][c] = 0.f;
  }
  const int n_tiles = (n_keys + FA_K - 1) / FA_K;
  for (int t = 0; t < n_tiles; ++t) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                         // tile t (and Q) is there; nobody still reads the other buffer
    if (t + 1 < n_tiles) fetch(t + 1);
    const int key0 = t * FA_K + warp * FA_KW;
    if (key0 >= n_keys) continue;                            // (warp-uniform; the barrier is at the top of the loop)
    const T* kt = tiles + (t & 1) * 2 * FA_K * ROW + warp * FA_KW * ROW;
    const T* vt = kt + FA_K * ROW;
    float s[4][4] = {};
#pragma unroll 4
    for (int e = 0; e < DH; e += 4) {
      float4 qa[4], kb[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) qa[a] = *reinterpret_cast<const float4*>(qs + (qi + 8 * a) * QROW + e);
#pragma unroll
      for (int j = 0; j < 4; ++j) kb[j] = load4<T>(kt + (ki + 4 * j) * ROW + e);
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          s[a][j] = fmaf(qa[a].x, kb[j].x, s[a][j]);
          s[a][j] = fmaf(qa[a].y, kb[j].y, s[a][j]);
          s[a][j] = fmaf(qa[a].z, kb[j].z, s[a][j]);
          s[a][j] = fmaf(qa[a].w, kb[j].w, s[a][j]);
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      float mx = -INFINITY;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (key0 + ki + 4 * j >= lim[a]) s[a][j] = -INFINITY;
        mx = fmaxf(mx, s[a][j]);
      }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float m_new = fmaxf(m[a], mx);
      const float m_use = m_new == -INFINITY ? 0.f : m_new;  // no visible key yet: every exponential below is zero
      const float corr = expf(m[a] - m_use);
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) { s[a][j] = expf(s[a][j] - m_use); sum += s[a][j]; }
      l[a] = l[a] * corr + sum;                              // this lane's keys only; the four lanes meet in the merge
      m[a] = m_new;
#pragma unroll
      for (int c = 0; c < COLS; ++c) o[a][c] *= corr;
    }
#pragma unroll
    for (int kk = 0; kk < FA_KW; ++kk) {                     // key kk: held by the lanes with ki == kk & 3, index kk >> 2
      float p[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) p[a] = __shfl_sync(0xffffffffu, s[a][kk >> 2], (lane & ~3) | (kk & 3));
#pragma unroll
      for (int c = 0; c < COLS / 4; ++c) {
        const float4 x = load4<T>(vt + kk * ROW + c * 16 + ki * 4);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          o[a][4 * c] = fmaf(p[a], x.x, o[a][4 * c]);
          o[a][4 * c + 1] = fmaf(p[a], x.y, o[a][4 * c + 1]);
          o[a][4 * c + 2] = fmaf(p[a], x.z, o[a][4 * c + 2]);
          o[a][4 * c + 3] = fmaf(p[a], x.w, o[a][4 * c + 3]);
        }
      }
    }
  }
  // merge: every warp leaves (m, l, o) of its 32 rows in shared memory, over the tiles
  __syncthreads();
  float* so = reinterpret_cast<float*>(fa_raw);              // [FA_WARPS][FA_Q][DH + 4]
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int row = warp * FA_Q + qi + 8 * a;
    float sum = l[a] + __shfl_xor_sync(0xffffffffu, l[a], 1);
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
    if (ki == 0) { s_m[row] = m[a]; s_l[row] = sum; }
#pragma unroll
    for (int c = 0; c < COLS / 4; ++c)
      *reinterpret_cast<float4*>(so + row * (DH + 4) + c * 16 + ki * 4) = make_float4(o[a][4 * c], o[a][4 * c + 1], o[a][4 * c + 2], o[a][4 * c + 3]);
  }
  __syncthreads();
  const int row = tid >> 3;
  if (row >= n_q) return;
  float mm = -INFINITY, ll = 0.f, w[FA_WARPS];
#pragma unroll
  for (int i = 0; i < FA_WARPS; ++i) mm = fmaxf(mm, s_m[i * FA_Q + row]);
#pragma unroll
  for (int i = 0; i < FA_WARPS; ++i) {
    w[i] = expf(s_m[i * FA_Q + row] - mm);                   // a warp without visible keys: exp(-inf) = 0
    ll = fmaf(s_l[i * FA_Q + row], w[i], ll);
  }
  const float inv = 1.f / ll;
#pragma unroll
  for (int c = 0; c < DH / 8; ++c) {
    const int e = (tid & 7) + 8 * c;
    float x = 0.f;
#pragma unroll
    for (int i = 0; i < FA_WARPS; ++i) x = fmaf(so[(i * FA_Q + row) * (DH + 4) + e], w[i], x);
    out[(long long)row * out_ld + e] = from_f32<T>(x * inv);
  }
}

template <typename T, int DH>
__global__ void __launch_bounds__(FA_THREADS)
attn_bidir_kernel(const T* qkv, T* __restrict__ out, const int* ctx_len, int gamma, int L_cap,
                  int n_head, const int* skip) {
  pdl_launch_dependents();
  pdl_wait();
  if (skip != nullptr && *skip) return;
  const int i0 = blockIdx.x * FA_Q, h = blockIdx.y, b = blockIdx.z;
  const int d = n_head * DH;
  const int L = ctx_len[b] + gamma;
  if (i0 >= L) return;                                       // padding rows are never read by valid ones; they stay as they are
  const long long row0 = (long long)b * L_cap;
  const T* base = qkv + row0 * 3 * d + h * DH;
  attn_rows<T, DH>(base + (long long)i0 * 3 * d, 3ll * d, base + d, base + 2 * d, 3ll * d, min(FA_Q, L - i0), L, L, 0,
                   out + (row0 + i0) * d + h * DH, d);
}

template <typename T, int DH>
__global__ void __launch_bounds__(FA_THREADS)
attn_cached_kernel(const T* qkv, const T* cache, T* __restrict__ out,
                   const int* ctx_len, int rows_per_seq, int mode, int n_ctx, int n_head) {
  pdl_launch_dependents();
  pdl_wait();
  const int j0 = blockIdx.x * FA_Q, h = blockIdx.y, b = blockIdx.z;
  const int d = n_head * DH;
  const int c = ctx_len[b];
  const long long row = (long long)b * rows_per_seq + j0;
  const int pos0 = mode == TARGET_VERIFY ? c - 1 + j0 : j0;  // position of the CTA's first row
  // rows past the last position (prefill: past the context; verify: past the table) do not exist
  int n_q = mode == TARGET_VERIFY ? min(rows_per_seq - j0, n_ctx - pos0) : min(rows_per_seq - j0, c - 1 - j0);
  n_q = min(n_q, FA_Q);
  if (n_q <= 0) return;
  const T* kb = cache + (long long)b * n_ctx * 2 * d + h * DH;
  attn_rows<T, DH>(qkv + row * 3 * d + h * DH, 3ll * d, kb, kb + d, 2ll * d, n_q, pos0 + n_q, pos0 + 1, 1, out + row * d + h * DH, d);
}

template <typename T>
static cudaError_t fa_prepare() {
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(attn_bidir_kernel<T, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, fa_smem<T, 64>())) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(attn_bidir_kernel<T, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, fa_smem<T, 32>())) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(attn_cached_kernel<T, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, fa_smem<T, 64>())) != cudaSuccess) return e;
  return cudaFuncSetAttribute(attn_cached_kernel<T, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, fa_smem<T, 32>());
}
cudaError_t prepare_attn() {
  static std::once_flag once;
  static cudaError_t prep = cudaSuccess;
  std::call_once(once, [] {
    prep = fa_prepare<float>();
    if (prep == cudaSuccess) prep = fa_prepare<__nv_bfloat16>();
  });
  return prep;
}

template <typename T>
cudaError_t launch_attn_bidir(const T* qkv, T* out, const int* ctx_len, int batch, int gamma, int L_cap, int n_head,
                              int d_head, cudaStream_t st, const int* skip) {
  cudaError_t e = prepare_attn();
  if (e != cudaSuccess) return e;
  const dim3 grid((L_cap + FA_Q - 1) / FA_Q, n_head, batch);
  if (d_head == 64) launch_k(attn_bidir_kernel<T, 64>, grid, dim3(FA_THREADS), fa_smem<T, 64>(), st, qkv, out, ctx_len, gamma, L_cap, n_head, skip);
  else if (d_head == 32) launch_k(attn_bidir_kernel<T, 32>, grid, dim3(FA_THREADS), fa_smem<T, 32>(), st, qkv, out, ctx_len, gamma, L_cap, n_head, skip);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_attn_cached(const T* qkv, const T* cache, T* out, const int* ctx_len, int batch, int rows_per_seq,
                               int mode, int n_ctx, int n_head, int d_head, cudaStream_t st) {
  if (rows_per_seq <= 0) return cudaSuccess;
  cudaError_t e = prepare_attn();
  if (e != cudaSuccess) return e;
  const dim3 grid((rows_per_seq + FA_Q - 1) / FA_Q, n_head, batch);
  if (d_head == 64)
    launch_k(attn_cached_kernel<T, 64>, grid, dim3(FA_THREADS), fa_smem<T, 64>(), st, qkv, cache, out, ctx_len, rows_per_seq, mode, n_ctx, n_head);
  else if (d_head == 32)
    launch_k(attn_cached_kernel<T, 32>, grid, dim3(FA_THREADS), fa_smem<T, 32>(), st, qkv, cache, out, ctx_len, rows_per_seq, mode, n_ctx, n_head);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

#define SDD_INSTANTIATE_ATTN(T)                                                                                  \
  template cudaError_t launch_attn_bidir<T>(const T*, T*, const int*, int, int, int, int, int, cudaStream_t,   \
                                            const int*);                                                       \
  template cudaError_t launch_attn_cached<T>(const T*, const T*, T*, const int*, int, int, int, int, int, int, \
                                             cudaStream_t);
SDD_INSTANTIATE_ATTN(float)
SDD_INSTANTIATE_ATTN(__nv_bfloat16)

}  // namespace sdd

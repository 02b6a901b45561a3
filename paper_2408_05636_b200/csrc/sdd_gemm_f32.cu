// fp32 GEMM for sm_100a on the bf16 tensor cores:  C[M, N] = A[M, K] * W[N, K]^T  with fp32 operands and results.
//
// Every fp32 operand element is split exactly into three bf16 terms, x = h + m + l (8 + 8 + 8 significant bits), and the
// product is the sum of the six bf16 products hh, hm, mh, mm, hl, lh; the three left out are about 2^-24 of |x||w|, the
// rounding of one fp32 addition.  The tensor core rounds its accumulator towards zero at every step, which adds
// up to a bias (measured on K = 3072: 3.2e-6 of the result against 5.0e-7 for a chain of fp32 FMAs), so the accumulator of
// the hh products only lives for 128 of K (8 steps) and is then added, rounded to nearest, to running sums in registers;
// the small products, 2^-8 of the result, keep one accumulator for the whole K range.  Relative 2-norm error against fp64:
// 1.4e-7 at K = 3072.
//
// One CTA: a 128 x BN tile.  Warp 0 brings fp32 tiles of 32 of K to a shared-memory ring by TMA, teams of four or eight warps
// split them -- the 128-row operand into tensor memory, the other into 64-byte-swizzled bf16 planes in shared memory --,
// warp 1 issues the MMAs, and the sixteen warps drain the accumulator of the chunk before while the next one is multiplied.
// What bounds it: a 128 x 128 x 32 block moves 136 KB through shared memory at 128 bytes a clock (208 KB when both operands
// went through it) and takes 1370 clocks; narrower tiles take 840 to 990, which is the round trip of a stage through TMA,
// splitting and MMA.  4096 x 4096 x 1024: 179 TFLOP/s; 384 x 3072 x 768: 15 us (CUDA-core kernel before: 90 us).
//
// Orientation as in sdd_gemm_tc.cu: NORMAL puts the activation rows on the MMA M axis, SWAP (64 rows or fewer) the weight
// rows.  The K range of a tile may be shared out over a cluster of up to 8 CTAs, which fills the chip when there are few
// tiles: their partial tiles meet in distributed shared memory (each CTA adds up and stores its own slice of the tile's
// columns, in a fixed order, so results do not depend on timing) and every epilogue works under the split.
#include <cstdlib>
#include <mutex>

#include "sdd_kernels.h"
#include "sdd_tc.cuh"

namespace sdd {
namespace tc {

constexpr int FX_WARPS = 16;                          // warps that split, accumulate and store
constexpr int FX_THREADS = 64 + 32 * FX_WARPS;        // warp 0: TMA, warp 1: MMA + TMEM owner
constexpr int FX_BK = 32;                             // 32 fp32 = one 128-byte row of the fp32 ring
constexpr int FX_CHUNK = 4;                           // k-blocks per life of an accumulator
constexpr int FX_PAD = 129;                           // rows per column group of the exchange area (conflict-free both ways)

template <int BN> constexpr int fx_f32_bytes() { return (128 + BN) * 128; }
template <int BN> constexpr int fx_bf16_bytes() { return 3 * BN * 64; }
template <int BN> constexpr int fx_f32_stages() { return BN == 128 ? 4 : 6; }
// tensor memory: two hh accumulators, one of the small products, 48 columns (three planes) of the A operand per stage
template <int BN> constexpr int fx_bf16_stages() { return BN == 128 ? 2 : 6; }
// teams of warps that split alternate k-blocks: as many as there are stages for, since a team's waits and fences cost more
// than its arithmetic (128 x 32 tiles: 930 clocks a k-block with two teams)
template <int BN> constexpr int fx_teams() { return BN == 128 ? 2 : 4; }
template <int BN> constexpr int fx_bar_off() {
  return fx_f32_stages<BN>() * fx_f32_bytes<BN>() + fx_bf16_stages<BN>() * fx_bf16_bytes<BN>();
}
template <int BN> constexpr int fx_smem() { return fx_bar_off<BN>() + 256 + 1024; }

// K-major, 64-byte swizzle: 8-row groups are 512 bytes apart
__device__ __forceinline__ uint64_t make_smem_desc64(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | (1ull << 16) | (32ull << 32) | (1ull << 46) | (4ull << 61);
}

__device__ __forceinline__ void tmem_ld8_issue(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(v[0]), "r"(v[1]),
               "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// MMA with the A operand in tensor memory (lane = row, two bf16 of K per column)
__device__ __forceinline__ void umma_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// ties registers loaded by tmem_ld8_issue to the wait in front of it
__device__ __forceinline__ void tmem_tie8(uint32_t (&v)[8]) {
  asm volatile("" : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7])::"memory");
}

// x = h + m + l for a pair of elements, packed bf16x2 (low half = first element).  Each term is the upper half of what is
// left of x, so the split is two masks, two exact subtractions and a byte permutation per packed pair; conversions
// (cvt.rn.bf16x2.f32) run at a quarter of that rate and bound the kernel when they did this (154 -> 290 TFLOP/s).
__device__ __forceinline__ void split_pair(float a, float b, uint32_t& h, uint32_t& m, uint32_t& l) {
  const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
  h = __byte_perm(ua, ub, 0x7632);
  const float ra = a - __uint_as_float(ua & 0xffff0000u), rb = b - __uint_as_float(ub & 0xffff0000u);
  const uint32_t va = __float_as_uint(ra), vb = __float_as_uint(rb);
  m = __byte_perm(va, vb, 0x7632);
  l = __byte_perm(__float_as_uint(ra - __uint_as_float(va & 0xffff0000u)), __float_as_uint(rb - __uint_as_float(vb & 0xffff0000u)),
                  0x7632);
}

__device__ __forceinline__ void st_cluster_f4(uint32_t cluster_addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// grid = (column tiles x splits, row tiles), cluster = splits CTAs along x
template <int BN, bool SWAP>
__global__ void __launch_bounds__(FX_THREADS)
gemm_f32_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, int rows_a, int rows_b,
                int K, int splits, int epi, const float* __restrict__ bias, float* __restrict__ out, int ldc, int* status,
                const int* skip) {
  constexpr int FS = fx_f32_stages<BN>(), BS = fx_bf16_stages<BN>();
  constexpr int F_BYTES = fx_f32_bytes<BN>(), B_BYTES = fx_bf16_bytes<BN>();
  constexpr int BF_OFF = FS * F_BYTES, BAR_OFF = fx_bar_off<BN>();
  constexpr int TEAMS = fx_teams<BN>(), TEAM_WARPS = FX_WARPS / TEAMS;
  constexpr int COLS = BN / 4;                        // columns of the tile per thread of the sixteen warps
  constexpr uint32_t TMEM_COLS = 512;
  constexpr uint32_t SMALL_COL = 2 * BN, A_COL = 3 * BN;
  static_assert(3 * BN + 48 * BS <= 512, "tensor memory");
  static_assert(FS >= BS && BS >= TEAMS, "barrier phases, see the splitting loop");
  static_assert((BN / 4 + 8) * FX_PAD * 16 <= BAR_OFF, "exchange area");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t bars = base + BAR_OFF;
  auto ffull = [&](int s) { return bars + 8u * s; };
  auto fempty = [&](int s) { return bars + 8u * (FS + s); };
  auto bfull = [&](int s) { return bars + 8u * (2 * FS + s); };
  auto bempty = [&](int s) { return bars + 8u * (2 * FS + BS + s); };
  auto afull = [&](int b) { return bars + 8u * (2 * FS + 2 * BS + b); };
  auto aempty = [&](int b) { return bars + 8u * (2 * FS + 2 * BS + 2 + b); };
  constexpr int N_BARS = 2 * FS + 2 * BS + 4;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(gbase + BAR_OFF + 8 * N_BARS);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gbase + BAR_OFF + 8 * N_BARS + 8);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)blockIdx.x % splits;
  const int m0 = blockIdx.y * 128, n0 = ((int)blockIdx.x / splits) * BN;
  const int total_kb = (K + FX_BK - 1) / FX_BK;
  const int kb_per = (total_kb + splits - 1) / splits;
  const int kb0 = rank * kb_per;
  const int num_kb = min(kb_per, total_kb - kb0);     // host guarantees >= 1
  const int num_ch = (num_kb + FX_CHUNK - 1) / FX_CHUNK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < FS; ++s) { mbar_init(ffull(s), 1); mbar_init(fempty(s), TEAM_WARPS); }
    for (int s = 0; s < BS; ++s) { mbar_init(bfull(s), TEAM_WARPS); mbar_init(bempty(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(afull(b), 1); mbar_init(aempty(b), FX_WARPS); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(tmem_slot, TMEM_COLS);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  // weight tiles of the first ring fill start before the wait for the kernel ahead (see gemm_tc_kernel)
  constexpr uint32_t W_BYTES = (SWAP ? 128 : BN) * 128;
  int n_pre = 0;
  if (warp == 0 && (skip == nullptr || *reinterpret_cast<const volatile int*>(skip) == 0)) n_pre = min(num_kb, FS);
  n_pre = __shfl_sync(0xffffffffu, n_pre, 0);
  if (warp == 0 && elect_one()) {
    for (int kb = 0; kb < n_pre; ++kb) {
      mbar_expect_tx_only(ffull(kb), W_BYTES);
      const uint32_t sa = base + kb * F_BYTES;
      if (SWAP) tma_load_2d(sa, &map_a, ffull(kb), (kb0 + kb) * FX_BK, m0);
      else tma_load_2d(sa + 128 * 128, &map_b, ffull(kb), (kb0 + kb) * FX_BK, n0);
    }
  }
  __syncwarp();
  pdl_launch_dependents();
  pdl_wait();
  if (warp == 0 && elect_one()) {
    for (int kb = 0; kb < n_pre; ++kb) {
      mbar_expect_tx(ffull(kb), (uint32_t)F_BYTES - W_BYTES);
      const uint32_t sa = base + kb * F_BYTES;
      if (SWAP) tma_load_2d(sa + 128 * 128, &map_b, ffull(kb), (kb0 + kb) * FX_BK, n0);
      else tma_load_2d(sa, &map_a, ffull(kb), (kb0 + kb) * FX_BK, m0);
    }
  }
  const bool active = skip == nullptr || *skip == 0;  // the same in every CTA of the cluster

  if (!active) {
    for (int kb = 0; threadIdx.x == 0 && kb < n_pre; ++kb) {   // tiles fetched ahead must have landed
      const long long t0 = clock64();
      while (!mbar_try(ffull(kb), 0u) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
    }
  } else if (warp == 0) {
    int issued = n_pre;
    for (int kb = n_pre; kb < num_kb; ++kb) {
      const int s = kb % FS;
      if (!__all_sync(0xffffffffu, mbar_wait(fempty(s), ((uint32_t)(kb / FS) & 1u) ^ 1u, abort_flag, status))) break;
      if (elect_one()) {
        mbar_expect_tx(ffull(s), (uint32_t)F_BYTES);
        const uint32_t sa = base + s * F_BYTES;
        tma_load_2d(sa, &map_a, ffull(s), (kb0 + kb) * FX_BK, m0);
        tma_load_2d(sa + 128 * 128, &map_b, ffull(s), (kb0 + kb) * FX_BK, n0);
      }
      __syncwarp();
      issued = kb + 1;
    }
    if (lane == 0 && *abort_flag) {                   // do not leave while copies may still be in flight
      for (int kb = issued > FS ? issued - FS : 0; kb < issued; ++kb) {
        const long long t0 = clock64();
        while (!mbar_try(ffull(kb % FS), (uint32_t)(kb / FS) & 1u) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
      }
    }
    __syncwarp();
    if (splits > 1) { cluster_sync_all(); cluster_sync_all(); }
  } else if (warp == 1) {
    {
      constexpr uint32_t idesc = make_idesc<BN>();
      bool ok = true;
      for (int kb = 0; kb < num_kb && ok; ++kb) {
        const int s = kb % BS, ch = kb / FX_CHUNK, buf = ch & 1;
        if (kb % FX_CHUNK == 0) {                     // the sixteen warps have drained this pair of accumulators
          ok = __all_sync(0xffffffffu, mbar_wait(aempty(buf), ((uint32_t)(ch >> 1) & 1u) ^ 1u, abort_flag, status));
          if (!ok) break;
        }
        ok = __all_sync(0xffffffffu, mbar_wait(bfull(s), (uint32_t)(kb / BS) & 1u, abort_flag, status));
        if (!ok) break;
        fence_after_sync();
        const uint32_t sw = base + BF_OFF + s * B_BYTES;
        const uint32_t acc_hh = tmem_base + (uint32_t)(buf * BN), acc_s = tmem_base + SMALL_COL;
        const uint32_t ta = tmem_base + A_COL + (uint32_t)(s * 48);
        if (elect_one()) {
#pragma unroll
        for (int k = 0; k < FX_BK / 16; ++k) {
          const uint32_t ah = ta + 8u * k, am = ah + 16u, al = ah + 32u;
          const uint64_t bh = make_smem_desc64(sw) + 2u * k, bm = make_smem_desc64(sw + BN * 64) + 2u * k,
                         bl = make_smem_desc64(sw + 2 * BN * 64) + 2u * k;
          umma_ts(acc_s, al, bh, idesc, (kb > 0 || k > 0) ? 1u : 0u);
          umma_ts(acc_s, ah, bl, idesc, 1u);
          umma_ts(acc_s, am, bm, idesc, 1u);
          umma_ts(acc_s, am, bh, idesc, 1u);
          umma_ts(acc_s, ah, bm, idesc, 1u);
          umma_ts(acc_hh, ah, bh, idesc, (kb % FX_CHUNK != 0 || k > 0) ? 1u : 0u);
        }
        umma_commit(bempty(s));
        if (kb % FX_CHUNK == FX_CHUNK - 1 || kb == num_kb - 1) umma_commit(afull(buf));
        }
        __syncwarp();
      }
    }
    __syncwarp();
    if (splits > 1) { cluster_sync_all(); cluster_sync_all(); }
  } else {
    const int ct = (int)threadIdx.x - 64;
    const int q = warp & 3, grp = (warp - 2) >> 2;    // TMEM lane quarter, column group
    float acc[COLS];
#pragma unroll
    for (int j = 0; j < COLS; ++j) acc[j] = 0.f;
    bool ok = true;
    const uint32_t t_lane = tmem_base + ((uint32_t)(q * 32) << 16);
    auto add_columns = [&](uint32_t col) {            // acc += this thread's columns of an accumulator
      uint32_t v[COLS / 8][8];
#pragma unroll
      for (int i = 0; i < COLS / 8; ++i) tmem_ld8_issue(t_lane + col + (uint32_t)(grp * COLS + 8 * i), v[i]);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < COLS / 8; ++i) {
        tmem_tie8(v[i]);
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[8 * i + j] += __uint_as_float(v[i][j]);
      }
    };
    auto drain = [&](int ch) {
      const int buf = ch & 1;
      ok = __all_sync(0xffffffffu, ok && mbar_wait(afull(buf), (uint32_t)(ch >> 1) & 1u, abort_flag, status));
      if (!ok) return;
      fence_after_sync();
      add_columns((uint32_t)(buf * BN));
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(aempty(buf));
    };
    // the teams split alternate k-blocks, so that one's waits and fences hide behind the others' arithmetic
    const int team = (warp - 2) / TEAM_WARPS, tt = ct % (32 * TEAM_WARPS);
    int drained = 0;
    for (int kb = team; kb < num_kb; kb += TEAMS) {
      const int fs = kb % FS, bs = kb % BS;
      // In this order: a stage of the fp32 ring passes from team to team and its tiles may land out of order, so a team
      // could take the phase before last of ffull for its own; once block kb - BS has been multiplied, the stage's phases up
      // to block kb - FS are behind everyone (FS >= BS >= TEAMS).
      ok = __all_sync(0xffffffffu, mbar_wait(bempty(bs), ((uint32_t)(kb / BS) & 1u) ^ 1u, abort_flag, status) &&
                                       mbar_wait(ffull(fs), (uint32_t)(kb / FS) & 1u, abort_flag, status));
      if (!ok) break;
      fence_after_sync();
      const uint8_t* src = gbase + fs * F_BYTES;
      // A operand: a thread takes halves (16 elements of K) of a row: one of them in a team of eight warps, both in one of
      // four (eight lanes of a row tile read all banks)
#pragma unroll
      for (int hv = 0; hv < 8 / TEAM_WARPS; ++hv) {
        const int row = q * 32 + lane, half = TEAM_WARPS == 8 ? ((warp - 2) >> 2) & 1 : hv;
        uint32_t h[8], m[8], l[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 x = *reinterpret_cast<const float4*>(src + row * 128 + (((half * 4 + i) ^ (row & 7)) << 4));
          split_pair(x.x, x.y, h[2 * i], m[2 * i], l[2 * i]);
          split_pair(x.z, x.w, h[2 * i + 1], m[2 * i + 1], l[2 * i + 1]);
        }
        const uint32_t ta = t_lane + A_COL + (uint32_t)(bs * 48 + half * 8);
        tmem_st8(ta, h);
        tmem_st8(ta + 16, m);
        tmem_st8(ta + 32, l);
      }
      // B operand: eight elements of K per step; four lanes share a row, so a quarter-warp covers two rows and all banks,
      // both ways
      uint8_t* dst = gbase + BF_OFF + bs * B_BYTES;
#pragma unroll
      for (int i = 0; i < BN / (8 * TEAM_WARPS); ++i) {
        const int row = (tt >> 2) + i * 8 * TEAM_WARPS, u = tt & 3;
        const uint8_t* sr = src + (128 + row) * 128;
        const float4 x0 = *reinterpret_cast<const float4*>(sr + (((2 * u) ^ (row & 7)) << 4));
        const float4 x1 = *reinterpret_cast<const float4*>(sr + (((2 * u + 1) ^ (row & 7)) << 4));
        uint4 h, m, l;
        split_pair(x0.x, x0.y, h.x, m.x, l.x);
        split_pair(x0.z, x0.w, h.y, m.y, l.y);
        split_pair(x1.x, x1.y, h.z, m.z, l.z);
        split_pair(x1.z, x1.w, h.w, m.w, l.w);
        uint8_t* p = dst + row * 64 + ((u ^ ((row >> 1) & 3)) << 4);
        *reinterpret_cast<uint4*>(p) = h;
        *reinterpret_cast<uint4*>(p + BN * 64) = m;
        *reinterpret_cast<uint4*>(p + 2 * BN * 64) = l;
      }
      tmem_wait_st();
      fence_before_sync();
      fence_async_smem();
      __syncwarp();
      if (lane == 0) { mbar_arrive(fempty(fs)); mbar_arrive(bfull(bs)); }
      // past the team's last block of chunk c: the chunk before it has been multiplied by now
      if ((kb + TEAMS) / FX_CHUNK > kb / FX_CHUNK && kb / FX_CHUNK > drained) { drain(drained++); if (!ok) break; }
    }
    while (ok && drained < num_ch) drain(drained++);
    if (ok) add_columns(SMALL_COL);                   // complete with the last chunk
    ok = named_bar_and(1, 32 * FX_WARPS, ok);
    // The tile goes through shared memory as [source CTA][column / 4][row] of four columns; with a split every CTA of the
    // cluster receives its slice of columns from all of them.  Ring and planes are idle: the last accumulator is complete.
    const int r = q * 32 + lane;
    const int slice4 = (BN / 4 + splits - 1) / splits; // column groups of four per CTA: group c4 belongs to CTA c4 % splits
    float4* ex = reinterpret_cast<float4*>(gbase);
    if (splits > 1) cluster_sync_all();               // nobody's main loop still uses the memory written below
    if (ok) {
#pragma unroll
      for (int j = 0; j < COLS / 4; ++j) {
        const int c4 = grp * (COLS / 4) + j;
        const float4 v = make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
        if (splits == 1) {
          ex[c4 * FX_PAD + r] = v;
        } else {
          const int owner = c4 % splits, lc = c4 / splits;
          st_cluster_f4(map_to_cta(smem_u32(ex + (rank * slice4 + lc) * FX_PAD + r), (uint32_t)owner), v);
        }
      }
    }
    if (splits > 1) cluster_sync_all();
    else named_bar_sync(2, 32 * FX_WARPS);
    if (ok) {
      const int units = slice4 * 128;
      const bool vec = !SWAP && (ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
      for (int un = ct; un < units; un += 32 * FX_WARPS) {
        // NORMAL: consecutive lanes take consecutive columns of a row; SWAP: consecutive features of a token
        const int lc = SWAP ? un >> 7 : un % slice4, rr = SWAP ? un & 127 : un / slice4;
        float4 v = ex[lc * FX_PAD + rr];
        for (int p = 1; p < splits; ++p) {
          const float4 w = ex[(p * slice4 + lc) * FX_PAD + rr];
          v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
        }
        const int c4 = lc * splits + rank, c = n0 + c4 * 4, row = m0 + rr;
        if (c4 >= BN / 4 || row >= rows_a || c >= rows_b) continue;
        float x[4] = {v.x, v.y, v.z, v.w};
        if (bias != nullptr) {
#pragma unroll
          for (int e = 0; e < 4; ++e) x[e] += SWAP ? bias[row] : (c + e < rows_b ? bias[c + e] : 0.f);
        }
        if (epi == EPI_GELU) {
#pragma unroll
          for (int e = 0; e < 4; ++e) x[e] = gelu_tanh(x[e]);
        }
        if (vec && c + 3 < rows_b) {
          float4* o = reinterpret_cast<float4*>(out + (long long)row * ldc + c);
          float4 y = make_float4(x[0], x[1], x[2], x[3]);
          if (epi == EPI_RESIDUAL) { const float4 h4 = *o; y.x += h4.x; y.y += h4.y; y.z += h4.z; y.w += h4.w; }
          *o = y;
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (c + e >= rows_b) break;
            float* o = out + (SWAP ? (long long)(c + e) * ldc + row : (long long)row * ldc + c + e);
            if (epi == EPI_RESIDUAL) *o += x[e]; else *o = x[e];
          }
        }
      }
    }
  }
  fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    fence_after_sync();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

template <int BN, bool SWAP>
static cudaError_t fx_prepare() {
  return cudaFuncSetAttribute(gemm_f32_kernel<BN, SWAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, fx_smem<BN>());
}

template <int BN, bool SWAP>
static cudaError_t fx_launch(const float* a, long long a_rows, const float* b, long long b_rows, int rows_a, int rows_b, int K,
                             int splits, int epi, const float* bias, float* out, int ldc, int* status, cudaStream_t st,
                             const int* skip) {
  CUtensorMap ma, mb;
  cudaError_t e;
  if ((e = get_tensor_map(a, a_rows, K, K, 128, FX_BK, &ma, 4)) != cudaSuccess) return e;
  if ((e = get_tensor_map(b, b_rows, K, K, BN, FX_BK, &mb, 4)) != cudaSuccess) return e;
  const dim3 grid((unsigned)((rows_b + BN - 1) / BN * splits), (unsigned)((rows_a + 127) / 128));
  if (splits > 1)
    return launch_k_cluster(gemm_f32_kernel<BN, SWAP>, grid, dim3(FX_THREADS), fx_smem<BN>(), st, (unsigned)splits, ma, mb, rows_a,
                            rows_b, K, splits, epi, bias, out, ldc, status, skip);
  return launch_k(gemm_f32_kernel<BN, SWAP>, grid, dim3(FX_THREADS), fx_smem<BN>(), st, ma, mb, rows_a, rows_b, K, splits, epi, bias,
                  out, ldc, status, skip);
}

}  // namespace tc

cudaError_t tc_prepare_gemm_f32() {
  using namespace tc;
  cudaError_t e;
  if ((e = fx_prepare<128, false>()) != cudaSuccess) return e;
  if ((e = fx_prepare<64, false>()) != cudaSuccess) return e;
  if ((e = fx_prepare<32, false>()) != cudaSuccess) return e;
  if ((e = fx_prepare<32, true>()) != cudaSuccess) return e;
  return fx_prepare<64, true>();
}

cudaError_t launch_gemm_f32(const float* A, long long a_cap, const float* W, const float* bias, int M, int N, int K, int epi,
                            float* out, int ldc, int* status, cudaStream_t st, const int* skip) {
  using namespace tc;
  if (M <= 0 || N <= 0) return cudaSuccess;
  static std::once_flag once;
  static cudaError_t prep = cudaSuccess;
  std::call_once(once, [] { prep = tc_prepare_gemm_f32(); });
  if (prep != cudaSuccess) return prep;
  constexpr int SMS = 148;
  const int total_kb = (K + FX_BK - 1) / FX_BK;
  // Tile width and K split by a cost model in SM clocks: measured clocks per k-block (tiles of 128 / 64 / 32 columns: 1370 /
  // 990 / 840), a fixed part (set-up, first tile, last drain), the two cluster barriers of a split, and the epilogue, times
  // the waves of the grid.  Clusters do not tile the chip's SM groups evenly: how many of each size run at a time (one CTA per SM) is what
  // the occupancy query reports on B200.
  constexpr int CLUSTERS[9] = {0, SMS, 74, 45, 33, 26, 22, 15, 15};
  const bool swap = M <= 64;
  const int rows_a = swap ? N : M, rows_b = swap ? M : N;
  int bn = 0, splits = 1;
  double best = 0.0;
  for (int cand : {128, 64, 32}) {
    if (swap && cand != (M <= 32 ? 32 : 64)) continue;
    const long long tiles = (long long)((rows_a + 127) / 128) * ((rows_b + cand - 1) / cand);
    for (int s = 1; s <= 8; ++s) {
      const int kb_per = (total_kb + s - 1) / s;
      if (s > 1 && kb_per < 2) break;
      if (kb_per * (s - 1) >= total_kb) continue;     // no empty split
      const double waves = (double)((tiles + CLUSTERS[s] - 1) / CLUSTERS[s]);
      const double cost = waves * (kb_per * (660.0 + 5.5 * cand) + 3000.0 + (s > 1 ? 1500.0 : 0.0) + 16.0 * cand / s);
      if (bn == 0 || cost < best * 0.97) { best = cost; bn = cand; splits = s; }
    }
  }
  if (swap) {
    if (bn == 32) return fx_launch<32, true>(W, N, A, a_cap, N, M, K, splits, epi, bias, out, ldc, status, st, skip);
    return fx_launch<64, true>(W, N, A, a_cap, N, M, K, splits, epi, bias, out, ldc, status, st, skip);
  }
  if (bn == 128) return fx_launch<128, false>(A, a_cap, W, N, M, N, K, splits, epi, bias, out, ldc, status, st, skip);
  if (bn == 64) return fx_launch<64, false>(A, a_cap, W, N, M, N, K, splits, epi, bias, out, ldc, status, st, skip);
  return fx_launch<32, false>(A, a_cap, W, N, M, N, K, splits, epi, bias, out, ldc, status, st, skip);
}

}  // namespace sdd

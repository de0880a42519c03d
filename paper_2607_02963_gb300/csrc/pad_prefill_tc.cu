// Whole-sequence forward attention under the event-factorized mask (Sec. 3.4, Fig. 3) on the
// 5th-generation tensor cores: the sequence of one video is [prefix of S tokens ; branch 0 ;
// ... ; branch E-1]; a prefix token attends causally within the prefix, a branch token to the
// prefix and causally to its own branch.
//
// One CTA per (query tile, kv-head).  A query tile is two slots of 128 rows: slot g holds
// 128 / G consecutive tokens x the G query heads of the kv-head (126 rows at G = 7), slot 1
// the tokens right after slot 0's.  The CTA walks the 128-key tiles its rows can see (the
// prefix up to its last token, then the keys from the start of its first branch token's
// branch to its last token) and masks per row only where a tile needs it.  Query tiles start
// in descending order, so that the longest key ranges go first.
//
// A short sequence (SPLIT) has one slot of queries per CTA and shares out its key tiles instead:
// the softmax warps 4-7 take the even ones, 8-11 the odd ones, each with an S buffer, a maximum
// and an O of their own, merged at the end.  There a CTA's chain of tiles, one after the other, is
// the whole time, and this halves it (512 + 160 tokens, 28/4 heads: 16.7 -> 14.5 us; 1100 + 160,
// 16/1 heads: 24.8 -> 16.8).
//
//   warps 0, 3  TMA producers of K and V tiles (64-column boxes, 128-byte swizzle); warp 3 clears
//               the rows of a branch's last V tile that no row here sees
//   warp 1      S issuer: S_g(k) = Q_g K(k)^T
//   warp 2      TMEM allocation (512 columns) and deallocation, and P.V issuer: O_g += P_g(k)
//               V(k), P read back from TMEM, 96 keys and then the last 32
//   warps 4-7   softmax of slot 0, warps 8-11 of slot 1: one query row per thread, all 128
//               scores of a tile in registers (setmaxnreg moves registers from warps 0-3 to
//               these); online sum in base 2 on a maximum that follows lazily.  At the end each
//               warp normalises its own 32 rows and writes them through its part of the
//               slot's (idle) Q stage.
//
// What bounds it, and why it looks like this (sequence of 34.7 k tokens, 28/4 heads, D 128: 7.08
// ms with one 128-row group per CTA, as it is 5.1 to 5.5 ms over several GPUs = 1.56 to 1.68 PFLOP/s of
// visible pairs, 0.83 to 0.89 of cuBLAS's rate; 8.7 k tokens, 14/2 heads, D 64: 724 us on the mma.sync
// kernel, 198 us here):
//   - Two slots share each K/V tile: with one 128-row group the MMAs' shared-memory operand
//     reads (S: 8 KB per K = 16 step, P.V: 4 KB) and the 64 KB that a tile brings in exceed 128
//     B per clock by a fifth; and one slot's softmax runs under the other's MMAs.
//   - What is left is the chain S -> softmax -> P.V of a slot, ~2900 cycles per tile against
//     2 x 1036 of MMAs.  So the softmax makes no pass for the maximum (the row sum tells
//     whether the running one still bounds the scores), tiles that need no mask run a loop
//     without mask code, and P is released in two unequal parts, so that little of P.V is
//     left to do once the last of P is written (halves: 5.67 ms).
//   - The issuer warps run their loops with all lanes and elect the issuing one (elect_one),
//     and the TMEM addresses are immediates: 6.34 -> 6.02 ms.
//
// TMEM columns: S_0 at 0, S_1 at 128, O_g at 256 + D g.  P_g goes over S_g (all of a row's
// scores are in registers by then), so S_g(k + 1) waits for P.V of tile k.
//
// head_dim 64 holds P as the sum of two bf16 numbers (columns 0-63 and 64-127 of S_g), each with
// its own P.V: one bf16 on the lazily followed maximum was 5-7 % less exact than the mma.sync
// kernel's, which follows it every 64 keys (relative error of the fp32 output against 64 bits
// 1.24e-3 to 1.40e-3 against 1.18e-3 to 1.32e-3; 140 us for the call above).  Two give 2e-6 to
// 4e-6.
//
// Barrier phases: every barrier is per slot or per stage, so that the completion a thread
// waits for by parity cannot be overtaken by the next one before the thread moves on.  Every
// wait is bounded (about one second of %globaltimer); one that runs out records
// PAD_ERR_DEVICE_TIMEOUT in the prefill status word, raises a CTA-wide abort flag, lets the
// producers and issuers drain what they started, frees TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "pad_internal.h"
#include "pad_tc_common.cuh"

namespace pad {

namespace {

using namespace tc;

constexpr int kMaxBranches = 1024;
constexpr int kBN = 128;        // keys per tile
constexpr int kThreads = 384;
constexpr int kLoGroups = 3;          // 32-key groups of a tile whose P is released first
constexpr float kRescaleSum = 256.0f; // a part of a row whose P sum to more is redone on a new maximum
constexpr float kNegInf = -__builtin_huge_valf();

template <int D>
struct Cfg {
  static constexpr int kHalves = D / 64;                      // 64-column boxes of a row
  static constexpr uint32_t kBoxBytes = kBN * 128;            // 128 rows x 64 bf16
  static constexpr uint32_t kTileBytes = kHalves * kBoxBytes; // a K or V tile, or Q of a slot
  static constexpr int kKS = D == 128 ? 3 : 4;                // K stages
  static constexpr int kVS = D == 128 ? 2 : 4;                // V stages
  static constexpr uint32_t kOffK = 2 * kTileBytes;           // Q_0, Q_1 first
  static constexpr uint32_t kOffV = kOffK + kKS * kTileBytes;
  static constexpr uint32_t kOffBar = kOffV + kVS * kTileBytes;
  static constexpr uint32_t kSmemBytes = kOffBar + 512;
  static constexpr bool kSplitP = D == 64;                    // P as two bf16 numbers
  static constexpr uint32_t kColO = 256;                      // + D g
  // Registers per thread after setmaxnreg: the launch gives 384 x 168 = 64512; 128 x 80 + 256 x
  // 208 = 63488, and 128 x 56 + 256 x 224 = 64512 where the softmax keeps both parts of P.
  static constexpr int kRegsIssue = kSplitP ? 56 : 80, kRegsSoftmax = kSplitP ? 224 : 208;
  static constexpr uint32_t kIdescS = make_idesc(128, kBN, false);  // B = K tile, K-major
  static constexpr uint32_t kIdescPV = make_idesc(128, D, true);    // B = V tile, N(=d)-major
  static_assert(kSmemBytes <= 232448, "fits the 227 KB opt-in shared memory");
};

struct PrefillTcParams {
  int32_t n_tokens, prefix_len, n_branches;
  int32_t h_q, h_kv, group, tps;        // tps: query tokens per slot (128 / group)
  int32_t tok_base, n_qt;               // the grid's query tiles: n_qt of them, from this token on
  int32_t release, after;               // mixed launch: this grid releases the next / ends after the one ahead
  float scale_log2;
  int32_t out_bf16;
  uint64_t gen;
  PadDevHeader* header;
  void* out;
  float* lse;
  int32_t bstart[kMaxBranches + 1];     // branch b occupies [bstart[b], bstart[b + 1]); bstart[0] = prefix_len
};

struct Bars {
  uint64_t kfull[4], kfree[4];
  uint64_t vfull[4], vfree[4];
  uint64_t qfull[2];
  uint64_t sfull[2];          // S of the slot's current tile has completed
  uint64_t plo[2], phi[2];    // P of its first 32 kLoGroups keys / of the rest is written (4 warp arrivals)
  uint64_t pvlo[2];           // P.V of its first part has completed
  uint64_t pvdone[2];         // its P.V has completed
  uint64_t drain_s, drain_pv; // every MMA of the S / P.V issuer has completed
  uint64_t tdone;             // the softmax warps are done with TMEM (8 warp arrivals)
  uint64_t vclear;            // the last V tile's rows past the last visible key are cleared
  uint32_t tmem_base;
  int32_t abort;
};
static_assert(sizeof(Bars) <= 512, "barrier block fits its slot");

// Bounded wait, inlined (setmaxnreg leaves no room for calls).
__device__ __forceinline__ bool pwait(uint64_t* bar, uint32_t parity, Bars* bars, const PrefillTcParams& p, int where) {
  unsigned long long t0 = 0;
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 255u) == 0) {
      if (*reinterpret_cast<volatile int32_t*>(&bars->abort)) return false;
      const unsigned long long now = globaltimer();
      if (t0 == 0) t0 = now;
      if (now - t0 > kWaitNs) {
        pad_set_error(p.header, p.gen, PAD_ERR_DEVICE_TIMEOUT, (int)blockIdx.x, where, (int)threadIdx.x);
        *reinterpret_cast<volatile int32_t*>(&bars->abort) = 1;
        return false;
      }
    }
  }
}

// The same for a whole warp (warp-uniform result).
__device__ __forceinline__ bool pwait_warp(uint64_t* bar, uint32_t parity, Bars* bars, const PrefillTcParams& p, int where) {
  return __all_sync(0xffffffffu, pwait(bar, parity, bars, p, where)) != 0;
}

// First token of the branch that holds token t (t >= prefix_len).
__device__ __forceinline__ int branch_start(const PrefillTcParams& p, int t) {
  int lo = 0, hi = p.n_branches - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (p.bstart[mid] <= t) lo = mid; else hi = mid - 1;
  }
  return p.bstart[lo];
}

// Maximum of a row's 128 raw scores (eight chains of three-input max).
__device__ __forceinline__ float row_max(const uint32_t (&s)[4][32]) {
  float m[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) m[u] = kNegInf;
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
      const int u = (i >> 1) & 7;
      m[u] = max3f(m[u], __uint_as_float(s[c][i]), __uint_as_float(s[c][i + 1]));
    }
  return fmaxf(max3f(m[0], m[1], m[2]), max3f(max3f(m[3], m[4], m[5]), m[6], m[7]));
}

// P = 2^(s * sl2 - m) of the 32-score groups [C0, C1) of a row, written as packed bf16 (two
// keys per column) to TMEM columns taddr + 16 C0 ..; returns their fp32 sums as four pairs.
// SPLIT: what the rounding leaves of P goes, rounded to bf16 too, 64 columns further on.
template <int C0, int C1, bool SPLIT>
__device__ __forceinline__ void part_exp(const uint32_t (&s)[4][32], uint64_t sc2, float m, uint32_t taddr,
                                         uint64_t (&sum)[4]) {
  const uint64_t nm2 = f2pack(-m, -m);
#pragma unroll
  for (int u = 0; u < 4; ++u) sum[u] = 0ull;
#pragma unroll
  for (int c = C0; c < C1; ++c) {
    if constexpr (SPLIT) {
      // (half the columns at a time: both parts of all sixteen did not fit the registers)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        uint32_t pk[8], rest[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int k = 2 * (8 * q + i);
          const uint64_t x = ffma2(f2pack(__uint_as_float(s[c][k]), __uint_as_float(s[c][k + 1])), sc2, nm2);
          const float a = ex2(f2lo(x)), b = ex2(f2hi(x));
          const uint64_t e = f2pack(a, b);
          sum[i & 3] = fadd2(sum[i & 3], e);
          pk[i] = pack_bf16(a, b);
          const uint64_t r = ffma2(f2pack(__uint_as_float(pk[i] << 16), __uint_as_float(pk[i] & 0xffff0000u)),
                                   f2pack(-1.f, -1.f), e);
          rest[i] = pack_bf16(f2lo(r), f2hi(r));
        }
        tmem_st8(taddr + 16 * c + 8 * q, pk);
        tmem_st8(taddr + 64 + 16 * c + 8 * q, rest);
      }
    } else {
      uint32_t pk[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const uint64_t x = ffma2(f2pack(__uint_as_float(s[c][2 * i]), __uint_as_float(s[c][2 * i + 1])), sc2, nm2);
        const float a = ex2(f2lo(x)), b = ex2(f2hi(x));
        sum[i & 3] = fadd2(sum[i & 3], f2pack(a, b));
        pk[i] = pack_bf16(a, b);
      }
      tmem_st16(taddr + 16 * c, pk);
    }
  }
}

template <int D, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 1)
    prefill_tc_kernel(const __grid_constant__ PrefillTcParams p, const __grid_constant__ CUtensorMap tmQ,
                      const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV) {
  using C = Cfg<D>;
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t sbase = smem_u32(smem);
  if (sbase & 1023u) {  // the 128-byte swizzle atoms need 1024-byte alignment (never expected)
    if (threadIdx.x == 0) pad_set_error(p.header, p.gen, PAD_ERR_UNSUPPORTED, (int)blockIdx.x, (int)sbase, 0);
    return;
  }
  Bars* bars = reinterpret_cast<Bars*>(smem + C::kOffBar);
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

  const int N = p.n_tokens, S = p.prefix_len, G = p.group;
  const int tpc = (SPLIT ? 1 : 2) * p.tps;                              // query tokens per CTA
  const int qt = p.n_qt - 1 - (int)blockIdx.x / p.h_kv;
  const int kvh = (int)blockIdx.x % p.h_kv;
  const int tok0 = p.tok_base + qt * tpc;
  const int last = min(tok0 + tpc, N) - 1;
  // key tiles: [0, a_end) of the prefix, then [b_lo, last] of the branches
  const int a_end = min(S, last + 1);
  const int a_tiles = (a_end + kBN - 1) / kBN;
  int b_lo = 0, b_tiles = 0;
  if (last >= S) {
    b_lo = branch_start(p, max(tok0, S));
    b_tiles = (last + 1 - b_lo + kBN - 1) / kBN;
  }
  const int n_tiles = a_tiles + b_tiles;                  // >= 1
  auto tile_tok = [&](int t) { return t < a_tiles ? min(t * kBN, a_end - kBN) : b_lo + (t - a_tiles) * kBN; };
  // Keys that no row of the CTA sees stay out of its V tiles (see zero_v_rows).  The last tile of the prefix
  // ends where the visible prefix does: it starts that much earlier (rows before the first token are
  // zero), and the columns that it shares with the tile before are masked.  The last tile of the branches
  // would run into the branch before instead: the V producer clears its rows past `last` (vclear).
  const bool part = b_tiles > 0 && (last + 1 - b_lo) % kBN != 0;
  auto load_tile = [&](const CUtensorMap* map, uint32_t off, int t, uint64_t* full) {
    mbar_expect_tx(full, C::kTileBytes);
#pragma unroll
    for (int h = 0; h < C::kHalves; ++h)
      tma_load_3d(sbase + off + h * C::kBoxBytes, map, 64 * h, kvh, tile_tok(t), full);
  };

  if (SPLIT && p.release) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (threadIdx.x == 0) {
    for (int s = 0; s < 4; ++s) {
      mbar_init(&bars->kfull[s], 1);
      mbar_init(&bars->kfree[s], 1);
      mbar_init(&bars->vfull[s], 1);
      mbar_init(&bars->vfree[s], 1);
    }
    for (int g = 0; g < 2; ++g) {
      mbar_init(&bars->qfull[g], 1);
      mbar_init(&bars->sfull[g], 1);
      mbar_init(&bars->plo[g], 4);
      mbar_init(&bars->phi[g], 4);
      mbar_init(&bars->pvlo[g], 1);
      mbar_init(&bars->pvdone[g], 1);
    }
    mbar_init(&bars->drain_s, 1);
    mbar_init(&bars->drain_pv, 1);
    mbar_init(&bars->tdone, 8);
    mbar_init(&bars->vclear, 1);
    bars->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // Q of both slots (box: 64 columns x G heads x tps tokens, so that smem row = token * G +
    // head; tokens past N are zero-filled) and the first K tile go out from here
    const uint32_t q_bytes = (uint32_t)C::kHalves * 128u * (uint32_t)(G * p.tps);
    for (int g = 0; g < (SPLIT ? 1 : 2); ++g) {
      mbar_expect_tx(&bars->qfull[g], q_bytes);
#pragma unroll
      for (int h = 0; h < C::kHalves; ++h)
        tma_load_3d(sbase + g * C::kTileBytes + h * C::kBoxBytes, &tmQ, 64 * h, kvh * G, tok0 + g * p.tps,
                    &bars->qfull[g]);
      if (g == 0) load_tile(&tmK, C::kOffK, 0, &bars->kfull[0]);
    }
    load_tile(&tmV, C::kOffV, 0, &bars->vfull[0]);
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  // an allocation of all 512 columns starts at TMEM address 0: known at compile time, so that
  // the MMAs' TMEM operands are immediates (a word read back from shared memory is not)
  constexpr uint32_t tmem = 0;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(C::kRegsIssue));
    bool ok = true;
    if (warp == 0 || warp == 3) {
      // ------------------------------------------------------------ TMA producers
      if (lane == 0) {
        const bool isK = warp == 0;
        const CUtensorMap* map = isK ? &tmK : &tmV;
        const int ns = isK ? C::kKS : C::kVS;
        uint64_t* full = isK ? bars->kfull : bars->vfull;
        uint64_t* freed = isK ? bars->kfree : bars->vfree;
        const uint32_t base = isK ? C::kOffK : C::kOffV;
        int s = 1, ph = 0, issued = 1;  // tile 0 went out in the prologue; ph: uses of stage s
        for (int t = 1; t < n_tiles; ++t) {
          if (s == ns) {
            s = 0;
            ++ph;
          }
          if (ph > 0) ok = pwait(&freed[s], (uint32_t)((ph - 1) & 1), bars, p, isK ? 1 : 2);
          if (!ok) break;
          load_tile(map, base + (uint32_t)s * C::kTileBytes, t, &full[s]);
          issued = t + 1;
          ++s;
        }
        if (!ok) {
          // the loads already issued must land before the CTA leaves
          for (int t = max(0, issued - ns); t < issued; ++t) drain_wait(&full[t % ns], (uint32_t)((t / ns) & 1));
        }
      }
      __syncwarp();
      if (warp == 3 && part && __shfl_sync(0xffffffffu, (int)ok, 0)) {
        const int s = (n_tiles - 1) % C::kVS;
        if (pwait_warp(&bars->vfull[s], (uint32_t)(((n_tiles - 1) / C::kVS) & 1), bars, p, 7)) {
          zero_v_rows<C::kHalves>(smem + C::kOffV + (uint32_t)s * C::kTileBytes, last + 1 - tile_tok(n_tiles - 1), lane, 32);
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars->vclear);
        }
      }
    } else if (warp == 1) {
      // ------------------------------------------------------------ S issuer
      const bool el = elect_one();
      const uint64_t dK = sdesc(sbase + C::kOffK, 16, 1024);
      int s = 0, ph = 0;
      for (int t = 0; t < n_tiles && ok; ++t) {
        ok = pwait_warp(&bars->kfull[s], (uint32_t)ph, bars, p, 3);
        const int j = SPLIT ? t >> 1 : t;      // the slot's how-manieth tile
#pragma unroll
        for (int i = 0; i < (SPLIT ? 1 : 2); ++i) {
          const int g = SPLIT ? t & 1 : i;
          if (!ok) break;
          if (j == 0)
            ok = pwait_warp(&bars->qfull[SPLIT ? 0 : g], 0u, bars, p, 11);
          else  // S_g holds P of the slot's previous tile until its P.V has completed
            ok = pwait_warp(&bars->pvdone[g], (uint32_t)((j - 1) & 1), bars, p, 6);
          if (!ok) break;
          fence_after();
          const uint64_t qd = sdesc(sbase + (SPLIT ? 0u : (uint32_t)g * C::kTileBytes), 16, 1024);
          const uint64_t kd = dK + ((uint32_t)s * C::kTileBytes >> 4);
          if (el) {
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
              const uint32_t off = (uint32_t)(kk >> 2) * C::kBoxBytes + (uint32_t)(kk & 3) * 32;
              mma_ss(tmem + 128u * g, qd + (off >> 4), kd + (off >> 4), C::kIdescS, kk > 0 ? 1u : 0u);
            }
            mma_commit(&bars->sfull[g]);
            if (SPLIT || g == 1) mma_commit(&bars->kfree[s]);
          }
          __syncwarp();
        }
        if (++s == C::kKS) {
          s = 0;
          ph ^= 1;
        }
      }
      if (el) mma_commit(&bars->drain_s);
      __syncwarp();
      drain_wait(&bars->drain_s, 0u);
    } else {
      // ------------------------------------------------------------ P.V issuer
      // V tile, N(=head-dim)-major: 16 keys per K-step (2048 bytes), a second 64-column box
      // at + kBoxBytes (leading byte offset), 8-row groups 1024 apart.
      const bool el = elect_one();
      const uint64_t dV = sdesc(sbase + C::kOffV, C::kBoxBytes, 1024);
      int s = 0, ph = 0;
      for (int t = 0; t < n_tiles && ok; ++t) {
        ok = pwait_warp(&bars->vfull[s], (uint32_t)ph, bars, p, 4);
        const uint64_t vd = dV + ((uint32_t)s * C::kTileBytes >> 4);
        const int j = SPLIT ? t >> 1 : t;
#pragma unroll
        for (int i = 0; i < (SPLIT ? 1 : 2); ++i) {
          const int g = SPLIT ? t & 1 : i;
          const uint32_t a = tmem + 128u * g;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (ok) ok = pwait_warp(h ? &bars->phi[g] : &bars->plo[g], (uint32_t)(j & 1), bars, p, 5);
            if (!ok) break;
            fence_after();
            if (el) {
#pragma unroll
              for (int kk = h ? 2 * kLoGroups : 0; kk < (h ? 8 : 2 * kLoGroups); ++kk)
                mma_ts(tmem + C::kColO + (uint32_t)D * g, a + kk * 8, vd + ((uint32_t)kk * 2048 >> 4), C::kIdescPV,
                       (j > 0 || kk > 0) ? 1u : 0u);
              if (C::kSplitP) {
#pragma unroll
                for (int kk = h ? 2 * kLoGroups : 0; kk < (h ? 8 : 2 * kLoGroups); ++kk)
                  mma_ts(tmem + C::kColO + (uint32_t)D * g, a + 64 + kk * 8, vd + ((uint32_t)kk * 2048 >> 4),
                         C::kIdescPV, 1u);
              }
              if (h == 0) mma_commit(&bars->pvlo[g]);
              if (h == 1) {
                mma_commit(&bars->pvdone[g]);
                if (SPLIT || g == 1) mma_commit(&bars->vfree[s]);
              }
            }
            __syncwarp();
          }
        }
        if (++s == C::kVS) {
          s = 0;
          ph ^= 1;
        }
      }
      if (el) mma_commit(&bars->drain_pv);
      __syncwarp();
      drain_wait(&bars->drain_pv, 0u);
    }
    __syncwarp();
    if (warp == 2) {
      // TMEM is freed only after every softmax warp has arrived
      drain_wait(&bars->tdone, 0u);
      __syncwarp();
      fence_after();
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
    // (a grid that ran beside the one ahead completes after it, as stream order has it)
    if (!SPLIT && warp == 0 && p.after) asm volatile("griddepcontrol.wait;" ::: "memory");
  } else {
    // ------------------------------------------------------------ softmax
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(C::kRegsSoftmax));
    const int g = (warp - 4) >> 2;             // slot
    const int wrow = 32 * (warp & 3);          // TMEM lanes wrow .. wrow + 31
    const int row = wrow + lane;               // row of the slot: token row / G, head row % G
    const int tl = row / G;
    const int tok = tok0 + (SPLIT ? 0 : g * p.tps) + tl;
    const bool active = tl < p.tps && tok < N;
    const int bs = active && tok >= S ? branch_start(p, tok) : -1;
    const uint32_t tb = tmem + ((uint32_t)wrow << 16);
    const uint32_t tS = tb + 128u * g;
    const uint32_t tO = tb + C::kColO + (uint32_t)D * g;
    const float sl2 = p.scale_log2;
    const uint64_t sc2 = f2pack(sl2, sl2);
    // an inactive row (past the slot's rows or the sequence) takes no part in any decision
    float m_run = active ? kNegInf : 0.f;
    uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
    bool ok = true;

    // One tile, in its two parts (h): P is computed on the running maximum m, and its sum,
    // which the row sum needs anyway, shows whether m still bounds the scores: a sum of at most
    // 2^8 means that every P is.  Only a part that exceeds it (and the first of all, which has
    // no m yet) finds the row's maximum, rescales O and l to it and is redone.
    auto tile = [&](int t, auto masked) -> bool {
      const int j = SPLIT ? t >> 1 : t;        // the slot's how-manieth tile
      if (!__all_sync(0xffffffffu, pwait(&bars->sfull[g], (uint32_t)(j & 1), bars, p, 8))) return false;
      fence_after();
      uint32_t s[4][32];
#pragma unroll
      for (int c = 0; c < 4; ++c) tmem_ld32(tS + 32 * c, s[c]);
#pragma unroll
      for (int c = 0; c < 4; ++c) tmem_wait_ld_dep(s[c]);
      if (decltype(masked)::value) {
        // the tile's columns this row sees: [lo, hi)
        int lo = 0, hi = kBN;
        if (active) {
          const int t0 = tile_tok(t);
          if (t < a_tiles) {
            lo = t * kBN - t0;
            hi = (bs < 0 ? tok + 1 : S) - t0;
          } else {
            lo = bs < 0 ? kBN : bs - t0;
            hi = tok + 1 - t0;
          }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const int col = 32 * c + i;
            if (col < lo || col >= hi) s[c][i] = 0xff800000u;  // -inf
          }
        if (part && t == n_tiles - 1 && !__all_sync(0xffffffffu, pwait(&bars->vclear, 0u, bars, p, 12))) return false;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint64_t sum[4];
        if (h == 0) part_exp<0, kLoGroups, C::kSplitP>(s, sc2, m_run == kNegInf ? 0.f : m_run, tS, sum);
        else part_exp<kLoGroups, 4, C::kSplitP>(s, sc2, m_run == kNegInf ? 0.f : m_run, tS, sum);
        const uint64_t s2 = fadd2(fadd2(sum[0], sum[1]), fadd2(sum[2], sum[3]));
        const bool grow = active && (m_run == kNegInf || f2lo(s2) + f2hi(s2) > kRescaleSum);
        if (__any_sync(0xffffffffu, grow)) {
          if (j > 0 || h == 1) {
            // every P.V issued on O so far has completed: O may be rescaled
            if (!__all_sync(0xffffffffu, h == 1 ? pwait(&bars->pvlo[g], (uint32_t)(j & 1), bars, p, 9)
                                                : pwait(&bars->pvdone[g], (uint32_t)((j - 1) & 1), bars, p, 9)))
              return false;
            fence_after();
          }
          const float m_new = fmaxf(m_run, row_max(s) * sl2);
          const bool need = grow && m_new > m_run;
          const float alpha = need ? ex2(m_run - m_new) : 1.f;
          if (j > 0 || h == 1) {
#pragma unroll 1
            for (int c = 0; c < D / 32; ++c) {
              uint32_t r[32];
              tmem_ld32(tO + 32 * c, r);
              tmem_wait_ld_dep(r);
#pragma unroll
              for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * alpha);
              tmem_st32(tO + 32 * c, r);
            }
          }
          const uint64_t al2 = f2pack(alpha, alpha);
#pragma unroll
          for (int u = 0; u < 4; ++u) acc[u] = fmul2(acc[u], al2);
          if (need) m_run = m_new;
          // (a row that has seen no visible key keeps m = -inf; its exponent base is 0)
          if (h == 0) part_exp<0, kLoGroups, C::kSplitP>(s, sc2, m_run == kNegInf ? 0.f : m_run, tS, sum);
          else part_exp<kLoGroups, 4, C::kSplitP>(s, sc2, m_run == kNegInf ? 0.f : m_run, tS, sum);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] = fadd2(acc[u], sum[u]);
        tmem_wait_st();
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(h ? &bars->phi[g] : &bars->plo[g]);
      }
      return true;
    };
    // the leading prefix tiles that every row of the warp sees in full need no mask
    int lim = active ? (bs < 0 ? tok + 1 : S) : 0x7fffffff;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lim = min(lim, __shfl_xor_sync(0xffffffffu, lim, o));
    const int n_full = min(a_tiles, lim / kBN);
    constexpr int kStep = SPLIT ? 2 : 1;
    int t = SPLIT ? g : 0;
    for (; t < n_full && ok; t += kStep) ok = tile(t, std::false_type{});
    for (; t < n_tiles && ok; t += kStep) ok = tile(t, std::true_type{});
    // O is final once the last P.V has completed; the slot's Q is idle by then too (its last S
    // completed before that P could be written)
    const int mine = SPLIT ? (n_tiles + 1 - g) >> 1 : n_tiles;  // tiles of this slot
    if (ok && mine > 0) ok = pwait(&bars->pvdone[g], (uint32_t)((mine - 1) & 1), bars, p, 10);
    ok = __all_sync(0xffffffffu, ok);
    const uint64_t a2 = fadd2(fadd2(acc[0], acc[1]), fadd2(acc[2], acc[3]));
    float l = f2lo(a2) + f2hi(a2);
    float wgt = 1.f;                           // of this slot's O in the result
    // SPLIT: slot g writes the columns from D/2 g on, and takes the other's share of them.  (m, l)
    // of both go through the second Q stage, which holds nothing here; then the O rows on the
    // common maximum through the K stages, idle once both slots' last P.V has completed: fp32,
    // row r's 16-byte chunk c at chunk c ^ (r % 16 or 8), so that both sides touch distinct banks.
    constexpr int kCo = D / 4;                 // 16-byte chunks of an fp32 row
    static_assert(128u * 4 * D <= C::kKS * C::kTileBytes, "the slots' O rows fit the K stages");
    float2* sml = reinterpret_cast<float2*>(smem + C::kTileBytes);
    uint8_t* so = smem + C::kOffK + (uint32_t)row * (4 * D);
    if (SPLIT) {
      sml[g * 128 + row] = make_float2(m_run, l);
      asm volatile("bar.sync 1, 256;" ::: "memory");
      const float2 other = sml[(g ^ 1) * 128 + row];
      const float m = fmaxf(m_run, other.x);
      wgt = mine > 0 && m_run > kNegInf ? ex2(m_run - m) : 0.f;
      l = fmaf(l, wgt, other.x > kNegInf ? other.y * ex2(other.x - m) : 0.f);
      m_run = m;
      if (ok) {
        fence_after();
#pragma unroll 1
        for (int c = (1 - g) * (D / 64); c < (2 - g) * (D / 64); ++c) {
          uint32_t r[32];
          if (mine > 0) {
            tmem_ld32(tO + 32 * c, r);
            tmem_wait_ld_dep(r);
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
            if (mine > 0)
              w = make_float4(__uint_as_float(r[4 * j]) * wgt, __uint_as_float(r[4 * j + 1]) * wgt,
                              __uint_as_float(r[4 * j + 2]) * wgt, __uint_as_float(r[4 * j + 3]) * wgt);
            *reinterpret_cast<float4*>(so + (((8 * c + j) ^ (lane & (kCo / 2 - 1))) << 4)) = w;
          }
        }
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
    }
    // O of 32 columns of the row, from c0 on
    auto load_o = [&](int c0, uint32_t* r) {
      if (!SPLIT || mine > 0) {
        tmem_ld32(tO + c0, r);
        tmem_wait_ld_dep(r);
      }
      if (SPLIT) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float4 w = *reinterpret_cast<const float4*>(so + (((c0 / 4 + j) ^ (lane & (kCo / 2 - 1))) << 4));
          const float a[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
          for (int u = 0; u < 4; ++u)
            r[4 * j + u] = __float_as_uint(mine > 0 ? fmaf(__uint_as_float(r[4 * j + u]), wgt, a[u]) : a[u]);
        }
      }
    };
    if (ok) {
      fence_after();
      const float inv = 1.0f / l;
      if (active && (!SPLIT || g == 0) && p.lse != nullptr)
        p.lse[(int64_t)tok * p.h_q + kvh * G + row % G] = (m_run + log2f(l)) * 0.69314718055994531f;
      // Rows out through this warp's 32 rows of the slot's Q stage (2 D bytes per row: all
      // columns in bf16, half of them in fp32): row r's 16-byte chunk c at chunk position
      // c ^ (r % chunks), so that both sides touch distinct banks; then coalesced rows.
      constexpr int kCh = 2 * D / 16;           // chunks per staged row
      uint8_t* stg = smem + (uint32_t)g * C::kTileBytes + (uint32_t)wrow * (2 * D);
      const int passes = p.out_bf16 ? 1 : 2;
      const int esz = p.out_bf16 ? 2 : 4;
#pragma unroll 1
      for (int ps = SPLIT && passes == 2 ? g : 0; ps < (SPLIT && passes == 2 ? g + 1 : passes); ++ps) {
        if (p.out_bf16) {
#pragma unroll 1
          for (int c = SPLIT ? g * (D / 64) : 0; c < (SPLIT ? g + 1 : 2) * (D / 64); ++c) {
            uint32_t r[32];
            load_o(32 * c, r);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              uint32_t w[4];
#pragma unroll
              for (int u = 0; u < 4; ++u)
                w[u] = pack_bf16(__uint_as_float(r[8 * j + 2 * u]) * inv, __uint_as_float(r[8 * j + 2 * u + 1]) * inv);
              *reinterpret_cast<uint4*>(stg + lane * (2 * D) + (((4 * c + j) ^ (lane & (kCh - 1))) << 4)) =
                  make_uint4(w[0], w[1], w[2], w[3]);
            }
          }
        } else {
#pragma unroll 1
          for (int c = 0; c < D / 64; ++c) {
            uint32_t r[32];
            load_o((D / 2) * ps + 32 * c, r);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              uint32_t w[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) w[u] = __float_as_uint(__uint_as_float(r[4 * j + u]) * inv);
              *reinterpret_cast<uint4*>(stg + lane * (2 * D) + (((8 * c + j) ^ (lane & (kCh - 1))) << 4)) =
                  make_uint4(w[0], w[1], w[2], w[3]);
            }
          }
        }
        __syncwarp();
#pragma unroll 1
        for (int i = lane; i < 32 * kCh / (SPLIT && p.out_bf16 ? 2 : 1); i += 32) {
          const int r = SPLIT && p.out_bf16 ? i / (kCh / 2) : i / kCh;
          const int c = SPLIT && p.out_bf16 ? g * (kCh / 2) + i % (kCh / 2) : i % kCh;
          const int rr = wrow + r, rt = rr / G, rtok = tok0 + (SPLIT ? 0 : g * p.tps) + rt;
          if (rt < p.tps && rtok < N) {
            const uint4 v = *reinterpret_cast<const uint4*>(stg + r * (2 * D) + ((c ^ (r & (kCh - 1))) << 4));
            const int64_t o = ((int64_t)rtok * p.h_q + kvh * G + (rr - rt * G)) * D * esz + (int64_t)ps * (2 * D) + 16 * c;
            *reinterpret_cast<uint4*>(static_cast<uint8_t*>(p.out) + o) = v;
          }
        }
        __syncwarp();
      }
    }
    fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(&bars->tdone);
  }
}

// (a CTA, and a round of two key tiles or a tile of its chain; the start and the end of a second grid)
constexpr double kSplitCtaUs = 8.5, kSplitRoundUs = 1.3, kPairCtaUs = 8.5, kPairTileUs = 1.54, kLateUs = 1.5, kTwoGridsUs = 3.0;

template <int D, bool SPLIT>
cudaError_t launch_slots(const PrefillTcParams& p, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv,
                         int dev, cudaStream_t s) {
  static bool configured[64] = {};
  if (dev >= 0 && dev < 64 && !configured[dev]) {
    cudaError_t e = cudaFuncSetAttribute(prefill_tc_kernel<D, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Cfg<D>::kSmemBytes);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  if ((int64_t)p.n_qt * p.h_kv > INT32_MAX) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.n_qt * p.h_kv));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = Cfg<D>::kSmemBytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = p.after ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, prefill_tc_kernel<D, SPLIT>, p, mq, mk, mv);
}

// SM count of a device (it does not change).
int sm_count(int dev) {
  static int n[64] = {};
  if (dev < 0 || dev >= 64) return 148;
  if (n[dev] == 0 && cudaDeviceGetAttribute(&n[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) n[dev] = 148;
  return n[dev];
}

template <int D>
cudaError_t launch(const PrefillTcParams& p, const void* q, const void* k, const void* v, cudaStream_t s) {
  CUtensorMap mq, mk, mv;
  if (!tma_map(&mq, q, D, p.h_q, p.n_tokens, p.group, p.tps) || !tma_map(&mk, k, D, p.h_kv, p.n_tokens, 1, kBN) ||
      !tma_map(&mv, v, D, p.h_kv, p.n_tokens, 1, kBN))
    return cudaErrorInvalidValue;
  int dev = 0;
  cudaGetDevice(&dev);
  // Two slots of queries per CTA are the better use of a full GPU, one slot with its key tiles
  // shared out of a short sequence: there a CTA's chain of tiles is the whole time.  Each is
  // costed as its longest CTA and, where it needs a second wave, the first CTA of that behind
  // the shortest of the first (CTAs start in descending order), with the costs measured on
  // GB300: us per call for 512 + 160 tokens, 28/4 heads, 16.9 with two slots, 14.5 split; 1500 +
  // 160, 16/1 heads, 29.0 and 22.8; but 1300 + 160, 28/4 heads, 29.0 and 32.7.  head_dim 64 is
  // costed the same: what it has more of P.V it has less of loads (800 + 160, 32/8 heads, 24.4 with
  // two slots, 22.7 split; 1200 + 160, 29.2 and 31.7; 512 + 160, 14/2 heads, 18.6 and 12.9).
  const int sms = sm_count(dev);
  auto tiles_upto = [&](int64_t last) {        // key tiles of a query tile whose last token this is
    return last < p.prefix_len ? last / kBN + 1 : (p.prefix_len + kBN - 1) / kBN + 1;
  };
  auto cost = [&](int tpc, int tiles_per_round, double cta_us, double round_us) {
    const int64_t n_qt = ((int64_t)p.n_tokens + tpc - 1) / tpc, n = n_qt * p.h_kv;
    auto rounds = [&](int64_t cta) {
      const int64_t last = std::min<int64_t>((n_qt - cta / p.h_kv) * tpc, p.n_tokens) - 1;
      return (double)((tiles_upto(last) + tiles_per_round - 1) / tiles_per_round);
    };
    double t = cta_us + round_us * rounds(0);
    // (the second of two CTAs finds its code and parameters cached)
    if (n > sms) t = std::max(t, 1.8 * cta_us + round_us * (rounds(sms - 1) + rounds(sms)));
    return n > 2 * (int64_t)sms + sms / 16 ? 1e30 : t;  // (a few over two waves, the shortest, are no third)
  };
  const int64_t n_one = ((int64_t)p.n_tokens + p.tps - 1) / p.tps;  // query tiles of one slot
  const double split_us = cost(p.tps, 2, kSplitCtaUs, kSplitRoundUs), pair_us = cost(2 * p.tps, 1, kPairCtaUs, kPairTileUs);
  // Where the split form is some CTAs over one wave, the first tokens, whose key ranges are the
  // shortest, go in pairs instead, just enough of them that everything runs at once: a second grid,
  // which starts when the first one's CTAs have.  (us per call, split or pairs / two grids: 600 + 160 tokens,
  // 28/4 heads 18.7 / 16.8; 500 + 160, 32/8 heads 18.6 / 16.5; 700 + 160, 32/8 heads 20.7 / 18.6.)
  const int64_t pairs = n_one - sms / p.h_kv;
  PrefillTcParams a = p;
  if (pairs > 0 && 2 * pairs <= n_one) {
    const double mixed_us = kTwoGridsUs + std::max(kSplitCtaUs + kSplitRoundUs * (double)((tiles_upto(p.n_tokens - 1) + 1) / 2),
                                                   kLateUs + kPairCtaUs + kPairTileUs * (double)tiles_upto(2 * pairs * p.tps - 1));
    if (mixed_us < split_us && mixed_us < pair_us) {
      a.tok_base = (int32_t)(2 * pairs * p.tps);
      a.n_qt = (int32_t)(n_one - 2 * pairs);
      a.release = a.n_qt > 0;
      cudaError_t e = a.n_qt > 0 ? launch_slots<D, true>(a, mq, mk, mv, dev, s) : cudaSuccess;
      if (e != cudaSuccess) return e;
      a.after = a.release;
      a.release = 0;
      a.tok_base = 0;
      a.n_qt = (int32_t)pairs;
      return launch_slots<D, false>(a, mq, mk, mv, dev, s);
    }
  }
  const bool split = split_us < pair_us;
  a.n_qt = (int32_t)((p.n_tokens + (int64_t)(split ? 1 : 2) * p.tps - 1) / ((split ? 1 : 2) * p.tps));
  return split ? launch_slots<D, true>(a, mq, mk, mv, dev, s) : launch_slots<D, false>(a, mq, mk, mv, dev, s);
}

}  // namespace

// Device status word of the whole-sequence prefill (no plan or workspace is involved).
__device__ PadDevHeader g_prefill_header;

cudaError_t prefill_header(PadDevHeader** out) {
  static PadDevHeader* ptr[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!ptr[dev]) {
    void* a = nullptr;
    e = cudaGetSymbolAddress(&a, g_prefill_header);
    if (e != cudaSuccess) return e;
    ptr[dev] = static_cast<PadDevHeader*>(a);
  }
  *out = ptr[dev];
  return cudaSuccess;
}

cudaError_t launch_prefill_tc(int32_t n_tokens, int32_t prefix_len, int32_t n_branches, const int32_t* branch_len,
                              int32_t h_q, int32_t h_kv, int32_t head_dim, float scale, int32_t out_bf16, uint64_t gen,
                              const void* q, const void* k, const void* v, void* out, float* lse, cudaStream_t s) {
  const int G = h_q / h_kv;
  if (G < 1 || G > 128 || n_tokens <= 0 || n_branches < 0 || n_branches > kMaxBranches) return cudaErrorInvalidValue;
  PrefillTcParams p;
  p.n_tokens = n_tokens;
  p.prefix_len = prefix_len;
  p.n_branches = n_branches;
  p.h_q = h_q;
  p.h_kv = h_kv;
  p.group = G;
  p.tps = 128 / G;
  p.scale_log2 = (float)((double)scale * 1.4426950408889634);
  p.out_bf16 = out_bf16;
  p.gen = gen;
  p.tok_base = p.n_qt = p.release = p.after = 0;
  cudaError_t e = prefill_header(&p.header);
  if (e != cudaSuccess) return e;
  p.out = out;
  p.lse = lse;
  p.bstart[0] = prefix_len;
  for (int b = 0; b < n_branches; ++b) p.bstart[b + 1] = p.bstart[b] + branch_len[b];
  if (head_dim == 128) return launch<128>(p, q, k, v, s);
  if (head_dim == 64) return launch<64>(p, q, k, v, s);
  return cudaErrorInvalidValue;
}

}  // namespace pad

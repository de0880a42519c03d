// a3 on the 5th-generation tensor cores: split-KV flash-decode over the shared
// prefix (the part of the event-factorized mask of Sec. 3.4 that every branch
// of a video sees: the multimodal prefix P and all planning tokens G^1..G^K, S).
//
// One CTA per (work item = video, kv-head, prefix split; group of <= 128 query
// rows).  The R = E_b * G query rows of the video's events that read this
// kv-head form the M dimension of the MMA, so each K/V tile brought from HBM
// serves every event and every GQA head of the group at once; the row groups of
// one item are adjacent CTAs that run together and share the tiles through L2.
//
//   warp 0      TMA producer of K tiles (128 tokens: two 64-column halves, 128-byte
//               swizzle) into a 3-stage ring; a stage is refilled once the S of
//               the tile it held has completed
//   warp 1      S issuer: S = Q K^T into one of three TMEM S buffers, up to three tiles
//               ahead of the softmax
//   warp 2      TMEM allocator (512 columns) and deallocator, and issuer of O += P V with P
//               read back from TMEM
//   warp 3      TMA producer of V tiles (refilled once the P.V of the tile completed); clears
//               the rows of the last one that lie past the split's end
//   warps 4-11  softmax: two warps per 32-row lane quarter, each with 16 of the quarter's rows
//               and all 128 columns of a tile (two rows per thread, a row shared by a quad of
//               lanes), so the warps never meet.  Online sum in base 2, P written as packed
//               bf16 over the S columns already read; the row maxima are found on the first
//               tile, and again only when a row's sum shows that a score outgrew them by more
//               than 2^8 (then O is rescaled and the tile redone).
//
// What bounds it: on a long split the softmax's own instructions (about 1280 cycles per tile and
// CTA at 32 and 64 events, 180 of them waits; 16 ragged videos, one row group each: 1760, a third
// waits for K/V from HBM), on a short one the fixed cost per CTA.  Electing the issuing lane of a
// uniform warp instead of branching to lane 0 (see elect_one) and skipping the maximum took,
// per step of that time: prefix 32768, 32 events 24.8 -> 23.7 us; 16384, 64 events 25.6 -> 23.9;
// 16384, 1 event 12.0 -> 11.4; 8192, 8 events 10.75 -> 10.6; 16 ragged videos 94.3 -> 93.0.  With
// what followed here and in the branch/merge pass: 22.5, 21.6, 9.3, 8.5 and 84.
//
// head_dim 64 (one 64-column box per tile, P.V with N = 64) takes the same pipeline: 14/2 heads,
// prefix 16384, 16 events 24.0 us per step on the mma.sync kernel, 8.7 here; 4/1 heads, 512
// tokens, 4 events 14.3 -> 6.3 (latency: programmatic dependent launch and the one-call order
// come with this path).
//
// Every MMA has N = 128 (S: 128 tokens; P.V: 128 head-dim columns; 64 at head_dim 64), the size at
// which one tcgen05.mma carries as much tensor work as it costs to issue.
// TMEM columns: S[b] at 128*b (b = 0, 1, 2), O at 384.  Output: the partial
// softmax state (m, l, O) of every row for this split, merged with the other
// splits and the branch by the branch/merge kernel, or, when the plan fuses them
// (every (event, kv-head) task has a CTA of its own and the grid is one wave), by
// the softmax warps of this kernel after their split: they publish the split on a
// counter, then run one task's branch pass, wait for the counters of the task's rows
// and merge (a4 + a5 as in the standalone kernel, same code).
//
// Barrier phases: a thread waits for completion #c of a barrier by its parity, which is
// only sound while completion #c+1 cannot yet have happened.  Every barrier here is
// therefore per slot (stage, S buffer, or tile parity) so that its next completion
// depends on progress of the waiting thread itself.
//
// Every mbarrier wait is bounded (about one second of %globaltimer); a wait
// that runs out records PAD_ERR_DEVICE_TIMEOUT in the status word, raises a
// CTA-wide abort flag, lets the producers and the MMA issuer drain what they
// already started, frees TMEM and returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <algorithm>
#include <cstddef>
#include <cstdint>

#include "pad_branch_merge.cuh"
#include "pad_internal.h"
#include "pad_tc_common.cuh"

namespace pad {

namespace {

using namespace tc;

constexpr int kBN = 128;       // prefix tokens per K/V tile
constexpr int kStages = 3;
constexpr int kSBuf = 3;       // S buffers in TMEM
constexpr int kThreads = 384;
constexpr uint32_t kHalfBytes = kBN * 128;         // 128 tokens x 64 bf16 = 16 KB
constexpr uint32_t kQHalfBytes = 128 * 128;        // 128 rows x 64 bf16 = 16 KB
template <int D>
struct Cfg {
  static constexpr int kHalves = D / 64;                        // 64-column boxes of a row
  static constexpr uint32_t kTileBytes = kHalves * kHalfBytes;  // one K (or V) tile
  static constexpr uint32_t kOffQ = 0;                          // Q of the 128-row group
  static constexpr uint32_t kOffK = kHalves * kQHalfBytes;
  static constexpr uint32_t kOffV = kOffK + kStages * kTileBytes;
  static constexpr uint32_t kOffBar = kOffV + kStages * kTileBytes;
  static constexpr uint32_t kSmemBytes = kOffBar + 256;
  // head_dim 64: P as the sum of two bf16 numbers, each with its own P.V.  The mma.sync kernel of
  // this head size, whose place this one takes (above 8 rows), holds P in one bf16 on maxima of 64
  // tokens; one bf16 on the lazily followed maxima here is less exact (relative error of the
  // output 1.6e-3 against 1.4e-3), two are far more so (2e-6 where the branch is one key; longer
  // branches add the branch pass's own rounding, up to 3e-4).
  static constexpr bool kSplitP = D == 64;
  static constexpr uint32_t kIdescS = make_idesc(128, kBN, false);  // S = Q K^T: B = K tile, K-major
  static constexpr uint32_t kIdescPV = make_idesc(128, D, true);    // O += P V: B = V tile, N(=d)-major
  static_assert(kSmemBytes <= 232448, "fits the 227 KB opt-in shared memory");
};
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColO = 384;
constexpr float kRescaleSum = 256.0f;                 // a tile whose P sum to more (per thread) is redone

struct TcBars {
  uint64_t kfull[kStages];
  uint64_t vfull[kStages];
  uint64_t pvfree[kStages];   // P.V of the tile in this stage / S buffer has completed
  uint64_t sfull[kSBuf];      // S of the tile in this buffer has completed (also frees its K stage)
  uint64_t pfull[kSBuf];      // P of the tile in this buffer is written (8 warp arrivals)
  uint64_t drain_s;           // every S MMA has completed (S issuer)
  uint64_t drain_pv;          // every P.V MMA has completed (P.V issuer)
  uint64_t qready;            // Q staged in shared memory (8 warp arrivals)
  uint64_t tdone;             // the softmax warps are done with TMEM (8 warp arrivals)
  uint64_t vpart;             // the last V tile, where the split ends inside it, has landed
  uint64_t gen;               // the plan's generation, for the status word
  uint32_t tmem_base;
  int32_t abort;
};
static_assert(sizeof(TcBars) <= 256, "barrier block fits its slot");

// The softmax warps split a 128-row group by rows: warp w of lane quarter q takes the 16
// rows 32q + 16h .. +15 (h = (w-4)/4) and every column of a tile, through the 16-lane TMEM
// shapes, so no row is shared by two warps and they never have to meet.  Thread t holds rows
// a = t/4 and a + 8 of the warp's 16 and, in each 8-column chunk, columns 2(t%4) and
// 2(t%4) + 1: s[x][4k..4k+3] = (a, c), (a, c+1), (a+8, c), (a+8, c+1) with
// c = 64x + 8k + 2(t%4).  A row's maximum and sum are shared by the four threads of its
// quad (lanes 4(t/4) .. +3).
// Visible columns of one row: a range, or the set bits of a 128-column mask.
struct ColsRange {
  int lo, hi;
  __device__ bool vis(int c) const { return c >= lo && c < hi; }
};
struct ColsBits {
  uint64_t lo, hi;  // columns 0-63, 64-127
  __device__ bool vis(int c) const { return ((c < 64 ? lo >> c : hi >> (c - 64)) & 1ull) != 0; }
};
__device__ __forceinline__ float quad_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// Columns of this thread's two rows that a row does not see go to -inf: they then get P = 0
// and no say in the maximum.
template <class CA, class CB>
__device__ __forceinline__ void mask_rows(uint32_t (&s)[2][32], int cq, CA ca, CB cb) {
#pragma unroll
  for (int x = 0; x < 2; ++x)
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int c = 64 * x + 8 * k + cq + i;
        if (!ca.vis(c)) s[x][4 * k + i] = 0xff800000u;
        if (!cb.vis(c)) s[x][4 * k + 2 + i] = 0xff800000u;
      }
}

// Maxima of the raw scores of this thread's two rows over all 128 columns, reduced over the quad.
__device__ __forceinline__ void rows_max(const uint32_t (&s)[2][32], float& ma, float& mb) {
  float xa[4], xb[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) xa[u] = xb[u] = -__builtin_huge_valf();
#pragma unroll
  for (int x = 0; x < 2; ++x)
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      xa[k & 3] = max3f(xa[k & 3], __uint_as_float(s[x][4 * k]), __uint_as_float(s[x][4 * k + 1]));
      xb[k & 3] = max3f(xb[k & 3], __uint_as_float(s[x][4 * k + 2]), __uint_as_float(s[x][4 * k + 3]));
    }
  ma = quad_max(fmaxf(fmaxf(xa[0], xa[1]), fmaxf(xa[2], xa[3])));
  mb = quad_max(fmaxf(fmaxf(xb[0], xb[1]), fmaxf(xb[2], xb[3])));
}

// P = 2^(s * scale_log2 - m) of this thread's two rows, written as packed bf16 (two tokens
// per column: column 4k + t%4 of chunk k holds tokens 8k + 2(t%4) and + 1, the layout the
// P.V MMA reads) to the 64 TMEM columns at taddr_p; la / lb: this thread's share of each row's
// sum of P.
// SPLIT: what the rounding to bf16 leaves of P goes, rounded to bf16 too, to the next 64 columns.
template <bool SPLIT>
__device__ __forceinline__ void rows_exp(const uint32_t (&s)[2][32], float sl2, float ma, float mb, uint32_t taddr_p,
                                         float& la, float& lb) {
  const uint64_t sc2 = f2pack(sl2, sl2), na = f2pack(-ma, -ma), nb = f2pack(-mb, -mb);
  uint64_t acc_a[2] = {0ull, 0ull}, acc_b[2] = {0ull, 0ull};
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    uint32_t pk[16], rest[16];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint64_t ya =
          ffma2(f2pack(__uint_as_float(s[x][4 * k]), __uint_as_float(s[x][4 * k + 1])), sc2, na);
      const uint64_t yb =
          ffma2(f2pack(__uint_as_float(s[x][4 * k + 2]), __uint_as_float(s[x][4 * k + 3])), sc2, nb);
      const float a0 = ex2(f2lo(ya)), a1 = ex2(f2hi(ya)), b0 = ex2(f2lo(yb)), b1 = ex2(f2hi(yb));
      acc_a[k & 1] = fadd2(acc_a[k & 1], f2pack(a0, a1));
      acc_b[k & 1] = fadd2(acc_b[k & 1], f2pack(b0, b1));
      pk[2 * k] = pack_bf16(a0, a1);
      pk[2 * k + 1] = pack_bf16(b0, b1);
      if (SPLIT) {
        rest[2 * k] = pack_bf16(a0 - __uint_as_float(pk[2 * k] << 16), a1 - __uint_as_float(pk[2 * k] & 0xffff0000u));
        rest[2 * k + 1] =
            pack_bf16(b0 - __uint_as_float(pk[2 * k + 1] << 16), b1 - __uint_as_float(pk[2 * k + 1] & 0xffff0000u));
      }
    }
    // P columns 32x + 4k + t%4 (tokens 64x + 8k + 2(t%4), + 1)
    tmem_st16x128_x8(taddr_p + 32 * x, pk);
    if (SPLIT) tmem_st16x128_x8(taddr_p + 64 + 32 * x, rest);
  }
  const uint64_t sa = fadd2(acc_a[0], acc_a[1]), sb = fadd2(acc_b[0], acc_b[1]);
  la = f2lo(sa) + f2hi(sa);
  lb = f2lo(sb) + f2hi(sb);
}

// Bounded wait of this kernel: gives up on the CTA's abort flag or after the time limit.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, TcBars* bars,
                                          PadDevHeader* hdr, int where) {
  return mbar_wait_b(bar, parity, &bars->abort, bars->gen, hdr, where);
}


// The same for a whole warp (warp-uniform result).
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, TcBars* bars, PadDevHeader* hdr,
                                               int where) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, bars, hdr, where)) != 0;
}

// Split counters of the fused tail, one per (video, kv-head, 128-row group): bits 15-0
// count the video's splits that have written their partial rows, bits 31-16 the tasks
// that have taken them.  The append kernel of the step zeroes them; the last task to
// take a counter zeroes it again for a launch of the same plan without an append.
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* a) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
  return v;
}
// Thread `leader` waits (bounded) until every split of video `vd` has published the rows
// [r0, r0 + G) of kv-head `kvh`, then takes them; the result is the same for all 256
// threads of the softmax group.
__device__ __forceinline__ bool tail_partials_ready(const KParams& p, const PadVideoDesc& vd, int kvh,
                                                    int r0, bool leader) {
  bool good = true;
  if (leader) {
    const int G = p.group;
    const int gb = (vd.n_events * G + 127) >> 7;
    const int g0 = r0 >> 7, g1 = (r0 + G - 1) >> 7;
    unsigned* base = p.counters + vd.cnt_base + (size_t)kvh * gb;
    const unsigned long long t0 = globaltimer();
    for (int g = g0; g <= g1 && good; ++g) {
      while ((int)(ld_acquire_u32(base + g) & 0xffffu) != vd.n_splits) {
        // give up at once if this plan's kernels already recorded an error (a split that
        // failed never publishes), else after the usual bound
        const unsigned long long hw = *reinterpret_cast<volatile unsigned long long*>(&p.header->word);
        if (((hw >> 8) == p.gen && (hw & 0xffull) != 0) || globaltimer() - t0 > kWaitNs) {
          pad_set_error(p.header, p.gen, PAD_ERR_DEVICE_TIMEOUT, (int)blockIdx.x, g, 20);
          good = false;
          break;
        }
        __nanosleep(64);
      }
    }
    if (good) {
      for (int g = g0; g <= g1; ++g) {
        const int lo = (g << 7) / G, hi = min(vd.n_events - 1, ((g << 7) + 127) / G);
        const unsigned old = atomicAdd(base + g, 1u << 16);
        if ((int)(old >> 16) + 1 == hi - lo + 1) atomicExch(base + g, 0u);
      }
    }
  }
  return bm::SyncNamed{1}.all(good);
}

template <int D, bool ROPE, bool GSELF>
__global__ void __launch_bounds__(kThreads, 1)
    prefix_tc_kernel(const __grid_constant__ KParams p, const __nv_bfloat16* __restrict__ q, const int n_groups,
                     const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                     const __nv_bfloat16* __restrict__ kpool, const __nv_bfloat16* __restrict__ vpool,
                     void* __restrict__ out, float* __restrict__ lse) {
  using C = Cfg<D>;
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t sbase = smem_u32(smem);
  if (sbase & 1023u) {  // the 128-byte swizzle atoms need 1024-byte alignment (never expected)
    if (threadIdx.x == 0) pad_set_error(p.header, p.gen, PAD_ERR_UNSUPPORTED, (int)blockIdx.x, (int)sbase, 0);
    return;
  }
  TcBars* bars = reinterpret_cast<TcBars*>(smem + C::kOffBar);
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  // Launched so that it may start while the grid before it (the previous step, this step's
  // append, or the caller's own kernel that wrote q) finishes.  Barrier set-up and TMEM
  // allocation overlap that grid, and so does the first K/V tile of a one-call step; every
  // thread that touches other global memory waits for it first (the Q loads), and the block
  // barrier after them orders everything else, including the release of the grid behind this one.

  // the CTA's work item and 128-row group: from the plan's CTA list, or the dense grid
  int item, group;
  if (p.cta_map) {
    const int v = plan_tasks(p)[blockIdx.x];
    item = v >> 6;
    group = v & 63;
  } else {
    item = blockIdx.x / n_groups;
    group = blockIdx.x - item * n_groups;
  }
  const PadWorkItem it = plan_items(p)[item];
  const int R = it.n_events * p.group;
  const int row0 = group * 128;
  if (row0 >= R) return;  // uniform over the CTA, before any barrier or allocation
  const int ntok = it.tok_end - it.tok_begin;
  const int n_tiles = (ntok + kBN - 1) / kBN;
  const int kvh = it.kvh;
  const int tok0 = (int)it.tok0;
  // Tokens past the split's end stay out of its V tiles (see zero_v_rows).  Where the prefix has 128
  // tokens up to there, the last tile ends with the split: it starts that much earlier, and the columns
  // that it shares with the tile before are masked.  A shorter prefix (one tile) would run into
  // whatever lies ahead of it instead: its V tile is loaded to a barrier of its own, and becomes full
  // (vfull) once the producer has cleared its rows past the end.  (Cleared so, 4000 tokens, 3 events
  // took 8.5 us per step instead of 8.2.)
  const bool whole = it.tok_end >= kBN, part = !whole && ntok % kBN != 0;
  const int last_tok = whole ? ntok - kBN : 0;   // of the split: where its last tile starts
  auto load_tile = [&](const CUtensorMap* map, uint32_t off, int t, uint64_t* full) {
    mbar_expect_tx(full, C::kTileBytes);
#pragma unroll
    for (int h = 0; h < C::kHalves; ++h)
      tma_load_3d(sbase + off + h * kHalfBytes, map, 64 * h, kvh, tok0 + min(t * kBN, last_tok), full);
  };

  // The softmax warps load their Q rows now, so that the loads overlap barrier set-up
  // and TMEM allocation; they are stored to shared memory after the block barrier.
  // Lane `lane` of warp w holds rows 32*(w&3) + (lane+32i)/8, 16-byte chunk (lane+32i)%8: of
  // head-dim half (w-4)/4 for i = 0 .. 7 (head_dim 128), or of the one half there is for the
  // four i from 4 ((w-4)/4) on (head_dim 64).  Rows past R are zero.
  constexpr int kQi = 4 * C::kHalves;
  uint4 qv[kQi];
  // RoPE: element d < D/2 pairs with d + D/2, i.e. 16-byte chunk cc with chunk cc + D/16 of the same
  // row.  A thread takes whole pairs instead (pair (t + 64 i) % (D/16) of the row (t + 64 i) /
  // (D/16) of the quarter, t over its two warps), with the table entries beside them, so that
  // everything is one round of loads and the rotation stays in registers (rotating rows already in
  // shared memory, with a barrier and a second round for the table: 2.1 us more per step).
  constexpr int kPairs = D / 16, kRi = 32 * kPairs / 64;
  float4 tbl[ROPE ? 4 * kRi : 1];
  if (warp >= 4) {
    // The addresses come first: their divisions, 8 to a thread, and the code for them, which a
    // launch finds in no instruction cache, took 1000 to 2000 cycles between the wait and the
    // loads (us per step: prefix 8192, 8 events 9.7, now 8.9; 32768, 32 events 23.1, now 22.2).
    const int lane_base = 32 * (warp & 3), half = (warp - 4) >> 2;
    constexpr int kLd = ROPE ? kRi : kQi;
    // this thread's 16-byte piece of its rows (with RoPE, and the one kPairs after it)
    const int cc = ROPE ? lane % kPairs : (D == 128 ? half * 8 : 0) + (lane & 7);
    const uint4* src[kLd];                    // in its rows of q, NULL past R
    int pos[ROPE ? kRi : 1];
#pragma unroll
    for (int i = 0; i < kLd; ++i) {
      const int qrow = row0 + lane_base +
                       (ROPE ? (half * 32 + lane + 64 * i) / kPairs : (lane + 32 * (D == 128 ? i : i + 4 * half)) >> 3);
      const int el = qrow / p.group, gh = qrow - el * p.group, ev = it.first_event + el;
      src[i] = qrow < R ? reinterpret_cast<const uint4*>(q) + (size_t)(ev * p.h_q + kvh * p.group + gh) * (D / 8) + cc : nullptr;
      if (ROPE) pos[i] = qrow < R ? plan_events(p)[ev].pos : 0;
    }
#pragma unroll
    for (int i = 0; i < kLd; ++i) asm volatile("" : "+l"(src[i]));  // (not sunk behind the wait)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // (past L1 and never through the read-only path, see rope_chunk8: the grid ahead may have
    // been writing q while this one was resident)
#pragma unroll
    for (int i = 0; i < kLd; ++i) {
      if constexpr (ROPE) {
        qv[2 * i] = qv[2 * i + 1] = make_uint4(0u, 0u, 0u, 0u);
        tbl[4 * i] = tbl[4 * i + 1] = tbl[4 * i + 2] = tbl[4 * i + 3] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (src[i] != nullptr) {
          qv[2 * i] = __ldcg(src[i]);
          qv[2 * i + 1] = __ldcg(src[i] + kPairs);
          const float4* cs = reinterpret_cast<const float4*>(p.rope_cs + (size_t)pos[i] * D + 8 * cc);
          tbl[4 * i] = __ldcg(cs);
          tbl[4 * i + 1] = __ldcg(cs + 1);
          tbl[4 * i + 2] = __ldcg(cs + D / 8);
          tbl[4 * i + 3] = __ldcg(cs + D / 8 + 1);
        }
      } else {
        qv[i] = src[i] != nullptr ? __ldcg(src[i]) : make_uint4(0u, 0u, 0u, 0u);
      }
    }
  }

  if (threadIdx.x == 0) {
    // The first K and V tile go out first (their barriers initialised, then the loads),
    // before the other barriers, TMEM allocation and the block barrier; the producer warps
    // issue the rest once that K tile has landed, so that every CTA's first tile is not
    // queued in DRAM behind the later tiles of all the others.  In a one-call step the prefix
    // K/V is written by no grid that may run ahead of this one (none of the library's own, and by
    // that call's contract none that releases its dependents before its writes), so that tile is
    // requested even before the wait for the grid ahead; nothing else is.  The attention call of
    // a two-call step has no such contract, and the append ahead of it releases this grid while
    // it still waits itself, for a grid that may be writing the prefix: there the tile is only
    // fetched into L2 ahead of the wait, and read after it.  (us per step, read ahead / fetched / neither:
    // 16384 tokens, 1 event 10.4 / 10.5 / 10.7; head_dim 64, 8000 tokens, 9 events 10.6 / 10.4 / 10.8;
    // 8219 tokens, 13 events with RoPE, which waits for q and its table anyway, 12.7 / 13.1 / 13.1.)
    mbar_init(&bars->kfull[0], 1);
    mbar_init(&bars->vfull[0], 1);
    mbar_init(&bars->vpart, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmK)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmV)) : "memory");
    if (p.k_new == nullptr) {
      if (n_tiles > 0) {
#pragma unroll
        for (int h = 0; h < C::kHalves; ++h) {
          tma_prefetch_3d(&tmK, 64 * h, kvh, tok0 + min(0, last_tok));
          tma_prefetch_3d(&tmV, 64 * h, kvh, tok0 + min(0, last_tok));
        }
      }
      asm volatile("griddepcontrol.wait;" ::: "memory");
    }
    if (n_tiles > 0) {
      load_tile(&tmK, C::kOffK, 0, &bars->kfull[0]);
      load_tile(&tmV, C::kOffV, 0, part && n_tiles == 1 ? &bars->vpart : &bars->vfull[0]);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int s = 0; s < kStages; ++s) {
      if (s > 0) {
        mbar_init(&bars->kfull[s], 1);
        mbar_init(&bars->vfull[s], 1);
      }
      mbar_init(&bars->pvfree[s], 1);
    }
    for (int b = 0; b < kSBuf; ++b) {
      mbar_init(&bars->sfull[b], 1);
      mbar_init(&bars->pfull[b], 8);  // one arrival per softmax warp
    }
    mbar_init(&bars->drain_s, 1);
    mbar_init(&bars->drain_pv, 1);
    mbar_init(&bars->qready, 8);
    mbar_init(&bars->tdone, 8);
    bars->abort = 0;
    bars->gen = p.gen;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&bars->tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }

  fence_before();
  __syncthreads();
  fence_after();
  // The grid launched after this one (the branch/merge pass) may start its own
  // prologue now; it waits for this grid's completion before it reads partials.  With
  // the fused tail of a two-call step the next grid is the next step's append, which
  // must not overwrite partials that the tail still reads: no early release there.  The
  // next one-call step waits for this grid before it touches anything, so it may start.
  if (p.k_new != nullptr || !p.fused) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // an allocation of all 512 columns starts at TMEM address 0: known at compile time, so that
  // the MMAs' TMEM operands are immediates (a word read back from shared memory is not)
  constexpr uint32_t tmem = 0;

  if (warp == 0 || warp == 3) {
    // ------------------------------------------------------------ TMA producers
    const bool isK = warp == 0;
    bool ok = true;
    if (lane == 0) {
      const CUtensorMap* map = isK ? &tmK : &tmV;
      int issued = min(1, n_tiles);  // tile 0 went out in the prologue
      // the other stages fill once the first K tile has landed
      ok = n_tiles <= 1 || mbar_wait(&bars->kfull[0], 0u, bars, p.header, isK ? 1 : 2);
      for (int t = 1; t < n_tiles && ok; ++t) {
        const int s = t % kStages;
        if (t >= kStages) {
          // K stage: S of tile t-3 done (sfull[s], completion t/3 - 1); V stage: its P.V done
          uint64_t* freed = isK ? &bars->sfull[s] : &bars->pvfree[s];
          ok = mbar_wait(freed, (uint32_t)((t / kStages - 1) & 1), bars, p.header, isK ? 1 : 2);
          if (!ok) break;
        }
        uint64_t* full = isK ? &bars->kfull[s] : (part && t == n_tiles - 1 ? &bars->vpart : &bars->vfull[s]);
        load_tile(map, (isK ? C::kOffK : C::kOffV) + s * C::kTileBytes, t, full);
        issued = t + 1;
      }
      if (!ok) {
        // the loads already issued must land before the CTA leaves
        for (int t = max(0, issued - kStages); t < issued; ++t) {
          uint64_t* full = isK ? &bars->kfull[t % kStages] : &bars->vfull[t % kStages];
          if (!isK && part && t == n_tiles - 1)
            drain_wait(&bars->vpart, 0u);
          else
            drain_wait(full, (uint32_t)((t / kStages) & 1));
        }
      }
    }
    __syncwarp();
    if (!isK && part && __shfl_sync(0xffffffffu, (int)ok, 0)) {
      const int s = (n_tiles - 1) % kStages;
      if (mbar_wait_warp(&bars->vpart, 0u, bars, p.header, 7)) {
        zero_v_rows<C::kHalves>(smem + C::kOffV + s * C::kTileBytes, ntok % kBN, lane, 32);
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->vfull[s]);
      } else {
        drain_wait(&bars->vpart, 0u);
      }
    }
    if (warp == 0 && !p.causal) prefetch_branch_tasks<D>(p, q, kpool, vpool, lane);
  } else if (warp == 1 || warp == 2) {
    // ------------------------------------------------------------ MMA issuers
    // Two warps feed the tensor pipe so that one's waits and commits overlap the other's MMAs:
    // warp 1 issues S = Q K^T, warp 2 (after allocating TMEM) issues O += P V.  Each runs its
    // loop with all lanes and lets the elected one issue (see elect_one).  A commit tracks
    // only its own thread's MMAs, so each has its own completion barriers (sfull / pvfree)
    // and drain.
    //
    // Descriptors are built once; a K-step moves the start address, i.e. adds
    // (byte offset >> 4) to the low field (no carry: addresses stay below 256 KB).
    const bool el = elect_one();
    bool ok = true;
    if (warp == 1) {
      const uint64_t dQ = sdesc(sbase + C::kOffQ, 16, 1024);
      const uint64_t dK = sdesc(sbase + C::kOffK, 16, 1024);
      ok = mbar_wait_warp(&bars->qready, 0u, bars, p.header, 11);
      int s = 0;
      uint32_t ph = 0;
      for (int t = 0; t < n_tiles && ok; ++t) {
        ok = mbar_wait_warp(&bars->kfull[s], ph, bars, p.header, 3);
        if (!ok) break;
        // S buffer s holds P of tile t-3 until that P.V completes
        if (t >= kStages) ok = mbar_wait_warp(&bars->pvfree[s], ph ^ 1u, bars, p.header, 6);
        if (!ok) break;
        fence_after();
        const uint32_t d = tmem + 128u * (uint32_t)s;
        const uint64_t kb = dK + ((uint32_t)s * C::kTileBytes >> 4);
        if (el) {
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            const uint32_t off = (uint32_t)(kk >> 2) * kQHalfBytes + (uint32_t)(kk & 3) * 32;
            mma_ss(d, dQ + (off >> 4), kb + (off >> 4), C::kIdescS, kk > 0 ? 1u : 0u);
          }
          mma_commit(&bars->sfull[s]);
        }
        __syncwarp();
        if (++s == kStages) {
          s = 0;
          ph ^= 1u;
        }
      }
      if (el) mma_commit(&bars->drain_s);
      __syncwarp();
      drain_wait(&bars->drain_s, 0u);
    } else {
      // V tile, N(=head-dim)-major: 16 tokens per step (2048 bytes), the second
      // 64-column half at +kHalfBytes (leading byte offset), 8-row groups 1024 apart.
      const uint64_t dV = sdesc(sbase + C::kOffV, kHalfBytes, 1024);
      int s = 0;
      uint32_t ph = 0;
      for (int j = 0; j < n_tiles && ok; ++j) {
        ok = mbar_wait_warp(&bars->vfull[s], ph, bars, p.header, 4);
        if (!ok) break;
        ok = mbar_wait_warp(&bars->pfull[s], ph, bars, p.header, 5);
        if (!ok) break;
        fence_after();
        const uint32_t a = tmem + 128u * (uint32_t)s;
        const uint64_t vb = dV + ((uint32_t)s * C::kTileBytes >> 4);
        if (el) {
#pragma unroll
          for (int kk = 0; kk < kBN / 16; ++kk)
            mma_ts(tmem + kColO, a + kk * 8, vb + ((uint32_t)kk * 2048 >> 4), C::kIdescPV, (j > 0 || kk > 0) ? 1u : 0u);
          if (C::kSplitP) {
#pragma unroll
            for (int kk = 0; kk < kBN / 16; ++kk)
              mma_ts(tmem + kColO, a + 64 + kk * 8, vb + ((uint32_t)kk * 2048 >> 4), C::kIdescPV, 1u);
          }
          mma_commit(&bars->pvfree[s]);
        }
        __syncwarp();
        if (++s == kStages) {
          s = 0;
          ph ^= 1u;
        }
      }
      // O is final once every P.V has completed
      if (el) mma_commit(&bars->drain_pv);
      __syncwarp();
      drain_wait(&bars->drain_pv, 0u);
    }
  } else if (warp >= 4) {
    // ------------------------------------------------------------ softmax
    const int quarter = warp & 3;              // TMEM lanes 32*quarter .. +31 (query rows)
    const int half = (warp - 4) >> 2;          // rows 16*half .. +15 of the quarter
    const int lane_base = 32 * quarter;
    // Q rows (loaded in the prologue) into the 128-byte-swizzled K-major layout the
    // MMA reads: row r, 16-byte chunk cc of half h at h*16K + r*128 + ((cc ^ (r & 7)) << 4).
    auto q_slot = [&](int r, int chunk) {  // chunk of the whole row
      return reinterpret_cast<uint4*>(smem + C::kOffQ + (chunk >> 3) * kQHalfBytes + r * 128 +
                                      (((chunk & 7) ^ (r & 7)) << 4));
    };
    if constexpr (ROPE) {
#pragma unroll
      for (int i = 0; i < kRi; ++i) {
        const int k = half * 32 + lane + 64 * i;
        const int r = lane_base + k / kPairs, cc = k % kPairs;
        const uint4 a = qv[2 * i], b = qv[2 * i + 1];
        const float4 c0 = tbl[4 * i], c1 = tbl[4 * i + 1], s0 = tbl[4 * i + 2], s1 = tbl[4 * i + 3];
        const float c[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
        const float s[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
        const uint32_t av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
        uint32_t ol[4], oh[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&av[j]));
          const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&bv[j]));
          const __nv_bfloat162 l2 = __floats2bfloat162_rn(rope_one(x.x, y.x, c[2 * j], s[2 * j], true),
                                                          rope_one(x.y, y.y, c[2 * j + 1], s[2 * j + 1], true));
          const __nv_bfloat162 h2 = __floats2bfloat162_rn(rope_one(y.x, x.x, c[2 * j], s[2 * j], false),
                                                          rope_one(y.y, x.y, c[2 * j + 1], s[2 * j + 1], false));
          ol[j] = *reinterpret_cast<const uint32_t*>(&l2);
          oh[j] = *reinterpret_cast<const uint32_t*>(&h2);
        }
        *q_slot(r, cc) = make_uint4(ol[0], ol[1], ol[2], ol[3]);
        *q_slot(r, cc + kPairs) = make_uint4(oh[0], oh[1], oh[2], oh[3]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < kQi; ++i) {
        const int idx = lane + 32 * (D == 128 ? i : i + 4 * half);
        *q_slot(lane_base + (idx >> 3), (D == 128 ? half * 8 : 0) + (idx & 7)) = qv[i];
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(&bars->qready);
    const float sl2 = p.scale_log2;
    bool ok = true;
    {
      // this warp's 16 rows (TMEM lanes), this thread's two of them and its first column of
      // every 8-column chunk
      const int wrow = lane_base + 16 * half;
      const int ra = wrow + (lane >> 2), rb = ra + 8;
      const int ga = row0 + ra, gb = row0 + rb;
      const int cq = 2 * (lane & 3);
      const bool warp_active = (row0 + wrow) < R;
      const uint32_t tl = tmem + ((uint32_t)wrow << 16);
      float m_a = -__builtin_huge_valf(), m_b = -__builtin_huge_valf(), l_a = 0.f, l_b = 0.f;
      // self G-token mask: the video's planning tokens G^1..G^K (prefix-relative [g_lo, g_hi))
      // and each row's own one
      int g_lo = 0, g_hi = 0, g_oa = -1, g_ob = -1;
      if (GSELF) {
        const PadVideoDesc vdg = plan_videos(p)[plan_events(p)[it.first_event].video];
        if (vdg.n_planning > 0) {
          g_lo = vdg.prefix_len - 1 - vdg.n_planning;
          g_hi = vdg.prefix_len - 1;
          if (ga < R) g_oa = g_lo + plan_events(p)[it.first_event + ga / p.group].gidx;
          if (gb < R) g_ob = g_lo + plan_events(p)[it.first_event + gb / p.group].gidx;
        }
      }
      uint32_t sr[2][32];
      for (int j = 0; j < n_tiles; ++j) {
        const uint32_t cS = 128u * (uint32_t)(j % kSBuf);
        ok = mbar_wait(&bars->sfull[j % kSBuf], (uint32_t)((j / kSBuf) & 1), bars, p.header, 8);
        ok = __all_sync(0xffffffffu, ok);  // tcgen05.ld/st below are warp-collective
        if (!ok) break;
        fence_after();
        if (warp_active) {
          const int valid = min(kBN, ntok - j * kBN);  // valid columns of the tile
          tmem_ld16x256_x8(tl + cS, sr[0]);
          tmem_ld16x256_x8(tl + cS + 64, sr[1]);
          tmem_wait_ld_dep(sr[0]);
          tmem_wait_ld_dep(sr[1]);
          // columns to mask: past the split's end, or (GSELF) hidden planning tokens of the
          // row's event; the path is chosen per warp (tcgen05.st below is warp-collective)
          // (the last tile's columns: those from `lo` on, or the first `hi`, see `whole`)
          const int lo = whole ? kBN - valid : 0, hi = whole ? kBN : valid;
          if (GSELF) {
            ColsBits ka{~0ull, ~0ull}, kb{~0ull, ~0ull};
            const int t0 = it.tok_begin + j * kBN - lo;
            if (valid < kBN || (t0 < g_hi && t0 + kBN > g_lo)) {
              const GMask gma{g_lo, g_hi, g_oa}, gmb{g_lo, g_hi, g_ob};
              const uint64_t f0 = lo >= 64 ? 0ull : ~0ull << lo, f1 = lo > 64 ? ~0ull << (lo - 64) : ~0ull;
              ka = ColsBits{keep_bits(hi, gma, t0) & f0, keep_bits(hi - 64, gma, t0 + 64) & f1};
              kb = ColsBits{keep_bits(hi, gmb, t0) & f0, keep_bits(hi - 64, gmb, t0 + 64) & f1};
            }
            if (__any_sync(0xffffffffu, (ka.lo & ka.hi & kb.lo & kb.hi) != ~0ull)) mask_rows(sr, cq, ka, kb);
          } else if (valid < kBN) {
            mask_rows(sr, cq, ColsRange{lo, hi}, ColsRange{lo, hi});
          }
          // P of the tile on the running maxima, over the first 64 columns of its S buffer, in
          // this warp's own rows.  The sums (ta, tb: this thread's share), which the row sums need
          // anyway, show whether the maxima still bound the scores: a sum of at most 2^8 means
          // that every P is.  Only a tile that exceeds it, and the first, which has no maxima
          // yet, finds its maxima (`fresh`), rescales O and l to them and is done on those.
          // (One copy of the exponentials in a loop over the two attempts, or the first tile's
          // maximum ahead of a shared copy, was 0.6-0.7 us slower per 32768-token step.)
          float ta, tb;
          auto exps = [&]() {
            // (a row with every key so far hidden keeps m = -inf; its exponent base is 0)
            rows_exp<C::kSplitP>(sr, sl2, m_a == -__builtin_huge_valf() ? 0.f : m_a, m_b == -__builtin_huge_valf() ? 0.f : m_b,
                     tl + cS, ta, tb);
          };
          bool fresh = j == 0;
          if (!fresh) {
            exps();
            fresh = __any_sync(0xffffffffu, (ga < R && (m_a == -__builtin_huge_valf() || ta > kRescaleSum)) ||
                                                (gb < R && (m_b == -__builtin_huge_valf() || tb > kRescaleSum)));
          }
          if (fresh) {
            if (j > 0) {
              // O must hold P.V of tile j-1 before its rows are rescaled
              ok = mbar_wait(&bars->pvfree[(j - 1) % kStages], (uint32_t)(((j - 1) / kStages) & 1), bars,
                             p.header, 9);
              ok = __all_sync(0xffffffffu, ok);
              if (!ok) break;
              fence_after();
            }
            float mxa, mxb;
            rows_max(sr, mxa, mxb);
            const float na = fmaxf(m_a, mxa * sl2), nb = fmaxf(m_b, mxb * sl2);
            if (j > 0) {
              const float al_a = na > m_a ? ex2(m_a - na) : 1.f, al_b = nb > m_b ? ex2(m_b - nb) : 1.f;
#pragma unroll 1
              for (int x = 0; x < D / 32; ++x) {
                uint32_t o[16];
                tmem_ld16x256_x4(tl + kColO + 32 * x, o);
                tmem_wait_ld_dep16(o);
#pragma unroll
                for (int i = 0; i < 16; ++i)
                  o[i] = __float_as_uint(__uint_as_float(o[i]) * ((i & 2) ? al_b : al_a));
                tmem_st16x256_x4(tl + kColO + 32 * x, o);
              }
              l_a *= al_a;
              l_b *= al_b;
            }
            m_a = na;
            m_b = nb;
            exps();
          }
          l_a += ta;
          l_b += tb;
          tmem_wait_st();
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->pfull[j % kSBuf]);
      }
      // the P.V issuer commits `drain_pv` after its last MMA: O is final once it lands
      if (ok) ok = mbar_wait(&bars->drain_pv, 0u, bars, p.header, 10);
      ok = __all_sync(0xffffffffu, ok);
      if (ok && warp_active) {
        fence_after();
        // O rows straight from the 16-lane layout: a quad writes 32 contiguous bytes of a
        // row, a warp instruction eight such segments
        float* po_a = p.part_o + ((int64_t)it.part_row0 + ga) * D;
        float* po_b = po_a + 8 * D;
#pragma unroll
        for (int x = 0; x < C::kHalves; ++x) {
          uint32_t o[32];
          tmem_ld16x256_x8(tl + kColO + 64 * x, o);
          tmem_wait_ld_dep(o);
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int c = 64 * x + 8 * k + cq;
            if (ga < R)
              *reinterpret_cast<float2*>(po_a + c) = make_float2(__uint_as_float(o[4 * k]), __uint_as_float(o[4 * k + 1]));
            if (gb < R)
              *reinterpret_cast<float2*>(po_b + c) =
                  make_float2(__uint_as_float(o[4 * k + 2]), __uint_as_float(o[4 * k + 3]));
          }
        }
        const float la = quad_sum(l_a), lb = quad_sum(l_b);
        if ((lane & 3) == 0) {
          if (ga < R) p.part_ml[(int64_t)it.part_row0 + ga] = make_float2(m_a, la);
          if (gb < R) p.part_ml[(int64_t)it.part_row0 + gb] = make_float2(m_b, lb);
        }
      }
    }
    // TMEM is freed by warp 2 only after every softmax warp has arrived here
    fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(&bars->tdone);
    // every softmax warp reaches this barrier exactly once (the loop above only breaks);
    // it orders the partial rows before the fused tail
    if (D == 128 && p.fused) asm volatile("bar.sync 1, 256;" ::: "memory");
    if (D == 128 && p.fused) {  // (head_dim 64 plans have no fused tail)
      // ---------------------------------------------------------- fused a4 + a5
      // Publish this split's rows (every softmax thread's partial stores are ordered
      // before the counter by the barrier and the fence), then run this CTA's (event,
      // kv-head) task with all of shared memory below the barriers (the Q, K and V
      // stages are idle once the last MMA has completed).
      const bm::SyncNamed sy{1};
      if (sy.all(ok)) {
        if (threadIdx.x == 128) {
          // the append kernel ahead zeroes the counters: wait for it (long complete by now)
          asm volatile("griddepcontrol.wait;" ::: "memory");
          __threadfence();
          const PadVideoDesc vd = plan_videos(p)[plan_events(p)[it.first_event].video];
          atomicAdd(p.counters + vd.cnt_base + (size_t)kvh * ((R + 127) >> 7) + group, 1u);
        }
        const int task = plan_tasks(p)[blockIdx.x];
        if (task >= 0) {
          const int te = task / p.h_kv, th = task - (task / p.h_kv) * p.h_kv;
          bm::run_task<D, ROPE, 2>(p, q, kpool, vpool, out, lse, te, th, (int)threadIdx.x - 128, smem, p.tail_chunk, sy,
                           false, [&]() {
                             const PadEventDesc ev = plan_events(p)[te];
                             const PadVideoDesc vd = plan_videos(p)[ev.video];
                             return tail_partials_ready(p, vd, th, ev.local * p.group, threadIdx.x == 128);
                           });
        }
      }
    }
  }

  __syncwarp();
  fence_before();
  __syncthreads();
  if (warp == 2) {
    // The block barrier above is not relied on to order the softmax warps' last TMEM
    // reads before the deallocation (it was measured to let the role warps through
    // before them); their own arrivals are.
    drain_wait(&bars->tdone, 0u);
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols)
                 : "memory");
  }
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess)
      ptr = nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
  }();
  return fn;
}

}  // namespace

bool tma_map(CUtensorMap* map, const void* base, int D, int heads, int64_t tokens, int box_heads, int box_tokens) {
  auto enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)heads, (cuuint64_t)tokens};
  cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)heads * D * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)box_heads, (cuuint32_t)box_tokens};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool prefix_tensor_maps(const void* kp, const void* vp, int D, int h_kv, int64_t tokens, CUtensorMap* mk, CUtensorMap* mv) {
  return tma_map(mk, kp, D, h_kv, tokens, 1, kBN) && tma_map(mv, vp, D, h_kv, tokens, 1, kBN);
}

int prefix_tc_tail_chunk(int branch_rows, int group, int max_splits) {
  int sch = std::min(bm::kMaxChunk, std::max(1, max_splits));
  while (sch > 1 && bm::smem_bytes<128>(branch_rows, group, sch) > Cfg<128>::kOffBar) --sch;
  return sch;
}

template <int D>
static cudaError_t launch_d(const KParams& p, int max_rows, const void* q, const CUtensorMap& mk, const CUtensorMap& mv,
                            const void* k_pool, const void* v_pool, void* out, float* lse, bool pdl, int dev,
                            cudaStream_t s) {
  constexpr uint32_t smem = Cfg<D>::kSmemBytes;
  static bool configured[64] = {};
  if (dev >= 0 && dev < 64 && !configured[dev]) {
    for (auto fn : {prefix_tc_kernel<D, false, false>, prefix_tc_kernel<D, true, false>,
                    prefix_tc_kernel<D, false, true>, prefix_tc_kernel<D, true, true>}) {
      cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    configured[dev] = true;
  }
  const int n_groups = (max_rows + 127) / 128;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.cta_map ? p.n_ctas : p.n_items * n_groups);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (p.fused && (D != 128 || bm::smem_bytes<D>(p.branch_rows, p.group, p.tail_chunk) > Cfg<D>::kOffBar))
    return cudaErrorInvalidValue;
  auto fn = p.rope_cs != nullptr ? (p.g_self ? prefix_tc_kernel<D, true, true> : prefix_tc_kernel<D, true, false>)
                                 : (p.g_self ? prefix_tc_kernel<D, false, true> : prefix_tc_kernel<D, false, false>);
  return cudaLaunchKernelEx(&cfg, fn, p, static_cast<const __nv_bfloat16*>(q), n_groups, mk, mv,
                            static_cast<const __nv_bfloat16*>(k_pool), static_cast<const __nv_bfloat16*>(v_pool),
                            out, lse);
}

cudaError_t launch_prefix_tc(const KParams& p, int max_rows, const void* q, const void* kp,
                             const void* vp, int64_t total_prefix_tokens, const void* k_pool,
                             const void* v_pool, void* out, float* lse, bool pdl, cudaStream_t s) {
  if (p.n_items == 0) return cudaSuccess;
  if ((p.head_dim != 128 && p.head_dim != 64) || total_prefix_tokens <= 0 || total_prefix_tokens > (int64_t)INT32_MAX)
    return cudaErrorInvalidValue;
  int dev = 0;
  cudaGetDevice(&dev);
  CUtensorMap mk, mv;
  if (!prefix_tensor_maps(kp, vp, p.head_dim, p.h_kv, total_prefix_tokens, &mk, &mv)) return cudaErrorInvalidValue;
  return p.head_dim == 128 ? launch_d<128>(p, max_rows, q, mk, mv, k_pool, v_pool, out, lse, pdl, dev, s)
                           : launch_d<64>(p, max_rows, q, mk, mv, k_pool, v_pool, out, lse, pdl, dev, s);
}

}  // namespace pad

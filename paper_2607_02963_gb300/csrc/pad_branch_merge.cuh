// a4 + a5 for one (event, kv-head), run by 256 threads (8 warps): used by the standalone
// branch/merge kernel (one CTA per task) and by the tensor-core prefix kernel, whose
// softmax warps take one task each after their prefix split.
//
//   a4, the own-branch part of the mask of Sec. 3.4: the branch's keys 0..len, its
//   private tokens and the one appended at this step (under the "causal attention" mask
//   of the ablation: the stored tokens of every branch of the video, then its own new
//   one), in rounds of up to kKeys.  Each warp takes 16 of a round's keys, all by itself: its
//   lanes hold the places of two rounds' keys (page ids read beside the event's descriptor), it
//   copies their K and V rows to its own part of shared memory (cp.async) and keeps a
//   flash-attention state in registers in the manner of the warp-level MMA
//   kernels (the G <= 16 query rows form one m16 tile, S = Q K^T, online softmax on the
//   accumulators in base 2, O += P V with P re-packed from the S accumulators).  No warp waits
//   for another between the staging of Q and the fold of the states.
//   a5: the warp states and the prefix splits' partial states are merged by
//   log-sum-exp (Eq. for combining softmax states: M = max of the maxima, every state
//   weighted by 2^(m - M)), and O and the LSE are written once.
//
//   a2, when the step is one call (KParams::k_new set): key `len` is read from k_new /
//   v_new instead of the pools, and this task writes it into them (its page-table entry
//   too, by the kv-head-0 task of an event that took a new page).  No other task reads
//   this (event, kv-head)'s branch, so nothing else waits for that write.
//
// Staging before griddepcontrol.wait reads nothing the grids ahead write: Q rows, the
// branch's page ids (key `len`'s page is the one this step took, else the table's entry
// of an earlier step) and the K/V rows of keys 0..len-1, and key `len` itself when it
// comes from k_new / v_new, or when the append kernel wrote it and the prefix grid waited for
// that kernel before it released this one (KParams::keys_ready; two-call step, prefix 8219, 13
// events with RoPE: 16.0 -> 13.9 us).  That is all the branch pass reads, so the whole pass (and the
// merge of its warp states) runs before the wait.  After it: key `len` in the other two-call
// steps (the branch pass follows), and the splits' (m, l) pairs and O rows once the caller says they are complete
// (`partials_ready`: at once for the standalone kernel, whose wait covers the prefix
// grid; after the split counters for the tensor-core kernel).
//
// What bounds a task is its chain of latencies (a few thousand bytes per step of it), so the chain
// is kept short.  Cycles from a task's start to its fold / the fold / the merge of its splits, 4
// CTAs per SM (16 ragged videos, 1032 tasks), with keys staged by the whole CTA behind barriers,
// unpadded O rows and rows weighted by single warps: 11800 / 2900 / 2500, now 10200 / 1500 / 1300.
// us per step: 88.9 -> 84.3; prefix 32768, 32 events 23.8 -> 22.5; 16384, 64 events 24.1 -> 21.7;
// 8192, 8 events 9.8 -> 9.5.
#pragma once

#include <cuda_bf16.h>
#include <cstddef>
#include <cstdint>

#include "pad_internal.h"

namespace pad {
namespace bm {

constexpr int kThreads = 256;                 // threads of one task (the default of 8 warps)
constexpr int kWarps = kThreads / 32;
constexpr int kKeys = 16 * kWarps;            // branch keys staged per round, at most
constexpr int kMaxChunk = 64;                 // prefix splits merged per staged chunk
constexpr float kNegInf = -__builtin_huge_valf();

__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) / 16 * 16; }
__host__ __device__ constexpr size_t max_sz(size_t a, size_t b) { return a > b ? a : b; }

// Shared memory of a task: this head, then three regions sized per launch (16-byte aligned):
//   kv   per warp that has keys (nkr / 16 of them, nkr = round_keys): its 16 K rows [16][LD] and
//        V rows [16][W + 8] of a round; after the branch pass its O rows, fp32 [G][W + 8]
//   ml   the splits' (m, l) pairs of a chunk, [G][sch]
//   po   the splits' O rows of a chunk, fp32 [sch][G][W]
template <int D>
struct Head {
  static constexpr int LD = D + 8;            // padded bf16 row: ldmatrix rows in distinct banks
  __nv_bfloat16 q[16][LD];
  float wm[kWarps][16], wl[kWarps][16];       // each warp's branch state per row
};
// Keys staged per round by a task of NW warps (16 per warp), for a launch's branch_rows.
__host__ __device__ constexpr int round_keys(int branch_rows, int NW) {
  return branch_rows < 16 * NW ? branch_rows : 16 * NW;
}
// (W: the output columns of the task, see run_task)
// One warp's part of kv.  Its O rows fit (G <= 16); they are padded so that the rows of a store lie
// in different banks (unpadded, 8 rows on the same ones: about 2000 cycles with 16 warps per SM).
template <int D, int W = D>
constexpr size_t kWarpKv = (size_t)16 * (Head<D>::LD + W + 8) * 2;
template <int D, int W = D>
__host__ __device__ constexpr size_t kv_bytes(int nkr) {
  static_assert((size_t)16 * (W + 8) * 4 <= kWarpKv<D, W>, "a warp's O rows fit over its keys");
  return (size_t)(nkr / 16) * kWarpKv<D, W>;
}
template <int D, int NW = kWarps, int W = D>
__host__ __device__ constexpr size_t smem_bytes(int branch_rows, int G, int sch) {
  return align16(sizeof(Head<D>)) + kv_bytes<D, W>(round_keys(branch_rows, NW)) + align16((size_t)G * sch * 8) +
         (size_t)sch * G * W * 4;
}
// A task whose branch pass ends before its partials are staged (OVER) lays po over kv: ml first,
// then one region for both.
template <int D, int NW = kWarps, int W = D>
__host__ __device__ constexpr size_t smem_bytes_over(int branch_rows, int G, int sch) {
  return align16(sizeof(Head<D>)) + align16((size_t)G * sch * 8) +
         max_sz(kv_bytes<D, W>(round_keys(branch_rows, NW)), (size_t)sch * G * W * 4);
}

#ifdef __CUDACC__
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool pred) {
  unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  int n = pred ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(n));
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}
__device__ __forceinline__ void ldsm_x4(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3,
                                        const void* p) {
  unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(p));
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(a));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3,
                                          const void* p) {
  unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(p));
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(a));
}
__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Partial row of part `split` of (video, kv-head), row r.
__device__ __forceinline__ int64_t part_row(const PadVideoDesc& vd, int kvh, int split, int R, int r) {
  return (int64_t)vd.part_base + ((int64_t)kvh * vd.n_splits + split) * R + r;
}

// Barriers over the task's 256 threads: the whole CTA, or a named barrier.
struct SyncCta {
  __device__ void sync() const { __syncthreads(); }
  __device__ bool all(bool v) const { return __syncthreads_and(v) != 0; }
};
struct SyncNamed {
  int id;
  __device__ void sync() const { asm volatile("bar.sync %0, 256;" ::"r"(id) : "memory"); }
  __device__ bool all(bool v) const {
    int r;
    asm volatile(
        "{\n .reg .pred pi, po;\n setp.ne.s32 pi, %1, 0;\n bar.red.and.pred po, %2, 256, pi;\n"
        " selp.s32 %0, 1, 0, po;\n}\n"
        : "=r"(r)
        : "r"((int)v), "r"(id)
        : "memory");
    return r != 0;
  }
};

// One task.  `tid` in [0, 256); `smem` 16-byte aligned, smem_bytes<D>(branch_rows, G, sch)
// long.  `partials_ready()` is called by all 256 threads and returns false if the
// partials cannot be read (then only the status word is written).
// CAUSAL: 0 = the method's own-branch keys, 1 = the causal-attention key list, 2 = read
// KParams::causal at run time (separate instantiations keep the common one lean).
// W < D: the task is shared by D / W CTAs, each with the output columns w0 .. w0 + W - 1: all of
// them find the scores and the weights, but each stages and merges its own columns of V and of
// the split partials, which is most of what a task moves.  The first also appends and writes
// the LSE.
// OVER: the caller knows that the branch pass ends before the partials are staged (`pre` below),
// so both use the same shared memory.
template <int D, bool ROPE, int CAUSAL, int NW = kWarps, int W = D, bool OVER = false, class Sync, class Ready>
__device__ __forceinline__ void run_task(const KParams& p, const __nv_bfloat16* __restrict__ q,
                                         const __nv_bfloat16* __restrict__ kpool,
                                         const __nv_bfloat16* __restrict__ vpool, void* __restrict__ out,
                                         float* __restrict__ lse, int e, int kvh, int tid,
                                         unsigned char* smem, int sch, const Sync& sy, bool early,
                                         Ready partials_ready, int w0 = 0) {
  static_assert(NW >= 1 && NW <= kWarps, "warps per task");
  constexpr int NT = 32 * NW;
  constexpr int CH = D / 8;                   // 16-byte pieces of a bf16 row
  constexpr int KS = D / 16;                  // k-steps of S = Q K^T
  constexpr int OT = W / 8;                   // n8 tiles of O
  constexpr int W4 = W / 4;
  constexpr int LDV = W + 8;                  // padded bf16 V row
  constexpr int LDO = W + 8;                  // padded fp32 O row
  constexpr int LD = Head<D>::LD;
  Head<D>& S = *reinterpret_cast<Head<D>*>(smem);
  const int G = p.group;
  const int nkr = round_keys(p.branch_rows, NW);  // keys per round (multiple of 16, <= 16 NW)
  unsigned char* kv_raw = smem + align16(sizeof(Head<D>)) + (OVER ? align16((size_t)G * sch * 8) : 0);
  float2* sml = reinterpret_cast<float2*>(OVER ? smem + align16(sizeof(Head<D>)) : kv_raw + kv_bytes<D, W>(nkr));
  float* spo = reinterpret_cast<float*>(OVER ? kv_raw : reinterpret_cast<unsigned char*>(sml) + align16((size_t)G * sch * 8));

  const int warp = tid >> 5, lane = tid & 31;
  const int gq = lane >> 2, t4 = lane & 3;
  const int ps = p.page_size;
  const int kb0 = 16 * warp;                  // this warp's keys within a round
  __nv_bfloat16 (*sK)[LD] = reinterpret_cast<__nv_bfloat16 (*)[LD]>(kv_raw + warp * kWarpKv<D, W>);
  __nv_bfloat16 (*sV)[LDV] = reinterpret_cast<__nv_bfloat16 (*)[LDV]>(&sK[16][0]);
  const bool causal = CAUSAL == 2 ? p.causal != 0 : CAUSAL == 1;
  // Lanes 0..15 hold the places of the warp's keys of an even round, lanes 16..31 of the odd
  // round after it.  For the first two rounds of a branch the page table is read beside the
  // event's descriptor (the row is the event's own, entries past its length are not used).
  const int key0 = (lane < 16 ? 0 : nkr - 16) + kb0 + lane;
  const int pi0 = key0 / ps;
  int page0 = -1;
  if (!causal && kb0 < nkr && pi0 < p.max_pages) page0 = __ldcg(p.page_table + (size_t)e * p.max_pages + pi0);
  if (!ROPE) {
    for (int i = tid; i < 16 * CH; i += NT) {
      const int g = i / CH, c = i - (i / CH) * CH;
      const bool in = g < G;
      cp_async16(&S.q[g][c * 8], q + ((size_t)e * p.h_q + kvh * G + (in ? g : 0)) * D + c * 8, in);
    }
  }
  const PadEventDesc ev = plan_events(p)[e];
  const PadVideoDesc vd = plan_videos(p)[ev.video];
  const int R = vd.n_events * G;
  const int ns = vd.n_splits;
  const int rbase = ev.local * G;
  const int len = ev.len;                     // keys before this step; key `len` is this step's
  // The task's keys: its own branch's len + 1, or (causal mask) the stored tokens of every
  // branch of the video, branch by branch, then its own token of this step.  `own` is the
  // index of that token among them.
  int own = len;
  if (causal) {
    own = 0;
    for (int f = 0; f < vd.n_events; ++f) own += plan_events(p)[vd.first_event + f].len;
  }
  const int nk = own + 1;

  // row of the pools (page, kv-head, offset in the page) of task key `key`, -1 if out of the pool
  auto pool_row = [&](int row, int pi, int slot, int entry) -> long long {
    const int page = (row == e && pi == len / ps && ev.new_page >= 0) ? ev.new_page : entry;
    if (page < 0 || page >= p.n_pages) {
      pad_set_error(p.header, p.gen, PAD_ERR_DEVICE_BOUNDS, row, pi, page);
      return -1;
    }
    return ((long long)page * p.h_kv + kvh) * ps + slot;
  };
  auto row_of = [&](int key) -> long long {
    int row = e, t = key;
    if (causal) {
      if (key == own) {
        t = len;
      } else {
        row = vd.first_event;
        for (int lf = plan_events(p)[row].len; t >= lf; lf = plan_events(p)[row].len) {
          t -= lf;
          ++row;
        }
      }
    }
    const int pi = t / ps;
    return pool_row(row, pi, t - pi * ps, __ldcg(p.page_table + (size_t)row * p.max_pages + pi));
  };
  long long place = -1;                       // pool row of this lane's key (see above)
  if (kb0 < nkr && key0 < nk) place = causal ? row_of(key0) : pool_row(e, pi0, key0 - pi0 * ps, page0);
  // (ROPE: the plan carries positions; a separate instantiation keeps the plain one lean)
  const float* cs = ROPE ? p.rope_cs + (size_t)ev.pos * D : nullptr;
  const __nv_bfloat16* knew = static_cast<const __nv_bfloat16*>(p.k_new);
  const __nv_bfloat16* vnew = static_cast<const __nv_bfloat16*>(p.v_new);
  const size_t new_row = ((size_t)e * p.h_kv + kvh) * D;
  // this step's key waits for the grids ahead only when the append kernel wrote it
  const bool len_in_first = own < nkr && knew == nullptr && !p.keys_ready;
  const bool own_here = own < nkr && warp == own / 16;  // it is among this warp's first keys
  // the warp's 16 keys from r0 + kb0 on, places in lanes src .. src + 15 (rows past the last key
  // are zero-filled), but for this step's key where that comes from elsewhere or later
  auto stage_keys = [&](int r0, int src, bool skip_own) {
#pragma unroll
    for (int i = 0; i < 16 * CH / 32; ++i) {
      const int k = (lane + 32 * i) / CH, c = (lane + 32 * i) % CH;
      const long long pl = __shfl_sync(0xffffffffu, place, src + k);
      const bool in = pl >= 0;
      if (skip_own && r0 + kb0 + k == own) continue;
      const size_t off = (size_t)(in ? pl : 0) * D + c * 8;
      cp_async16(&sK[k][c * 8], kpool + off, in);
      if (W == D || (unsigned)(c * 8 - w0) < (unsigned)W) cp_async16(&sV[k][c * 8 - w0], vpool + off, in);
    }
  };
  // this step's key, one of the warp's 16 of a round: from k_new / v_new or from the pools
  auto stage_own = [&](int src) {
    const int k = own & 15;
    const long long pl = __shfl_sync(0xffffffffu, place, src + k);
    const bool in = pl >= 0;
    if (lane < CH) {
      const size_t off = knew != nullptr ? new_row + lane * 8 : (size_t)(in ? pl : 0) * D + lane * 8;
      if (ROPE && knew != nullptr)
        *reinterpret_cast<uint4*>(&sK[k][lane * 8]) = in ? rope_chunk8(knew + new_row, D, lane * 8, cs)
                                                         : make_uint4(0u, 0u, 0u, 0u);
      else
        cp_async16(&sK[k][lane * 8], (knew != nullptr ? knew : kpool) + off, in);
      if (W == D || (unsigned)(lane * 8 - w0) < (unsigned)W)
        cp_async16(&sV[k][lane * 8 - w0], (knew != nullptr ? vnew : vpool) + off, in);
    }
  };
  if (kb0 < min(nkr, nk)) stage_keys(0, 0, knew != nullptr || len_in_first);
  if (knew != nullptr && own_here) stage_own(0);
  cp_async_commit();
  if (ROPE) {                                 // rotated here (rows past G are zero)
    for (int i = tid; i < 16 * CH; i += NT) {
      const int g = i / CH, c = i - (i / CH) * CH;
      const __nv_bfloat16* qr = q + ((size_t)e * p.h_q + kvh * G + (g < G ? g : 0)) * D;
      *reinterpret_cast<uint4*>(&S.q[g][c * 8]) = g < G ? rope_chunk8(qr, D, c * 8, cs) : make_uint4(0u, 0u, 0u, 0u);
    }
  }
  if (knew != nullptr && w0 == 0) {
    // a2: this task's row of the new token into the pools (16-byte pieces of K, then V), by the
    // warp that holds its place
    if (own_here || (own >= nkr && warp == 0)) {
      const long long at = __shfl_sync(0xffffffffu, place, own & 15);
      const long long pl = own_here ? at : row_of(own);
      if (pl >= 0 && lane < 2 * CH) {
        const int c = lane % CH;
        const bool isv = lane >= CH;
        const uint4 v = (ROPE && !isv) ? rope_chunk8(knew + new_row, D, c * 8, cs)
                                       : __ldcg(reinterpret_cast<const uint4*>((isv ? vnew : knew) + new_row + c * 8));
        *reinterpret_cast<uint4*>(const_cast<__nv_bfloat16*>(isv ? vpool : kpool) + (size_t)pl * D + c * 8) = v;
      }
    }
    if (kvh == 0 && tid == 0 && ev.new_page >= 0 && ev.new_page < p.n_pages)
      p.page_table[(size_t)e * p.max_pages + len / ps] = ev.new_page;
  }
  // Where nothing the branch pass reads is written by a grid still running, the whole pass
  // runs before the wait and only the merge of the splits' partials follows it;
  // unless the plan says this CTA cannot start before the prefix grid completes anyway
  // (merge_first), where waiting first lets the partials load during the branch pass.
  const bool pre = OVER || ((knew != nullptr || p.keys_ready) && !p.merge_first);

  // ---------------- after the grids ahead (at least the append) completed
  if (!pre) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (len_in_first && own_here) stage_own(0);
  }
  cp_async_commit();                          // this round's keys

  // the splits' O rows (the task's columns of them) and (m, l) pairs of chunk [s0, s0 + nch): per
  // split, the task's G rows are one block of G * D floats, R * D floats after the previous split's
  // (the flat index is advanced by NT without a division).  Where the copies begin is found ahead
  // of the wait, and the pairs go by whole rows to warps: divisions behind the wait are time lost
  // (us per step: prefix 16384, 1 event 9.8, now 9.4; 8192, 8 events 8.8, now 8.5).
  const int gd4 = G * W4;
  const float* po_base = nullptr;
  const float2* ml_base = nullptr;
  int po_sl = 0, po_r = 0;
  auto find_chunk = [&]() {                   // what of it needs no partials: ahead of the wait
    po_sl = tid / gd4;
    po_r = tid - po_sl * gd4;
    po_base = p.part_o + part_row(vd, kvh, 0, R, rbase) * D + w0;
    ml_base = p.part_ml + part_row(vd, kvh, 0, R, rbase);
    asm volatile("" : "+r"(po_sl), "+r"(po_r), "+l"(po_base), "+l"(ml_base));  // (not sunk behind it)
  };
  if (!OVER) find_chunk();                    // (where registers are short: at the wait)
  auto stage_chunk = [&](int s0, int nch) {
    const size_t split_stride = (size_t)R * D;
    const int adv_sl = NT / gd4, adv_r = NT - adv_sl * gd4;
    const float* base = po_base + s0 * split_stride;
    for (int sl = po_sl, r = po_r; sl < nch;) {
      // piece r of the G x W block: row r / W4, float4 r % W4 of the task's columns
      const size_t src = W == D ? (size_t)r * 4 : (size_t)(r / W4) * D + (size_t)(r % W4) * 4;
      cp_async16(spo + (size_t)sl * G * W + (size_t)r * 4, base + sl * split_stride + src, true);
      sl += adv_sl;
      r += adv_r;
      if (r >= gd4) {
        r -= gd4;
        ++sl;
      }
    }
    const float2* mbase = ml_base + (size_t)s0 * R;
    for (int g = warp; g < G; g += NW)
      for (int k = lane; k < nch; k += 32) cp_async8(&sml[g * sch + k], mbase + (size_t)k * R + g);
  };
  bool ok = true;
  if (early && !pre) {
    if (ns > 0) stage_chunk(0, min(sch, ns));
    cp_async_commit();                        // the first chunk, waited for in a5
  }

  // ---------------- a4: the branch pass
  float o[OT][4];
#pragma unroll
  for (int i = 0; i < OT; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  float m_lo = kNegInf, m_hi = kNegInf;       // rows gq, gq + 8 (log2 units)
  float l_lo = 0.f, l_hi = 0.f;               // this lane's share of the row sums
  uint32_t qa[KS][4];
  // the rows of q and the warp's own first keys; from here to the fold no warp waits for another
  if (early && !pre)
    cp_async_wait<1>();                       // all but the first chunk's group
  else
    cp_async_wait<0>();
  sy.sync();
#pragma unroll
  for (int kk = 0; kk < KS; ++kk)
    ldsm_x4(qa[kk][0], qa[kk][1], qa[kk][2], qa[kk][3], &S.q[lane & 15][kk * 16 + (lane >> 4) * 8]);
  int src = 0;
  for (int r0 = 0; kb0 < nkr && r0 + kb0 < nk; r0 += nkr) {
    if (r0 > 0) {
      src ^= 16;
      if (src == 0) {
        const int key = r0 + key0;
        place = key < nk ? row_of(key) : -1;
      }
      __syncwarp();                           // the previous round's keys have been read
      stage_keys(r0, src, knew != nullptr);
      if (knew != nullptr && (own - r0) >> 4 == warp) stage_own(src);
      cp_async_commit();
      cp_async_wait<0>();
      __syncwarp();
    }
    const uint32_t seen = __ballot_sync(0xffffffffu, place >= 0) >> src;  // bit k: the warp's key k
    float s[2][4];
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
#pragma unroll
      for (int kk = 0; kk < KS; kk += 2) {
        uint32_t b0, b1, b2, b3;
        ldsm_x4(b0, b1, b2, b3, &sK[nt * 8 + (lane & 7)][kk * 16 + (lane >> 3) * 8]);
        mma_bf16(s[nt], qa[kk], b0, b1);
        mma_bf16(s[nt], qa[kk + 1], b2, b3);
      }
    }
    float mx_lo = kNegInf, mx_hi = kNegInf;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const bool in = (seen >> (nt * 8 + 2 * t4 + j)) & 1u;
        s[nt][j] = in ? s[nt][j] * p.scale_log2 : kNegInf;
        s[nt][2 + j] = in ? s[nt][2 + j] * p.scale_log2 : kNegInf;
        mx_lo = fmaxf(mx_lo, s[nt][j]);
        mx_hi = fmaxf(mx_hi, s[nt][2 + j]);
      }
    }
    mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 1));
    mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 2));
    mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 1));
    mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 2));
    float mn_lo = fmaxf(m_lo, mx_lo), mn_hi = fmaxf(m_hi, mx_hi);
    if (mn_lo == kNegInf) mn_lo = 0.f;  // only while every key so far failed its bounds check
    if (mn_hi == kNegInf) mn_hi = 0.f;
    const float al_lo = ex2(m_lo - mn_lo), al_hi = ex2(m_hi - mn_hi);
    m_lo = mn_lo;
    m_hi = mn_hi;
    float pr[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int j = 0; j < 4; ++j) pr[h][j] = ex2(s[h][j] - (j < 2 ? mn_lo : mn_hi));
    l_lo = l_lo * al_lo + (pr[0][0] + pr[0][1]) + (pr[1][0] + pr[1][1]);
    l_hi = l_hi * al_hi + (pr[0][2] + pr[0][3]) + (pr[1][2] + pr[1][3]);
    uint32_t a[4];
    a[0] = pack_bf16(pr[0][0], pr[0][1]);
    a[1] = pack_bf16(pr[0][2], pr[0][3]);
    a[2] = pack_bf16(pr[1][0], pr[1][1]);
    a[3] = pack_bf16(pr[1][2], pr[1][3]);
#pragma unroll
    for (int i = 0; i < OT; i += 2) {
      uint32_t b0, b1, b2, b3;
      ldsm_x4_t(b0, b1, b2, b3, &sV[lane & 15][(i + (lane >> 4)) * 8]);
      o[i][0] *= al_lo;
      o[i][1] *= al_lo;
      o[i][2] *= al_hi;
      o[i][3] *= al_hi;
      o[i + 1][0] *= al_lo;
      o[i + 1][1] *= al_lo;
      o[i + 1][2] *= al_hi;
      o[i + 1][3] *= al_hi;
      mma_bf16(o[i], a, b0, b1);
      mma_bf16(o[i + 1], a, b2, b3);
    }
  }
  l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1);
  l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
  l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1);
  l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);
  // this warp's state: (m, l) per row and its O rows (over its own keys)
  __syncwarp();
  float* wo = reinterpret_cast<float*>(&sK[0][0]);
  if (t4 == 0) {
    S.wm[warp][gq] = m_lo;
    S.wl[warp][gq] = l_lo;
    S.wm[warp][gq + 8] = m_hi;
    S.wl[warp][gq + 8] = l_hi;
  }
  if (kb0 < nkr && gq < G) {
    float* dst = wo + gq * LDO;
#pragma unroll
    for (int i = 0; i < OT; ++i) *reinterpret_cast<float2*>(dst + i * 8 + 2 * t4) = make_float2(o[i][0], o[i][1]);
  }
  if (kb0 < nkr && gq + 8 < G) {
    float* dst = wo + (gq + 8) * LDO;
#pragma unroll
    for (int i = 0; i < OT; ++i) *reinterpret_cast<float2*>(dst + i * 8 + 2 * t4) = make_float2(o[i][2], o[i][3]);
  }
  sy.sync();

  // ---------------- a5: the warp states, then the prefix splits in chunks of `sch`.  A thread
  // keeps its float4s of the output rows, with their rows' M and L, in registers throughout and
  // finds the weights itself: a few exponentials more, but no pass over the rows by single warps
  // with barriers on both sides.
  constexpr int kOut = (16 * W4 + NT - 1) / NT;
  float4 acc[kOut];
  float M[kOut], L[kOut];
  const int nact = (min(nkr, nk) + 15) / 16;  // warps that had keys
#pragma unroll
  for (int it = 0; it < kOut; ++it) {
    const int i = tid + it * NT;
    acc[it] = make_float4(0.f, 0.f, 0.f, 0.f);
    M[it] = L[it] = 0.f;
    if (i < G * W4) {
      const int g = i / W4, d4 = i - g * W4;
      float mx = kNegInf;
      for (int w = 0; w < nact; ++w) mx = fmaxf(mx, S.wm[w][g]);
      if (mx == kNegInf) mx = 0.f;            // no key of the branch passed its bounds check
      for (int w = 0; w < nact; ++w) {
        const float c = ex2(S.wm[w][g] - mx);
        const float4 v = reinterpret_cast<const float4*>(kv_raw + w * kWarpKv<D, W>)[g * (LDO / 4) + d4];
        L[it] = fmaf(S.wl[w][g], c, L[it]);
        acc[it].x = fmaf(c, v.x, acc[it].x);
        acc[it].y = fmaf(c, v.y, acc[it].y);
        acc[it].z = fmaf(c, v.z, acc[it].z);
        acc[it].w = fmaf(c, v.w, acc[it].w);
      }
      M[it] = mx;
    }
  }

  if (early && pre) {
    if (OVER) find_chunk();
    // ---------------- after the grids ahead (the prefix pass) completed
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (OVER) sy.sync();                      // the warps' O rows have been read
    if (ns > 0) stage_chunk(0, min(sch, ns));
    cp_async_commit();
  }
  if (!early && ns > 0) {
    ok = partials_ready();
    if (ok) stage_chunk(0, min(sch, ns));
    cp_async_commit();
  }
  for (int s0 = 0; ok && s0 < ns; s0 += sch) {
    const int nch = min(sch, ns - s0);
    if (s0 > 0) {
      sy.sync();                              // the previous chunk's rows are consumed
      stage_chunk(s0, nch);
    }
    cp_async_commit();
    cp_async_wait<0>();
    sy.sync();
#pragma unroll
    for (int it = 0; it < kOut; ++it) {
      const int i = tid + it * NT;
      if (i < G * W4) {
        const int g = i / W4;
        const float2* ml = sml + g * sch;
        float mn = M[it];
        for (int sl = 0; sl < nch; ++sl) mn = fmaxf(mn, ml[sl].x);
        const float al = ex2(M[it] - mn);
        M[it] = mn;
        L[it] *= al;
        float4 a = acc[it];
        a.x *= al;
        a.y *= al;
        a.z *= al;
        a.w *= al;
        const float4* po = reinterpret_cast<const float4*>(spo) + i;
#pragma unroll 4
        for (int sl = 0; sl < nch; ++sl) {
          const float2 st = ml[sl];
          const float c = ex2(st.x - mn);
          const float4 v = po[sl * G * W4];
          L[it] = fmaf(st.y, c, L[it]);
          a.x = fmaf(c, v.x, a.x);
          a.y = fmaf(c, v.y, a.y);
          a.z = fmaf(c, v.z, a.z);
          a.w = fmaf(c, v.w, a.w);
        }
        acc[it] = a;
      }
    }
  }
  cp_async_wait<0>();
  if (!ok) return;

#pragma unroll
  for (int it = 0; it < kOut; ++it) {
    const int i = tid + it * NT;
    if (i >= G * W4) break;
    const int g = i / W4, d4 = i - g * W4;
    const float inv = 1.0f / L[it];
    float4 v = acc[it];
    v.x *= inv;
    v.y *= inv;
    v.z *= inv;
    v.w *= inv;
    const size_t oi = ((size_t)e * p.h_q + kvh * G + g) * D + w0 + 4 * d4;
    if (p.out_bf16)
      *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(out) + oi) =
          make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
    else
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + oi) = v;
    if (lse != nullptr && d4 == 0 && w0 == 0)
      lse[(size_t)e * p.h_q + kvh * G + g] = (M[it] + log2f(L[it])) * 0.69314718055994531f;
  }
}
#endif  // __CUDACC__

}  // namespace bm
}  // namespace pad

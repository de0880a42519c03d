// Grounding readout of the planning tokens (Sec. 3.3, and the paper's note on inference by
// similarity matching): each generated event token G^i is matched against the audio-visual
// prefix tokens after both went through the model's projection; the dot products of one
// time segment's tokens are summed into a segment score, and the segments whose score
// reaches a fraction of the event's best form its grounded interval.  Attention-guided
// aggregation (strategy (3) of Sec. 3.3) then pools the grounded tokens' hidden states with
// the last query token's attention weights and adds the result to the event embedding.
//
// The segment score is linear in the token features, so sum_t <g, f_t> = <g, sum_t f_t>:
// the prefix is read once, pooling each segment's projected features (ground_pool_kernel,
// HBM-bound; a thread has up to eight rows' loads in flight, four at d <= 256, since a latency-bound stream
// of single loads ran at a twentieth of the bandwidth), and scoring every event against the pooled rows is a small contraction over
// L2-resident data (ground_score_kernel).  The aggregation reads the hidden states once,
// pooling them per segment with the attention weights, and sums each event's segments
// (attn_seg_pool_kernel, attn_event_kernel).
#include <cuda_bf16.h>
#include <algorithm>
#include <cstdint>

#include "pad_internal.h"

// The kernels here run for 2 to 25 us each, so the gaps between them count: all are launched
// with programmatic dependent launch.  Each waits for the grid ahead before it reads or writes
// anything that grid may touch, and releases its dependents only after that wait, so that a
// kernel that has started knows every grid but the one right ahead of it to have completed.
// What the grid ahead may still write while a kernel here runs is read past L1 (not through
// the read-only path, which assumes that nobody writes).
namespace pad {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
constexpr int kMaxSegments = 1024;

// A kernel's parameters are cold in the constant cache at every launch, and each step of a
// binary search over a thousand of them is a dependent miss (the searches of the pooling
// kernels cost 3 us).  So the host also passes, for each 64th of a grid, the segment its first
// block falls into; the search then runs between two of these.
constexpr int kHints = 64;
struct Hints {
  uint16_t seg[kHints + 1];
  // range [lo, hi] of the segment of block b of nb
  __device__ void range(unsigned b, unsigned nb, int& lo, int& hi) const {
    const int g = (int)((unsigned long long)b * kHints / nb);
    lo = seg[g];
    hi = seg[g + 1];
  }
};

struct Offsets {
  int32_t n;                       // segments
  Hints hint;                      // by chunk of the pooling kernel
  int32_t off[kMaxSegments + 1];   // token ranges [off[s], off[s + 1])
};

// 16-byte streaming load, issued where it stands (asm volatile keeps a group of them ahead
// of their first use, so that they are in flight together).
__device__ __forceinline__ uint4 ld_stream(const void* p) {
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// Four such loads in one statement: all four are issued before any of them is used.
__device__ __forceinline__ void ld_stream4(uint4 (&v)[4], const void* p0, const void* p1, const void* p2,
                                           const void* p3) {
  asm volatile(
      "ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%16];\n"
      "ld.global.L1::no_allocate.v4.u32 {%4, %5, %6, %7}, [%17];\n"
      "ld.global.L1::no_allocate.v4.u32 {%8, %9, %10, %11}, [%18];\n"
      "ld.global.L1::no_allocate.v4.u32 {%12, %13, %14, %15}, [%19];"
      : "=r"(v[0].x), "=r"(v[0].y), "=r"(v[0].z), "=r"(v[0].w), "=r"(v[1].x), "=r"(v[1].y), "=r"(v[1].z),
        "=r"(v[1].w), "=r"(v[2].x), "=r"(v[2].y), "=r"(v[2].z), "=r"(v[2].w), "=r"(v[3].x), "=r"(v[3].y),
        "=r"(v[3].z), "=r"(v[3].w)
      : "l"(p0), "l"(p1), "l"(p2), "l"(p3));
}

// A row that a grid ahead wrote: through L1 where the kernel is launched in plain stream order only.
template <bool L1>
__device__ __forceinline__ float4 ld_row(const float4* p) {
  return L1 ? __ldg(p) : __ldcg(p);
}

// One bf16 element past L1.  (The header's __ldcg of this type may be moved ahead of the wait.)
__device__ __forceinline__ float ld_bf16(const __nv_bfloat16* p) {
  return __bfloat162float(__ushort_as_bfloat16(__ldcg(reinterpret_cast<const unsigned short*>(p))));
}

__device__ __forceinline__ void unpack8(const uint4 v, float* f) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 t = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[j]));
    f[2 * j] = t.x;
    f[2 * j + 1] = t.y;
  }
}

// Zeroes the sums ahead of the pooling kernel.
__global__ void __launch_bounds__(kThreads) ground_zero_kernel(float4* __restrict__ out, int n4) {
  grid_wait();
  grid_release();
  for (int i = blockIdx.x * kThreads + threadIdx.x; i < n4; i += gridDim.x * kThreads)
    out[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// One CTA per chunk of pool_chunk tokens, whatever segments they belong to: the 256 threads
// cover the row's 16-byte chunks (CH = d / 8 of them) and RP = 256 / CH rows at a
// time.  For each segment that overlaps the chunk (if they are few, see kFewSegments) a thread adds up
// its rows (up to four for d <= 256, 32 beyond), and the RP partial sums are added in shared memory and
// then into seg_sum (zeroed by the kernel ahead) with atomics, so the chunks of a segment add up in
// no fixed order.  It starts while that kernel runs (which has seen everything before it complete)
// and waits for it before the first atomic.  Chunks instead of slices of each segment keep the CTAs equal: a grid of segments x
// (longest segment / slice) is mostly CTAs with nothing to do.
// Tokens of a chunk: 16 KB of them, so that the grid is several CTAs per SM (four or two times as
// much: 6 or 0.9 us more per readout at d = 256), but at least 32, since every chunk adds a
// row of d floats per segment to the sums.
__host__ __device__ constexpr int pool_chunk(int RP) { return 4 * RP > 32 ? 4 * RP : 32; }
// A segment of a chunk costs a round of loads and two barriers, one after the other.  A chunk of more
// than kFewSegments goes the other way: each row group takes rows that follow one another and adds
// up on its own, straight into the sums wherever a segment ends: more atomics, but no barrier.  1024
// tokens in 1024 segments, us per call by segments and by rows: d = 8 2842, 11.6; d = 64 127, 11.6; d =
// 256 27.5, 11.6; d = 2048 36.0, 14.5; 32768 tokens in 128 segments at d = 8 (five per chunk) 27.9,
// 11.0.  (Limits of 2 and 8 are within 15 % of this one wherever a chunk is not just short of 8.)
constexpr int kFewSegments = 4;
__global__ void __launch_bounds__(kThreads) ground_pool_kernel(const __grid_constant__ Offsets so,
                                                               const __nv_bfloat16* __restrict__ f, int d,
                                                               float* __restrict__ seg_sum) {
  extern __shared__ __align__(16) float red[];  // [RP][d]
  const int CH = d / 8, RP = kThreads / CH;
  const int c = threadIdx.x % CH, rg = threadIdx.x / CH;
  const int chunk = pool_chunk(RP);
  const int t_lo = so.off[0] + (int)blockIdx.x * chunk, t_hi = t_lo + min(so.off[so.n] - t_lo, chunk);
  int s, sh;  // the segment of token t_lo: the last s with off[s] <= t_lo
  so.hint.range(blockIdx.x, gridDim.x, s, sh);
  while (s < sh) {
    const int mid = (s + sh + 1) >> 1;
    if (so.off[mid] <= t_lo)
      s = mid;
    else
      sh = mid - 1;
  }
  if (s + kFewSegments < so.n && so.off[s + kFewSegments] < t_hi) {
    int* off = reinterpret_cast<int*>(red);    // off[s ..]: at most 1025 of them (red has 129 * 8 floats or more)
    const int ns = so.n - s;
    for (int i = threadIdx.x; i <= ns; i += kThreads) off[i] = so.off[s + i];
    grid_wait();
    grid_release();
    __syncthreads();
    const int rows = (chunk + RP - 1) / RP;    // of a row group
    int t = t_lo + rg * rows;
    const int te = min(t_hi, t + rows);
    if (rg >= RP || t >= te) return;
    auto find = [&](int lo, int tok) {         // the segment of tok: the last u >= lo with off[u] <= tok
      int hi = ns - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= tok)
          lo = mid;
        else
          hi = mid - 1;
      }
      return lo;
    };
    int u = find(0, t);
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    auto flush = [&] {
      float4* dst = reinterpret_cast<float4*>(seg_sum + (size_t)(s + u) * d + c * 8);
      atomicAdd(dst, make_float4(acc[0], acc[1], acc[2], acc[3]));
      atomicAdd(dst + 1, make_float4(acc[4], acc[5], acc[6], acc[7]));
    };
    for (; t < te; t += 4) {
      uint4 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[k] = make_uint4(0u, 0u, 0u, 0u);
        if (t + k < te) v[k] = ld_stream(reinterpret_cast<const uint4*>(f + (size_t)(t + k) * d) + c);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (t + k >= te) break;
        if (t + k >= off[u + 1]) {
          flush();
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[j] = 0.f;
          ++u;
          if (t + k >= off[u + 1]) u = find(u + 1, t + k);  // (a run of empty segments)
        }
        float x[8];
        unpack8(v[k], x);
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] += x[j];
      }
    }
    flush();
    return;
  }
  bool waited = false;
  for (int t0 = t_lo; t0 < t_hi; ++s) {
    const int t1 = min(t_hi, so.off[s + 1]);
    if (t1 <= t0) continue;  // an empty segment
    const int n = t1 - t0;
    const __nv_bfloat16* row0 = f + (size_t)t0 * d;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (rg < RP) {
      for (int t = rg; t < n; t += 8 * RP) {
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          v[u] = make_uint4(0u, 0u, 0u, 0u);
          if (t + u * RP < n) v[u] = ld_stream(reinterpret_cast<const uint4*>(row0 + (size_t)(t + u * RP) * d) + c);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          float x[8];
          unpack8(v[u], x);
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[j] += x[j];
        }
      }
      float4* dst = reinterpret_cast<float4*>(red + rg * d + c * 8);
      dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    }
    if (!waited) {
      grid_wait();
      grid_release();
      waited = true;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < d / 4; i += kThreads) {
      float4 tot = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int r = 0; r < RP; ++r) {
        const float4 v = *reinterpret_cast<const float4*>(red + r * d + 4 * i);
        tot.x += v.x;
        tot.y += v.y;
        tot.z += v.z;
        tot.w += v.w;
      }
      atomicAdd(reinterpret_cast<float4*>(seg_sum + (size_t)s * d) + i, tot);
    }
    __syncthreads();
    t0 = t1;
  }
  if (!waited) grid_wait();
}

// One CTA per event: scores against every pooled segment row, the best score, the salient
// set (score >= fraction * best when best > 0, else the first best segment alone) and the
// first and last salient segments.
// A warp takes ROWS segments at a time.  32 warps of four rows (a hundred segments are one round of
// loads) are best while every CTA finds room, two per SM, and where an event's own work is long.
// More events than that over few segments take eight warps of eight rows, eight CTAs per SM, and where
// the rows of all events are more than 64 MB they come through L1, which the CTAs of an SM share (the
// kernel is then launched in plain stream order).  us per call, 32 x 4, 8 x 8, 8 x 8 through L1: 1024 events, 8
// segments, d = 64: 17.5, 6.1, -; 310, 128, 256: 10.5, 8.3, 10.4; 310, 1024, 256: 41.1, 48.2, 38.2; 1024,
// 128, 256: 24.1, 13.9, 14.5; 620, 1024, 1024: 147.8, 168, 186.
template <int WARPS, int ROWS, bool L1>
__global__ void __launch_bounds__(32 * WARPS) ground_score_kernel(const __nv_bfloat16* __restrict__ g, int S, int d,
                                                                const float* __restrict__ seg_sum, float frac,
                                                                float* __restrict__ scores,
                                                                uint8_t* __restrict__ salient,
                                                                int32_t* __restrict__ interval) {
  constexpr int kThr = 32 * WARPS;
  extern __shared__ float gs[];  // [d] the event's projected token, then [S] scores
  float* sc = gs + d;
  __shared__ float wbest[WARPS];
  __shared__ int wlo[WARPS], whi[WARPS], warg[WARPS];
  const int i = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  grid_wait();
  grid_release();
  for (int c = threadIdx.x; c < d; c += kThr) gs[c] = L1 ? __bfloat162float(g[(size_t)i * d + c]) : ld_bf16(g + (size_t)i * d + c);
  __syncthreads();
  // a warp per segment row (lanes over its float4 columns), ROWS rows in flight per warp
  float best = -__builtin_huge_valf();
  const int d4 = d / 4;
  for (int s0 = warp * ROWS; s0 < S; s0 += ROWS * WARPS) {
    float part[ROWS] = {};
#pragma unroll 8 / ROWS
    for (int c = lane; c < d4; c += 32) {
      float4 v[ROWS];
#pragma unroll
      for (int u = 0; u < ROWS; ++u)
        v[u] = s0 + u < S ? ld_row<L1>(reinterpret_cast<const float4*>(seg_sum + (size_t)(s0 + u) * d) + c)
                          : make_float4(0.f, 0.f, 0.f, 0.f);
      const float g0 = gs[4 * c], g1 = gs[4 * c + 1], g2 = gs[4 * c + 2], g3 = gs[4 * c + 3];
#pragma unroll
      for (int u = 0; u < ROWS; ++u) part[u] += (g0 * v[u].x + g1 * v[u].y) + (g2 * v[u].z + g3 * v[u].w);
    }
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
      float v = part[u];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (s0 + u < S) {
        if (lane == 0) {
          sc[s0 + u] = v;
          scores[(size_t)i * S + s0 + u] = v;
        }
        best = fmaxf(best, v);
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
  if (lane == 0) wbest[warp] = best;
  __syncthreads();
  best = wbest[0];
  for (int w = 1; w < WARPS; ++w) best = fmaxf(best, wbest[w]);
  // the first best segment (used alone when no score is positive)
  int arg = S;
  for (int s = threadIdx.x; s < S; s += kThr)
    if (sc[s] == best) arg = min(arg, s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) arg = min(arg, __shfl_xor_sync(0xffffffffu, arg, o));
  if (lane == 0) warg[warp] = arg;
  __syncthreads();
  arg = warg[0];
  for (int w = 1; w < WARPS; ++w) arg = min(arg, warg[w]);
  const float cut = frac * best;
  int lo = S, hi = -1;
  for (int s = threadIdx.x; s < S; s += kThr) {
    const bool on = best > 0.f ? sc[s] >= cut : s == arg;
    salient[(size_t)i * S + s] = on ? 1 : 0;
    if (on) {
      lo = min(lo, s);
      hi = max(hi, s);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (lane == 0) {
    wlo[warp] = lo;
    whi[warp] = hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < WARPS; ++w) {
      lo = min(lo, wlo[w]);
      hi = max(hi, whi[w]);
    }
    lo = min(lo, wlo[0]);
    hi = max(hi, whi[0]);
    interval[2 * i] = lo;
    interval[2 * i + 1] = hi;
  }
}

// Attention-guided aggregation.  The weights attn[t] belong to the tokens, not to the
// events, so an event's weighted sum over its grounded segments lo..hi is the sum of the
// segments' own weighted sums: the hidden states are read once (attn_seg_pool_kernel,
// HBM-bound), and every event then adds up its segments' rows, which stay in L2
// (attn_event_kernel).  For balance the token axis is cut into pieces of at most
// kAggPiece tokens, each inside one segment (segment s owns pieces pbeg[s] .. pbeg[s+1]-1),
// and the pooled rows are per piece: W[p] = sum_{t in p} attn[t] x[t], A[p] = sum_{t in p}
// attn[t].  Every element is written once and summed in a fixed order, so the results are
// the same from run to run.
constexpr int kAggCols = 256;
constexpr int kAggPiece = 256;
constexpr int kAggGroups = kThreads / 32;

struct Pieces {
  int32_t n;                          // segments
  Hints hint;                         // by piece
  int32_t off[kMaxSegments + 1];      // token ranges of the segments
  int32_t pbeg[kMaxSegments + 1];     // first piece of each segment; pbeg[n] = pieces
};

// attn_seg_pool_kernel: grid (piece, slice of kAggCols columns).  Eight row groups of 32
// threads; a thread owns one 16-byte piece (8 columns) of every eighth row and keeps eight
// rows' loads in flight; the row groups' sums are added in shared memory, in order.  HBM-bound:
// about 25 us for 134 MB with five CTAs per SM (four: 1.5 us more).  Slices of 128 or 512 columns,
// or a last batch of predicated loads (more registers, so fewer CTAs), were 4 to 10 us slower.
__global__ void __launch_bounds__(kThreads, 5) attn_seg_pool_kernel(const __grid_constant__ Pieces pm,
                                                                 const __nv_bfloat16* __restrict__ x, int d,
                                                                 const float* __restrict__ attn,
                                                                 float* __restrict__ wsum, float* __restrict__ asum) {
  __shared__ float red[kAggGroups][kAggCols];
  __shared__ float ared[kAggGroups];
  grid_wait();
  grid_release();
  const int pc = blockIdx.x;
  int sl, sh;  // the segment owning piece pc: the last s with pbeg[s] <= pc
  pm.hint.range(blockIdx.x, gridDim.x, sl, sh);
  while (sl < sh) {
    const int mid = (sl + sh + 1) >> 1;
    if (pm.pbeg[mid] <= pc)
      sl = mid;
    else
      sh = mid - 1;
  }
  const int lo = pm.off[sl] + (pc - pm.pbeg[sl]) * kAggPiece, hi = min(pm.off[sl + 1], lo + kAggPiece);
  const int lane = threadIdx.x & 31, rg = threadIdx.x >> 5;
  const int c = blockIdx.y * (kAggCols / 8) + lane;  // 16-byte piece of the row
  const bool cin = c < d / 8;
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  float wacc = 0.f;
  const uint4* xc = reinterpret_cast<const uint4*>(x) + (cin ? c : 0);
  const size_t rs = (size_t)d / 8;  // row stride in pieces
  int t = lo + rg;
  for (; t + 7 * kAggGroups < hi; t += 8 * kAggGroups) {
    uint4 v[2][4];
    ld_stream4(v[0], xc + (size_t)t * rs, xc + (size_t)(t + kAggGroups) * rs, xc + (size_t)(t + 2 * kAggGroups) * rs,
               xc + (size_t)(t + 3 * kAggGroups) * rs);
    ld_stream4(v[1], xc + (size_t)(t + 4 * kAggGroups) * rs, xc + (size_t)(t + 5 * kAggGroups) * rs,
               xc + (size_t)(t + 6 * kAggGroups) * rs, xc + (size_t)(t + 7 * kAggGroups) * rs);
    float w[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) w[u] = __ldcg(attn + t + u * kAggGroups);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      float f[8];
      unpack8(v[u >> 2][u & 3], f);
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[j] = fmaf(w[u], f[j], acc[j]);
      wacc += w[u];
    }
  }
  for (; t < hi; t += kAggGroups) {
    const float w0 = __ldcg(attn + t);
    float f[8];
    unpack8(ld_stream(xc + (size_t)t * rs), f);
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = fmaf(w0, f[j], acc[j]);
    wacc += w0;
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) red[rg][lane * 8 + j] = acc[j];
  if (lane == 0) ared[rg] = wacc;  // (every lane of the group summed the same weights)
  __syncthreads();
  const int col = blockIdx.y * kAggCols + threadIdx.x;
  if (col < d) {
    float tot = 0.f;
#pragma unroll
    for (int r = 0; r < kAggGroups; ++r) tot += red[r][threadIdx.x];
    wsum[(size_t)pc * d + col] = tot;
  }
  if (blockIdx.y == 0 && threadIdx.x == 0) {
    float a = 0.f;
    for (int r = 0; r < kAggGroups; ++r) a += ared[r];
    asum[pc] = a;
  }
}

// attn_event_kernel: grid (event, slice of kAggCols columns).  The pieces of the event's
// interval (lo, hi), clamped to the segments, are spread over 16 warps (warp w takes every
// 16th piece from the first, four in flight; eight or 32 warps were 1.4 us slower per readout); a lane
// adds 8 columns; the warps' sums are added in shared memory, in order, and out = g_emb + sum W / sum A
// (g_emb alone when sum A is 0).  A grid of more than twelve CTAs per SM has eight warps with one piece at a
// time, through L1, which the events share (in plain stream order, then): 1024 events, 32768 tokens,
// d = 2048, 128 segments 65.4 us per call with 16 warps, 45.4 so; 400 events 38.2, 33.0; 200 (ten per
// SM) 30.4, 31.0.
template <int WARPS, bool L1>
__global__ void __launch_bounds__(32 * WARPS) attn_event_kernel(const __grid_constant__ Pieces pm, int d,
                                                              const int32_t* __restrict__ interval,
                                                              const float* wsum, const float* asum,
                                                              const __nv_bfloat16* __restrict__ g_emb,
                                                              float* __restrict__ out) {
  __shared__ float red[WARPS][kAggCols];
  __shared__ float ared[WARPS];
  const int i = blockIdx.x, S = pm.n;
  const int s_lo = min(max(__ldcg(interval + 2 * i), 0), S - 1);
  const int s_hi = min(max(__ldcg(interval + 2 * i + 1), s_lo), S - 1);
  const int p0 = pm.pbeg[s_lo], p1 = pm.pbeg[s_hi + 1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c8 = blockIdx.y * kAggCols + lane * 8;  // first of this lane's 8 columns
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  float a = 0.f;
  grid_wait();  // (the interval was written before the pooling kernel started)
  grid_release();
  if (L1 && c8 < d) {
    for (int pc = p0 + w; pc < p1; pc += WARPS) {
      const float4* src = reinterpret_cast<const float4*>(wsum + (size_t)pc * d + c8);
      const float4 u0 = __ldg(src), u1 = __ldg(src + 1);
      acc[0] += u0.x;
      acc[1] += u0.y;
      acc[2] += u0.z;
      acc[3] += u0.w;
      acc[4] += u1.x;
      acc[5] += u1.y;
      acc[6] += u1.z;
      acc[7] += u1.w;
      a += __ldg(asum + pc);
    }
  } else if (c8 < d) {
    // four pieces' loads in flight
    for (int pc = p0 + w; pc < p1; pc += 4 * WARPS) {
      float4 u0[4], u1[4];
      float av[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int q = pc + k * WARPS;
        u0[k] = u1[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        av[k] = 0.f;
        if (q < p1) {
          const float4* src = reinterpret_cast<const float4*>(wsum + (size_t)q * d + c8);
          u0[k] = __ldcg(src);
          u1[k] = __ldcg(src + 1);
          av[k] = __ldcg(asum + q);
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        acc[0] += u0[k].x;
        acc[1] += u0[k].y;
        acc[2] += u0[k].z;
        acc[3] += u0[k].w;
        acc[4] += u1[k].x;
        acc[5] += u1[k].y;
        acc[6] += u1[k].z;
        acc[7] += u1[k].w;
        a += av[k];
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) red[w][lane * 8 + j] = acc[j];
  if (lane == 0) ared[w] = a;
  __syncthreads();
  const int col = blockIdx.y * kAggCols + threadIdx.x;
  if (threadIdx.x < kAggCols && col < d) {
    float num = 0.f, den = 0.f;
#pragma unroll
    for (int r = 0; r < WARPS; ++r) {
      num += red[r][threadIdx.x];
      den += ared[r];
    }
    const float base = ld_bf16(g_emb + (size_t)i * d + col);
    out[(size_t)i * d + col] = den > 0.f ? base + num / den : base;
  }
}

// SM count of the current device (it does not change).
int sm_count() {
  static int n[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
  if (n[dev] == 0 && cudaDeviceGetAttribute(&n[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) n[dev] = 152;
  return n[dev];
}

// A launch that may start while the grid ahead of it runs (early), or in plain stream order.
template <class... KArgs, class... Args>
cudaError_t launch_early(bool early, void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                         Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <class... KArgs, class... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t s, Args... args) {
  return launch_early(true, kernel, grid, threads, smem, s, args...);
}

// hint.seg[g]: the last segment whose `first` entry is at most that of the first block of the
// g-th 64th of `blocks` (Hints::range's split); the entry after the last is the last segment.
template <class Of>
void fill_hints(Hints& h, const int32_t* first, int n, int64_t blocks, Of value_of) {
  int s = 0;
  for (int g = 0; g < kHints; ++g) {
    const int64_t b = (blocks * g + kHints - 1) / kHints;  // the first block b with b * kHints / blocks >= g
    if (b >= blocks) {
      h.seg[g] = (uint16_t)(n - 1);
      continue;
    }
    const int64_t v = value_of(b);
    while (s + 1 < n && first[s + 1] <= v) ++s;
    h.seg[g] = (uint16_t)s;
  }
  h.seg[kHints] = (uint16_t)(n - 1);
}

bool fill_offsets(Offsets& so, const int32_t* offsets, int32_t n_segments, int64_t n_tokens) {
  if (n_segments < 1 || n_segments > kMaxSegments || !offsets) return false;
  so.n = n_segments;
  for (int s = 0; s <= n_segments; ++s) {
    if (offsets[s] < 0 || offsets[s] > n_tokens || (s > 0 && offsets[s] < offsets[s - 1])) return false;
    so.off[s] = offsets[s];
  }
  return true;
}

}  // namespace

cudaError_t launch_ground_pool(const void* f_proj, int64_t n_tokens, int32_t d, const int32_t* offsets,
                               int32_t n_segments, float* seg_sum, cudaStream_t s) {
  Offsets so;
  if (!fill_offsets(so, offsets, n_segments, n_tokens)) return cudaErrorInvalidValue;
  const int CH = d / 8, RP = kThreads / CH;
  // (a segment of more than 65535 x 16 RP tokens has always been refused)
  int longest = 0;
  for (int i = 0; i < n_segments; ++i) longest = std::max(longest, so.off[i + 1] - so.off[i]);
  if (longest > (int64_t)65535 * 16 * RP) return cudaErrorInvalidValue;
  const int n4 = n_segments * (d / 4);
  cudaError_t e = launch_pdl(ground_zero_kernel, dim3(std::min(64, (n4 + kThreads - 1) / kThreads)), kThreads, 0, s,
                             reinterpret_cast<float4*>(seg_sum), n4);
  if (e != cudaSuccess) return e;
  const int64_t tokens = (int64_t)so.off[n_segments] - so.off[0], chunk = pool_chunk(RP);
  if (tokens == 0) return cudaSuccess;
  const int64_t blocks = (tokens + chunk - 1) / chunk;
  fill_hints(so.hint, so.off, n_segments, blocks, [&](int64_t b) { return so.off[0] + b * chunk; });
  return launch_pdl(ground_pool_kernel, dim3((unsigned)blocks), kThreads,
                    (size_t)RP * d * sizeof(float), s, so, static_cast<const __nv_bfloat16*>(f_proj), d, seg_sum);
}

cudaError_t launch_ground_score(const void* g_proj, int32_t n_events, const float* seg_sum, int32_t n_segments,
                                int32_t d, float frac, float* scores, uint8_t* salient, int32_t* interval,
                                cudaStream_t s) {
  if (n_events == 0) return cudaSuccess;
  const size_t smem = (size_t)(d + n_segments) * sizeof(float);
  const bool many = n_events > 2 * sm_count() && n_segments * d < (1 << 19);
  const bool l1 = many && (int64_t)n_events * n_segments * d > (16 << 20);  // 64 MB of rows
  auto* kernel = l1 ? ground_score_kernel<8, 8, true> : many ? ground_score_kernel<8, 8, false> : ground_score_kernel<32, 4, false>;
  return launch_early(!l1, kernel, dim3(n_events), many ? 256 : 1024, smem, s, static_cast<const __nv_bfloat16*>(g_proj),
                      n_segments, d, seg_sum, frac, scores, salient, interval);
}

size_t attn_aggregate_ws_floats(int64_t n_tokens, int32_t n_segments, int32_t d) {
  return ((size_t)n_segments + (size_t)(n_tokens + kAggPiece - 1) / kAggPiece) * ((size_t)d + 1);
}

cudaError_t launch_attn_aggregate(const void* x, int64_t n_tokens, int32_t d, const float* attn,
                                  const int32_t* offsets, int32_t n_segments, const int32_t* interval,
                                  int32_t n_events, const void* g_emb, float* seg_ws, float* out, cudaStream_t s) {
  Offsets so;
  if (!fill_offsets(so, offsets, n_segments, n_tokens)) return cudaErrorInvalidValue;
  if (n_events == 0) return cudaSuccess;
  Pieces pm;
  pm.n = n_segments;
  pm.pbeg[0] = 0;
  for (int i = 0; i < n_segments; ++i) {
    pm.off[i] = so.off[i];
    pm.pbeg[i + 1] = pm.pbeg[i] + (so.off[i + 1] - so.off[i] + kAggPiece - 1) / kAggPiece;
  }
  pm.off[n_segments] = so.off[n_segments];
  const int pieces = pm.pbeg[n_segments];
  const int slices = (d + kAggCols - 1) / kAggCols;
  if (slices > 65535) return cudaErrorInvalidValue;
  // (pieces <= n_segments + n_tokens / kAggPiece: within attn_aggregate_ws_floats)
  float* wsum = seg_ws;
  float* asum = seg_ws + (size_t)std::max(pieces, 1) * d;
  if (pieces > 0) {
    fill_hints(pm.hint, pm.pbeg, n_segments, pieces, [](int64_t b) { return b; });
    cudaError_t e = launch_pdl(attn_seg_pool_kernel, dim3(pieces, slices), kThreads, 0, s, pm,
                               static_cast<const __nv_bfloat16*>(x), d, attn, wsum, asum);
    if (e != cudaSuccess) return e;
  }
  const bool many = (int64_t)n_events * slices > 12 * sm_count();
  return launch_early(!many, many ? attn_event_kernel<8, true> : attn_event_kernel<16, false>, dim3(n_events, slices),
                      many ? 256 : 512, 0, s, pm, d, interval, wsum, asum, static_cast<const __nv_bfloat16*>(g_emb), out);
}

}  // namespace pad

// Ranking and keep/drop sets, Algorithm 1 steps 1 and 3.
//
// A sort problem is (request, KV head) in the shared mode, (request, layer, KV
// head) in the layer-specific mode.  Scores become 32-bit keys whose ascending
// order is descending score; rank[v] = position of token v in the order
// "descending score, lower index first on exact ties".
//
// prunekv_select returns the ranks.  chunk_sort_kernel + chunk_rank_kernel:
// sorted 1024-key chunks, then each element's rank by counting (binary search)
// in every other chunk of its problem; many CTAs per problem, ranks exact and
// schedule-independent.
//
// The fused pass needs no ranks, only where the order is cut: threshold_kernel
// finds, per problem, the element at each cut (position B_l - 1 of every
// layer, Nq - 1), and a token is kept or dropped by comparing it with them.
//
// compact_kernel: one CTA per (request, layer <= h, KV head) with B_l > 0.
// Warps take runs of consecutive tokens; ballots and the block's counts per
// warp place keep = {rank < B_l} and drop = {B_l <= rank < Nq} in ascending
// position, whatever the thread scheduling.
#include <algorithm>
#include <climits>

#include "vc_common.cuh"
#include "kernels.h"
#include "profile.h"

namespace vc {
namespace {

__device__ __forceinline__ uint32_t desc_key(float s) {
  // monotone map float -> uint32 (ascending), then invert for descending order
  uint32_t u = __float_as_uint(s);
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  return ~u;
}

// chunk_sort_kernel: CTA (chunk c, problem p) forms the composite keys
// (desc_key(score) << 32 | token) of tokens c*1024 ... c*1024+1023 (missing
// tokens: all ones) and sorts them ascending with a bitonic network in shared
// memory; composite keys are unique, so "ascending composite" is exactly
// "descending score, lower index first on exact ties".
// chunk_rank_kernel: CTA (c, p) holds its sorted chunk, one element per thread,
// and streams every other chunk of the problem through shared memory; a
// binary search counts that chunk's elements below the thread's element.  The
// element's rank is its position in its own chunk plus those counts: the
// number of elements of the whole problem below it.

// Ranking problem p: its request, score offset and chunk base; false when
// the problem's layer is not scored (per-layer ranking of an evicted layer in
// the fused pass), so the CTA has nothing to do.
__device__ __forceinline__ bool problem_of(const Shape& sh, const Tables& tb, int p, Req& rq,
                                           int64_t& off, int64_t& chunk_base, int& nchunks) {
  const bool per_layer = sh.rank_mode == VC_RANK_PER_LAYER;
  const int per_req = per_layer ? sh.L * sh.Hkv : sh.Hkv;
  const int r = p / per_req, k = p % per_req;
  rq = tb.req[r];
  nchunks = (rq.n + kSortChunk - 1) / kSortChunk;
  off = rq.s_off + (int64_t)k * rq.n;
  chunk_base = ((int64_t)rq.chunk0 + (int64_t)k * nchunks) * kSortChunk;
  return !per_layer || k / sh.Hkv < rq.Ls;
}

// Compare-exchange of the bitonic network between lanes t and t ^ j of a
// warp (j < 32): the lower lane keeps min/max as the direction bit says.
__device__ __forceinline__ uint64_t bitonic_lane(uint64_t a, int t, int j, int k) {
  const uint64_t b = __shfl_xor_sync(0xffffffffu, a, j);
  const bool up = (t & k) == 0;
  const bool lower = (t & j) == 0;
  return (lower == up) ? (a < b ? a : b) : (a < b ? b : a);
}

__global__ void __launch_bounds__(kSortChunk) chunk_sort_kernel(Shape sh, Tables tb,
                                                                const float* __restrict__ scores,
                                                                uint64_t* __restrict__ chunks) {
  __shared__ uint64_t e[kSortChunk];
  dep_wait();                                      // the scores
  if (threadIdx.x == 0) dep_launch();
  Req rq;
  int64_t off, base;
  int nchunks;
  const bool scored = problem_of(sh, tb, blockIdx.y, rq, off, base, nchunks);
  const int c = blockIdx.x;
  if (c >= nchunks || !scored) return;
  const int t = threadIdx.x;
  const int v = c * kSortChunk + t;
  uint64_t a = v < rq.n ? ((uint64_t)desc_key(scores[off + v]) << 32) | (uint32_t)v : ~0ull;
  // strides below 32 stay in the warp (shuffles), larger ones go through
  // shared memory with a block barrier
  for (int k = 2; k <= kSortChunk; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= 32) {
        e[t] = a;
        __syncthreads();
        const uint64_t b = e[t ^ j];
        const bool up = (t & k) == 0;
        const bool lower = (t & j) == 0;
        a = (lower == up) ? (a < b ? a : b) : (a < b ? b : a);
        __syncthreads();
      } else {
        a = bitonic_lane(a, t, j, k);
      }
    }
  }
  chunks[base + (int64_t)c * kSortChunk + t] = a;
}

// Other chunks are staged kRankGroup at a time (8 KB each) so a group costs
// one barrier pair; each thread then runs its binary searches back to back.
constexpr int kRankGroup = 12;

__global__ void __launch_bounds__(kSortChunk) chunk_rank_kernel(Shape sh, Tables tb,
                                                                const uint64_t* __restrict__ chunks,
                                                                int32_t* __restrict__ rank) {
  extern __shared__ uint64_t other[];               // [kRankGroup][kSortChunk]
  dep_wait();                                      // the sorted chunks
  if (threadIdx.x == 0) dep_launch();
  Req rq;
  int64_t off, base;
  int nchunks;
  const bool scored = problem_of(sh, tb, blockIdx.y, rq, off, base, nchunks);
  const int c = blockIdx.x;
  if (c >= nchunks || !scored) return;
  const int t = threadIdx.x;
  const uint64_t mine = chunks[base + (int64_t)c * kSortChunk + t];
  int count = t;                                   // elements of its own chunk below it
  for (int g0 = 0; g0 < nchunks; g0 += kRankGroup) {
    const int gn = min(kRankGroup, nchunks - g0);
    __syncthreads();
    for (int i = 0; i < gn; ++i)
      other[i * kSortChunk + t] = chunks[base + (int64_t)(g0 + i) * kSortChunk + t];
    __syncthreads();
    for (int i = 0; i < gn; ++i) {
      if (g0 + i == c) continue;
      const uint64_t* o = other + i * kSortChunk;
      int pos = 0;                                 // elements of chunk g0 + i below `mine`
#pragma unroll
      for (int s = kSortChunk; s > 0; s >>= 1)
        if (pos + s <= kSortChunk && o[pos + s - 1] < mine) pos += s;
      count += pos;
    }
  }
  if (mine != ~0ull) {
    const uint32_t v = (uint32_t)mine;
    if (v < (uint32_t)rq.n && count < rq.n) rank[off + v] = count;
    else set_status(tb.status, VC_ERR_DEVICE_INDEX);
  }
}

// threshold_kernel: CTA p cuts problem p.  Composites (desc_key(score) << 16 |
// token) are unique and ascend in ranking order; cut j is the composite at
// sorted position pos[j].  A round takes a range of composites: a histogram of
// kSelBuckets equal parts, a scan, and each cut's part is found by bisection;
// the elements of the cuts' parts are collected and each cut picks the one
// with the right number of smaller ones.  A part with more than kSelCap
// elements (many equal or nearly equal scores) becomes the range of another
// round; ranges shrink 16,384-fold, to single composites after four.
// Bound by the latency of one SM's shared memory and barriers, as four
// problems leave the other SMs idle.  Measured against the chunk kernels it
// replaces in the fused pass (event times, compaction not included): 7B shape,
// n = 12,544, 4 problems 25.3 -> 16.3 us; n = 3,136 18.8 -> 12.5 us; 112 problems
// (layer-specific ranking) 109 -> 16.6 us; 72B shape, n = 32,768 58 -> 34 us; the
// pass with layer-specific ranking 548 -> 461 us.
constexpr int kSelThreads = 1024;
constexpr int kSelBuckets = 16384;
constexpr int kSelCap = 512;
constexpr int kSelPool = 8192;
constexpr int kSelCuts = 257;                // 256 layers and Nq
constexpr int kSelHeld = 16384;              // tokens whose keys are kept in shared memory
// Every round finishes its first open cut or narrows that cut's range to one of
// 16,384 parts, and 48 bits of composite are gone after four: with scores that
// stand still no search takes more rounds than this.  Scores that change under
// it (a caller that shares a workspace between streams; past kSelHeld tokens
// they are read again) could leave a cut's range empty and the search without an end.
constexpr int kSelRounds = 4 * kSelCuts;

struct SelSmem {
  uint32_t count[kSelBuckets];               // counts, then first positions; a collected part: top bit | its cut
  uint64_t pool[kSelPool];                   // collected elements
  uint32_t key[kSelHeld];
  uint64_t lo[kSelCuts], hi[kSelCuts];       // a cut's range, its answer in lo once it is done
  int32_t base[kSelCuts], pos[kSelCuts];     // elements below the range; sorted position wanted, -1 done
  int32_t part[kSelCuts], first[kSelCuts], size[kSelCuts];   // a cut's part, its first position and size
  int32_t seg[kSelCuts], fill[kSelCuts];     // collected parts: offset in the pool, elements so far
  uint32_t wsum[32], wmin[32], wmax[32];
  int32_t todo;
};

// Exclusive sum over the block of one value per thread (two barriers).
__device__ __forceinline__ uint32_t block_before(uint32_t x, uint32_t* wsum) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  __syncthreads();                           // wsum's last readers are done
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  return __reduce_add_sync(0xffffffffu, lane < warp ? wsum[lane] : 0u) + incl - x;
}

__global__ void __launch_bounds__(kSelThreads, 1) threshold_kernel(Shape sh, Tables tb,
                                                                   const float* __restrict__ scores,
                                                                   uint64_t* __restrict__ cuts) {
  extern __shared__ __align__(16) uint8_t sel_sm[];
  SelSmem& sm = *reinterpret_cast<SelSmem*>(sel_sm);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const bool per_layer = sh.rank_mode == VC_RANK_PER_LAYER;
  const int ncut = per_layer ? 2 : sh.L + 1;
  auto zero = [&]() {
#pragma unroll
    for (int i = 0; i < kSelBuckets / 4 / kSelThreads; ++i)
      reinterpret_cast<uint4*>(sm.count)[t + i * kSelThreads] = make_uint4(0u, 0u, 0u, 0u);
  };
  zero();
  dep_wait();                                // the scores
  if (t == 0) dep_launch();
  Req rq;
  int64_t off, unused;
  int nchunks;
  if (!problem_of(sh, tb, blockIdx.x, rq, off, unused, nchunks)) return;
  const int n = rq.n;
  const float* sc = scores + off;
  // cuts: 0 the survivors, then the layers' budgets (non-increasing)
  {
    const int per_req = per_layer ? sh.L * sh.Hkv : sh.Hkv;
    const int r = blockIdx.x / per_req, l0 = per_layer ? blockIdx.x % per_req / sh.Hkv : 0;
    if (t < ncut) {
      sm.pos[t] = (t == 0 ? rq.Nq : tb.layer[r * sh.L + l0 + t - 1].B) - 1;
      sm.base[t] = 0;
    }
  }
  // range of the keys
  uint32_t kmin = 0xffffffffu, kmax = 0u;
  // the first kSelHeld keys stay in shared memory; visit(key, token) of this
  // thread's tokens (loops kept short: a launch starts with a cold
  // instruction cache, and straight-line code for 16 tokens cost more than it saved)
  const int held = min(n, kSelHeld);
#pragma unroll 4
  for (int v = t; v < held; v += kSelThreads) sm.key[v] = desc_key(sc[v]);
  auto each = [&](auto visit) {
#pragma unroll 4
    for (int v = t; v < held; v += kSelThreads) visit(sm.key[v], v);
#pragma unroll 2
    for (int v = kSelHeld + t; v < n; v += kSelThreads) visit(desc_key(sc[v]), v);
  };
  each([&](uint32_t k, int) {
    kmin = min(kmin, k);
    kmax = max(kmax, k);
  });
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if (lane == 0) {
    sm.wmin[warp] = kmin;
    sm.wmax[warp] = kmax;
  }
  __syncthreads();
  kmin = __reduce_min_sync(0xffffffffu, sm.wmin[lane]);
  kmax = __reduce_max_sync(0xffffffffu, sm.wmax[lane]);
  if (t < ncut) {
    sm.lo[t] = (uint64_t)kmin << 16;
    sm.hi[t] = (uint64_t)kmax << 16 | 0xffffu;
  }
  for (int round = 0; round < kSelRounds; ++round) {
    if (t == 0) sm.todo = kSelCuts;
    __syncthreads();
    if (t < ncut && sm.pos[t] >= 0) atomicMin(&sm.todo, t);
    __syncthreads();
    const int lead = sm.todo;                // the first cut not done: this round's range is its
    if (lead == kSelCuts) break;
    if (round > 0) {
      zero();
      __syncthreads();
    }
    const uint64_t lo = sm.lo[lead], hi = sm.hi[lead];
    const int shift = max(0, 64 - __clzll((long long)(hi - lo)) - 14);   // hi - lo >> shift < kSelBuckets
    each([&](uint32_t k, int v) {
      const uint64_t c = (uint64_t)k << 16 | (uint32_t)v;
      if (c >= lo && c <= hi) atomicAdd(&sm.count[(uint32_t)((c - lo) >> shift)], 1u);
    });
    __syncthreads();
    {                                        // exclusive scan: thread t owns 16 counts
      uint4* mine = reinterpret_cast<uint4*>(sm.count) + 4 * t;
      uint4 c[4];
      uint32_t sum = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        c[i] = mine[i];
        sum += c[i].x + c[i].y + c[i].z + c[i].w;
      }
      uint32_t run = block_before(sum, sm.wsum);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint4 x = c[i];
        mine[i] = make_uint4(run, run + x.x, run + x.x + x.y, run + x.x + x.y + x.z);
        run += x.x + x.y + x.z + x.w;
      }
    }
    __syncthreads();
    const uint32_t total = __reduce_add_sync(0xffffffffu, sm.wsum[lane]);
    // each cut of this range: its part
    int part = -1, first = 0, size = 0;
    if (t < ncut && sm.pos[t] >= 0 && sm.lo[t] == lo && sm.hi[t] == hi) {
      const uint32_t k = (uint32_t)(sm.pos[t] - sm.base[t]);
      int a = 0, b = kSelBuckets - 1;        // largest part whose first position is <= k
      while (a < b) {
        const int mid = (a + b + 1) >> 1;
        if (sm.count[mid] <= k) a = mid; else b = mid - 1;
      }
      part = a;
      first = (int)sm.count[a];
      size = (int)(a + 1 < kSelBuckets ? sm.count[a + 1] : total) - first;
    }
    if (t < ncut) {
      sm.part[t] = part;
      sm.first[t] = first;
      sm.size[t] = size;
    }
    __syncthreads();
    // the first cut of a part small enough collects it, if the pool has room
    // (the round's first always has); a later round takes the others
    const bool leads = part >= 0 && shift > 0 && size <= kSelCap && (t == 0 || sm.part[t - 1] != part);
    const uint32_t at = block_before(leads ? (uint32_t)size : 0u, sm.wsum);
    if (leads && at + size <= kSelPool) {
      sm.seg[t] = (int)at;
      sm.fill[t] = 0;
      sm.count[part] = 0x80000000u | (uint32_t)t;
    }
    __syncthreads();
    if (shift > 0)
      each([&](uint32_t k, int v) {
        const uint64_t c = (uint64_t)k << 16 | (uint32_t)v;
        if (c < lo || c > hi) return;
        const uint32_t w = sm.count[(uint32_t)((c - lo) >> shift)];
        if (w >> 31) {
          const int j = (int)(w & 0xffffu);
          const int i = atomicAdd(&sm.fill[j], 1);
          if (i < sm.size[j]) sm.pool[sm.seg[j] + i] = c;
        }
      });
    __syncthreads();
    for (int j = warp; j < ncut; j += kSelThreads / 32) {
      const int b = sm.part[j];
      if (b < 0) continue;
      const int m = sm.size[j];
      const uint32_t w = sm.count[b];
      if (shift == 0) {                      // the part is one composite
        if (lane == 0) {
          sm.lo[j] = lo + (uint32_t)b;
          sm.pos[j] = -1;
        }
      } else if (w >> 31) {
        const uint64_t* e = sm.pool + sm.seg[w & 0xffffu];
        const int k = sm.pos[j] - sm.base[j] - sm.first[j];
        __syncwarp();
        for (int i = lane; i < m; i += 32) {
          const uint64_t x = e[i];
          int below = 0;
          for (int q = 0; q < m; ++q) below += e[q] < x;
          if (below == k) {
            sm.lo[j] = x;
            sm.pos[j] = -1;
          }
        }
      } else if (m > kSelCap && lane == 0) { // narrow the range
        const uint64_t l = lo + ((uint64_t)b << shift);
        sm.lo[j] = l;
        sm.hi[j] = min((unsigned long long)hi, (unsigned long long)(l + (1ull << shift) - 1));
        sm.base[j] += sm.first[j];
      }
    }
    __syncthreads();
  }
  if (t < ncut) {
    if (sm.pos[t] >= 0) set_status(tb.status, VC_ERR_DEVICE_INDEX);
    cuts[(int64_t)blockIdx.x * ncut + t] = sm.lo[t];
  }
}

// One CTA per (request, layer, KV head); layers with B_l == 0 exit at once.
// RANKED: the ranks are given; else scores and cuts (threshold_kernel).  A
// segment is 32 warps x up to kScanPer x 32 consecutive tokens each.
constexpr int kScanThreads = 1024;
constexpr int kScanPer = 16;

template <bool RANKED>
__global__ void __launch_bounds__(kScanThreads) compact_kernel(Shape sh, Tables tb,
                                                               const int32_t* __restrict__ rank,
                                                               const float* __restrict__ scores,
                                                               const uint64_t* __restrict__ cuts,
                                                               int32_t* __restrict__ keep_idx,
                                                               int32_t* __restrict__ drop_idx) {
  constexpr int kWarps = kScanThreads / 32;
  __shared__ int32_t wk[2][kWarps], wd[2][kWarps];
  dep_wait();                                // the ranks or cuts
  if (threadIdx.x == 0) dep_launch();        // the gather may be scheduled
  const int g = blockIdx.y;
  const int rl = blockIdx.x;                 // request * L + layer
  const int r = rl / sh.L, l = rl % sh.L;
  const Req rq = tb.req[r];
  const Layer ly = tb.layer[rl];
  if (ly.B <= 0) return;
  const int n = rq.n;
  const bool per_layer = sh.rank_mode == VC_RANK_PER_LAYER;
  const int64_t at = rq.s_off + (per_layer ? (int64_t)l * sh.Hkv + g : (int64_t)g) * n;
  uint64_t ck = 0, cd = 0;                   // last composites kept and surviving
  if (!RANKED) {
    const int64_t p = per_layer ? (int64_t)rl * sh.Hkv + g : (int64_t)r * sh.Hkv + g;
    cd = cuts[per_layer ? 2 * p : p * (sh.L + 1)];
    ck = cuts[per_layer ? 2 * p + 1 : p * (sh.L + 1) + 1 + l];
  }
  int32_t* ko = keep_idx + rq.out_row0 + (int64_t)sh.Hkv * ly.P + (int64_t)g * ly.B;
  int32_t* dro = drop_idx + rq.drop_row0 + (int64_t)sh.Hkv * ly.Qd + (int64_t)g * ly.D;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t below = (1u << lane) - 1u;
  int base_k = 0, base_d = 0, flip = 0;
  for (int s0 = 0; s0 < n; flip ^= 1) {
    const int kk = min(kScanPer, (n - s0 + kScanThreads - 1) / kScanThreads);   // rounds of 32 tokens a warp
    const int v0 = s0 + warp * 32 * kk + lane;
    uint32_t x[kScanPer];
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
      const int v = v0 + 32 * k;
      x[k] = 0u;
      if (k < kk && v < n) x[k] = RANKED ? (uint32_t)rank[at + v] : __float_as_uint(scores[at + v]);
    }
    uint32_t keep = 0, drop = 0;             // bit k: token v0 + 32 k
    int nk = 0, nd = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
      if (k >= kk) break;
      const int v = v0 + 32 * k;
      bool is_k, is_s;
      if (RANKED) {
        is_k = (int)x[k] < ly.B;
        is_s = (int)x[k] < rq.Nq;
      } else {
        const uint64_t c = (uint64_t)desc_key(__uint_as_float(x[k])) << 16 | (uint32_t)v;
        is_k = c <= ck;
        is_s = c <= cd;
      }
      is_k = is_k && v < n;
      is_s = is_s && v < n && !is_k;
      keep |= (uint32_t)is_k << k;
      drop |= (uint32_t)is_s << k;
      nk += __popc(__ballot_sync(0xffffffffu, is_k));
      nd += __popc(__ballot_sync(0xffffffffu, is_s));
    }
    if (lane == 0) { wk[flip][warp] = nk; wd[flip][warp] = nd; }
    __syncthreads();
    const int a = wk[flip][lane], b = wd[flip][lane];
    int pk = base_k + (int)__reduce_add_sync(0xffffffffu, lane < warp ? a : 0);
    int pd = base_d + (int)__reduce_add_sync(0xffffffffu, lane < warp ? b : 0);
    base_k += (int)__reduce_add_sync(0xffffffffu, a);
    base_d += (int)__reduce_add_sync(0xffffffffu, b);
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
      if (k >= kk) break;
      const bool is_k = (keep >> k) & 1u, is_d = (drop >> k) & 1u;
      const uint32_t mk = __ballot_sync(0xffffffffu, is_k), md = __ballot_sync(0xffffffffu, is_d);
      if (is_k) {
        const int i = pk + __popc(mk & below);
        if (i < ly.B) ko[i] = v0 + 32 * k; else set_status(tb.status, VC_ERR_DEVICE_INDEX);
      }
      if (is_d) {
        const int i = pd + __popc(md & below);
        if (i < ly.D) dro[i] = v0 + 32 * k; else set_status(tb.status, VC_ERR_DEVICE_INDEX);
      }
      pk += __popc(mk);
      pd += __popc(md);
    }
    s0 += kScanThreads * kk;
  }
}

}  // namespace

cudaError_t launch_select(const Shape& sh, const Tables& tb, int n_problems, int max_chunks,
                          const float* scores, int32_t* rank, uint64_t* chunks, int32_t* keep_idx,
                          int32_t* drop_idx, cudaStream_t st) {
  const dim3 grid((unsigned)max_chunks, (unsigned)n_problems);
  {
    ProfileScope ps("chunk_sort", st);
    cudaError_t el = launch_dep(chunk_sort_kernel, grid, dim3(kSortChunk), 0, st, sh, tb, scores, chunks);
    if (el != cudaSuccess) return el;
  }
  cudaError_t e0 = cudaGetLastError();
  if (e0 != cudaSuccess) return e0;
  {
    const size_t smem = sizeof(uint64_t) * kSortChunk * (size_t)std::min(kRankGroup, std::max(max_chunks, 1));
    cudaError_t ea = cudaFuncSetAttribute(chunk_rank_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (ea != cudaSuccess) return ea;
    ProfileScope ps("chunk_rank", st);
    cudaError_t el = launch_dep(chunk_rank_kernel, grid, dim3(kSortChunk), smem, st, sh, tb,
                                static_cast<const uint64_t*>(chunks), rank);
    if (el != cudaSuccess) return el;
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  {
    ProfileScope ps("compact_keep_drop", st);
    // an ordinary launch: it starts once the ranks are complete.  Measured on
    // the ragged 8-request batch, the chain of dependent launches from the
    // column sums through the gather cost ~60 us per call when every link
    // of it was dependent, and nothing when any one of them was not; here
    // the break costs nothing on the single-request workloads.
    compact_kernel<true><<<dim3(sh.n_req * sh.L, sh.Hkv), kScanThreads, 0, st>>>(sh, tb, rank, nullptr, nullptr,
                                                                                 keep_idx, drop_idx);
  }
  return cudaGetLastError();
}

cudaError_t launch_cut(const Shape& sh, const Tables& tb, int n_problems, const float* scores, uint64_t* cuts,
                       int32_t* keep_idx, int32_t* drop_idx, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(threshold_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(SelSmem));
  if (e != cudaSuccess) return e;
  {
    ProfileScope ps("threshold", st);
    e = launch_dep(threshold_kernel, dim3((unsigned)n_problems), dim3(kSelThreads), sizeof(SelSmem), st, sh, tb,
                   scores, cuts);
    if (e != cudaSuccess) return e;
  }
  ProfileScope ps("compact_keep_drop", st);
  // dependent: without the sort and the rank before it the chain loses nothing
  // on ragged batches (launch_select), and a short call gains the gap (n = 3,136,
  // 28 layers: 158.4 -> 156.6 us; one fp32 layer of 1,024: 47.2 -> 45.2 us)
  return launch_dep(compact_kernel<false>, dim3(sh.n_req * sh.L, sh.Hkv), dim3(kScanThreads), 0, st, sh, tb,
                    static_cast<const int32_t*>(nullptr), scores, static_cast<const uint64_t*>(cuts), keep_idx,
                    drop_idx);
}

}  // namespace vc

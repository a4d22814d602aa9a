// Scout keyframe selection, Eq. (mmr) (Sec. 3.1): for each video, frame
// embeddings h_f and a prompt embedding h_t; frames join the selected set
// Omega greedily by
//     lambda * sim(h_f, h_t) - (1 - lambda) * max_{f' in Omega} sim(h_f, h_f')
// (cosine similarity) until k = ceil(p * F) frames are chosen.  Readings: the
// redundancy term is 0 while Omega is empty, ties go to the lower frame index,
// a zero vector has similarity 0 with everything.
//
// Three kernels, fp32 arithmetic:
//   scout_norm_kernel  one warp per frame / prompt row: the row scaled to unit
//                      length (zero rows stay zero);
//   scout_sim_kernel   per video the F x F cosine matrix S = Hn Hn^T, 64 x 64
//                      tiles (CUDA cores: the matrix is small and every later
//                      pick compares entries of it, so it is kept in fp32);
//   scout_mmr_kernel   one 1024-thread CTA per video runs the greedy loop:
//                      each thread holds up to four frames' relevance and
//                      running redundancy in registers, a block-wide argmax of
//                      (score, -index) picks the frame, and the picked frame's
//                      row of S updates the redundancies.  The picks are
//                      written in selection order, then (a block scan over the
//                      frame flags) in ascending frame order.
// Videos are independent: the batch is the data-parallel axis (one CTA each).
//
// Short videos (F <= 128 frames whose rows and S fit in 224 KB: the paper's 64 CLIP frames of
// width 512) take one fused kernel instead, scout_small_kernel: a cluster of two
// CTAs per video, each with the raw rows d-major in its shared memory (dot
// products are scaled by the two inverse norms afterwards).  The CTAs share the
// 4 x 4 tiles of S's upper triangle (four lanes per tile, each summing a quarter
// of the width, parts added in a fixed order); the second writes its part into
// the first's S through distributed shared memory.  The first CTA also computes
// the relevances, on warps that have no tile, and runs the greedy loop inside
// one warp (two or four frames per lane; the warp argmax is a max reduction of
// the score key and a min reduction of the frame index; no block barriers).
// Each video takes one path by its own size, so a batch returns what its videos
// return one by one.
// Bound by latency: the load, half of S's serial sums and k picks follow one
// another.  64 videos of 64 frames (48 picks): 32.7 us with one CTA a video (64
// of 152 SMs busy, packed fmas at a quarter of the scalar rate, transposed 4-byte
// stores with 4-way conflicts), 20.5 us now (8.2 us
// of it at 32 dimensions and one pick: launch, cluster start and exit).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include <cooperative_groups.h>

#include "profile.h"
#include "tc_common.cuh"
#include "viscache.h"

namespace vc {
namespace {

constexpr int kScoutMaxReq = 64;
constexpr int kScoutMaxFrames = 4096;
constexpr int kMmrThreads = 1024;
constexpr int kFpt = kScoutMaxFrames / kMmrThreads;   // frames per thread
constexpr int kSimTile = 64;
constexpr int kSimChunk = 32;
constexpr size_t kWsAlign = 256;

struct ScoutTable {            // kernel parameter: per-video sizes and offsets
  int32_t n_req, D;
  float lam;
  int32_t F[kScoutMaxReq];     // frames
  int32_t k[kScoutMaxReq];     // keyframes
  int32_t k_off[kScoutMaxReq]; // first output row
  int64_t h_off[kScoutMaxReq]; // first frame row of H
  int64_t s_off[kScoutMaxReq]; // first element of the video's F x F matrix
};

constexpr int kSmallMaxFrames = 128;
constexpr int kSmallMaxFloats = 56000;       // shared memory of the fused kernel, in floats
constexpr int kSmallThreads = 768;

// Row strides of the fused kernel's d-major rows.  small_ld (F rounded up to 4
// plus 4) decides by its size which videos take the kernel; wide_ld, 8 or 24
// words mod 32, keeps the four parts of a tile's 16-byte loads on different
// banks and is used where it still fits.
__host__ __device__ __forceinline__ int small_ld(int F) { return ((F + 3) & ~3) + 4; }
__host__ __device__ __forceinline__ int wide_ld(int F) { return ((F + 7) & ~15) + 8; }
__host__ __device__ __forceinline__ int64_t small_floats(int F, int D, int ld) {
  return (int64_t)D * ld + (int64_t)F * F + D + F;
}
__host__ __device__ __forceinline__ int used_ld(int F, int D) {
  return small_floats(F, D, wide_ld(F)) <= kSmallMaxFloats ? wide_ld(F) : small_ld(F);
}
// A video small enough for the fused kernel (the paper's 64 frames of width 512 are).
__host__ __device__ __forceinline__ bool small_video(int F, int D) {
  return F <= kSmallMaxFrames && small_floats(F, D, small_ld(F)) <= kSmallMaxFloats;
}

__global__ void __launch_bounds__(256) scout_norm_kernel(const float* __restrict__ H,
                                                         const float* __restrict__ P, int64_t frames,
                                                         int n_req, int D, float* __restrict__ Hn,
                                                         float* __restrict__ Tn) {
  const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= frames + n_req) return;
  const float* src = row < frames ? H + row * D : P + (row - frames) * D;
  float* dst = row < frames ? Hn + row * D : Tn + (row - frames) * D;
  float ss = 0.f;
  for (int j = lane; j < D; j += 32) ss = fmaf(src[j], src[j], ss);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  const float inv = ss > 0.f ? 1.f / sqrtf(ss) : 0.f;
  for (int j = lane; j < D; j += 32) dst[j] = src[j] * inv;
}

// S_r = Hn_r Hn_r^T; block (tile row, tile col, video), 256 threads, 4 x 4
// outputs each.
__global__ void __launch_bounds__(256) scout_sim_kernel(const __grid_constant__ ScoutTable tb,
                                                        const float* __restrict__ Hn,
                                                        float* __restrict__ S) {
  __shared__ float a[kSimChunk][kSimTile + 1], b[kSimChunk][kSimTile + 1];
  const int r = blockIdx.z;
  const int F = tb.F[r], D = tb.D;
  const int i0 = blockIdx.y * kSimTile, j0 = blockIdx.x * kSimTile;
  if (i0 >= F || j0 >= F || small_video(F, D)) return;
  const float* h = Hn + tb.h_off[r] * D;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc[4][4] = {};
  for (int d0 = 0; d0 < D; d0 += kSimChunk) {
    for (int e = threadIdx.x; e < kSimChunk * kSimTile; e += 256) {
      const int row = e / kSimChunk, col = e % kSimChunk;   // consecutive threads read one row
      const int d = d0 + col;
      a[col][row] = (i0 + row < F && d < D) ? h[(int64_t)(i0 + row) * D + d] : 0.f;
      b[col][row] = (j0 + row < F && d < D) ? h[(int64_t)(j0 + row) * D + d] : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int c = 0; c < kSimChunk; ++c) {
      float x[4], y[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        x[u] = a[c][ty * 4 + u];
        y[u] = b[c][tx * 4 + u];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(x[u], y[v], acc[u][v]);
    }
    __syncthreads();
  }
  float* s = S + tb.s_off[r];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int i = i0 + ty * 4 + u, j = j0 + tx * 4 + v;
      if (i < F && j < F) s[(int64_t)i * F + j] = acc[u][v];
    }
}

// Order-preserving map of a float onto uint32 (ascending) and back.
__device__ __forceinline__ uint32_t ord_key(float x) {
  const uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord_value(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

// Block-wide maximum of a 64-bit key; every thread gets the result.
__device__ __forceinline__ unsigned long long block_max(unsigned long long v, unsigned long long* warp_max,
                                                        unsigned long long* result) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  if (lane == 0) warp_max[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = warp_max[lane];                      // 32 warps
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
      v = w > v ? w : v;
    }
    if (lane == 0) *result = v;
  }
  __syncthreads();
  return *result;
}

// Exclusive prefix count of a per-thread flag over the block (thread order);
// *total gets the block's count.
__device__ __forceinline__ int block_exclusive_count(bool flag, int* warp_cnt, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned m = __ballot_sync(0xffffffffu, flag);
  if (lane == 0) warp_cnt[warp] = __popc(m);
  __syncthreads();
  if (warp == 0) {
    const int c = warp_cnt[lane];
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    warp_cnt[lane] = incl - c;
    if (lane == 31) *total = incl;
  }
  __syncthreads();
  const int before = warp_cnt[warp] + __popc(m & ((1u << lane) - 1u));
  __syncthreads();                           // warp_cnt is reused by the next call
  return before;
}

__global__ void __launch_bounds__(kMmrThreads, 1) scout_mmr_kernel(const __grid_constant__ ScoutTable tb,
                                                                   const float* __restrict__ Hn,
                                                                   const float* __restrict__ Tn,
                                                                   const float* __restrict__ S,
                                                                   int32_t* __restrict__ order,
                                                                   int32_t* __restrict__ keyframes,
                                                                   float* __restrict__ gains) {
  __shared__ unsigned long long warp_max[32];
  __shared__ unsigned long long winner;
  __shared__ int warp_cnt[32];
  __shared__ int seg_total;
  const int r = blockIdx.x;
  const int F = tb.F[r], k = tb.k[r], D = tb.D;
  if (small_video(F, D)) return;               // the fused kernel takes it
  const float lam = tb.lam;
  const float* hn = Hn + tb.h_off[r] * D;
  const float* tn = Tn + (int64_t)r * D;
  const float* s = S + tb.s_off[r];
  const int t = threadIdx.x;

  float rel[kFpt], red[kFpt];
  bool sel[kFpt];
#pragma unroll
  for (int j = 0; j < kFpt; ++j) {
    const int f = t + j * kMmrThreads;
    float acc = 0.f;
    if (f < F)
      for (int d = 0; d < D; ++d) acc = fmaf(hn[(int64_t)f * D + d], tn[d], acc);
    rel[j] = acc;
    red[j] = 0.f;                            // empty selected set: no redundancy
    sel[j] = false;
  }
  for (int i = 0; i < k; ++i) {
    unsigned long long best = 0;             // below every real key
#pragma unroll
    for (int j = 0; j < kFpt; ++j) {
      const int f = t + j * kMmrThreads;
      if (f < F && !sel[j]) {
        const float sc = fmaf(-(1.f - lam), red[j], lam * rel[j]);   // same rounding in both paths
        const unsigned long long key = ((unsigned long long)ord_key(sc) << 32) | (0xffffffffu - (uint32_t)f);
        best = key > best ? key : best;
      }
    }
    const unsigned long long w = block_max(best, warp_max, &winner);
    const int fs = (int)(0xffffffffu - (uint32_t)w);
    if (t == 0) {
      order[tb.k_off[r] + i] = fs;
      if (gains) gains[tb.k_off[r] + i] = ord_value((uint32_t)(w >> 32));
    }
    const float* row = s + (int64_t)fs * F;   // S is symmetric: row fs = column fs
#pragma unroll
    for (int j = 0; j < kFpt; ++j) {
      const int f = t + j * kMmrThreads;
      if (f < F) {
        const float x = row[f];
        red[j] = i == 0 ? x : fmaxf(red[j], x);
        if (f == fs) sel[j] = true;
      }
    }
  }
  // ascending frame order: frame f = t + j*1024 goes to (selected frames
  // before it), counted segment by segment
  int base = 0;
#pragma unroll
  for (int j = 0; j < kFpt; ++j) {
    const int before = block_exclusive_count(sel[j], warp_cnt, &seg_total);
    if (sel[j]) keyframes[tb.k_off[r] + base + before] = t + j * kMmrThreads;
    base += seg_total;
    __syncthreads();                         // seg_total is rewritten by the next segment
  }
}

// The greedy loop of one warp: the lane holds frames lane, lane + 32, ... (J of
// them); pick[i] and pick_gain[i] get the i-th frame and its score.
template <int J>
__device__ __forceinline__ void pick_frames(const float* S, const float* rel, int F, int k, float lam, int* pick,
                                            float* pick_gain, bool (&sel)[kSmallMaxFrames / 32]) {
  const int lane = threadIdx.x & 31;
  float lr[J], red[J];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int f = lane + 32 * j;
    lr[j] = f < F ? lam * rel[f] : 0.f;
    red[j] = 0.f;                                // empty selected set: no redundancy
    sel[j] = f >= F;                             // frames past F are never picked
  }
  for (int i = 0; i < k; ++i) {
    // this lane's best frame (highest score, then lowest index), then the
    // warp's: the highest score key, and the lowest frame holding it
    uint32_t kb = 0, fb = 0xffffffffu;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const uint32_t key = sel[j] ? 0u : ord_key(fmaf(-(1.f - lam), red[j], lr[j]));
      if (key > kb) {
        kb = key;
        fb = (uint32_t)(lane + 32 * j);
      }
    }
    const uint32_t kmax = __reduce_max_sync(0xffffffffu, kb);
    const int fs = (int)__reduce_min_sync(0xffffffffu, kb == kmax ? fb : 0xffffffffu);
    if (lane == 0) {
      pick[i] = fs;
      pick_gain[i] = ord_value(kmax);
    }
    const float* row = S + (size_t)fs * F;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int f = lane + 32 * j;
      if (f < F) {
        red[j] = i == 0 ? row[f] : fmaxf(red[j], row[f]);
        if (f == fs) sel[j] = true;
      }
    }
  }
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kSmallThreads, 1)
    scout_small_kernel(const __grid_constant__ ScoutTable tb, const float* __restrict__ H, const float* __restrict__ P,
                       int32_t* __restrict__ order, int32_t* __restrict__ keyframes, float* __restrict__ gains) {
  extern __shared__ __align__(16) float sm[];
  __shared__ float inv_norm[kSmallMaxFrames + 1];
  __shared__ int pick[kSmallMaxFrames];
  __shared__ float pick_gain[kSmallMaxFrames];
  const int r = blockIdx.x >> 1, rank = blockIdx.x & 1;
  const int F = tb.F[r], D = tb.D;
  if (!small_video(F, D)) return;              // the three-kernel path takes it (both CTAs leave)
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  tc::cluster_arrive();                            // "started": waited for before S is written remotely
  const int k = tb.k[r], ld = used_ld(F, D);
  const float lam = tb.lam;
  float* hT = sm;                              // [D][ld] rows, d-major
  float* S = hT + (size_t)D * ld;              // [F][F] (the first CTA's is used)
  float* tn = S + (size_t)F * F;               // [D] prompt
  float* rel = tn + D;                         // [F] relevance
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* h = H + tb.h_off[r] * D;
  const int nt = (F + 3) / 4;
  // raw rows into shared memory (four rows of a warp as one 16-byte piece per
  // dimension; the prompt as group nt) and each row's inverse norm
  for (int q = warp; q <= nt; q += kSmallThreads / 32) {
    float ss[4] = {};
    const float* src[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) src[u] = q < nt ? (4 * q + u < F ? h + (int64_t)(4 * q + u) * D : nullptr)
                                               : (u == 0 ? P + (int64_t)r * D : nullptr);
#pragma unroll 8
    for (int j = lane; j < D; j += 32) {
      float x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = src[u] ? src[u][j] : 0.f;
#pragma unroll
      for (int u = 0; u < 4; ++u) ss[u] = fmaf(x[u], x[u], ss[u]);
      if (q < nt) *reinterpret_cast<float4*>(hT + (size_t)j * ld + 4 * q) = make_float4(x[0], x[1], x[2], x[3]);
      else tn[j] = x[0];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ss[u] += __shfl_xor_sync(0xffffffffu, ss[u], o);
      const int row = q < nt ? 4 * q + u : F + u;
      if (lane == 0 && row <= F && (q == nt || row < F)) inv_norm[row] = ss[u] > 0.f ? 1.f / sqrtf(ss[u]) : 0.f;
    }
  }
  __syncthreads();
  tc::cluster_wait();
  float* S0 = cluster.map_shared_rank(S, 0);
  // S = hn hn^T: 4 x 4 tiles of the upper triangle, mirrored; this CTA takes
  // every second one.  Four adjacent lanes share a tile, lane part p summing
  // widths p, p+4, ...; the parts are added as (p0 + p1) + (p2 + p3) by two
  // shuffles, and lane p scales and writes the tile's row p.
  const int ntri = nt * (nt + 1) / 2;
  const int mine = (ntri + 1 - rank) / 2;
  for (int item = threadIdx.x; item < 4 * ((mine + 7) / 8) * 8; item += kSmallThreads) {
    const int part = item & 3;
    const bool live = (item >> 2) < mine;
    int a = 0, rem = live ? 2 * (item >> 2) + rank : 0;
    while (rem >= nt - a) {
      rem -= nt - a;
      ++a;
    }
    const int i0 = a * 4, j0 = (a + rem) * 4;
    float acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
    if (live) {
#pragma unroll 8
      for (int d = part; d < D; d += 4) {
        const float4 x = *reinterpret_cast<const float4*>(hT + (size_t)d * ld + i0);
        const float4 y = *reinterpret_cast<const float4*>(hT + (size_t)d * ld + j0);
        const float xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(xs[u], ys[v], acc[u][v]);
      }
    }
    float out[4] = {};                         // row `part` of the tile
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        float w = acc[u][v];
        w += __shfl_xor_sync(0xffffffffu, w, 1);
        w += __shfl_xor_sync(0xffffffffu, w, 2);
        if (part == u) out[v] = w;
      }
    const int i = i0 + part;
    if (live && i < F) {
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int j = j0 + v;
        if (j < F && (i0 != j0 || j <= i)) {   // a diagonal tile's pairs once, the larger index first
          const float c = (out[v] * inv_norm[i]) * inv_norm[j];
          S0[(size_t)i * F + j] = c;
          S0[(size_t)j * F + i] = c;
        }
      }
    }
  }
  // relevance, from the last warp down (the tiles fill from the first): four
  // lanes per frame, parts combined as for S
  if (rank == 0)
    for (int item = kSmallThreads - 32 - 32 * warp + lane; item < 4 * ((F + 7) / 8) * 8; item += kSmallThreads) {
      const int f = item >> 2, part = item & 3;
      float acc = 0.f;
      if (f < F) {
#pragma unroll 8
        for (int d = part; d < D; d += 4) acc = fmaf(hT[(size_t)d * ld + f], tn[d], acc);
      }
      acc += __shfl_xor_sync(0xffffffffu, acc, 1);
      acc += __shfl_xor_sync(0xffffffffu, acc, 2);
      if (f < F && part == 0) rel[f] = (acc * inv_norm[f]) * inv_norm[F];
    }
  __syncwarp();
  tc::cluster_arrive();
  tc::cluster_wait();                              // S and the relevances are complete in the first CTA
  if (rank != 0 || warp != 0) return;
  // greedy loop in warp 0: lane holds frames lane, lane + 32, ...
  constexpr int kLaneFrames = kSmallMaxFrames / 32;
  bool sel[kLaneFrames] = {};
  if (F <= 64) pick_frames<2>(S, rel, F, k, lam, pick, pick_gain, sel);
  else pick_frames<kLaneFrames>(S, rel, F, k, lam, pick, pick_gain, sel);
  const int o0 = tb.k_off[r];
  __syncwarp();
  for (int i = lane; i < k; i += 32) {
    order[o0 + i] = pick[i];
    if (gains) gains[o0 + i] = pick_gain[i];
  }
  // ascending frame order: frame lane + 32 j after the picks of lower frames
  int base = 0;
#pragma unroll
  for (int j = 0; j < kLaneFrames; ++j) {
    const bool mine = sel[j] && lane + 32 * j < F;
    const unsigned m = __ballot_sync(0xffffffffu, mine);
    if (mine) keyframes[o0 + base + __popc(m & ((1u << lane) - 1u))] = lane + 32 * j;
    base += __popc(m);
  }
}

inline size_t align_up(size_t x) { return (x + kWsAlign - 1) / kWsAlign * kWsAlign; }

struct ScoutLayout {
  size_t o_hn = 0, o_tn = 0, o_s = 0, total = 0;
  int64_t frames = 0, s_elems = 0;
};

// Host checks and the per-video table; returns VC_OK or an error code.
int scout_plan(int32_t n_req, const int32_t* n_frames, int32_t D, uint32_t p_num, uint32_t p_den,
               float lam, ScoutTable* tb, ScoutLayout* lay) {
  if (n_req < 1 || n_req > kScoutMaxReq || !n_frames || D < 1 || D > 8192) return VC_ERR_INVALID_ARG;
  if (p_den == 0 || p_num == 0 || p_num > p_den || !(lam >= 0.f && lam <= 1.f)) return VC_ERR_INVALID_ARG;
  tb->n_req = n_req;
  tb->D = D;
  tb->lam = lam;
  int64_t frames = 0, s_elems = 0;
  int32_t k_off = 0;
  for (int r = 0; r < n_req; ++r) {
    const int32_t F = n_frames[r];
    if (F < 1 || F > kScoutMaxFrames) return VC_ERR_INVALID_ARG;
    // k = ceil(p F), at least 1 (p > 0 and F >= 1 give k >= 1), at most F
    const int64_t k = ((int64_t)p_num * F + p_den - 1) / p_den;
    tb->F[r] = F;
    tb->k[r] = (int32_t)k;
    tb->k_off[r] = k_off;
    tb->h_off[r] = frames;
    tb->s_off[r] = s_elems;
    k_off += (int32_t)k;
    frames += F;
    s_elems += (int64_t)F * F;
  }
  lay->frames = frames;
  lay->s_elems = s_elems;
  lay->o_hn = 0;
  lay->o_tn = align_up(sizeof(float) * frames * D);
  lay->o_s = lay->o_tn + align_up(sizeof(float) * (size_t)n_req * D);
  lay->total = lay->o_s + align_up(sizeof(float) * s_elems);
  return VC_OK;
}

}  // namespace
}  // namespace vc

using namespace vc;

extern "C" size_t viscache_scout_workspace_size(int32_t n_req, const int32_t* n_frames, int32_t D) {
  ScoutTable tb;
  ScoutLayout lay;
  return scout_plan(n_req, n_frames, D, 1, 1, 0.5f, &tb, &lay) == VC_OK ? lay.total : 0;
}

extern "C" int viscache_scout_sizes(int32_t n_req, const int32_t* n_frames, uint32_t p_num,
                                    uint32_t p_den, int32_t* k_out) {
  if (!k_out) return VC_ERR_INVALID_ARG;
  ScoutTable tb;
  ScoutLayout lay;
  const int rc = scout_plan(n_req, n_frames, 1, p_num, p_den, 0.5f, &tb, &lay);
  if (rc != VC_OK) return rc;
  for (int r = 0; r < n_req; ++r) k_out[r] = tb.k[r];
  return VC_OK;
}

extern "C" int viscache_scout_mmr(const float* H, const float* prompt, int32_t n_req,
                                  const int32_t* n_frames, int32_t D, float lambda, uint32_t p_num,
                                  uint32_t p_den, int32_t* order_out, int32_t* keyframes_out,
                                  float* gains_out, int32_t* k_out, void* ws, size_t ws_bytes,
                                  void* stream) {
  ScoutTable tb;
  ScoutLayout lay;
  const int rc = scout_plan(n_req, n_frames, D, p_num, p_den, lambda, &tb, &lay);
  if (rc != VC_OK) return rc;
  if (!H || !prompt || !order_out || !keyframes_out) return VC_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(H) | reinterpret_cast<uintptr_t>(prompt)) & 3u) return VC_ERR_INVALID_ARG;
  if (!ws || (reinterpret_cast<uintptr_t>(ws) & (kWsAlign - 1)) != 0 || ws_bytes < lay.total)
    return VC_ERR_WORKSPACE;
  if (k_out)
    for (int r = 0; r < n_req; ++r) k_out[r] = tb.k[r];
  uint8_t* w = static_cast<uint8_t*>(ws);
  float* Hn = reinterpret_cast<float*>(w + lay.o_hn);
  float* Tn = reinterpret_cast<float*>(w + lay.o_tn);
  float* S = reinterpret_cast<float*>(w + lay.o_s);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // each video goes to the fused kernel or to the three-kernel path by its size
  int fmax_large = 0;
  int64_t floats_small = 0;
  for (int r = 0; r < n_req; ++r) {
    if (small_video(tb.F[r], D)) floats_small = std::max(floats_small, small_floats(tb.F[r], D, used_ld(tb.F[r], D)));
    else fmax_large = std::max(fmax_large, tb.F[r]);
  }
  if (floats_small > 0) {
    ProfileScope ps("scout_small", st);
    const size_t smem = sizeof(float) * (size_t)floats_small;
    if (cudaFuncSetAttribute(scout_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
      return VC_ERR_CUDA;
    scout_small_kernel<<<2u * (unsigned)n_req, kSmallThreads, smem, st>>>(tb, H, prompt, order_out, keyframes_out,
                                                                    gains_out);
    if (cudaGetLastError() != cudaSuccess) return VC_ERR_CUDA;
  }
  if (fmax_large == 0) return VC_OK;
  {
    ProfileScope ps("scout_norm", st);
    const int64_t rows = lay.frames + n_req;
    scout_norm_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(H, prompt, lay.frames, n_req, D, Hn, Tn);
    if (cudaGetLastError() != cudaSuccess) return VC_ERR_CUDA;
  }
  {
    ProfileScope ps("scout_sim", st);
    const unsigned tiles = (unsigned)((fmax_large + kSimTile - 1) / kSimTile);
    scout_sim_kernel<<<dim3(tiles, tiles, (unsigned)n_req), 256, 0, st>>>(tb, Hn, S);
    if (cudaGetLastError() != cudaSuccess) return VC_ERR_CUDA;
  }
  {
    ProfileScope ps("scout_mmr", st);
    scout_mmr_kernel<<<(unsigned)n_req, kMmrThreads, 0, st>>>(tb, Hn, Tn, S, order_out, keyframes_out,
                                                              gains_out);
    if (cudaGetLastError() != cudaSuccess) return VC_ERR_CUDA;
  }
  return VC_OK;
}

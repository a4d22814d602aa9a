// Decode attention over the compressed cache (Sec. 2 "VLLM Decoding", with the
// visual part of layer l's cache replaced by PruneKV's (K_new, V_new), Sec. 3.2):
//     out_j = softmax(q_j K_g^T * scale) V_g,  g = j // G,
// over KV head g's B kept visual rows of the layer followed by its T text rows.
//
// A decode step reads the whole layer cache once for a handful of query rows:
// bound by those reads.
//   decode_tiles_kernel    (bf16 caches, and its Q4 form over the 4-bit cache)
//                          warps stream tiles of 32 keys on the tensor cores,
//                          a cluster of CTAs per (request, KV head) merges
//                          them (below)
//   decode_partial_kernel  (fp32 caches, splits of 256 keys) on CUDA cores, one
//                          256-thread CTA per unit (request, KV head, split):
//                          K, then V rows staged in one shared buffer by
//                          16-byte asynchronous copies, the row's pieces
//                          XOR-permuted so that the reads hit distinct banks;
//                          two threads per key pair form the logits with
//                          packed fp32 FMAs against duplicated query values;
//                          threads own 16-byte pieces of the V rows for a key
//                          slice; decode_combine_kernel (one warp per request
//                          and query head) then merges the splits: the
//                          unnormalised partial output and (max, sum) per
//                          query.
// A query with no keys at all (an evicted layer, no text) gets zeros.
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "decode_plan.h"
#include "kernels.h"
#include "profile.h"
#include "tc_common.cuh"
#include "vc_common.cuh"

namespace vc {
namespace {

constexpr int kSplitF = 256;                  // keys per CTA, fp32 caches (CUDA cores)
constexpr int kDecThreads = 256;
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kGm = kDecodeMaxGroup;
constexpr float kLog2eF = 1.4426950408889634f;

template <typename T, int D>
struct DecCfg {
  static constexpr int RB = D * (int)sizeof(T);          // bytes of a cache row
  static constexpr int PR = RB / 16;                     // 16-byte pieces of a row
  static constexpr int EPP = 16 / (int)sizeof(T);        // elements of a piece
  static constexpr int RW = 32 / PR;                     // rows a warp reads at once (phase 3)
  static constexpr int KS = kDecWarps * RW;              // phase-3 key slices
  static constexpr size_t BUF = (size_t)kSplitF * RB;     // K rows, then V rows, then partials
  static constexpr size_t QS = (size_t)D * kGm * 8;      // (q, q) pairs [D][kGm]
  static constexpr size_t PS = (size_t)kSplitF * kGm * 8; // (p, p) pairs [kSplitF][kGm]
  static constexpr size_t RED = (size_t)2 * kDecWarps * kGm * 4;
  static constexpr size_t SMEM = BUF + QS + PS + RED;
  static_assert(PR >= 8 && PR <= 32, "row of 8..32 pieces");
  static_assert(kSplitF == kDecThreads, "two threads per key pair (p, p + kSplitF / 2)");
  static_assert((size_t)kDecWarps * kGm * D * 4 <= BUF, "warp partials fit the row buffer");
};

__device__ __forceinline__ int piece_slot(int r, int c) { return c ^ ((r & 3) << 1); }

__device__ __forceinline__ void unpack(const uint4& u, const float*, float (&v)[4]) {
  v[0] = __uint_as_float(u.x); v[1] = __uint_as_float(u.y);
  v[2] = __uint_as_float(u.z); v[3] = __uint_as_float(u.w);
}

__device__ __forceinline__ int find_req(const DecodeTable& tb, int unit) {
  int lo = 0, hi = tb.n_req - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tb.req[mid].unit0 <= unit) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Stage rows [0, nk) of the split (visual rows first, then text rows) into buf.
template <typename T, int D>
__device__ __forceinline__ void stage_rows(uint8_t* buf, const T* vis, const T* txt, int nv, int nk) {
  using C = DecCfg<T, D>;
  for (int i = (int)threadIdx.x; i < nk * C::PR; i += kDecThreads) {
    const int r = i / C::PR, c = i % C::PR;
    const T* src = r < nv ? vis + (int64_t)r * D : txt + (int64_t)(r - nv) * D;
    tc::cp_async16(buf + (size_t)r * C::RB + piece_slot(r, c) * 16, src + c * C::EPP, 16);
  }
  tc::cp_async_commit();
}

template <typename T, int D>
__global__ void __launch_bounds__(kDecThreads, 1) decode_partial_kernel(
    const __grid_constant__ DecodeTable tb, const T* __restrict__ q, const T* __restrict__ Kc,
    const T* __restrict__ Vc, const T* __restrict__ Kt, const T* __restrict__ Vt,
    float* __restrict__ part_o, float2* __restrict__ part_ml) {
  using C = DecCfg<T, D>;
  extern __shared__ __align__(128) uint8_t dsm[];
  uint8_t* buf = dsm;
  float2* qs = reinterpret_cast<float2*>(dsm + C::BUF);               // [D][kGm]
  float2* ps = reinterpret_cast<float2*>(dsm + C::BUF + C::QS);       // [kSplitF][kGm]
  float* wmax = reinterpret_cast<float*>(dsm + C::BUF + C::QS + C::PS);
  float* wsum = wmax + kDecWarps * kGm;
  const int unit = blockIdx.x;
  const int r = find_req(tb, unit);
  const DecodeReq rq = tb.req[r];
  const int u = unit - rq.unit0;
  const int g = u / rq.nsplit, s = u % rq.nsplit;
  const int G = tb.G;
  const int k0 = s * tb.split;                // tb.split == kSplitF on this path
  const int nk = min(tb.split, rq.B + rq.T - k0);
  const int nv = max(0, min(nk, rq.B - k0));  // the split's visual keys come first
  const int64_t vis0 = rq.vis_row0 + (int64_t)g * rq.B + k0;
  const int64_t txt0 = rq.txt_row0 + (int64_t)g * rq.T + (k0 + nv - rq.B);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  stage_rows<T, D>(buf, Kc + vis0 * D, Kt + txt0 * D, nv, nk);
  // query rows g*G ... of request r in log2 units, each value duplicated
  const float c2 = tb.scale * kLog2eF;
  for (int e = t; e < kGm * D; e += kDecThreads) {
    const int jj = e % kGm, d = e / kGm;
    const float x = jj < G ? Elem<T>::to_f(q[((int64_t)r * tb.Hq + g * G + jj) * D + d]) * c2 : 0.f;
    qs[d * kGm + jj] = make_float2(x, x);
  }
  tc::cp_async_wait<0>();
  __syncthreads();
  // phase 1: logits of keys kA = p and kB = p + kSplitF/2 over this thread's pieces
  const int p = t >> 1, h = t & 1;
  const int kA = p, kB = p + kSplitF / 2;
  float2 acc[kGm];
#pragma unroll
  for (int jj = 0; jj < kGm; ++jj) acc[jj] = make_float2(0.f, 0.f);
#pragma unroll 2
  for (int i = 0; i < C::PR / 2; ++i) {
    const int c = 2 * i + h;
    const uint4 ua = *reinterpret_cast<const uint4*>(buf + (size_t)kA * C::RB + piece_slot(kA, c) * 16);
    const uint4 ub = *reinterpret_cast<const uint4*>(buf + (size_t)kB * C::RB + piece_slot(kB, c) * 16);
    float va[C::EPP], vb[C::EPP];
    unpack(ua, (const T*)nullptr, va);
    unpack(ub, (const T*)nullptr, vb);
#pragma unroll
    for (int e = 0; e < C::EPP; ++e) {
      const float2 kv = make_float2(va[e], vb[e]);
      const float4* qrow = reinterpret_cast<const float4*>(qs + (c * C::EPP + e) * kGm);
#pragma unroll
      for (int j2 = 0; j2 < kGm / 2; ++j2) {
        if (2 * j2 < G) {
          const float4 qq = qrow[j2];
          acc[2 * j2] = __ffma2_rn(kv, make_float2(qq.x, qq.y), acc[2 * j2]);
          if (2 * j2 + 1 < G) acc[2 * j2 + 1] = __ffma2_rn(kv, make_float2(qq.z, qq.w), acc[2 * j2 + 1]);
        }
      }
    }
  }
  // the two halves of the row; thread h keeps key h ? kB : kA
  const int kmine = h ? kB : kA;
  const bool valid = kmine < nk;
  float x[kGm];
#pragma unroll
  for (int jj = 0; jj < kGm; ++jj) {
    const float ax = acc[jj].x + __shfl_xor_sync(0xffffffffu, acc[jj].x, 1);
    const float ay = acc[jj].y + __shfl_xor_sync(0xffffffffu, acc[jj].y, 1);
    x[jj] = valid ? (h ? ay : ax) : -INFINITY;
  }
  __syncthreads();                              // K rows no longer read: stage V
  stage_rows<T, D>(buf, Vc + vis0 * D, Vt + txt0 * D, nv, nk);
  // phase 2: split max per query, exp2 terms and their sum
  float m[kGm];
#pragma unroll
  for (int jj = 0; jj < kGm; ++jj) {
    m[jj] = x[jj];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m[jj] = fmaxf(m[jj], __shfl_xor_sync(0xffffffffu, m[jj], o));
  }
  if (lane == 0) {
#pragma unroll
    for (int jj = 0; jj < kGm; ++jj) wmax[warp * kGm + jj] = m[jj];
  }
  __syncthreads();
  float l[kGm];
#pragma unroll
  for (int jj = 0; jj < kGm; ++jj) {
    float M = wmax[jj];
#pragma unroll
    for (int w = 1; w < kDecWarps; ++w) M = fmaxf(M, wmax[w * kGm + jj]);
    const float e = valid && jj < G ? exp2f(x[jj] - M) : 0.f;
    if (kmine < kSplitF) ps[kmine * kGm + jj] = make_float2(e, e);
    l[jj] = e;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l[jj] += __shfl_xor_sync(0xffffffffu, l[jj], o);
  }
  if (lane == 0) {
#pragma unroll
    for (int jj = 0; jj < kGm; ++jj) wsum[warp * kGm + jj] = l[jj];
  }
  tc::cp_async_wait<0>();
  __syncthreads();
  if (t < G) {
    float M = wmax[t], L = 0.f;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) {
      M = fmaxf(M, wmax[w * kGm + t]);
      L += wsum[w * kGm + t];
    }
    part_ml[(int64_t)unit * kGm + t] = make_float2(M, L);
  }
  // phase 3: O[jj][piece c] over key slice ks
  const int c = lane % C::PR, ks = warp * C::RW + lane / C::PR;
  float2 o[kGm][C::EPP / 2];
#pragma unroll
  for (int jj = 0; jj < kGm; ++jj)
#pragma unroll
    for (int e = 0; e < C::EPP / 2; ++e) o[jj][e] = make_float2(0.f, 0.f);
#pragma unroll 2
  for (int kk = ks; kk < nk; kk += C::KS) {
    const uint4 uv = *reinterpret_cast<const uint4*>(buf + (size_t)kk * C::RB + piece_slot(kk, c) * 16);
    float v[C::EPP];
    unpack(uv, (const T*)nullptr, v);
    const float4* prow = reinterpret_cast<const float4*>(ps + kk * kGm);
#pragma unroll
    for (int j2 = 0; j2 < kGm / 2; ++j2) {
      if (2 * j2 < G) {
        const float4 pp = prow[j2];
#pragma unroll
        for (int e = 0; e < C::EPP / 2; ++e) {
          const float2 ve = make_float2(v[2 * e], v[2 * e + 1]);
          o[2 * j2][e] = __ffma2_rn(ve, make_float2(pp.x, pp.y), o[2 * j2][e]);
          if (2 * j2 + 1 < G) o[2 * j2 + 1][e] = __ffma2_rn(ve, make_float2(pp.z, pp.w), o[2 * j2 + 1][e]);
        }
      }
    }
  }
  // rows of a warp, then warps, are added
#pragma unroll
  for (int jj = 0; jj < kGm; ++jj)
#pragma unroll
    for (int e = 0; e < C::EPP / 2; ++e)
#pragma unroll
      for (int sh = C::PR; sh < 32; sh <<= 1) {
        o[jj][e].x += __shfl_xor_sync(0xffffffffu, o[jj][e].x, sh);
        o[jj][e].y += __shfl_xor_sync(0xffffffffu, o[jj][e].y, sh);
      }
  __syncthreads();                              // V rows no longer read: warp partials
  float* wpart = reinterpret_cast<float*>(buf);  // [kDecWarps][kGm][D]
  if (lane < C::PR) {
#pragma unroll
    for (int jj = 0; jj < kGm; ++jj) {
      if (jj < G) {
        float4* dst = reinterpret_cast<float4*>(wpart + ((size_t)warp * kGm + jj) * D + c * C::EPP);
#pragma unroll
        for (int e = 0; e < C::EPP / 4; ++e)
          dst[e] = make_float4(o[jj][2 * e].x, o[jj][2 * e].y, o[jj][2 * e + 1].x, o[jj][2 * e + 1].y);
      }
    }
  }
  __syncthreads();
  for (int i = t; i < G * D; i += kDecThreads) {
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) sum += wpart[(size_t)w * kGm * D + i];
    part_o[(int64_t)unit * kGm * D + i] = sum;
  }
}

// ---------------------------------------------------------------------------
// bf16 caches: every warp streams tiles of 32 keys of its (request, KV head)
// on its own (no block barrier until the merge) through a ring of slots in
// shared memory, so the loads of the next items run under the current one's
// arithmetic.
//
// Both contractions are mma.sync m16n8k16 with the G <= 8 query heads as M:
// rows 0-7 carry the bf16 high parts of the query rows (then of the
// probabilities), rows 8-15 the low parts, so one instruction forms both
// products and their sum keeps ~16 mantissa bits (K and V are exact in
// bf16).  N is 8 keys (QK) or 8 output dimensions (PV).  The logits' C
// fragment is the probabilities' A fragment, so P never leaves registers.
// A k-step's four columns of a thread are four adjacent dimensions, half of
// a 16-byte piece of a K row: one 16-byte shared load serves two k-steps.
// Slots store piece c of row r at c ^ (r & 7), which makes those loads and
// ldmatrix (V) free of bank conflicts.
//
// The 4-bit form (Q4) keeps codes and parameters in the slots and expands
// them straight into B fragments: a thread's K columns as above; for PV a
// thread takes D / 8 adjacent dimensions of its keys, one per output tile
// (which dimension a tile's column stands for changes no sum).  The expanded
// values are fma(code, scale, min) rounded to bf16, the rows
// viscache_kv4_dequantize writes, and enter the same products in the same
// order, so the result equals the bf16 kernel's over those rows bit for bit.
//
// A cluster of C CTAs shares a pair: warp w of the cluster takes tiles w,
// w + 4 C, ..., each CTA merges its warps' (max, sum, output) states, sends
// every item of four outputs to the CTA that owns it through distributed
// shared memory, and after one cluster barrier the owners finish them.  No
// counters or partial outputs in global memory, one kernel a call, launched
// dependently (it waits for the previous kernel before it reads anything).
// Batches of very unequal requests (decode_plan.h) take the PARTS form: every CTA
// takes a part of a pair's tiles and leaves its state in the workspace, and
// decode_merge_kernel adds the parts up.
//
// Measured on a GB300 (28 layers as a graph, 7B shape, n = 12,544 at 19% + 512
// text rows; before: splits of 256 keys merged through global memory): one
// request 368 -> 145 us a step, 16 requests 790 -> 496 us (5.4 TB/s of 6.8),
// 4-bit cache of 16 requests 923 -> 528 us (556 with packed fp32 expansion).  A large
// layer runs at the memory rate (143 MB in 24 us) plus ~3 us that the launch, the
// first loads and the merge take; the 4-bit form is bound by instruction latency
// and issue (~1,400 warp instructions a tile, most of them the expansion, on two
// warps a scheduler; issue slots 45% busy).

constexpr int kWarps = kDecTileWarps;          // warps per CTA
constexpr int kMaxCluster = 16;                // CTAs per pair
constexpr float kRise = 8.f;                   // log2 units

template <int D, bool Q4>
struct TileCfg {
  static constexpr int RB = D * 2;                        // bytes of a bf16 row
  static constexpr int PR = RB / 16;                      // 16-byte pieces of a row
  static constexpr int KS = D / 16;                       // QK k-steps
  static constexpr int NT = D / 8;                        // output tiles of 8 dimensions
  static constexpr int ROWS = Q4 ? 16 : 32;               // bf16 rows of a ring slot
  static constexpr int PARTS = kTileKeys / ROWS;          // slots of a tile's K (or V) rows
  static constexpr int SLOT = ROWS * RB;
  static constexpr int SLOTS = 3 * PARTS;                 // slots of a warp's ring (24 KB at D = 128)
  static constexpr int RING = SLOTS * SLOT;
  static constexpr int ITEMS = kGm * D / 4;               // outputs of a pair, four adjacent ones an item
  // after the rings: the warps' (max, sum), the CTAs', and the CTAs' outputs of this CTA's items
  static constexpr int TAIL = (kWarps + kMaxCluster) * kGm * 8 + (ITEMS + kMaxCluster) * 16;
  static constexpr int SMEM = kWarps * RING + TAIL;
  static_assert(kGm * D * 4 <= RING, "a warp's output state fits its ring");
  // 4-bit items: codes [32][D / 2], then parameters (K: [D][2] floats, V: [32][D / 32][2])
  static constexpr int CODES = kTileKeys * D / 2;
  static_assert(CODES + D * 8 <= SLOT && CODES + kTileKeys * (D / 32) * 8 <= SLOT, "a 4-bit item fits a slot");
};

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t (&a)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp16_or_zero(uint32_t dst, const void* src, bool live) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(live ? 16u : 0u)
               : "memory");
}

// Place of 16-byte piece c of bf16 row r in a slot.
template <int D>
__device__ __forceinline__ uint32_t row_at(int r, int c) {
  return (uint32_t)(r * (D * 2) + ((c ^ (r & 7)) << 4));
}

// Rows [0, valid) of an item (contiguous rows at src) into a slot by the
// whole warp, zeros after them (finite values under the zero probabilities).
// `src` is read only where rows are valid.
template <int D, bool Q4>
__device__ __forceinline__ void load_rows(uint32_t slot, const __nv_bfloat16* src, int valid, int lane) {
  using C = TileCfg<D, Q4>;
  constexpr int RPI = 32 / C::PR;               // rows per warp instruction
  const int c = lane % C::PR, r0 = lane / C::PR;
  const __nv_bfloat16* p = src + lane * 8;
  if (valid >= C::ROWS) {
#pragma unroll
    for (int i = 0; i < C::ROWS / RPI; ++i) cp16(slot + row_at<D>(r0 + RPI * i, c), p + i * 256);
  } else {
#pragma unroll 2
    for (int i = 0; i < C::ROWS / RPI; ++i) {
      const int r = r0 + RPI * i;
      const bool live = r < valid;
      cp16_or_zero(slot + row_at<D>(r, c), live ? p + i * 256 : src, live);
    }
  }
}

// Places in a 4-bit item: byte b of code row r (D = 128: 16-byte pieces
// flipped by bit 1 of r), and 16-byte piece p of the key parameters (flipped
// by the thread that reads it); the value parameters lie in order.
template <int D>
__device__ __forceinline__ uint32_t code_at(int r, int b) {
  return (uint32_t)(r * (D / 2) + (D == 128 ? b ^ (((r >> 1) & 1) << 5) : b));
}
__device__ __forceinline__ uint32_t kpar_at(int p) { return (uint32_t)((p ^ ((p >> 3) & 7)) << 4); }

// `valid` rows of codes and `pars` 16-byte pieces of parameters.
template <int D>
__device__ __forceinline__ void load_q4(uint32_t slot, const uint8_t* codes, const void* par, int valid, int pars,
                                        bool keys, int lane) {
  constexpr int CP = D / 32;                    // 16-byte pieces of a code row
  const uint8_t* cl = codes + 16 * lane;
  const uint32_t dc = slot + code_at<D>(lane / CP, lane % CP * 16);
  const int nc = valid * CP - lane;
#pragma unroll
  for (int i = 0; i < CP; ++i)                  // 32 / CP rows each: the flip is the same
    cp16_or_zero(dc + i * 512, nc > 32 * i ? cl + 512 * i : codes, nc > 32 * i);
  const uint8_t* pp = static_cast<const uint8_t*>(par);
#pragma unroll
  for (int i = 0; i < D / 64; ++i) {
    const int p = lane + 32 * i;
    cp16_or_zero(slot + TileCfg<D, true>::CODES + (keys ? kpar_at(p) : (uint32_t)p << 4), p < pars ? pp + 16 * p : pp,
                 p < pars);
  }
}

// 2^23 + byte b of x as a float's bits (asm: as intrinsics the compiler turns
// most of these permutations into a shift and a logic operation).
__device__ __forceinline__ uint32_t magic_byte(uint32_t x, int b) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(0x4B000000u), "r"(0x7440 | b));
  return r;
}
// Byte b of x and of y as codes (exactly: 2^23 + code, minus 2^23), then
// fma(code, scale, lo) rounded to bf16.  Scalar: packed fp32 operations issue
// at a quarter of the rate.
__device__ __forceinline__ uint32_t expand_pair(uint32_t x, uint32_t y, int b, float sx, float sy, float lx, float ly) {
  const float cx = __fsub_rn(__uint_as_float(magic_byte(x, b)), 8388608.f);
  const float cy = __fsub_rn(__uint_as_float(magic_byte(y, b)), 8388608.f);
  return pack_bf16(fmaf(cx, sx, lx), fmaf(cy, sy, ly));
}

// Logits of the part h of a tile: s[n] += (Q high; Q low) K^T for the tile's
// keys 8 n ... 8 n + 7.  Piece j of a thread is 2 tig + (j & 1) + 8 (j / 2).
template <int D, bool Q4>
__device__ __forceinline__ void qk_rows(const uint8_t* slot, const uint32_t (&qa)[D / 16][4], float (&s)[4][4],
                                        int h, int gid, int tig) {
  using C = TileCfg<D, Q4>;
#pragma unroll
  for (int j = 0; j < C::KS / 2; ++j)
#pragma unroll
    for (int n = 0; n < C::ROWS / 8; ++n) {
      const uint4 u = *reinterpret_cast<const uint4*>(slot + row_at<D>(8 * n + gid, 2 * tig + (j & 1) + 8 * (j >> 1)));
      mma_bf16(s[C::ROWS / 8 * h + n], qa[2 * j], u.x, u.y);
      mma_bf16(s[C::ROWS / 8 * h + n], qa[2 * j + 1], u.z, u.w);
    }
}
template <int D>
__device__ __forceinline__ void qk_q4(const uint8_t* slot, const uint32_t (&qa)[D / 16][4], float (&s)[4][4],
                                      int gid, int tig) {
  using C = TileCfg<D, true>;
  const uint8_t* par = slot + C::CODES + 128 * tig;
#pragma unroll
  for (int j = 0; j < C::KS / 2; ++j) {
    float4 f[4];                                // (scale, minimum) of the piece's channels 2 i, 2 i + 1
    const int flip = 4 * ((j & 1) ^ (j >> 1));  // kpar_at(32 (j / 2) + 8 tig + 4 (j & 1) + i)
#pragma unroll
    for (int i = 0; i < 4; ++i)
      f[i] = *reinterpret_cast<const float4*>(par + 16 * (i ^ tig) + 512 * (j >> 1) + 16 * flip);
    const uint8_t* codes = slot + code_at<D>(gid, 32 * (j >> 1) + 8 * tig);
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const uint32_t w = *reinterpret_cast<const uint32_t*>(codes + n * 4 * D + 4 * (j & 1));
      const uint32_t a = w & 0x0f0f0f0fu, b = (w >> 4) & 0x0f0f0f0fu;
      uint32_t u[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) u[i] = expand_pair(a, b, i, f[i].x, f[i].z, f[i].y, f[i].w);
      mma_bf16(s[n], qa[2 * j], u[0], u[1]);
      mma_bf16(s[n], qa[2 * j + 1], u[2], u[3]);
    }
  }
}

// o[t] += (P high; P low) V for 16 keys, rows 16 h ... of the slot; column n
// of output tile t is dimension 8 t + n.
template <int D>
__device__ __forceinline__ void pv_rows(uint32_t slot, const uint32_t (&pa)[4], int h, float (&o)[D / 8][4], int lane) {
  const int r = 16 * h + (lane & 15), cs = lane >> 4;
#pragma unroll
  for (int c = 0; c < D / 8; c += 2) {
    uint32_t v[4];
    ldsm_x4_t(slot + row_at<D>(r, c + cs), v);
    mma_bf16(o[c], pa, v[0], v[1]);
    mma_bf16(o[c + 1], pa, v[2], v[3]);
  }
}
// The 4-bit kernel's columns: column n of tile t is dimension (D / 8) n + t.
template <int D>
__device__ __forceinline__ void pv_rows_q4(const uint8_t* slot, const uint32_t (&pa)[4], float (&o)[D / 8][4], int gid,
                                           int tig) {
#pragma unroll
  for (int c = 0; c < D / 64; ++c) {
    uint32_t w[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = 2 * tig + (i & 1) + (i >> 1) * 8;
      const uint4 u = *reinterpret_cast<const uint4*>(slot + row_at<D>(r, gid * (D / 64) + c));
      w[i][0] = u.x; w[i][1] = u.y; w[i][2] = u.z; w[i][3] = u.w;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      mma_bf16(o[8 * c + 2 * i], pa, __byte_perm(w[0][i], w[1][i], 0x5410), __byte_perm(w[2][i], w[3][i], 0x5410));
      mma_bf16(o[8 * c + 2 * i + 1], pa, __byte_perm(w[0][i], w[1][i], 0x7632),
               __byte_perm(w[2][i], w[3][i], 0x7632));
    }
  }
}
template <int D>
__device__ __forceinline__ void pv_q4(const uint8_t* slot, const uint32_t (&pa)[4], int h, float (&o)[D / 8][4],
                                      int gid, int tig) {
  using C = TileCfg<D, true>;
  constexpr int WPK = D / 64;                   // code words of a thread's D / 8 dimensions
  uint32_t w[4][WPK];                           // keys 2 tig, + 1, + 8, + 9 of the 16
  float2 pr[4];
  const uint8_t* codes = slot + code_at<D>(2 * tig, gid * (D / 16)) + h * 8 * D;
  const uint8_t* par = slot + C::CODES + tig * (D / 2) + gid * D / 256 * 8 + h * 4 * D;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = (i & 1) + (i >> 1) * 8;
    if constexpr (WPK == 2) {
      const uint2 u = *reinterpret_cast<const uint2*>(codes + r * (D / 2));
      w[i][0] = u.x;
      w[i][WPK - 1] = u.y;
    } else {
      w[i][0] = *reinterpret_cast<const uint32_t*>(codes + r * (D / 2));
    }
    pr[i] = *reinterpret_cast<const float2*>(par + r * (D / 4));
  }
  auto expand = [&](const uint32_t (&c)[4], int b, int k) {   // byte b of keys k, k + 1
    return expand_pair(c[k], c[k + 1], b, pr[k].x, pr[k + 1].x, pr[k].y, pr[k + 1].y);
  };
#pragma unroll
  for (int k = 0; k < WPK; ++k) {
    uint32_t a[4], b[4];                        // even and odd dimensions of the four keys
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      a[i] = w[i][k] & 0x0f0f0f0fu;
      b[i] = (w[i][k] >> 4) & 0x0f0f0f0fu;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      mma_bf16(o[8 * k + 2 * i], pa, expand(a, i, 0), expand(a, i, 2));
      mma_bf16(o[8 * k + 2 * i + 1], pa, expand(b, i, 0), expand(b, i, 2));
    }
  }
}

// Stores to another CTA of the cluster (address from map_to_rank).
__device__ __forceinline__ void st_cluster2(uint32_t addr, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void st_cluster4(uint32_t addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
               : "memory");
}

template <int D, bool Q4, bool PARTS>
__global__ void __launch_bounds__(32 * kWarps, 2) decode_tiles_kernel(
    const __grid_constant__ DecodeTable tb, int cluster_or_1, const __nv_bfloat16* __restrict__ q,
    const __nv_bfloat16* __restrict__ Kc, const __nv_bfloat16* __restrict__ Vc,
    const __nv_bfloat16* __restrict__ Kt, const __nv_bfloat16* __restrict__ Vt,
    const uint8_t* __restrict__ Kq, const uint8_t* __restrict__ Vq, const float* __restrict__ Kqp,
    const float* __restrict__ Vqp, __nv_bfloat16* __restrict__ out, float* __restrict__ part_o,
    float2* __restrict__ part_ml) {
  using C = TileCfg<D, Q4>;
  extern __shared__ __align__(128) uint8_t dsm[];
  const int cluster = PARTS ? 1 : cluster_or_1;
  const int warp = (int)threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gid = lane >> 2, tig = lane & 3;
  const int rank = (int)blockIdx.x % cluster, pair = (int)blockIdx.x / cluster;
  // PARTS: CTA u of a request's units is part u % nsplit of its pair u / nsplit
  const int r = PARTS ? find_req(tb, pair) : pair / tb.Hkv;
  const int nparts = PARTS ? tb.req[r].nsplit : 1, u = PARTS ? pair - tb.req[r].unit0 : pair % tb.Hkv;
  const int g = u / nparts, G = tb.G;
  const int B = tb.req[r].B, T = tb.req[r].T;
  const int64_t vis0 = tb.req[r].vis_row0 + (int64_t)g * B, txt0 = tb.req[r].txt_row0 + (int64_t)g * T;
  const int64_t kg0 = tb.req[r].kg0 + (int64_t)g * tb.req[r].nkg;
  const int nvt = (B + kTileKeys - 1) / kTileKeys, nt = nvt + (T + kTileKeys - 1) / kTileKeys;
  // this CTA's tiles [lo, hi)
  const int per = PARTS ? decode_tiles_per_part(nt, nparts) : nt;
  const int lo = PARTS ? u % nparts * per : 0, hi = PARTS ? min(nt, lo + per) : nt;
  const int first = lo + rank * kWarps + warp, step = cluster * kWarps;
  const int mine = hi > first ? (hi - first + step - 1) / step : 0;
  uint8_t* ring = dsm + warp * C::RING;
  const uint32_t ring_s = tc::smem_u32(ring);
  float2* ml = reinterpret_cast<float2*>(dsm + kWarps * C::RING);            // [warp][query] (max, sum)
  float2* cml = ml + kWarps * kGm;                                       // [CTA of the cluster][query]
  float4* cout = reinterpret_cast<float4*>(cml + kMaxCluster * kGm);        // [CTA][item of this CTA]
  if (cluster > 1) tc::cluster_arrive();        // met before the merge: every CTA has started

  dep_wait();                                   // queries and cache may be the previous kernel's output
  if (threadIdx.x == 0) dep_launch();

  // Ring items, a commit group each: a tile of bf16 rows is PARTS items of K
  // rows and as many of V rows, a 4-bit tile one of each (those come first).
  const int q4_end = min(nvt, hi);
  const int q4_tiles = Q4 && q4_end > first ? (q4_end - first + step - 1) / step : 0;
  auto issue = [&](int item, int slot) {
    const uint32_t dst = ring_s + slot * C::SLOT;
    if (Q4 && item < 2 * q4_tiles) {
      const int t = first + (item >> 1) * step;
      const int64_t row = vis0 + t * kTileKeys;
      const int valid = min(kTileKeys, B - t * kTileKeys);
      const bool v = item & 1;
      load_q4<D>(dst, (v ? Vq : Kq) + row * (D / 2), v ? Vqp + row * (D / 32) * 2 : Kqp + (kg0 + t) * D * 2, valid,
                 v ? valid * (D / 64) : D / 2, !v, lane);
    } else {
      const int e = item - 2 * q4_tiles, i = q4_tiles + e / (2 * C::PARTS);
      if (i < mine) {
        const int t = first + i * step;
        const bool text = Q4 || t >= nvt, v = e & C::PARTS;
        const int k0 = (text ? t - nvt : t) * kTileKeys + (e & (C::PARTS - 1)) * C::ROWS;
        const __nv_bfloat16* base = text ? (v ? Vt : Kt) : (v ? Vc : Kc);
        load_rows<D, Q4>(dst, base + ((text ? txt0 : vis0) + k0) * D, (text ? T : B) - k0, lane);
      }
    }
    tc::cp_async_commit();
  };
#pragma unroll 1
  for (int i = 0; i < C::SLOTS; ++i) issue(i, i);

  // A fragments of the query rows in log2 units: rows 0-7 high, 8-15 low parts
  uint32_t qa[C::KS][4];
  {
    const float c2 = tb.scale * kLog2eF;
    const __nv_bfloat16* qr = q + ((int64_t)r * tb.Hq + g * G + min(gid, G - 1)) * D + 16 * tig;
#pragma unroll
    for (int j = 0; j < C::KS / 2; ++j) {
      uint4 u = *reinterpret_cast<const uint4*>(qr + 64 * (j >> 1) + 8 * (j & 1));
      if (gid >= G) u = make_uint4(0u, 0u, 0u, 0u);
      const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float x0 = __uint_as_float(w[i] << 16) * c2, x1 = __uint_as_float(w[i] & 0xffff0000u) * c2;
        const float h0 = __bfloat162float(__float2bfloat16_rn(x0));
        const float h1 = __bfloat162float(__float2bfloat16_rn(x1));
        qa[2 * j + (i >> 1)][2 * (i & 1)] = pack_bf16(h0, h1);
        qa[2 * j + (i >> 1)][2 * (i & 1) + 1] = pack_bf16(x0 - h0, x1 - h1);
      }
    }
  }

  float m = -INFINITY, l = 0.f;                 // of query gid; l over this thread's keys
  float o[C::NT][4];
#pragma unroll
  for (int t = 0; t < C::NT; ++t)
#pragma unroll
    for (int i = 0; i < 4; ++i) o[t][i] = 0.f;
  int slot = 0, item = 0;                       // the oldest item and its slot
  auto refill = [&](int n) {                    // the n oldest items are read
    __syncwarp();
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
      issue(item + C::SLOTS, slot);
      ++item;
      slot = slot == C::SLOTS - 1 ? 0 : slot + 1;
    }
  };
  // softmax of a tile's logits (keys 8 n + 2 tig, + 1 of query gid): P as A fragments
  auto softmax = [&](const float (&s)[4][4], int valid, uint32_t (&pa)[2][4]) {
    float x[4][2], mt = -INFINITY;
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int e = 0; e < 2; ++e) x[n][e] = s[n][e] + s[n][2 + e];
    if (valid < kTileKeys) {
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (8 * n + 2 * tig + e >= valid) x[n][e] = -INFINITY;
    }
#pragma unroll
    for (int n = 0; n < 4; ++n) mt = tc::fmax3(mt, x[n][0], x[n][1]);
    mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 1));
    mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 2));
    // the reference rises only past 2^kRise times the terms it allows, so a
    // rescale of the outputs is rare; sums and products stay far below overflow
    const bool rise = mt > m + kRise;
    if (__any_sync(0xffffffffu, rise)) {
      const float corr = rise ? tc::ex2(m - mt) : 1.f;
      if (rise) m = mt;
      l *= corr;
#pragma unroll
      for (int k = 0; k < C::NT; ++k)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[k][e] *= corr;
    }
    const float mg = m == -INFINITY ? 0.f : m;  // no finite logit yet: every term is 0
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const float p0 = tc::ex2(x[n][0] - mg), p1 = tc::ex2(x[n][1] - mg);
      l += p0 + p1;
      const float h0 = __bfloat162float(__float2bfloat16_rn(p0)), h1 = __bfloat162float(__float2bfloat16_rn(p1));
      pa[n >> 1][2 * (n & 1)] = pack_bf16(h0, h1);
      pa[n >> 1][2 * (n & 1) + 1] = pack_bf16(p0 - h0, p1 - h1);
    }
  };
  if constexpr (Q4) {
#pragma unroll 1
    for (int i = 0; i < q4_tiles; ++i) {
      float s[4][4] = {};
      uint32_t pa[2][4];
      tc::cp_async_wait<C::SLOTS - 1>();
      __syncwarp();
      qk_q4<D>(ring + slot * C::SLOT, qa, s, gid, tig);
      refill(1);
      softmax(s, B - (first + i * step) * kTileKeys, pa);
      tc::cp_async_wait<C::SLOTS - 1>();
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; ++h) pv_q4<D>(ring + slot * C::SLOT, pa[h], h, o, gid, tig);
      refill(1);
    }
  }
#pragma unroll 1
  for (int i = q4_tiles; i < mine; ++i) {
    const int t = first + i * step;
    float s[4][4] = {};
    uint32_t pa[2][4];
    tc::cp_async_wait<C::SLOTS - 1>();
    __syncwarp();
    qk_rows<D, Q4>(ring + slot * C::SLOT, qa, s, 0, gid, tig);
    if constexpr (C::PARTS == 2) {
      tc::cp_async_wait<C::SLOTS - 2>();
      __syncwarp();
      qk_rows<D, Q4>(ring + (slot + 1) % C::SLOTS * C::SLOT, qa, s, 1, gid, tig);
    }
    refill(C::PARTS);
    softmax(s, t >= nvt ? T - (t - nvt) * kTileKeys : B - t * kTileKeys, pa);
    tc::cp_async_wait<C::SLOTS - 1>();
    __syncwarp();
    if constexpr (Q4) {
      pv_rows_q4<D>(ring + slot * C::SLOT, pa[0], o, gid, tig);
      tc::cp_async_wait<C::SLOTS - 2>();
      __syncwarp();
      pv_rows_q4<D>(ring + (slot + 1) % C::SLOTS * C::SLOT, pa[1], o, gid, tig);
    } else {
#pragma unroll
      for (int h = 0; h < 2; ++h) pv_rows<D>(ring_s + slot * C::SLOT, pa[h], h, o, lane);
    }
    refill(C::PARTS);
  }
  // this warp's state: (max, sum) and the unnormalised output [query][D] over its ring
  l += __shfl_xor_sync(0xffffffffu, l, 1);
  l += __shfl_xor_sync(0xffffffffu, l, 2);
  if (tig == 0) ml[warp * kGm + gid] = make_float2(m, l);
  {
    float* po = reinterpret_cast<float*>(ring) + gid * D;
    if constexpr (Q4) {
#pragma unroll
      for (int t = 0; t < C::NT; t += 4)
#pragma unroll
        for (int e = 0; e < 2; ++e)
          *reinterpret_cast<float4*>(po + (D / 8) * (2 * tig + e) + t) =
              make_float4(o[t][e] + o[t][2 + e], o[t + 1][e] + o[t + 1][2 + e], o[t + 2][e] + o[t + 2][2 + e],
                          o[t + 3][e] + o[t + 3][2 + e]);
    } else {
#pragma unroll
      for (int t = 0; t < C::NT; ++t)
        *reinterpret_cast<float2*>(po + 8 * t + 2 * tig) = make_float2(o[t][0] + o[t][2], o[t][1] + o[t][3]);
    }
  }
  __syncthreads();
  // Merge.  The CTA's warps first, four adjacent outputs an item: with one CTA
  // that is the result; else each item goes to the CTA that owns it (CTA c
  // owns `own` items from c own), and the (max, sum) to every CTA.
  const int own = (C::ITEMS + cluster - 1) / cluster;
  auto store = [&](int item, float4 v, float M, float L) {
    // no keys: zeros; keys without a finite logit: no softmax
    const float f = L > 0.f ? 1.f / L : M == -INFINITY && nt > 0 ? NAN : 0.f;
    const int jj = item / (D / 4), d0 = item % (D / 4) * 4;
    *reinterpret_cast<uint2*>(out + ((int64_t)r * tb.Hq + g * G + jj) * D + d0) =
        make_uint2(pack_bf16(v.x * f, v.y * f), pack_bf16(v.z * f, v.w * f));
  };
  auto fold = [](float4& acc, float& L, float4 v, float2 st, float M) {
    const float w = st.x == -INFINITY ? 0.f : tc::ex2(st.x - M);
    L = fmaf(st.y, w, L);
    acc.x = fmaf(v.x, w, acc.x);
    acc.y = fmaf(v.y, w, acc.y);
    acc.z = fmaf(v.z, w, acc.z);
    acc.w = fmaf(v.w, w, acc.w);
  };
  if (cluster > 1) tc::cluster_wait();
#pragma unroll 1
  for (int item = threadIdx.x; item < G * (D / 4); item += 32 * kWarps) {
    const int jj = item / (D / 4), d4 = item % (D / 4);
    float M = -INFINITY, L = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) M = fmaxf(M, ml[w * kGm + jj].x);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < kWarps; ++w)
      fold(acc, L, *reinterpret_cast<const float4*>(dsm + w * C::RING + item * 16), ml[w * kGm + jj], M);
    if (PARTS) {
      *reinterpret_cast<float4*>(part_o + (int64_t)pair * kGm * D + item * 4) = acc;
      if (d4 == 0) part_ml[(int64_t)pair * kGm + jj] = make_float2(M, L);
    } else if (cluster == 1) {
      store(item, acc, M, L);
    } else {
      st_cluster4(tc::map_to_rank(tc::smem_u32(cout + rank * own + item % own), item / own), acc);
      if (d4 < cluster) st_cluster2(tc::map_to_rank(tc::smem_u32(cml + rank * kGm + jj), d4), make_float2(M, L));
    }
  }
  if (cluster == 1) return;
  __syncwarp();
  tc::cluster_sync();                           // the cluster's states have arrived; nothing remote after it
  for (int i = threadIdx.x; i < own; i += 32 * kWarps) {
    const int item = rank * own + i, jj = item / (D / 4);
    if (jj >= G) break;
    float M = -INFINITY, L = 0.f;
    for (int c = 0; c < cluster; ++c) M = fmaxf(M, cml[c * kGm + jj].x);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int c = 0; c < cluster; ++c) fold(acc, L, cout[c * own + i], cml[c * kGm + jj], M);
    store(item, acc, M, L);
  }
}

// One warp per (request, query head): merge the splits of its KV head.  Lane
// s holds split s's state (s = lane, lane + 32, ...); the weighted partial
// outputs are then summed with several splits' loads in flight.
template <typename T, int D>
__global__ void __launch_bounds__(128) decode_combine_kernel(const __grid_constant__ DecodeTable tb,
                                                             const float* __restrict__ part_o,
                                                             const float2* __restrict__ part_ml,
                                                             T* __restrict__ out) {
  constexpr int EPL = D / 32;                   // output elements per lane
  const int w = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (w >= tb.n_req * tb.Hq) return;
  const int r = w / tb.Hq, j = w % tb.Hq;
  const DecodeReq rq = tb.req[r];
  const int g = j / tb.G, jj = j % tb.G;
  const int64_t u0 = rq.unit0 + (int64_t)g * rq.nsplit;
  const int ns = rq.B + rq.T > 0 ? rq.nsplit : 0;
  float M = -INFINITY;
  for (int s = lane; s < ns; s += 32) M = fmaxf(M, part_ml[(u0 + s) * kGm + jj].x);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  float Lsum = 0.f;
  float acc[EPL];
#pragma unroll
  for (int i = 0; i < EPL; ++i) acc[i] = 0.f;
  for (int s0 = 0; s0 < ns; s0 += 32) {
    const int sl = s0 + lane;
    float wl = 0.f;
    if (sl < ns) {
      const float2 ml = part_ml[(u0 + sl) * kGm + jj];
      wl = exp2f(ml.x - M);
      Lsum = fmaf(ml.y, wl, Lsum);
    }
    const int cnt = min(32, ns - s0);
#pragma unroll 4
    for (int i = 0; i < cnt; ++i) {
      const float ws = __shfl_sync(0xffffffffu, wl, i);
      const float* o = part_o + ((u0 + s0 + i) * kGm + jj) * D + lane * EPL;
      if constexpr (EPL == 4) {
        const float4 v = *reinterpret_cast<const float4*>(o);
        acc[0] = fmaf(v.x, ws, acc[0]);
        acc[1] = fmaf(v.y, ws, acc[1]);
        acc[2] = fmaf(v.z, ws, acc[2]);
        acc[3] = fmaf(v.w, ws, acc[3]);
      } else {
        const float2 v = *reinterpret_cast<const float2*>(o);
        acc[0] = fmaf(v.x, ws, acc[0]);
        acc[1] = fmaf(v.y, ws, acc[1]);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) Lsum += __shfl_xor_sync(0xffffffffu, Lsum, o);
  const float inv = Lsum > 0.f ? 1.f / Lsum : 0.f;
  T* dst = out + ((int64_t)r * tb.Hq + j) * D + lane * EPL;
#pragma unroll
  for (int i = 0; i < EPL; ++i) dst[i] = Elem<T>::from_f(acc[i] * inv);
}

// One CTA per (request, query head): merge the parts of its KV head.  Warp w
// sums parts w, w + 4, ... with eight parts' loads in flight; the four sums are
// added in order.  (1,024 parts a pair took 380 us on a warp with four in flight.)
constexpr int kMergeWarps = 4;
template <int D>
__global__ void __launch_bounds__(32 * kMergeWarps) decode_merge_kernel(const __grid_constant__ DecodeTable tb,
                                                                        const float* __restrict__ part_o,
                                                                        const float2* __restrict__ part_ml,
                                                                        __nv_bfloat16* __restrict__ out) {
  constexpr int EPL = D / 32;                   // output elements per lane
  __shared__ float wmax[kMergeWarps], wsum[kMergeWarps], wo[kMergeWarps][D];
  dep_wait();                                   // the parts' states
  if (threadIdx.x == 0) dep_launch();
  const int warp = (int)threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = (int)blockIdx.x / tb.Hq, j = (int)blockIdx.x % tb.Hq, g = j / tb.G, jj = j % tb.G;
  const int ns = tb.req[r].B + tb.req[r].T > 0 ? tb.req[r].nsplit : 0;
  const int64_t u0 = tb.req[r].unit0 + (int64_t)g * tb.req[r].nsplit;
  const float2* ml = part_ml + u0 * kGm + jj;
  const float* po = part_o + (u0 * kGm + jj) * D + lane * EPL;
  float M = -INFINITY;
  for (int s = threadIdx.x; s < ns; s += 32 * kMergeWarps) M = fmaxf(M, ml[(int64_t)s * kGm].x);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  if (lane == 0) wmax[warp] = M;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kMergeWarps; ++w) M = fmaxf(M, wmax[w]);
  float L = 0.f, acc[EPL] = {};
#pragma unroll 8
  for (int s = warp; s < ns; s += kMergeWarps) {
    const float2 st = ml[(int64_t)s * kGm];
    const float wt = exp2f(st.x - M);           // no part with a finite logit: NaN, as the softmax
    L = fmaf(st.y, wt, L);
    const float* o = po + (int64_t)s * kGm * D;
    if constexpr (EPL == 4) {
      const float4 v = *reinterpret_cast<const float4*>(o);
      acc[0] = fmaf(v.x, wt, acc[0]);
      acc[1] = fmaf(v.y, wt, acc[1]);
      acc[EPL - 2] = fmaf(v.z, wt, acc[EPL - 2]);
      acc[EPL - 1] = fmaf(v.w, wt, acc[EPL - 1]);
    } else {
      const float2 v = *reinterpret_cast<const float2*>(o);
      acc[0] = fmaf(v.x, wt, acc[0]);
      acc[1] = fmaf(v.y, wt, acc[1]);
    }
  }
#pragma unroll
  for (int i = 0; i < EPL; ++i) wo[warp][lane * EPL + i] = acc[i];
  if (lane == 0) wsum[warp] = L;
  __syncthreads();
  for (int d = threadIdx.x; d < D; d += 32 * kMergeWarps) {
    float sum = 0.f, total = 0.f;
#pragma unroll
    for (int w = 0; w < kMergeWarps; ++w) {
      sum += wo[w][d];
      total += wsum[w];
    }
    const float inv = total > 0.f ? 1.f / total : 0.f;
    out[((int64_t)r * tb.Hq + j) * D + d] = __float2bfloat16_rn(sum * inv);
  }
}

template <typename T, int D>
cudaError_t launch_decode_t(const DecodeTable& tb, const void* q, const void* Kc, const void* Vc,
                            const void* Kt, const void* Vt, void* out, float* part_o, float2* part_ml,
                            cudaStream_t st) {
  if (tb.units > 0) {
    constexpr size_t smem = DecCfg<T, D>::SMEM;
    static bool attr = false;
    if (!attr) {
      cudaError_t e = cudaFuncSetAttribute(decode_partial_kernel<T, D>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      // the whole unified L1 as shared memory: a d = 64 CTA is 87 KB, two an SM
      e = cudaFuncSetAttribute(decode_partial_kernel<T, D>,
                               cudaFuncAttributePreferredSharedMemoryCarveout, 100);
      if (e != cudaSuccess) return e;
      attr = true;
    }
    ProfileScope ps("decode_partial", st);
    decode_partial_kernel<T, D><<<(unsigned)tb.units, kDecThreads, smem, st>>>(
        tb, static_cast<const T*>(q), static_cast<const T*>(Kc), static_cast<const T*>(Vc),
        static_cast<const T*>(Kt), static_cast<const T*>(Vt), part_o, part_ml);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  ProfileScope ps("decode_combine", st);
  const int warps = tb.n_req * tb.Hq;
  decode_combine_kernel<T, D><<<(unsigned)((warps + 3) / 4), 128, 0, st>>>(tb, part_o, part_ml,
                                                                          static_cast<T*>(out));
  return cudaGetLastError();
}

template <int D, bool Q4, bool PARTS>
cudaError_t prepare_decode_tiles() {
  auto kernel = decode_tiles_kernel<D, Q4, PARTS>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TileCfg<D, Q4>::SMEM);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  // the whole unified L1 as shared memory: two CTAs per SM
  return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
}

// Prepares the forms of the kernel on the current device at its first call
// and returns what fits (the same for all: one shared-memory size).
template <int D>
cudaError_t decode_fit(DecodeFit* fit) {
  static_assert(TileCfg<D, false>::SMEM == TileCfg<D, true>::SMEM, "both forms occupy an SM alike");
  static bool known[64];
  static DecodeFit fits[64];
  static std::mutex guard;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> hold(guard);
  if (!known[dev]) {
    e = prepare_decode_tiles<D, false, false>();
    if (e == cudaSuccess) e = prepare_decode_tiles<D, true, false>();
    if (e == cudaSuccess) e = prepare_decode_tiles<D, false, true>();
    if (e == cudaSuccess) e = prepare_decode_tiles<D, true, true>();
    if (e != cudaSuccess) return e;
    for (int k = 0; k < kClusterKinds; ++k) {
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = (unsigned)kClusterSizes[k];
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)kClusterSizes[k], 1, 1);
      cfg.blockDim = dim3(32 * kWarps, 1, 1);
      cfg.dynamicSmemBytes = TileCfg<D, false>::SMEM;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&fits[dev].n[k], decode_tiles_kernel<D, false, false>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        fits[dev].n[k] = 0;
      }
    }
    known[dev] = true;
  }
  *fit = fits[dev];
  return cudaSuccess;
}

// The 4-bit form takes the same clusters and parts as the bf16 form, so that its
// tiles are split and merged alike.
template <int D, bool Q4>
cudaError_t launch_decode_tiles(const DecodeTable& tb, const void* q, const void* Kc, const void* Vc,
                                const void* Kt, const void* Vt, const uint8_t* Kq, const uint8_t* Vq,
                                const float* Kqp, const float* Vqp, void* out, float* part_o, float2* part_ml,
                                cudaStream_t st) {
  using B16 = __nv_bfloat16;
  if (tb.n_req < 1) return cudaSuccess;
  DecodeFit fit;
  cudaError_t e = decode_fit<D>(&fit);
  if (e != cudaSuccess) return e;
  int64_t tiles[kDecodeMaxReq];
  for (int r = 0; r < tb.n_req; ++r) tiles[r] = decode_tiles(tb.req[r].B, tb.req[r].T);
  const DecodePlan plan = plan_decode(tiles, tb.n_req, tb.Hkv, fit);
  auto launch = [&](auto in_parts, const DecodeTable& table, int ctas) {
    ProfileScope ps(Q4 ? "decode_attn_kv4" : "decode_attn", st);
    return launch_dep_clusters(decode_tiles_kernel<D, Q4, decltype(in_parts)::value>, dim3((unsigned)ctas),
                               dim3(32 * kWarps), (size_t)TileCfg<D, Q4>::SMEM, plan.cluster, st, table, plan.cluster,
                               static_cast<const B16*>(q), static_cast<const B16*>(Kc), static_cast<const B16*>(Vc),
                               static_cast<const B16*>(Kt), static_cast<const B16*>(Vt), Kq, Vq, Kqp, Vqp,
                               static_cast<B16*>(out), part_o, part_ml);
  };
  if (plan.part_tiles == 0)
    return launch(std::false_type{}, tb, tb.n_req * tb.Hkv * plan.cluster);
  // the table's units become the parts: one for every kPartMin * kWarps tiles at
  // most, so never more than the 256-key splits the workspace is sized for
  static_assert(kPartMin * kWarps * kTileKeys >= 2 * kSplitF, "the parts' states fit the workspace of the splits");
  DecodeTable parts = tb;
  parts.units = 0;
  for (int r = 0; r < tb.n_req; ++r) {
    parts.req[r].unit0 = parts.units;
    parts.req[r].nsplit = decode_parts(tiles[r], plan.part_tiles);
    parts.units += tb.Hkv * parts.req[r].nsplit;
  }
  e = launch(std::true_type{}, parts, parts.units);
  if (e != cudaSuccess) return e;
  ProfileScope ps("decode_merge", st);
  return launch_dep(decode_merge_kernel<D>, dim3((unsigned)(tb.n_req * tb.Hq)), dim3(32 * kMergeWarps), 0, st, parts,
                    static_cast<const float*>(part_o), static_cast<const float2*>(part_ml), static_cast<B16*>(out));
}

}  // namespace

int decode_split_keys() { return kSplitF; }

cudaError_t launch_decode(const DecodeTable& tb, int dtype, int d, const void* q, const void* Kc,
                          const void* Vc, const void* Kt, const void* Vt, void* out, float* part_o,
                          float2* part_ml, cudaStream_t st) {
  if (dtype == VC_BF16) {
    if (d == 128)
      return launch_decode_tiles<128, false>(tb, q, Kc, Vc, Kt, Vt, nullptr, nullptr, nullptr, nullptr, out, part_o,
                                            part_ml, st);
    return launch_decode_tiles<64, false>(tb, q, Kc, Vc, Kt, Vt, nullptr, nullptr, nullptr, nullptr, out, part_o,
                                            part_ml, st);
  }
  if (d == 128) return launch_decode_t<float, 128>(tb, q, Kc, Vc, Kt, Vt, out, part_o, part_ml, st);
  return launch_decode_t<float, 64>(tb, q, Kc, Vc, Kt, Vt, out, part_o, part_ml, st);
}

cudaError_t launch_decode_kv4(const DecodeTable& tb, int d, const void* q, const uint8_t* Kq,
                              const uint8_t* Vq, const float* Kqp, const float* Vqp, const void* Kt,
                              const void* Vt, void* out, float* part_o, float2* part_ml, cudaStream_t st) {
  if (d == 128)
    return launch_decode_tiles<128, true>(tb, q, nullptr, nullptr, Kt, Vt, Kq, Vq, Kqp, Vqp, out, part_o, part_ml, st);
  return launch_decode_tiles<64, true>(tb, q, nullptr, nullptr, Kt, Vt, Kq, Vq, Kqp, Vqp, out, part_o, part_ml, st);
}

}  // namespace vc

// 4-bit quantisation of the compacted cache (the Appendix "Quantization"
// combination: the compressed visual KV under a 4-bit KV cache quantiser) and
// its inverse.  Asymmetric round-to-nearest with a per-group scale and
// minimum:
//     scale = (max - min) / 15,  code = clamp(rint((x - min) / scale), 0, 15),
//     x_hat = code * scale + min  (one fused multiply-add),
// keys per channel over groups of 32 consecutive rows of one (request, layer,
// KV head) segment (the last group of a segment may be shorter), values per
// row over groups of 32 channels.  Codes are packed two per byte, the even
// channel in the low nibble; parameters are fp32 (scale, min) pairs.  The
// code is decided in fp32 with IEEE subtraction and division and rint.
//
// One warp per key group (up to 32 rows of one segment).  The work is a
// streaming pass (read 2 x 2 bytes, write 2 x ~0.75 bytes per element pair).
#include <cuda_bf16.h>
#include <stdint.h>

#include <type_traits>

#include "kernels.h"
#include "profile.h"
#include "vc_common.cuh"

namespace vc {
namespace {

constexpr int kGroup = 32;
constexpr int kQuantWarps = 4;                // key groups (one per warp) per CTA

__device__ __forceinline__ int find_entry(const QuantTable& tb, int unit) {
  int lo = 0, hi = tb.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tb.e[mid].unit0 <= unit) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// rint((x - lo) / scale) with an IEEE quotient, clamped to [0, 15]; inv is
// the correctly rounded 1 / scale.  t = (x - lo) * inv is within 1.5 ulp of
// the exact quotient (the IEEE quotient within 0.5 ulp), so for |t| <= 16
// both lie within 4e-6 of it: unless t is within 1e-5 of a half-integer
// they round to the same integer, and only then is the division done.
__device__ __forceinline__ uint32_t code_of(float x, float lo, float scale, float inv) {
  if (!(scale > 0.f)) return 0u;
  const float a = __fsub_rn(x, lo);
  float t = __fmul_rn(a, inv);
  if (fabsf(t - floorf(t) - 0.5f) < 1e-5f || !(fabsf(t) <= 16.f)) t = __fdiv_rn(a, scale);
  return (uint32_t)fminf(fmaxf(rintf(t), 0.f), 15.f);
}

// The same decision without branches.  With inv the correctly rounded 1 / scale,
// t0 = (x - lo) inv, rem = (x - lo) - t0 scale (exact) and t = t0 + rem inv, t is
// the IEEE quotient (Markstein, "Computation of elementary functions on the IBM
// RISC System/6000 processor", 1990), and t + 1.5 * 2^23 holds rint(t) in its low
// bits.  The group must be regular: scale 0 (every t is 0) or finite and at least
// 2^-96, which keeps rem clear of underflow; then 0 <= t < 15.5 for every number
// of the group.  A NaN gives the low bits 0xffff.
constexpr float kRound = 12582912.f;                 // 1.5 * 2^23
__device__ __forceinline__ bool regular_scale(float scale) {
  return scale == 0.f || (scale >= 1.2621774e-29f && scale < INFINITY);
}
__device__ __forceinline__ uint32_t code_bits(float x, float lo, float scale, float inv) {
  const float a = __fsub_rn(x, lo), t0 = __fmul_rn(a, inv);
  return __float_as_uint(__fadd_rn(__fmaf_rn(__fmaf_rn(-t0, scale, a), inv, t0), kRound));
}

// Codes r0[0 .. N) in nibbles 0 .. N-1 and r1[0 .. N) in nibbles 4 .. 3 + N of
// the result; seen collects the bits of all, for any_nan.
template <int N>
__device__ __forceinline__ uint32_t pack_codes(const uint32_t (&r0)[N], const uint32_t (&r1)[N], uint32_t& seen) {
  uint32_t s = 0;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const uint32_t w = __byte_perm(r0[j], r1[j], 0x5410);
    seen |= w;
    s += w << (4 * j);
  }
  return s;
}
__device__ __forceinline__ bool any_nan(uint32_t seen) { return (seen & 0xfff0fff0u) != 0; }

// Elementwise minimum and maximum of bf16 pairs (exact: no rounding).
__device__ __forceinline__ __nv_bfloat162 as_bf162(uint32_t u) {
  return *reinterpret_cast<const __nv_bfloat162*>(&u);
}

struct GroupRows {
  int64_t row;   // first row of the key group
  int nrows;     // rows in the group (1..32)
  int64_t kg;    // global index of the key group (its parameter row)
};
__device__ __forceinline__ GroupRows group_rows(const QuantTable& tb, int unit) {
  const QuantEntry e = tb.e[find_entry(tb, unit)];
  const int local = unit - e.unit0;
  const int nb = (e.B + kGroup - 1) / kGroup;
  const int g = local / nb, b = local % nb;
  GroupRows x;
  x.row = e.row0 + (int64_t)g * e.B + (int64_t)b * kGroup;
  x.nrows = min(kGroup, e.B - b * kGroup);
  x.kg = tb.unit_base + unit;
  return x;
}

// CPT adjacent channels of one row as floats (CPT = 2 or 4; 4 or 8 bf16 bytes,
// 8 or 16 fp32 bytes).
template <typename T, int CPT>
__device__ __forceinline__ void load_cpt(const T* p, float (&v)[CPT]);
template <>
__device__ __forceinline__ void load_cpt<__nv_bfloat16, 4>(const __nv_bfloat16* p, float (&v)[4]) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  v[0] = __uint_as_float(u.x << 16); v[1] = __uint_as_float(u.x & 0xffff0000u);
  v[2] = __uint_as_float(u.y << 16); v[3] = __uint_as_float(u.y & 0xffff0000u);
}
template <>
__device__ __forceinline__ void load_cpt<__nv_bfloat16, 2>(const __nv_bfloat16* p, float (&v)[2]) {
  const uint32_t u = *reinterpret_cast<const uint32_t*>(p);
  v[0] = __uint_as_float(u << 16); v[1] = __uint_as_float(u & 0xffff0000u);
}
template <>
__device__ __forceinline__ void load_cpt<float, 4>(const float* p, float (&v)[4]) {
  const float4 u = *reinterpret_cast<const float4*>(p);
  v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w;
}
template <>
__device__ __forceinline__ void load_cpt<float, 2>(const float* p, float (&v)[2]) {
  const float2 u = *reinterpret_cast<const float2*>(p);
  v[0] = u.x; v[1] = u.y;
}

// One warp per key group.  Keys: lane t owns channels CPT t .. CPT t + CPT - 1
// of the group's rows; bf16 rows are read once and stay in registers between
// the minimum and maximum of each channel and the codes (fp32 rows are read
// again, from cache).  Rows past a short group repeat its last one, and are not
// stored.  Values: each lane takes whole (row, 32-channel group) pairs.  Groups
// with a NaN, an infinity or a scale below 2^-96 go through code_of.
// Bound by HBM.  At 16 requests of 3,136 tokens (28 layers, bf16; 3.0 GB) the
// whole call took 981 us when the codes' branches and a second read of the rows
// kept the issue slots busy at 45% of the copy rate, and takes 484 us now
// (92% of the copy rate).
// BYTES: code arrays of any alignment, stored byte by byte (a word of 2 or 16
// bytes otherwise).
template <typename T, int D, bool BYTES>
__global__ void __launch_bounds__(kQuantWarps * 32) quant_kernel(
    const __grid_constant__ QuantTable tb, int units, const T* __restrict__ K, const T* __restrict__ V,
    uint8_t* __restrict__ Kc, uint8_t* __restrict__ Vc, float2* __restrict__ Kp, float2* __restrict__ Vp) {
  constexpr int CPT = D / 32;
  const int unit = blockIdx.x * kQuantWarps + (threadIdx.x >> 5);
  if (unit >= units) return;
  const int lane = threadIdx.x & 31, c0 = lane * CPT;
  const GroupRows gr = group_rows(tb, unit);
  const T* kp = K + gr.row * D + c0;
  constexpr bool kBf16 = std::is_same<T, __nv_bfloat16>::value;
  constexpr int kHeld = kBf16 ? kGroup : 1, kHalf = CPT / 2;
  uint32_t held[kHeld][kHalf];                 // the lane's pieces of the rows, as bf16 pairs
  float mn[CPT], mx[CPT];
  if constexpr (kBf16) {
#pragma unroll
    for (int i = 0; i < kGroup; ++i) {
      const T* p = kp + min(i, gr.nrows - 1) * D;
      if constexpr (CPT == 4) {
        const uint2 u = *reinterpret_cast<const uint2*>(p);
        held[i][0] = u.x;
        held[i][kHalf - 1] = u.y;
      } else {
        held[i][0] = *reinterpret_cast<const uint32_t*>(p);
      }
    }
#pragma unroll
    for (int j = 0; j < kHalf; ++j) {
      __nv_bfloat162 lo2 = __floats2bfloat162_rn(INFINITY, INFINITY), hi2 = __floats2bfloat162_rn(-INFINITY, -INFINITY);
#pragma unroll
      for (int i = 0; i < kGroup; ++i) {
        lo2 = __hmin2(lo2, as_bf162(held[i][j]));
        hi2 = __hmax2(hi2, as_bf162(held[i][j]));
      }
      const float2 l = __bfloat1622float2(lo2), h = __bfloat1622float2(hi2);
      mn[2 * j] = l.x;
      mn[2 * j + 1] = l.y;
      mx[2 * j] = h.x;
      mx[2 * j + 1] = h.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
      mn[j] = INFINITY;
      mx[j] = -INFINITY;
    }
#pragma unroll 8
    for (int i = 0; i < gr.nrows; ++i) {
      float v[CPT];
      load_cpt<T, CPT>(kp + i * D, v);
#pragma unroll
      for (int j = 0; j < CPT; ++j) {
        mn[j] = fminf(mn[j], v[j]);
        mx[j] = fmaxf(mx[j], v[j]);
      }
    }
  }
  float ks[CPT], ki[CPT];
  bool plain = true;                           // every group of the lane is regular
#pragma unroll
  for (int j = 0; j < CPT; ++j) {
    ks[j] = __fdiv_rn(__fsub_rn(mx[j], mn[j]), 15.f);
    ki[j] = ks[j] > 0.f ? __frcp_rn(ks[j]) : 0.f;
    plain = plain && regular_scale(ks[j]);
    Kp[gr.kg * D + c0 + j] = make_float2(ks[j], mn[j]);
  }
  uint8_t* kc = Kc + gr.row * (D / 2) + c0 / 2;
  auto store_row = [&](int i, uint32_t q) {    // the lane's CPT codes of a row
    if (i >= gr.nrows) return;
    if constexpr (CPT == 4 && !BYTES) {
      *reinterpret_cast<uint16_t*>(kc + i * (D / 2)) = (uint16_t)q;
    } else {
      kc[i * (D / 2)] = (uint8_t)q;
      if constexpr (CPT == 4) kc[i * (D / 2) + 1] = (uint8_t)(q >> 8);
    }
  };
  uint32_t seen = 0;
#pragma unroll
  for (int i = 0; i < kGroup; i += 2) {
    float x[2][CPT];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if constexpr (kBf16) {
#pragma unroll
        for (int j = 0; j < kHalf; ++j) {
          x[u][2 * j] = __uint_as_float(held[i + u][j] << 16);
          x[u][2 * j + 1] = __uint_as_float(held[i + u][j] & 0xffff0000u);
        }
      } else {
        load_cpt<T, CPT>(kp + min(i + u, gr.nrows - 1) * D, x[u]);
      }
    }
    uint32_t r0[CPT], r1[CPT];
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
      r0[j] = code_bits(x[0][j], mn[j], ks[j], ki[j]);
      r1[j] = code_bits(x[1][j], mn[j], ks[j], ki[j]);
    }
    const uint32_t s = pack_codes<CPT>(r0, r1, seen);
    store_row(i, s & 0xffffu);
    store_row(i + 1, s >> 16);
  }
  if (!plain || any_nan(seen)) {
    for (int i = 0; i < gr.nrows; ++i) {
      float v[CPT];
      load_cpt<T, CPT>(kp + i * D, v);
      uint32_t q = 0;
#pragma unroll
      for (int j = 0; j < CPT; ++j) q |= code_of(v[j], mn[j], ks[j], ki[j]) << (4 * j);
      store_row(i, q);
    }
  }
  // values: lane (row i, 32-channel group gv) takes the group whole (NG groups
  // a row, 32 / NG rows a pass): 16-byte loads, its own minimum and maximum,
  // 16 bytes of codes
  constexpr int NG = D / kGroup, RPP = 32 / NG;
  const int gv = lane % NG;
  for (int i = lane / NG; i < gr.nrows; i += RPP) {
    float v[kGroup];
    const T* src = V + (gr.row + i) * D + gv * kGroup;
    float lo, hi;
    if constexpr (kBf16) {
      // the group's 32 values as 16 bf16 pairs: minimum and maximum on pairs
      uint32_t w[kGroup / 2];
#pragma unroll
      for (int k = 0; k < kGroup / 2; k += 4) {
        const uint4 u = *reinterpret_cast<const uint4*>(src + 2 * k);
        w[k] = u.x; w[k + 1] = u.y; w[k + 2] = u.z; w[k + 3] = u.w;
      }
      __nv_bfloat162 l2 = as_bf162(w[0]), h2 = as_bf162(w[0]);
#pragma unroll
      for (int k = 1; k < kGroup / 2; ++k) {
        l2 = __hmin2(l2, as_bf162(w[k]));
        h2 = __hmax2(h2, as_bf162(w[k]));
      }
      const float2 lf = __bfloat1622float2(l2), hf = __bfloat1622float2(h2);
      lo = fminf(lf.x, lf.y);
      hi = fmaxf(hf.x, hf.y);
#pragma unroll
      for (int k = 0; k < kGroup / 2; ++k) {
        v[2 * k] = __uint_as_float(w[k] << 16);
        v[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
      }
    } else {
#pragma unroll
      for (int k = 0; k < kGroup; k += CPT) {
        float u[CPT];
        load_cpt<T, CPT>(src + k, u);
#pragma unroll
        for (int j = 0; j < CPT; ++j) v[k + j] = u[j];
      }
      lo = v[0];
      hi = v[0];
#pragma unroll
      for (int k = 1; k < kGroup; ++k) {
        lo = fminf(lo, v[k]);
        hi = fmaxf(hi, v[k]);
      }
    }
    const float vs = __fdiv_rn(__fsub_rn(hi, lo), 15.f);
    const float vi = vs > 0.f ? __frcp_rn(vs) : 0.f;
    Vp[(gr.row + i) * NG + gv] = make_float2(vs, lo);
    uint32_t w[4];
    seen = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      uint32_t r0[4], r1[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        r0[k] = code_bits(v[8 * b + k], lo, vs, vi);
        r1[k] = code_bits(v[8 * b + 4 + k], lo, vs, vi);
      }
      w[b] = pack_codes<4>(r0, r1, seen);
    }
    if (!regular_scale(vs) || any_nan(seen)) {
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        w[b] = 0u;
#pragma unroll 1
        for (int k = 0; k < 8; ++k) w[b] |= code_of(Elem<T>::to_f(src[8 * b + k]), lo, vs, vi) << (4 * k);
      }
    }
    uint8_t* vc = Vc + (gr.row + i) * (D / 2) + gv * (kGroup / 2);
    if constexpr (BYTES) {
#pragma unroll
      for (int b = 0; b < 16; ++b) vc[b] = (uint8_t)(w[b >> 2] >> (8 * (b & 3)));
    } else {
      *reinterpret_cast<uint4*>(vc) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// 8 reconstructed channels (codes in the nibbles of q) to 8 adjacent outputs of
// a live row; in fp32 the whole warp calls it.  Two lanes hold 64 adjacent bytes of
// an fp32 row: they swap halves, so that each store instruction writes whole
// 32-byte sectors of it (8 requests of 6,000 tokens, d = 128: 186 us; with each
// lane's own two 16-byte stores 267, with 4 channels a lane 199).
template <typename T>
__device__ __forceinline__ void store8(T* p, bool live, uint32_t q, const float (&scale)[8], const float (&lo)[8]) {
  float x[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {                // 2^23 + code, exact
    const float c = __fsub_rn(__uint_as_float(0x4B000000u | ((q >> (4 * j)) & 15u)), 8388608.f);
    x[j] = fmaf(c, scale[j], lo[j]);
  }
  if constexpr (std::is_same<T, __nv_bfloat16>::value) {
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(x[2 * j], x[2 * j + 1]);
      w[j] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
  } else {
    const bool odd = threadIdx.x & 1;
    float y[4];                                // the other lane's half: its first if this one is even
#pragma unroll
    for (int j = 0; j < 4; ++j) y[j] = __shfl_xor_sync(0xffffffffu, odd ? x[j] : x[4 + j], 1);
    // even: bytes 0-15 (its own) and 32-47 (the other's first half) of the 64;
    // odd: 16-31 (the other's second half) and 48-63 (its own)
    float4* at = reinterpret_cast<float4*>(p) - (odd ? 1 : 0);
    if (live) {
      at[0] = odd ? make_float4(y[0], y[1], y[2], y[3]) : make_float4(x[0], x[1], x[2], x[3]);
      at[2] = odd ? make_float4(x[4], x[5], x[6], x[7]) : make_float4(y[0], y[1], y[2], y[3]);
    }
  }
}

// 8 codes; code arrays need no alignment of their own
__device__ __forceinline__ uint32_t load_codes8(const uint8_t* p, bool aligned4) {
  if (aligned4) return *reinterpret_cast<const uint32_t*>(p);
  return p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) | ((uint32_t)p[3] << 24);
}

// One warp per key group; a lane takes 8 adjacent channels (4 bytes of codes) of
// every RPW-th row, so that a warp's stores are 512 or 1,024 contiguous bytes.
// Bound by HBM.  At 16 requests of 3,136 tokens (28 layers, bf16; 3.0 GB): 527 us
// with 4 channels a lane (84% of the copy rate) and 64 bytes a lane in
// flight, 442 us (all of it) with the loads of the whole group sent at once.
template <typename T, int D>
__global__ void __launch_bounds__(kQuantWarps * 32) dequant_kernel(
    const __grid_constant__ QuantTable tb, int units, const uint8_t* __restrict__ Kc,
    const uint8_t* __restrict__ Vc, const float2* __restrict__ Kp, const float2* __restrict__ Vp,
    T* __restrict__ Kh, T* __restrict__ Vh) {
  constexpr int LPR = D / 8, RPW = 32 / LPR;   // lanes of a row, rows of a step
  constexpr bool kBf16 = std::is_same<T, __nv_bfloat16>::value;
  const int unit = blockIdx.x * kQuantWarps + (threadIdx.x >> 5);
  if (unit >= units) return;
  const int lane = threadIdx.x & 31, c0 = (lane % LPR) * 8, i0 = lane / LPR;
  const GroupRows gr = group_rows(tb, unit);
  const bool al = ((reinterpret_cast<uintptr_t>(Kc) | reinterpret_cast<uintptr_t>(Vc)) & 3u) == 0;
  constexpr int U = kGroup / RPW;              // steps; all loads of the group go out together
  uint32_t kq[U], vq[U];
  float2 vp[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t r = gr.row + min(i0 + u * RPW, gr.nrows - 1);
    kq[u] = load_codes8(Kc + r * (D / 2) + c0 / 2, al);
    vq[u] = load_codes8(Vc + r * (D / 2) + c0 / 2, al);
    vp[u] = Vp[r * (D / kGroup) + c0 / kGroup];
  }
  float ks[8], kl[8];
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    const float4 p = *reinterpret_cast<const float4*>(Kp + gr.kg * D + c0 + j);
    ks[j] = p.x;
    kl[j] = p.y;
    ks[j + 1] = p.z;
    kl[j + 1] = p.w;
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = i0 + u * RPW;
    if (kBf16 && i >= gr.nrows) continue;      // fp32: the whole warp stays, its lanes swap halves
    store8(Kh + (gr.row + i) * D + c0, i < gr.nrows, kq[u], ks, kl);
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = i0 + u * RPW;
    if (kBf16 && i >= gr.nrows) continue;
    float vs[8], vl[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      vs[j] = vp[u].x;
      vl[j] = vp[u].y;
    }
    store8(Vh + (gr.row + i) * D + c0, i < gr.nrows, vq[u], vs, vl);
  }
}

template <typename T, int D>
cudaError_t launch_t(const QuantTable& tb, int units, bool quantize, const void* K, const void* V,
                     uint8_t* Kc, uint8_t* Vc, float* Kp, float* Vp, void* Kh, void* Vh,
                     cudaStream_t st) {
  const unsigned grid = (unsigned)((units + kQuantWarps - 1) / kQuantWarps);
  if (quantize) {
    ProfileScope ps("kv4_quantize", st);
    const bool words = reinterpret_cast<uintptr_t>(Kc) % (D == 128 ? 2 : 1) == 0 &&
                       reinterpret_cast<uintptr_t>(Vc) % 16 == 0;
    auto kernel = words ? quant_kernel<T, D, false> : quant_kernel<T, D, true>;
    kernel<<<grid, kQuantWarps * 32, 0, st>>>(tb, units, static_cast<const T*>(K), static_cast<const T*>(V), Kc, Vc,
                                              reinterpret_cast<float2*>(Kp), reinterpret_cast<float2*>(Vp));
  } else {
    ProfileScope ps("kv4_dequantize", st);
    dequant_kernel<T, D><<<grid, kQuantWarps * 32, 0, st>>>(
        tb, units, Kc, Vc, reinterpret_cast<const float2*>(Kp), reinterpret_cast<const float2*>(Vp),
        static_cast<T*>(Kh), static_cast<T*>(Vh));
  }
  return cudaGetLastError();
}

}  // namespace

int kv4_group_rows() { return kGroup; }

cudaError_t launch_kv4(const QuantTable& tb, int units, int dtype, int d, bool quantize,
                       const void* K, const void* V, uint8_t* Kc, uint8_t* Vc, float* Kp, float* Vp,
                       void* Kh, void* Vh, cudaStream_t st) {
  if (units < 1) return cudaSuccess;
  if (dtype == VC_BF16) {
    if (d == 128) return launch_t<__nv_bfloat16, 128>(tb, units, quantize, K, V, Kc, Vc, Kp, Vp, Kh, Vh, st);
    return launch_t<__nv_bfloat16, 64>(tb, units, quantize, K, V, Kc, Vc, Kp, Vp, Kh, Vh, st);
  }
  if (d == 128) return launch_t<float, 128>(tb, units, quantize, K, V, Kc, Vc, Kp, Vp, Kh, Vh, st);
  return launch_t<float, 64>(tb, units, quantize, K, V, Kc, Vc, Kp, Vp, Kh, Vh, st);
}

}  // namespace vc

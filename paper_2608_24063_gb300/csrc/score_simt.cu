// Token scoring on CUDA cores (fp32 FFMA), Eq. (token_score).
//
// Two passes per (request, layer, KV head):
//   pass 1  lse2[l][j][i] = log2 sum_v exp2(x2_{j,i,v}),  x2 = scale*log2(e) * q_{j,i}.k_v
//   pass 2  s[g][v] += sum_{j in group g} sum_i exp2(x2_{j,i,v} - lse2[l][j][i])
// In the shared ranking mode pass 2 keeps each token's sum over all layers in
// registers (compensated) and writes s = sum / L once; in the layer-specific
// mode it writes one row per layer.  This path serves fp32 inputs and is the
// portable reference path for bf16.
//
// Few, short problems (one layer of 1,024 fp32 tokens) are bound by latency: a
// CTA then takes a row a warp (pass 1) or a key a lane (pass 2) instead of four
// and two, so that more of them share the work, and the next tile loads into
// registers while the current one is used.  Larger problems are bound by the
// fma and shared-memory pipes with several CTAs an SM: there the registers that
// hold a tile would cost CTAs (24 layers of 12,544 bf16 tokens, d = 64: pass 2
// 2,055 us with them, 1,362 without).  Every row's and key's arithmetic is the
// same in all forms.  Tiles are read from shared memory 16 bytes at a time (rows
// padded to 4 words mod 32, free of bank conflicts).
// Measured on the 1,024-token layer (event times, before -> now): pass 1 44.9 ->
// 22.3 us, pass 2 11.7 -> 9.1 us.  Whole calls, bf16, d = 64, 24 layers of 14 / 2
// heads, window 64, against tiles read 4 bytes at a time by ordinary launches:
// n = 3,136 1,268 -> 1,162 us, 12,544 3,944 -> 3,778; fp32, d = 128, 8 layers of
// 8 / 4 heads, n = 3,136 582 -> 502.
// The next kernel may be scheduled only once a CTA has its sums: triggered
// at the start, its CTAs filled whichever SMs came free first (n = 3,136 of
// the above: 1,525 us instead of 1,252).
#include "vc_common.cuh"
#include "kernels.h"
#include "profile.h"

namespace vc {
namespace {

constexpr int kThreads = 256;   // 8 warps
constexpr int kRows = 32;       // query rows per unit of the plan tables (4 per warp)
constexpr int kKeys = 64;       // keys per unit of the plan tables, and per pass-1 tile (2 per lane)

// ROWS rows of D values of a tile, as float4 pieces held by the CTA's threads
// between their loads and their stores to shared memory (row stride D + 4).
template <typename T, int D, int ROWS>
struct TilePieces {
  static constexpr int N = ROWS * (D / 4) / kThreads > 0 ? ROWS * (D / 4) / kThreads : 1;
  float4 v[N];
  // row(r) gives row r's address, or nullptr for a row of zeros
  template <typename Row>
  __device__ __forceinline__ void load(Row row) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int e = threadIdx.x + i * kThreads, r = e / (D / 4), c4 = (e % (D / 4)) * 4;
      const T* p = r < ROWS ? row(r) : nullptr;
      v[i] = p ? load4(p + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __device__ __forceinline__ void store(float* dst) const {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int e = threadIdx.x + i * kThreads, r = e / (D / 4), c4 = (e % (D / 4)) * 4;
      if (r < ROWS) *reinterpret_cast<float4*>(dst + r * (D + 4) + c4) = v[i];
    }
  }
};

// acc[a][b] = q_row(a) . k_key(lane + 32 b), summed in order of the dimension;
// q and k point at the warp's first row and the lane's first key.
template <int D, int R, int KPL>
__device__ __forceinline__ void tile_dots(float (&acc)[R][KPL], const float* q, const float* k) {
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < KPL; ++b) acc[a][b] = 0.f;
#pragma unroll 4
  for (int c = 0; c < D; c += 4) {
    float4 kv[KPL];
#pragma unroll
    for (int b = 0; b < KPL; ++b) kv[b] = *reinterpret_cast<const float4*>(k + 32 * b * (D + 4) + c);
#pragma unroll
    for (int a = 0; a < R; ++a) {
      const float4 qv = *reinterpret_cast<const float4*>(q + a * (D + 4) + c);
#pragma unroll
      for (int b = 0; b < KPL; ++b) {
        acc[a][b] = fmaf(qv.x, kv[b].x, acc[a][b]);
        acc[a][b] = fmaf(qv.y, kv[b].y, acc[a][b]);
        acc[a][b] = fmaf(qv.z, kv[b].z, acc[a][b]);
        acc[a][b] = fmaf(qv.w, kv[b].w, acc[a][b]);
      }
    }
  }
}

// First query row of a (request, layer, KV head) row set; row rho of the set is
// query head g*G + rho / W, window row rho % W, and the set is contiguous.
template <typename T, int D>
__device__ __forceinline__ const T* row_set(const T* Qw, const Req& rq, const Shape& sh, int l, int g) {
  return Qw + rq.q_off + (int64_t)(l * sh.Hq + g * sh.G) * rq.W * D;
}

// Pass 1: grid (units over (request, row tile) x 32 / (8 R), L, Hkv); R rows a warp.
template <typename T, int D, int R, int BLOCKS>
__global__ void __launch_bounds__(kThreads, BLOCKS) lse_simt_kernel(const T* __restrict__ Qw,
                                                            const T* __restrict__ K, Shape sh,
                                                            Tables tb, float* __restrict__ lse) {
  extern __shared__ float4 smem4[];
  constexpr int kBlockRows = 8 * R, kSub = kRows / kBlockRows;
  constexpr bool kAhead = R == 1;                              // next tile loads under the current one
  float* qs = reinterpret_cast<float*>(smem4);                 // [kBlockRows][D + 4]
  float* ks = qs + kBlockRows * (D + 4);                       // [kAhead ? 2 : 1][kKeys][D + 4]
  dep_wait();                                                  // the plan tables
  const int unit = blockIdx.x / kSub;
  const int r = upper_index(tb.unit0_lse, sh.n_req, (int32_t)unit);
  const Req& rq = tb.req[r];
  const int l = blockIdx.y, g = blockIdx.z, n = rq.n;
  const int rows = sh.G * rq.W;
  const int r0 = (unit - tb.unit0_lse[r]) * kRows + (blockIdx.x % kSub) * kBlockRows;
  if (r0 >= rows) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const T* Kl = K + rq.kv_off + (int64_t)(l * sh.Hkv + g) * n * D;
  const T* Ql = row_set<T, D>(Qw, rq, sh, l, g);
  TilePieces<T, D, kBlockRows> qp;
  qp.load([&](int i) { return r0 + i < rows ? Ql + (int64_t)(r0 + i) * D : nullptr; });
  TilePieces<T, D, kKeys> kp;
  auto load_keys = [&](int v0) {
    kp.load([&](int i) { return v0 + i < n ? Kl + (int64_t)(v0 + i) * D : nullptr; });
  };
  qp.store(qs);
  if (kAhead) {
    load_keys(0);
    kp.store(ks);
    __syncthreads();
  }
  float m[R], z[R];
#pragma unroll
  for (int a = 0; a < R; ++a) { m[a] = -INFINITY; z[a] = 0.f; }

  int buf = 0;
  for (int v0 = 0; v0 < n; v0 += kKeys, buf ^= kAhead ? 1 : 0) {
    const bool more = v0 + kKeys < n;
    if (!kAhead) {
      load_keys(v0);
      kp.store(ks);
      __syncthreads();
    } else if (more) {
      load_keys(v0 + kKeys);
    }
    float acc[R][2];
    tile_dots<D, R, 2>(acc, qs + R * warp * (D + 4), ks + (buf * kKeys + lane) * (D + 4));
    const bool ok0 = v0 + lane < n, ok1 = v0 + lane + 32 < n;
#pragma unroll
    for (int a = 0; a < R; ++a) {
      const float x0 = ok0 ? acc[a][0] * sh.scale_log2 : -INFINITY;
      const float x1 = ok1 ? acc[a][1] * sh.scale_log2 : -INFINITY;
      const float mn = fmaxf(m[a], fmaxf(x0, x1));
      if (mn != -INFINITY) {
        z[a] = z[a] * exp2f(m[a] - mn) + exp2f(x0 - mn) + exp2f(x1 - mn);
        m[a] = mn;
      }
    }
    if (kAhead && more) kp.store(ks + (buf ^ 1) * kKeys * (D + 4));
    __syncthreads();
  }
  if (threadIdx.x == 0) dep_launch();
  // merge the 32 lanes' partial (max, sum) of each row
#pragma unroll
  for (int a = 0; a < R; ++a) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float mo = __shfl_xor_sync(0xffffffffu, m[a], off);
      const float zo = __shfl_xor_sync(0xffffffffu, z[a], off);
      const float mn = fmaxf(m[a], mo);
      if (mn != -INFINITY) {
        z[a] = z[a] * exp2f(m[a] - mn) + zo * exp2f(mo - mn);
        m[a] = mn;
      }
    }
    const int rho = r0 + R * warp + a;
    if (lane == 0 && rho < rows) {
      const int j = g * sh.G + rho / rq.W, i = rho % rq.W;
      lse[rq.lse_off + (int64_t)(l * sh.Hq + j) * rq.W + i] = m[a] + log2f(z[a]);
    }
  }
}

// Pass 2: grid (units over (request, key tile) x 64 / (32 KPL), Hkv), KPL keys a
// lane.  Loops over all layers.  lse_nat != nullptr: normalisers come from the
// caller (natural log, [L][Hq][W]).
template <typename T, int D, int KPL>
__global__ void __launch_bounds__(kThreads) colsum_simt_kernel(const T* __restrict__ Qw,
                                                               const T* __restrict__ K, Shape sh,
                                                               Tables tb,
                                                               const float* __restrict__ lse,
                                                               const float* __restrict__ lse_nat,
                                                               float* __restrict__ scores) {
  extern __shared__ float4 smem4[];
  constexpr int kBlockKeys = 32 * KPL, kSub = kKeys / kBlockKeys;
  constexpr bool kAhead = KPL == 1;                            // next rows and keys load under the current ones
  constexpr int kBufs = kAhead ? 2 : 1;
  float* qs = reinterpret_cast<float*>(smem4);                 // [kBufs][kRows][D + 4]
  float* ks = qs + kBufs * kRows * (D + 4);                    // [kBlockKeys][D + 4]
  float* ls = ks + kBlockKeys * (D + 4);                       // [kBufs][kRows]
  float (*red)[kBlockKeys] = reinterpret_cast<float (*)[kBlockKeys]>(ls + kBufs * kRows);
  dep_wait();                                                  // the tables and pass 1's normalisers
  const int unit = blockIdx.x / kSub;
  const int r = upper_index(tb.unit0_col, sh.n_req, (int32_t)unit);
  const Req& rq = tb.req[r];
  const int g = blockIdx.y, n = rq.n;
  const int v0 = (unit - tb.unit0_col[r]) * kKeys + (blockIdx.x % kSub) * kBlockKeys;
  if (v0 >= n) return;
  const int rows = sh.G * rq.W;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // steps (layer, row tile); a step's rows and normalisers load during the step before
  const int tiles = (rows + kRows - 1) / kRows, steps = sh.L * tiles;
  TilePieces<T, D, kRows> qp;
  float lp = INFINITY;
  auto load_rows = [&](int step) {
    const int l = step / tiles, r0 = (step % tiles) * kRows;
    const T* Ql = row_set<T, D>(Qw, rq, sh, l, g);
    qp.load([&](int i) { return r0 + i < rows ? Ql + (int64_t)(r0 + i) * D : nullptr; });
    if (threadIdx.x < kRows) {
      const int rho = r0 + threadIdx.x;
      lp = INFINITY;   // padded rows contribute exp2(-inf) = 0
      if (rho < rows) {
        const int64_t o = rq.lse_off + (int64_t)(l * sh.Hq + g * sh.G) * rq.W + rho;
        lp = lse_nat ? lse_nat[o] * kLog2e : lse[o];
      }
    }
  };
  auto store_rows = [&](int buf) {
    qp.store(qs + buf * kRows * (D + 4));
    if (threadIdx.x < kRows) ls[buf * kRows + threadIdx.x] = lp;
  };
  TilePieces<T, D, kBlockKeys> kp;
  auto load_keys = [&](int l) {
    const T* Kl = K + rq.kv_off + (int64_t)(l * sh.Hkv + g) * n * D;
    kp.load([&](int i) { return v0 + i < n ? Kl + (int64_t)(v0 + i) * D : nullptr; });
  };
  if (kAhead) {
    load_rows(0);
    load_keys(0);
    store_rows(0);
  }
  Kahan tot[KPL], lay[KPL];
#pragma unroll
  for (int b = 0; b < KPL; ++b) { tot[b].init(); lay[b].init(); }
  for (int step = 0; step < steps; ++step) {
    const int l = step / tiles, tile = step % tiles, buf = kAhead ? step & 1 : 0;
    if (!kAhead) {
      load_rows(step);
      store_rows(0);
    }
    if (tile == 0) {
      if (!kAhead) load_keys(l);
      kp.store(ks);                              // the layer's keys (their readers are past the last barrier)
#pragma unroll
      for (int b = 0; b < KPL; ++b) lay[b].init();
    }
    __syncthreads();
    if (kAhead && step + 1 < steps) {
      load_rows(step + 1);
      if (tile == tiles - 1) load_keys(l + 1);
    }
    float acc[4][KPL];
    tile_dots<D, 4, KPL>(acc, qs + (buf * kRows + 4 * warp) * (D + 4), ks + lane * (D + 4));
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const float lz = ls[buf * kRows + 4 * warp + a];
#pragma unroll
      for (int b = 0; b < KPL; ++b) lay[b].add(exp2f(fmaf(acc[a][b], sh.scale_log2, -lz)));
    }
    if (kAhead && step + 1 < steps) store_rows(buf ^ 1);
    if (tile < tiles - 1) {
      if (!kAhead) __syncthreads();              // the rows are read: the next ones may come
      continue;
    }
    if (sh.rank_mode == VC_RANK_PER_LAYER) {
#pragma unroll
      for (int b = 0; b < KPL; ++b) red[warp][lane + 32 * b] = lay[b].s;
      __syncthreads();
      if (threadIdx.x < kBlockKeys && v0 + threadIdx.x < n) {
        Kahan k; k.init();
        for (int w = 0; w < 8; ++w) k.add(red[w][threadIdx.x]);
        scores[rq.s_off + ((int64_t)l * sh.Hkv + g) * n + v0 + threadIdx.x] = k.s;
      }
    } else {
#pragma unroll
      for (int b = 0; b < KPL; ++b) tot[b].add(lay[b].s);
    }
    __syncthreads();                             // keys (and partial sums) read: the next layer's may come
  }
  if (threadIdx.x == 0) dep_launch();
  if (sh.rank_mode != VC_RANK_PER_LAYER) {
#pragma unroll
    for (int b = 0; b < KPL; ++b) red[warp][lane + 32 * b] = tot[b].s;
    __syncthreads();
    if (threadIdx.x < kBlockKeys && v0 + threadIdx.x < n) {
      Kahan k; k.init();
      for (int w = 0; w < 8; ++w) k.add(red[w][threadIdx.x]);
      scores[rq.s_off + (int64_t)g * n + v0 + threadIdx.x] = k.s / (float)sh.L;
    }
  }
}

template <typename T, int D, int R, int BLOCKS>
cudaError_t launch_lse(const T* q, const T* k, const Shape& sh, const Tables& tb, int units, float* lse,
                       cudaStream_t st) {
  const size_t smem = sizeof(float) * (8 * R + (R == 1 ? 2 : 1) * kKeys) * (D + 4);
  cudaError_t e = cudaFuncSetAttribute(lse_simt_kernel<T, D, R, BLOCKS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  ProfileScope ps("score_lse_simt", st);
  return launch_dep(lse_simt_kernel<T, D, R, BLOCKS>, dim3(units * (kRows / (8 * R)), sh.L, sh.Hkv), dim3(kThreads),
                    smem, st, q, k, sh, tb, lse);
}

template <typename T, int D, int KPL>
cudaError_t launch_colsum(const T* q, const T* k, const Shape& sh, const Tables& tb, int units, const float* lse,
                          const float* lse_nat, float* scores, cudaStream_t st) {
  constexpr int kBufs = KPL == 1 ? 2 : 1;
  const size_t smem = sizeof(float) * ((kBufs * kRows + 32 * KPL) * (D + 4) + kBufs * kRows + 8 * 32 * KPL);
  cudaError_t e = cudaFuncSetAttribute(colsum_simt_kernel<T, D, KPL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  ProfileScope ps("score_colsum_simt", st);
  return launch_dep(colsum_simt_kernel<T, D, KPL>, dim3(units * (kKeys / (32 * KPL)), sh.Hkv), dim3(kThreads), smem, st,
                    q, k, sh, tb, lse, lse_nat, scores);
}

template <typename T, int D>
cudaError_t launch_t(const void* Qw, const void* K, const Shape& sh, const Tables& tb,
                     int units_lse, int units_col, float* lse, const float* lse_nat,
                     float* scores, cudaStream_t st) {
  const T* q = static_cast<const T*>(Qw);
  const T* k = static_cast<const T*>(K);
  // Blocks of the larger tiles.  The smaller ones read shared memory twice as
  // often per product, so they serve only where the others leave the chip half
  // empty.  Pass 1, four for one (us, large | small): d = 64, 16 blocks 54 | 31,
  // 48 78 | 68, 72 99 | 86, 96 147 | 168; d = 128, 32 123 | 72, 64 204 | 206, 80
  // 124 | 186.  Pass 2, two for one: 64 15 | 12, 76 33 | 25 (d = 128), 100 15 | 18,
  // 152 33 | 43 (d = 128).
  const int sms = sm_count();
  const int64_t blocks1 = (int64_t)units_lse * sh.L * sh.Hkv, blocks2 = (int64_t)units_col * sh.Hkv;
  cudaError_t e;
  if (!lse_nat) {
    // d = 64, more than two blocks an SM: five fit with 48 registers (12,544 bf16
    // tokens, 672 blocks: 1,671 -> 1,374 us; 72 blocks: 99 -> 119)
    if (2 * blocks1 <= sms) e = launch_lse<T, D, 1, 1>(q, k, sh, tb, units_lse, lse, st);
    else if (D == 128 || blocks1 <= 2 * sms) e = launch_lse<T, D, 4, 4>(q, k, sh, tb, units_lse, lse, st);
    else e = launch_lse<T, D, 4, D == 128 ? 4 : 5>(q, k, sh, tb, units_lse, lse, st);
    if (e != cudaSuccess) return e;
  }
  return 2 * blocks2 <= sms ? launch_colsum<T, D, 1>(q, k, sh, tb, units_col, lse, lse_nat, scores, st)
                            : launch_colsum<T, D, 2>(q, k, sh, tb, units_col, lse, lse_nat, scores, st);
}

}  // namespace

int score_rows_per_tile_simt() { return kRows; }
int score_keys_per_tile_simt() { return kKeys; }

int sm_count() {
  static std::atomic<int> cached[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
  int n = cached[dev].load(std::memory_order_relaxed);
  if (n > 0) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 1;
  cached[dev].store(n, std::memory_order_relaxed);
  return n;
}

cudaError_t launch_score_simt(int dtype, const void* Qw, const void* K, const Shape& sh,
                              const Tables& tb, int units_lse, int units_col, float* lse,
                              const float* lse_nat, float* scores, cudaStream_t st) {
  if (dtype == VC_F32) {
    if (sh.d == 64) return launch_t<float, 64>(Qw, K, sh, tb, units_lse, units_col, lse, lse_nat, scores, st);
    return launch_t<float, 128>(Qw, K, sh, tb, units_lse, units_col, lse, lse_nat, scores, st);
  }
  if (sh.d == 64)
    return launch_t<__nv_bfloat16, 64>(Qw, K, sh, tb, units_lse, units_col, lse, lse_nat, scores, st);
  return launch_t<__nv_bfloat16, 128>(Qw, K, sh, tb, units_lse, units_col, lse, lse_nat, scores, st);
}

}  // namespace vc

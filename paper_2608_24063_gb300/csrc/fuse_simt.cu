// Prune keys, fuse values, compact -- Algorithm 1 step 3.
//
// fuse_v_simt_kernel: per (request, layer, KV head, tile of 8 R kept rows, R
//   rows a warp) O = softmax_row(V_k V_d^T / tau) V_d with an online (running
//   max / sum) softmax over tiles of 64 dropped rows, then
//   V_out = mu V_k + (1-mu) O, Eq. (redistribution) and Eq. (weight_fusion).
//   Empty drop set: V_out = V_k.  The CTA also copies its kept keys, K_out =
//   K[keep] (bit-exact 16-byte pieces).
// R is 4, or 1 where that would leave SMs idle (one layer of 1,024 fp32 tokens:
// 32 CTAs of 32 rows); rows in shared memory are read 16 bytes at a time.  Measured on
// that problem, with the key copy (a kernel of its own before): 23.0 -> 12.7 us.
#include "vc_common.cuh"
#include "kernels.h"
#include "profile.h"

namespace vc {
namespace {

constexpr int kFuseThreads = 256;   // 8 warps
constexpr int kFuseRows = 32;       // kept rows per unit of the plan tables
constexpr int kFuseKeys = 64;       // dropped rows per tile (2 per lane)

template <typename T, int D, int R>
__global__ void __launch_bounds__(kFuseThreads) fuse_v_simt_kernel(
    const T* __restrict__ K, const T* __restrict__ V, Shape sh, Tables tb, const int32_t* __restrict__ keep_idx,
    const int32_t* __restrict__ drop_idx, float mu, float inv_tau_log2, T* __restrict__ K_out,
    T* __restrict__ V_out) {
  extern __shared__ float4 smem4[];
  constexpr int kBlockRows = 8 * R, kSub = kFuseRows / kBlockRows;
  constexpr int PR = D * (int)sizeof(T) / 16;                  // 16-byte pieces of a row
  float* vk = reinterpret_cast<float*>(smem4);                 // [kBlockRows][D + 4]
  float* vd = vk + kBlockRows * (D + 4);                       // [kFuseKeys][D + 4]
  float* ps = vd + kFuseKeys * (D + 4);                        // [kBlockRows][kFuseKeys + 4]
  dep_wait();                                                  // the keep and drop lists
  if (threadIdx.x == 0) dep_launch();
  // unit -> (request, layer), then (KV head, row tile)
  const int unit = blockIdx.x / kSub;
  const int rl = upper_index(tb.unit0_fuse, sh.n_req * sh.L, (int32_t)unit);
  const int r = rl / sh.L, l = rl % sh.L;
  const Req& rq = tb.req[r];
  const Layer ly = tb.layer[rl];
  const int n = rq.n;
  const int tiles = (ly.B + kFuseRows - 1) / kFuseRows;
  const int u = unit - tb.unit0_fuse[rl];
  const int g = u / tiles;
  const int r0 = (u % tiles) * kFuseRows + (blockIdx.x % kSub) * kBlockRows;
  const int rows = min(kBlockRows, ly.B - r0);
  if (rows <= 0) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  const int64_t src = rq.kv_off + (int64_t)(l * sh.Hkv + g) * n * D;
  const T* Vl = V + src;
  const int64_t row0 = rq.out_row0 + (int64_t)sh.Hkv * ly.P + (int64_t)g * ly.B + r0;
  const int32_t* kp = keep_idx + row0;
  const int32_t* dp = drop_idx + rq.drop_row0 + (int64_t)sh.Hkv * ly.Qd + (int64_t)g * ly.D;
  T* out = V_out + row0 * D;

  // kept rows, and their keys
  for (int e = threadIdx.x; e < kBlockRows * (D / 4); e += kFuseThreads) {
    const int rr = e / (D / 4), c4 = (e % (D / 4)) * 4;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (rr < rows) {
      const int v = kp[rr];
      if (v >= 0 && v < n) x = load4(Vl + (int64_t)v * D + c4);
      else set_status(tb.status, VC_ERR_DEVICE_INDEX);
    }
    *reinterpret_cast<float4*>(vk + rr * (D + 4) + c4) = x;
  }
  for (int e = threadIdx.x; e < rows * PR; e += kFuseThreads) {
    const int v = kp[e / PR];
    if (v >= 0 && v < n)
      reinterpret_cast<uint4*>(K_out + row0 * D)[e] = reinterpret_cast<const uint4*>(K + src + (int64_t)v * D)[e % PR];
    else
      set_status(tb.status, VC_ERR_DEVICE_INDEX);
  }

  constexpr int CPL = D / 32;   // output columns per lane
  float o[R][CPL];
  float m[R], zs[R];
#pragma unroll
  for (int a = 0; a < R; ++a) {
    m[a] = -INFINITY; zs[a] = 0.f;
#pragma unroll
    for (int c = 0; c < CPL; ++c) o[a][c] = 0.f;
  }
  const float* q = vk + R * warp * (D + 4);
  float* p = ps + R * warp * (kFuseKeys + 4);

  for (int j0 = 0; j0 < ly.D; j0 += kFuseKeys) {
    __syncthreads();
    for (int e = threadIdx.x; e < kFuseKeys * (D / 4); e += kFuseThreads) {
      const int rr = e / (D / 4), c4 = (e % (D / 4)) * 4;
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j0 + rr < ly.D) {
        const int v = dp[j0 + rr];
        if (v >= 0 && v < n) x = load4(Vl + (int64_t)v * D + c4);
        else set_status(tb.status, VC_ERR_DEVICE_INDEX);
      }
      *reinterpret_cast<float4*>(vd + rr * (D + 4) + c4) = x;
    }
    __syncthreads();
    // logits for R kept rows x 2 dropped rows
    float acc[R][2];
#pragma unroll
    for (int a = 0; a < R; ++a) acc[a][0] = acc[a][1] = 0.f;
#pragma unroll 4
    for (int c = 0; c < D; c += 4) {
      const float4 d0 = *reinterpret_cast<const float4*>(vd + lane * (D + 4) + c);
      const float4 d1 = *reinterpret_cast<const float4*>(vd + (lane + 32) * (D + 4) + c);
#pragma unroll
      for (int a = 0; a < R; ++a) {
        const float4 x = *reinterpret_cast<const float4*>(q + a * (D + 4) + c);
        acc[a][0] = fmaf(x.w, d0.w, fmaf(x.z, d0.z, fmaf(x.y, d0.y, fmaf(x.x, d0.x, acc[a][0]))));
        acc[a][1] = fmaf(x.w, d1.w, fmaf(x.z, d1.z, fmaf(x.y, d1.y, fmaf(x.x, d1.x, acc[a][1]))));
      }
    }
    const bool ok0 = j0 + lane < ly.D, ok1 = j0 + lane + 32 < ly.D;
#pragma unroll
    for (int a = 0; a < R; ++a) {
      const float x0 = ok0 ? acc[a][0] * inv_tau_log2 : -INFINITY;
      const float x1 = ok1 ? acc[a][1] * inv_tau_log2 : -INFINITY;
      float tm = fmaxf(x0, x1);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) tm = fmaxf(tm, __shfl_xor_sync(0xffffffffu, tm, off));
      const float mn = fmaxf(m[a], tm);          // finite: at least one valid key per tile
      const float corr = exp2f(m[a] - mn);
      const float p0 = exp2f(x0 - mn), p1 = exp2f(x1 - mn);
      float ts = p0 + p1;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) ts += __shfl_xor_sync(0xffffffffu, ts, off);
      zs[a] = zs[a] * corr + ts;
      m[a] = mn;
#pragma unroll
      for (int c = 0; c < CPL; ++c) o[a][c] *= corr;
      p[a * (kFuseKeys + 4) + lane] = p0;
      p[a * (kFuseKeys + 4) + lane + 32] = p1;
    }
    __syncwarp();
    // O[row][col] += sum_k P[row][k] V_d[k][col]  (cols lane + 32 c); rows are warp-private
#pragma unroll 2
    for (int k = 0; k < kFuseKeys; k += 4) {
      float4 pv[R];
#pragma unroll
      for (int a = 0; a < R; ++a) pv[a] = *reinterpret_cast<const float4*>(p + a * (kFuseKeys + 4) + k);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float dv[CPL];
#pragma unroll
        for (int c = 0; c < CPL; ++c) dv[c] = vd[(k + i) * (D + 4) + lane + 32 * c];
#pragma unroll
        for (int a = 0; a < R; ++a) {
          const float x = i == 0 ? pv[a].x : i == 1 ? pv[a].y : i == 2 ? pv[a].z : pv[a].w;
#pragma unroll
          for (int c = 0; c < CPL; ++c) o[a][c] = fmaf(x, dv[c], o[a][c]);
        }
      }
    }
  }
  __syncthreads();
  // epilogue: V_out = mu V_k + (1 - mu) O / Z   (V_k itself when the drop set is empty)
#pragma unroll
  for (int a = 0; a < R; ++a) {
    const int rr = R * warp + a;
    if (rr >= rows) continue;
    const float inv = ly.D > 0 ? 1.f / zs[a] : 0.f;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const int col = lane + 32 * c;
      const float vkc = vk[rr * (D + 4) + col];
      const float y = ly.D > 0 ? fmaf(mu, vkc, (1.f - mu) * (o[a][c] * inv)) : vkc;
      out[(int64_t)rr * D + col] = Elem<T>::from_f(y);
    }
  }
}

template <typename T, int D, int R>
cudaError_t launch_fuse_r(const void* K, const void* V, const Shape& sh, const Tables& tb, const int32_t* keep_idx,
                          const int32_t* drop_idx, float mu, float tau, void* K_out, void* V_out, int units,
                          cudaStream_t st) {
  const size_t smem = sizeof(float) * ((8 * R + kFuseKeys) * (D + 4) + 8 * R * (kFuseKeys + 4));
  cudaError_t e = cudaFuncSetAttribute(fuse_v_simt_kernel<T, D, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  ProfileScope ps("fuse_v_simt", st);
  return launch_dep(fuse_v_simt_kernel<T, D, R>, dim3(units * (kFuseRows / (8 * R))), dim3(kFuseThreads), smem, st,
                    static_cast<const T*>(K), static_cast<const T*>(V), sh, tb, keep_idx, drop_idx, mu, kLog2e / tau,
                    static_cast<T*>(K_out), static_cast<T*>(V_out));
}

template <typename T, int D>
cudaError_t launch_fuse_t(const void* K, const void* V, const Shape& sh, const Tables& tb, const int32_t* keep_idx,
                          const int32_t* drop_idx, float mu, float tau, void* K_out, void* V_out, int units,
                          cudaStream_t st) {
  // 8 rows a CTA while all of those fit at once, five an SM at d = 128: fewer of
  // them leave SMs idle, more read the dropped rows too often (us, 32 | 8 rows:
  // 114 units 52 | 43, 171 54 | 39, 238 127 | 228, 342 48 | 61)
  if (4 * (int64_t)units <= 5 * (int64_t)sm_count())
    return launch_fuse_r<T, D, 1>(K, V, sh, tb, keep_idx, drop_idx, mu, tau, K_out, V_out, units, st);
  return launch_fuse_r<T, D, 4>(K, V, sh, tb, keep_idx, drop_idx, mu, tau, K_out, V_out, units, st);
}

}  // namespace

int fuse_rows_per_tile_simt() { return kFuseRows; }

cudaError_t launch_fuse_simt(int dtype, const void* K, const void* V, const Shape& sh, const Tables& tb,
                             const int32_t* keep_idx, const int32_t* drop_idx, float mu, float tau,
                             void* K_out, void* V_out, int units, cudaStream_t st) {
  if (units == 0) return cudaSuccess;
  if (dtype == VC_F32) {
    if (sh.d == 64) return launch_fuse_t<float, 64>(K, V, sh, tb, keep_idx, drop_idx, mu, tau, K_out, V_out, units, st);
    return launch_fuse_t<float, 128>(K, V, sh, tb, keep_idx, drop_idx, mu, tau, K_out, V_out, units, st);
  }
  if (sh.d == 64)
    return launch_fuse_t<__nv_bfloat16, 64>(K, V, sh, tb, keep_idx, drop_idx, mu, tau, K_out, V_out, units, st);
  return launch_fuse_t<__nv_bfloat16, 128>(K, V, sh, tb, keep_idx, drop_idx, mu, tau, K_out, V_out, units, st);
}

}  // namespace vc

// Token scoring on the tcgen05 tensor cores, Eq. (token_score); bf16 inputs, d = 128.
//
// Per (request, layer, KV head) the G*W window rows (contiguous in Qw) meet
// the n visual keys (contiguous in K).  Logits come from tcgen05.mma (bf16 x
// bf16 -> fp32 in tensor memory), operands staged by TMA with 128-byte
// swizzling.  The exact softmax column sum needs every row's normaliser
// first, so the score takes two passes over the logits:
//
//   pass 1 (score_lse_tc)    persistent CTA pairs, rows in TMEM lanes: per row,
//                            running max and compensated sum of exp2 over a
//                            range of 256-key tiles -> partial (m, z) per key
//                            split;
//   merge  (lse_merge)       -lse2 = -(m + log2 z) over the splits (or minus
//                            the caller's natural-log normaliser * log2 e),
//                            written per (layer, KV head) padded with -inf to
//                            whole pass-2 chunks; with a single key split
//                            pass 1 writes these values itself and the merge
//                            is skipped;
//   pass 2 (score_colsum_tc) CTA pairs, keys in TMEM lanes: each thread owns
//                            one key and sums exp2(x*scale*log2e - lse2[row])
//                            over all rows of all layers (compensated),
//                            s = sum / L.  Each 256-row chunk's normalisers
//                            arrive beside its Q rows (one bulk copy per
//                            CTA), padding rows contribute 0.
//
// Warp roles in both passes (384 threads, one CTA per SM): warps 0-3 and 4-7
// are two consumer warpgroups (one TMEM lane per thread), warp 8 issues TMA and
// owns the tensor-memory allocation, one thread of warp 9 issues the MMAs (in
// both passes only the even CTA of each pair issues them, as 2-SM MMAs).
// Each consumer thread takes a whole tile (up to 128 accumulators) per step,
// so its exps and sums form many independent chains.  Every wait is bounded: on a
// timeout the CTA stops issuing, waits for its own copies and MMAs, frees its
// tensor memory and records VC_ERR_DEVICE_TIMEOUT.
#include <cudaTypedefs.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "kernels.h"
#include "profile.h"
#include "tc_common.cuh"
#include "vc_common.cuh"

namespace vc {
namespace {

using namespace tc;

constexpr int kThreads = 384;                   // three warpgroups (warps 10 and 11 idle)
// Registers per thread: the launch's 168 x 384 threads, moved from the third
// warpgroup to the consumers, who hold 128 accumulators each (pass 2 at 168:
// 154.4 us for n = 12,544 and 4,430 us for the 72B shape, now 150.5 and 4,315;
// pass 1 the same either way; event times).
constexpr int kConsumerRegs = 232, kOtherRegs = 40;
static_assert(256 * kConsumerRegs + 128 * kOtherRegs <= 384 * 168, "the split fits what the launch gets");
constexpr int kProducerWarp = 8, kMmaWarp = 9;
constexpr uint32_t kTile = 128;                 // keys per tile, rows per block / chunk
constexpr uint32_t kKBlockBytes = kTile * 128;  // 128 rows x 64 bf16
constexpr uint32_t kTileBytes = 2 * kKBlockBytes;
constexpr uint32_t kTmemCols = 512;




// sum_j exp2(x_j * s + b_j) over 16 values, with packed fp32x2 FMA and adds
// (pairwise, so the rounding error stays a few ulp).
__device__ __forceinline__ float exp2_sum16(const float (&x)[16], float2 s, const float2 (&b)[8]) {
  float2 e[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float2 t = __ffma2_rn(make_float2(x[2 * j], x[2 * j + 1]), s, b[j]);
    e[j] = make_float2(ex2(t.x), ex2(t.y));
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) e[j] = __fadd2_rn(e[2 * j], e[2 * j + 1]);
  e[0] = __fadd2_rn(e[0], e[1]);
  e[2] = __fadd2_rn(e[2], e[3]);
  e[0] = __fadd2_rn(e[0], e[2]);
  return e[0].x + e[0].y;
}

// ---------------------------------------------------------------------------
// pass 1 on CTA pairs
//
// Persistent: as many pairs as the device holds, each taking its units (256
// window rows of a (request, layer, KV head) and a range of 256-key tiles) one
// after the other, longest first and dealt back and forth, so nothing starts
// or drains between them.  A pair covers 256 window rows (128 per CTA, rows in
// TMEM lanes); each CTA loads its 128 query rows of the unit (double buffered
// across units) and, per tile, its own 128 keys; one 2-SM MMA chain (M = 256,
// N = 256, K = 128) leaves every row's 256 logits in its own CTA's tensor
// memory.  Tensor memory: 2 slots x 256 columns; consumer warpgroup wg takes
// the tiles i with i % 2 == wg of each unit from slot wg, so the MMA fills one
// slot while the other is read.  A slot is always the same warpgroup's, which
// waits for its uses in order, so no waiter can be two phases ahead of a
// barrier.  The two warpgroups' per-row (max, sum) pairs are merged at the end
// of a unit.
//
// Bound by the consumers: per half tile and warp ~1,030 cycles of exps, 400 of
// TMEM load and maximum, ~150 waiting for the slot (clock stamps; two warps share
// a sub-partition's exp2 unit, which the 256 exps of both keep busy for 1,024).
// Slots of 128 columns, freed as soon as they are in registers, were slower
// (153 us): an N = 128 MMA takes ~120 cycles, hardly less than an N = 256 one.
// Measured (event times), one unit per launched pair -> now: n = 3,136 58.1 -> 47.3
// us, n = 12,544 147.7 -> 140.4, layer-specific ranking 144.3 -> 118.3, ragged batch
// 1,348 -> 1,257, 72B shape 4,456 -> 4,061.

constexpr uint32_t kPairKeys = 256;             // keys per pass-1 tile (both CTAs)
constexpr int kStagesPair = 4;                  // K ring of pass 1 (per CTA: 32 KB a stage)
constexpr int kSlots1 = 2;                      // tensor-memory slots of 256 columns
constexpr int kMaxUnits1 = 256;                 // units per pair and launch (descriptor table)

struct Unit1 {                                  // one unit as this CTA sees it
  int32_t qrow, krow;                           // Qw row of this CTA's first window row; K row of its first key
  int32_t ntiles, keys;                         // 256-key tiles; valid keys from the unit's first on
  int32_t rho0, rows, prow;                     // this CTA's first row in the row set; the set's rows, padded rows
  int32_t split;
  int64_t out;                                  // S > 1: first row of the set in `part`; else in `nlse`
};

struct P1Smem {
  uint8_t q[2][2][kKBlockBytes];                // this CTA's 128 query rows of unit k in q[k % 2] [K-block]
  uint8_t k[kStagesPair][2][kKBlockBytes];      // this CTA's 128 keys of the tile [stage][K-block]
  Unit1 unit[kMaxUnits1];
  float2 half[2][4][32];                        // [unit & 1]: (max, sum) of warpgroup 1
  uint64_t q_full[2];                           // even CTA: both CTAs' Q rows landed
  uint64_t q_empty[2];                          // both: the MMAs of the unit are done
  uint64_t k_full[kStagesPair];                 // even CTA: both CTAs' keys landed
  uint64_t k_empty[kStagesPair];                // both: the MMAs reading the stage are done
  uint64_t tm_full[kSlots1];                    // both: the slot's logits are ready
  uint64_t tm_empty[kSlots1];                   // even CTA: the slot's 8 consumer warps copied it out
  uint64_t mma_done;                            // both: every MMA of the pair is done
  uint64_t never;                               // test support: never completes
  uint64_t peer_done;                           // even CTA: the odd CTA's fill counts landed (8 bytes)
  int2 peer_fills;                              // even CTA: (unit rows, key tiles) the odd CTA issued
  uint32_t tmem_base;
  int abort;
};

// Named barriers of the per-unit merge: warpgroup 1 arrives at kHalfFull + b
// when its statistics are in half[b], warpgroup 0 at kHalfEmpty + b when it
// has read them.
constexpr uint32_t kHalfFull = 1, kHalfEmpty = 3;

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
score_lse_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    Shape sh, Tables tb, int S, int u_lo, int u_cnt, float2* __restrict__ part,
                    float* __restrict__ nlse, int32_t* __restrict__ split_counts) {
  extern __shared__ uint8_t smem_raw[];
  P1Smem& sm = *reinterpret_cast<P1Smem*>(align1024(smem_raw));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) { mbar_init(&sm.q_full[i], 1); mbar_init(&sm.q_empty[i], 1); }
    for (int i = 0; i < kStagesPair; ++i) { mbar_init(&sm.k_full[i], 1); mbar_init(&sm.k_empty[i], 1); }
    for (int i = 0; i < kSlots1; ++i) { mbar_init(&sm.tm_full[i], 1); mbar_init(&sm.tm_empty[i], 8); }
    mbar_init(&sm.mma_done, 1);
    mbar_init(&sm.never, 1);
    mbar_init(&sm.peer_done, 1);
    sm.abort = 0;
    fence_mbar_init();
    if (rank == 0) mbar_arrive_expect_tx(&sm.peer_done, 8);
  }
  if (warp == kProducerWarp) {
    tmem_alloc_pair(&sm.tmem_base, kTmemCols);
    tmem_relinquish_pair();
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync();                  // barriers of both CTAs, TMEM
  tc_fence_after();
  // the plan tables come from the kernel just before this one
  dep_wait();
  if (split_counts && blockIdx.x == 0) {       // pass 2's counts, before it can be scheduled
    if (threadIdx.x < 2 * kMaxPairs2) split_counts[threadIdx.x] = 0;
    __syncthreads();
  }
  if (threadIdx.x == 0) dep_launch();
  // this pair's units: positions of the longest-first order [u_lo, u_lo + u_cnt)
  // dealt to the pairs back and forth
  const int pair = (int)(blockIdx.x >> 1), npairs = (int)(gridDim.x >> 1);
  const int rounds = u_cnt / npairs, rem = u_cnt % npairs;
  const int nunits = min(kMaxUnits1, rounds + ((rounds & 1) ? (pair >= npairs - rem) : (pair < rem)));
  for (int i = threadIdx.x; i < nunits; i += kThreads) {
    const int unit = u_lo + i * npairs + ((i & 1) ? npairs - 1 - pair : pair);
    const int place = upper_index(tb.unit0_tc1, sh.n_req, (int32_t)unit);
    const Req& rq = tb.req[sh.n_req > 1 ? tb.req[place].by_length : 0];
    int u = unit - tb.unit0_tc1[place];
    const int split = u % S;
    u /= S;
    const int rbp = u % rq.nrb;
    u /= rq.nrb;
    const int g = u % sh.Hkv, l = u / sh.Hkv;
    const int ntiles_all = (rq.n + (int)kPairKeys - 1) / (int)kPairKeys;
    const int tps = (ntiles_all + S - 1) / S;
    const int t_begin = split * tps;
    Unit1 d;
    d.rho0 = rbp * 256 + (int)rank * (int)kTile;
    d.rows = sh.G * rq.W;
    d.prow = rq.C * rq.cw;
    d.split = split;
    d.qrow = (int)(rq.q_off / 128 + ((int64_t)l * sh.Hq + g * sh.G) * rq.W) + d.rho0;
    d.krow = (int)(rq.kv_off / 128 + ((int64_t)l * sh.Hkv + g) * rq.n) + t_begin * (int)kPairKeys +
             (int)rank * (int)kTile;
    d.ntiles = max(0, min(ntiles_all, t_begin + tps) - t_begin);
    d.keys = rq.n - t_begin * (int)kPairKeys;
    d.out = S > 1 ? rq.lse_off + ((int64_t)l * sh.Hq + g * sh.G) * rq.W
                  : rq.lsep_off + ((int64_t)l * sh.Hkv + g) * d.prow;
    sm.unit[i] = d;
  }
  __syncthreads();                 // descriptors
  const uint32_t tbase = sm.tmem_base;
  volatile int* abort = &sm.abort;

  if (warp >= 8) {
    give_registers<kOtherRegs>();
    if (warp == kProducerWarp && lane == 0) {
      // ---- TMA producer (both CTAs): own rows and keys, counted on the even CTA's barriers
      prefetch_tmap(&tmQ);
      prefetch_tmap(&tmK);
      int t = 0, kq = 0;
      bool ok = true;
      for (int k = 0; ok && k < nunits; ++k) {
        const Unit1 d = sm.unit[k];
        const int b = k & 1;
        if (!mbar_wait(&sm.q_empty[b], ((k >> 1) & 1) ^ 1, abort)) break;
        if (rank == 0) mbar_arrive_expect_tx(&sm.q_full[b], 2 * kTileBytes);
        const uint32_t q_full0 = map_to_rank(smem_u32(&sm.q_full[b]), 0);
        for (int kb = 0; kb < 2; ++kb) tma_load_2d_pair(sm.q[b][kb], &tmQ, kb * 64, d.qrow, q_full0);
        ++kq;
        for (int i = 0; i < d.ntiles; ++i) {
          const int st = t % kStagesPair;
          if (!mbar_wait(&sm.k_empty[st], ((t / kStagesPair) & 1) ^ 1, abort)) { ok = false; break; }
          if (rank == 0) mbar_arrive_expect_tx(&sm.k_full[st], 2 * kTileBytes);
          const uint32_t k_full0 = map_to_rank(smem_u32(&sm.k_full[st]), 0);
          for (int kb = 0; kb < 2; ++kb)
            tma_load_2d_pair(sm.k[st][kb], &tmK, kb * 64, d.krow + i * (int)kPairKeys, k_full0);
          ++t;
        }
      }
      // the even CTA waits until every copy of both CTAs has landed
      if (rank == 1) report_fills(&sm.peer_fills, &sm.peer_done, kq, t);
      if (rank == 0) {
        const int2 f = peer_fills(&sm.peer_done, &sm.peer_fills, make_int2(kq, t), abort);
        drain_pair_ring(sm.q_full, 2, kq, f.x, kTileBytes);
        drain_pair_ring(sm.k_full, kStagesPair, t, f.y, kTileBytes);
      }
    } else if (warp == kMmaWarp && lane == 0 && rank == 0) {
      // ---- MMA issuer (even CTA): D[row][key] for 256 rows x 128 keys per half tile
      const uint32_t idesc = idesc_bf16_f32(2 * kTile, kPairKeys);
      bool ok = true;
      int t = 0;
      uint32_t uses[2] = {0u, 0u};                  // tiles of each warpgroup so far
      for (int k = 0; ok && k < nunits; ++k) {
        const int ntiles = sm.unit[k].ntiles, b = k & 1;
        if (!mbar_wait(&sm.q_full[b], (k >> 1) & 1, abort)) break;
        for (int i = 0; ok && i < ntiles; ++i, ++t) {
          const int st = t % kStagesPair;
          if (!mbar_wait(&sm.k_full[st], (t / kStagesPair) & 1, abort)) { ok = false; break; }
          const uint32_t use = (i & 1) ? uses[1]++ : uses[0]++;
          const int slot = i & 1;
          if (!mbar_wait(&sm.tm_empty[slot], (use & 1) ^ 1, abort)) { ok = false; break; }
          tc_fence_after();
          const uint32_t d = tbase + (uint32_t)slot * kPairKeys;
  #pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            mma_bf16_pair(d, desc_sw128(smem_u32(sm.q[b][kk >> 2]) + (kk & 3) * 32),
                          desc_sw128(smem_u32(sm.k[st][kk >> 2]) + (kk & 3) * 32), idesc, kk ? 1u : 0u);
          mma_commit_pair(&sm.tm_full[slot], 3);
          mma_commit_pair(&sm.k_empty[st], 3);
        }
        if (ok) mma_commit_pair(&sm.q_empty[b], 3);
      }
      mma_commit_pair(&sm.mma_done, 3);
      drain_wait(&sm.mma_done, 0);
    } else if (warp == kMmaWarp && lane == 0) {
      // odd CTA: the pair's MMAs (and their arrivals on this CTA's barriers) are done
      drain_wait(&sm.mma_done, 0);
    }
  } else {
    take_registers<kConsumerRegs>();
    if ((sh.test_wait & VC_TEST_WAIT_SCORE_LSE) && warp == 0) {
      if (lane == 0 && injected_wait_gives_up(&sm.never)) {
        set_status(tb.status, VC_ERR_DEVICE_TIMEOUT);
        *abort = 1;
      }
      __syncwarp();
    }
    // ---- row statistics: one thread per row (= TMEM lane).  Warpgroup wg
    // takes the tiles i with i % 2 == wg of every unit, half by half, so the
    // two warpgroups on a sub-partition run a tile apart and one's waits and
    // TMEM loads overlap the other's exps.  After a give-up a warp stays in
    // its loops without waiting or touching tensor memory, but still meets the
    // other warps at the named barriers.
    const int wg = warp >> 2;
    const int lrow = ((warp & 3) << 5) + lane;
    const uint32_t lane_off = (uint32_t)((warp & 3) << 5) << 16;
    const uint32_t tm_empty0 = lane == 0 ? map_to_rank(smem_u32(&sm.tm_empty[wg]), 0) : 0u;
    const float s2 = sh.scale_log2;
    bool ok = true;
    uint32_t use = 0;                             // this warpgroup's tiles so far
    for (int k = 0; k < nunits; ++k) {
      const int ntiles = sm.unit[k].ntiles, keys = sm.unit[k].keys;
      float m = -INFINITY;
      Kahan z;
      z.init();
      // The half's exp2 sum is added to z only after the next half's exp2 terms
      // are issued (its terms have arrived by then); adding it at once would
      // stall the warp until the exp2 unit has worked through its queue.
      float pend = 0.f;
      for (int i = wg; ok && i < ntiles; i += 2, ++use) {
        ok = warp_wait(&sm.tm_full[wg], use & 1, abort);
        if (!ok) break;
        tc_fence_after();
#pragma unroll 1
        for (int hf = 0; hf < 2; ++hf) {
          const int valid = min((int)kTile, keys - i * (int)kPairKeys - hf * (int)kTile);
          const uint32_t col0 = tbase + lane_off + (uint32_t)wg * kPairKeys + (uint32_t)hf * kTile;
          float x[8][16];
          {
            uint32_t v[8][16];
#pragma unroll
            for (int p = 0; p < 8; ++p) tmem_ld16(col0 + p * 16, v[p]);
            tmem_wait_only();
#pragma unroll
            for (int p = 0; p < 8; ++p) {
              reg_fence(v[p]);
#pragma unroll
              for (int j = 0; j < 16; ++j) x[p][j] = __uint_as_float(v[p][j]);
            }
          }
          if (hf == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(tm_empty0);   // slot copied out
          }
          if (valid < (int)kTile) {                 // keys >= n (ragged last tile)
#pragma unroll
            for (int p = 0; p < 8; ++p)
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (p * 16 + j >= valid) x[p][j] = -INFINITY;
          }
          float pm[8];
#pragma unroll
          for (int p = 0; p < 8; ++p) {
            float a = fmaxf(x[p][0], x[p][1]);
#pragma unroll
            for (int j = 2; j < 16; j += 2) a = fmax3(a, x[p][j], x[p][j + 1]);
            pm[p] = a;
          }
          const float cm =
              fmax3(fmax3(pm[0], pm[1], pm[2]), fmax3(pm[3], pm[4], pm[5]), fmaxf(pm[6], pm[7]));
          const float xm = cm * s2;
          if (xm > m) {
            const float c = ex2(m - xm);
            z.s *= c;
            z.c *= c;
            pend *= c;
            m = xm;
          }
          if (m != -INFINITY) {
            float2 nb[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) nb[j] = make_float2(-m, -m);
            float ps[8];
#pragma unroll
            for (int p = 0; p < 8; ++p) ps[p] = exp2_sum16(x[p], make_float2(s2, s2), nb);
            z.add(pend);
            pend = ((ps[0] + ps[1]) + (ps[2] + ps[3])) + ((ps[4] + ps[5]) + (ps[6] + ps[7]));
          }
        }
      }
      z.add(pend);
      // merge the two warpgroups' statistics of each row
      const int b = k & 1;
      if (wg == 1) {
        if (k >= 2) named_sync(kHalfEmpty + b, 256);
        sm.half[b][warp & 3][lane] = make_float2(m, z.s);
        __syncwarp();
        named_arrive(kHalfFull + b, 256);
      } else {
        named_sync(kHalfFull + b, 256);
        const float2 o = sm.half[b][warp & 3][lane];
        __syncwarp();
        if (k + 2 < nunits) named_arrive(kHalfEmpty + b, 256);
        const float mm = fmaxf(m, o.x);
        float zz = 0.f;
        if (mm != -INFINITY) {
          if (m != -INFINITY) zz += z.s * ex2(m - mm);
          if (o.x != -INFINITY) zz += o.y * ex2(o.x - mm);
        }
        const Unit1& d = sm.unit[k];
        const int rho = d.rho0 + lrow;
        if (S > 1) {
          if (rho < d.rows) part[(d.out + rho) * S + d.split] = make_float2(mm, zz);
        } else if (rho < d.prow) {
          // one key split: the merge's result directly, same arithmetic
          float out = -INFINITY;                      // padding rows: exp2(x + -inf) = 0
          if (rho < d.rows) {
            const float z1 = mm != -INFINITY ? zz * exp2f(0.f) : 0.f;
            out = -(mm + log2f(z1));
          }
          nlse[d.out + rho] = out;
        }
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync();                  // no CTA leaves while the pair's MMAs or copies may touch it
  if (warp == kProducerWarp) {
    tc_fence_after();
    tmem_dealloc_pair(tbase, kTmemCols);
  }
  if (threadIdx.x == 0 && sm.abort) set_status(tb.status, VC_ERR_DEVICE_TIMEOUT);
}

// ---------------------------------------------------------------------------
// merge: minus lse2 per window row into the chunk-padded layout; grid
// (padded rows / 256, n_req)

__global__ void lse_merge_kernel(Shape sh, Tables tb, int S, const float2* __restrict__ part,
                                 const float* __restrict__ lse_nat, float* __restrict__ nlse) {
  dep_wait();                                 // the partial statistics of pass 1
  if (threadIdx.x == 0) dep_launch();
  const Req rq = tb.req[blockIdx.y];
  const int rows = rq.C * rq.cw;              // padded rows of one (layer, KV head)
  const int64_t per = (int64_t)sh.L * sh.Hkv * rows;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= per) return;
  const int p = (int)(i % rows);
  const int grp = (int)(i / rows);
  const int l = grp / sh.Hkv, g = grp % sh.Hkv;
  float out = -INFINITY;                      // padding rows: exp2(x + -inf) = 0
  if (p < sh.G * rq.W) {
    const int64_t o = rq.lse_off + ((int64_t)l * sh.Hq + g * sh.G) * rq.W + p;
    if (lse_nat) {
      out = -lse_nat[o] * kLog2e;
    } else {
      float m = -INFINITY;
      for (int s = 0; s < S; ++s) m = fmaxf(m, part[o * S + s].x);
      float z = 0.f;
      for (int s = 0; s < S; ++s) {
        const float2 q = part[o * S + s];
        if (q.x != -INFINITY) z += q.y * exp2f(q.x - m);
      }
      out = -(m + log2f(z));
    }
  }
  nlse[rq.lsep_off + i] = out;
}

// ---------------------------------------------------------------------------
// pass 2 on CTA pairs
//
// A unit is a tile of 256 keys of a (request, KV head) (128 per CTA, keys in
// TMEM lanes), walked over all layers: per layer its K rows (each CTA its own
// 128 keys, double buffered), then the layer's G*W window rows in C chunks of
// cw <= 256 rows (G*W spread evenly, rounded up to 16, so a 448-row set is two
// chunks of 224, not two of 256; CTA r uses rows r*cw/2 ... of the chunk from a
// 128-row box).  One 2-SM MMA chain (M = 256 keys, N = cw rows, K = 128)
// leaves each key's cw logits in its own CTA's tensor memory.  Every CTA
// also loads the chunk's cw row normalisers into its own shared memory (rows
// past the row set carry -inf and add 0).  Warpgroup wg takes the chunks q
// with q % 2 == wg (TMEM slot wg; q = layer * C + chunk), the cw columns in up
// to two halves of 128.
//
// A launch with few units per resident pair is persistent: the (unit, layer)
// sequence is cut into equal shares, one per pair, so a share may begin and end
// inside a unit and no pair is idle in a last, partly filled wave (worth_sharing).  Whole units
// end in their scores.  The pairs that share a unit leave each layer's column
// sums in the workspace, and the CTA that comes last (a count per unit and CTA
// rank; nobody waits) adds them in layer order: the same additions in the same
// order as for a whole unit, so the scores do not depend on the cuts.  A
// longer sequence, or one without room for those sums, launches one pair per
// unit.
//
// Bound by the consumers, two warps per sub-partition: ~14 cycles a column
// and warp pair where the exp2 unit needs 8 and the packed multiply-adds and
// adds, at 4 cycles each, 8 as well.  Measured (event times), whole units in
// every launch -> now: n = 3,136 (52 units on 76 pairs) 57.5 -> 52.7 us; n = 12,544
// (196 units) 159.4 -> 150.5, layer-specific ranking 141.7 -> 125.0; whole units in
// both: ragged batch 1,218 -> 1,235, 72B shape 4,422 -> 4,315.

constexpr uint32_t kChunkRows = 256;            // window rows per pass-2 chunk (both CTAs)

// One pass-2 consumer step over NP groups of 16 TMEM columns (one key per
// lane, one window row per column) starting at col0: load, optionally free
// the slot (last load of the chunk), then sum exp2(x * s2 + nl[col]) over the
// columns.  NP is a compile-time count so the loads and sums unroll fully.
template <int NP>
__device__ __forceinline__ float colsum_group(uint32_t col0, const float* nl_col, float s2, bool release,
                                              uint32_t tm_empty0, int lane) {
  float x[NP][16];
  {
    uint32_t vv[NP][16];
#pragma unroll
    for (int p = 0; p < NP; ++p) tmem_ld16(col0 + p * 16, vv[p]);
    tmem_wait_only();
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      reg_fence(vv[p]);
#pragma unroll
      for (int j = 0; j < 16; ++j) x[p][j] = __uint_as_float(vv[p][j]);
    }
  }
  if (release) {
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive_cluster(tm_empty0);   // slot copied out
  }
  const float4* nl = reinterpret_cast<const float4*>(nl_col);
  float ps[8];
#pragma unroll
  for (int p = 0; p < 8; ++p) ps[p] = 0.f;
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    float2 nb[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 f = nl[p * 4 + j];
      nb[2 * j] = make_float2(f.x, f.y);
      nb[2 * j + 1] = make_float2(f.z, f.w);
    }
    ps[p] = exp2_sum16(x[p], make_float2(s2, s2), nb);
  }
  return ((ps[0] + ps[1]) + (ps[2] + ps[3])) + ((ps[4] + ps[5]) + (ps[6] + ps[7]));
}
constexpr int kQStagesPair = 4;                 // Q ring of pass 2 (per CTA: 32 KB + 1 KB a stage)

struct Seg2 {                                   // layers [l0, l1) of one unit as this CTA sees it
  int64_t score;                                // first score of this CTA's keys (layer 0)
  int64_t nl;                                   // first row normaliser (layer 0, chunk 0)
  int32_t krow, kstep;                          // K row of this CTA's first key in layer 0; rows per layer
  int32_t qrow, qstep;                          // Qw row of this CTA's half of chunk 0, layer 0; rows per layer
  int32_t nlstep;                               // normalisers per layer
  int32_t keys;                                 // valid keys of this CTA
  int32_t sstep;                                // scores per layer (layer-specific ranking)
  int32_t C, cw;
  int16_t l0, l1, Ls;
  int16_t slot, parts;                          // split unit: its place among the launch's split units, its segments
};

struct P2Smem {
  uint8_t k[2][2][kKBlockBytes];              // this CTA's 128 keys of a layer [item & 1][K-block]
  uint8_t q[kQStagesPair][2][kKBlockBytes];   // this CTA's 128 rows of the chunk [stage][K-block]
  float nlse[kQStagesPair][kChunkRows];       // minus lse2 of all 256 rows of the chunk
  float red[2][2][kTile];                     // [segment & 1][warpgroup][key]
  Seg2 seg[kMaxSegs];
  uint64_t k_full[2];                         // even CTA: both CTAs' keys of the layer landed
  uint64_t k_empty[2];                        // both: the layer's MMAs are done
  uint64_t q_full[kQStagesPair];              // even CTA: both CTAs' rows of the chunk landed
  uint64_t nl_full[kQStagesPair];             // both: this CTA's copy of the normalisers landed
  uint64_t q_empty[kQStagesPair];             // both: MMAs done and this CTA's warpgroup read the normalisers
  uint64_t tm_full[2];                        // both: the slot's logits are ready
  uint64_t tm_empty[2];                       // even CTA: the slot's 8 consumer warps copied it out
  uint64_t mma_done;                          // both: every MMA of the pair is done
  uint64_t never;                             // test support: never completes
  uint64_t peer_done;                         // even CTA: the odd CTA's fill counts landed (8 bytes)
  int2 peer_fills;                            // even CTA: (key, chunk) tiles the odd CTA issued
  uint32_t tmem_base;
  int abort;
  int last;                                   // this CTA finished a split unit last
};

// Counts of finished segments per (split unit, CTA rank), zeroed by pass 1,
// then the split units' column sums [unit][layer][warpgroup][256 keys].
constexpr size_t kSplitCountBytes = sizeof(int32_t) * 2 * kMaxPairs2;
__device__ __forceinline__ float* split_sums(void* scratch, int slot, int Ls, int l, int wg) {
  return reinterpret_cast<float*>(static_cast<uint8_t*>(scratch) + kSplitCountBytes) +
         (((int64_t)slot * Ls + l) * 2 + wg) * kPairKeys;
}

// CUT: the pairs take the shares' segments; else pair p walks unit p.
struct NoShares {};
template <bool CUT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
score_colsum_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                       const __grid_constant__ std::conditional_t<CUT, Shares, NoShares> shares, Shape sh,
                       Tables tb, const float* __restrict__ nlse,
                       float* __restrict__ scores, void* __restrict__ scratch) {
  extern __shared__ uint8_t smem_raw[];
  P2Smem& sm = *reinterpret_cast<P2Smem*>(align1024(smem_raw));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int pair = (int)(blockIdx.x >> 1), npairs = (int)(gridDim.x >> 1);
  const bool per_layer = sh.rank_mode == VC_RANK_PER_LAYER;

  // this pair's segments
  int nsegs = 1;
  if constexpr (CUT) nsegs = min(kMaxSegs, share_segments(shares, pair));
  for (int i = (int)threadIdx.x - 32; i < nsegs; i += kThreads) {   // warp 0 sets up the barriers meanwhile
    if (i < 0) continue;
    int unit = pair;
    if constexpr (CUT) unit = shares.unit[pair] + i;
    const int r = upper_index(tb.unit0_tc2, sh.n_req, (int32_t)unit);
    const Req& rq = tb.req[r];
    ShareSegment part = {unit, 0, rq.Ls, 0, 1};
    if constexpr (CUT) part = share_segment(shares, npairs, pair, i, rq.Ls);
    const int u = unit - tb.unit0_tc2[r];
    const int g = u / rq.tiles, kt = u % rq.tiles;
    const int key0 = kt * (int)kPairKeys + (int)rank * (int)kTile;
    Seg2 d;
    d.Ls = (int16_t)rq.Ls;
    d.l0 = (int16_t)part.l0;
    d.l1 = (int16_t)part.l1;
    d.slot = (int16_t)part.slot;
    d.parts = (int16_t)part.parts;
    d.C = rq.C;
    d.cw = rq.cw;
    d.keys = rq.n - key0;
    d.score = rq.s_off + (int64_t)g * rq.n + key0;
    d.sstep = sh.Hkv * rq.n;
    d.nlstep = sh.Hkv * rq.C * rq.cw;
    d.nl = rq.lsep_off + (int64_t)g * (rq.C * rq.cw);
    d.krow = (int)(rq.kv_off / 128 + (int64_t)g * rq.n) + key0;
    d.kstep = sh.Hkv * rq.n;
    d.qrow = (int)(rq.q_off / 128 + (int64_t)g * sh.G * rq.W) + (int)rank * (rq.cw >> 1);
    d.qstep = sh.Hq * rq.W;
    sm.seg[i] = d;
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sm.k_full[i], 1);
      mbar_init(&sm.k_empty[i], 1);
      mbar_init(&sm.tm_full[i], 1);
      mbar_init(&sm.tm_empty[i], 8);
    }
    for (int i = 0; i < kQStagesPair; ++i) {
      mbar_init(&sm.q_full[i], 1);
      mbar_init(&sm.nl_full[i], 1);
      mbar_init(&sm.q_empty[i], 1 + 4);   // MMA commit + the stage's 4 consumer warps of this CTA
    }
    mbar_init(&sm.mma_done, 1);
    mbar_init(&sm.never, 1);
    mbar_init(&sm.peer_done, 1);
    sm.abort = 0;
    fence_mbar_init();
    if (rank == 0) mbar_arrive_expect_tx(&sm.peer_done, 8);
  }
  if (warp == kProducerWarp) {
    tmem_alloc_pair(&sm.tmem_base, kTmemCols);
    tmem_relinquish_pair();
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync();                  // segments, barriers of both CTAs, TMEM
  tc_fence_after();
  const uint32_t tbase = sm.tmem_base;
  volatile int* abort = &sm.abort;

  if (warp >= 8) {
    give_registers<kOtherRegs>();
    if (warp == kProducerWarp && lane == 0) {
      // ---- TMA producer (both CTAs): K half of a layer, then the layer's row chunks
      prefetch_tmap(&tmQ);
      prefetch_tmap(&tmK);
      int ki = 0, qi = 0;
      bool ok = true, waited = false;
      for (int s = 0; ok && s < nsegs; ++s) {
        const Seg2 d = sm.seg[s];
        for (int l = d.l0; ok && l < d.l1; ++l) {
          const int ks = ki & 1;
          if (!mbar_wait(&sm.k_empty[ks], ((ki >> 1) & 1) ^ 1, abort)) { ok = false; break; }
          if (rank == 0) mbar_arrive_expect_tx(&sm.k_full[ks], 2 * kTileBytes);
          const uint32_t k_full0 = map_to_rank(smem_u32(&sm.k_full[ks]), 0);
          const int ky = d.krow + l * d.kstep;
          tma_load_2d_pair(sm.k[ks][0], &tmK, 0, ky, k_full0);
          tma_load_2d_pair(sm.k[ks][1], &tmK, 64, ky, k_full0);
          ++ki;
          for (int c = 0; c < d.C; ++c) {
            const int qs = qi % kQStagesPair;
            if (!mbar_wait(&sm.q_empty[qs], ((qi / kQStagesPair) & 1) ^ 1, abort)) { ok = false; break; }
            if (rank == 0) mbar_arrive_expect_tx(&sm.q_full[qs], 2 * kTileBytes);
            const uint32_t q_full0 = map_to_rank(smem_u32(&sm.q_full[qs]), 0);
            const int qy = d.qrow + l * d.qstep + c * d.cw;
            tma_load_2d_pair(sm.q[qs][0], &tmQ, 0, qy, q_full0);
            tma_load_2d_pair(sm.q[qs][1], &tmQ, 64, qy, q_full0);
            if (!waited) {
              // the keys and the first rows are inputs and load while the
              // kernel before this one drains; the normalisers are its output
              dep_wait();
              dep_launch();
              waited = true;
            }
            mbar_arrive_expect_tx(&sm.nl_full[qs], (uint32_t)d.cw * 4);
            bulk_load(sm.nlse[qs], nlse + d.nl + (int64_t)l * d.nlstep + c * d.cw, (uint32_t)d.cw * 4, &sm.nl_full[qs]);
            ++qi;
          }
        }
      }
      if (!waited) {                 // no chunk (nothing scored, or an abort)
        dep_wait();
        dep_launch();
      }
      // every copy this CTA started has landed before the pair may leave: the
      // normalisers on this CTA's barriers, the tiles on the even CTA's
      if (rank == 1) report_fills(&sm.peer_fills, &sm.peer_done, ki, qi);
      for (int i = max(0, qi - kQStagesPair); i < qi; ++i)
        drain_wait(&sm.nl_full[i % kQStagesPair], (i / kQStagesPair) & 1);
      if (rank == 0) {
        const int2 f = peer_fills(&sm.peer_done, &sm.peer_fills, make_int2(ki, qi), abort);
        drain_pair_ring(sm.k_full, 2, ki, f.x, kTileBytes);
        drain_pair_ring(sm.q_full, kQStagesPair, qi, f.y, kTileBytes);
      }
    } else if (warp == kMmaWarp && lane == 0 && rank == 0) {
      // ---- MMA issuer (even CTA): D[key][row] = K_tile . Q_chunk^T, 256 x cw
      bool ok = true;
      int ki = 0, qi = 0;
      uint32_t uses[2] = {0u, 0u};                  // chunks of each warpgroup (slot) so far
      for (int s = 0; ok && s < nsegs; ++s) {
        const int C = sm.seg[s].C, l0 = sm.seg[s].l0, l1 = sm.seg[s].l1;
        const uint32_t idesc = idesc_bf16_f32(2 * kTile, (uint32_t)sm.seg[s].cw);
        for (int l = l0; ok && l < l1; ++l, ++ki) {
          const int ks = ki & 1;
          if (!mbar_wait(&sm.k_full[ks], (ki >> 1) & 1, abort)) { ok = false; break; }
          for (int c = 0; c < C; ++c, ++qi) {
            const int qs = qi % kQStagesPair, slot = (l * C + c) & 1;
            const uint32_t use = slot ? uses[1]++ : uses[0]++;
            if (!mbar_wait(&sm.q_full[qs], (qi / kQStagesPair) & 1, abort)) { ok = false; break; }
            if (!mbar_wait(&sm.tm_empty[slot], (use & 1) ^ 1, abort)) { ok = false; break; }
            tc_fence_after();
            const uint32_t d = tbase + (uint32_t)slot * kChunkRows;
  #pragma unroll
            for (int kk = 0; kk < 8; ++kk)
              mma_bf16_pair(d, desc_sw128(smem_u32(sm.k[ks][kk >> 2]) + (kk & 3) * 32),
                            desc_sw128(smem_u32(sm.q[qs][kk >> 2]) + (kk & 3) * 32), idesc, kk ? 1u : 0u);
            mma_commit_pair(&sm.tm_full[slot], 3);
            mma_commit_pair(&sm.q_empty[qs], 3);
          }
          if (ok) mma_commit_pair(&sm.k_empty[ks], 3);
        }
      }
      mma_commit_pair(&sm.mma_done, 3);
      drain_wait(&sm.mma_done, 0);
    } else if (warp == kMmaWarp && lane == 0) {
      // odd CTA: the pair's MMAs (and their arrivals on this CTA's barriers) are done
      drain_wait(&sm.mma_done, 0);
    }
  } else {
    take_registers<kConsumerRegs>();
    if ((sh.test_wait & VC_TEST_WAIT_SCORE_COLSUM) && warp == 0) {
      if (lane == 0 && injected_wait_gives_up(&sm.never)) {
        set_status(tb.status, VC_ERR_DEVICE_TIMEOUT);
        *abort = 1;
      }
      __syncwarp();
    }
    // ---- column sums: one thread per key (= TMEM lane)
    const int wg = warp >> 2;
    const int key = ((warp & 3) << 5) + lane;
    const uint32_t lane_off = (uint32_t)((warp & 3) << 5) << 16;
    const uint32_t tm_empty0 = lane == 0 ? map_to_rank(smem_u32(&sm.tm_empty[wg]), 0) : 0u;
    const float s2 = sh.scale_log2;
    int qi = 0;                                     // chunks so far
    uint32_t use = 0;                               // this warpgroup's chunks so far
    for (int s = 0; s < nsegs; ++s) {
      const int C = sm.seg[s].C, cw = sm.seg[s].cw, Ls = sm.seg[s].Ls;
      const int l0 = CUT ? sm.seg[s].l0 : 0, l1 = CUT ? sm.seg[s].l1 : Ls;
      const int parts = CUT ? sm.seg[s].parts : 1, slot = CUT ? sm.seg[s].slot : 0;
      // Split units' sums and counts go to memory the kernel before this one may be
      // clearing: every consumer is ordered behind it, also one without a chunk
      // whose normalisers it would wait for.
      if (!per_layer && parts > 1) dep_wait();
      const bool valid = key < sm.seg[s].keys;
      float* out = scores + sm.seg[s].score + key;
      const int nhalf = (cw + (int)kTile - 1) / (int)kTile;   // 1 or 2 halves of 128 columns
      // The sum of a group of exp2 terms is ready only once the exp2 unit has
      // worked through the warp's queue, which takes long after the last one
      // is issued.  So nothing waits for a sum right after issuing it: the last
      // half-sum of a chunk stays pending until the next chunk's first half is
      // issued, and a layer is added to the total only after the next layer's
      // chunk is issued.  Layer l accumulates into a[l & 1]; the additions keep
      // their order (halves in order into the layer, layers in order into the
      // total).
      Kahan tot, a0, a1;
      tot.init();
      a0.init();
      a1.init();
      float pend = 0.f;                             // last half-sum of the latest chunk
      int pend_l = -1;                              // its layer (-1: none)
      auto add_to_layer = [&](int l, float x) {
        if (l & 1) a1.add(x);
        else a0.add(x);
      };
      auto flush = [&](int l) {                     // the pending half-sum, if it is layer l's
        if (pend_l == l) {
          add_to_layer(l, pend);
          pend_l = -1;
        }
      };
      auto half_sum = [&](int qs, int hf) -> float {
        const int np = min(8, (cw >> 4) - hf * 8);  // 16-column groups of this half
        const uint32_t col0 = tbase + lane_off + (uint32_t)wg * kChunkRows + (uint32_t)hf * kTile;
        const float* nl = sm.nlse[qs] + hf * (int)kTile;
        const bool rel = hf == nhalf - 1;           // the slot is free after this load
        switch (np) {
          case 8: return colsum_group<8>(col0, nl, s2, rel, tm_empty0, lane);
          case 7: return colsum_group<7>(col0, nl, s2, rel, tm_empty0, lane);
          case 6: return colsum_group<6>(col0, nl, s2, rel, tm_empty0, lane);
          case 5: return colsum_group<5>(col0, nl, s2, rel, tm_empty0, lane);
          case 4: return colsum_group<4>(col0, nl, s2, rel, tm_empty0, lane);
          case 3: return colsum_group<3>(col0, nl, s2, rel, tm_empty0, lane);
          case 2: return colsum_group<2>(col0, nl, s2, rel, tm_empty0, lane);
          default: return colsum_group<1>(col0, nl, s2, rel, tm_empty0, lane);
        }
      };
      // one chunk (layer l) of this warpgroup: wait for its logits and
      // normalisers, issue its exp2 terms, release the normaliser stage
      auto run_chunk = [&](int l) {
        const int qs = qi % kQStagesPair;
        const bool go = __all_sync(0xffffffffu, *abort == 0);
        if (go && warp_wait(&sm.tm_full[wg], use & 1, abort) &&
            warp_wait(&sm.nl_full[qs], (qi / kQStagesPair) & 1, abort)) {
          tc_fence_after();
          const float h0 = half_sum(qs, 0);
          if (pend_l >= 0) {                        // the previous chunk's last half
            add_to_layer(pend_l, pend);
            pend_l = -1;
          }
          if (nhalf == 2) {
            const float h1 = half_sum(qs, 1);
            add_to_layer(l, h0);
            pend = h1;
          } else {
            pend = h0;
          }
          pend_l = l;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.q_empty[qs]);   // this warp is done with the stage's normalisers
        ++use;
      };
      auto run_layer = [&](int l) {
        for (int c = 0; c < C; ++c, ++qi)
          if (((l * C + c) & 1) == wg) run_chunk(l);
      };
      auto layer_total = [&](int l) -> float {      // layer l's sum, its accumulator reset
        flush(l);
        const float t = (l & 1) ? a1.s : a0.s;
        if (l & 1) a1.init();
        else a0.init();
        return t;
      };
      float (*red)[kTile] = sm.red[s & 1];
      if (per_layer) {
        for (int l = l0; l < l1; ++l) {
          run_layer(l);
          red[wg][key] = layer_total(l);
          __syncwarp();
          named_sync(1, 2 * kTile);
          if (wg == 0 && valid) out[(int64_t)l * sm.seg[s].sstep] = red[0][key] + red[1][key];
          named_sync(1, 2 * kTile);
        }
        continue;
      }
      // (Ls == L here: the shared ranking averages every layer)
      auto take = [&](int l) {                      // layer l is complete
        const float t = layer_total(l);
        if (parts == 1) tot.add(t);
        else split_sums(scratch, slot, Ls, l, wg)[rank * kTile + key] = t;
      };
      for (int l = l0; l < l1; ++l) {
        run_layer(l);
        if (l > l0) take(l - 1);
      }
      if (l1 > l0) take(l1 - 1);
      if (parts > 1) {
        // the last of the unit's segments adds up its layers
        __threadfence();
        named_sync(1, 2 * kTile);
        if (threadIdx.x == 0) {
          int32_t* count = static_cast<int32_t*>(scratch) + 2 * slot + rank;
          sm.last = atomicAdd(count, 1) == parts - 1;
          __threadfence();
        }
        named_sync(1, 2 * kTile);
        const bool last = *(volatile int*)&sm.last != 0;
        if (last) {
#pragma unroll 8
          for (int l = 0; l < Ls; ++l)
            tot.add(__ldcg(split_sums(scratch, slot, Ls, l, wg) + rank * kTile + key));
        }
        red[wg][key] = tot.s;
        __syncwarp();
        named_sync(1, 2 * kTile);
        if (!last) continue;
      } else {
        red[wg][key] = tot.s;
        __syncwarp();
        named_sync(1, 2 * kTile);
      }
      if (wg == 0 && valid) *out = (red[0][key] + red[1][key]) / (float)sh.L;
    }
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync();                  // no CTA leaves while the pair's MMAs or copies may touch it
  if (warp == kProducerWarp) {
    tc_fence_after();
    tmem_dealloc_pair(tbase, kTmemCols);
  }
  if (threadIdx.x == 0 && sm.abort) set_status(tb.status, VC_ERR_DEVICE_TIMEOUT);
}

// ---------------------------------------------------------------------------
// host side

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// [rows][128] bf16 tensor, boxes of 128 rows x 64 elements, 128-byte swizzle.
bool make_rows_map(CUtensorMap* m, const void* base, uint64_t rows) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  if (!enc || rows == 0 || rows > 0x7fffffffull) return false;
  cuuint64_t dims[2] = {128, rows};
  cuuint64_t strides[1] = {256};
  cuuint32_t box[2] = {64, kTile};
  cuuint32_t es[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

int score_tc_max_splits() { return 4; }

// CTA pairs of the lse pass that fit on the device at once (pairs must sit on
// one TPC, so this can be below half the SM count).
int score_tc_pair_slots() {
  static int cached[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
  if (cached[dev] > 0) return cached[dev];
  const size_t smem1 = sizeof(P1Smem) + 1024;
  if (cudaFuncSetAttribute(score_lse_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem1) !=
      cudaSuccess)
    return 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, score_lse_tc_kernel, &cfg) != cudaSuccess || n <= 0) {
    cudaGetLastError();
    int sms = 2;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    n = std::max(1, sms / 2);
  }
  cached[dev] = n;
  return n;
}

cudaError_t launch_score_tc(const void* Qw, const void* K, const Shape& sh, const Tables& tb,
                            const TcPlan& tp, float2* part, float* nlse_pad, const float* lse_nat,
                            float* scores, void* scratch, size_t scratch_bytes, cudaStream_t st) {
  CUtensorMap mq, mk;
  if (!make_rows_map(&mq, Qw, tp.q_rows) || !make_rows_map(&mk, K, tp.k_rows))
    return cudaErrorInvalidValue;
  // shared ranking only: a layer-specific score needs no other layer's sums
  const int pairs = std::max(1, score_tc_pair_slots());
  const bool per_layer = sh.rank_mode == VC_RANK_PER_LAYER;
  const int pairs2 = std::min(pairs, kMaxPairs2);
  const bool split = !per_layer && !lse_nat && scratch &&
                     scratch_bytes >= kSplitCountBytes + sizeof(float) * 2 * kPairKeys * (size_t)sh.L *
                                                             (size_t)std::min(tp.units2, pairs2);
  Shares shares;
  const bool whole = !(split || per_layer) || !worth_sharing(tp.units2, pairs2, per_layer) ||
                     !plan_shares(tp.req, tp.n_req, tp.units2, pairs2, &shares) ||
                     (tp.units2 <= pairs2 && !cuts_a_unit(shares, pairs2));
  cudaError_t e;
  if (!lse_nat) {
    const size_t smem1 = sizeof(P1Smem) + 1024;
    e = cudaFuncSetAttribute(score_lse_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem1);
    if (e != cudaSuccess) return e;
    ProfileScope ps("score_lse_tc", st);
    // one launch per slice of at most pairs * kMaxUnits1 units
    const int64_t per_launch = (int64_t)pairs * kMaxUnits1;
    for (int64_t u = 0; u < tp.units1; u += per_launch) {
      const int cnt = (int)std::min<int64_t>(per_launch, tp.units1 - u);
      e = launch_dep(score_lse_tc_kernel, dim3(2 * std::min(pairs, cnt)), dim3(kThreads), smem1, st, mq, mk, sh, tb,
                     tp.S, (int)u, cnt, part, nlse_pad, split ? static_cast<int32_t*>(scratch) : nullptr);
      if (e != cudaSuccess) return e;
    }
  }
  if (lse_nat || tp.S > 1) {
    ProfileScope ps("lse_merge", st);
    e = launch_dep(lse_merge_kernel, dim3((unsigned)((tp.max_prows + 255) / 256), sh.n_req), dim3(256), 0, st,
                   sh, tb, tp.S, static_cast<const float2*>(part), lse_nat, nlse_pad);
    if (e != cudaSuccess) return e;
  }
  if (tp.units2 == 0) return cudaSuccess;      // no layer is scored (layer-specific ranking, all budgets 0)
  const size_t smem2 = sizeof(P2Smem) + 1024;
  auto colsum = [&](auto cut, const auto& cuts, int ctas) -> cudaError_t {
    constexpr bool kCut = decltype(cut)::value;
    e = cudaFuncSetAttribute(score_colsum_tc_kernel<kCut>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2);
    if (e != cudaSuccess) return e;
    ProfileScope ps("score_colsum_tc", st);
    return launch_dep(score_colsum_tc_kernel<kCut>, dim3(ctas), dim3(kThreads), smem2, st, mq, mk, cuts, sh, tb,
                      static_cast<const float*>(nlse_pad), scores, scratch);
  };
  return whole ? colsum(std::false_type{}, NoShares{}, 2 * tp.units2) : colsum(std::true_type{}, shares, 2 * pairs2);
}

}  // namespace vc

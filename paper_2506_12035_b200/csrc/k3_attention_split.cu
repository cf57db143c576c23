// K3 for few (sample, head) items and up to 64 query rows: every key tile of an item on its way at once, and the keys
// split over a cluster of CTAs and over groups of warps.
//
// What bounds it: latency.  One image (2 rows of guidance, 12 or 16 heads) makes 24 or 32 items; a CTA per item with a
// three-slot ring leaves most SMs idle while each of the others walks the 5 (S 320) to 17 (S 1088) key tiles one after
// the other, 0.9 us each.  Here a CTA holds all of its 64-key tiles in shared memory (no ring, no slot to wait for), a
// cluster of up to eight CTAs shares an item where SMs would idle, and nk groups of warps share a CTA's tiles.  Every
// (CTA, group) computes the unnormalised output of its queries over its keys with a reference maximum of its own; the
// partial results go (through distributed shared memory) to the CTA that owns the query row, which merges them in a
// fixed order (Eq. 6-10's merge, bit-reproducible) and stores.  The tiles are prefetched into L2 before the
// dependency wait: the L2 is where a concurrent write-back of fresh rows lands too, so nothing stale can be kept.
// Arithmetic as in the ring kernel (mma.sync m16n8k16, fp32 softmax statistics).  16 heads, head_dim 64, us before -> after:
// 32 items: S 320, 41 rows 6.9 -> 4.5, 5 rows 5.5 -> 3.1; S 1088, 41 rows 17.8 -> 6.8; 160 items, S 320, 41 rows 8.7 -> 7.0.
// Every wait is bounded; all threads of a cluster reach both cluster barriers, whatever happened, and no CTA of a cluster
// stores a row after one of them gave up.
#include <cuda.h>

#include "attention_common.cuh"
#include "kernels.h"
#include "launch_pdl.h"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace marche {

namespace {

using namespace att;

constexpr int kMaxTiles = 12;                            // per CTA
constexpr int kMaxThreads = 512;
constexpr int kFewParts = 5;                             // partial results of a row that are merged without a loop
enum { ST_ATTENTION_SPLIT = 0x24 };

template <bool Q_TMA> struct QueryMaps { CUtensorMap main, tail; };   // columns 0-63 and 64-79 of a head
template <> struct QueryMaps<false> {};

// NQ * nk consumer warps (NQ groups of 16 query rows, nk shares of the CTA's tiles) and a producer warp.  Grid: cs * B * H
// CTAs in clusters of cs.
// Q_TMA: the query rows come by TMA (16-byte aligned rows), for many groups of warps (see the launch).
template <int DH, int NQ, bool Q_TMA>
__global__ void __launch_bounds__(kMaxThreads)
attention_split_kernel(const __grid_constant__ CUtensorMap tmap_kv, const __grid_constant__ CUtensorMap tmap_tail,
                       const __grid_constant__ QueryMaps<Q_TMA> tmap_q,
                       const bf16* __restrict__ q, int ld_q, int n, int S, int H, int B, int cs, int nk, int tiles_max, int q_off,
                       uint16_t* __restrict__ o, bool o_bf16, int* __restrict__ status) {
  using Cfg = AttCfg<DH>;
  constexpr int ROW = DH + 4;                            // a row's partial result: DH sums, maximum, sum of weights
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = ptx::smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  const int own = (NQ * 16 + cs - 1) / cs;               // query rows merged per CTA
  const int n_parts = cs * nk;                           // partial results of a row
  // [n_parts][own][ROW] floats: over the tiles once they are used up, or behind them where other CTAs may be earlier
  // (a query tile, where TMA can address the rows, behind both)
  const uint32_t recv = cs > 1 ? base + (uint32_t)tiles_max * Cfg::STAGE_BYTES : base;
  const uint32_t q_tile = base + (uint32_t)q_off;
  const float* recv_gen = reinterpret_cast<const float*>(smem_raw + (recv - raw));
  __shared__ __align__(8) uint64_t full_bars[kMaxTiles + 1];   // the tiles', the queries'
  __shared__ int abort_flags[2];
  const uint32_t full0 = ptx::smem_u32(full_bars);
  volatile int* abort_flag = abort_flags;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_cons = NQ * nk, wq = warp % NQ, wk = warp / NQ;
  const int g = lane >> 2, tg = lane & 3;
  const int rank = cs > 1 ? (int)ptx::cluster_ctarank() : 0, item = (int)blockIdx.x / cs;
  const int b = item / H, h = item - b * H, D = H * DH;
  const int n_kv = (S + KT - 1) / KT;
  const int kt0 = rank * n_kv / cs, n_tiles = (rank + 1) * n_kv / cs - kt0;
  const float scale_log2 = rsqrtf((float)DH) * 1.4426950408889634f;

  if (threadIdx.x == 0) {
    for (int s = 0; s <= kMaxTiles; ++s) ptx::mbar_init(full0 + 8u * s, 1);
    abort_flags[0] = abort_flags[1] = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
  }
  if (warp == n_cons && lane == 0) {
    ptx::prefetch_tensormap(&tmap_kv);
    for (int i = 0; i < n_tiles; ++i) {
      ptx::tma_prefetch_l2_3d(&tmap_kv, h * DH, (kt0 + i) * KT, b);
      ptx::tma_prefetch_l2_3d(&tmap_kv, h * DH, (kt0 + i) * KT, B + b);
    }
  }
  __syncwarp();
  if (cs > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  __syncthreads();
  pdl_sync();                                            // everything above overlaps the previous kernel's tail

  bool ok = true;
  float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};   // maximum of the RAW logits, sum of the weights
  float oacc[Cfg::ONT][4];
#pragma unroll
  for (int j = 0; j < Cfg::ONT; ++j) oacc[j][0] = oacc[j][1] = oacc[j][2] = oacc[j][3] = 0.f;
  const bool warp_active = warp < n_cons && wq * 16 < n;
  if (warp == n_cons) {
    if (lane == 0) {
      if constexpr (Q_TMA) {
        const uint32_t bar = full0 + 8u * kMaxTiles;
        ptx::mbar_expect_tx(bar, (uint32_t)(NQ * 16 * DH * 2));
        ptx::tma_load_3d(q_tile, &tmap_q.main, h * DH, 0, b, bar);
        if (DH > 64) ptx::tma_load_3d(q_tile + KT * 128, &tmap_q.tail, h * DH + 64, 0, b, bar);
      }
      for (int i = 0; i < n_tiles; ++i) {
        const uint32_t dst = base + i * Cfg::STAGE_BYTES, bar = full0 + 8u * i;
        ptx::mbar_expect_tx(bar, Cfg::STAGE_BYTES);
        ptx::tma_load_3d(dst, &tmap_kv, h * DH, (kt0 + i) * KT, b, bar);
        if (DH > 64) ptx::tma_load_3d(dst + KT * 128, &tmap_tail, h * DH + 64, (kt0 + i) * KT, b, bar);
        ptx::tma_load_3d(dst + Cfg::TILE_BYTES, &tmap_kv, h * DH, (kt0 + i) * KT, B + b, bar);
        if (DH > 64) ptx::tma_load_3d(dst + Cfg::TILE_BYTES + KT * 128, &tmap_tail, h * DH + 64, (kt0 + i) * KT, B + b, bar);
      }
    }
    __syncwarp();
  } else if (warp_active) {
    uint32_t qf[Cfg::KSTEPS][4];                         // this warp's 16 query rows as A fragments
    if constexpr (Q_TMA) {
      ok = ptx::mbar_wait(full0 + 8u * kMaxTiles, 0, abort_flag);
#pragma unroll
      for (int kk = 0; kk < Cfg::KSTEPS; ++kk)
        ldsm_x4(q_tile + kv_off<DH>(wq * 16 + (lane & 15), 2 * kk + (lane >> 4)), qf[kk][0], qf[kk][1], qf[kk][2], qf[kk][3]);
    } else {
      const int r0 = wq * 16 + g, r1 = r0 + 8;
      const bf16* q0 = q + ((size_t)b * n + r0) * ld_q + h * DH;
      const bf16* q1 = q + ((size_t)b * n + r1) * ld_q + h * DH;
#pragma unroll
      for (int kk = 0; kk < Cfg::KSTEPS; ++kk) {
        qf[kk][0] = r0 < n ? *reinterpret_cast<const uint32_t*>(q0 + kk * 16 + 2 * tg) : 0u;
        qf[kk][1] = r1 < n ? *reinterpret_cast<const uint32_t*>(q1 + kk * 16 + 2 * tg) : 0u;
        qf[kk][2] = r0 < n ? *reinterpret_cast<const uint32_t*>(q0 + kk * 16 + 8 + 2 * tg) : 0u;
        qf[kk][3] = r1 < n ? *reinterpret_cast<const uint32_t*>(q1 + kk * 16 + 8 + 2 * tg) : 0u;
      }
    }
    for (int i = wk; i < n_tiles && ok; i += nk) {
      if (!ptx::mbar_wait(full0 + 8u * i, 0, abort_flag)) { ok = false; break; }
      const uint32_t k_tile = base + i * Cfg::STAGE_BYTES, v_tile = k_tile + Cfg::TILE_BYTES;
      // ---- raw logits of 16 rows x 64 keys
      float sacc[8][4];
#pragma unroll
      for (int j = 0; j < 8; ++j) sacc[j][0] = sacc[j][1] = sacc[j][2] = sacc[j][3] = 0.f;
#pragma unroll
      for (int kk = 0; kk < Cfg::KSTEPS; ++kk) {
#pragma unroll
        for (int jp = 0; jp < 4; ++jp) {
          const int mi = lane >> 3;
          const int key = 8 * (2 * jp + (mi >> 1)) + (lane & 7);
          uint32_t b0, b1, b2, b3;
          ldsm_x4(k_tile + kv_off<DH>(key, 2 * kk + (mi & 1)), b0, b1, b2, b3);
          mma_bf16(sacc[2 * jp], qf[kk], b0, b1);
          mma_bf16(sacc[2 * jp + 1], qf[kk], b2, b3);
        }
      }
      const int t_base = (kt0 + i) * KT;
      if (t_base + KT > S) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (t_base + 8 * j + 2 * tg + (e & 1) >= S) sacc[j][e] = -INFINITY;
      }
      // ---- online softmax; every tile has a key below S, so the maxima are finite
      float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        mx[0] = fmaxf(mx[0], fmaxf(sacc[j][0], sacc[j][1]));
        mx[1] = fmaxf(mx[1], fmaxf(sacc[j][2], sacc[j][3]));
      }
      float corr[2], neg_ms[2], rs[2] = {0.f, 0.f};
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
        const float m_new = fmaxf(m_run[r], mx[r]);
        corr[r] = ex2_approx((m_run[r] - m_new) * scale_log2);
        m_run[r] = m_new;
        neg_ms[r] = -m_new * scale_log2;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float p = ex2_approx(fmaf(sacc[j][e], scale_log2, neg_ms[e >> 1]));
          sacc[j][e] = p;
          rs[e >> 1] += p;
        }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        rs[r] += __shfl_xor_sync(0xffffffffu, rs[r], 1);
        rs[r] += __shfl_xor_sync(0xffffffffu, rs[r], 2);
        l_run[r] = l_run[r] * corr[r] + rs[r];
      }
#pragma unroll
      for (int j = 0; j < Cfg::ONT; ++j) {
        oacc[j][0] *= corr[0]; oacc[j][1] *= corr[0];
        oacc[j][2] *= corr[1]; oacc[j][3] *= corr[1];
      }
      // ---- O += P V
#pragma unroll
      for (int k2 = 0; k2 < KT / 16; ++k2) {
        uint32_t pf[4];
        pf[0] = pack_bf16x2(sacc[2 * k2][0], sacc[2 * k2][1]);
        pf[1] = pack_bf16x2(sacc[2 * k2][2], sacc[2 * k2][3]);
        pf[2] = pack_bf16x2(sacc[2 * k2 + 1][0], sacc[2 * k2 + 1][1]);
        pf[3] = pack_bf16x2(sacc[2 * k2 + 1][2], sacc[2 * k2 + 1][3]);
#pragma unroll
        for (int jd = 0; jd < Cfg::ONT; jd += 2) {
          const int mi = lane >> 3;
          const int key = 16 * k2 + 8 * (mi & 1) + (lane & 7);
          uint32_t b0, b1, b2, b3;
          ldsm_x4_trans(v_tile + kv_off<DH>(key, jd + (mi >> 1)), b0, b1, b2, b3);
          mma_bf16(oacc[jd], pf, b0, b1);
          mma_bf16(oacc[jd + 1], pf, b2, b3);
        }
      }
    }
  }
  if (!ok && lane == 0) {
    *(volatile int*)status = ST_ATTENTION_SPLIT;
    // let copies already issued land before the CTA's shared memory is released
    for (int i = 0; i < n_tiles; ++i) ptx::mbar_wait(full0 + 8u * i, 0, abort_flag + 1, 20000000LL);
    if (Q_TMA) ptx::mbar_wait(full0 + 8u * kMaxTiles, 0, abort_flag + 1, 20000000LL);
  }

  if (n_parts == 1) {
    if (warp_active && ok) {
      const float f0 = 1.0f / l_run[0], f1 = 1.0f / l_run[1];
      const int r0 = wq * 16 + g, r1 = r0 + 8;
      uint16_t* o0 = o + ((size_t)b * n + r0) * D + h * DH + 2 * tg;
      uint16_t* o1 = o + ((size_t)b * n + r1) * D + h * DH + 2 * tg;
#pragma unroll
      for (int j = 0; j < Cfg::ONT; ++j) {
        if (r0 < n) *reinterpret_cast<uint32_t*>(o0 + 8 * j) = pack_a16x2(oacc[j][0] * f0, oacc[j][1] * f0, o_bf16);
        if (r1 < n) *reinterpret_cast<uint32_t*>(o1 + 8 * j) = pack_a16x2(oacc[j][2] * f1, oacc[j][3] * f1, o_bf16);
      }
    }
  } else {
    // ---- partial results to the owners of the rows
    if (cs > 1) {
      __syncwarp();                                      // (lane 0 may have been waiting for copies)
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");                // every CTA of the cluster has started
      if (!ok) ptx::cluster_raise(ptx::smem_u32(abort_flags), cs);                       // nobody merges what is missing
    } else {
      __syncthreads();                                   // the tiles are used up
    }
    if (warp_active && ok) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int row = wq * 16 + g + 8 * r;
        if (row < n) {
          const int owner = cs > 1 ? row / own : 0;
          uint32_t dst = recv + 4u * (uint32_t)(((rank * nk + wk) * own + row - owner * own) * ROW);
          if (cs > 1) dst = ptx::mapa(dst, (uint32_t)owner);
#pragma unroll
          for (int j = 0; j < Cfg::ONT; ++j)
            asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(dst + 4u * (8 * j + 2 * tg)), "f"(oacc[j][2 * r]),
                         "f"(oacc[j][2 * r + 1]) : "memory");
          if (tg == 0)
            asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(dst + 4u * DH), "f"(m_run[r]), "f"(l_run[r])
                         : "memory");
        }
      }
    }
    if (cs > 1) {
      __syncwarp();
      ptx::cluster_sync_all();
    } else {
      __syncthreads();
    }
    // ---- merge, in rank order: one thread per four columns of a row this CTA owns
    if (!*abort_flag) {
      const int stride = own * ROW;
      for (int e = threadIdx.x; e < own * (DH / 4); e += (int)blockDim.x) {
        const int j = e / (DH / 4), c = e % (DH / 4) * 4, row = rank * own + j;
        if (row >= n) continue;
        const float* p = recv_gen + j * ROW;
        float m = -INFINITY, l = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        auto add = [&](float w, float l_s, const float4& v) {
          l = fmaf(w, l_s, l);
          acc.x = fmaf(w, v.x, acc.x); acc.y = fmaf(w, v.y, acc.y);
          acc.z = fmaf(w, v.z, acc.z); acc.w = fmaf(w, v.w, acc.w);
        };
        if constexpr (Q_TMA) {                        // all loads at once (a loop of loads took 2500 cycles for five parts)
          float2 ml[kFewParts];
          float4 v[kFewParts];
#pragma unroll
          for (int s = 0; s < kFewParts; ++s) {
            ml[s] = s < n_parts ? *reinterpret_cast<const float2*>(p + s * stride + DH) : make_float2(-INFINITY, 0.f);
            v[s] = s < n_parts ? *reinterpret_cast<const float4*>(p + s * stride + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            m = fmaxf(m, ml[s].x);
          }
#pragma unroll
          for (int s = 0; s < kFewParts; ++s) add(ex2_approx((ml[s].x - m) * scale_log2), ml[s].y, v[s]);
        } else {
          for (int s = 0; s < n_parts; ++s) m = fmaxf(m, p[s * stride + DH]);
          for (int s = 0; s < n_parts; ++s)
            add(ex2_approx((p[s * stride + DH] - m) * scale_log2), p[s * stride + DH + 1], *reinterpret_cast<const float4*>(p + s * stride + c));
        }
        const float f = 1.0f / l;
        uint2 u;
        u.x = pack_a16x2(acc.x * f, acc.y * f, o_bf16);
        u.y = pack_a16x2(acc.z * f, acc.w * f, o_bf16);
        *reinterpret_cast<uint2*>(o + ((size_t)b * n + row) * D + h * DH + c) = u;
      }
    }
  }
}

template <int DH, int NQ, bool Q_TMA>
cudaError_t launch_split(const CUtensorMap& tm, const CUtensorMap& tail, const bf16* q, int ld_q, int B, int n, int S, int H,
                         int cs, int nk, uint16_t* o, bool o_bf16, int* status, cudaStream_t st) {
  const int n_kv = (S + KT - 1) / KT, tiles = (n_kv + cs - 1) / cs, own = (NQ * 16 + cs - 1) / cs, threads = (NQ * nk + 1) * 32;
  const size_t ring = (size_t)tiles * AttCfg<DH>::STAGE_BYTES, recv = cs * nk > 1 ? (size_t)cs * nk * own * (DH + 4) * 4 : 0;
  const size_t used = cs > 1 ? ring + recv : (ring > recv ? ring : recv);
  const size_t q_off = (used + 1023) / 1024 * 1024, smem = 1024 + (Q_TMA ? q_off + AttCfg<DH>::TILE_BYTES : used);
  QueryMaps<Q_TMA> tq;
  if constexpr (Q_TMA) {
    const uint64_t dims[3] = {(uint64_t)ld_q, (uint64_t)n, (uint64_t)B};
    const uint64_t strides[2] = {(uint64_t)ld_q * 2, (uint64_t)n * ld_q * 2};
    const uint32_t box[3] = {64, NQ * 16, 1}, box_tail[3] = {16, NQ * 16, 1};
    if (!tma_make_map_bf16(&tq.main, q, 3, dims, strides, box, true)) return cudaErrorInvalidValue;
    tq.tail = tq.main;
    if (DH > 64 && !tma_make_map_bf16(&tq.tail, q, 3, dims, strides, box_tail, false, false, true)) return cudaErrorInvalidValue;
  }
  if (tiles > kMaxTiles || threads > kMaxThreads || smem > 226 * 1024) return cudaErrorInvalidValue;
  static size_t smem_set[kMaxDevices] = {};
  cudaError_t e = ensure_dynamic_smem(attention_split_kernel<DH, NQ, Q_TMA>, smem, smem_set);
  if (e != cudaSuccess) return e;
  return launch_pdl_cluster(attention_split_kernel<DH, NQ, Q_TMA>, dim3(cs * B * H), dim3(threads), smem, cs, st, tm, tail, tq, q, ld_q, n, S, H, B, cs, nk, tiles, (int)q_off, o, o_bf16, status);
}

}  // namespace

// How an item of this shape is split: cs CTAs, nk groups of consumer warps in each.  False: shared memory cannot hold it.
bool attention_split_plan(int n, int S, int dh, int items, int* cs, int* nk) {
  const int n_kv = (S + KT - 1) / KT, nq = (n + 15) / 16, stage = 4 * KT * dh;
  if (n < 1 || n > 64 || (dh != 64 && dh != 80)) return false;
  // CTAs per item while the launch still is one CTA per SM or less.  The exchange through the cluster costs about 1.3 us,
  // two or three key tiles of a warp (S 320, 41 rows, 16 heads: 32 items 4.5 us on pairs and 4.8 on single CTAs, 64 items
  // 4.8 either way, 128 items 7.3 and 5.3; S 1088: 6.8 us on four, 7.1 on two CTAs at 32 items).
  int c = 1;
  if (n_kv > (nq == 1 ? 5 : 3))
    while (c < 4 && 2 * c * items <= device_sm_count()) c *= 2;
  // (... four query warps at head_dim 80 over five tiles or fewer: where clusters would take more than half of the SMs, single
  // CTAs do better.  64 rows, S 320, eight blocks of a step: 64 items 342 us on pairs, 315 on one, mma.sync kernel 320; 32 items
  // 295 either way; 16 items on four CTAs 6.4 us against 6.7 back to back.)
  if (dh == 80 && nq == 4 && n_kv <= 5 && 2 * c * items > device_sm_count()) c = 1;
  // Two or three groups of query rows over four or five tiles: a single CTA whose groups of warps take a tile each, in place of clusters of
  // four (up to a quarter of the SMs in items) and of two.  A block of a step, us, clusters and single CTAs: five tiles, 43 rows: 32 items
  // (of four) 33.5 and 32.1, 48 items (of two) 34.4 and 33.7, 72 items 34.3 and 33.6, 20 rows, 64 items 32.8 and 30.5; four tiles, 43 rows:
  // 32 items 31.9 and 31.3, 48 items 30.7 and 29.1, 72 items 33.7 and 32.6; head_dim 80, 43 rows, 32 items: five tiles 39.2 and 36.7, four
  // 37.4 and 36.0.  (Back to back, without the launches around it, four tiles of 32 items are slower: 4.0 and 4.2, head_dim 80 4.7 and 5.2.)
  // With fewer items clusters of four do better (43 rows, 24 items 26.6 and 27.2); 25 to 31 were not measured.  At head_dim 80 three groups
  // from 49 items on stay on pairs of CTAs.
  if ((nq == 2 || nq == 3) && (n_kv == 4 || n_kv == 5) && items > 28 && 2 * items <= device_sm_count() && !(dh == 80 && nq == 3 && items > 48)) {
    *cs = 1;
    *nk = n_kv;
    return true;
  }
  while (c < 8 && (n_kv + c - 1) / c > (dh == 64 ? 10 : 8)) c *= 2;
  const int tiles = (n_kv + c - 1) / c;
  if (tiles > kMaxTiles || tiles * stage > 160 * 1024) return false;
  // Warps beyond the query groups: free where the merge over the cluster happens anyway; in a single CTA, with the queries by loads and the
  // merge in a loop, they pay for one group (S 320, 5 rows: 4.5 -> 3.1 us) and two groups of queries with four tiles or more, not for
  // three (4.8 -> 5.3).
  int k = 1;
  if (nq == 1) k = tiles < 5 ? tiles : 5;
  else if ((c > 1 && tiles > 1) || (nq == 2 && tiles > 3)) k = 2;
  *cs = c;
  *nk = k;
  return true;
}

// Where it beats the other kernels (us, 45 rows unless stated): always below one CTA per SM (S 320: 6.9 -> 4.5 at 32 items;
// S 1088: 17.8 -> 6.8); up to two per SM for five key tiles (288 items: 9.6 -> 8.2; 384 items, 60 rows: 13.5 against 12.5 of
// the tcgen05 kernel); for three tiles, which leave room for four CTAs, up to four per SM (512 items, 20 rows: 7.8 -> 7.0; 576
// items, 60 rows: 11.2 either way) and with three groups of queries at head_dim 64 without limit (2048 items: 29.7 -> 26.6).
// With two tiles and up to 32 rows up to three and a half items per SM (eight blocks of a step, 24 rows: 384 items 301 and 309 with
// the persistent kernel, 512 items 350 and 355, 576 items 386 and 372).  At head_dim 80 up to one and a half items per SM with 33
// rows or more (S 320: 192 items 9.6 against 9.9, 288 items 11.5 and 10.4), and up to one and three quarters with up to 16 rows of
// three tiles (eight blocks: 256 items, 8 rows 285 and 298, 288 items, 12 rows 325 and 322).
bool attention_split_wins(int n, int S, int dh, int items) {
  int cs, nk;
  if (!attention_split_plan(n, S, dh, items, &cs, &nk)) return false;
  const int n_kv = (S + KT - 1) / KT, nq = (n + 15) / 16, sms = device_sm_count();
  if (items * cs <= sms) return true;
  if (cs > 1 || n_kv > 5) return false;
  if (dh == 80 && nq >= 3) return 2 * items <= 3 * sms;
  if (dh == 80 && nq == 1 && n_kv == 3) return 4 * items <= 7 * sms;
  if (dh == 64 && n_kv <= 3) return nq == 3 || 2 * items <= (n_kv == 2 && nq <= 2 ? 7 : 8) * sms;
  return items <= 2 * sms;
}

cudaError_t launch_attention_split(const void* q, int ld_q, int B, int n, int S, int H, int dh, const void* cache_layer,
                                   void* o, bool o_bf16, int* status, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  int cs, nk;
  if (!attention_split_plan(n, S, dh, B * H, &cs, &nk) || ld_q % 2 || ((uintptr_t)q & 3) || ((uintptr_t)cache_layer & 15) || ((uintptr_t)o & 15))
    return cudaErrorInvalidValue;
  const int D = H * dh;
  CUtensorMap tm, tail;
  const uint64_t dims[3] = {(uint64_t)D, (uint64_t)S, (uint64_t)2 * B};
  const uint64_t strides[2] = {(uint64_t)D * 2, (uint64_t)S * D * 2};
  const uint32_t box[3] = {64, KT, 1};                   // columns 0-63 of a head: 128-byte rows, swizzled
  if (!tma_make_map_bf16(&tm, cache_layer, 3, dims, strides, box, true)) return cudaErrorInvalidValue;
  tail = tm;
  if (dh == 80) {                                        // columns 64-79: 32-byte rows, 32-byte swizzle
    const uint32_t box_tail[3] = {16, KT, 1};
    if (!tma_make_map_bf16(&tail, cache_layer, 3, dims, strides, box_tail, false, false, true)) return cudaErrorInvalidValue;
  }
  const int nq = (n + 15) / 16;
  // Groups of warps for every tile: the queries by TMA, 700 cycles earlier in registers than by loads of four bytes, and a merge without
  // loops (up to five partial results).  With fewer groups the loads overlap the wait for the tiles and the larger kernel costs
  // (120 items, 43 rows on single CTAs: a block 36.4 -> 37.1 us).
  if (cs == 1 && nk > 2 && nk <= kFewParts && (nq == 2 || nq == 3) && ld_q % 8 == 0 && ((uintptr_t)q & 15) == 0) {
    if (dh == 64)
      return nq == 2 ? launch_split<64, 2, true>(tm, tail, (const bf16*)q, ld_q, B, n, S, H, cs, nk, (uint16_t*)o, o_bf16, status, st)
                     : launch_split<64, 3, true>(tm, tail, (const bf16*)q, ld_q, B, n, S, H, cs, nk, (uint16_t*)o, o_bf16, status, st);
    return nq == 2 ? launch_split<80, 2, true>(tm, tail, (const bf16*)q, ld_q, B, n, S, H, cs, nk, (uint16_t*)o, o_bf16, status, st)
                   : launch_split<80, 3, true>(tm, tail, (const bf16*)q, ld_q, B, n, S, H, cs, nk, (uint16_t*)o, o_bf16, status, st);
  }
#define MARCHE_SPLIT_CASE(DH_, NW_) \
  if (dh == DH_ && nq == NW_)       \
    return launch_split<DH_, NW_, false>(tm, tail, (const bf16*)q, ld_q, B, n, S, H, cs, nk, (uint16_t*)o, o_bf16, status, st);
  MARCHE_SPLIT_CASE(64, 1) MARCHE_SPLIT_CASE(64, 2) MARCHE_SPLIT_CASE(64, 3) MARCHE_SPLIT_CASE(64, 4)
  MARCHE_SPLIT_CASE(80, 1) MARCHE_SPLIT_CASE(80, 2) MARCHE_SPLIT_CASE(80, 3) MARCHE_SPLIT_CASE(80, 4)
#undef MARCHE_SPLIT_CASE
  return cudaErrorInvalidValue;
}

}  // namespace marche

// K3, relevance scores alone (Section 4.2): per key, the sum over the generating tokens' queries of the softmax weight.
//
// Only a few of the active rows generate (at most a seventh of them in the middle of a run, two of 320 in its first step),
// but a flavour of the attention that also sums weights has to take every row twice over the keys, since a weight is
// final only once the row's maximum and sum are.  So the scoring block runs the plain attention for its output, and this
// kernel for the generating rows: it picks them by their flags, holds all K tiles of the (sample, head) item in shared
// memory (V is not needed), and takes the rows through Q K^T twice, first for maximum and sum, then for the weights.
// With 16 generating rows or fewer four warps share the tiles, else two and two.  Weights are added over the 16 rows of a
// warp by shuffles and over row groups in a fixed order: bit-reproducible.  Every wait is bounded.
// Scoring block, us, one kernel -> plain attention and this one: 64 x 16 items, S 1088, 151 rows of which 21 generate
// 387 -> 281; 128 x 16, S 320, 320 rows of which 2 generate 238 -> 174; 2 x 12, S 320, 10 rows of which 5 generate 16.1 -> 9.7.
#include <cuda.h>

#include "attention_common.cuh"
#include "kernels.h"
#include "launch_pdl.h"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace marche {

namespace {

using namespace att;

constexpr int kWarps = 4, kThreads = (kWarps + 1) * 32;  // consumers and a producer warp
constexpr int kGroups = 2;                               // groups of 16 rows taken at a time
constexpr int kMaxTiles = 32;                            // S <= 2048
enum { ST_ATTENTION_SCORES = 0x25 };

// Raw logits of 16 rows x 64 keys; keys beyond S become -inf.
template <int DH>
MARCHE_DEVINL void logits(float (&s)[8][4], const uint32_t (&qf)[AttCfg<DH>::KSTEPS][4], uint32_t k_tile, int t_base, int S,
                          int lane) {
#pragma unroll
  for (int j = 0; j < 8; ++j) s[j][0] = s[j][1] = s[j][2] = s[j][3] = 0.f;
#pragma unroll
  for (int kk = 0; kk < AttCfg<DH>::KSTEPS; ++kk) {
#pragma unroll
    for (int jp = 0; jp < 4; ++jp) {
      const int mi = lane >> 3, key = 8 * (2 * jp + (mi >> 1)) + (lane & 7);
      uint32_t b0, b1, b2, b3;
      ldsm_x4(k_tile + kv_off<DH>(key, 2 * kk + (mi & 1)), b0, b1, b2, b3);
      mma_bf16(s[2 * jp], qf[kk], b0, b1);
      mma_bf16(s[2 * jp + 1], qf[kk], b2, b3);
    }
  }
  if (t_base + KT > S) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (t_base + 8 * j + 2 * (lane & 3) + (e & 1) >= S) s[j][e] = -INFINITY;
  }
}

MARCHE_DEVINL void consumers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kWarps * 32) : "memory"); }

template <int DH>
__global__ void __launch_bounds__(kThreads)
attention_scores_kernel(const __grid_constant__ CUtensorMap tmap_k, const __grid_constant__ CUtensorMap tmap_tail,
                        const bf16* __restrict__ q, int ld_q, int n, int S, int H, const uint8_t* __restrict__ is_new,
                        float* __restrict__ score_partial, int* __restrict__ status) {
  using Cfg = AttCfg<DH>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = ptx::smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;
  const int n_kv = (S + KT - 1) / KT;
  float* colsum = reinterpret_cast<float*>(smem_raw + (base - raw) + n_kv * Cfg::TILE_BYTES);   // [kGroups][S]
  uint16_t* rows = reinterpret_cast<uint16_t*>(colsum + kGroups * S);                            // the generating rows
  __shared__ __align__(8) uint64_t full_bars[kMaxTiles];
  __shared__ float2 stats[kWarps][16];                   // maximum and sum of a row over a warp's tiles
  __shared__ int counts[kWarps];
  __shared__ int abort_flags[2];
  const uint32_t full0 = ptx::smem_u32(full_bars);
  volatile int* abort_flag = abort_flags;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, tg = lane & 3;
  const int b = blockIdx.x / H, h = blockIdx.x - b * H;
  const float scale_log2 = rsqrtf((float)DH) * 1.4426950408889634f;

  if (threadIdx.x == 0) {
    for (int s = 0; s < n_kv; ++s) ptx::mbar_init(full0 + 8u * s, 1);
    abort_flags[0] = abort_flags[1] = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
  }
  for (int t = threadIdx.x; t < kGroups * S; t += kThreads) colsum[t] = 0.f;
  __syncthreads();
  pdl_sync();

  // ---- the list of generating rows: every warp counts and then writes those of a quarter of the rows
  const uint8_t* flags = is_new + (size_t)b * n;
  const int chunk = (n + 32 * kWarps - 1) / (32 * kWarps) * 32, r_begin = warp * chunk, r_end = min(r_begin + chunk, n);
  if (warp < kWarps) {
    int c = 0;
    for (int r = r_begin; r < r_end; r += 32) c += __popc(__ballot_sync(0xffffffffu, r + lane < r_end && flags[r + lane]));
    if (lane == 0) counts[warp] = c;
  } else if (ptx::elect_one()) {
    ptx::prefetch_tensormap(&tmap_k);
    for (int i = 0; i < n_kv; ++i) {
      const uint32_t dst = base + i * Cfg::TILE_BYTES, bar = full0 + 8u * i;
      ptx::mbar_expect_tx(bar, Cfg::TILE_BYTES);
      ptx::tma_load_3d(dst, &tmap_k, h * DH, i * KT, b, bar);
      if (DH > 64) ptx::tma_load_3d(dst + KT * 128, &tmap_tail, h * DH + 64, i * KT, b, bar);
    }
  }
  __syncthreads();
  int n_rows = 0;
  if (warp < kWarps) {
    int at = 0;
    for (int w = 0; w < kWarps; ++w) { if (w < warp) at += counts[w]; n_rows += counts[w]; }
    for (int r = r_begin; r < r_end; r += 32) {
      const bool f = r + lane < r_end && flags[r + lane];
      const unsigned m = __ballot_sync(0xffffffffu, f);
      if (f) rows[at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(r + lane);
      at += __popc(m);
    }
  }
  __syncthreads();

  bool ok = true;
  if (warp < kWarps) {
    for (int g0 = 0; g0 < n_rows; g0 += 16 * kGroups) {
      const int ks = n_rows - g0 > 16 ? kWarps / kGroups : kWarps;   // warps that share a group's tiles
      const int wr = warp / ks, wk = warp - wr * ks;
      const int i0 = g0 + wr * 16 + g, i1 = i0 + 8;
      const bool v0 = i0 < n_rows, v1 = i1 < n_rows;
      uint32_t qf[Cfg::KSTEPS][4];
      float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
      const bf16* q0 = q + ((size_t)b * n + (v0 ? rows[i0] : 0)) * ld_q + h * DH;
      const bf16* q1 = q + ((size_t)b * n + (v1 ? rows[i1] : 0)) * ld_q + h * DH;
#pragma unroll
      for (int kk = 0; kk < Cfg::KSTEPS; ++kk) {
        qf[kk][0] = v0 ? *reinterpret_cast<const uint32_t*>(q0 + kk * 16 + 2 * tg) : 0u;
        qf[kk][1] = v1 ? *reinterpret_cast<const uint32_t*>(q1 + kk * 16 + 2 * tg) : 0u;
        qf[kk][2] = v0 ? *reinterpret_cast<const uint32_t*>(q0 + kk * 16 + 8 + 2 * tg) : 0u;
        qf[kk][3] = v1 ? *reinterpret_cast<const uint32_t*>(q1 + kk * 16 + 8 + 2 * tg) : 0u;
      }
      // ---- maximum and sum over this warp's tiles
      for (int kt = wk; kt < n_kv && ok; kt += ks) {
        if (!ptx::mbar_wait(full0 + 8u * kt, 0, abort_flag)) { ok = false; break; }
        float s[8][4];
        logits<DH>(s, qf, base + kt * Cfg::TILE_BYTES, kt * KT, S, lane);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          float mx = -INFINITY, sum = 0.f;
#pragma unroll
          for (int j = 0; j < 8; ++j) mx = fmaxf(mx, fmaxf(s[j][2 * r], s[j][2 * r + 1]));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
          const float m_new = fmaxf(m_run[r], mx), neg = -m_new * scale_log2;
#pragma unroll
          for (int j = 0; j < 8; ++j)
            sum += ex2_approx(fmaf(s[j][2 * r], scale_log2, neg)) + ex2_approx(fmaf(s[j][2 * r + 1], scale_log2, neg));
          sum += __shfl_xor_sync(0xffffffffu, sum, 1);
          sum += __shfl_xor_sync(0xffffffffu, sum, 2);
          l_run[r] = l_run[r] * ex2_approx((m_run[r] - m_new) * scale_log2) + sum;
          m_run[r] = m_new;
        }
      }
      if (tg == 0) {
        stats[warp][g] = make_float2(m_run[0], l_run[0]);
        stats[warp][g + 8] = make_float2(m_run[1], l_run[1]);
      }
      consumers_sync();
      float neg[2], inv[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float m = -INFINITY, l = 0.f;
        for (int w = 0; w < ks; ++w) m = fmaxf(m, stats[wr * ks + w][g + 8 * r].x);
        for (int w = 0; w < ks; ++w) {
          const float2 x = stats[wr * ks + w][g + 8 * r];
          l += x.y * ex2_approx((x.x - m) * scale_log2);
        }
        neg[r] = -m * scale_log2;
        inv[r] = (r ? v1 : v0) ? 1.0f / l : 0.f;
      }
      // ---- final weights, added over the 16 rows
      float* cs = colsum + wr * S;
      for (int kt = wk; kt < n_kv && ok; kt += ks) {
        float s[8][4];
        logits<DH>(s, qf, base + kt * Cfg::TILE_BYTES, kt * KT, S, lane);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          float c0 = ex2_approx(fmaf(s[j][0], scale_log2, neg[0])) * inv[0] + ex2_approx(fmaf(s[j][2], scale_log2, neg[1])) * inv[1];
          float c1 = ex2_approx(fmaf(s[j][1], scale_log2, neg[0])) * inv[0] + ex2_approx(fmaf(s[j][3], scale_log2, neg[1])) * inv[1];
#pragma unroll
          for (int sh = 4; sh < 32; sh <<= 1) {
            c0 += __shfl_xor_sync(0xffffffffu, c0, sh);
            c1 += __shfl_xor_sync(0xffffffffu, c1, sh);
          }
          const int t = kt * KT + 8 * j + 2 * tg;
          if (g == 0) {
            if (t < S) cs[t] += c0;
            if (t + 1 < S) cs[t + 1] += c1;
          }
        }
      }
      consumers_sync();                                    // the statistics may be overwritten
    }
    if (!ok && lane == 0) *(volatile int*)status = ST_ATTENTION_SCORES;
  }
  // every tile has landed before the CTA leaves, also where no row generates
  if (threadIdx.x == 0)
    for (int i = 0; i < n_kv; ++i) ptx::mbar_wait(full0 + 8u * i, 0, abort_flag + 1, 20000000LL);
  __syncthreads();
  if (!*abort_flag) {
    float* dst = score_partial + ((size_t)b * H + h) * S;
    for (int t = threadIdx.x; t < S; t += kThreads) {
      float sum = 0.f;
#pragma unroll
      for (int w = 0; w < kGroups; ++w) sum += colsum[w * S + t];
      dst[t] = sum;
    }
  }
}

size_t scores_smem(int n, int S, int dh) {
  return 1024 + (size_t)((S + KT - 1) / KT) * KT * dh * 2 + (size_t)kGroups * S * 4 + (size_t)(n + 1) / 2 * 4;
}

template <int DH>
cudaError_t launch_scores(const CUtensorMap& tm, const CUtensorMap& tail, const void* q, int ld_q, int B, int n, int S, int H,
                          const uint8_t* is_new, float* score_partial, int* status, cudaStream_t st) {
  const size_t smem = scores_smem(n, S, DH);
  static size_t smem_set[kMaxDevices] = {};
  cudaError_t e = ensure_dynamic_smem(attention_scores_kernel<DH>, smem, smem_set);
  if (e != cudaSuccess) return e;
  return launch_pdl(attention_scores_kernel<DH>, dim3(B * H), dim3(kThreads), smem, st, tm, tail, (const bf16*)q, ld_q, n, S, H,
                    is_new, score_partial, status);
}

}  // namespace

// A launch of its own costs 2 to 4 us (rows listed, K tiles loaded, two passes over them; twice that with a second group of 16
// generating rows), and saves what the one-kernel flavour costs over the plain one.  Difference of a one-block step, us, one group
// unless stated (few: one item per SM or less; many: more than two; beyond 13 tiles, at head_dim 80 11, an SM holds one CTA of it):
//   head_dim 64  up to 64 rows   few: one tile +2.4, two +0.4, three -2, five -4, 17 -30; 256 items: three 0, five -2 to -4; 64 rows
//                                three +2, four +1, five -2, with two groups five +1.5, ten -4.5, 17 +7
//                65 to 128 rows  (the two-pass tcgen05 kernel is close to the plain one) few +2 to +5, 256 items +5, at 17 tiles -11;
//                                many -0 to -58, with two groups -3 to +10, at 17 tiles -4
//                more            few: three tiles -1, ten -11; 256 items: three +3, five +1, ten -7; many -7 to -270
//   head_dim 80  up to 64 rows   few: as head_dim 64; 256 items: up to 16 rows three tiles +0.4, five -3, 17 +4; 17 to 32 rows two -1.3,
//                                three -3.4; 33 to 48 three +1.4, five -4.5; more two -4, five -14
//                more            few: two tiles +1, three -1, with two groups four -1; else -5 to -720 (no tcgen05 two-pass kernel)
bool attention_scores_wins(int n, int n_new, int S, int dh, int items) {
  const size_t smem = scores_smem(n, S, dh);
  if (n < 1 || (dh != 64 && dh != 80) || S > kMaxTiles * KT || smem > 224 * 1024 || n_new > 16 * kGroups) return false;
  const int n_kv = (S + KT - 1) / KT, sms = device_sm_count();
  const bool two = n_new > 16, few = items <= sms, many = items > 2 * sms, pair = smem <= 113 * 1024;   // two CTAs per SM
  const bool long_enough = n_kv >= (two ? 4 : 3);
  if (dh == 80 && (n > 96 || (n > 64 && !few))) return true;
  if (dh == 64 && n > 128) return many || (few ? long_enough : n_kv >= 10 || n > 256);
  if (dh == 64 && n > 64) return n_kv >= 16 ? many || (!two && !few) : many && !two;
  if (many) return false;
  if (few) return long_enough;
  if (dh == 80) return n <= 16 ? n_kv >= 4 && pair : n_kv >= (n > 32 && n <= 48 ? 4 : 2);
  if (n > 48) return two ? n_kv >= 8 && pair : n_kv >= 5;
  return n_kv >= (n > 16 ? 4 : 3);
}

cudaError_t launch_attention_scores(const void* q, int ld_q, int B, int n, int S, int H, int dh, const void* cache_layer,
                                    const uint8_t* is_new, float* score_partial, int* status, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  if ((dh != 64 && dh != 80) || S > kMaxTiles * KT || scores_smem(n, S, dh) > 224 * 1024 || ld_q % 2 || ((uintptr_t)q & 3) || ((uintptr_t)cache_layer & 15))
    return cudaErrorInvalidValue;
  const int D = H * dh;
  CUtensorMap tm, tail;
  const uint64_t dims[3] = {(uint64_t)D, (uint64_t)S, (uint64_t)2 * B};
  const uint64_t strides[2] = {(uint64_t)D * 2, (uint64_t)S * D * 2};
  const uint32_t box[3] = {64, KT, 1}, box_tail[3] = {16, KT, 1};   // as in the attention kernels
  if (!tma_make_map_bf16(&tm, cache_layer, 3, dims, strides, box, true)) return cudaErrorInvalidValue;
  tail = tm;
  if (dh == 80 && !tma_make_map_bf16(&tail, cache_layer, 3, dims, strides, box_tail, false, false, true))
    return cudaErrorInvalidValue;
  return dh == 64 ? launch_scores<64>(tm, tail, q, ld_q, B, n, S, H, is_new, score_partial, status, st)
                  : launch_scores<80>(tm, tail, q, ld_q, B, n, S, H, is_new, score_partial, status, st);
}

}  // namespace marche

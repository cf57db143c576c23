// K3 (SIMT): attention of the active queries over all S cached rows of one block
// (Algorithm 1 lines 6-8; by Appendix A this is plain softmax attention, Eq. 5, once
// the active rows' fresh K, V are in the cache), with the relevance reduction of
// Section 4.2 fused in.  fp32 arithmetic and storage; serves the fp32 configuration only.
//
// Bound by latency at that configuration's sizes (a handful of samples, 4 heads, about a hundred rows), then by shared
// memory, from which every warp reads every key and value: the queries of a (sample, head) item are dealt to up to eight
// CTAs (a cluster where they add scores together), and a warp takes two, for which it reads a key once.  K and V tiles (64
// keys, coalesced cp.async) are on their way up to four at once.  A warp's logits, softmax and output never leave it.  The
// probabilities of a CTA's queries stay in shared memory, so the softmax is the exact two-pass form and the column sums
// use final probabilities; they are added in query order within a CTA and in rank order over the cluster: scores are
// bit-reproducible.  (One CTA per item, reading a key row per lane and a value row at a time from global memory, was most
// of the 7.4 ms that an eight-step run took.)
#include "common.cuh"
#include "kernels.h"
#include "launch_pdl.h"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace marche {

namespace {

constexpr int kAttWarps = 8, kAttThreads = kAttWarps * 32, kKeys = 64;
constexpr int RW = 2, kRows = RW * kAttWarps;            // queries per warp and per CTA at a time

struct SimtLayout {                                      // in floats
  int ld, p_ld, tile, q, p, colsum, kv, total;
};
__host__ __device__ inline SimtLayout simt_layout(int S, int dh, int stages) {
  SimtLayout l;
  l.ld = dh + 4;                                         // rows 16 bytes apart modulo 128: conflict-free 128-bit reads
  l.p_ld = (S + kKeys - 1) / kKeys * kKeys + 4;
  l.tile = kKeys * l.ld;
  l.q = 0;
  l.p = l.q + kRows * l.ld;
  l.colsum = l.p + kRows * l.p_ld;
  l.kv = l.colsum + (S + 3) / 4 * 4;
  l.total = l.kv + stages * l.tile;
  return l;
}

MARCHE_DEVINL float dot4(float4 x, float4 y, float acc) {
  return fmaf(x.w, y.w, fmaf(x.z, y.z, fmaf(x.y, y.y, fmaf(x.x, y.x, acc))));
}

// NST K/V tiles in flight; HALVES 64-column halves of a head.  vec: the cache allows 16-byte copies.
template <int NST, int HALVES>
__global__ void __launch_bounds__(kAttThreads)
attention_simt_kernel(const float* __restrict__ q, int ld_q, int n, int S, int H, int dh, int cs,
                      const float* __restrict__ cache_layer, long kv_stride, const uint8_t* __restrict__ is_new,
                      float* __restrict__ score_partial, float* __restrict__ o, int vec) {
  extern __shared__ float4 smem_f4[];
  float* smem = reinterpret_cast<float*>(smem_f4);
  const SimtLayout l = simt_layout(S, dh, NST);
  float *qs = smem + l.q, *p = smem + l.p, *colsum = smem + l.colsum, *kv = smem + l.kv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int item = (int)blockIdx.x / cs, rank = (int)blockIdx.x - item * cs;   // (clusters are consecutive CTAs)
  const int b = item / H, h = item - b * H, D = H * dh;
  const int row_begin = (int)((long)n * rank / cs), row_end = (int)((long)n * (rank + 1) / cs);
  const float* Kb = cache_layer + (long)b * S * D + h * dh;
  const int n_kv = (S + kKeys - 1) / kKeys;
  const float scale = rsqrtf((float)dh);
  const uint32_t kv_base = ptx::smem_u32(kv);
  __shared__ bool flag[kRows];                           // scoring queries among the CTA's
  if (is_new)
    for (int t = tid; t < S; t += kAttThreads) colsum[t] = 0.f;
  pdl_sync();

  for (int r0 = row_begin; r0 < row_end; r0 += kRows) {
    const int rows = row_end - r0 < kRows ? row_end - r0 : kRows;
    // tile i of K tiles 0 .. n_kv - 1, then the V tiles; whole groups of four keys, zeros beyond S
    auto load = [&](int i) {
      if (i < 2 * n_kv) {
        const int t0 = (i < n_kv ? i : i - n_kv) * kKeys;
        const float* src = Kb + (i < n_kv ? 0 : kv_stride);
        const uint32_t dst = kv_base + 4u * (uint32_t)((i % NST) * l.tile);
        const int keys4 = S - t0 < kKeys ? (S - t0 + 3) & ~3 : kKeys;
        const float* s = src + (t0 + (tid >> 4)) * D + 4 * (tid & 15);
        uint32_t d = dst + 4u * (uint32_t)((tid >> 4) * l.ld + 4 * (tid & 15));
        for (int t = tid >> 4; t < keys4; t += kAttThreads / 16, s += kAttThreads / 16 * D, d += 4u * (kAttThreads / 16) * l.ld) {
          const bool ok = t0 + t < S;
#pragma unroll
          for (int half = 0; half < HALVES; ++half) {
            if (64 * half + 4 * (tid & 15) >= dh) break;
            const float* from = ok ? s + 64 * half : src;
            if (vec) {
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d + 256u * half), "l"(from), "r"(ok ? 16 : 0) : "memory");
            } else {
#pragma unroll
              for (int e = 0; e < 4; ++e)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d + 256u * half + 4 * e), "l"(from + (ok ? e : 0)),
                             "r"(ok ? 4 : 0) : "memory");
            }
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // a warp's queries are rows RW * warp, ...; it loads them itself, so no barrier stands between
    bool live[RW];
    const float* qr[RW];
    float* pr[RW];
    float qv[RW][2 * HALVES];
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const int row = RW * warp + r;
      live[r] = row < rows;
      if (is_new && lane == 0) flag[row] = live[r] && is_new[(long)b * n + r0 + row];
      qr[r] = qs + row * l.ld;
      pr[r] = p + row * l.p_ld;
#pragma unroll
      for (int e = 0; e < 2 * HALVES; ++e)
        qv[r][e] = live[r] && lane + 32 * e < dh ? q[((long)b * n + r0 + row) * ld_q + h * dh + lane + 32 * e] : 0.f;
    }
    for (int i = 0; i < NST - 1; ++i) load(i);
#pragma unroll
    for (int r = 0; r < RW; ++r)
#pragma unroll
      for (int e = 0; e < 2 * HALVES; ++e)
        if (lane + 32 * e < dh) qs[(RW * warp + r) * l.ld + lane + 32 * e] = qv[r][e] * scale;
    __syncwarp();
    float o_acc[RW][HALVES][2] = {};                     // [query][64-column half of the head][column of the lane's pair]

    for (int i = 0; i < 2 * n_kv; ++i) {
      asm volatile("cp.async.wait_group %0;" ::"n"(NST - 2) : "memory");
      __syncthreads();                                   // tile i has landed; every warp is done with tile i - 1
      load(i + NST - 1);
      const float* tile = kv + (i % NST) * l.tile;
      const int t0 = (i < n_kv ? i : i - n_kv) * kKeys, keys = S - t0 < kKeys ? S - t0 : kKeys;
      if (i < n_kv) {
        if (live[0]) {
          float s[2][RW] = {};                           // logits: this warp's queries x keys lane, lane + 32
          const float* kr = tile + lane * l.ld;
          if (keys > 32) {
#pragma unroll 4
            for (int c = 0; c < dh; c += 4) {
              const float4 x0 = *reinterpret_cast<const float4*>(kr + c), x1 = *reinterpret_cast<const float4*>(kr + 32 * l.ld + c);
#pragma unroll
              for (int r = 0; r < RW; ++r) {
                const float4 y = *reinterpret_cast<const float4*>(qr[r] + c);
                s[0][r] = dot4(x0, y, s[0][r]);
                s[1][r] = dot4(x1, y, s[1][r]);
              }
            }
          } else {
#pragma unroll 4
            for (int c = 0; c < dh; c += 4) {
              const float4 x0 = *reinterpret_cast<const float4*>(kr + c);
#pragma unroll
              for (int r = 0; r < RW; ++r) s[0][r] = dot4(x0, *reinterpret_cast<const float4*>(qr[r] + c), s[0][r]);
            }
          }
#pragma unroll
          for (int r = 0; r < RW; ++r) {
            pr[r][t0 + lane] = lane < keys ? s[0][r] : -INFINITY;
            pr[r][t0 + lane + 32] = lane + 32 < keys ? s[1][r] : -INFINITY;
          }
        }
        if (i == n_kv - 1) {
          // ---- exact softmax (each lane reads back what it wrote itself)
#pragma unroll
          for (int r = 0; r < RW; ++r) {
            if (!live[r]) continue;
            float mx = -INFINITY, sum = 0.f;
#pragma unroll 4
            for (int u = lane; u < n_kv * kKeys; u += 32) mx = fmaxf(mx, pr[r][u]);
            mx = warp_max(mx);
#pragma unroll 2
            for (int u = lane; u < n_kv * kKeys; u += 32) {
              const float e = expf(pr[r][u] - mx);
              pr[r][u] = e;
              sum += e;
            }
            const float inv = 1.0f / warp_sum(sum);
#pragma unroll 4
            for (int u = lane; u < n_kv * kKeys; u += 32) pr[r][u] *= inv;
          }
          __syncwarp();
          if (is_new) {
            __syncthreads();                             // the CTA's probabilities, added in query order
            for (int t = tid; t < S; t += kAttThreads) {
              float sum = colsum[t];
#pragma unroll
              for (int r = 0; r < kRows; ++r)
                if (flag[r]) sum += p[r * l.p_ld + t];
              colsum[t] = sum;
            }
          }
        }
      } else if (live[0]) {
#pragma unroll 4
        for (int t = 0; t < keys; t += 4) {              // (the last group may reach beyond S: zero weights times zeros)
          float w[RW][4];
#pragma unroll
          for (int r = 0; r < RW; ++r) {
            const float4 x = *reinterpret_cast<const float4*>(pr[r] + t0 + t);
            w[r][0] = x.x; w[r][1] = x.y; w[r][2] = x.z; w[r][3] = x.w;
          }
#pragma unroll
          for (int half = 0; half < HALVES; ++half) {
            const int c = 64 * half + 2 * lane;
            if (c < dh) {
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const float2 x = *reinterpret_cast<const float2*>(tile + (t + u) * l.ld + c);
#pragma unroll
                for (int r = 0; r < RW; ++r) {
                  o_acc[r][half][0] = fmaf(w[r][u], x.x, o_acc[r][half][0]);
                  o_acc[r][half][1] = fmaf(w[r][u], x.y, o_acc[r][half][1]);
                }
              }
            }
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < RW; ++r)
#pragma unroll
      for (int half = 0; half < HALVES; ++half) {
        const int c = 64 * half + 2 * lane;
        if (live[r] && c < dh) {
          float* dst = o + ((long)b * n + r0 + RW * warp + r) * D + h * dh + c;
          dst[0] = o_acc[r][half][0];
          dst[1] = o_acc[r][half][1];
        }
      }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                     // the next queries reuse the buffers
  }

  if (is_new) {
    // ---- column sums of the cluster, rank r finishing every cs-th group of keys
    __syncthreads();
    if (cs > 1) ptx::cluster_sync_all();
    for (int t = rank * kAttThreads + tid; t < S; t += cs * kAttThreads) {
      float sum = 0.f;
      for (int src = 0; src < cs; ++src) {
        float v;
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(ptx::mapa(ptx::smem_u32(colsum + t), (uint32_t)src)) : "memory");
        sum += v;
      }
      score_partial[((long)b * H + h) * S + t] = sum;
    }
    if (cs > 1) ptx::cluster_sync_all();                 // nobody leaves while its sums are read
  }
}

template <int NST, int HALVES>
cudaError_t launch_stages(const float* q, int ld_q, int B, int n, int S, int H, int dh, int cs, const float* cache_layer,
                          const uint8_t* is_new, float* score_partial, float* o, cudaStream_t st) {
  const size_t smem = (size_t)simt_layout(S, dh, NST).total * sizeof(float);
  static size_t smem_set[kMaxDevices] = {};
  cudaError_t e = ensure_dynamic_smem(attention_simt_kernel<NST, HALVES>, smem, smem_set);
  if (e != cudaSuccess) return e;
  const int vec = (((uintptr_t)cache_layer) & 15) == 0;
  return launch_pdl_cluster(attention_simt_kernel<NST, HALVES>, dim3(B * H * cs), dim3(kAttThreads), smem, is_new ? cs : 1, st, q, ld_q, n, S, H,
                            dh, cs, cache_layer, (long)B * S * H * dh, is_new, score_partial, o, vec);
}

}  // namespace

cudaError_t launch_attention_simt(const float* q, int ld_q, int B, int n, int S, int H, int dh,
                                  const float* cache_layer, const uint8_t* is_new, float* score_partial,
                                  float* o, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  // CTAs per item: one per eight queries (four warps) while the launch stays within a few CTAs per SM
  int cs = 1;
  while (cs < 8 && cs * kAttWarps < n && B * H * cs * 2 <= 4 * device_sm_count()) cs *= 2;
  // four tiles in flight where two CTAs per SM still fit, else two
  const bool deep = simt_layout(S, dh, 4).total * sizeof(float) <= 112 * 1024;
  if (dh <= 64)
    return deep ? launch_stages<4, 1>(q, ld_q, B, n, S, H, dh, cs, cache_layer, is_new, score_partial, o, st)
                : launch_stages<2, 1>(q, ld_q, B, n, S, H, dh, cs, cache_layer, is_new, score_partial, o, st);
  return deep ? launch_stages<4, 2>(q, ld_q, B, n, S, H, dh, cs, cache_layer, is_new, score_partial, o, st)
              : launch_stages<2, 2>(q, ld_q, B, n, S, H, dh, cs, cache_layer, is_new, score_partial, o, st);
}

}  // namespace marche

// K3 (SIMT): attention of the active queries over all S cached rows of one block
// (Algorithm 1 lines 6-8; by Appendix A this is plain softmax attention, Eq. 5, once
// the active rows' fresh K, V are in the cache), with the relevance reduction of
// Section 4.2 fused in.  fp32 arithmetic and storage; serves the fp32 configuration only.
//
// Bound by latency at that configuration's sizes (a handful of samples, 4 heads, about a hundred rows): the queries of
// a (sample, head) item are therefore dealt to a cluster of up to eight CTAs, 16 queries at a time, and the K and V
// tiles (64 keys, coalesced cp.async) are all on their way at once where shared memory holds them.  A warp owns two
// queries: their logits, softmax and output never leave it.  The probabilities of a tile's 16 queries stay in shared
// memory, so the softmax is the exact two-pass form and the column sums use final probabilities; they are added in
// query order within a CTA and in rank order over the cluster: scores are bit-reproducible.  (One CTA per item, reading
// a key row per lane and a value row at a time from global memory, was most of the 7.4 ms that an eight-step run took.)
#include "common.cuh"
#include "kernels.h"
#include "launch_pdl.h"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace marche {

namespace {

constexpr int kAttWarps = 8, kRows = 16, kKeys = 64;

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

// NST K/V tiles in flight.  vec: q and the cache allow 16-byte copies.
template <int NST>
__global__ void __launch_bounds__(kAttWarps * 32)
attention_simt_kernel(const float* __restrict__ q, int ld_q, int n, int S, int H, int dh, int cs,
                      const float* __restrict__ cache_layer, long kv_stride, const uint8_t* __restrict__ is_new,
                      float* __restrict__ score_partial, float* __restrict__ o, int vec) {
  extern __shared__ float4 smem_f4[];
  float* smem = reinterpret_cast<float*>(smem_f4);
  const SimtLayout l = simt_layout(S, dh, NST);
  float *qs = smem + l.q, *p = smem + l.p, *colsum = smem + l.colsum, *kv = smem + l.kv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = cs > 1 ? (int)ptx::cluster_ctarank() : 0, item = (int)blockIdx.x / cs;
  const int b = item / H, h = item - b * H, D = H * dh;
  const int row_begin = (int)((long)n * rank / cs), row_end = (int)((long)n * (rank + 1) / cs);
  const float* Kb = cache_layer + (long)b * S * D + h * dh;
  const int n_kv = (S + kKeys - 1) / kKeys, dv = dh / 4;
  const float scale = rsqrtf((float)dh);
  const uint32_t kv_base = ptx::smem_u32(kv);
  if (is_new)
    for (int t = tid; t < S; t += kAttWarps * 32) colsum[t] = 0.f;
  pdl_sync();

  for (int r0 = row_begin; r0 < row_end; r0 += kRows) {
    const int rows = row_end - r0 < kRows ? row_end - r0 : kRows;
    auto load = [&](int i) {                             // K tiles 0 .. n_kv - 1, then the V tiles
      if (i < 2 * n_kv) {
        const int t0 = (i < n_kv ? i : i - n_kv) * kKeys;
        const float* src = Kb + (i < n_kv ? 0 : kv_stride);
        const uint32_t dst = kv_base + 4u * (uint32_t)((i % NST) * l.tile);
        for (int e = tid; e < kKeys * dv; e += kAttWarps * 32) {
          const int t = e / dv, v = e - t * dv, bytes = t0 + t < S ? (vec ? 16 : 4) : 0;
          const float* s = src + (long)(t0 + t < S ? t0 + t : 0) * D + 4 * v;
          const uint32_t d = dst + 4u * (uint32_t)(t * l.ld + 4 * v);
          if (vec) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(s), "r"(bytes) : "memory");
          } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d + 4 * j), "l"(s + j), "r"(bytes) : "memory");
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int i = 0; i < NST - 1; ++i) load(i);
    for (int e = tid; e < kRows * dh; e += kAttWarps * 32) {
      const int r = e / dh, c = e - r * dh;
      qs[r * l.ld + c] = r < rows ? q[((long)b * n + r0 + r) * ld_q + h * dh + c] * scale : 0.f;
    }
    const int ra = warp, rb = warp + kAttWarps;          // this warp's two queries
    float o_acc[2][2][2] = {};                           // [query][64-column half of the head][column of the lane's pair]

    for (int i = 0; i < 2 * n_kv; ++i) {
      asm volatile("cp.async.wait_group %0;" ::"n"(NST - 2) : "memory");
      __syncthreads();                                   // tile i has landed; every warp is done with tile i - 1
      load(i + NST - 1);
      const float* tile = kv + (i % NST) * l.tile;
      if (i < n_kv) {
        float s[2][2] = {};                              // logits: queries ra, rb x keys lane, lane + 32
        const float *qa = qs + ra * l.ld, *qb = qs + rb * l.ld, *k0 = tile + lane * l.ld, *k1 = k0 + 32 * l.ld;
#pragma unroll 4
        for (int c = 0; c < dh; c += 4) {
          const float4 x0 = *reinterpret_cast<const float4*>(k0 + c), x1 = *reinterpret_cast<const float4*>(k1 + c);
          const float4 ya = *reinterpret_cast<const float4*>(qa + c), yb = *reinterpret_cast<const float4*>(qb + c);
          s[0][0] = dot4(x0, ya, s[0][0]);
          s[0][1] = dot4(x1, ya, s[0][1]);
          s[1][0] = dot4(x0, yb, s[1][0]);
          s[1][1] = dot4(x1, yb, s[1][1]);
        }
        const int t = i * kKeys + lane;
        p[ra * l.p_ld + t] = t < S ? s[0][0] : -INFINITY;
        p[ra * l.p_ld + t + 32] = t + 32 < S ? s[0][1] : -INFINITY;
        p[rb * l.p_ld + t] = t < S ? s[1][0] : -INFINITY;
        p[rb * l.p_ld + t + 32] = t + 32 < S ? s[1][1] : -INFINITY;
        if (i == n_kv - 1) {
          // ---- exact softmax of the two queries (each lane reads back what it wrote itself)
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            float* pr = p + (r ? rb : ra) * l.p_ld;
            float mx = -INFINITY, sum = 0.f;
            for (int u = lane; u < n_kv * kKeys; u += 32) mx = fmaxf(mx, pr[u]);
            mx = warp_max(mx);
            for (int u = lane; u < n_kv * kKeys; u += 32) {
              const float e = expf(pr[u] - mx);
              pr[u] = e;
              sum += e;
            }
            const float inv = 1.0f / warp_sum(sum);
            for (int u = lane; u < n_kv * kKeys; u += 32) pr[u] *= inv;
          }
          __syncwarp();
          if (is_new) {
            __syncthreads();                             // all 16 queries' probabilities
            for (int t2 = tid; t2 < S; t2 += kAttWarps * 32) {
              float cs_t = colsum[t2];
              for (int r = 0; r < rows; ++r)
                if (is_new[(long)b * n + r0 + r]) cs_t += p[r * l.p_ld + t2];
              colsum[t2] = cs_t;
            }
          }
        }
      } else {
        const int t0 = (i - n_kv) * kKeys;
        const float *pa = p + ra * l.p_ld + t0, *pb = p + rb * l.p_ld + t0;
#pragma unroll 4
        for (int t = 0; t < kKeys; t += 4) {             // (keys beyond S: zero probabilities times zeros)
          const float4 wa = *reinterpret_cast<const float4*>(pa + t), wb = *reinterpret_cast<const float4*>(pb + t);
          const float va[4] = {wa.x, wa.y, wa.z, wa.w}, vb[4] = {wb.x, wb.y, wb.z, wb.w};
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            const int c = 64 * half + 2 * lane;
            if (c < dh) {
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const float2 x = *reinterpret_cast<const float2*>(tile + (t + u) * l.ld + c);
                o_acc[0][half][0] = fmaf(va[u], x.x, o_acc[0][half][0]);
                o_acc[0][half][1] = fmaf(va[u], x.y, o_acc[0][half][1]);
                o_acc[1][half][0] = fmaf(vb[u], x.x, o_acc[1][half][0]);
                o_acc[1][half][1] = fmaf(vb[u], x.y, o_acc[1][half][1]);
              }
            }
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int row = r ? rb : ra, c = 64 * half + 2 * lane;
        if (row < rows && c < dh) {
          float* dst = o + ((long)b * n + r0 + row) * D + h * dh + c;
          dst[0] = o_acc[r][half][0];
          dst[1] = o_acc[r][half][1];
        }
      }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                     // the next 16 queries reuse the buffers
  }

  if (is_new) {
    // ---- column sums of the cluster, rank r finishing every cs-th group of keys
    __syncthreads();
    if (cs > 1) ptx::cluster_sync_all();
    for (int t = rank * kAttWarps * 32 + tid; t < S; t += cs * kAttWarps * 32) {
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

template <int NST>
cudaError_t launch_stages(const float* q, int ld_q, int B, int n, int S, int H, int dh, int cs, const float* cache_layer,
                          const uint8_t* is_new, float* score_partial, float* o, cudaStream_t st) {
  const size_t smem = (size_t)simt_layout(S, dh, NST).total * sizeof(float);
  static size_t smem_set[kMaxDevices] = {};
  cudaError_t e = ensure_dynamic_smem(attention_simt_kernel<NST>, smem, smem_set);
  if (e != cudaSuccess) return e;
  const int vec = (((uintptr_t)cache_layer) & 15) == 0;
  return launch_pdl_cluster(attention_simt_kernel<NST>, dim3(B * H * cs), dim3(kAttWarps * 32), smem, cs, st, q, ld_q, n, S, H,
                            dh, cs, cache_layer, (long)B * S * H * dh, is_new, score_partial, o, vec);
}

}  // namespace

cudaError_t launch_attention_simt(const float* q, int ld_q, int B, int n, int S, int H, int dh,
                                  const float* cache_layer, const uint8_t* is_new, float* score_partial,
                                  float* o, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  // CTAs per item: one per 16 queries, as long as the launch stays within a few CTAs per SM
  int cs = 1;
  while (cs < 8 && cs * kRows < n && B * H * cs * 2 <= 4 * device_sm_count()) cs *= 2;
  // four tiles in flight where two CTAs per SM still fit, else two
  return simt_layout(S, dh, 4).total * sizeof(float) <= 112 * 1024
             ? launch_stages<4>(q, ld_q, B, n, S, H, dh, cs, cache_layer, is_new, score_partial, o, st)
             : launch_stages<2>(q, ld_q, B, n, S, H, dh, cs, cache_layer, is_new, score_partial, o, st);
}

}  // namespace marche

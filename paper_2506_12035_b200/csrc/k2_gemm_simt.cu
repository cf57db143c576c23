// K2 (SIMT): out = epilogue(a * w^T + bias) with fp32 FMA arithmetic.
//
// fp32 operands and outputs only: this is the projection kernel of the fp32 configuration (the
// tensor cores have no full-fp32 mode, and TF32 would not meet an fp32-level tolerance).  The
// 16-bit contexts never come here.
//
// What bounds it at the sizes of that configuration (some hundred rows, width 256) is latency, then the FMA pipes.  A
// CTA computes a T x T tile of the output; its four groups of 64 threads take a quarter of every K chunk each, so that
// a small tile still keeps eight warps busy, and the partial sums meet in shared memory in group order.  Where the
// tiles leave SMs idle, a cluster of CS CTAs shares a tile, each with a slice of K, and the slices are added in rank
// order through distributed shared memory: bit-reproducible either way.  K chunks of 128 arrive by cp.async, two in
// flight, the weights' first ones before the dependency wait (no kernel writes weights).  With this and the fp32 attention
// in clusters a tiny eight-step run (2 x 68 tokens, width 256, 4 blocks) went from 7.38 ms to 0.98 ms.
#include <cmath>

#include "common.cuh"
#include "kernels.h"
#include "launch_pdl.h"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace marche {

namespace {

constexpr int kGemmThreads = 256, kGroups = 4, KC = 128, kRowPad = 4, kStagesSimt = 2;

// Four consecutive floats into shared memory; `valid` false writes zeros.
MARCHE_DEVINL void copy4(uint32_t dst, const float* src, bool valid, bool vec) {
  const int bytes = valid ? (vec ? 16 : 4) : 0;
  if (vec) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4 * i), "l"(valid ? src + i : src), "r"(bytes) : "memory");
  }
}

// T x T output tile, micro-tiles of T / 8 x T / 8.  vec: a, w and their row strides allow 16-byte copies.
template <int T, int CS, int EPI>
__global__ void __launch_bounds__(kGemmThreads)
gemm_simt_kernel(const float* __restrict__ a, int lda, int M, const float* __restrict__ w, const float* __restrict__ bias,
                 int N, int K, float* __restrict__ out, const KvScatter kv, int vec) {
  constexpr int TM = T / 8, LD = KC + kRowPad, STAGE = 2 * T * LD;
  constexpr int NV = T * T / 4 / kGemmThreads;           // float4s of the tile per thread
  constexpr int OWN = T * T / 4 / CS;                    // float4s of the tile that one CTA of the cluster finishes
  extern __shared__ float4 smem_f4[];
  float* smem = reinterpret_cast<float*>(smem_f4);
  float4* red = smem_f4;                                 // [kGroups][T * T / 4], over the (finished) ring
  float4* recv = smem_f4 + kStagesSimt * STAGE / 4;      // [CS][OWN]
  const int tid = threadIdx.x, grp = tid >> 6, tx = tid & 7, ty = (tid >> 3) & 7;
  const int rank = CS > 1 ? (int)ptx::cluster_ctarank() : 0;
  const int n_n = N / T, tile = (int)blockIdx.x / CS;
  const int m0 = tile / n_n * T, n0 = tile % n_n * T;
  const int k_begin = rank * (K / CS), k_end = k_begin + K / CS, n_chunks = (K / CS + KC - 1) / KC;
  const uint32_t smem_base = ptx::smem_u32(smem);

  auto load = [&](const float* src, long ld, int rows, int r0, int c, int offset) {   // T rows of chunk c
    const int k0 = k_begin + c * KC, q = (k_end - k0 < KC ? k_end - k0 : KC) / 4;
    const uint32_t dst = smem_base + 4u * (uint32_t)((c & 1) * STAGE + offset);
    for (int i = tid; i < T * (KC / 4); i += kGemmThreads) {
      const int r = i / (KC / 4), v = i % (KC / 4);
      if (v < q) {
        const bool ok = r0 + r < rows;
        copy4(dst + 4u * (uint32_t)(r * LD + 4 * v), ok ? src + (long)(r0 + r) * ld + k0 + 4 * v : src, ok, vec != 0);
      }
    }
  };
  // weights of both chunks ahead of the wait; a group per chunk once its activations are on their way too
  for (int c = 0; c < kStagesSimt && c < n_chunks; ++c) load(w, K, N, n0, c, T * LD);
  if (CS > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  pdl_sync();
  for (int c = 0; c < kStagesSimt; ++c) {
    if (c < n_chunks) load(a, lda, M, m0, c, 0);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // what the epilogue will need: this thread's float4s are e = tid + 256 i (of the CTA's own ones when CS > 1)
  constexpr int NF = CS > 1 ? (OWN + kGemmThreads - 1) / kGemmThreads : NV;
  float4 bv[NF], res[NF];
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    const int e = tid + kGemmThreads * i, f = rank * OWN + e, row = m0 + f / (T / 4), col = n0 + f % (T / 4) * 4;
    bv[i] = res[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < OWN) {
      bv[i] = *reinterpret_cast<const float4*>(bias + col);
      if (EPI == 1 && row < M) res[i] = *reinterpret_cast<const float4*>(out + (long)row * N + col);
    }
  }

  float acc[TM][TM];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) acc[i][j] = 0.f;
  for (int c = 0; c < n_chunks; ++c) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const int kc = k_end - (k_begin + c * KC) < KC ? k_end - (k_begin + c * KC) : KC;
    const float* as = smem + (c & 1) * STAGE + ty * LD + grp * (kc / 4);
    const float* ws = smem + (c & 1) * STAGE + (T + tx) * LD + grp * (kc / 4);
#pragma unroll (T == 32 ? 2 : 1)
    for (int k = 0; k < kc / 4; k += 4) {
      float4 av[TM], wv[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i) av[i] = *reinterpret_cast<const float4*>(as + i * 8 * LD + k);
#pragma unroll
      for (int j = 0; j < TM; ++j) wv[j] = *reinterpret_cast<const float4*>(ws + j * 8 * LD + k);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TM; ++j) {
          acc[i][j] = fmaf(av[i].x, wv[j].x, acc[i][j]);
          acc[i][j] = fmaf(av[i].y, wv[j].y, acc[i][j]);
          acc[i][j] = fmaf(av[i].z, wv[j].z, acc[i][j]);
          acc[i][j] = fmaf(av[i].w, wv[j].w, acc[i][j]);
        }
    }
    __syncthreads();                                     // the chunk's buffer is free
    if (c + kStagesSimt < n_chunks) {
      load(w, K, N, n0, c + kStagesSimt, T * LD);
      load(a, lda, M, m0, c + kStagesSimt, 0);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }

  // ---- sum over the groups, then over the cluster
  float* my = reinterpret_cast<float*>(red) + grp * (T * T);
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) my[(ty + 8 * i) * T + tx + 8 * j] = acc[i][j];
  __syncthreads();
  float4 sum[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int e = tid + kGemmThreads * i;
    sum[i] = red[e];
#pragma unroll
    for (int g = 1; g < kGroups; ++g) {
      const float4 p = red[g * (T * T / 4) + e];
      sum[i].x += p.x; sum[i].y += p.y; sum[i].z += p.z; sum[i].w += p.w;
    }
  }
  if (CS > 1) {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");      // every CTA of the cluster has started
    const uint32_t slot = ptx::smem_u32(recv + rank * OWN);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int e = tid + kGemmThreads * i;
      const uint32_t dst = ptx::mapa(slot, (uint32_t)(e / OWN)) + 16u * (uint32_t)(e % OWN);
      asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "f"(sum[i].x), "f"(sum[i].y),
                   "f"(sum[i].z), "f"(sum[i].w) : "memory");
    }
    ptx::cluster_sync_all();
  }
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    const int e = tid + kGemmThreads * i, f = rank * OWN + e, row = m0 + f / (T / 4), col = n0 + f % (T / 4) * 4;
    if (e >= OWN || row >= M) continue;
    float4 v = sum[i < NV ? i : 0];
    if (CS > 1) {
      v = recv[e];
#pragma unroll
      for (int src = 1; src < CS; ++src) {
        const float4 p = recv[src * OWN + e];
        v.x += p.x; v.y += p.y; v.z += p.z; v.w += p.w;
      }
    }
    v.x += bv[i].x; v.y += bv[i].y; v.z += bv[i].z; v.w += bv[i].w;
    if (EPI == 1) { v.x += res[i].x; v.y += res[i].y; v.z += res[i].z; v.w += res[i].w; }
    if (EPI == 2) { v.x = gelu_erf(v.x); v.y = gelu_erf(v.y); v.z = gelu_erf(v.z); v.w = gelu_erf(v.w); }
    float* dst = out + (long)row * N + col;
    if (EPI == 4 && col >= kv.D) {                       // a K or V column: into the cache row of the token
      const int which = col / kv.D - 1, b = row / kv.n, token = kv.idx ? kv.idx[row] : row - b * kv.n;
      dst = reinterpret_cast<float*>(kv.cache) + (((long)which * kv.B + b) * kv.S + token) * kv.D + col - (which + 1) * kv.D;
    }
    *reinterpret_cast<float4*>(dst) = v;
  }
}

template <int T, int CS, int EPI>
cudaError_t launch_one(const float* a, int lda, int M, const float* w, const float* bias, int N, int K, float* out,
                       const KvScatter& kv, cudaStream_t st) {
  const size_t smem = ((size_t)kStagesSimt * 2 * T * (KC + kRowPad) + (CS > 1 ? T * T : 0)) * sizeof(float);
  static_assert(kStagesSimt * 2 * (KC + kRowPad) >= kGroups * T, "the groups' partial sums lie over the ring");
  static size_t smem_set[kMaxDevices] = {};
  cudaError_t e = ensure_dynamic_smem(gemm_simt_kernel<T, CS, EPI>, smem, smem_set);
  if (e != cudaSuccess) return e;
  const int vec = lda % 4 == 0 && ((((uintptr_t)a | (uintptr_t)w)) & 15) == 0;
  return launch_pdl_cluster(gemm_simt_kernel<T, CS, EPI>, dim3(CS * (N / T) * ((M + T - 1) / T)), dim3(kGemmThreads), smem, CS,
                            st, a, lda, M, w, bias, N, K, out, kv, vec);
}

// Estimated microseconds, fitted to the measured times of every tile and cluster size (M 10 to 1700, N 256 to 1024, K 256 and
// 1024): a K column of a 32 x 32 tile takes 14.6 ns alone on an SM and 12.1 with others, one of a 64 x 64 tile 35 and 42
// (LDS.128 issue bounds both: 8 loads per 64 and 16 per 256 FMAs); a cluster costs its start and exchange, more so where
// CTAs queue.  M x N x K, us, one CTA per tile -> chosen: 20 x 256 x 1024 15.6 -> 3.6, 40 x 768 x 256 4.4 -> 3.9.
double simt_cost(int M, int N, int K, int t, int cs) {
  if (N % t || K % (16 * cs)) return 1e30;
  const double load = (double)((M + t - 1) / t) * (N / t) * cs / device_sm_count(), k = (double)K / cs;
  const double cost = load <= 1.0 ? 0.8 + k * (t == 32 ? 14.6e-3 : 35e-3) : 0.6 + std::ceil(load) * k * (t == 32 ? 12.1e-3 : 42e-3);
  return cs == 1 ? cost : cost + 0.4 + 0.15 * cs + (load > 1.0 ? 2.0 : 0.0);
}

}  // namespace

cudaError_t launch_gemm_simt(const float* a, int lda, int M, const float* w, const float* bias,
                             int N, int K, int epilogue, float* out, cudaStream_t st, const KvScatter* kv_scatter) {
  if (M == 0) return cudaSuccess;
  if (N % 64 || K % 16) return cudaErrorInvalidValue;
  KvScatter kv = {nullptr, nullptr, 1, 1, 1, 1 << 30};
  if (epilogue == 4) {
    if (!kv_scatter || !kv_scatter->cache || N != 3 * kv_scatter->D || ((uintptr_t)kv_scatter->cache & 15)) return cudaErrorInvalidValue;
    kv = *kv_scatter;
  }
  int t = 64, cs = 1;
  double best = 1e30;
  for (int ti = 32; ti <= 64; ti *= 2)
    for (int c = 1; c <= (ti == 32 ? 8 : 1); c *= 2) {
      const double cost = simt_cost(M, N, K, ti, c);
      if (cost < best) { best = cost; t = ti; cs = c; }
    }
#define MARCHE_SIMT_CASE(T_, CS_)                                                                          \
  if (t == T_ && cs == CS_) {                                                                              \
    if (epilogue == 0) return launch_one<T_, CS_, 0>(a, lda, M, w, bias, N, K, out, kv, st);               \
    if (epilogue == 1) return launch_one<T_, CS_, 1>(a, lda, M, w, bias, N, K, out, kv, st);               \
    if (epilogue == 2) return launch_one<T_, CS_, 2>(a, lda, M, w, bias, N, K, out, kv, st);               \
    if (epilogue == 4) return launch_one<T_, CS_, 4>(a, lda, M, w, bias, N, K, out, kv, st);               \
  }
  MARCHE_SIMT_CASE(32, 1) MARCHE_SIMT_CASE(32, 2) MARCHE_SIMT_CASE(32, 4)
  MARCHE_SIMT_CASE(32, 8) MARCHE_SIMT_CASE(64, 1)
#undef MARCHE_SIMT_CASE
  return cudaErrorInvalidValue;
}

}  // namespace marche

// K2 for few rows: out = epilogue(a * w^T + bias), the projections of up to about a thousand active rows.
//
// What bounds it: latency.  One image (2 rows of guidance, about 40 active tokens each) gives 82 rows; the 128 x 256
// or 256 x 256 tiles of the large-batch kernels then leave all but 8 to 16 SMs idle while those walk the whole K
// range one 64-wide block after the other.  Here one CTA computes a 128 x BN piece of the output over a SLICE of K,
// and the CTAs that share an output tile form a cluster: each sends its fp32 partial sums through
// distributed shared memory to the CTA that owns the columns, which adds them in rank order (bit-reproducible),
// applies the epilogue and stores.  No second launch, no atomics, no partials in global memory.
//
//   warp 0 (one lane)  TMA producer.  Weights are never written by a kernel, so the ring's first W tiles are loaded,
//                      and the rest of the slice is prefetched into L2, BEFORE the dependency wait, under the
//                      predecessor's tail; only the A tiles wait for it.
//   warp 1 (one lane)  issues tcgen05.mma (M 128, N BN, K 16), accumulator in BN columns of tensor memory
//   warps 2-5          partial sums to the owners, reduction, epilogue; one thread per output row
// A CTA takes at most 112 KB of shared memory (but for clusters on 128-column tiles) and BN columns of tensor memory, so
// the next kernel's CTAs become resident beside it and run their set-up early (programmatic dependent launch).  A tiles are
// only as high as their share of the rows: the MMA's remaining rows read whatever the ring holds and are never stored.
// All waits are bounded; a CTA that gave up stays until its cluster has left, so nobody writes to a CTA that is gone.
#include <cuda.h>

#include <cmath>
#include <type_traits>

#include "gemm_epilogue.cuh"
#include "kernels.h"
#include "launch_pdl.h"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace marche {

namespace {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int kThreads = 192;
constexpr int kMaxStages = 8;
constexpr int kSmemBudget = 112 * 1024;   // two CTAs per SM
constexpr int kSmemBudgetWide = 224 * 1024;   // one: a 128-column tile's partial sums take 64 KB
enum { STK_PRODUCER = 0x61, STK_MMA = 0x62, STK_EPILOGUE = 0x63 };

MARCHE_DEVINL void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
MARCHE_DEVINL void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
MARCHE_DEVINL void st_cluster_v4(uint32_t addr, const uint32_t* v) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3])
               : "memory");
}
MARCHE_DEVINL float4 ld_shared_v4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

MARCHE_DEVINL void st_global_v8(void* dst, const uint32_t* v) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
               "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}

// 32 bytes of one finished output row (8 fp32 or 16 16-bit columns, the sums in f): epilogue and store.  A lane holds a
// row, so that a warp's store touches 32 rows whatever its width: whole sectors where the output is so aligned.
template <int EPI>
MARCHE_DEVINL void finish32(float4 (&f)[EPI == 1 ? 2 : 4], uint8_t* dst, bool sector, bool a_bf16) {
  uint32_t v[8];
#pragma unroll
  for (int j = 0; j < (EPI == 1 ? 2 : 4); ++j) {
    if (EPI == 1) {
      v[4 * j % 8] = __float_as_uint(f[j].x); v[(4 * j + 1) % 8] = __float_as_uint(f[j].y);
      v[(4 * j + 2) % 8] = __float_as_uint(f[j].z); v[(4 * j + 3) % 8] = __float_as_uint(f[j].w);
    } else if (EPI == 2) {
      gelu_erf_pair(f[j].x, f[j].y);
      gelu_erf_pair(f[j].z, f[j].w);
      v[2 * j] = pack_a16x2(f[j].x, f[j].y, a_bf16);
      v[2 * j + 1] = pack_a16x2(f[j].z, f[j].w, a_bf16);
    } else {
      v[2 * j] = pack_bf16x2(f[j].x, f[j].y);
      v[2 * j + 1] = pack_bf16x2(f[j].z, f[j].w);
    }
  }
  if (sector) {
    st_global_v8(dst, v);
  } else {
    reinterpret_cast<uint4*>(dst)[0] = make_uint4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<uint4*>(dst)[1] = make_uint4(v[4], v[5], v[6], v[7]);
  }
}

// The same for eight 16-bit columns.
template <int EPI>
MARCHE_DEVINL void finish16(float4 a, float4 b, uint8_t* dst, bool a_bf16) {
  if (EPI == 2) { gelu_erf_pair(a.x, a.y); gelu_erf_pair(a.z, a.w); gelu_erf_pair(b.x, b.y); gelu_erf_pair(b.z, b.w); }
  const bool bf = EPI != 2 || a_bf16;
  *reinterpret_cast<uint4*>(dst) = make_uint4(pack_a16x2(a.x, a.y, bf), pack_a16x2(a.z, a.w, bf), pack_a16x2(b.x, b.y, bf),
                                              pack_a16x2(b.z, b.w, bf));
}

// TMA stores the output only where no cluster finishes it: the other launches do not carry its map.
template <int CS> using OutMap = typename std::conditional<CS == 1, CUtensorMap, char>::type;

// Grid: x = CS * (n_m * n_n) CTAs, clusters of CS consecutive ones share an output tile and split its K blocks.
template <int BN, int CS, int EPI>
__global__ void __launch_bounds__(kThreads, BN == 128 && CS > 1 ? 1 : 2)
gemm_splitk_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w,
                   const __grid_constant__ OutMap<CS> tmap_out, int M, int N, int K, int a_rows, int n_stages,
                   int ring_bytes, const float* __restrict__ bias, void* __restrict__ out,
                   const KvScatter kv, int a_bf16, int* __restrict__ status) {
  constexpr int W_BYTES = BN * BK * 2;
  constexpr int OWN = BN / CS;                             // columns this CTA finishes
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = ptx::smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  const uint32_t a_bytes = (uint32_t)a_rows * (BK * 2);
  const uint32_t w_base = base + (uint32_t)n_stages * a_bytes;
  const uint32_t recv = base + ring_bytes;                 // partial sums [CS][OWN / 4][128 rows] float4 (CS > 1)
  const uint32_t bar_base = recv + (CS > 1 ? BM * BN * 4u : BN * 4u);            // CS == 1: the bias instead
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (kMaxStages + s); };
  const uint32_t tfull_bar = bar_base + 8u * (2 * kMaxStages), recv_bar = tfull_bar + 8u;
  uint8_t* gen = smem_raw + (bar_base - raw) + 8 * (2 * kMaxStages + 2);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(gen);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gen + 8);

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int rank = CS > 1 ? (int)ptx::cluster_ctarank() : 0;
  const int n_n = N / BN, n_kb = K / BK;
  const int tile = (int)blockIdx.x / CS;
  const int m_blk = tile / n_n, n_blk = tile - m_blk * n_n;
  const int kb0 = rank * n_kb / CS, kb1 = (rank + 1) * n_kb / CS, n_it = kb1 - kb0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < n_stages; ++s) {
      ptx::mbar_init(full_bar(s), 1);
      ptx::mbar_init(empty_bar(s), 1);
    }
    ptx::mbar_init(tfull_bar, 1);
    ptx::mbar_init(recv_bar, 4 * CS);                      // one arrival per epilogue warp of every CTA of the cluster
    abort_flag[0] = 0;
    abort_flag[1] = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
  }
  if (warp == 2) {
    ptx::tmem_alloc(ptx::smem_u32((const void*)tmem_slot), BN);
    ptx::tmem_relinquish();
  }
  int loaded = 0;                                          // ring slots whose W tile is on its way
  if (warp == 0 && ptx::elect_one()) {
    ptx::prefetch_tensormap(&tmap_a);
    ptx::prefetch_tensormap(&tmap_w);
    for (; loaded < n_it && loaded < n_stages; ++loaded) {
      ptx::mbar_expect_tx(full_bar(loaded), a_bytes + W_BYTES);
      ptx::tma_load_2d(w_base + loaded * W_BYTES, &tmap_w, (kb0 + loaded) * BK, n_blk * BN, full_bar(loaded));
    }
    for (int i = loaded; i < n_it; ++i) ptx::tma_prefetch_l2_2d(&tmap_w, (kb0 + i) * BK, n_blk * BN);
  }
  __syncwarp();
  if (CS > 1) cluster_arrive();                            // our barriers exist
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  constexpr int NQ = CS > 1 ? OWN / 4 : 1;                 // float4s that a thread finishes of its row
  float4 bv[NQ];                                           // (the bias, too, is never written)
  if (CS > 1 && warp >= 2) {
#pragma unroll
    for (int j = 0; j < NQ; ++j) bv[j] = __ldg(reinterpret_cast<const float4*>(bias + n_blk * BN + rank * OWN) + j);
  }
  pdl_sync();                                              // everything above overlapped the previous kernel's tail

  bool ok = true;
  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (ptx::elect_one()) {
      int s = 0, x = kb0 * BK, i = 0;
      uint32_t phase = 1;                                  // an empty slot's first wait passes at once
      for (; i < n_it; ++i, x += BK) {
        if (i >= loaded) {
          if (!ptx::mbar_wait(empty_bar(s), phase, abort_flag)) { ok = false; break; }
          ptx::mbar_expect_tx(full_bar(s), a_bytes + W_BYTES);
          ptx::tma_load_2d(w_base + s * W_BYTES, &tmap_w, x, n_blk * BN, full_bar(s));
        }
        ptx::tma_load_2d(base + s * a_bytes, &tmap_a, x, m_blk * a_rows, full_bar(s));
        if (++s == n_stages) { s = 0; phase ^= 1u; }
      }
      if (!ok) {
        *(volatile int*)status = STK_PRODUCER;
        // let copies already issued land before the CTA's shared memory is released
        for (int j = 1; j <= n_stages && j <= i; ++j) {
          const int i2 = i - j;
          ptx::mbar_wait(full_bar(i2 % n_stages), (uint32_t)(i2 / n_stages) & 1u, abort_flag + 1, 20000000LL);
        }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    // One K block is 4 MMAs of BN / 2 cycles or so: slot, phase and descriptors are stepped, not divided out (with the
    // usual i % stages and descriptors built per MMA a block cost 680 cycles, with these 240).
    if (ptx::elect_one()) {
      const uint32_t idesc = ptx::idesc_16_f32(BM, BN, a_bf16 != 0);
      const uint64_t a_desc0 = ptx::smem_desc_k_sw128(base), w_desc0 = ptx::smem_desc_k_sw128(w_base);
      uint64_t da = a_desc0, dw = w_desc0;
      int s = 0;
      uint32_t phase = 0;
      for (int i = 0; i < n_it; ++i) {
        if (!ptx::mbar_wait(full_bar(s), phase, abort_flag)) { ok = false; break; }
        ptx::tc_fence_after();
#pragma unroll
        for (int k = 0; k < BK / 16; ++k) ptx::umma_f16(tmem_base, da + 2 * k, dw + 2 * k, idesc, (i | k) ? 1u : 0u);
        if (i + n_stages < n_it) ptx::umma_commit(empty_bar(s));
        da += a_bytes >> 4;
        dw += W_BYTES >> 4;
        if (++s == n_stages) { s = 0; phase ^= 1u; da = a_desc0; dw = w_desc0; }
      }
      if (ok) ptx::umma_commit(tfull_bar);
      else *(volatile int*)status = STK_MMA;
    }
  } else {
    // ---------------------------------------------------------------- epilogue (warps 2..5)
    const int quarter = warp & 3;
    const int r = quarter * 32 + lane, row = m_blk * a_rows + r;
    const bool valid = r < a_rows && row < M;
    const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const int col0 = n_blk * BN + rank * OWN;              // first output column this CTA finishes
    const bool to_cache = EPI == 4 && col0 >= kv.D;        // a K or V column: into the cache row of the token
    const int which = to_cache ? col0 / kv.D - 1 : 0;
    const int kv_col = col0 - (which + 1) * kv.D;
    long kv_row = -1;
    if (to_cache && valid) {
      const int b = row / kv.n;
      const int t = kv.idx ? kv.idx[row] : row - b * kv.n;
      kv_row = ((long)which * kv.B + b) * kv.S + t;
    }
    if constexpr (CS == 1) {
      epilogue_bias_store(epilogue_bias_load(bias + col0, BN, lane), BN, recv, lane);
      ok = ptx::mbar_wait(tfull_bar, 0, abort_flag);
      ptx::tc_fence_after();
      // every MMA has completed, so the ring is free: it becomes the warps' staging boxes
      const uint32_t stage = base + (uint32_t)(warp - 2) * 8192u;
      const int row0 = m_blk * a_rows + quarter * 32;
      if (ok && quarter * 32 < a_rows && row0 < M) {
        int n_box = 0;
        if (to_cache)
          epilogue_columns<0, true>(t_row, 0, BN, recv, &tmap_out, col0, row0, stage, n_box, lane,
                                    false, (bf16*)kv.cache, kv_row < 0 ? -1L : kv_row * kv.D + kv_col);
        else
          epilogue_columns<EPI == 4 ? 0 : EPI, false>(t_row, 0, BN, recv, &tmap_out, col0, row0,
                                                      stage, n_box, lane, a_bf16 != 0);
        if (lane == 0) ptx::bulk_wait_read_all();
      }
    } else {
      // what the residual sum will need is fetched under the main loop: the old values
      constexpr int OB = EPI == 1 ? 4 : 2;
      uint8_t* dst = !valid ? nullptr
                     : to_cache ? reinterpret_cast<uint8_t*>(kv.cache) + (kv_row * kv.D + kv_col) * OB
                                : reinterpret_cast<uint8_t*>(out) + ((size_t)row * N + col0) * OB;
      float4 res[NQ];
#pragma unroll
      for (int j = 0; j < NQ; ++j)
        res[j] = EPI == 1 && valid ? reinterpret_cast<const float4*>(dst)[j] : make_float4(0.f, 0.f, 0.f, 0.f);
      cluster_wait();                                      // every CTA of the cluster has started
      ok = ptx::mbar_wait(tfull_bar, 0, abort_flag);
      if (ok) {
        ptx::tc_fence_after();
        // ---- partial sums to the owners of the columns (consecutive lanes write consecutive 16 bytes)
        const uint32_t slot = recv + (uint32_t)(rank * NQ * BM + r) * 16u;
        uint32_t v[BN / 32][32];
#pragma unroll
        for (int c = 0; c < BN / 32; ++c) ptx::tmem_ld_32x32(t_row + 32u * c, v[c]);
#pragma unroll
        for (int c = 0; c < BN / 32; ++c) ptx::tmem_ld_wait(v[c]);
        ptx::tc_fence_before();
        if (valid) {
#pragma unroll
          for (int c = 0; c < BN / 32; ++c)
#pragma unroll
            for (int q = 0; q < 8; ++q)
              st_cluster_v4(ptx::mapa(slot, (uint32_t)((32 * c + 4 * q) / OWN)) + (uint32_t)((32 * c + 4 * q) % OWN) * (BM * 4u),
                            v[c] + 4 * q);
        }
        __syncwarp();
        if (lane < CS) ptx::mbar_arrive_cluster(ptx::mapa(recv_bar, (uint32_t)lane));
      }
      // tensor memory is given back while the other CTAs' partial sums arrive, not after them
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (warp == 2) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, BN);
      }
      if (ok) {
        // ---- the sum over the cluster, in rank order
        ok = ptx::mbar_wait_cluster(recv_bar, 0, abort_flag);
        if (ok && valid) {
          constexpr int NG = EPI == 1 ? 2 : 4;              // float4s per 32 bytes of output
          const bool sector = (reinterpret_cast<uintptr_t>(dst) & 31) == 0;
          auto total = [&](int j) -> float4 {
            float4 f = ld_shared_v4(recv + (uint32_t)(j * BM + r) * 16u);
#pragma unroll
            for (int src = 1; src < CS; ++src) {
              const float4 p = ld_shared_v4(recv + (uint32_t)((src * NQ + j) * BM + r) * 16u);
              f.x += p.x; f.y += p.y; f.z += p.z; f.w += p.w;
            }
            f.x += bv[j].x; f.y += bv[j].y; f.z += bv[j].z; f.w += bv[j].w;
            if (EPI == 1) { f.x += res[j].x; f.y += res[j].y; f.z += res[j].z; f.w += res[j].w; }
            return f;
          };
          if (NQ % NG == 0) {
#pragma unroll
            for (int j = 0; j < NQ / NG; ++j) {
              float4 f[NG];
#pragma unroll
              for (int e = 0; e < NG; ++e) f[e] = total((NG * j + e) % NQ);
              finish32<EPI>(f, dst + 32 * j, sector, a_bf16 != 0);
            }
          } else {                                         // eight 16-bit columns: half of that
            float4 f[NG] = {};
#pragma unroll
            for (int e = 0; e < NQ && e < NG; ++e) f[e] = total(e);
            finish16<EPI>(f[0], f[1], dst, a_bf16 != 0);
          }
        }
      }
    }
    if (!ok && lane == 0) *(volatile int*)status = STK_EPILOGUE;
  }
  if (CS > 1 && warp < 2) cluster_wait();
  ptx::tc_fence_before();
  __syncthreads();
  if (CS == 1 && warp == 2) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, BN);
  }
  if (CS > 1 && *abort_flag) {                             // gave up: stay until no CTA of the cluster can write here
    cluster_arrive();
    cluster_wait();
  }
}

template <int BN, int CS, int EPI>
cudaError_t launch_one(const CUtensorMap& ta, const CUtensorMap& tw, int M, int N, int K, int a_rows, const float* bias,
                       void* out, const KvScatter& kv, int a_bf16, int* status, cudaStream_t st) {
  const int n_tiles = ((M + BM - 1) / BM) * (N / BN);
  const int fixed = 1024 + 256 + (CS > 1 ? BM * BN * 4 : BN * 4);
  const int stage = a_rows * BK * 2 + BN * BK * 2;
  const int n_it = (K / BK + CS - 1) / CS;
  constexpr int budget = BN == 128 && CS > 1 ? kSmemBudgetWide : kSmemBudget;
  int stages = (budget - fixed) / stage;
  if (stages > kMaxStages) stages = kMaxStages;
  if (stages > n_it) stages = n_it;
  // The MMA reads 128 rows of A from the last slot on, whatever they hold, and without a cluster the ring ends as the
  // epilogue's 32 KB of staging boxes.
  size_t ring = (size_t)stages * stage;
  const size_t reach = (size_t)(stages - 1) * a_rows * BK * 2 + BM * BK * 2;
  if (CS > 1 ? reach > ring + BM * BN * 4 : reach > ring) ring = reach;
  if (CS == 1 && ring < 32768) ring = 32768;
  const size_t smem = fixed + ring;
  OutMap<CS> to = {};
  if constexpr (CS == 1)
    if (!tma_make_store_map(&to, out, (uint64_t)M, (uint64_t)N, EPI == 1 ? 4 : 2)) return cudaErrorInvalidValue;
  static size_t smem_set[kMaxDevices] = {};
  cudaError_t e = ensure_dynamic_smem(gemm_splitk_kernel<BN, CS, EPI>, (size_t)budget, smem_set);
  if (e != cudaSuccess) return e;
  return launch_pdl_cluster(gemm_splitk_kernel<BN, CS, EPI>, dim3(n_tiles * CS), dim3(kThreads), smem, CS, st, ta, tw, to, M, N,
                            K, a_rows, stages, (int)ring, bias, out, kv, a_bf16, status);
}

}  // namespace

// Rows of A per tile: the row blocks share the rows evenly, so that the last one is not a tile of padding that costs as
// much to feed as the others.  A whole number of 8-row swizzle atoms, or of 32-row store boxes where TMA stores.
static int rows_per_tile(int M, int cs) {
  const int n_m = (M + BM - 1) / BM, step = cs > 1 || n_m == 1 ? 8 : 32;
  return ((M + n_m - 1) / n_m + step - 1) / step * step;
}

// Estimated time of one shape in microseconds: a fixed cost, the K loop (hand-overs of a 64-wide block, or its bytes at
// the 114 KB/us that an SM is fed with from L2, whichever is more), and with a cluster its start, the exchange of partial
// sums through distributed shared memory and the second CTA of an SM (without one, two CTAs of an SM hide each other).
// The constants are fitted to 156 measured shapes (M 8 to 5248, the projections of widths 768, 1024 and 1280, every tile
// and cluster size): the choice costs 0.5 % over the fastest shape on average; before the fit, without the 128-column
// clusters, 3.6 %.  M x N x K, us: 8 x 4096 x 1024 5.0 -> 4.0, 82 x 2304 x 768 4.3 -> 4.0, 390 x 4096 x 1024 9.5 -> 7.7,
// 390 x 1024 x 4096 12.4 -> 10.1, 520 x 1024 x 4096 15.4 -> 12.6, 390 x 1280 x 5120 18.7 -> 15.0.
double gemm_splitk_cost(int M, int N, int K, SplitKShape shape) {
  const int bn = shape.bn, cs = shape.cs;
  const int n_kb = K / BK, rows = rows_per_tile(M, cs);
  if (N % bn || n_kb < cs) return 1e30;
  const double ctas = (double)((M + BM - 1) / BM) * (N / bn) * cs, load = ctas / device_sm_count();
  const double share = load <= 1.0 ? 1.0 : (cs == 1 && load <= 2.0 ? 0.956 + 0.044 * load : std::ceil(load));
  const double feed = (rows + bn) * 128 / 114e3, hand_over = rows > 32 ? 0.11 : 0.184;
  double t = 1.81 + 0.006 * ctas + share * ((n_kb + cs - 1) / cs) * (feed > hand_over ? feed : hand_over);
  if (cs == 1) return t + 0.41 * bn / 64;
  t += 0.68 + 0.157 * cs + share * rows * bn * 4 * (cs - 1) / cs / 28.6e3;
  if (load > 1.0) t += 1.34;
  return bn == 128 ? t + 0.15 : t;
}

SplitKShape gemm_splitk_pick(int M, int N, int K) {
  static const SplitKShape shapes[] = {{64, 1}, {64, 2}, {64, 4}, {64, 8}, {32, 2}, {32, 4}, {128, 1}, {128, 2}, {128, 4}, {128, 8}};
  SplitKShape best = {128, 1};
  double t = 1e30;
  for (const SplitKShape& s : shapes) {
    const double c = gemm_splitk_cost(M, N, K, s);
    if (c < t) { t = c; best = s; }
  }
  return best;
}

cudaError_t launch_gemm_splitk(const void* a, int lda, int M, const void* w, const float* bias, int N, int K, int epilogue,
                               void* out, bool a_bf16, int* status, cudaStream_t st, SplitKShape shape,
                               const KvScatter* kv_scatter) {
  if (M == 0) return cudaSuccess;
  const int bn = shape.bn, cs = shape.cs;
  if ((bn != 32 && bn != 64 && bn != 128) || N % bn || K % BK || K / BK < cs || lda % 8 ||
      (((uintptr_t)a | (uintptr_t)w | (uintptr_t)out | (uintptr_t)bias) & 15))
    return cudaErrorInvalidValue;
  KvScatter kv = {nullptr, nullptr, 1, 1, 1, 1 << 30};
  if (epilogue == 4) {
    if (!kv_scatter || !kv_scatter->cache || N != 3 * kv_scatter->D || kv_scatter->D % bn || ((uintptr_t)kv_scatter->cache & 15))
      return cudaErrorInvalidValue;
    kv = *kv_scatter;
  }
  const int a_rows = rows_per_tile(M, cs);
  CUtensorMap ta, tw;
  {
    const uint64_t dims[2] = {(uint64_t)K, (uint64_t)M}, strides[1] = {(uint64_t)lda * 2};
    const uint32_t box[2] = {BK, (uint32_t)a_rows};
    if (!tma_make_map_bf16(&ta, a, 2, dims, strides, box, true, !a_bf16)) return cudaErrorInvalidValue;
  }
  {
    const uint64_t dims[2] = {(uint64_t)K, (uint64_t)N}, strides[1] = {(uint64_t)K * 2};
    const uint32_t box[2] = {BK, (uint32_t)bn};
    if (!tma_make_map_bf16(&tw, w, 2, dims, strides, box, true, !a_bf16)) return cudaErrorInvalidValue;
  }
#define MARCHE_SPLITK_CASE(BN_, CS_)                                                                                   \
  if (bn == BN_ && cs == CS_) {                                                                                        \
    if (epilogue == 0) return launch_one<BN_, CS_, 0>(ta, tw, M, N, K, a_rows, bias, out, kv, a_bf16, status, st);      \
    if (epilogue == 1) return launch_one<BN_, CS_, 1>(ta, tw, M, N, K, a_rows, bias, out, kv, a_bf16, status, st);      \
    if (epilogue == 2) return launch_one<BN_, CS_, 2>(ta, tw, M, N, K, a_rows, bias, out, kv, a_bf16, status, st);      \
    if (epilogue == 4) return launch_one<BN_, CS_, 4>(ta, tw, M, N, K, a_rows, bias, out, kv, a_bf16, status, st);      \
  }
  MARCHE_SPLITK_CASE(32, 2) MARCHE_SPLITK_CASE(32, 4)
  MARCHE_SPLITK_CASE(64, 1) MARCHE_SPLITK_CASE(64, 2) MARCHE_SPLITK_CASE(64, 4) MARCHE_SPLITK_CASE(64, 8)
  MARCHE_SPLITK_CASE(128, 1) MARCHE_SPLITK_CASE(128, 2) MARCHE_SPLITK_CASE(128, 4) MARCHE_SPLITK_CASE(128, 8)
#undef MARCHE_SPLITK_CASE
  return cudaErrorInvalidValue;
}

}  // namespace marche

// K2 for a handful of rows (up to 16, or 32, by size: gemm_few_wins): out = epilogue(a * w^T + bias), with the LayerNorm of the rows (K1)
// in the same launch where the caller has the fp32 rows.
//
// What bounds it: latency.  One image without refresh has 4 to 26 active rows; a launch is a chain of hand-over, first operands,
// products, exchange and store.  Stamps in the tcgen05 split-K kernel at 16 x 2304 x 768 say where that goes once the rows are
// there: 1450 cycles until the MMAs of three K blocks are issued, 390 until the accumulator is complete, 1450 until it has been
// read from tensor memory and sent.  Here the products are mma.sync's and none of these links exists:
//   * a cluster of CS CTAs shares 16 rows x 8 NT columns and splits K, a CTA's warps split its slice of K in 32-wide blocks;
//   * every thread copies, with cp.async ahead of the dependency wait, the very 16 bytes of W that it will multiply, into a
//     slot of its own: no barrier, no swizzle, and the weights are on chip when the rows arrive;
//   * the rows go from L2 to registers as mma.sync fragments without shared memory: a dot product does not mind in which order
//     k is taken, so a thread's eight consecutive values of a row serve as its pairs of two k16 steps, as the same eight
//     columns of W do on the other side;
//   * with the fp32 rows at hand the cluster normalises them: mean and squared deviations of a CTA's slice of every row go to the
//     other CTAs, and the LayerNorm launch before it is gone;
//   * partial sums meet in the CTA's shared memory, then in the CTA that owns the pair of columns, both in a fixed order; what
//     crosses the cluster goes by st.async, whose bytes the receiver's barrier counts (no fence, no barrier of the cluster).
// A block of a step (six blocks over 320 tokens; 7 launches with the split-K kernel, 5 with this one), us: width 768, 4 rows 24.9 and 18.8,
// 16 rows 24.6 and 19.6, 32 rows 24.9 and 22.8; width 1024, 16 rows 27.9 and 23.2; width 1280, 16 rows 31.2 and 27.9.  Waits on barriers
// of shared memory are bounded; those on the cluster's barrier return once every CTA has arrived or left, which none of them delays.
#include "common.cuh"
#include "kernels.h"
#include "launch_pdl.h"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace marche {

namespace {

constexpr int kBlockK = 32;                // K block of a warp: four lanes of a row hold eight values each
constexpr int kMaxWarps = 16;              // all along K; two CTAs of 64 registers a thread per SM
constexpr int kRows = 16;                  // of a tile
constexpr int kSmemMax = 110 * 1024;       // two CTAs per SM, this launch's and the next one's
constexpr int kSmemSm = 228 * 1024;        // of an SM, 1 KB of it for every CTA

MARCHE_DEVINL void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
MARCHE_DEVINL void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
MARCHE_DEVINL void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
MARCHE_DEVINL void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
MARCHE_DEVINL uint4 ld_shared_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
template <bool BF>
MARCHE_DEVINL void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  if (BF)
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  else
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Columns of a CTA's slice of a row (LayerNorm), and the reciprocals that the statistics' merges need.
struct NormShape { float inv_cols, cols_cta, inv_warps; };
enum { ST_GEMM_FEW = 0x64 };

// Grid: CS * N / (8 NT) * n_m CTAs (n_m groups of 16 rows); the CS CTAs of a cluster share a tile.  NORM: a is fp32 [M][lda], to be
// normalised first, and every warp has one K block.
// The code runs once per launch, so what it costs is its instructions, fetched cold, and its dependent steps: nothing behind the
// dependency wait divides by a runtime value (the first version spent 4600 of 10 500 cycles on such divisions).
template <int NT, int CS, bool NORM, bool BF>
__global__ void __launch_bounds__(kMaxWarps * 32, 2)
gemm_few_kernel(const void* __restrict__ a, int lda, int M, const uint16_t* __restrict__ w, const float* __restrict__ bias, int N,
                int K, int epi, void* __restrict__ out, const KvScatter kv, const float* __restrict__ gamma,
                const float* __restrict__ beta, float eps, const NormShape sh, int kbw, int n_m, int* __restrict__ status) {
  static_assert(!NORM || CS % 2 == 0, "the statistics go through the cluster");
  constexpr int cs = CS, pairs = NT * 64, own = pairs / cs;  // output pairs of the cluster's tile, of this CTA
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ __align__(8) uint64_t bars[2];                // statistics there, partial sums there
  __shared__ int abort_flags[1];
  const int threads = blockDim.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, warps = threads >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  const int rank = cs > 1 ? (int)ptx::cluster_ctarank() : 0;
  const int tile = (int)blockIdx.x / cs, n_blk = tile / n_m, m0 = (tile - n_blk * n_m) * kRows;
  const int n_kb = K / kBlockK, kb0 = rank * n_kb / cs, kb1 = (rank + 1) * n_kb / cs;
  // shared memory: per warp its W slots [K block][NT][lane] of 16 bytes, then over them its partial sums | received [rank][own] |
  // statistics: of the warps [warp][16], of the CTAs [rank][16] | gamma, beta of the slice
  constexpr int w_step = 512;
  const int area = kbw * NT * w_step;                     // bytes of a warp
  const uint32_t w_slot = ptx::smem_u32(smem) + (uint32_t)(warp * area + lane * 16);
  float2* recv = reinterpret_cast<float2*>(smem + warps * area);
  float2* s_warp = recv + (cs > 1 ? pairs : 0);
  float2* s_cta = s_warp + warps * kRows;
  float* s_gamma = reinterpret_cast<float*>(s_cta + cs * kRows);
  float* s_beta = s_gamma + (kb1 - kb0) * kBlockK;
  const uint32_t bar_stats = ptx::smem_u32(bars), bar_sums = bar_stats + 8u;
  volatile int* abort_flag = abort_flags;

  if (tid == 0) {
    ptx::mbar_init(bar_stats, 1);
    ptx::mbar_init(bar_sums, 1);
    abort_flags[0] = 0;
    ptx::fence_barrier_init();
    if (NORM) ptx::mbar_expect_tx(bar_stats, (uint32_t)(cs * kRows) * 8u);
    ptx::mbar_expect_tx(bar_sums, (uint32_t)pairs * 8u);
  }
  if (NORM) {
    const uint32_t sg = ptx::smem_u32(s_gamma), sb = ptx::smem_u32(s_beta);
    for (int i = tid; i < (kb1 - kb0) * (kBlockK / 4); i += threads) {
      cp_async16(sg + 16u * i, gamma + kb0 * kBlockK + 4 * i);
      cp_async16(sb + 16u * i, beta + kb0 * kBlockK + 4 * i);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  const int mine = (kb1 - kb0 - warp + warps - 1) / warps;      // K blocks of this warp
  {
    const uint16_t* src = w + (size_t)(n_blk * 8 * NT + g) * K + (kb0 + warp) * kBlockK + t4 * 8;
    for (int i = 0; i < mine; ++i, src += warps * kBlockK)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) cp_async16(w_slot + (i * NT + nt) * w_step, src + (size_t)nt * 8 * K);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // pair q of the tile: column group of 8 * 64 + accumulator half * 32 + lane
  auto row_of = [&](int q) { return m0 + ((q >> 5) & 1) * 8 + ((q & 31) >> 2); };
  auto col_of = [&](int q) { return (n_blk * NT + (q >> 6)) * 8 + 2 * (q & 3); };
  // Where a finished pair goes: for a K or V column the cache row of its token, which is known after the wait.
  auto out_of = [&](int row, int col, const int32_t*& token) -> uint8_t* {
    token = nullptr;
    if (epi == 1) return reinterpret_cast<uint8_t*>(out) + ((size_t)row * N + col) * 4;
    if (epi != 4 || col < kv.D) return reinterpret_cast<uint8_t*>(out) + ((size_t)row * N + col) * 2;
    const int which = col >= 2 * kv.D ? 1 : 0, b = row / kv.n;
    if (kv.idx) token = kv.idx + row;
    return reinterpret_cast<uint8_t*>(kv.cache) +
           ((((size_t)which * kv.B + b) * kv.S + (kv.idx ? 0 : row - b * kv.n)) * kv.D + (col - (which + 1) * kv.D)) * 2;
  };
  const int row_q = row_of(rank * own + tid), col_q = col_of(rank * own + tid);
  const bool has_q = tid < own && row_q < M;               // this thread's first pair
  const int32_t* token = nullptr;
  uint8_t* dst_q = has_q ? out_of(row_q, col_q, token) : nullptr;
  float2 bias_q = has_q ? __ldg(reinterpret_cast<const float2*>(bias + col_q)) : make_float2(0.f, 0.f), res_q = make_float2(0.f, 0.f);
  __syncthreads();                                         // the barriers exist
  if (cs > 1) cluster_arrive();                            // ... and the cluster may know
  pdl_sync();                                              // everything above overlapped the previous kernel's tail

  bool ok = true;
  const int t_q = token ? *token : 0;
  float acc[NT][4] = {};
  if constexpr (!NORM) {
    constexpr int AHEAD = 2;
    const uint4* rows[2];
#pragma unroll
    for (int h = 0; h < 2; ++h)                            // (rows beyond M repeat the last one and are not stored)
      rows[h] = reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(a) + (size_t)min(m0 + 8 * h + g, M - 1) * lda +
                                               (kb0 + warp) * kBlockK + t4 * 8);
    uint4 v[AHEAD][2];
    auto fetch = [&](int i, uint4 (&x)[2]) {
      if (i < mine) {
#pragma unroll
        for (int h = 0; h < 2; ++h) x[h] = rows[h][(size_t)i * (warps * (kBlockK / 8))];
      }
    };
#pragma unroll
    for (int i = 0; i < AHEAD; ++i) fetch(i, v[i]);
    if (epi == 1 && has_q) res_q = *reinterpret_cast<const float2*>(dst_q);
    cp_async_wait_all();                                   // (a thread reads nobody's slots but its own)
#pragma unroll 1
    for (int i0 = 0; i0 < mine; i0 += AHEAD) {
#pragma unroll
      for (int j = 0; j < AHEAD; ++j) {
        if (i0 + j < mine) {
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            const uint4 b = ld_shared_v4(w_slot + ((i0 + j) * NT + nt) * w_step);
            mma_16816<BF>(acc[nt], v[j][0].x, v[j][1].x, v[j][0].y, v[j][1].y, b.x, b.y);
            mma_16816<BF>(acc[nt], v[j][0].z, v[j][1].z, v[j][0].w, v[j][1].w, b.z, b.w);
          }
          fetch(i0 + j + AHEAD, v[j]);
        }
      }
    }
  } else {
    // ---- one K block: the rows, the statistics of the warp's 32 columns
    float x[2][8];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4* src = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(a) + (size_t)min(m0 + 8 * h + g, M - 1) * lda +
                                                          (kb0 + warp) * kBlockK + t4 * 8);
      const float4 u = src[0], v = src[1];
      x[h][0] = u.x; x[h][1] = u.y; x[h][2] = u.z; x[h][3] = u.w;
      x[h][4] = v.x; x[h][5] = v.y; x[h][6] = v.z; x[h][7] = v.w;
    }
    float s[2], m2[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) s[h] = ((x[h][0] + x[h][1]) + (x[h][2] + x[h][3])) + ((x[h][4] + x[h][5]) + (x[h][6] + x[h][7]));
#pragma unroll
    for (int h = 0; h < 2; ++h) s[h] += __shfl_xor_sync(0xffffffffu, s[h], 1);
#pragma unroll
    for (int h = 0; h < 2; ++h) s[h] = (s[h] + __shfl_xor_sync(0xffffffffu, s[h], 2)) * (1.0f / kBlockK);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      m2[h] = 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) { const float d = x[h][e] - s[h]; m2[h] = fmaf(d, d, m2[h]); }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) m2[h] += __shfl_xor_sync(0xffffffffu, m2[h], 1);
#pragma unroll
    for (int h = 0; h < 2; ++h) m2[h] += __shfl_xor_sync(0xffffffffu, m2[h], 2);
    if (t4 == 0) {
#pragma unroll
      for (int h = 0; h < 2; ++h) s_warp[warp * kRows + 8 * h + g] = make_float2(s[h], m2[h]);
    }
    asm volatile("cp.async.wait_group 1;" ::: "memory");   // gamma and beta (W is another group)
    __syncthreads();                                       // the warps' statistics, and everybody's gamma and beta
    cluster_wait();                                        // every CTA of the cluster has started
    if (warp == 0) {                                       // the CTA's share of a row, to all CTAs of the cluster
      // Two lanes a row, every other warp's part each.  Squared deviations are summed around the merged mean and not as a
      // difference of sums: nothing cancels (variance off by 3e-7 where the difference left 6e-6, one warp's columns 50 deviations from the
      // others'), and a deviation whose square overflows leaves infinity, i.e. a row of beta, as in the LayerNorm launch.  The second
      // pass costs 120 cycles of 5000 (one image of 64 steps as a graph 28.7 -> 28.9 ms).
      const int row = lane & 15, odd = lane >> 4;
      const float pivot = s_warp[row].x;                   // (all counts are equal: the mean, around one of the means)
      float s1 = 0.f, dev = 0.f;
#pragma unroll
      for (int v = 0; v < kMaxWarps; v += 2)
        if (v + odd < warps) s1 += s_warp[(v + odd) * kRows + row].x - pivot;
      s1 += __shfl_xor_sync(0xffffffffu, s1, 16);
      const float mean = fmaf(s1, sh.inv_warps, pivot);
#pragma unroll
      for (int v = 0; v < kMaxWarps; v += 2)
        if (v + odd < warps) {
          const float2 p = s_warp[(v + odd) * kRows + row];
          const float d = p.x - mean;
          dev += fmaf(d * d, (float)kBlockK, p.y);
        }
      dev += __shfl_xor_sync(0xffffffffu, dev, 16);
      const uint32_t dst = ptx::smem_u32(s_cta + rank * kRows + row);
#pragma unroll
      for (int c = 0; c < cs; c += 2)
        ptx::st_async_v2(ptx::mapa(dst, (uint32_t)(c + odd)), mean, dev, ptx::mapa(bar_stats, (uint32_t)(c + odd)));
    }
    __syncwarp();                                          // (lanes that wait must not keep those that send from running)
    const float* gm = s_gamma + warp * kBlockK + t4 * 8;
    const float* bt = s_beta + warp * kBlockK + t4 * 8;
    const float4 g0 = *reinterpret_cast<const float4*>(gm), g1 = *reinterpret_cast<const float4*>(gm + 4);
    const float4 b0 = *reinterpret_cast<const float4*>(bt), b1 = *reinterpret_cast<const float4*>(bt + 4);
    ok = ptx::mbar_wait_cluster(bar_stats, 0, abort_flag);
    uint32_t u[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float2 q[cs];                                        // the CTAs' slices, merged in pairs
#pragma unroll
      for (int c = 0; c < cs; ++c) q[c] = s_cta[c * kRows + 8 * h + g];
#pragma unroll
      for (int n = 1; n < cs; n *= 2)
#pragma unroll
        for (int c = 0; c + n < cs; c += 2 * n) {
          const float d = q[c + n].x - q[c].x;
          q[c].x = fmaf(d, 0.5f, q[c].x);
          q[c].y = fmaf(d * d, 0.5f * n * sh.cols_cta, q[c].y + q[c + n].y);
        }
      const float mean = q[0].x, rstd = rsqrtf(q[0].y * sh.inv_cols + eps);
      const float* y = x[h];
      u[h][0] = pack_a16x2((y[0] - mean) * rstd * g0.x + b0.x, (y[1] - mean) * rstd * g0.y + b0.y, BF);
      u[h][1] = pack_a16x2((y[2] - mean) * rstd * g0.z + b0.z, (y[3] - mean) * rstd * g0.w + b0.w, BF);
      u[h][2] = pack_a16x2((y[4] - mean) * rstd * g1.x + b1.x, (y[5] - mean) * rstd * g1.y + b1.y, BF);
      u[h][3] = pack_a16x2((y[6] - mean) * rstd * g1.z + b1.z, (y[7] - mean) * rstd * g1.w + b1.w, BF);
    }
    cp_async_wait_all();
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const uint4 b = ld_shared_v4(w_slot + nt * w_step);
      mma_16816<BF>(acc[nt], u[0][0], u[1][0], u[0][1], u[1][1], b.x, b.y);
      mma_16816<BF>(acc[nt], u[0][2], u[1][2], u[0][3], u[1][3], b.z, b.w);
    }
  }

  // ---- the sum over the CTA's warps, to the CTA that owns the pair
  {
    __syncwarp();                                          // (every lane has read its slots)
    float2* dst = reinterpret_cast<float2*>(smem + warp * area) + lane;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      dst[nt * 64] = make_float2(acc[nt][0], acc[nt][1]);
      dst[nt * 64 + 32] = make_float2(acc[nt][2], acc[nt][3]);
    }
  }
  // A CTA whose statistics did not come sends no sums and tells the cluster, all of which waits for them: nobody stores anything.
  // (The others are still there for the same reason.)
  if (NORM && !ok) ptx::cluster_raise(ptx::smem_u32(abort_flags), cs);
  bool silent = false;
  if (NORM) silent = __syncthreads_or(!ok);
  else __syncthreads();
  auto sum_warps = [&](int q) {
    const uint8_t* p = smem + q * 8;
    float2 f = *reinterpret_cast<const float2*>(p);
#pragma unroll
    for (int v = 1; v < kMaxWarps; ++v)
      if (v < warps) {
        const float2 o = *reinterpret_cast<const float2*>(p + v * area);
        f.x += o.x;
        f.y += o.y;
      }
    return f;
  };
  if (cs > 1) {
    if (!NORM) cluster_wait();                             // every CTA of the cluster has started
    const uint32_t dst = ptx::smem_u32(recv + rank * own);
    for (int q = silent ? pairs : tid; q < pairs; q += threads) {
      const float2 f = sum_warps(q);
      const uint32_t o = (uint32_t)q / own;
      ptx::st_async_v2(ptx::mapa(dst + (uint32_t)q % own * 8u, o), f.x, f.y, ptx::mapa(bar_sums, o));
    }
    __syncwarp();
    ok = ptx::mbar_wait_cluster(bar_sums, 0, abort_flag) && ok;
    if (!ok) *(volatile int*)status = ST_GEMM_FEW;
  }
  // ---- the sum over the CTAs, in rank order, and the epilogue
  dst_q += (size_t)t_q * kv.D * 2;
  for (int q = tid; q < own && ok; q += threads) {
    if (q != tid) {                                        // (tiles of more pairs than threads)
      const int row = row_of(rank * own + q), col = col_of(rank * own + q);
      dst_q = row < M ? out_of(row, col, token) : nullptr;
      if (dst_q && token) dst_q += (size_t)*token * kv.D * 2;
      bias_q = __ldg(reinterpret_cast<const float2*>(bias + col));
      if (epi == 1 && dst_q) res_q = *reinterpret_cast<const float2*>(dst_q);
    }
    if (row_of(rank * own + q) >= M) continue;
    float2 f;
    if (cs > 1) {
      f = recv[q];
#pragma unroll
      for (int c = 1; c < cs; ++c) {
        f.x += recv[c * own + q].x;
        f.y += recv[c * own + q].y;
      }
    } else {
      f = sum_warps(q);
    }
    f.x += bias_q.x;
    f.y += bias_q.y;
    if (epi == 1) {
      f.x += res_q.x;
      f.y += res_q.y;
      *reinterpret_cast<float2*>(dst_q) = f;
    } else if (epi == 2) {
      gelu_erf_pair(f.x, f.y);
      *reinterpret_cast<uint32_t*>(dst_q) = pack_a16x2(f.x, f.y, BF);
    } else {
      *reinterpret_cast<uint32_t*>(dst_q) = pack_bf16x2(f.x, f.y);
    }
  }
  if (cs > 1) {
    __syncthreads();
    if (*abort_flag) {                                     // gave up: stay until no CTA of the cluster can write here
      cluster_arrive();
      cluster_wait();
    }
  }
}

struct Plan { int nt, cs, warps, kbw, n_m, ctas; size_t smem; };

// Columns per CTA and CTAs per cluster.  With the LayerNorm every warp has one K block, so that the slice of K is at most 512 columns, and
// as many columns as the registers hold, since every CTA reads and normalises the rows anew (16 rows, a block of a step of 24 blocks, us, as the
// kernel was when the plan was chosen: 8 NT = 64 columns and pairs of CTAs 17.3, 48 columns 17.1, 32 columns 17.9, clusters of four 17.6;
// width 1024 19.7, 20.6, 21.3 and 21.5).
// Without it 16 columns: whole K up to 2048 (17.2 us; pairs 17.1, of 32 columns 17.1), then pairs (17.1; whole K 18.6, of 32
// columns 17.4; width 1024 19.7 and 21.8), with two groups of rows pairs of 32 columns (21.8 -> 21.2).
bool make_plan(int M, int N, int K, bool norm, Plan* p) {
  const int n_kb = K / kBlockK, n_m = (M + kRows - 1) / kRows;
  const int cs = norm ? (n_kb <= 2 * kMaxWarps ? 2 : 4) : (K > 2048 ? 2 : 1), nt = norm ? 8 : (cs > 1 && n_m > 1 ? 4 : 2);
  const int per = (n_kb + cs - 1) / cs, kbw = (per + kMaxWarps - 1) / kMaxWarps, warps = (per + kbw - 1) / kbw;
  if (N % (8 * nt) || n_kb < cs || (norm && (kbw > 1 || n_kb % cs))) return false;
  *p = {nt, cs, warps, kbw, n_m, n_m * (N / (8 * nt)) * cs,
        (size_t)kbw * nt * warps * 512 + (cs > 1 ? nt * 512 : 0) + (norm ? (size_t)(warps + cs) * kRows * 8 + (size_t)per * kBlockK * 8 : 0)};
  return p->smem <= kSmemMax;
}

template <int NT, int CS, bool NORM, bool BF>
cudaError_t launch_one(const Plan& p, const void* a, int lda, int M, const void* w, const float* bias, int N, int K, int epi, void* out,
                       const KvScatter& kv, const float* gamma, const float* beta, float eps, int* status, cudaStream_t st) {
  static size_t smem_set[kMaxDevices] = {};
  static bool carved[kMaxDevices] = {};
  const auto kernel = gemm_few_kernel<NT, CS, NORM, BF>;
  cudaError_t e = ensure_dynamic_smem(kernel, (size_t)kSmemMax, smem_set);
  if (e == cudaSuccess) e = prefer_shared_memory(kernel, carved);
  if (e != cudaSuccess) return e;
  const float cta_cols = (float)(p.warps * kBlockK);
  const NormShape sh = {1.0f / K, cta_cols, 1.0f / p.warps};
  return launch_pdl_cluster(kernel, dim3(p.ctas), dim3(p.warps * 32), p.smem, CS, st,
                            a, lda, M, (const uint16_t*)w, bias, N, K, epi, out, kv, gamma, beta, eps, sh, p.kbw, p.n_m, status);
}

template <bool BF, typename... Args>
cudaError_t launch_any(const Plan& p, bool norm, Args... args) {
  if (norm) return p.cs == 2 ? launch_one<8, 2, true, BF>(p, args...) : launch_one<8, 4, true, BF>(p, args...);
  if (p.cs == 1) return launch_one<2, 1, false, BF>(p, args...);
  return p.nt == 2 ? launch_one<2, 2, false, BF>(p, args...) : launch_one<4, 2, false, BF>(p, args...);
}

}  // namespace

// One group of rows where the whole launch runs at once: 32 warps of 64 registers a thread fit an SM, and their shared memory has to.
// (Beyond, us, split-K and this kernel: 16 x 5120 x 1280 4.8 and 8.1, 16 x 6144 x 1536 5.5 and 9.7, 16 x 2560 x 4096 6.4 and 10.9; with the
// LayerNorm, a block of a step of 16 rows: width 1792, MLP 7168, 39.4 with LayerNorm launches, 42.9 without.  CTAs of 16 warps, which fill
// the SM, may be a third more: the QKV projection of width 2048 is level, 37.2 and 37.8 at MLP 4096, 49.9 and 47.8 in front of fc1 at 8192.)
// And not where a warp has many K blocks, so that every CTA reads long rows for its 16 columns: 16 x 2048 x 2048 3.7 and 4.3 (8 rows 5 %
// slower, one row level), 16 x 1536 x 6144 6.1 and 7.2, 1 row 6.1 and 6.3; with few columns the few CTAs are fed anyway (16 x 1024 x 6144
// 5.3 either way), and with more the split-K kernel's clusters of eight do not all fit (16 x 2048 x 6144 11.1 and 8.0, 16 x 4608 x 2048
// 9.5 and 6.7).
// Two groups of rows where the launch has no more warps than one CTA of 16 per SM (a block of a step, 32 rows: width 768, 192 CTAs of 12
// warps 24.0 -> 22.3; width 1024, 192 CTAs of 16 26.6 -> 27.0; width 1280, 640 CTAs 31.8 -> 43.6), and without the LayerNorm only for up
// to 1024 columns or a K of up to 1024 (24 rows: width 1280, MLP 2560, 27.9 and 30.6; width 1152, MLP 4608, 29.8 and 30.2; width 1024
// 25.1 and 25.0 to 25.6, by rows); three never (48 rows, width 768 25.5 -> 26.2).
bool gemm_few_wins(int M, int N, int K, bool norm) {
  Plan p;
  if (M > 2 * kRows || !make_plan(M, N, K, norm, &p)) return false;
  if (M > kRows) return p.ctas * p.warps <= kMaxWarps * device_sm_count() && (norm || N <= 1024 || K <= 1024);
  const int by_smem = kSmemSm / ((int)p.smem + 1024), by_regs = 2 * kMaxWarps / p.warps;
  const int fit = device_sm_count() * (by_smem < by_regs ? by_smem : by_regs);
  if (p.ctas > (norm && p.warps == kMaxWarps ? fit * 4 / 3 : fit)) return false;
  if (norm || N <= 1024) return true;
  return p.cs == 1 ? p.kbw <= 3 || M <= kRows / 2 || N >= 4096 : p.kbw <= 5 || N >= 2048;
}

cudaError_t launch_gemm_few(const void* a, int lda, int M, const void* w, const float* bias, int N, int K, int epilogue, void* out,
                            bool a_bf16, int* status, cudaStream_t st, const KvScatter* kv_scatter, const float* gamma, const float* beta,
                            float eps) {
  if (M == 0) return cudaSuccess;
  const bool norm = gamma != nullptr;
  if (N % 128 || K % 64 || lda % (norm ? 4 : 8) ||
      (((uintptr_t)a | (uintptr_t)w | (uintptr_t)out | (uintptr_t)bias | (uintptr_t)gamma | (uintptr_t)beta) & 15))
    return cudaErrorInvalidValue;
  KvScatter kv = {nullptr, nullptr, 1, 1, 1, 1 << 30};
  if (epilogue == 4) {
    if (!kv_scatter || !kv_scatter->cache || N != 3 * kv_scatter->D || ((uintptr_t)kv_scatter->cache & 15)) return cudaErrorInvalidValue;
    kv = *kv_scatter;
  }
  Plan p;
  if (!make_plan(M, N, K, norm, &p)) return cudaErrorInvalidValue;
  if (norm && epilogue == 1) return cudaErrorInvalidValue;
  return a_bf16 ? launch_any<true>(p, norm, a, lda, M, w, bias, N, K, epilogue, out, kv, gamma, beta, eps, status, st)
                : launch_any<false>(p, norm, a, lda, M, w, bias, N, K, epilogue, out, kv, gamma, beta, eps, status, st);
}

}  // namespace marche

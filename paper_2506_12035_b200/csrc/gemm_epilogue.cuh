// Epilogue of the tcgen05 GEMM kernels.  One warp owns 32 accumulator rows (TMEM lanes); it walks over its columns
// in chunks of 32, turns them into 128-byte-wide row pieces (32 fp32 or 64 16-bit output columns) in one of its two
// private 4 KB staging boxes in shared memory, in the TMA 128-byte swizzle (conflict-free: lane = row), and one lane
// hands the box to the TMA engine, which writes full 128-byte lines to global memory (rows beyond M are clipped by the
// tensor map).
//   EPI 0: out bf16 = acc + bias
//   EPI 1: out fp32 += acc + bias   -- TMA reduce-add in L2, no read in the SM, one add per element
//   EPI 2: out = GELU_erf(acc + bias) in the operand type, fp16 (saturating) or bf16 (feeds the next
//          projection as its A operand)
//   EPI 4: as EPI 0 for the q columns; the K and V columns go straight into scattered rows of the
//          K/V cache, so no separate write-back launch is needed
// It is a chain of latencies, not of bytes: the accumulator of the next chunk is on its way from tensor memory while
// a chunk is processed, the bias waits in shared memory, and a box is filled while the other one is still being read.
// With one box, and bias and accumulator fetched when needed, a 256 x 256 tile of a CTA pair took 5260 (bias),
// 7300 (GELU) and 8070 cycles (residual), exposed after the last tile of every launch and, for K = 1024, as long as the
// tile's main loop (8400 cycles).
#pragma once

#include "kernels.h"
#include "sm100_ptx.cuh"

namespace marche {

// One chunk of 32 columns (accumulator bits r, bias at shared address bias_s) into the box row at row_base: eight
// 16-byte pieces of fp32 (EPI 1), or pieces 4 half .. 4 half + 3 of a 16-bit row.
template <int EPI>
MARCHE_DEVINL void epilogue_chunk(const uint32_t (&r)[32], uint32_t bias_s, uint32_t row_base, int half, int lane, bool a_bf16) {
  auto bias4 = [&](int j) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(bias_s + 16u * j));
    return v;
  };
  if (EPI == 1) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float4 bv = bias4(j);
      const uint32_t dst = row_base + (uint32_t)((j ^ (lane & 7)) << 4);
      asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "f"(__uint_as_float(r[4 * j + 0]) + bv.x),
                   "f"(__uint_as_float(r[4 * j + 1]) + bv.y), "f"(__uint_as_float(r[4 * j + 2]) + bv.z),
                   "f"(__uint_as_float(r[4 * j + 3]) + bv.w) : "memory");
    }
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 b0 = bias4(2 * j), b1 = bias4(2 * j + 1);
      float v0 = __uint_as_float(r[8 * j + 0]) + b0.x, v1 = __uint_as_float(r[8 * j + 1]) + b0.y;
      float v2 = __uint_as_float(r[8 * j + 2]) + b0.z, v3 = __uint_as_float(r[8 * j + 3]) + b0.w;
      float v4 = __uint_as_float(r[8 * j + 4]) + b1.x, v5 = __uint_as_float(r[8 * j + 5]) + b1.y;
      float v6 = __uint_as_float(r[8 * j + 6]) + b1.z, v7 = __uint_as_float(r[8 * j + 7]) + b1.w;
      if (EPI == 2) {
        gelu_erf_pair(v0, v1); gelu_erf_pair(v2, v3); gelu_erf_pair(v4, v5); gelu_erf_pair(v6, v7);
      }
      const uint32_t dst = row_base + (uint32_t)(((half * 4 + j) ^ (lane & 7)) << 4);
      uint32_t p0, p1, p2, p3;
      if (EPI == 2) { p0 = pack_a16x2(v0, v1, a_bf16); p1 = pack_a16x2(v2, v3, a_bf16); p2 = pack_a16x2(v4, v5, a_bf16); p3 = pack_a16x2(v6, v7, a_bf16); }
      else { p0 = pack_bf16x2(v0, v1); p1 = pack_bf16x2(v2, v3); p2 = pack_bf16x2(v4, v5); p3 = pack_bf16x2(v6, v7); }
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(p0), "r"(p1), "r"(p2), "r"(p3) : "memory");
    }
  }
}

// A finished box of 64 bf16 columns into scattered cache rows: every quarter warp copies one whole 128-byte row piece
// per instruction (lane l: chunk l % 8 of row l / 8 + 4 i), so each global store instruction of the warp writes four
// full 128-byte lines.  dst_elem = element offset of this lane's row in the cache plus the column of this box, or -1
// for a row beyond M.
MARCHE_DEVINL void scatter_box(bf16* cache, long dst_elem, uint32_t box, int lane) {
  __syncwarp();
  const int chunk = lane & 7;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = (lane >> 3) + 4 * i;
    const long dst = __shfl_sync(0xffffffffu, dst_elem, row);
    uint32_t v0, v1, v2, v3;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v0), "=r"(v1), "=r"(v2), "=r"(v3)
                 : "r"(box + (uint32_t)row * 128u + (uint32_t)((chunk ^ (row & 7)) << 4)) : "memory");
    if (dst >= 0) *reinterpret_cast<uint4*>(cache + dst + chunk * 8) = make_uint4(v0, v1, v2, v3);
  }
  __syncwarp();                                         // the box may be refilled
}

// This lane's share of the bias of up to 128 columns (columns 4 lane .. 4 lane + 3; zeros for nullptr, a partial sum of
// a split K range whose bias another piece adds): loaded before the accumulator is waited for, stored to the slot that
// epilogue_columns reads after it.  Warps that work on the same columns share a slot: they write the same values.
MARCHE_DEVINL float4 epilogue_bias_load(const float* __restrict__ bias, int n, int lane) {
  return bias && 4 * lane < n ? __ldg(reinterpret_cast<const float4*>(bias) + lane) : make_float4(0.f, 0.f, 0.f, 0.f);
}
MARCHE_DEVINL void epilogue_bias_store(float4 v, int n, uint32_t bias_s, int lane) {
  if (4 * lane < n)
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(bias_s + 16u * lane), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
  __syncwarp();
}

// Columns [c_begin, c_end) of the accumulator whose row starts at TMEM address t_row; column 0 is output column `col`.
// Whole boxes only: multiples of 32 (EPI 1) or 64 columns.  bias_s: the bias of c_begin.  stage: this warp's two
// boxes (1024-byte aligned); n_box counts the boxes handed to the TMA engine so far.  SCATTER (EPI 0 only): the columns
// are K or V values and go to cache + dst_elem + column (dst_elem -1: no such row).
template <int EPI, bool SCATTER>
MARCHE_DEVINL void epilogue_columns(uint32_t t_row, int c_begin, int c_end, uint32_t bias_s, const CUtensorMap* out_map,
                                    int col, int row0, uint32_t stage, int& n_box, int lane, bool a_bf16,
                                    bf16* cache = nullptr, long dst_elem = -1) {
  uint32_t ra[32], rb[32];
  uint32_t box = stage;
  auto open_box = [&]() {
    box = stage + (uint32_t)(n_box & 1) * 4096u;
    // the box that was handed over two boxes ago must have been read out of shared memory
    if (lane == 0) { if (SCATTER) ptx::bulk_wait_read_all(); else ptx::bulk_wait_read_one(); }
    __syncwarp();
  };
  auto close_box = [&](int c) {
    if (SCATTER) {
      scatter_box(cache, dst_elem < 0 ? -1L : dst_elem + c, box, lane);
    } else {
      ptx::fence_proxy_async();                         // generic-proxy writes -> visible to the TMA engine
      __syncwarp();
      if (lane == 0) {
        if (EPI == 1) ptx::tma_reduce_add_2d(out_map, col + c, row0, box);
        else ptx::tma_store_2d(out_map, col + c, row0, box);
        ptx::bulk_commit();
      }
      ++n_box;
    }
  };
  if (c_begin >= c_end) return;
  ptx::tmem_ld_32x32(t_row + (uint32_t)c_begin, ra);
#pragma unroll 1
  for (int c = c_begin; c < c_end; c += 64) {
    ptx::tmem_ld_wait(ra);
    if (c + 32 < c_end) ptx::tmem_ld_32x32(t_row + (uint32_t)(c + 32), rb);
    open_box();
    epilogue_chunk<EPI>(ra, bias_s + 4u * (uint32_t)(c - c_begin), box + (uint32_t)lane * 128u, 0, lane, a_bf16);
    if (EPI == 1) close_box(c);
    if (c + 32 < c_end) {
      ptx::tmem_ld_wait(rb);
      if (c + 64 < c_end) ptx::tmem_ld_32x32(t_row + (uint32_t)(c + 64), ra);
      if (EPI == 1) open_box();
      epilogue_chunk<EPI>(rb, bias_s + 4u * (uint32_t)(c + 32 - c_begin), box + (uint32_t)lane * 128u, 1, lane, a_bf16);
      close_box(EPI == 1 ? c + 32 : c);
    }
  }
}

template <int EPI> struct EpiCols { static constexpr int value = (EPI == 1) ? 32 : 64; };

}  // namespace marche

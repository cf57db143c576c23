// K3 on the 5th-generation tensor cores, single pass (head_dim 64 or 80, no relevance scores): attention of
// the active queries over all S cached rows of one block (Algorithm 1 lines 6-8 == Eq. 5 by
// Appendix A), with the running-maximum / running-sum merge of Eq. 6-10 applied tile by tile.
//
// Persistent CTAs (one per SM).  The work of a CTA is a list of units, one unit = one 128-row query
// tile of one (sample, head) item against all S keys; three independent streams inside the CTA (one where a CTA has a single unit,
// four where that saves rounds that count, see attention_tc_streams) take the units in turn.  A unit is a latency chain (Q K^T -> read logits -> exponentials -> write
// weights -> P V), and the exponentials - 16 per clock and SM - are the scarce resource once the active set
// is large; the chains in flight per SM partition keep those units busy while each waits on its hand-overs.
// Each stream owns a query buffer, TMA rings of 64-key tiles (three of K, two of V: a K tile is used up a step earlier)
// that run ahead across units and 160 columns of tensor memory: S_j 64 columns (fp32 logits), P_j 32 (the weights, packed bf16),
// O_j 64.  The logits are free as soon as they have been read, so Q K^T of the next tile runs under the
// exponentials of this one and only the softmax itself is left of the chain.  Four streams, and three at head_dim 80 (O_j 80
// columns), have no columns to spare: there P_j overwrites S_j, P V of a tile and Q K^T of the next are issued together, in the
// order in which the tensor core executes them, and both are part of the chain.  Three streams with columns for P_j against four
// without, 128 x 16 items, S 320, us: 320 rows 107 and 122, 128 rows 42.5 and 50.5, 60 rows 36 and 40; 64 x 16 items, S 1088: 151
// rows 98 and 104, 1088 rows 528 and 590; one stream, with and without: S 1088, 144 items, 116 rows 17.1 and 19.5, S 2048, 64
// items, 200 rows 28.2 and 33.0.
// Roles, for three streams (18 warps of 96 registers a thread, 112 would fit; for four, in brackets, 24 of 80):
//   warps 0-11    [0-15] softmax: warps 4j .. 4j+3 serve stream j, one thread per query row.  A thread pulls its
//                 S row into registers (tcgen05.ld; without columns for P_j the first half again for its exponentials, since 80
//                 registers do not hold a row and its weights) and writes the weights to tensor memory
//                 (tcgen05.st), from where the tensor core reads them as the A operand of P V
//   warps 12-14   [16-19] TMA producer of stream 0, 1, ..: Q tile per unit, K and V rings
//   warps 15-17   [20-23] issue tcgen05.mma for stream 0, 1, ..: S_j = Q_j K^T (M128 x N64 x K64) of the next tile as soon as the
//                 last one has been read, O_j += P_j V (M128 x N64 x K64, V as an MN-major operand from
//                 shared memory) as soon as the weights are there; the last warp also allocates / frees tensor memory
// A warp can only reach the tensor-memory lanes of its quarter, and a quarter is one SM partition.  A query tile of
// fewer than 97 rows is therefore placed on other lanes by other streams, so that the partitions share the work.
// head_dim 80: a tile arrives as two boxes, columns 0-63 in rows of 128 bytes under the 128-byte swizzle and columns 64-79
// behind them in rows of 32 bytes under the 32-byte swizzle; Q K^T takes a fifth K = 16 step from the second one, P V a second
// MMA of 16 columns per step.
// Online softmax with a lazy reference maximum: the exponent reference of a row only moves when a
// tile's maximum exceeds it by more than 2^8 in the exponent, and only then is the row's O accumulator
// rescaled in tensor memory (by the row's own thread); weights
// therefore never exceed 256 and the final division by the row sum makes the result exact up to
// rounding.  All waits are bounded and report through the status word.
#include <cuda.h>

#include "kernels.h"
#include "launch_pdl.h"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace marche {

namespace {

constexpr int QT = 128;                    // query rows per unit (= TMEM lanes)
constexpr int KT = 64;                     // keys per tile
constexpr int NK = 3, NV = 2;              // K and V tiles in flight per stream
enum { ST_ATT_STREAM = 0x51 };
// barriers of one stream (8 bytes each); stream j's block starts at j * NB
enum { B_K_FULL = 0, B_K_EMPTY = B_K_FULL + NK, B_V_FULL = B_K_EMPTY + NK, B_V_EMPTY = B_V_FULL + NV, B_Q_FULL = B_V_EMPTY + NV,
       B_Q_EMPTY, B_S_FULL, B_S_FREE, B_P_FULL, B_O_FULL, NB };

constexpr int kStreams = 3;                // per CTA, but for launches of few units
template <int DH, int NS> struct Cfg {
  // The weights P_j have columns of their own where a stream's share leaves room: then Q K^T of the next tile runs under the
  // exponentials of this one.  Else they overwrite the logits, and P V and Q K^T are both part of the chain.
  static constexpr bool OWN_P = NS < (DH == 64 ? 4 : 3);
  static constexpr uint32_t COL_P = OWN_P ? KT : 0, COL_O = OWN_P ? KT + KT / 2 : KT;
  static constexpr int THREADS = NS * 6 * 32;                // per stream four softmax warps, a producer, an MMA issuer
  static constexpr int W_PROD = NS * 4, W_MMA = NS * 5;
  static constexpr int T_MAIN = KT * 128, T_BYTES = KT * DH * 2;   // a K or V tile; its columns 0-63
  static constexpr int Q_MAIN = QT * 128, Q_BYTES = QT * DH * 2;
  static constexpr uint32_t COL_STREAM = DH == 64 ? (OWN_P ? 160 : 128) : (OWN_P ? 192 : 160);
  static constexpr int TMEM_COLS = NS > 1 ? 512 : 256;
  // shared memory (from a 1024-byte aligned base)
  static constexpr int OFF_Q = 0;                            // [stream]
  static constexpr int OFF_K = OFF_Q + NS * Q_BYTES;         // [stream][slot]
  static constexpr int OFF_V = OFF_K + NS * NK * T_BYTES;    // [stream][slot]
  static constexpr int OFF_BAR = OFF_V + NS * NV * T_BYTES;
  static constexpr int OFF_MISC = OFF_BAR + 8 * NS * NB;     // tmem slot (4), abort flags (8)
  // (A CTA of one stream asks for more than it uses: two of them on an SM, where the kernel before has left room on one and
  // none yet on another, would share its exponential units; in the step 20 us became 37.)
  static constexpr int USED_BYTES = OFF_MISC + 32 + 1024, SMEM_BYTES = USED_BYTES > 120 * 1024 ? USED_BYTES : 120 * 1024;
  static_assert(NS * COL_STREAM <= TMEM_COLS && COL_O + DH <= COL_STREAM, "tensor memory budget");
  static_assert(SMEM_BYTES <= 227 * 1024 && T_BYTES % 1024 == 0 && Q_BYTES % 1024 == 0, "shared memory of one CTA");
};

MARCHE_DEVINL constexpr uint32_t idesc_bf16(int M, int N, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (b_mn_major ? (1u << 16) : 0u) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}
// MN-major operand tile written by TMA as [k rows][64 elements = 128 bytes] with the 128-byte
// swizzle: 8 k-rows form a 1024-byte atom (stride byte offset), one atom wide in MN.
MARCHE_DEVINL uint64_t smem_desc_mn_sw128(uint32_t addr) {
  const uint32_t lo = ((addr & 0x3FFFFu) >> 4) | ((1024u >> 4) << 16);
  const uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);
  return ((uint64_t)hi << 32) | lo;
}
// The same for tiles of 32-byte rows (16 elements) under the 32-byte swizzle: 8 rows form a 256-byte atom.  K-major: one
// K = 16 step of an operand; MN-major: 16 columns.
MARCHE_DEVINL uint64_t smem_desc_sw32(uint32_t addr) {
  const uint32_t lo = ((addr & 0x3FFFFu) >> 4) | ((256u >> 4) << 16);
  const uint32_t hi = (256u >> 4) | (1u << 14) | (6u << 29);
  return ((uint64_t)hi << 32) | lo;
}
// D[tmem] (+)= A[tmem] * B[smem desc]: the A operand (128 lanes x K 16-bit values, two per column) is
// read from tensor memory.
MARCHE_DEVINL void umma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
      "}\n"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// 32 lanes x N consecutive 32-bit columns: thread i of the warp accesses lane (base + i).
MARCHE_DEVINL void tmem_ld_32x16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
MARCHE_DEVINL void tmem_st_32x16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
MARCHE_DEVINL void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
MARCHE_DEVINL float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// Packed fp32 pairs (one instruction for two values): (a0, a1) * m + (b, b), and pairwise accumulate.
MARCHE_DEVINL void ffma2_bcast(float a0, float a1, float m, float b, float& r0, float& r1) {
  asm("{\n"
      ".reg .b64 ra, rm, rb, rr;\n"
      "mov.b64 ra, {%2, %3};\n"
      "mov.b64 rm, {%4, %4};\n"
      "mov.b64 rb, {%5, %5};\n"
      "fma.rn.f32x2 rr, ra, rm, rb;\n"
      "mov.b64 {%0, %1}, rr;\n"
      "}\n"
      : "=f"(r0), "=f"(r1) : "f"(a0), "f"(a1), "f"(m), "f"(b));
}
MARCHE_DEVINL void fadd2(float& acc0, float& acc1, float p0, float p1) {
  asm("{\n"
      ".reg .b64 ra, rp;\n"
      "mov.b64 ra, {%0, %1};\n"
      "mov.b64 rp, {%2, %3};\n"
      "add.f32x2 ra, ra, rp;\n"
      "mov.b64 {%0, %1}, ra;\n"
      "}\n"
      : "+f"(acc0), "+f"(acc1) : "f"(p0), "f"(p1));
}
MARCHE_DEVINL float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Units are dealt to the CTAs in turn: the k-th of a CTA is one of units k * grid .. k * grid + grid - 1, and unit i is query tile
// i % n_qt of item i / n_qt, so that CTAs that run at the same time read the same or neighbouring heads of the same cache rows.
// (Whole items dealt instead leave CTAs without work where items are few, S 1088, 512 items, 151 rows 70 us and 61; S 900, 320
// items, 300 rows 62 and 55; S 320, 512 items, 230 rows 25.4 and 24.1; level with many.)  Stream j of a CTA takes k = j, j + NS, ...
// An item's last tile can be much shorter than the others, and no CTA or stream should get the short ones only, or none: where
// there is more than one turn, a CTA's place in the row of CTAs moves on by `rotate` with every k and by `rotate_turn` with
// every turn of its streams (attention_tc_rotation chooses them so that the tile number changes along both).
struct Deal {
  int units, grid, rotate, rotate_turn;
  template <int NS> MARCHE_DEVINL int place(int k) const {
    return ((int)blockIdx.x + k * rotate + k / NS * rotate_turn) % grid;
  }
};
struct Unit { int b, h, start, row0; };    // the tile's first query row; the row on lane 0 (up to 96 before it)
template <int NS>
MARCHE_DEVINL Unit unit_of(int j, int u, const Deal& deal, int n_qt, int n, int H) {
  const int k = NS * u + j, i = k * deal.grid + deal.place<NS>(k);
  const int item = i / n_qt, qt = i - item * n_qt;
  Unit r;
  r.b = item / H;
  r.h = item - r.b * H;
  r.start = qt * QT;
  // a tile that needs one, two or three of the four lane quarters starts at another quarter in another stream
  const int quarters = n - r.start >= QT ? 4 : (n - r.start + 31) / 32;
  r.row0 = r.start - 32 * (quarters == 1 ? j : (quarters == 4 ? 0 : (j & 1) * (4 - quarters)));
  return r;
}

// tmap_kv, tmap_q: columns 0-63 of a head; the tails: columns 64-79 (unused at head_dim 64).
template <int DH, int NS>
__global__ void __launch_bounds__(Cfg<DH, NS>::THREADS, 1)
attention_tc_stream_kernel(const __grid_constant__ CUtensorMap tmap_kv, const __grid_constant__ CUtensorMap tmap_q,
                           const __grid_constant__ CUtensorMap tmap_kv_tail, const __grid_constant__ CUtensorMap tmap_q_tail, int n, int S, int H, int B, uint16_t* __restrict__ o, int o_bf16, int* __restrict__ status, int rotate,
                           int rotate_turn) {
  using C = Cfg<DH, NS>;
  constexpr bool OWN_P = C::OWN_P;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = ptx::smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - raw);
  auto bar = [&](int j, int i) { return base + C::OFF_BAR + 8u * (uint32_t)(j * NB + i); };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(gen + C::OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gen + C::OFF_MISC + 8);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int D = H * DH;
  const int n_kv = (S + KT - 1) / KT, n_qt = (n + QT - 1) / QT;
  const Deal deal = {B * H * n_qt, (int)gridDim.x, rotate, rotate_turn};
  const int units_cta = deal.units / deal.grid +           // (the last turn over the CTAs may not reach this one)
                        (deal.place<NS>(deal.units / deal.grid) < deal.units % deal.grid ? 1 : 0);
  constexpr float c_log2 = (DH == 64 ? 0.125f : 0.111803399f) * 1.4426950408889634f;   // log2(e) / sqrt(head_dim)

  if (threadIdx.x == 0) {
    for (int j = 0; j < NS; ++j) {
      for (int i = 0; i < NB; ++i) ptx::mbar_init(bar(j, i), i == B_P_FULL || i == B_S_FREE ? 4 : 1);
    }
    abort_flag[0] = 0;
    abort_flag[1] = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
  }
  if (warp == C::W_MMA + NS - 1) {
    ptx::tmem_alloc(ptx::smem_u32((const void*)tmem_slot), C::TMEM_COLS);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_sync();
  if (warp >= C::W_PROD) {
   if (warp < C::W_MMA) {
    // ---------------------------------------------------------------- TMA producer of stream j
    if (ptx::elect_one()) {
      const int j = warp - C::W_PROD, n_units = (units_cta + NS - 1 - j) / NS;
      ptx::prefetch_tensormap(&tmap_kv);
      ptx::prefetch_tensormap(&tmap_q);
      const uint64_t stream_once = ptx::l2_policy_evict_first();
      const uint32_t k0 = base + C::OFF_K + j * NK * C::T_BYTES, v0 = base + C::OFF_V + j * NV * C::T_BYTES;
      int n_k = 0, n_v = 0, ks = 0, vs = 0;                // K and V tiles issued so far; slots of the next
      uint32_t k_phase = 1, v_phase = 1;                   // an empty slot's first wait passes at once
      bool ok = true;
      for (int u = 0; u < n_units && ok; ++u) {
        const Unit un = unit_of<NS>(j, u, deal, n_qt, n, H);
        if (!ptx::mbar_wait(bar(j, B_Q_EMPTY), ((uint32_t)u & 1u) ^ 1u, abort_flag)) { ok = false; break; }
        ptx::mbar_expect_tx(bar(j, B_Q_FULL), C::Q_BYTES);
        ptx::tma_load_3d(base + C::OFF_Q + j * C::Q_BYTES, &tmap_q, un.h * DH, un.row0, un.b, bar(j, B_Q_FULL));
        if (DH > 64)
          ptx::tma_load_3d(base + C::OFF_Q + j * C::Q_BYTES + C::Q_MAIN, &tmap_q_tail, un.h * DH + 64, un.row0, un.b,
                           bar(j, B_Q_FULL));
        for (int kt = 0; kt < n_kv; ++kt) {
          if (!ptx::mbar_wait(bar(j, B_K_EMPTY + ks), k_phase, abort_flag)) { ok = false; break; }
          ptx::mbar_expect_tx(bar(j, B_K_FULL + ks), C::T_BYTES);
          ptx::tma_load_3d_hint(k0 + ks * C::T_BYTES, &tmap_kv, un.h * DH, kt * KT, un.b, bar(j, B_K_FULL + ks), stream_once);
          if (DH > 64)
            ptx::tma_load_3d_hint(k0 + ks * C::T_BYTES + C::T_MAIN, &tmap_kv_tail, un.h * DH + 64, kt * KT, un.b,
                                  bar(j, B_K_FULL + ks), stream_once);
          ++n_k;
          if (++ks == NK) { ks = 0; k_phase ^= 1u; }
          if (!ptx::mbar_wait(bar(j, B_V_EMPTY + vs), v_phase, abort_flag)) { ok = false; break; }
          ptx::mbar_expect_tx(bar(j, B_V_FULL + vs), C::T_BYTES);
          ptx::tma_load_3d_hint(v0 + vs * C::T_BYTES, &tmap_kv, un.h * DH, kt * KT, B + un.b, bar(j, B_V_FULL + vs), stream_once);
          if (DH > 64)
            ptx::tma_load_3d_hint(v0 + vs * C::T_BYTES + C::T_MAIN, &tmap_kv_tail, un.h * DH + 64, kt * KT, B + un.b,
                                  bar(j, B_V_FULL + vs), stream_once);
          ++n_v;
          if (++vs == NV) { vs = 0; v_phase ^= 1u; }
        }
      }
      if (!ok) {
        *(volatile int*)status = ST_ATT_STREAM;
        // let copies already issued land before the CTA's shared memory is released
        for (int back = 1; back <= NK && back <= n_k; ++back)
          ptx::mbar_wait(bar(j, B_K_FULL + (n_k - back) % NK), (uint32_t)((n_k - back) / NK) & 1u, abort_flag + 1, 20000000LL);
        for (int back = 1; back <= NV && back <= n_v; ++back)
          ptx::mbar_wait(bar(j, B_V_FULL + (n_v - back) % NV), (uint32_t)((n_v - back) / NV) & 1u, abort_flag + 1, 20000000LL);
      }
    }
   } else if (warp < C::W_MMA + NS) {
    // ---------------------------------------------------------------- MMA issuer of stream j
    // Slots, phases and descriptors are stepped and the branch is an elected one: with divisions by the tile count and
    // descriptors built per MMA in a lane-0 branch the issuer's own instructions were a fifth of a tile's chain.
    if (ptx::elect_one()) {
      const int j = warp - C::W_MMA, n_units = (units_cta + NS - 1 - j) / NS;
      constexpr uint32_t idesc_s = idesc_bf16(QT, KT, false);
      constexpr uint32_t idesc_o = idesc_bf16(QT, 64, true), idesc_tail = idesc_bf16(QT, 16, true);
      const int total = n_units * n_kv;
      const uint32_t d_s = tmem_base + (uint32_t)j * C::COL_STREAM, d_p = d_s + C::COL_P, d_o = d_s + C::COL_O;
      const uint64_t dq = ptx::smem_desc_k_sw128(base + C::OFF_Q + j * C::Q_BYTES),
                     dk0 = ptx::smem_desc_k_sw128(base + C::OFF_K + j * NK * C::T_BYTES),
                     dv0 = smem_desc_mn_sw128(base + C::OFF_V + j * NV * C::T_BYTES),
                     dq_tail = smem_desc_sw32(base + C::OFF_Q + j * C::Q_BYTES + C::Q_MAIN),
                     dk_tail0 = smem_desc_sw32(base + C::OFF_K + j * NK * C::T_BYTES + C::T_MAIN),
                     dv_tail0 = smem_desc_sw32(base + C::OFF_V + j * NV * C::T_BYTES + C::T_MAIN);
      bool ok = true;
      int s_slot = 0, s_i = 0, o_slot = 0, o_i = 0;        // ring slot and tile of the unit, of the next S and of the next O
      uint32_t k_phase = 0, v_phase = 0, q_phase = 0;
      // operands of the next S = Q K^T are there
      auto wait_s = [&]() -> bool {
        if (s_i == 0) {
          if (!ptx::mbar_wait(bar(j, B_Q_FULL), q_phase, abort_flag)) return false;
          q_phase ^= 1u;
        }
        return ptx::mbar_wait(bar(j, B_K_FULL + s_slot), k_phase, abort_flag);
      };
      auto issue_s = [&]() {
        const uint64_t dk = dk0 + (uint32_t)(s_slot * (C::T_BYTES >> 4));
#pragma unroll
        for (int k = 0; k < 4; ++k) ptx::umma_f16(d_s, dq + 2 * k, dk + 2 * k, idesc_s, k ? 1u : 0u);
        if (DH > 64) ptx::umma_f16(d_s, dq_tail, dk_tail0 + (uint32_t)(s_slot * (C::T_BYTES >> 4)), idesc_s, 1u);
        ptx::umma_commit(bar(j, B_S_FULL));                // (covers the P V before it, too, where they are issued together)
        ptx::umma_commit(bar(j, B_K_EMPTY + s_slot));
        if (++s_i == n_kv) {                               // the unit's last Q K^T: Q_j may be overwritten
          s_i = 0;
          ptx::umma_commit(bar(j, B_Q_EMPTY));
        }
        if (++s_slot == NK) { s_slot = 0; k_phase ^= 1u; }
      };
      if (total > 0) {
        ok = wait_s();
        ptx::tc_fence_after();
        if (ok) issue_s();
      }
      for (int t = 0; t < total && ok; ++t) {
        // a wait costs 110 cycles even if nothing is waited for, so those for the tiles come before the one for the weights
        if (t + 1 < total && !wait_s()) { ok = false; break; }
        if (OWN_P && t + 1 < total) {                      // the logits are in registers: the next ones may come
          if (!ptx::mbar_wait(bar(j, B_S_FREE), (uint32_t)t & 1u, abort_flag)) { ok = false; break; }
          ptx::tc_fence_after();
          issue_s();
        }
        if (!ptx::mbar_wait(bar(j, B_V_FULL + o_slot), v_phase, abort_flag) ||
            // (for a unit's first tile the previous output has been read out: every softmax warp did so before it wrote)
            !ptx::mbar_wait(bar(j, B_P_FULL), (uint32_t)t & 1u, abort_flag)) { ok = false; break; }
        ptx::tc_fence_after();
        const uint64_t dv = dv0 + (uint32_t)(o_slot * (C::T_BYTES >> 4));
#pragma unroll
        for (int k = 0; k < KT / 16; ++k) {
          umma_f16_ts(d_o, d_p + 8u * k, dv + 128 * k, idesc_o, (o_i | k) ? 1u : 0u);
          if (DH > 64)
            umma_f16_ts(d_o + 64u, d_p + 8u * k, dv_tail0 + (uint32_t)(o_slot * (C::T_BYTES >> 4)) + 32 * k, idesc_tail,
                        (o_i | k) ? 1u : 0u);
        }
        if (++o_i == n_kv) o_i = 0;
        if (OWN_P || o_i == 0) ptx::umma_commit(bar(j, B_O_FULL));
        // behind it, in the order of execution, the next logits over these weights
        if (!OWN_P && t + 1 < total) issue_s();
        ptx::umma_commit(bar(j, B_V_EMPTY + o_slot));
        if (++o_slot == NV) { o_slot = 0; v_phase ^= 1u; }
      }
      if (!ok) *(volatile int*)status = ST_ATT_STREAM;
    }
   }
  } else {
    // ---------------------------------------------------------------- softmax streams (one thread per row)
    const int j = warp >> 2;                               // stream (warps 4j .. 4j+3)
    const int n_units = (units_cta + NS - 1 - j) / NS;
    const int quarter = warp & 3;
    const int r = quarter * 32 + lane;                     // row inside the query tile = TMEM lane
    const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const uint32_t t_s = t_lane + (uint32_t)j * C::COL_STREAM, t_p = t_s + C::COL_P, t_o = t_s + C::COL_O;
    bool ok = true;
    int t = 0;                                             // tiles of this stream so far
    for (int u = 0; u < n_units && ok; ++u) {
      const Unit un = unit_of<NS>(j, u, deal, n_qt, n, H);
      const int row = un.row0 + r, row_w = un.row0 + quarter * 32;   // this thread's query row, the warp's first one
      const bool warp_valid = row_w >= un.start && row_w < n;
      float m_ref = -INFINITY, l = 0.f;                    // exponent reference (raw logit units), running sum
      for (int i = 0; i < n_kv; ++i, ++t) {
        // S_j of this tile is there (and without columns for P_j the previous P V is done)
        if (!ptx::mbar_wait(bar(j, B_S_FULL), (uint32_t)t & 1u, abort_flag)) { ok = false; break; }
        ptx::tc_fence_after();
        const int lim = S - i * KT;                        // keys of this tile that exist
        // The previous P V of this unit has read its weights and added to O_j.  (Without it no warp may announce this tile's
        // weights, not even one without rows: its arrival would count for the tile before.)
        auto previous_done = [&]() { return i == 0 || ptx::mbar_wait(bar(j, B_O_FULL), (uint32_t)(t - 1) & 1u, abort_flag); };
        if (warp_valid) {
          uint32_t va[KT / 2], vb[KT / 2];                 // logits of the first and second 32 keys
          ptx::tmem_ld_32x32(t_s, va);
          ptx::tmem_ld_32x32(t_s + KT / 2, vb);
          ptx::tmem_ld_wait(va);
          ptx::tmem_ld_wait(vb);
          if (OWN_P) {
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(j, B_S_FREE));
          }
          float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
          if (lim >= KT) {
#pragma unroll
            for (int c = 0; c < KT / 2; c += 2) {
              mx[c & 2] = max3(mx[c & 2], __uint_as_float(va[c]), __uint_as_float(va[c + 1]));
              mx[(c & 2) + 1] = max3(mx[(c & 2) + 1], __uint_as_float(vb[c]), __uint_as_float(vb[c + 1]));
            }
          } else {
#pragma unroll
            for (int c = 0; c < KT / 2; ++c) {
              if (c < lim) mx[c & 1] = fmaxf(mx[c & 1], __uint_as_float(va[c]));
              if (c + KT / 2 < lim) mx[2 + (c & 1)] = fmaxf(mx[2 + (c & 1)], __uint_as_float(vb[c]));
            }
          }
          if (!OWN_P) ptx::tmem_ld_32x32(t_s, va);         // again, for the exponentials
          const float tmax = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
          // lazy reference maximum: move it only when this tile exceeds it by more than 2^8
          const bool move = (tmax - m_ref) * c_log2 > 8.0f;   // also true for a unit's first tile (m_ref = -inf)
          const bool rescale = i > 0 && __any_sync(0xffffffffu, move);
          const float f = move ? ex2_approx((m_ref - tmax) * c_log2) : 1.0f;
          if (move) m_ref = tmax;
          const float neg = -m_ref * c_log2;
          // weights: p = 2^((s - m_ref) / sqrt(d) * log2 e), packed bf16 pairs, in place (pair c -> v[c])
          float ls[4] = {0.f, 0.f, 0.f, 0.f};
          auto weights = [&](uint32_t (&v)[KT / 2], int left) {   // left: keys of this half that exist
            if (left >= KT / 2) {                          // (two copies: no per-element selects for the full half)
#pragma unroll
              for (int c = 0; c < KT / 4; ++c) {
                float x0, x1;
                ffma2_bcast(__uint_as_float(v[2 * c]), __uint_as_float(v[2 * c + 1]), c_log2, neg, x0, x1);
                const float p0 = ex2_approx(x0), p1 = ex2_approx(x1);
                fadd2(ls[2 * (c & 1)], ls[2 * (c & 1) + 1], p0, p1);
                v[c] = pack_bf16x2(p0, p1);
              }
            } else {
#pragma unroll
              for (int c = 0; c < KT / 4; ++c) {
                float p0 = ex2_approx(fmaf(__uint_as_float(v[2 * c]), c_log2, neg));
                float p1 = ex2_approx(fmaf(__uint_as_float(v[2 * c + 1]), c_log2, neg));
                if (2 * c >= left) p0 = 0.f;
                if (2 * c + 1 >= left) p1 = 0.f;
                ls[c & 3] += p0 + p1;
                v[c] = pack_bf16x2(p0, p1);
              }
            }
          };
          weights(vb, lim - KT / 2);
          if (OWN_P) {
            ok = previous_done();
            ptx::tc_fence_after();
          } else {
            ptx::tmem_ld_wait(va);
          }
          tmem_st_32x16(t_p + KT / 4, vb);                 // (without columns of their own: over logits that have been read)
          weights(va, lim);
          tmem_st_32x16(t_p, va);
          if (rescale) {
            // this row's accumulator in tensor memory moves to the new reference
#pragma unroll 1
            for (int qc = 0; qc < DH / 16; ++qc) {
              uint32_t ov[16];
              tmem_ld_32x16(t_o + (uint32_t)(qc * 16), ov);
              ptx::tmem_ld_wait();
#pragma unroll
              for (int c = 0; c < 16; ++c) ov[c] = __float_as_uint(__uint_as_float(ov[c]) * f);
              tmem_st_32x16(t_o + (uint32_t)(qc * 16), ov);
            }
            l *= f;
          }
          l += (ls[0] + ls[1]) + (ls[2] + ls[3]);
          tmem_st_wait();
        } else if (OWN_P) {
          if (lane == 0) ptx::mbar_arrive(bar(j, B_S_FREE));
          ok = previous_done();
        }
        if (!ok) break;
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(bar(j, B_P_FULL));
      }
      if (!ok) break;
      // ---- end of the unit: O / l -> output rows
      if (!ptx::mbar_wait(bar(j, B_O_FULL), (uint32_t)(OWN_P ? t - 1 : u) & 1u, abort_flag)) { ok = false; break; }
      ptx::tc_fence_after();
      if (warp_valid) {
        const float inv = 1.0f / l;
        uint16_t* dst = o + ((size_t)un.b * n + row) * D + un.h * DH;
        uint32_t oa[32], ob[32], oc[16];
        ptx::tmem_ld_32x32(t_o, oa);
        ptx::tmem_ld_32x32(t_o + 32u, ob);
        ptx::tmem_ld_wait(oa);
        ptx::tmem_ld_wait(ob);
        // 16 columns per store, a whole 32-byte sector where the output is so aligned
        auto store = [&](const uint32_t* x, uint16_t* to) {
          uint32_t w[8];
#pragma unroll
          for (int e = 0; e < 8; ++e)
            w[e] = pack_a16x2(__uint_as_float(x[2 * e]) * inv, __uint_as_float(x[2 * e + 1]) * inv, o_bf16 != 0);
          if ((reinterpret_cast<uintptr_t>(o) & 31) == 0) {
            asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(to), "r"(w[0]), "r"(w[1]),
                         "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
          } else {
            reinterpret_cast<uint4*>(to)[0] = make_uint4(w[0], w[1], w[2], w[3]);
            reinterpret_cast<uint4*>(to)[1] = make_uint4(w[4], w[5], w[6], w[7]);
          }
        };
        if (row < n) {
          store(oa, dst);
          store(oa + 16, dst + 16);
          store(ob, dst + 32);
          store(ob + 16, dst + 48);
        }
        if (DH > 64) {
          tmem_ld_32x16(t_o + 64u, oc);
          ptx::tmem_ld_wait();
          if (row < n) store(oc, dst + 64);
        }
      }
    }
    if (!ok && lane == 0) *(volatile int*)status = ST_ATT_STREAM;
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (warp == C::W_MMA + NS - 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

}  // namespace

// How the units of a launch are dealt (Deal).  A CTA's next unit is grid + rotate units on, a stream's NS (grid + rotate) + rotate_turn:
// neither a multiple of an item's tiles.
// Items of one tile have no tiles to mix: there the units of the last turn should go to the CTAs that started first, as long as there are
// few turns (head_dim 80, 448 items, 80 rows, S 100 11.6 and 10.9 us, S 320 18.8 and 18.2; head_dim 64, 600 items, 116 rows, S 256 16.8
// and 15.8); over more than two turns of the streams rotation spreads the CTAs' reads (head_dim 80, 2048 items, 64 rows, S 1088 132 and 137).
int attention_tc_rotation(long units, int n_qt, int grid, int streams, int* rotate_turn) {
  *rotate_turn = 0;
  if (units <= (n_qt > 1 ? 1L : 2L) * streams * grid) return 0;
  const int rotate = n_qt > 1 && (grid + 1) % n_qt == 0 ? 2 : 1;
  *rotate_turn = n_qt > 1 && streams * (grid + rotate) % n_qt == 0 ? 1 : 0;
  return rotate;
}

namespace {

template <int DH, int NS>
cudaError_t launch_stream(const void* q, int ld_q, int B, int n, int S, int H, const void* cache_layer, void* o, bool o_bf16,
                          int* status, cudaStream_t st) {
  using C = Cfg<DH, NS>;
  const int D = H * DH;
  // columns 0-63 of a head as 128-byte rows, columns 64-79 as 32-byte rows, both swizzled
  CUtensorMap tkv, tq, tkv_tail, tq_tail;
  auto make = [&](CUtensorMap* map, const void* p, int ld, int rows, int samples, uint32_t box_rows, bool tail) {
    const uint64_t dims[3] = {(uint64_t)ld, (uint64_t)rows, (uint64_t)samples};
    const uint64_t strides[2] = {(uint64_t)ld * 2, (uint64_t)rows * ld * 2};
    const uint32_t box[3] = {tail ? 16u : 64u, box_rows, 1};
    return tma_make_map_bf16(map, p, 3, dims, strides, box, !tail, false, tail);
  };
  if (!make(&tkv, cache_layer, D, S, 2 * B, KT, false) || !make(&tq, q, ld_q, n, B, QT, false)) return cudaErrorInvalidValue;
  tkv_tail = tkv;
  tq_tail = tq;
  if (DH > 64 && (!make(&tkv_tail, cache_layer, D, S, 2 * B, KT, true) || !make(&tq_tail, q, ld_q, n, B, QT, true)))
    return cudaErrorInvalidValue;
  static size_t smem_set[kMaxDevices] = {};
  cudaError_t e = ensure_dynamic_smem(attention_tc_stream_kernel<DH, NS>, (size_t)C::SMEM_BYTES, smem_set);
  if (e != cudaSuccess) return e;
  const int sms = device_sm_count();
  const long units = (long)B * H * ((n + QT - 1) / QT);
  const int grid = units < sms ? (int)units : sms, n_qt = (n + QT - 1) / QT;
  int rotate_turn;
  const int rotate = attention_tc_rotation(units, n_qt, grid, NS, &rotate_turn);
  return launch_pdl(attention_tc_stream_kernel<DH, NS>, dim3(grid), dim3(C::THREADS), (size_t)C::SMEM_BYTES, st, tkv, tq, tkv_tail,
                    tq_tail, n, S, H, B, (uint16_t*)o, o_bf16 ? 1 : 0, status, rotate, rotate_turn);
}

}  // namespace

// Against the mma.sync kernels (alone, us, 2048 items over 320 keys), which take 48 rows or fewer (min_rows, marche_tuning) with up to
// five CTAs per SM and drop to two from 49 rows: head_dim 64: 60 rows 37 and 56, 77 rows 42 and 109, 320 rows 107 and 307; head_dim 80: 60
// rows 47 and 99, 320 rows 133 and 352.  33 to 48 rows at head_dim 64: over long sequences (S 1088, 1024 items, 41 rows: 56 and 62).  Over
// shorter ones the line dates from four streams whose weights shared the logits' columns (41 and 42, nothing in a step); the streams of today are
// faster there, too, from about 700 items on: S 320, 41 rows, 2048 items 36.5 and 40.9, 1024 items 22.3 and 24.0, 512 items 13.4 and 13.5,
// and a block of a step: width 1024, 128 samples 199 and 205, 64 samples 116 and 117, 32 samples 74.0 and 73.6; width 768, 64 samples 78.5 and
// 82.4.  At head_dim 80 over five key tiles or more (S 320, 2048 items, 41 rows: 46 and 52), unless the last round of units leaves the streams
// (three per SM) idle: 512 items on 444 streams 18.2 and 15.3, 1024 items 27.1 and 27.9.
// One item per SM or fewer at head_dim 80, 49 to 64 rows: the mma.sync kernel's four warps take an item faster than a stream that
// nothing overlaps with (S 1088, 128 items, 60 rows, back to back 18.1 and 20.5, eight blocks of a step 465 and 503; 41 rows, on three
// warps, 530 and 481).  At head_dim 64 the one-stream CTAs are slower back to back (S 1088, 128 items, 41 rows 18.6 and 17.8, 64 rows
// 18.7 and 16.5) but faster in a step, in which up to four of the mma.sync kernel's small CTAs fit an SM that is free early (eight
// blocks, 41 rows 404 and 431, 64 rows 442 and 472).
bool attention_tc_stream_wins(int n, int S, int dh, int items, int min_rows) {
  if (dh == 80 && items <= device_sm_count() && n > min_rows && 3 * n <= 4 * min_rows) return false;
  if (n > min_rows) return true;
  if (3 * n <= 2 * min_rows) return false;
  if (dh == 64) return S >= 512;
  const int streams = kStreams * device_sm_count(), rounds = (items + streams - 1) / streams;
  return S > 4 * KT && (rounds == 1 || 4 * items >= 3 * rounds * streams);
}

// Streams per CTA.  No more units than SMs: a CTA has one, and a CTA of one stream is smaller and starts sooner.  Head_dim 80: 144
// items, S 100, 80 rows 5.4 and 5.8 us; not over longer sequences.
// Head_dim 64: four streams take more units at a time than three, each more slowly, since their weights share the logits' columns.  That
// counts where it saves a round of two (192 items, S 320, 320 rows: 576 units on 444 or 592 streams 16.0 and 14.4 us), and over long
// sequences, where the tiles come from HBM and a fourth stream's are on their way meanwhile, also a round of three (64 x 16 items, us on
// three and four: S 640, 48 rows 38.7 and 37.0; S 1088, 64 rows 59.8 and 57.1, 116 rows 66.7 and 63.8; S 2048, 80 rows 110 and 104; 448
// items, S 1536, 200 rows 83.0 and 78.0; 116 rows over S 448 32.4 and 32.6, S 320 25.7 and 26.4), or of four behind a short last tile
// (S 1088, 2048 items, 151 rows 205 and 192, 800 items 83.5 and 81.2, with 200 rows 88.4 and 90.0; S 2048, 800 items, 151 rows 150 and 141).
// One in five costs (S 1088, 1024 items, 151 rows 98 and 104).
int attention_tc_streams(int n, int S, int dh, int items) {
  const long units = (long)items * ((n + QT - 1) / QT);
  const int sms = device_sm_count();
  if (units <= sms && (dh == 64 || S <= 2 * KT)) return 1;
  if (dh != 64) return kStreams;
  const long r3 = (units + kStreams * sms - 1) / (kStreams * sms), r4 = (units + 4L * sms - 1) / (4L * sms);
  const bool short_tile = n > QT && n % QT > 0 && n % QT <= 32;
  return r3 >= 2 * r4 || (S >= 8 * KT && 2 * r3 >= 3 * r4) || (S >= 14 * KT && short_tile && 3 * r3 >= 4 * r4) ? 4 : kStreams;
}

cudaError_t launch_attention_tc_stream(const void* q, int ld_q, int B, int n, int S, int H, int dh,
                                       const void* cache_layer, void* o, bool o_bf16, int* status, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  if ((dh != 64 && dh != 80) || ld_q % 8 || ((uintptr_t)q & 15) || ((uintptr_t)cache_layer & 15) || ((uintptr_t)o & 15) || S > 2048)
    return cudaErrorInvalidValue;
  switch (attention_tc_streams(n, S, dh, B * H)) {
    case 1:
      return dh == 64 ? launch_stream<64, 1>(q, ld_q, B, n, S, H, cache_layer, o, o_bf16, status, st)
                      : launch_stream<80, 1>(q, ld_q, B, n, S, H, cache_layer, o, o_bf16, status, st);
    case 4:
      return launch_stream<64, 4>(q, ld_q, B, n, S, H, cache_layer, o, o_bf16, status, st);
    default:
      return dh == 64 ? launch_stream<64, kStreams>(q, ld_q, B, n, S, H, cache_layer, o, o_bf16, status, st)
                      : launch_stream<80, kStreams>(q, ld_q, B, n, S, H, cache_layer, o, o_bf16, status, st);
  }
}

}  // namespace marche

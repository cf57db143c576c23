// K4: relevance-score reduction and top-K refresh selection (Section 4.2).
//
// One CTA per sample.  The per-head score partials [H][S] written by the attention
// kernel are summed in fixed head order (bit-reproducible run to run, unlike atomics),
// then the K-th best candidate under (score descending, index ascending) is found by a
// radix select and the K best are emitted in ascending index order through a block
// scan.  S <= 2048: a thread keeps its share of the candidates, at most eight, in registers.
//
// Bound by latency (64 samples of 1088 tokens are 0.3 MB): what counts is how many barriers stand in a row.  The
// tokens that must not be chosen are marked in shared memory by the same launch; the digits start at the first bit
// in which the candidates differ, which leaves one to three of a thousand scores in the crossing bin of the first pass;
// every warp scans the 512 bins for itself.  Six to eight barriers and one launch, where four fixed passes of four
// barriers took two launches.
#include "common.cuh"
#include "kernels.h"
#include "launch_pdl.h"
#include "tma_host.h"

namespace marche {

constexpr int kTopkThreads = 256;

// Order-preserving map of a finite float to uint32 (larger float -> larger key), with
// -0 mapped onto +0.
MARCHE_DEVINL uint32_t score_key(float f) {
  uint32_t u = __float_as_uint(f);
  if ((u << 1) == 0u) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Counter-based 32-bit mix of (seed, sample, token) for the random-selection ablation: xor the
// three words with odd multipliers, then two xorshift-multiply rounds.
MARCHE_DEVINL uint32_t mix32(uint32_t seed, uint32_t b, uint32_t t) {
  uint32_t x = seed ^ (b * 0x9E3779B1u) ^ (t * 0x85EBCA77u);
  x ^= x >> 16; x *= 0x7FEB352Du;
  x ^= x >> 15; x *= 0x846CA68Bu;
  x ^= x >> 16;
  return x;
}

// policy 0: highest score first (Section 4.2); 1: lowest score first and 2: random order (the
// selection ablations of Section 5.3).  Ties always go to the lower token index.
//
// Every candidate gets a 43-bit composite (32-bit order key, then 2047 - index); composites are distinct, a larger one
// ranks earlier.  Each pass deals those in the current range over 512 bins by their next nine bits and keeps the bin in
// which the k-th largest lies; it is over when that bin is wanted whole or holds one value.
constexpr int kIdxBits = 11, kBinBits = 9, kBins = 1 << kBinBits, kMaxPasses = (32 + kIdxBits + kBinBits - 1) / kBinBits;
constexpr int kPerThread = 2048 / kTopkThreads, kTopkWarps = kTopkThreads / 32;

// MANY: more samples than run at once, where what a sample costs counts beside its latency: a crowded bin is looked at (64
// samples of 1088 tokens 5.4 us without that, 5.6 with it).  48 registers, five CTAs per SM: left alone the compiler takes 64
// and four, 16 384 samples of 320 tokens 158 -> 169 us.
template <bool MANY>
__global__ void __launch_bounds__(kTopkThreads, MANY ? 5 : 0)
topk_kernel(const float* __restrict__ partial, int H, float* __restrict__ scores, const int32_t* __restrict__ new_idx,
            int n_new, const int32_t* __restrict__ excl_idx, int n_excl, int S, int k, int policy, uint32_t seed,
            int32_t* __restrict__ refresh_idx) {
  __shared__ uint4 hist[kMaxPasses][kBins / 4];          // one histogram per pass: none has to be cleared again
  __shared__ uint32_t taken[2048 / 4];                   // a byte per token: generating or excluded
  __shared__ uint32_t warp_min[kTopkWarps], warp_max[kTopkWarps];
  __shared__ int warp_tot[kTopkWarps];
  __shared__ uint32_t least[kMaxPasses];                 // key of the crossing bin after a pass, where it is crowded
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < kMaxPasses * kBins / 4; i += kTopkThreads) (&hist[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int i = tid; i < 2048 / 4; i += kTopkThreads) taken[i] = 0u;
  if (MANY && tid < kMaxPasses) least[tid] = 0xffffffffu;
  __syncthreads();
  pdl_sync();

  uint8_t* mark = reinterpret_cast<uint8_t*>(taken);
  if (k > 0) {
    for (int i = tid; i < n_new; i += kTopkThreads) mark[new_idx[(long)b * n_new + i]] = 1;
    for (int i = tid; i < n_excl; i += kTopkThreads) mark[excl_idx[(long)b * n_excl + i]] = 1;
  }
  // a thread owns consecutive tokens, so that the selected ones come out in ascending order
  const int per = (S + kTopkThreads - 1) / kTopkThreads, t0 = tid * per;
  uint32_t key[kPerThread];
#pragma unroll
  for (int i = 0; i < kPerThread; ++i) {
    const int t = t0 + i;
    key[i] = 0u;
    if (i < per && t < S) {
      float s;
      if (partial) {
        s = 0.f;
        for (int h = 0; h < H; ++h) s += partial[((long)b * H + h) * S + t];
        scores[(long)b * S + t] = s;
      } else {
        s = scores[(long)b * S + t];
      }
      key[i] = policy == 0 ? score_key(s) : (policy == 1 ? ~score_key(s) : ~mix32(seed, (uint32_t)b, (uint32_t)t));
    }
  }
  if (k <= 0) return;
  __syncthreads();                                       // the marks
  unsigned cand = 0;                                     // bit i: token t0 + i is a candidate
  uint32_t lo32 = 0xffffffffu, hi32 = 0u;
#pragma unroll
  for (int i = 0; i < kPerThread; ++i)
    if (i < per && t0 + i < S && !mark[t0 + i]) {
      cand |= 1u << i;
      lo32 = min(lo32, key[i]);
      hi32 = max(hi32, key[i]);
    }
  lo32 = __reduce_min_sync(0xffffffffu, lo32);
  hi32 = __reduce_max_sync(0xffffffffu, hi32);
  if (lane == 0) { warp_min[warp] = lo32; warp_max[warp] = hi32; }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kTopkWarps; ++w) { lo32 = min(lo32, warp_min[w]); hi32 = max(hi32, warp_max[w]); }

  // ---- radix select of the k-th largest composite; with fewer than k candidates all of them stay
  auto composite = [&](int i) { return ((unsigned long long)key[i] << kIdxBits) | (unsigned)((1 << kIdxBits) - 1 - (t0 + i)); };
  unsigned long long lo = (unsigned long long)lo32 << kIdxBits;
  unsigned long long range = hi32 >= lo32 ? (((unsigned long long)(hi32 - lo32) << kIdxBits) | ((1 << kIdxBits) - 1)) : 0ull;
  unsigned int remaining = (unsigned)k;
  unsigned in_range = cand;
#pragma unroll 1
  for (int pass = 0; pass < kMaxPasses; ++pass) {
    const int bits = 64 - __clzll((long long)range), shift = bits > kBinBits ? bits - kBinBits : 0;
    unsigned int* h = reinterpret_cast<unsigned int*>(hist[pass]);
#pragma unroll
    for (int i = 0; i < kPerThread; ++i)
      if (in_range & (1u << i)) atomicAdd(&h[(unsigned)((composite(i) - lo) >> shift)], 1u);
    __syncthreads();
    unsigned int c[kBins / 32], mine = 0u;               // a lane's consecutive bins
#pragma unroll
    for (int j = 0; j < kBins / 128; ++j) {
      const uint4 v = hist[pass][lane * (kBins / 128) + j];
      c[4 * j] = v.x; c[4 * j + 1] = v.y; c[4 * j + 2] = v.z; c[4 * j + 3] = v.w;
      mine += (v.x + v.y) + (v.z + v.w);
    }
    unsigned int above = mine;                           // suffix sums from the top bin downwards
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int v = __shfl_down_sync(0xffffffffu, above, o);
      if (lane + o < 32) above += v;
    }
    const bool here = above >= remaining && above - mine < remaining;
    const unsigned who = __ballot_sync(0xffffffffu, here);
    if (who == 0u) break;                                // fewer candidates than remaining
    above -= mine;
    int digit = 0;
    unsigned int before = 0u, held = 0u;
#pragma unroll
    for (int j = kBins / 32 - 1; j >= 0; --j) {
      if (above < remaining && above + c[j] >= remaining) { digit = lane * (kBins / 32) + j; before = above; held = c[j]; }
      above += c[j];
    }
    const int src = __ffs((int)who) - 1;
    digit = __shfl_sync(0xffffffffu, digit, src);
    before = __shfl_sync(0xffffffffu, before, src);
    held = __shfl_sync(0xffffffffu, held, src);
    lo += (unsigned long long)digit << shift;
    range = (1ull << shift) - 1ull;
    remaining -= before;
    if (held == remaining || shift == 0) break;
#pragma unroll
    for (int i = 0; i < kPerThread; ++i)
      if ((in_range & (1u << i)) && (composite(i) < lo || composite(i) - lo > range)) in_range &= ~(1u << i);
    if (MANY && held > 32u) {
      // A crowded bin, most likely one score: then only the indices are left to compare, where up to three passes over bits in
      // common would follow.  Scores of three values, 16 384 samples of 320 tokens: 324 -> 206 us.
#pragma unroll
      for (int i = 0; i < kPerThread; ++i)
        if (in_range & (1u << i)) atomicMin(&least[pass], key[i]);
      __syncthreads();
      bool differ = false;
#pragma unroll
      for (int i = 0; i < kPerThread; ++i) differ |= (in_range & (1u << i)) && key[i] != least[pass];
      if (!__syncthreads_or(differ)) {
        lo = (unsigned long long)least[pass] << kIdxBits;
        range = (1ull << kIdxBits) - 1ull;
      }
    }
  }

  // ---- every candidate at or above the bound, in ascending order of index
  unsigned sel = 0;
#pragma unroll
  for (int i = 0; i < kPerThread; ++i)
    if ((cand & (1u << i)) && composite(i) >= lo) sel |= 1u << i;
  const int cnt = __popc(sel);
  int inc = cnt;                                         // inclusive scan over the block
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  int pos = inc - cnt;
  for (int w = 0; w < warp; ++w) pos += warp_tot[w];
#pragma unroll
  for (int i = 0; i < kPerThread; ++i)
    if (sel & (1u << i)) refresh_idx[(long)b * k + pos++] = t0 + i;
}

cudaError_t launch_topk(const float* partial, int H, float* scores, const int32_t* new_idx, int n_new,
                        const int32_t* excl_idx, int n_excl, int B, int S, int k, int32_t* refresh_idx, cudaStream_t st,
                        int policy, uint32_t seed) {
  if (S > 2048) return cudaErrorInvalidValue;
  static bool carved[2][kMaxDevices] = {};
  const bool many = B > 512 && B > 5 * device_sm_count();   // (the first test saves the usual call the query of its device)
  auto* kernel = many ? topk_kernel<true> : topk_kernel<false>;
  const cudaError_t e = prefer_shared_memory(kernel, carved[many]);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3(B), dim3(kTopkThreads), 0, st, partial, H, scores, new_idx, n_new, excl_idx, n_excl, S,
                    k, policy, seed, refresh_idx);
}

}  // namespace marche

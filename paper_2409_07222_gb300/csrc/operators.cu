// operators.cu -- labs_sequence_operators: the end-element operators that move candidates to the
// neighbouring lengths (Section 3: appending or removing an element at either end gives sequences of
// length L+1 and L-1 with comparable merit factor, which re-enter step 2; the loop of Fig. 4).
//
// Lane w owns 32-bit word w of the sequence: an append sets bit L, a prepend shifts every word up by one bit, a
// removal clears the last bit or shifts down by one.  The energy is that of labs_energy_batch (energy_words.cuh).
// A warp takes one of an input's six results, so that even one input fills six warps (step 2's best sequence is what
// a search hands over), or all six where there are inputs enough: the sequence is then read and the loop's index
// divided once, which for short sequences is most of the work.  Measured, 65,536 inputs: L = 64: 72.6 us with a warp a
// result, 22.5 us with a warp an input; L = 451: 254 and 231 us.
#include <algorithm>

#include "energy_words.cuh"
#include "labs_internal.h"

namespace labsg {
namespace {

constexpr int kOpWarps = 8;

// Writes the variant in vbits (length Lv) as packed 64-bit words.
__device__ __forceinline__ void store_words(const uint32_t* vbits, int Lv, uint64_t* dst) {
  const int lane = lane_id();
  const int W = (Lv + 63) >> 6;
  if (lane < W) dst[lane] = (uint64_t)vbits[2 * lane] | ((uint64_t)vbits[2 * lane + 1] << 32);
}

// Result v of an input: 0, 1 append +1 / -1, 2, 3 prepend +1 / -1, 4 without the last element, 5 without the
// first.  NG, NS: 32-bit words of L + 1 and of L - 1 positions.  ALL: a warp takes all six results of an input, else
// one of them.
template <int NG, int NS, bool ALL>
__global__ void __launch_bounds__(32 * kOpWarps) operators_kernel(const uint64_t* __restrict__ seqs, int L, int64_t n,
                                                                  uint64_t* __restrict__ grow, int32_t* __restrict__ E_grow,
                                                                  uint64_t* __restrict__ shrink,
                                                                  int32_t* __restrict__ E_shrink) {
  __shared__ __align__(16) uint32_t vb[kOpWarps][kBitWords];
  uint32_t* v = vb[threadIdx.x >> 5];
  const int lane = lane_id();
  const int W = (L + 63) >> 6, Wg = (L + 64) >> 6, Ws = (L + 62) >> 6;
  const int W32 = (L + 31) >> 5;
  const int64_t warps_total = (int64_t)gridDim.x * kOpWarps, items = ALL ? n : 6 * n;
  for (int64_t it = (int64_t)blockIdx.x * kOpWarps + (threadIdx.x >> 5); it < items; it += warps_total) {
    const int64_t q = ALL ? it : it / 6;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(seqs + q * W);
    uint32_t x = 0;
    if (lane < W32) {
      x = src[lane];
      const int rem = L - 32 * lane;
      if (rem < 32) x &= (1u << rem) - 1u;
    }
    const uint32_t below = __shfl_up_sync(kFull, x, 1), above = __shfl_down_sync(kFull, x, 1);
    auto result = [&](int var) {
      const uint32_t bit = (var & 1) ? 0u : 1u;  // value of a new element (1 = +1)
      uint32_t w;
      if (var < 2)
        w = lane == (L >> 5) ? x | bit << (L & 31) : x;
      else if (var < 4)
        w = (x << 1) | (lane ? below >> 31 : bit);
      else if (var == 4)
        w = lane == ((L - 1) >> 5) ? x & ~(1u << ((L - 1) & 31)) : x;
      else
        w = (x >> 1) | (above << 31);
      __syncwarp();  // the previous result's readers of v are done
      if (lane < kBitWords) v[lane] = w;
      __syncwarp();
      const int Lv = var < 4 ? L + 1 : L - 1;
      const int E = var < 4 ? energy_words<NG>(v, Lv) : energy_words<NS>(v, Lv);
      if (var < 4) {
        if (grow) store_words(v, Lv, grow + (q * 4 + var) * Wg);
        if (E_grow && lane == 0) E_grow[q * 4 + var] = E;
      } else {
        if (shrink) store_words(v, Lv, shrink + (q * 2 + var - 4) * Ws);
        if (E_shrink && lane == 0) E_shrink[q * 2 + var - 4] = E;
      }
    };
    if constexpr (!ALL) {
      result((int)(it - 6 * q));
    } else if constexpr (NG <= 4) {
#pragma unroll
      for (int var = 0; var < 6; var++) result(var);
    } else {
#pragma unroll 1
      for (int var = 0; var < 6; var++) result(var);
    }
  }
}

}  // namespace

int launch_sequence_operators(labs_ctx* ctx, const uint64_t* seqs, int L, int64_t n, uint64_t* grow, int32_t* E_grow,
                              uint64_t* shrink, int32_t* E_shrink, cudaStream_t st) {
  if (n == 0) return LABS_OK;
  // All six results a warp once the warps that the chip holds have an input each (64 an SM); from 16 an SM where a
  // result is short work.  A warp a result against a warp an input, in us: 3,000 inputs of L = 200: 8.0 and 7.5, of
  // L = 451: 14.5 and 16.1; 10,000 of L = 451: 41.5 and 41.0.
  const bool all = n >= (int64_t)ctx->num_sms * (L + 1 <= 320 ? 16 : 64);
  const int64_t items = all ? n : 6 * n;
  const unsigned nb = (unsigned)std::min<int64_t>((items + kOpWarps - 1) / kOpWarps, (int64_t)ctx->num_sms * 16);
  return by_words((L + 32) >> 5, [&](auto nw) {
    constexpr int NG = decltype(nw)::value, NL = NG > 1 ? NG - 1 : 1;
    auto run = [&](auto* kernel) {
      kernel<<<nb, 32 * kOpWarps, 0, st>>>(seqs, L, n, grow, E_grow, shrink, E_shrink);
      return cuda_status(cudaGetLastError());
    };
    if ((L + 30) >> 5 == NG) return run(all ? operators_kernel<NG, NG, true> : operators_kernel<NG, NG, false>);
    // L - 1 positions end one word earlier
    return run(all ? operators_kernel<NG, NL, true> : operators_kernel<NG, NL, false>);
  });
}

}  // namespace labsg

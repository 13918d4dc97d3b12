// operators.cu -- labs_sequence_operators: the end-element operators that move candidates to the
// neighbouring lengths (Section 3: appending or removing an element at either end gives sequences of
// length L+1 and L-1 with comparable merit factor, which re-enter step 2; the loop of Fig. 4).
//
// One warp per result.  Lane w owns 32-bit word w of the sequence: an append sets bit L, a prepend shifts
// every word up by one bit, a removal clears the last bit or shifts down by one.  The energy is that of
// labs_energy_batch (energy_words.cuh).  Six results per input, so that even one input fills six warps (step
// 2's best sequence is what a search hands over).
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
// first.  NG, NS: 32-bit words of L + 1 and of L - 1 positions.
template <int NG, int NS>
__global__ void __launch_bounds__(32 * kOpWarps) operators_kernel(const uint64_t* __restrict__ seqs, int L, int64_t n,
                                                                  uint64_t* __restrict__ grow, int32_t* __restrict__ E_grow,
                                                                  uint64_t* __restrict__ shrink,
                                                                  int32_t* __restrict__ E_shrink) {
  __shared__ __align__(16) uint32_t vb[kOpWarps][kBitWords];
  uint32_t* v = vb[threadIdx.x >> 5];
  const int lane = lane_id();
  const int W = (L + 63) >> 6, Wg = (L + 64) >> 6, Ws = (L + 62) >> 6;
  const int W32 = (L + 31) >> 5;
  const int64_t warps_total = (int64_t)gridDim.x * kOpWarps;
  for (int64_t r = (int64_t)blockIdx.x * kOpWarps + (threadIdx.x >> 5); r < 6 * n; r += warps_total) {
    const int64_t q = r / 6;
    const int var = (int)(r - 6 * q);
    const uint32_t* src = reinterpret_cast<const uint32_t*>(seqs + q * W);
    uint32_t x = 0;
    if (lane < W32) {
      x = src[lane];
      const int rem = L - 32 * lane;
      if (rem < 32) x &= (1u << rem) - 1u;
    }
    const uint32_t below = __shfl_up_sync(kFull, x, 1), above = __shfl_down_sync(kFull, x, 1);
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
  }
}

}  // namespace

int launch_sequence_operators(labs_ctx* ctx, const uint64_t* seqs, int L, int64_t n, uint64_t* grow, int32_t* E_grow,
                              uint64_t* shrink, int32_t* E_shrink, cudaStream_t st) {
  if (n == 0) return LABS_OK;
  const unsigned nb = (unsigned)std::min<int64_t>((6 * n + kOpWarps - 1) / kOpWarps, (int64_t)ctx->num_sms * 16);
  return by_words((L + 32) >> 5, [&](auto nw) {
    constexpr int NG = decltype(nw)::value, NL = NG > 1 ? NG - 1 : 1;
    if ((L + 30) >> 5 == NG)
      operators_kernel<NG, NG><<<nb, 32 * kOpWarps, 0, st>>>(seqs, L, n, grow, E_grow, shrink, E_shrink);
    else  // L - 1 positions end one word earlier
      operators_kernel<NG, NL><<<nb, 32 * kOpWarps, 0, st>>>(seqs, L, n, grow, E_grow, shrink, E_shrink);
    return cuda_status(cudaGetLastError());
  });
}

}  // namespace labsg

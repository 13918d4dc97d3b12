// energy.cu -- labs_energy_batch: C_k and E = sum C_k^2 for a batch of bit-packed sequences
// (Section 1 definitions; ENERGY in Algorithms 1 and 2).
//
// One warp per sequence, its words in registers (energy_words.cuh).  8 B per word in, 4 B out (plus the C_k
// when asked for); the next sequence's words are loaded while this one is worked on.
#include <algorithm>

#include "energy_words.cuh"
#include "labs_internal.h"

namespace labsg {
namespace {

constexpr int kEnergyWarps = 8;

template <int NW, bool WITH_C>
__global__ void __launch_bounds__(32 * kEnergyWarps) energy_batch_kernel(const uint64_t* __restrict__ seqs, int L,
                                                                          int64_t n, int32_t* __restrict__ E_out,
                                                                          int32_t* __restrict__ C_out) {
  __shared__ __align__(16) uint32_t bits_all[kEnergyWarps][(NW + 3) / 4 * 4];
  uint32_t* sb = bits_all[threadIdx.x >> 5];
  const int lane = lane_id();
  const int W = (L + 63) >> 6;
  const int64_t warps_total = (int64_t)gridDim.x * kEnergyWarps;
  auto fetch = [&](int64_t q) {
    if (lane >= NW || q >= n) return 0u;
    const uint32_t v = reinterpret_cast<const uint32_t*>(seqs + q * W)[lane];
    const int rem = L - 32 * lane;
    return rem < 32 ? v & ((1u << rem) - 1u) : v;
  };
  int64_t q = (int64_t)blockIdx.x * kEnergyWarps + (threadIdx.x >> 5);
  uint32_t own = fetch(q);
  for (; q < n; q += warps_total) {
    __syncwarp();  // the previous sequence's readers of sb are done
    if (lane < NW) sb[lane] = own;
    __syncwarp();
    own = fetch(q + warps_total);
    const int e = energy_words<NW, WITH_C>(sb, L, WITH_C ? C_out + q * (L - 1) : nullptr);
    if (lane == 0) E_out[q] = e;
  }
}

}  // namespace

int launch_energy_batch(labs_ctx* ctx, const uint64_t* seqs, int L, int64_t n, int32_t* E_out, int32_t* C_out,
                        cudaStream_t st) {
  if (n == 0) return LABS_OK;
  const unsigned nb = (unsigned)std::min<int64_t>((n + kEnergyWarps - 1) / kEnergyWarps, (int64_t)ctx->num_sms * 16);
  return by_words((L + 31) >> 5, [&](auto nw) {
    constexpr int NW = decltype(nw)::value;
    if (C_out)
      energy_batch_kernel<NW, true><<<nb, 32 * kEnergyWarps, 0, st>>>(seqs, L, n, E_out, C_out);
    else
      energy_batch_kernel<NW, false><<<nb, 32 * kEnergyWarps, 0, st>>>(seqs, L, n, E_out, nullptr);
    return cuda_status(cudaGetLastError());
  });
}

}  // namespace labsg

// flip_deltas.cu -- labs_flip_deltas: exact Delta E of every single-flip neighbour (BEST_NEIGHBOUR of
// Algorithm 1, the neighbourhood loop of Algorithm 2), stand-alone.
//
// One warp per sequence: its correlations by carry-save counting (energy_words.cuh), the neighbours' sums T by
// a Toeplitz product on the tensor cores (scan_mma.cuh), then the Delta E of walk.cu's incremental
// neighbourhood (same names): of a skew sequence from the class correlations R^e, of an unrestricted one from
// the self-convolution V.
//
// Measured against the dp4a scan of all neighbours x lags (one lane per tile of eight neighbours): 32,768 skew
// sequences of L = 451, p = 24: 217 -> 72 us; 8,192 unrestricted ones of L = 452: 123 -> 38 us, of L = 576: 191
// -> 46 us.  Bound: issue slots (1,646 warp instructions a skew sequence, 67% busy at 20 warps an SM), the
// tensor cores 16% busy.
#include <algorithm>

#include "labs_internal.h"
#include "scan_mma.cuh"

namespace labsg {
namespace {

constexpr int kFdWarps = 4;

// Shared memory of one warp, in 32-bit words from its slab's start.
struct FdPlan {
  ScanMmaPlan mma;
  int q, x, z, words;  // q: two copies; x: class sequences; z: int16 tables; bits, classes in front
};
constexpr int kFdBits = 0, kFdClass = kBitWords, kFdRev = kFdClass + 2 * kClassWords,
              kFdOdd = kFdRev + 2 * kClassWords, kFdTables = kFdOdd + 4;  // kFdOdd: the warp met such a table

// Entries of a table of up to these bits (and a sign) are exact as FP16 operands: a sequence's own are (|C| <= 575).
constexpr int kHalfBits = 11;

// A caller's table is used as it is given (16 bits of every entry).  A warp that met one that the kernels' fast way
// does not serve goes over its sequences once more: Delta E of the neighbours p + 1 .. last by plain loops over the
// lags that are multiples of lam (2: skew pairs; their mirror's product drops out).  No table of a sequence's own
// correlations comes here, so this is small rather than fast, and behind the loop that needs the registers: inside
// it, 8,192 unrestricted sequences of L = 576 took 44.5 us with a table, behind it 42.3 (41.4 without the check).
__device__ __forceinline__ void odd_tables(const uint64_t* seqs, const int32_t* Cin, int L, int64_t n, int lam, int p,
                                           int last, uint32_t* bits, int32_t* dE) {
  const int W = (L + 63) >> 6, lane = lane_id();
  const int64_t warps_total = (int64_t)gridDim.x * kFdWarps;
  auto s_at = [&](int i) { return i < 1 || i > L ? 0 : ((bits[(i - 1) >> 5] >> ((i - 1) & 31)) & 1u) ? 1 : -1; };
  for (int64_t s = (int64_t)blockIdx.x * kFdWarps + (threadIdx.x >> 5); s < n; s += warps_total) {
    const int32_t* C = Cin + s * (L - 1);
    if (lane < (L + 31) >> 5) bits[lane] = reinterpret_cast<const uint32_t*>(seqs + s * W)[lane];
    __syncwarp();
    for (int m = p + 1 + lane; m <= last; m += 32) {
      const int mirror = lam == 2 && 2 * m != L + 1 ? L + 1 - m : 0, alpha = mirror ? 4 : 2;
      const int sm = s_at(m);
      int linear = 0, square = 0;  // C_k changes by - alpha s_m y
      for (int k = lam; k < L; k += lam) {
        const int y = (m + k == mirror ? 0 : s_at(m + k)) + s_at(m - k);
        linear += (int16_t)C[k - 1] * y;
        square += y * y;
      }
      dE[s * L + m - 1] = alpha * (alpha * square - 2 * sm * linear);
    }
    __syncwarp();
  }
}

// NC: 32-bit words of the longer parity class; NT: tiles of 128 neighbours per class; GIVEN: with a caller's table.
template <int NC, int NT, bool GIVEN>
__global__ void __launch_bounds__(32 * kFdWarps, NT == 1 ? 6 : 5) flip_deltas_skew_kernel(const uint64_t* __restrict__ seqs,
                                                                          const int32_t* __restrict__ Cin, int L, int64_t n,
                                                                          int p, FdPlan fp, int32_t* __restrict__ dE) {
  extern __shared__ __align__(16) uint32_t fd_smem[];
  uint32_t* slab = fd_smem + (size_t)(threadIdx.x >> 5) * fp.words;
  uint32_t *bits = slab + kFdBits, *cw = slab + kFdClass, *q = slab + fp.q;
  // Z^e_g = 2 R^e_g + C_{2g} of the two parities e of the distance from the centre
  int16_t* z0 = reinterpret_cast<int16_t*>(slab + fp.z);
  int16_t* z1 = z0 + 32 * NC;
  const int lane = lane_id();
  const int W = (L + 63) >> 6, W32 = (L + 31) >> 5, k = (L - 1) / 2, c = k + 1;
  const int n_odd = (L + 1) / 2, n_even = L / 2;       // positions 1, 3, .. and 2, 4, ..
  const int e_odd = (c - 1) & 1;                       // parity of the distance of the odd positions
  const int nh[2] = {2 * (k >> 1) + 1, 2 * ((k + 1) >> 1)};  // positions at even and odd distance
  for (int i = lane; i < fp.words; i += 32) slab[i] = 0u;
  __syncwarp();
  const uint32_t* const xs[2] = {slab + fp.x, slab + fp.x + fp.mma.x_words};
  const int64_t warps_total = (int64_t)gridDim.x * kFdWarps;
  for (int64_t s = (int64_t)blockIdx.x * kFdWarps + (threadIdx.x >> 5); s < n; s += warps_total) {
    if (lane < W32) {
      const uint32_t v = reinterpret_cast<const uint32_t*>(seqs + s * W)[lane];
      const int rem = L - 32 * lane;
      bits[lane] = rem < 32 ? v & ((1u << rem) - 1u) : v;
    }
    __syncwarp();
    split_classes(bits, cw);
    // class correlations at lag g (twice the class index): positions of one parity are one class of distances
    int16_t* zo = e_odd ? z1 : z0;
    int16_t* ze = e_odd ? z0 : z1;
    int odd = 0;  // whether the given table differs from the sequence's own, which the sums below are formed from
    corr_words<NC>(cw, cw, n_odd, [&](int g, int r) { zo[g] = (int16_t)r; });
    corr_words<NC>(cw + kClassWords, cw + kClassWords, n_even, [&](int g, int r) {
      const int r_odd = zo[g];  // the lane's own
      const int cg = r_odd + r;
      if (GIVEN && g >= 1 && g <= k) odd |= Cin[s * (L - 1) + 2 * g - 1] ^ cg;
      zo[g] = (int16_t)(2 * r_odd + cg);
      ze[g] = (int16_t)(2 * r + cg);
      if (g >= 1 && g <= k) put_q(q, fp.mma, g, cg);
    });
    put_x(slab + fp.x, cw, n_odd);
    put_x(slab + fp.x + fp.mma.x_words, cw + kClassWords, n_even);
    if (GIVEN && odd) slab[kFdOdd] = 1u;
    __syncwarp();
    float acc[2][NT][4];
    scan_mma<2, NT>(q, xs, fp.mma, n_odd, acc);
    int32_t* out = dE + s * L;
    for (int i = lane; i < p; i += 32) out[i] = INT32_MAX;
    for (int i = c + lane; i < L; i += 32) out[i] = INT32_MAX;
#pragma unroll
    for (int x = 0; x < 2; x++) {
      // positions m = 2 j + 1 + x: distances h = c - m of one parity e
      const int h0 = c - 1 - x, e = h0 & 1, eta = e ? -1 : 1;
      const int16_t* zt = e ? z1 : z0;
      const uint32_t* xw = cw + x * kClassWords;
      const int base = 16 * (nh[e] - 3);
#pragma unroll
      for (int T = 0; T < NT; T++) {
        // the tile's four outputs of the lane lie in one word of the class: bits 0, 16, 8, 24 above g
        const int jl = fp.mma.j0 + 128 * T + 32 * (lane & 3);
        const uint32_t own = xw[jl >> 5] >> (lane >> 2);
#pragma unroll
        for (int r = 0; r < 4; r++) {
          const int o = 16 * (r & 1) + 8 * (r >> 1), j = jl + (lane >> 2) + o, m = 2 * j + 1 + x, h = h0 - 2 * j;
          if (m > p && h >= 0) {
            const int sm = (own >> o & 1u) ? 1 : -1, st = sm * (int)acc[x][T][r];
            int d = 8 * (eta * zt[h] - st) + base;
            const int j3 = j - h;  // - 32 (-1)^h S[h] S[3h]: position c - 3h is class index j - h
            if (j3 >= 0) d += ((xw[j3 >> 5] >> (j3 & 31)) & 1u) ? -32 * eta * sm : 32 * eta * sm;
            out[m - 1] = h == 0 ? 8 * nh[0] - 8 - 4 * st : d;
          }
        }
      }
    }
    __syncwarp();
  }
  if (GIVEN && slab[kFdOdd]) odd_tables(seqs, Cin, L, n, 2, p, c, bits, dE);
}

// NW: 32-bit words of the sequence; NT: tiles of 128 neighbours; GIVEN: with a caller's table.
template <int NW, int NT, bool GIVEN>
__global__ void __launch_bounds__(32 * kFdWarps, NT <= 2 ? 6 : 4) flip_deltas_kernel(const uint64_t* __restrict__ seqs,
                                                                     const int32_t* __restrict__ Cin, int L, int64_t n,
                                                                     int p, FdPlan fp, int32_t* __restrict__ dE) {
  extern __shared__ __align__(16) uint32_t fd_smem[];
  uint32_t* slab = fd_smem + (size_t)(threadIdx.x >> 5) * fp.words;
  uint32_t *bits = slab + kFdBits, *cw = slab + kFdClass, *q = slab + fp.q;
  int16_t* v = reinterpret_cast<int16_t*>(slab + fp.z);
  const int lane = lane_id();
  const int W = (L + 63) >> 6, W32 = (L + 31) >> 5;
  for (int i = lane; i < fp.words; i += 32) slab[i] = 0u;
  __syncwarp();
  const uint32_t* const xs[1] = {slab + fp.x};
  const int64_t warps_total = (int64_t)gridDim.x * kFdWarps;
  for (int64_t s = (int64_t)blockIdx.x * kFdWarps + (threadIdx.x >> 5); s < n; s += warps_total) {
    if (lane < W32) {
      const uint32_t w = reinterpret_cast<const uint32_t*>(seqs + s * W)[lane];
      const int rem = L - 32 * lane;
      bits[lane] = rem < 32 ? w & ((1u << rem) - 1u) : w;
    }
    __syncwarp();
    if constexpr (GIVEN) {
      int odd = 0;  // ones above kHalfBits where an entry has more bits
      for (int d = lane + 1; d < L; d += 32) {
        const int cd = Cin[s * (L - 1) + d - 1];
        odd |= cd ^ (cd >> 31);
        put_q(q, fp.mma, d, cd);
      }
      if (odd >> kHalfBits) slab[kFdOdd] = 1u;
    } else {
      corr_words<NW>(bits, bits, L, [&](int d, int cd) {
        if (d >= 1 && d < L) put_q(q, fp.mma, d, cd);
      });
    }
    put_x(slab + fp.x, bits, L);
    split_classes(bits, cw);
    self_convolution<(NW + 1) / 2>(cw, slab + kFdRev, L, v);
    __syncwarp();
    float acc[1][NT][4];
    scan_mma<1, NT>(q, xs, fp.mma, L, acc);
    int32_t* out = dE + s * L;
    for (int i = lane; i < p; i += 32) out[i] = INT32_MAX;
#pragma unroll
    for (int T = 0; T < NT; T++) {
      const int jl = fp.mma.j0 + 128 * T + 32 * (lane & 3);
      const uint32_t own = jl < L ? bits[jl >> 5] >> (lane >> 2) : 0u;
#pragma unroll
      for (int r = 0; r < 4; r++) {
        const int o = 16 * (r & 1) + 8 * (r >> 1), m = jl + (lane >> 2) + o + 1;
        if (m > p && m <= L) {
          const int t = (int)acc[0][T][r];
          out[m - 1] = 4 * ((int)v[m] + L - 2 - ((own >> o & 1u) ? t : -t));
        }
      }
    }
    __syncwarp();
  }
  if (GIVEN && slab[kFdOdd]) odd_tables(seqs, Cin, L, n, 1, p, L, bits, dE);
}

template <class Kernel>
int launch_fd(labs_ctx* ctx, Kernel* kern, const uint64_t* seqs, const int32_t* C, int L, int64_t n, int p, const FdPlan& fp,
              int32_t* dE, cudaStream_t st) {
  const size_t smem = sizeof(uint32_t) * (size_t)fp.words * kFdWarps;
  if (allow_smem(ctx, kern) != cudaSuccess) return LABS_ERR_CUDA;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kFdWarps, smem) != cudaSuccess || per_sm < 1)
    return LABS_ERR_CUDA;
  const unsigned blocks = (unsigned)std::min<int64_t>((n + kFdWarps - 1) / kFdWarps, (int64_t)ctx->num_sms * per_sm);
  kern<<<blocks, 32 * kFdWarps, smem, st>>>(seqs, C, L, n, p, fp, dE);
  return cuda_status(cudaGetLastError());
}

}  // namespace

int launch_flip_deltas(labs_ctx* ctx, const uint64_t* seqs, const int32_t* C, int L, int64_t n, int skew, int p,
                       int32_t* dE_out, cudaStream_t st) {
  if (n == 0) return LABS_OK;
  FdPlan fp;
  if (skew) {
    const int c = (L + 1) / 2;
    // class indices of the neighbours p + 1 .. c in either class
    fp.mma = scan_mma_plan((L + 1) / 2, p / 2, (c - 1) / 2);
    fp.q = kFdTables;
    fp.x = fp.q + 2 * fp.mma.q_words;
    fp.z = fp.x + 2 * fp.mma.x_words;
  } else {
    fp.mma = scan_mma_plan(L, p, L - 1);
    fp.q = kFdTables;
    fp.x = fp.q + 2 * fp.mma.q_words;
    fp.z = fp.x + fp.mma.x_words;
  }
  return by_words((L + 31) >> 5, [&](auto nw) {
    constexpr int NW = decltype(nw)::value, NC = (NW + 1) / 2;
    if (skew) {
      fp.words = fp.z + 32 * NC;  // two tables of 32 NC halves
      constexpr int kMost = (16 * NW / 2 + 63 + 128) / 128;  // tiles when nothing is fixed, j0 rounded down
      if constexpr (kMost >= 2)
        if (fp.mma.nt == 2)
          return launch_fd(ctx, C ? flip_deltas_skew_kernel<NC, 2, true> : flip_deltas_skew_kernel<NC, 2, false>, seqs, C, L,
                           n, p, fp, dE_out, st);
      return launch_fd(ctx, C ? flip_deltas_skew_kernel<NC, 1, true> : flip_deltas_skew_kernel<NC, 1, false>, seqs, C, L, n,
                       p, fp, dE_out, st);
    }
    fp.words = (fp.z + L / 2 + 1 + 3) / 4 * 4;  // v[1 .. L]
    constexpr int kMost = NW / 4 + 1;  // tiles when nothing is fixed
    auto run = [&](auto nt) {
      constexpr int NT = decltype(nt)::value;
      if constexpr (NT <= kMost)
        return launch_fd(ctx, C ? flip_deltas_kernel<NW, NT, true> : flip_deltas_kernel<NW, NT, false>, seqs, C, L, n, p, fp,
                         dE_out, st);
      return (int)LABS_ERR_INVALID_ARG;
    };
    switch (fp.mma.nt) {
      case 1: return run(std::integral_constant<int, 1>{});
      case 2: return run(std::integral_constant<int, 2>{});
      case 3: return run(std::integral_constant<int, 3>{});
      case 4: return run(std::integral_constant<int, 4>{});
      default: return run(std::integral_constant<int, 5>{});
    }
  });
}

}  // namespace labsg

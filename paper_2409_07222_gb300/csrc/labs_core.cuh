// labs_core.cuh -- device building blocks shared by the LABS kernels (sm_103a): random streams, warp reductions,
// walk starts, fingerprints, one correlation by popcounts, and the tile plan by which the walk entry points accept
// or refuse their sizes.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "labs.h"

namespace labsg {

constexpr int kMaxL = LABS_MAX_L;
constexpr int kQOff = 3;             // class index of the first position of a class
constexpr int kDirBytes = 1216;      // tile plan: byte-window array per direction (two 608-byte classes when skew)
constexpr int kClassBytes = 608;
constexpr int kCLen = 608;           // tile plan: correlation table slots (>= 4 * padded group count, L <= 576)
constexpr int kBitWords = 20;        // 18 words for 576 bits + 2 zero words for funnel shifts
constexpr int kMaxR = 32;

// ------------------------------------------------------------------------------------------------
// SplitMix64 (Steele, Lea & Flood, OOPSLA 2014), counter form: output i of the generator whose state
// starts at `key`.  Streams are keyed by chaining at(at(at(seed, purpose), a), b).
// ------------------------------------------------------------------------------------------------
constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;
enum : uint64_t { kPurposeWalk = 1, kPurposeThresh = 2, kPurposeZobrist = 0x5A0B };

__host__ __device__ __forceinline__ uint64_t sm64_at(uint64_t key, uint64_t i) {
  uint64_t z = key + (i + 1) * kGamma;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__host__ __device__ __forceinline__ uint64_t stream_key(uint64_t seed, uint64_t purpose, uint64_t a, uint64_t b) {
  return sm64_at(sm64_at(sm64_at(seed, purpose), a), b);
}

// Zobrist key of position i (1-based) for length L, given zkey = stream_key(0, Zobrist, L, 0).
__device__ __forceinline__ uint64_t zobrist(uint64_t zkey, int i) { return sm64_at(zkey, (uint64_t)(i - 1)); }

// ------------------------------------------------------------------------------------------------
// Warp helpers
// ------------------------------------------------------------------------------------------------
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

__device__ __forceinline__ int warp_sum_i32(int v) { return __reduce_add_sync(kFull, v); }
__device__ __forceinline__ int warp_min_i32(int v) { return __reduce_min_sync(kFull, v); }
__device__ __forceinline__ int warp_max_i32(int v) { return __reduce_max_sync(kFull, v); }
__device__ __forceinline__ unsigned warp_min_u32(unsigned v) { return __reduce_min_sync(kFull, v); }

__device__ __forceinline__ uint64_t warp_xor_u64(uint64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v ^= __shfl_xor_sync(kFull, v, o);
  return v;
}

// ------------------------------------------------------------------------------------------------
// Tile plan of (L, skew, p, M, H): a pure function of its inputs.
// ------------------------------------------------------------------------------------------------
struct Layout {
  int n_tasks;  // tiles x lag ranges
};

// Tiles of M neighbours per position class (class indices start at 3 mod 4), H lag ranges per tile, groups of four
// lags in turns of M/4 + 1: false where the byte windows of the tiled scan would not hold the length.
__host__ __device__ inline bool make_layout(Layout& ly, int L, int skew, int p, int M, int H = 1) {
  const int R = M / 4 + 1;
  const int G = skew ? (L - 1) >> 1 : L - 1, NG = (G + 3) / 4;
  const int mlast = skew ? (L + 1) / 2 : L;
  auto pos_q = [&](int i) { return (skew ? (i - ((i & 1) ? 1 : 2)) >> 1 : i - 1) + kQOff; };
  int n_tiles = 0, qmax_end = 0;
  for (int cls = 0; cls < (skew ? 2 : 1); cls++) {
    int i_lo = p + 1, i_hi = mlast;
    if (skew) {
      if ((i_lo & 1) != cls) i_lo++;
      if ((i_hi & 1) != cls) i_hi--;
    }
    if (i_lo > i_hi) continue;
    const int first = ((pos_q(i_lo) - 3) / 4) * 4 + 3;
    const int nt = (pos_q(i_hi) - first + 1 + M - 1) / M;
    n_tiles += nt;
    const int end = first + nt * M - 1;
    if (end > qmax_end) qmax_end = end;
  }
  const int Qr = qmax_end + ((2 - (qmax_end & 3)) & 3);
  ly.n_tasks = n_tiles * H;
  int NGend;  // padded end of the groups
  if (H == 1) {
    NGend = ((NG + R - 1) / R) * R;
  } else {
    const int half = (NG + 1) / 2, NGh = ((half + R - 1) / R) * R, rest = NG - NGh;
    NGend = NGh + (rest > 0 ? ((rest + R - 1) / R) * R : 0);
  }
  const int cap = skew ? kClassBytes : kDirBytes;
  return (H == 1 || H == 2) && M % 4 == 0 && qmax_end + 4 * NGend + 8 < cap && Qr + 4 * NGend + 8 < cap &&
         2 * qmax_end < cap && 4 * NGend <= kCLen && L >= 2 && L <= kMaxL;
}

// ------------------------------------------------------------------------------------------------
// Correlations, starts, fingerprints
// ------------------------------------------------------------------------------------------------
// C_k = (L-k) - 2 popc((x XOR (x >> k)) restricted to the low L-k bits) from the packed bits.
__device__ __forceinline__ int corr_lag(const uint32_t* bits, int L, int k) {
  const int n = L - k;  // number of products s_i s_{i+k}
  const int ws = k >> 5, sh = k & 31;
  const int nw = (n + 31) >> 5;
  int dis = 0;
  for (int w = 0; w < nw; w++) {
    uint32_t x = bits[w] ^ __funnelshift_r(bits[w + ws], bits[w + ws + 1], sh);
    int rem = n - 32 * w;
    if (rem < 32) x &= (1u << rem) - 1u;
    dis += __popc(x);
  }
  return n - 2 * dis;
}

// Builds a walk start into the bits (kBitWords words): s_1..s_p from the prefix, free element j (position
// p+1+j) is +1 iff bit j%64 of output j/64 of stream `key`; skew walks fill the last k by Eq. (2) around the
// centre c.  Lane w forms word w: the outputs' words shifted by p, then for skew sequences the mirrored half,
// its bits reversed and every other one negated.  scr: kBitWords + 2 words of scratch.
__device__ inline void build_start(uint32_t* bits, uint32_t* scr, int L, bool skew, int c, int p, const uint64_t* prefix,
                                   uint64_t key) {
  const int lane = lane_id();
  __syncwarp();
  if (lane < 11) {
    const uint64_t o = lane < LABS_MAX_W ? sm64_at(key, (uint64_t)lane) : 0ull;
    scr[2 * lane] = (uint32_t)o;
    scr[2 * lane + 1] = (uint32_t)(o >> 32);
  }
  __syncwarp();
  const int i0 = 32 * lane;  // 0-based position of the word's first bit
  // the low n bits, n of any sign
  auto low = [](int n) { return n >= 32 ? 0xffffffffu : (n <= 0 ? 0u : (1u << n) - 1u); };
  // 32 bits of `w` from bit o on; bits in front of w are zero
  auto window = [](const uint32_t* w, int o) {
    if (o < 0) return o > -32 ? w[0] << -o : 0u;
    return __funnelshift_r(w[o >> 5], w[(o >> 5) + 1], o & 31);
  };
  uint32_t x = 0;
  const int n = skew ? c : L;  // positions drawn
  if (i0 < n) {
    x = window(scr, i0 - p);
    if (i0 < p) x = (x & ~low(p - i0)) | ((uint32_t)(prefix[lane >> 1] >> (32 * (lane & 1))) & low(p - i0));
    x &= low(n - i0);
  }
  if (lane < kBitWords) bits[lane] = x;
  __syncwarp();
  if (skew) {
    const int k = c - 1;
    uint32_t y = 0;
    if (i0 < L && i0 + 31 > k)  // position k + j mirrors k - j, negated for odd j
      y = (__brev(window(bits, 2 * k - i0 - 31)) ^ (k & 1 ? 0x55555555u : 0xAAAAAAAAu)) & low(L - i0) & ~low(c - i0);
    __syncwarp();
    if (lane < kBitWords) bits[lane] = x | y;
    __syncwarp();
  }
}

// Zobrist fingerprint of the sequence in the bits.
__device__ inline uint64_t fingerprint(const uint32_t* bits, int L, uint64_t zkey) {
  uint64_t h = 0;
  for (int i = lane_id() + 1; i <= L; i += 32)
    if (!((bits[(i - 1) >> 5] >> ((i - 1) & 31)) & 1u)) h ^= zobrist(zkey, i);
  return warp_xor_u64(h);
}

}  // namespace labsg

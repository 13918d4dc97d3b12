// scan_mma.cuh -- the neighbour scan of one sequence from scratch on the tensor cores: T_m = sum_{i != m}
// c_{|m-i|} x_i for a class sequence x (every position, or the positions of one parity) and its correlation
// table c, the O(L) sum of every neighbour's Delta E.
//
// T is a Toeplitz product.  With m = j0 + 128 T + 16 a + b (tile T, column a < 8, row b < 16),
//     T_m = sum_i q(b - i) x_{j0 + 128 T + 16 a + i},      q(d) = c_{|d|}, q(0) = 0,
// a 16 x K matrix of q that depends on b - i alone times a K x 8 matrix of x (mma.sync m16n8k16, FP16 operands:
// |c| <= 576 and +-1 are exact, the FP32 sums stay below 2^19).  Sequences share neither operand, so there is
// nothing for a 128-row tcgen05 tile to reuse.
//
// Loads: a thread's A words for step i are q at i + 2t - g (+ 8, - 8), the last the previous step's + 8, and
// the fourth equals the first (two words a step; a second copy shifted by one element serves the odd rows).
// Its B words are x at i + 16 g + 2t (+ 8), shared by all tiles of the class; 4 words of padding per 64
// elements keep the eight columns on different banks.
//
// Bound: shared-memory reads (2 + 2 tiles per step, or 4 + 2 for the two classes of a skew sequence) and the
// HMMA rate, 1,012 multiply-adds per clock and SM: L = 451 skew, 23 steps of 2 MMAs; unrestricted, 37 of 4 --
// the dp4a scan issued 8,000 instructions for the latter.
#pragma once

#include <cuda_fp16.h>

#include "energy_words.cuh"

namespace labsg {

constexpr int kXPad = 128;  // zero elements on either side of a class sequence

// Sizes of one warp's operands for class sequences of up to n elements, tiles from j0 on.
struct ScanMmaPlan {
  int j0, nt;       // first output (a multiple of 64), tiles of 128 outputs
  int off;          // element of q(0) in a copy (even)
  int q_words;      // 32-bit words of one copy
  int x_words;      // 32-bit words of one class sequence
};

// Storage word of the element pair (e, e + 1), e even, of a class sequence.
__host__ __device__ __forceinline__ int x_word(int e) { return ((e + kXPad) >> 1) + 4 * ((e + kXPad) >> 6); }

// n: longest class sequence; outputs j_lo .. j_hi.
__host__ inline ScanMmaPlan scan_mma_plan(int n, int j_lo, int j_hi) {
  ScanMmaPlan sp;
  sp.j0 = j_lo / 64 * 64;
  sp.nt = (j_hi - sp.j0) / 128 + 1;
  // i = 64 u + 16 s - j0 - 128 T from -128 - j0 - 128 (nt - 1) up to (n rounded up to 64) - 16 - j0, and i - b + 1
  // .. of the pairs: 24 below and above
  sp.off = sp.j0 + 128 * (sp.nt - 1) + 128 + 24;
  sp.q_words = ((sp.off + (n + 63) / 64 * 64 + 24) / 2 + 31) / 32 * 32 + 16;  // the copies 16 banks apart
  sp.x_words = (x_word((n + 63) / 64 * 64 + kXPad + 16) + 4) / 4 * 4;
  return sp;
}

// Stores q(d) = q(-d) = c (d >= 1).
__device__ __forceinline__ void put_q(uint32_t* q, const ScanMmaPlan& sp, int d, int c) {
  const __half v = __int2half_rn(c);
  __half* c0 = reinterpret_cast<__half*>(q) + sp.off;
  __half* c1 = reinterpret_cast<__half*>(q + sp.q_words) + sp.off + 1;
  c0[d] = v;
  c1[d] = v;
  if (d < sp.off) {  // lower elements are not read
    c0[-d] = v;
    c1[-d] = v;
  }
}

// Stores the +-1 sequence of n elements given by its bits (words readable up to word n / 32).
__device__ __forceinline__ void put_x(uint32_t* x, const uint32_t* bits, int n) {
  for (int w = lane_id(); 2 * w < n; w += 32) {
    const uint32_t b = bits[w >> 4] >> (2 * (w & 15));
    uint32_t v = 0x3C003C00u ^ ((~b & 1u) << 15) ^ ((~b & 2u) << 30);
    if (2 * w + 1 >= n) v &= 0xffffu;
    x[x_word(2 * w)] = v;
  }
}

// acc[x][T][r]: T of class sequence x at output j0 + 128 T + 16 (2 t + (r & 1)) + g + 8 (r >> 1), g = lane / 4,
// t = lane % 4.  q: the two copies; xs[x]: the class sequences, of at most n elements.
template <int NX, int NT>
__device__ __forceinline__ void scan_mma(const uint32_t* q, const uint32_t* const (&xs)[NX], const ScanMmaPlan& sp, int n,
                                         float (&acc)[NX][NT][4]) {
  const int lane = lane_id(), g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int x = 0; x < NX; x++)
#pragma unroll
    for (int T = 0; T < NT; T++)
#pragma unroll
      for (int r = 0; r < 4; r++) acc[x][T][r] = 0.f;
  // word of q at i = -j0 (the copy of odd rows holds element e at e + 1)
  const uint32_t* qa = q + (g & 1) * sp.q_words + ((sp.off + (g & 1) + 2 * t - g - sp.j0) >> 1);
  int xo[4];
#pragma unroll
  for (int s = 0; s < 4; s++) xo[s] = x_word(16 * (g + s) + 2 * t);
  uint32_t below[NT];  // q eight elements below the step's (the last step's upper word)
#pragma unroll
  for (int T = 0; T < NT; T++) below[T] = qa[-64 - 64 * T - 4];
  const int u_end = (n + 63) >> 6;
  for (int u = -2; u < u_end; u++) {
#pragma unroll
    for (int s = 0; s < 4; s++) {
      uint32_t b0[NX], b1[NX];
#pragma unroll
      for (int x = 0; x < NX; x++) {
        b0[x] = xs[x][xo[s] + 36 * u];
        b1[x] = xs[x][xo[s] + 36 * u + 4];
      }
#pragma unroll
      for (int T = 0; T < NT; T++) {
        const uint32_t a0 = qa[32 * u + 8 * s - 64 * T], a2 = qa[32 * u + 8 * s - 64 * T + 4];
#pragma unroll
        for (int x = 0; x < NX; x++)
          asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
              "{%0, %1, %2, %3};"
              : "+f"(acc[x][T][0]), "+f"(acc[x][T][1]), "+f"(acc[x][T][2]), "+f"(acc[x][T][3])
              : "r"(a0), "r"(below[T]), "r"(a2), "r"(a0), "r"(b0[x]), "r"(b1[x]));
        below[T] = a2;
      }
    }
  }
}

// Every other bit of x, from bit 0, in the low half.
__device__ __forceinline__ uint32_t even_bits(uint32_t x) {
  x &= 0x55555555u;
  x = (x | (x >> 1)) & 0x33333333u;
  x = (x | (x >> 2)) & 0x0F0F0F0Fu;
  x = (x | (x >> 4)) & 0x00FF00FFu;
  return (x | (x >> 8)) & 0xFFFFu;
}

constexpr int kClassWords = 12;  // 32-bit words kept per parity class (288 positions and zeros above)

// Parity classes of the sequence in bits (kBitWords words, zero above L): cw[0 ..] the odd positions 1, 3, ..,
// cw[kClassWords ..] the even ones.
__device__ __forceinline__ void split_classes(const uint32_t* bits, uint32_t* cw) {
  const int lane = lane_id();
  if (lane < kClassWords) {
    const uint32_t lo = 2 * lane < kBitWords ? bits[2 * lane] : 0u, hi = 2 * lane + 1 < kBitWords ? bits[2 * lane + 1] : 0u;
    cw[lane] = even_bits(lo) | (even_bits(hi) << 16);
    cw[kClassWords + lane] = even_bits(lo >> 1) | (even_bits(hi >> 1) << 16);
  }
  __syncwarp();
}

// rw: the sequence of n elements in w (kClassWords words) reversed.
__device__ __forceinline__ void reverse_class(const uint32_t* w, uint32_t* rw, int n) {
  const int lane = lane_id();
  if (lane < kClassWords) {
    const int o = n - 32 * lane - 32;  // element n-1-j of bits j = 32 lane ..
    uint32_t y = 0;
    if (o >= 0)
      y = __funnelshift_r(w[o >> 5], (o >> 5) + 1 < kClassWords ? w[(o >> 5) + 1] : 0u, o & 31);
    else if (o > -32)
      y = w[0] << -o;
    rw[lane] = __brev(y);
  }
}

// v[m] = V_{2m} = sum_i s_i s_{2m-i}, m = 1 .. L.  i and 2m - i have one parity, so each parity class contributes
// its own convolution, at index m - 1 (odd positions, m < 2 n) and m - 2 (even ones, 1 < m): the correlation with
// its reversal.  NC: class words; cw as split_classes left it, rw: scratch of the same size.
template <int NC>
__device__ __forceinline__ void self_convolution(const uint32_t* cw, uint32_t* rw, int L, int16_t* v) {
  reverse_class(cw, rw, (L + 1) / 2);
  reverse_class(cw + kClassWords, rw + kClassWords, L / 2);
  if (lane_id() == 0) v[L] = 0;  // even L: the odd positions end at L - 1
  __syncwarp();
#pragma unroll 1
  for (int e = 0; e < 2; e++) {
    const int n = e ? L / 2 : (L + 1) / 2;
    int16_t* out = v + n + e;  // index sum n - 1 -+ d is position n + e -+ d
    const uint32_t *a = cw + e * kClassWords, *b = rw + e * kClassWords;
    corr_words<NC>(a, b, n, [&](int d, int c) {
      if (d < n) out[-d] = (int16_t)(e ? out[-d] + c : c);
    });
    corr_words<NC>(b, a, n, [&](int d, int c) {
      if (d >= 1 && d < n) out[d] = (int16_t)(e ? out[d] + c : c);
    });
    __syncwarp();
  }
}

// Word `lane` of the sequence of L elements (NW words in `bits`, zero above L, readable to word 19) rotated left
// by r, 0 <= r < L: element i is element i + r (mod L).
template <int NW>
__device__ __forceinline__ uint32_t rotated_word(const uint32_t* bits, int L, int r) {
  const int lane = lane_id(), o = 32 * lane + r, ow = o - L;
  if (lane >= NW) return 0u;
  uint32_t y = 0;
  if (o < L) y = __funnelshift_r(bits[o >> 5], bits[(o >> 5) + 1], o & 31);
  if (ow >= 0)  // elements past the end come from the start
    y = __funnelshift_r(bits[ow >> 5], bits[(ow >> 5) + 1], ow & 31);
  else if (ow > -32)
    y |= bits[0] << -ow;
  return lane == NW - 1 ? y & (0xffffffffu >> (32 * NW - L)) : y;
}

}  // namespace labsg

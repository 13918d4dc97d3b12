// energy_words.cuh -- C_k and E = sum_k C_k^2 (Section 1) of one bit-packed sequence by one warp, the sequence
// held in registers.
//
// Lane l takes the lags k = 32 j + l (j = 0 .. NW - 1): for a given j every lane's word offset is j and its bit
// shift is l, so the shifted words f_v = (s >> l) of word v are formed once and the loops over j and the words
// unroll.  C_k = (L - k) - 2 d, d counting the disagreeing pairs (s_i != s_{i+k}, i < L - k): the words of
// s ^ f, those at the sequence's end masked to its positions in the same instruction.
//
// Popcounts issue at 16 lanes per clock and SM, logic at 64, so the words of a lag are added up by carry-save
// adders first (sum and majority, two LOP3 each): seven words become one of weight 1, one of weight 2 and one
// of weight 4, three popcounts instead of seven for eight LOP3.  Bound: the ALU pipe (about 270 warp
// instructions a sequence at L = 451, 136 cycles; 51 popcounts, 102 cycles; a popcount per word: 240 cycles).
// Measured, 2^20 sequences of L = 451: 574 us (992 us with a popcount per word).
// The tensor cores gain less: f16 mma.sync measured 1,012 multiply-adds per clock and SM, 160 cycles for the product
// whose outputs are the C_k; a form in E4M3 took 510 us for 2^19 sequences, a popcount per word 502 us.
#pragma once

#include "labs_core.cuh"

namespace labsg {

// Sum and carry of three bits, lane by lane, as one three-input operation each (written as a ^ b ^ c and
// (a & b) | (c & (a ^ b)), 2^20 energies of L = 451 measured 12% more time).
__device__ __forceinline__ uint32_t add3(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0x96;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0xE8;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// Counts the ones of N words x(0) .. x(N - 1) (compile-time N and indices).
template <int N, int FROM = 0, class X>
__device__ __forceinline__ int count_words(X&& x) {
  constexpr int n = N - FROM;
  if constexpr (n <= 0) {
    return 0;
  } else if constexpr (n >= 7) {
    const uint32_t a = x(FROM), b = x(FROM + 1), c = x(FROM + 2), d = x(FROM + 3), e = x(FROM + 4), f = x(FROM + 5),
                   g = x(FROM + 6);
    const uint32_t s1 = add3(a, b, c), c1 = maj3(a, b, c), s2 = add3(d, e, f), c2 = maj3(d, e, f), s = add3(s1, s2, g),
                   c3 = maj3(s1, s2, g);
    return __popc(s) + 2 * __popc(add3(c1, c2, c3)) + 4 * __popc(maj3(c1, c2, c3)) + count_words<N, FROM + 7>(x);
  } else if constexpr (n >= 5) {
    const uint32_t a = x(FROM), b = x(FROM + 1), c = x(FROM + 2), d = x(FROM + 3), e = x(FROM + 4);
    const uint32_t s1 = add3(a, b, c);
    return __popc(add3(s1, d, e)) + 2 * (__popc(maj3(a, b, c)) + __popc(maj3(s1, d, e))) + count_words<N, FROM + 5>(x);
  } else if constexpr (n >= 3) {
    const uint32_t a = x(FROM), b = x(FROM + 1), c = x(FROM + 2);
    return __popc(add3(a, b, c)) + 2 * __popc(maj3(a, b, c)) + count_words<N, FROM + 3>(x);
  } else {
    return __popc(x(FROM)) + count_words<N, FROM + 1>(x);
  }
}

// Lag groups J, J + 1, .. of corr_words (compile-time recursion).
template <int NW, int J, class Emit>
__device__ __forceinline__ void corr_lags(const uint32_t (&a)[NW], const uint32_t (&f)[NW], uint32_t m1, uint32_t m2,
                                          int left, Emit&& emit) {
  if constexpr (J < NW) {
    const int d = count_words<NW - J>([&](int w) {
      if (w + J < NW - 2) return a[w] ^ f[w + J];
      uint32_t x;  // (a ^ f) & m
      asm("lop3.b32 %0, %1, %2, %3, 0x28;" : "=r"(x) : "r"(a[w]), "r"(f[w + J]), "r"(w + J == NW - 1 ? m1 : m2));
      return x;
    });
    emit(32 * J + lane_id(), max(left - 32 * J, 0) - 2 * d);
    corr_lags<NW, J + 1>(a, f, m1, m2, left, emit);
  }
}

// emit(k, sum_{i < n-k} a_i b_{i+k}) for the lane's lags k = 32 j + lane, j < NW (0 for k >= n), of two
// sequences of length n, 32 (NW - 1) <= n <= 32 NW, given by their NW 32-bit words in shared memory (16-byte
// aligned), bits at and above n zero.
template <int NW, class Emit>
__device__ __forceinline__ void corr_words(const uint32_t* a, const uint32_t* b, int n, Emit&& emit) {
  const int lane = lane_id();
  uint32_t av[NW], bv[NW], f[NW];
#pragma unroll
  for (int w = 0; w < NW; w++) av[w] = a[w];
#pragma unroll
  for (int w = 0; w < NW; w++) bv[w] = b[w];
#pragma unroll
  for (int v = 0; v < NW; v++) f[v] = __funnelshift_r(bv[v], v + 1 < NW ? bv[v + 1] : 0u, lane);
  // positions of the last two shifted words inside the sequence
  auto low = [](int m) { return m >= 32 ? 0xffffffffu : (m <= 0 ? 0u : (1u << m) - 1u); };
  const int r = n - 32 * (NW - 1) - lane;
  corr_lags<NW, 0>(av, f, low(r), low(r + 32), n - lane, emit);
}

// E of the sequence in sb (as in corr_words, 32 (NW - 1) < L <= 32 NW), on every lane; WITH_C: C_out receives
// C_k at C_out[k - 1], k = 1 .. L-1.
template <int NW, bool WITH_C = false>
__device__ __forceinline__ int energy_words(const uint32_t* sb, int L, int32_t* C_out = nullptr) {
  int e = 0;
  corr_words<NW>(sb, sb, L, [&](int k, int c) {
    e += c * c;
    if (WITH_C && k >= 1 && k < L) C_out[k - 1] = c;
  });
  return warp_sum_i32(e) - L * L;  // without k = 0
}

}  // namespace labsg

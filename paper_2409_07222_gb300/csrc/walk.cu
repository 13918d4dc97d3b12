// walk.cu -- step 1 of the dual-step search: Algorithm 1's self-avoiding walks (labs_skew_search,
// labs_batched_search) and the sieve bound E_l (labs_sample_threshold).
//
// GB300 mapping.  The paper runs one walk per thread block and evaluates every neighbour in time linear in L
// (Section III); here one walk is one warp and a flip changes every neighbour's Delta E by a constant number
// of table values (below), so a step is linear in L instead of quadratic.  A persistent grid of one block per
// SM pulls work items (length, walk) from a device counter, so walks of different lengths and cost balance
// across the 152 SMs in one launch.  A walk's sequence bytes, tables and Bloom filter of 2^bloom_log2 bits
// live in its warp's shared-memory slab (7 KB at L = 451: 32 walks an SM), its neighbours' sums in registers;
// a step is
//   select -- Delta E of the lane's neighbours, warp argmin of (Delta E, m), Bloom test of the winner's
//             fingerprint; on a hit the owner lane looks for its next smallest (same result as testing all),
//   apply  -- the flip, the O(L) tables, then every neighbour's sum from them,
//   sieve  -- the walk's R best distinct (E, fp) states with E <= E_thr.
// Measured (L = 451, p = 24, 65,536 walks x 2,000 flips, sieve bound of 10^6 samples included): 77.6 ms, where
// the scan of every neighbour took 337 ms; 256 walks x 8,192 flips 11.3 ms (74.6 ms: its blocks filled 11 SMs).
#include <algorithm>
#include <cstring>
#include <memory>
#include <mutex>
#include <vector>

#include "energy_words.cuh"
#include "labs_internal.h"

namespace labsg {
namespace {

constexpr int kMaxLens = 96;  // lengths in one launch (kernel parameter table)

// Slots (values of T) a lane of a walk kernel holds, and the threads per block it is compiled for (one block
// per SM): 32 walks of up to 10 slots a lane (64 registers a thread), 24 walks of up to 18 slots (80).  Every
// instantiation spills some registers: 104 bytes a thread at <4, 16, 0>, the slots of L = 451, 276 to 380 at <4, 16, 1>,
// <4, 18, 2>, <5, 18, 1> and <5, 18, 2>.  Measured with 24 walks (80 registers, 48 bytes) in place of 32 for <4, 16, 0>:
// 65,536 walks x 2,000 flips 76.4 ms against 77.6, 256 walks x 8,192 flips 10.3 against 11.4; learned, 8,192 walks in
// chunks of 64, 8.55 against 8.33.  The 32 were chosen for what an SM holds, not for these times.
__host__ __device__ constexpr int walk_slots(int mode, int ns, int nu) {
  return mode == 0 ? 2 * ns : (mode == 1 || nu > 2 * ns ? nu : 2 * ns);
}
__host__ __device__ constexpr int walk_block_threads(int mode, int ns, int nu) {
  return walk_slots(mode, ns, nu) <= 10 ? 1024 : 768;
}

// Halves of a packed table word hold value + kBias, so that adding packed changes never borrows across
// them: |Z| <= 2 * 288 + 576, |X| <= 288, |2 C_d| <= 1152 and |V| <= 576 for every L <= 576.
constexpr int kBias = 2048;

// What a walk changes rarely (its busy values are registers), and with it the values saved between launches.
struct WalkCtl {
  long long skips, skips0;  // skips0 .. dead0: the values when the launch took the walk up
  unsigned long long fp, wfp;
  int E, bestE, first_hit, aprev, dprev;
  int wE, wlane;          // the sieve's worst slot: key (wE, wfp), lane
  unsigned flips, flips0, segs, segs0, dead, dead0;
  unsigned seg0;          // flips at the segment's beginning
  unsigned logged, log_next;  // chunks logged, flips at the beginning of the next
  int need_start, done;
};

// Shared-memory slab of one walk, sized per launch for its lengths (byte offsets, 16-byte aligned): the
// sequence bits at 0, the control block, the sequence bytes, the tables, the Bloom filter (at least kScratch
// bytes: the table builds use its words before a segment's filter is cleared).
struct SlabPlan {
  int off_ctl, off_S, off_tab, off_bloom, bytes;
};
constexpr int kScratch = 96;

// One length of a launch.  Skew walks (odd L = 2k + 1, c = k + 1) address positions by their distance h from
// the centre: S[h] = s_{c-h} for |h| <= k, S[-h] = (-1)^h S[h] (Eq. 2), neighbours h = 0 .. hmax = k - p.
// Unrestricted walks address positions m = p + 1 .. L.
struct WalkLen {
  int L, skew, p, k, c, hmax;
  int so, sn;   // byte of S[0] inside the sequence bytes, their number
  int t1, t2;   // entries of the first table(s) and of all tables: Z0 | Z1 | X at 0, t1, 2 t1 (skew); Z | V (else)
  int T_i;
  int32_t E_thr_value;  // used when WalkParams::E_thr_dev is null
  int64_t item_begin;   // first work item of this length
  int64_t walk_begin;   // global walk id of its first walk
};

struct WalkParams {
  int n_len, R, bloom_log2, bloom_k, prefix_words, n_prefix;
  int32_t E_target;
  int64_t n_items, flip_budget;
  uint64_t seed;
  const uint64_t* prefixes;
  const uint64_t* zpair;     // [n_len][kMaxL]: fingerprint change of neighbour m at m - 1 (walk_init_kernel)
  const int32_t* E_thr_dev;  // nullable: per-length sieve bounds in device memory
  labs_candidate* out;       // [n_items][R]
  int64_t* walk_stats;       // nullable: [n_items][6]
  labs_walk_stats* stats;
  unsigned long long* counter;
  // logs of a plain chunked run (nullable): every `log_chunk` flips the sequence and the next move
  int log_chunk;
  uint64_t* state_log;  // [n_chunks][n_items][W]
  int32_t* move_log;    // [n_chunks][n_items][2]: a chunk's first move (position, Delta E)
  // resumable chunks (learned proposal); all nullable / zero for a plain run to the end
  unsigned char* state;  // [n_items][state_stride]: a walk's slab and its T values ([slot][lane]) between launches
  int state_stride;
  int chunk;             // > 0: at most `chunk` accepted flips per walk and launch; < 0: set-up only
  const float* bias;     // [n_items][L] proposal logits biasing the choice (null: plain walk)
  float lambda;
  uint64_t* seq_out;     // [n_items][W]: the walk's sequence when the launch leaves it
  SlabPlan slab;
  WalkLen len[kMaxLens];
};

// Order-preserving int32 image of a float (-0 folded onto +0 first).
__device__ __forceinline__ int float_key(float f) {
  const int i = __float_as_int(f + 0.0f);
  return i ^ ((i >> 31) & 0x7fffffff);
}

__device__ __forceinline__ uint32_t bloom_idx(uint64_t fp, int j, uint32_t mask) {
  uint32_t lo = (uint32_t)fp, hi = (uint32_t)(fp >> 32);
  return (lo + (uint32_t)j * (hi | 1u)) & mask;
}

// Whether all K probes of fp are set; a lane beyond K repeats the last probe.  Each lane's probe word and
// bit go to `at` and `bit`.
__device__ __forceinline__ bool bloom_test(const uint32_t* bloom, uint64_t fp, int probe, uint32_t mask, uint32_t& at,
                                           uint32_t& bit) {
  const uint32_t b = bloom_idx(fp, probe, mask);
  at = b >> 5;
  bit = 1u << (b & 31);
  return __all_sync(kFull, bloom[at] & bit);
}

__device__ __forceinline__ bool key_less(int Ea, uint64_t fa, int Eb, uint64_t fb) {
  return Ea < Eb || (Ea == Eb && fa < fb);
}

// sum_{j < cnt} a_j b_{j + d} of two +-1 sequences given by bits, d >= 0.
__device__ __forceinline__ int corr_bits(const uint32_t* a, const uint32_t* b, int cnt, int d) {
  if (cnt <= 0) return 0;
  const int ws = d >> 5, sh = d & 31;
  int dis = 0;
  for (int w = 0; 32 * w < cnt; w++) {
    uint32_t x = a[w] ^ __funnelshift_r(b[w + ws], b[w + ws + 1], sh);
    const int rem = cnt - 32 * w;
    if (rem < 32) x &= (1u << rem) - 1u;
    dis += __popc(x);
  }
  return cnt - 2 * dis;
}

// ------------------------------------------------------------------------------------------------
// The incremental neighbourhood.
//
// With T_m = sum_{j != m} C_{|m-j|} s_j (the linear-time sum of a neighbour's Delta E), a flip of f changes
// every T_m by a second difference of E, and that is a constant number of table values: for
// y_d(m) = s_{m+d} + s_{m-d},
//     sum_d y_d(f) y_d(m) = C_{|m-f|} + V_{m+f} - 2 s_f s_m,      V_t = sum_i s_i s_{t-i},
// because the products s_{f+d} s_{m+d} and s_{f-d} s_{m-d} run over all pairs at distance |m - f| but the
// flipped one, and s_{f+d} s_{m-d}, s_{f-d} s_{m+d} over all pairs with index sum m + f.  One flip is then
// O(L): the tables change in one or two products per entry, every T_m in a few table values, and Delta E of
// every neighbour follows.  With the values after the flip (s_f = s, tables C and V updated):
//
// unrestricted, Z_d = 2 C_d with Z_0 := L + 4:
//     T_m += 2 s (Z_{|m-f|} + V_{m+f}) - 8 s_m - 4 s_{2f-m}                          (m = f included)
//     Delta E_m = 4 (V_{2m} + L - 2 - s_m T_m)
//     flip of f:  Z_d += 4 s (s_{f+d} + s_{f-d}),   V_{f+j} += 4 s s_j (j != f)
//
// skew-symmetric, flips of the pair (a, -a) in distances from the centre, e = a mod 2, eta = (-1)^a:
// correlations inside one parity class R^e_g = sum_{h = e (2)} S[h] S[h+2g], C_{2g} = R^0_g + R^1_g,
// Z^e_g = 2 R^e_g + C_{2g} with Z^e_0 := 2 n_e + 12 (n_e = positions of the class), and across the classes
// X_d = sum_{h even} S[h] S[h+d], d odd (odd C vanish, so X of odd h is -X_d).  By Eq. 2 the index-sum
// products are class correlations too.  T_h carries + 4 (-1)^h S[3h] (h > 0):
//     h = e (2):  T_h += 2 s (Z^e_{|h-a|/2} + eta Z^e_{(h+a)/2}) - 24 S[h] - 12 eta y,   y = S[h+2a] + S[h-2a]
//                 and + 8 eta s more for h = 3a and for 3h = a
//     else:       T_h += 4 s (eta sgn(h-a) X_{|h-a|} + X_{h+a}) - 8 S[h] - 4 eta y
//     Delta E_h = 8 ((-1)^h Z^h_h - S[h] T_h) + 16 (n_h - 3),  centre: Delta E_0 = -4 S[0] T_0 + 8 n_0 - 8
//     flip:       R^e_g += 4 s (S[a+2g] + S[a-2g]) without the mirror's product (g = a),
//                 X_d += 2 s eta (S[a+d] - S[a-d])
// The centre alone (a = 0): half of all the above and no y term, T_0 -= 16 s.
//
// Delta E is a multiple of 4 and |Delta E| < 2^23 for every L <= 576 (|T| <= sqrt(E sum y^2), E < 2^26), so
// (Delta E / 4) * 1024 + m orders the neighbours by (Delta E, m) in one int32.
// ------------------------------------------------------------------------------------------------

// One walk per warp.  A lane holds NS slots (values of T) per parity class of a skew walk, NU slots of an
// unrestricted one.  MODE 0: a launch of one skew length, 1: one unrestricted length, 2: several lengths of
// either kind; BIASED: the choice key is the proposal score of WalkParams::bias.
//
// Bound (L = 451, skew): issue slots (88% used) and shared-memory instructions -- a flip is about 75 shared-memory
// accesses and 608 warp instructions (623 with its share of a segment's start), where scanning every neighbour took
// 2,285.
template <int NS, int NU, int MODE, bool BIASED>
__global__ void __launch_bounds__(walk_block_threads(MODE, NS, NU), 1)
    walk_kernel(const __grid_constant__ WalkParams P) {
  constexpr int SL = walk_slots(MODE, NS, NU);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* slab = smem_raw + (size_t)(threadIdx.x >> 5) * P.slab.bytes;
  uint32_t* bits = reinterpret_cast<uint32_t*>(slab);
  WalkCtl* ctl = reinterpret_cast<WalkCtl*>(slab + P.slab.off_ctl);
  uint8_t* Sraw = slab + P.slab.off_S;
  uint16_t* tab = reinterpret_cast<uint16_t*>(slab + P.slab.off_tab);
  uint32_t* bloom = reinterpret_cast<uint32_t*>(slab + P.slab.off_bloom);
  const int lane = lane_id();
  const uint32_t bmask = (1u << P.bloom_log2) - 1u;
  const int bwords = 1 << (P.bloom_log2 - 5);
  const int R = P.R;
  const unsigned budget = (unsigned)P.flip_budget;  // < 2^32, checked by the host

  while (true) {
    unsigned item = 0;  // n_items < 2^32, checked by the host
    if (lane == 0) item = (unsigned)min(atomicAdd(P.counter, 1ull), (unsigned long long)P.n_items);
    item = __shfl_sync(kFull, item, 0);
    if (item >= P.n_items) break;
    int li = 0;
    if (MODE == 2)
      while (li + 1 < P.n_len && P.len[li + 1].item_begin <= (long long)item) li++;
    const WalkLen& le = MODE == 2 ? P.len[li] : P.len[0];
    const int L = le.L, p = le.p;
    const bool skew = MODE == 0 || (MODE == 2 && le.skew);
    const uint64_t* zp = P.zpair + (size_t)li * kMaxL;
    unsigned char* saved = P.state ? P.state + (size_t)item * P.state_stride : nullptr;
    const bool resumed = saved && P.chunk > 0;
    if (resumed && reinterpret_cast<const WalkCtl*>(saved + P.slab.off_ctl)->done) continue;

    uint8_t* S = Sraw + le.so;  // S[h] (skew) or S[position], value + 1 in {0, 2}, 1 outside the sequence
    // skew: Z^0 | Z^1 | X (entry d >> 1); unrestricted: Z | V
    uint16_t* T1 = tab + le.t1;
    uint16_t* TX = tab + 2 * le.t1;
    const int k = le.k, c = le.c, hmax = le.hmax;
    const int n0 = 2 * (k >> 1) + 1, n1 = 2 * ((k + 1) >> 1);  // positions of the even and odd class
    // skew: T[j] is class 0, slot j (h = 2 (lane + 32 j)), T[NS + j] class 1 (h + 1); unrestricted: position
    // p + 1 + lane + 32 j.  sg: the slot's element, 0 without one
    int T[SL], sg[SL];

    unsigned flips = 0, skips = 0;  // skips: Bloom skips since they were last added to ctl
    int bestE = INT32_MAX, E = 0;
    int aprev = -1, dprev = 0;  // neighbour flipped by the previous move of this segment (h or position), its Delta E
    uint64_t fp = 0;
    bool need_start = true;

    // elements of the lane's slots, from the sequence bytes
    auto load_signs = [&]() {
      if (skew) {
#pragma unroll
        for (int j = 0; j < NS; j++)
          {
            const int h = 2 * (lane + 32 * j);
            sg[j] = (int)S[h] - 1;
            sg[NS + j] = (int)S[h + 1] - 1;
          }
      } else if (MODE != 0) {
#pragma unroll
        for (int j = 0; j < NU; j++)
          sg[j] = (int)S[p + 1 + lane + 32 * j] - 1;
      }
    };
    // everything derived from the bits: sequence bytes, tables, energy, T
    auto build_state = [&]() {
      uint32_t* scr = bloom;
      for (int b = lane; b < le.sn; b += 32) {
        const int x = b - le.so;
        const int i = skew ? c - x : x;  // position
        Sraw[b] = (i >= 1 && i <= L) ? (uint8_t)(2 * ((bits[(i - 1) >> 5] >> ((i - 1) & 31)) & 1u)) : (uint8_t)1;
      }
      __syncwarp();
      int e_part = 0;
      if (skew) {
        // class bits: a_j = S[2j - k0], b_j = S[2j - k1], k0 / k1 the largest even / odd distance
        const int k0 = k & ~1, k1 = (k - 1) | 1;
        uint32_t *ab = scr, *bb = scr + 12;
        for (int t = 0; t < 12; t++) {
          const int j = 32 * t + lane;
          const unsigned wa = __ballot_sync(kFull, j < n0 && S[2 * j - k0] == 2);
          const unsigned wb = __ballot_sync(kFull, j < n1 && S[2 * j - k1] == 2);
          if (lane == 0) {
            ab[t] = wa;
            bb[t] = wb;
          }
        }
        __syncwarp();
        for (int g = lane; g < le.t1; g += 32) {
          const int r0 = corr_bits(ab, ab, n0 - g, g), r1 = corr_bits(bb, bb, n1 - g, g);
          const int cg = r0 + r1;
          tab[g] = (uint16_t)(kBias + (g ? 2 * r0 + cg : 2 * n0 + 12));
          T1[g] = (uint16_t)(kBias + (g ? 2 * r1 + cg : 2 * n1 + 12));
          const int sh = (2 * g + 1 + k1 - k0) / 2;
          TX[g] = (uint16_t)(kBias + corr_bits(ab, bb, min(n0, n1 - sh), sh));
          if (g >= 1 && g <= k) e_part += cg * cg;
        }
      } else if (MODE != 0) {
        for (int t = 0; t < kBitWords; t++) {  // the reversed sequence
          const int j = 32 * t + lane;
          const unsigned wr = __ballot_sync(kFull, j < L && S[L - j] == 2);
          if (lane == 0) scr[t] = wr;
        }
        __syncwarp();
        for (int d = lane; d < le.t1; d += 32) {
          const int cd = d < L ? corr_bits(bits, bits, L - d, d) : 0;
          tab[d] = (uint16_t)(kBias + (d ? 2 * cd : L + 4));
          if (d >= 1) e_part += cd * cd;
        }
        for (int t = lane; t < le.t2 - le.t1; t += 32) {  // V_t: the correlation with the reversal at L + 1 - t
          const int d = L + 1 - t;
          int v = 0;
          if (t >= 2 && t <= 2 * L) v = d >= 0 ? corr_bits(bits, scr, L - d, d) : corr_bits(scr, bits, L + d, -d);
          T1[t] = (uint16_t)(kBias + v);
        }
      }
      E = warp_sum_i32(e_part);
      __syncwarp();
      load_signs();
      int csum = 0;
#pragma unroll
      for (int j = 0; j < SL; j++) T[j] = 0;
      if (skew) {
        const uint8_t* s0 = S + 2 * lane;
        for (int g = 1; g <= k; g++) {
          const int cg = ((int)tab[g] + (int)T1[g] - 2 * kBias) >> 2;
          csum += cg;
#pragma unroll
          for (int j = 0; j < NS; j++)
            {
              const int yy = (int)*reinterpret_cast<const uint16_t*>(s0 + 64 * j + 2 * g) +
                             (int)*reinterpret_cast<const uint16_t*>(s0 + 64 * j - 2 * g);
              T[j] += cg * (yy & 255);
              T[NS + j] += cg * (yy >> 8);
            }
        }
#pragma unroll
        for (int j = 0; j < NS; j++)
          {
            const int h = 2 * (lane + 32 * j);
            T[j] -= 2 * csum;
            T[NS + j] -= 2 * csum;
            if (h > 0 && 3 * h <= k) T[j] += 4 * ((int)S[3 * h] - 1);
            if (3 * h + 3 <= k) T[NS + j] -= 4 * ((int)S[3 * h + 3] - 1);
          }
      } else if (MODE != 0) {
        const uint8_t* s0 = S + p + 1 + lane;
        for (int d = 1; d < L; d++) {
          const int cd = ((int)tab[d] - kBias) >> 1;
          csum += cd;
#pragma unroll
          for (int j = 0; j < NU; j++)
            T[j] += cd * ((int)s0[32 * j + d] + (int)s0[32 * j - d]);
        }
#pragma unroll
        for (int j = 0; j < NU; j++) T[j] -= 2 * csum;
      }
    };
    // INIT_PARTITIONED_SEQUENCE of a new segment (Algorithm 1)
    auto start_segment = [&]() {
      const int64_t w = le.walk_begin + ((long long)item - le.item_begin);
      const unsigned seg = ctl->segs;
      build_start(bits, bloom, L, skew, c, p, P.prefixes + (w % P.n_prefix) * P.prefix_words,
                  stream_key(P.seed, kPurposeWalk, (uint64_t)w, (uint64_t)seg));
      build_state();
      __syncwarp();
      for (int t = lane; t < bwords; t += 32) bloom[t] = 0u;
      fp = fingerprint(bits, L, stream_key(0, kPurposeZobrist, (uint64_t)L, 0));
      __syncwarp();
      if (lane < P.bloom_k) {
        const uint32_t b = bloom_idx(fp, lane, bmask);
        atomicOr(&bloom[b >> 5], 1u << (b & 31));
      }
      if (lane == 0) {
        ctl->segs = seg + 1;
        ctl->seg0 = flips;
        ctl->skips += skips;
      }
      skips = 0;
      __syncwarp();
      aprev = -1;
      need_start = false;
    };
    // The tables and T after the flip of neighbour a (already flipped in S; s its new value; own: the bit of
    // its slot in the lane that holds it).
    auto apply_flip = [&](const int a, const int s, const unsigned own) {
      if (skew) {
        const int e = a & 1, es = e ? -s : s;  // es: eta s, the mirror's element
        {
          // lane entry pair g = 2u, 2u + 1 (X: d = 4u + 1, 4u + 3), u = lane + 32 i: the four elements
          // S[a + 4u ..] and the four S[a - 4u - 3 ..], as bytes; 16-bit halves hold the pair
          const int m4 = a ? 4 * s : 2 * s, mz0 = e ? m4 : 3 * m4, mz1 = e ? 3 * m4 : m4, mx = a ? 2 * es : s;
          const int n_it = (min((k + a) >> 1, hmax) >> 6) + 1;
          const int bf = le.so + a, bb = le.so + a - 3;
          const uint32_t* wf = reinterpret_cast<const uint32_t*>(Sraw) + (bf >> 2) + lane;
          const uint32_t* wb = reinterpret_cast<const uint32_t*>(Sraw) + (bb >> 2) - lane;
          const int sf = 8 * (bf & 3), sb = 8 * (bb & 3);
          uint32_t* z0 = reinterpret_cast<uint32_t*>(tab) + lane;
          uint32_t* z1 = reinterpret_cast<uint32_t*>(T1) + lane;
          uint32_t* xx = reinterpret_cast<uint32_t*>(TX) + lane;
          const int ua = (a >> 1) - lane;                               // the pair holding g = a
          const int corr = a ? (e ? es * 65536 : es) : 0;               // its mirror product
#pragma unroll
          for (int i = 0; i < NS; i++) {
            if (i >= n_it) break;
            const uint32_t f = __funnelshift_r(wf[32 * i], wf[32 * i + 1], sf);
            const uint32_t b = __funnelshift_r(wb[-32 * i], wb[-32 * i + 1], sb);
            // even lags: sums of elements 0, 2 of f and 3, 1 of b; odd lags: differences of 1, 3 and 2, 0
            int dy = (int)(__byte_perm(f, 0, 0x4240) + __byte_perm(b, 0, 0x4143) - 0x00020002u);
            const int dx = (int)(__byte_perm(f, 0, 0x4341) - __byte_perm(b, 0, 0x4042));
            if (ua == 32 * i) dy -= corr;
            if (i == 0 && lane == 0) dy -= 2 * s;  // g = 0 is no lag
            z0[32 * i] += (uint32_t)(dy * mz0);
            z1[32 * i] += (uint32_t)(dy * mz1);
            xx[32 * i] += (uint32_t)(dx * mx);
          }
        }
        __syncwarp();
        // T of the class of a, then of the other class; the biases of the bytes and the tables are taken
        // out with the table values (2 cy / cz, 2 cy / cx)
        const int a1 = a >> 1, a2 = (a + 1) >> 1;
        const uint8_t* sp = S + 2 * lane + 2 * a;
        const uint8_t* sm = S + 2 * lane - 2 * a;
        const uint16_t* zq = (e ? T1 : tab) + lane + a2;
        const uint16_t* zm = e ? T1 : tab;
        const uint16_t* xq = TX + lane + a1;
        const int u1 = lane - a1, u2 = lane - a2;
        // odd: a is odd; pair: a > 0 (compile-time)
        auto classes = [&](const bool odd, const bool pair) {
          const int bs = odd ? NS : 0, bo = odd ? 0 : NS;  // first slot of the class of a / of the other class
          const int s2 = pair ? 2 * s : s, s4 = 2 * s2;    // cz, cx
          const int q = odd ? -s4 : s4;                    // eta cx
          const int ky = pair ? (odd ? -12 * s : 12 * s - 2 * kBias) : -2 * kBias;
          const int kx = pair ? (odd ? -2 * s : 2 * s) - kBias : -kBias;
          constexpr int cs = 24, cso = 8, cy = 12, cyo = 4;
#pragma unroll
          for (int j = 0; j < NS; j++) {
            int ylo = 0, yhi = 0;
            if (pair) {
              const int yy = (int)*reinterpret_cast<const uint16_t*>(sp + 64 * j) +
                             (int)*reinterpret_cast<const uint16_t*>(sm + 64 * j);
              ylo = yy & 255;
              yhi = yy >> 8;
            }
            const int vm = zm[abs(u1 + 32 * j)], vq = zq[32 * j];
            int t = T[bs + j] - (pair ? cs : cs / 2) * sg[bs + j];
            t += s2 * (odd ? vm - vq + ky : vm + vq + ky);
            if (pair) t += (odd ? cy : -cy) * (odd ? yhi : ylo);
            T[bs + j] = t;
            const int u = u2 + 32 * j, mk = u >> 31;
            int o = T[bo + j] - (pair ? cso : cso / 2) * sg[bo + j];
            o += (mk ? -q : q) * ((int)TX[u ^ mk] - kBias);
            o += s4 * ((int)xq[32 * j] + kx);
            if (pair) o += (odd ? cyo : -cyo) * (odd ? ylo : yhi);
            T[bo + j] = o;
          }
        };
        // the flipped element's own slot
#pragma unroll
        for (int t = 0; t < SL; t++)
          if (t < 2 * NS && (own >> t & 1)) sg[t] = s;
        if (e)
          classes(true, true);
        else if (a)
          classes(false, true);
        else
          classes(false, false);
        if (a == 0) {
          if (lane == 0) T[0] -= 16 * s;
        } else if (3 * a <= hmax || a % 3 == 0) {  // h = 3a and 3h = a: 8 eta s more, in the class of a
          const int i3 = ((3 * a) >> 1) - lane, id3 = a % 3 == 0 ? (a / 3 >> 1) - lane : -1;
#pragma unroll
          for (int j = 0; j < NS; j++)
            if (i3 == 32 * j || id3 == 32 * j) {
              if (e)
                T[NS + j] += 8 * es;
              else
                T[j] += 8 * es;
            }
        }
      } else if (MODE != 0) {
        const int f = a;  // position
        {
          // Z_d, four lags d = 4u .. 4u + 3 per lane
          const int n_it = (max(f - 1, L - f) >> 7) + 1;
          const int bf = le.so + f, bb = le.so + f - 3;
          const uint32_t* wf = reinterpret_cast<const uint32_t*>(Sraw) + (bf >> 2) + lane;
          const uint32_t* wb = reinterpret_cast<const uint32_t*>(Sraw) + (bb >> 2) - lane;
          const int sf = 8 * (bf & 3), sb = 8 * (bb & 3);
          uint2* z = reinterpret_cast<uint2*>(tab) + lane;
          for (int i = 0; i < n_it; i++) {
            const uint32_t fw = __funnelshift_r(wf[32 * i], wf[32 * i + 1], sf);
            const uint32_t bw = __funnelshift_r(wb[-32 * i], wb[-32 * i + 1], sb);
            int dlo = (int)(__byte_perm(fw, 0, 0x4140) + __byte_perm(bw, 0, 0x4243)) - 0x00020002;
            const int dhi = (int)(__byte_perm(fw, 0, 0x4342) + __byte_perm(bw, 0, 0x4041)) - 0x00020002;
            if (lane + 32 * i == 0) dlo -= 2 * s;  // d = 0 is no lag
            uint2 v = z[32 * i];
            v.x += (uint32_t)(dlo * 4 * s);
            v.y += (uint32_t)(dhi * 4 * s);
            z[32 * i] = v;
          }
          // V_t, four sums t = t0 + 4u .. + 3 per lane, elements j = t - f
          const int t0 = (f + 1) & ~3;
          const int m_it = ((f + L - t0) >> 7) + 1;
          const int bj = le.so + t0 - f;
          const uint32_t* wj = reinterpret_cast<const uint32_t*>(Sraw) + (bj >> 2) + lane;
          const int sj = 8 * (bj & 3);
          uint2* vv = reinterpret_cast<uint2*>(T1 + t0) + lane;
          const int own = 2 * f - t0;  // t = 2f: the square of the flipped element, unchanged
          for (int i = 0; i < m_it; i++) {
            const uint32_t x = __funnelshift_r(wj[32 * i], wj[32 * i + 1], sj);
            int dlo = (int)__byte_perm(x, 0, 0x4140) - 0x00010001, dhi = (int)__byte_perm(x, 0, 0x4342) - 0x00010001;
            if (lane + 32 * i == (own >> 2)) {
              const int d = own & 1 ? s * 65536 : s;
              if (own & 2)
                dhi -= d;
              else
                dlo -= d;
            }
            uint2 v = vv[32 * i];
            v.x += (uint32_t)(dlo * 4 * s);
            v.y += (uint32_t)(dhi * 4 * s);
            vv[32 * i] = v;
          }
        }
        __syncwarp();
        const int af = f - p - 1;  // slot index of f
        const uint16_t* vt = T1 + f + p + 1 + lane;
        const uint8_t* sr = S + 2 * f - p - 1 - lane;
#pragma unroll
        for (int j = 0; j < NU; j++)
          {
            const int idx = lane + 32 * j;
            if (own >> j & 1) sg[j] = s;
            const int z = (int)tab[abs(idx - af)] + (int)vt[32 * j] - 2 * kBias;
            T[j] += 2 * s * z - 8 * sg[j] - 4 * ((int)sr[-32 * j] - 1);
          }
      }
    };
    // (Delta E / 4) * 1024 + m of every slot t (compile-time after unrolling) of the lane, as the sum of a
    // value and a compile-time constant: take(t, value, constant)
    const int b0 = (4 * (n0 - 3) - 2 * kBias) * 1024 + c - 2 * lane;
    const int b1 = (4 * (n1 - 3) + 2 * kBias) * 1024 + c - 1 - 2 * lane;
    const int bu = (L - 2 - kBias) * 1024 + p + 1 + lane;
    auto lane_keys = [&](auto&& take) {
      if (skew) {
        const uint16_t* z0 = tab + 2 * lane;
        const uint16_t* z1 = T1 + 2 * lane + 1;
#pragma unroll
        for (int j = 0; j < NS; j++) {
          int v = ((int)z0[64 * j] - sg[j] * T[j]) * 2048 + b0;
          if (j == 0 && lane == 0) v = (2 * n0 - 2 - sg[0] * T[0]) * 1024 + c;
          take(j, v, -64 * j);
          take(NS + j, ((int)z1[64 * j] + sg[NS + j] * T[NS + j]) * -2048 + b1, -64 * j);
        }
      } else if (MODE != 0) {
        const uint16_t* v = T1 + 2 * (p + 1 + lane);
#pragma unroll
        for (int j = 0; j < NU; j++) take(j, ((int)v[64 * j] - sg[j] * T[j]) * 1024 + bu, 32 * j);
      }
    };
    // bit of neighbour a's slot in the lane that holds it, 0 in the others
    auto own_bit = [&](int a) {
      const int idx = skew ? a >> 1 : a - p - 1;
      const int t = (idx >> 5) + (skew && (a & 1) ? NS : 0);
      return lane == (idx & 31) ? 1u << t : 0u;
    };
    unsigned act = 0;  // the lane's slots that hold a neighbour
#pragma unroll
    for (int t = 0; t < SL; t++) {
      const bool on = skew ? t < 2 * NS && 2 * (lane + 32 * (t % NS)) + t / NS <= hmax : lane + 32 * t <= hmax;
      if (on) act |= 1u << t;
    }
    const int probe = min(lane, P.bloom_k - 1);
    // largest (E, fp) of the R sieve slots (lane r holds slot r), lowest lane among equals, into ctl
    auto find_worst = [&](int cE, uint64_t cfp) {
      const int mE = warp_max_i32(lane < R ? cE : INT32_MIN);
      uint64_t mf = (lane < R && cE == mE) ? cfp : 0ull;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const uint64_t other = __shfl_xor_sync(kFull, mf, o);
        mf = other > mf ? other : mf;
      }
      const unsigned who = __ballot_sync(kFull, lane < R && cE == mE && cfp == mf);
      if (lane == 0) {
        ctl->wE = mE;
        ctl->wfp = mf;
        ctl->wlane = __ffs(who) - 1;
      }
      __syncwarp();
    };
    // sequence words of the walk, to global memory
    auto store_seq = [&](uint64_t* dst) {
      if (lane < (L + 63) >> 6) dst[lane] = (uint64_t)bits[2 * lane] | ((uint64_t)bits[2 * lane + 1] << 32);
    };
    auto record = [&](int r) { return P.out + (size_t)item * R + r; };

    __syncwarp();  // the previous walk of this warp is done with ctl
    if (!resumed) {
      if (lane == 0) {
        WalkCtl z{};
        z.wE = INT32_MAX;
        z.wfp = ~0ull;
        z.first_hit = -1;
        *ctl = z;
      }
      if (lane < R) {  // empty sieve slots
        labs_candidate* r = record(lane);
        r->E = INT32_MAX;
        r->walk = 0;
        r->step = 0;
        r->pad = 0;
        r->fp = ~0ull;
#pragma unroll
        for (int t = 0; t < LABS_MAX_W; t++) r->seq[t] = 0;
      }
      __syncwarp();
    } else {
      for (int t = lane; t < P.slab.bytes / 4; t += 32)
        reinterpret_cast<uint32_t*>(slab)[t] = reinterpret_cast<const uint32_t*>(saved)[t];
      const int* gt = reinterpret_cast<const int*>(saved + P.slab.bytes) + lane;
#pragma unroll
      for (int j = 0; j < SL; j++) T[j] = gt[32 * j];
      __syncwarp();
      flips = ctl->flips;
      fp = ctl->fp;
      E = ctl->E;
      bestE = ctl->bestE;
      aprev = ctl->aprev;
      dprev = ctl->dprev;
      need_start = ctl->need_start;
      load_signs();
      __syncwarp();
      if (lane == 0) {
        ctl->skips0 = ctl->skips;
        ctl->flips0 = ctl->flips;
        ctl->segs0 = ctl->segs;
        ctl->dead0 = ctl->dead;
        ctl->logged = 0;
        ctl->log_next = ctl->flips;
      }
      __syncwarp();
    }
    // the launch's last flip; a set-up launch only builds the first state
    const unsigned stop = P.chunk == 0 ? budget : (unsigned)min((unsigned long long)budget, (unsigned long long)flips + (P.chunk > 0 ? P.chunk : 0));
    const int32_t E_thr = P.E_thr_dev ? P.E_thr_dev[li] : le.E_thr_value;
    // a state with E <= gate is looked at: the sieve takes states inside its bound that beat its worst slot,
    // and the first one at the target is noted
    auto gate_of = [&]() {
      const int g = min(E_thr, ctl->wE);
      return ctl->first_hit < 0 ? max(g, P.E_target) : g;
    };
    int gate = gate_of();
    bool log_move = false;  // the next accepted move is a chunk's first

    while (true) {  // stretches of flips between the events: restarts, chunk logs, the end
      if (P.log_chunk > 0) {
        if (log_move && flips != ctl->log_next) {  // the chunk's first move has been made
          const unsigned lg = ctl->logged;
          __syncwarp();
          if (lane == 0) {
            if (P.move_log) {
              int32_t* ml = P.move_log + ((size_t)lg * P.n_items + item) * 2;
              ml[0] = skew ? c - aprev : aprev;
              ml[1] = dprev;
            }
            ctl->logged = lg + 1;
            ctl->log_next = P.chunk > 0 ? 0xffffffffu : (lg + 1) * (unsigned)P.log_chunk;
          }
          __syncwarp();
          log_move = false;
        }
        if (!log_move && flips == ctl->log_next && flips < stop) {
          if (ctl->logged == 0 && need_start) start_segment();  // the first chunk begins with the first state
          if (P.state_log) store_seq(P.state_log + ((size_t)ctl->logged * P.n_items + item) * ((L + 63) >> 6));
          log_move = true;
        }
      }
      if (need_start && (flips < stop || (P.chunk < 0 && flips < budget))) start_segment();
      if (flips >= stop) break;
      if (lane == 0) ctl->skips += skips;
      skips = 0;
      // flips of this stretch (at most 2^20, so that skips cannot overflow)
      unsigned long long next = min((unsigned long long)stop, flips + (1ull << 20));
      next = min(next, ctl->seg0 + (unsigned long long)le.T_i);
      if (P.log_chunk > 0) next = min(next, log_move ? flips + 1ull : (unsigned long long)ctl->log_next);
      const unsigned until = (unsigned)next;
      do {
        // ---- select: smallest (key, m) whose neighbour is not in the Bloom filter.  A hit makes the owner
        //      lane look for its next smallest.  The move back is certainly in the filter: its slot is left
        //      out, and as its Delta E undoes the last move's, it is known without its slot whether it ranked
        //      ahead of the chosen move and counts as a skip.
        const unsigned own_prev = aprev >= 0 ? own_bit(aprev) : 0u;
        const unsigned use = act & ~own_prev;
        int astar = -1, dstar = 0;
        uint64_t nfp = 0;
        uint32_t b_at = 0, b_bit = 0;
        if (!BIASED) {
          int best = INT32_MAX, cmin;
          lane_keys([&](int t, int v, int k) {
            if (use >> t & 1) best = min(best, v + k);
          });
          while (true) {
            cmin = warp_min_i32(best);
            if (cmin == INT32_MAX) break;
            const int m = cmin & 1023;
            nfp = fp ^ zp[m - 1];
            if (!bloom_test(bloom, nfp, probe, bmask, b_at, b_bit)) {
              astar = skew ? c - m : m;
              dstar = (cmin >> 10) * 4;
              break;
            }
            skips++;
            if (best == cmin) {  // the lane's smallest key above cmin
              best = INT32_MAX;
              lane_keys([&](int t, int v, int k) {
                if ((use >> t & 1) && v + k > cmin) best = min(best, v + k);
              });
            }
          }
          const int mprev = skew ? c - aprev : aprev;
          if (aprev >= 0 && -(dprev >> 2) * 1024 + mprev < cmin) skips++;
        } else {
          const float* bias = P.bias + (size_t)item * L;
          auto key_of = [&](int m, int d) {
            float l = bias[m - 1];
            if (!isfinite(l)) l = 0.f;  // a missing or broken proposal falls back to the plain choice
            return float_key(fmaf(-P.lambda, l, (float)d));
          };
          int bk = INT32_MAX, bm = INT32_MAX, bd = 0;
          int kmin = INT32_MIN, mm = 0;
          bool mine = true;
          while (true) {
            if (mine) {  // the lane's smallest (key, m) ranked after (kmin, mm)
              bk = INT32_MAX;
              bm = INT32_MAX;
              lane_keys([&](int t, int v, int k) {
                if (!(use >> t & 1)) return;
                const int m = (v + k) & 1023, d = ((v + k) >> 10) * 4;
                const int key = key_of(m, d);
                if ((key > kmin || (key == kmin && m > mm)) && (key < bk || (key == bk && m < bm))) {
                  bk = key;
                  bm = m;
                  bd = d;
                }
              });
            }
            kmin = warp_min_i32(bk);
            if (kmin == INT32_MAX) break;
            mm = (int)warp_min_u32(bk == kmin ? (unsigned)bm : 0xffffffffu);
            mine = bk == kmin && bm == mm;
            const int d = __shfl_sync(kFull, bd, __ffs(__ballot_sync(kFull, mine)) - 1);
            nfp = fp ^ zp[mm - 1];
            if (!bloom_test(bloom, nfp, probe, bmask, b_at, b_bit)) {
              astar = skew ? c - mm : mm;
              dstar = d;
              break;
            }
            skips++;
          }
          if (aprev >= 0) {
            const int mprev = skew ? c - aprev : aprev;
            const int bkey = key_of(mprev, -dprev);
            if (bkey != INT32_MAX && (astar < 0 || bkey < kmin || (bkey == kmin && mprev < mm))) skips++;
          }
        }
        if (astar < 0) {
          if (lane == 0) ctl->dead++;
          need_start = true;
          break;
        }
        // ---- apply
        const int s = 1 - (int)S[astar];  // the element's new value
        __syncwarp();                     // every lane has read what the flip changes
        if (lane < (skew && astar ? 2 : 1)) {
          const int x = lane ? -astar : astar;
          const int i = (skew ? c - x : x) - 1;
          S[x] = (uint8_t)(2 - S[x]);
          atomicXor(&bits[i >> 5], 1u << (i & 31));
        }
        if (lane < P.bloom_k) atomicOr(&bloom[b_at], b_bit);
        E += dstar;
        fp = nfp;
        __syncwarp();
        apply_flip(astar, s, own_bit(astar));
        aprev = astar;
        dprev = dstar;
        flips++;
        bestE = min(bestE, E);
        if (E <= gate) {
          if (E <= P.E_target && ctl->first_hit < 0) {
            __syncwarp();
            if (lane == 0) ctl->first_hit = (int)flips;
            __syncwarp();
          }
          // ---- sieve
          if (E <= E_thr && key_less(E, fp, ctl->wE, ctl->wfp)) {
            int cE = INT32_MAX;
            uint64_t cfp = ~0ull;
            if (lane < R) {
              cE = record(lane)->E;
              cfp = record(lane)->fp;
            }
            if (!__any_sync(kFull, cE != INT32_MAX && cfp == fp)) {  // not kept yet
              const int wl = ctl->wlane;
              labs_candidate* rr = record(wl);
              if (lane == wl) {
                cE = E;
                cfp = fp;
                rr->E = E;
                rr->walk = (uint32_t)(le.walk_begin + ((long long)item - le.item_begin));
                rr->step = (uint32_t)flips;
                rr->fp = fp;
              }
              store_seq(rr->seq);
              find_worst(cE, cfp);
            }
          }
          gate = gate_of();
        }
      } while (flips != until);
      if (flips - ctl->seg0 >= (unsigned)le.T_i) need_start = true;
      __syncwarp();
    }
    __syncwarp();
    if (lane == 0) {
      ctl->skips += skips;
      ctl->flips = flips;
      ctl->bestE = bestE;
      ctl->E = E;
      ctl->fp = fp;
      ctl->aprev = aprev;
      ctl->dprev = dprev;
      ctl->need_start = need_start ? 1 : 0;
    }
    __syncwarp();
    if (P.seq_out) store_seq(P.seq_out + (size_t)item * ((L + 63) >> 6));
    if (flips < budget) {
      // ---- leave the walk for the next launch
      if (saved) {
        for (int t = lane; t < P.slab.bytes / 4; t += 32)
          reinterpret_cast<uint32_t*>(saved)[t] = reinterpret_cast<const uint32_t*>(slab)[t];
        int* gt = reinterpret_cast<int*>(saved + P.slab.bytes) + lane;
#pragma unroll
        for (int j = 0; j < SL; j++) gt[32 * j] = T[j];
      }
    } else {
      // ---- final: sort the R slots by (E, fp) (ties between empty slots by lane) and rewrite in place
      labs_candidate mine;
      mine.E = INT32_MAX;
      mine.fp = ~0ull;
      if (lane < R) mine = *record(lane);
      int rank = 0;
      for (int r = 0; r < R; r++) {
        const int oE = __shfl_sync(kFull, mine.E, r);
        const uint64_t of = __shfl_sync(kFull, mine.fp, r);
        if (key_less(oE, of, mine.E, mine.fp) || (oE == mine.E && of == mine.fp && r < lane)) rank++;
      }
      __syncwarp();
      if (lane < R) *record(rank) = mine;
      if (lane == 0) {
        if (P.walk_stats) {
          int64_t* st = P.walk_stats + (int64_t)item * 6;
          st[0] = (int64_t)flips;
          st[1] = (int64_t)ctl->segs;
          st[2] = ctl->skips;
          st[3] = (int64_t)ctl->dead;
          st[4] = bestE;
          st[5] = ctl->first_hit;
        }
        if (saved) reinterpret_cast<WalkCtl*>(saved + P.slab.off_ctl)->done = 1;
      }
    }
    if (lane == 0) {
      atomicAdd(reinterpret_cast<unsigned long long*>(&P.stats->flips), (unsigned long long)(flips - ctl->flips0));
      atomicAdd(reinterpret_cast<unsigned long long*>(&P.stats->segments), (unsigned long long)(ctl->segs - ctl->segs0));
      atomicAdd(reinterpret_cast<unsigned long long*>(&P.stats->bloom_skips), (unsigned long long)(ctl->skips - ctl->skips0));
      atomicAdd(reinterpret_cast<unsigned long long*>(&P.stats->dead_ends), (unsigned long long)(ctl->dead - ctl->dead0));
      atomicMin(&P.stats->best_E, bestE);
    }
  }
}

// One block per length: the fingerprint change of every neighbour (the Zobrist keys of its flipped
// positions).  Block 0 also zeroes the aggregates and the work counter; E_thr reports the first length's
// sieve bound.
__global__ void __launch_bounds__(128) walk_init_kernel(const __grid_constant__ WalkParams P, uint64_t* zpair) {
  const WalkLen& le = P.len[blockIdx.x];
  const uint64_t zk = stream_key(0, kPurposeZobrist, (uint64_t)le.L, 0);
  const int n = le.skew ? le.c : le.L;
  for (int m = 1 + threadIdx.x; m <= n; m += blockDim.x)
    zpair[(size_t)blockIdx.x * kMaxL + m - 1] =
        zobrist(zk, m) ^ (le.skew && m != le.c ? zobrist(zk, le.L + 1 - m) : 0ull);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    labs_walk_stats* stats = P.stats;
    stats->flips = 0;
    stats->segments = 0;
    stats->bloom_skips = 0;
    stats->dead_ends = 0;
    stats->E_thr = P.E_thr_dev ? P.E_thr_dev[0] : le.E_thr_value;
    stats->best_E = INT32_MAX;
    stats->status = LABS_OK;
    stats->reserved = 0;
    *P.counter = 0ull;
  }
}

// ---------------------------------------------------------------------------------------------
// Sieve bound: sample energies, then an exact two-level radix select (13 + 13 bits; E < 2^26).
// ---------------------------------------------------------------------------------------------
constexpr int kSampleWarps = 8;
constexpr int kHistBins = 8192;

// One warp per sample: the start's bits and its energy (all lags: a skew start's odd ones are zero).  The
// energies crowd into a few of the first level's bins, so a block counts in shared memory and adds its counts
// once (an atomic per sample would serialise on them).
template <int NW>
__global__ void __launch_bounds__(32 * kSampleWarps) sample_kernel(int L, int skew, int p,
                                                                    const uint64_t* __restrict__ prefixes, int n_prefix,
                                                                    int prefix_words, uint64_t seed, int64_t n,
                                                                    int32_t* __restrict__ E_out,
                                                                    unsigned* __restrict__ hist) {
  __shared__ unsigned counts[kHistBins];
  __shared__ __align__(16) uint32_t bits_all[kSampleWarps][kBitWords], scr_all[kSampleWarps][kBitWords + 2];
  uint32_t* bits = bits_all[threadIdx.x >> 5];
  for (int b = threadIdx.x; b < kHistBins; b += blockDim.x) counts[b] = 0u;
  __syncthreads();
  const int64_t warps_total = (int64_t)gridDim.x * kSampleWarps;
  for (int64_t i = (int64_t)blockIdx.x * kSampleWarps + (threadIdx.x >> 5); i < n; i += warps_total) {
    build_start(bits, scr_all[threadIdx.x >> 5], L, skew != 0, (L + 1) / 2, p, prefixes + (i % n_prefix) * prefix_words,
                stream_key(seed, kPurposeThresh, (uint64_t)i, 0));
    const int E = energy_words<NW>(bits, L);
    if (lane_id() == 0) {
      E_out[i] = E;
      atomicAdd(&counts[E >> 13], 1u);
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < kHistBins; b += blockDim.x)
    if (counts[b]) atomicAdd(&hist[b], counts[b]);
}

// One block of 1024 threads: the bin of hist (kHistBins bins, eight a thread) that holds `rank`, and the
// rank inside it.  Returns true on the one thread that found it.
__device__ __forceinline__ bool find_bin(const unsigned* __restrict__ hist, unsigned long long rank, int* bin,
                                         unsigned long long* inside) {
  __shared__ unsigned long long warp_sum[32];
  const int t = threadIdx.x, lane = lane_id();
  unsigned own[8];
  unsigned long long s = 0;
#pragma unroll
  for (int b = 0; b < 8; b++) {
    own[b] = hist[t * 8 + b];
    s += own[b];
  }
  unsigned long long incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) warp_sum[t >> 5] = incl;
  __syncthreads();
  unsigned long long before = incl - s;
  for (int w = 0; w < t >> 5; w++) before += warp_sum[w];
  if (!(before <= rank && rank < before + s)) return false;
  int b = 0;
  while (b < 7 && before + own[b] <= rank) before += own[b++];
  *bin = t * 8 + b;
  *inside = rank - before;
  return true;
}

__global__ void __launch_bounds__(1024) select_bin_kernel(const unsigned* __restrict__ hist, int64_t rank, long long* sel) {
  int bin;
  unsigned long long inside;
  if (find_bin(hist, (unsigned long long)rank, &bin, &inside)) {
    sel[0] = bin;
    sel[1] = (long long)inside;
  }
}

__global__ void hist_low_kernel(const int32_t* __restrict__ E, int64_t n, const long long* sel,
                                unsigned* __restrict__ hist2) {
  const int bin = (int)sel[0];
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int e = E[i];
    if ((e >> 13) == bin) atomicAdd(&hist2[e & 8191], 1u);
  }
}

__global__ void __launch_bounds__(1024) finish_select_kernel(const unsigned* __restrict__ hist2, const long long* sel,
                                                             int32_t* E_thr_out) {
  int low;
  unsigned long long inside;
  if (find_bin(hist2, (unsigned long long)sel[1], &low, &inside)) *E_thr_out = (int32_t)((sel[0] << 13) | low);
}

// The whole bound on `st`: samples into Es [n_samples], the two histograms at hist, the selected bin at sel.
static int issue_threshold(int sms, int L, int skew, int p, const uint64_t* prefixes, int n_prefix, int prefix_words,
                           uint64_t seed, int64_t n_samples, int64_t rank, int32_t* E_thr_out, int32_t* Es,
                           unsigned* hist, long long* sel, cudaStream_t st) {
  if (cudaMemsetAsync(hist, 0, sizeof(unsigned) * 2 * kHistBins, st) != cudaSuccess) return LABS_ERR_CUDA;
  const unsigned blocks = (unsigned)std::min<int64_t>((n_samples + kSampleWarps - 1) / kSampleWarps, (int64_t)sms * 4);
  const int s = by_words((L + 31) >> 5, [&](auto nw) {
    sample_kernel<decltype(nw)::value>
        <<<blocks, 32 * kSampleWarps, 0, st>>>(L, skew, p, prefixes, n_prefix, prefix_words, seed, n_samples, Es, hist);
    return cuda_status(cudaGetLastError());
  });
  if (s != LABS_OK) return s;
  select_bin_kernel<<<1, 1024, 0, st>>>(hist, rank, sel);
  const int64_t hb = std::min<int64_t>((n_samples + 255) / 256, (int64_t)sms * 8);
  hist_low_kernel<<<(unsigned)hb, 256, 0, st>>>(Es, n_samples, sel, hist + kHistBins);
  finish_select_kernel<<<1, 1024, 0, st>>>(hist + kHistBins, sel, E_thr_out);
  return cuda_status(cudaGetLastError());
}

// ---------------------------------------------------------------------------------------------
// Which configurations are accepted.  The tile parameters (tile_m, lanes_per_walk) select nothing in the incremental
// walk; they were those of a tiled scan of all neighbours, and what that scan had no plan for was refused.  Callers
// may rely on the refusals, so they are kept exactly: make_layout, the eight tiles and the ranking by scan work below
// answer nothing else.  The ranking matters for one of them: with lanes_per_walk 0, more than eight warps per CTA are
// accepted where the plan of least work had 16 lanes a walk.
// ---------------------------------------------------------------------------------------------
constexpr int kMaxPasses = 3;  // lane passes over the tiles of one walk
struct Variant {
  int M, H, GL;  // tile, lag ranges per tile, lanes per walk
};
static const Variant kVariants[] = {{8, 1, 32}, {12, 1, 32}, {16, 1, 32}, {16, 2, 32},
                                    {8, 1, 16}, {12, 1, 16}, {16, 1, 16}, {16, 2, 16}};

// Passes a length needs with variant v (0 if the layout does not fit).
static int passes_for(int L, int skew, int p, const Variant& v) {
  Layout ly;
  if (!make_layout(ly, L, skew, p, v.M, v.H)) return 0;
  int np = (ly.n_tasks + v.GL - 1) / v.GL;
  return np < 1 ? 1 : np;
}

// One launch's lengths.
struct LenSpec {
  int L, skew, p, T_i;
  int64_t walks, walk_begin;
};

// The plan of least scan work, sum(walks * NP * M / H * GL / 32), that the requested parameters allow; ties
// to fewer lanes per walk, fewer passes, more lanes per tile, the larger tile.  False if there is none: refused.
// req_m / req_gl: 0 or the tile size / lanes per walk the caller fixed; R: sieve slots per walk.
static bool choose_variant(const std::vector<LenSpec>& lens, int req_m, int req_gl, int R, Variant* out) {
  bool found = false;
  long double best_cost = 0;
  int best_np = 0;
  Variant best{0, 0, 0};
  for (const Variant& v : kVariants) {
    if (req_m && v.M != req_m) continue;
    if (req_gl && v.GL != req_gl) continue;
    if (R > v.GL) continue;
    long double cost = 0;
    int max_np = 0;
    bool ok = true;
    for (const LenSpec& s : lens) {
      int np = passes_for(s.L, s.skew, s.p, v);
      if (np == 0 || np > kMaxPasses) {
        ok = false;
        break;
      }
      max_np = std::max(max_np, np);
      cost += (long double)std::max<int64_t>(s.walks, 1) * np * v.M / v.H * v.GL / 32;
    }
    if (!ok) continue;
    const bool better =
        !found || cost < best_cost ||
        (cost == best_cost &&
         (v.GL < best.GL ||
          (v.GL == best.GL && (max_np < best_np || (max_np == best_np && (v.H > best.H || (v.H == best.H && v.M > best.M)))))));
    if (better) {
      best = v;
      best_cost = cost;
      best_np = max_np;
      found = true;
    }
  }
  *out = best;
  return found;
}

static bool accepted(const std::vector<LenSpec>& lens, int req_m, int req_gl, int R, int warps) {
  Variant v;
  return choose_variant(lens, req_m, req_gl, R, &v) && 32 * warps <= (v.GL == 32 ? 256 : 384);
}

// A launch's kernel (slots per lane, mode) and shape.
struct Launch {
  int ns, nu, mode, warps;
  long long blocks;
  size_t smem;
};

typedef void (*WalkKernel)(const WalkParams);
template <int NS, int NU>
static WalkKernel walk_fn_of(int mode, bool biased) {  // biased launches hold one length
  if (mode == 0) return biased ? walk_kernel<NS, NU, 0, true> : walk_kernel<NS, NU, 0, false>;
  if (mode == 1) return biased ? walk_kernel<NS, NU, 1, true> : walk_kernel<NS, NU, 1, false>;
  return walk_kernel<NS, NU, 2, false>;
}
// Compiled slot counts: lengths to 128, 256, 384, 512 and 576 (fewer slots where a prefix leaves fewer
// neighbours); a launch takes the smallest that holds all its lengths.
static const int kSlots[][2] = {{1, 4}, {2, 8}, {3, 12}, {4, 16}, {4, 18}, {5, 18}};
static WalkKernel walk_fn(const Launch& ln, bool biased) {
  switch (100 * ln.ns + ln.nu) {
    case 104: return walk_fn_of<1, 4>(ln.mode, biased);
    case 208: return walk_fn_of<2, 8>(ln.mode, biased);
    case 312: return walk_fn_of<3, 12>(ln.mode, biased);
    case 416: return walk_fn_of<4, 16>(ln.mode, biased);
    case 418:  // for unrestricted lengths beyond 512; the skew part of a mixed launch has four slots
      return ln.mode == 2 ? walk_kernel<4, 18, 2, false> : ln.mode == 1 ? walk_fn_of<5, 18>(1, biased) : walk_fn_of<4, 16>(0, biased);
    default: return walk_fn_of<5, 18>(ln.mode, biased);
  }
}

// Fills the per-length table and the slab plan, and picks the kernel.  Every index that the kernel forms
// from these sizes is checked on the CPU for all lengths (tests/test_walk_tables.py mirrors this plan).
static void fill_params(WalkParams& P, const std::vector<LenSpec>& lens, int bloom_log2, Launch* ln) {
  P.n_len = (int)lens.size();
  int need_s = 0, need_u = 0;  // slots a lane needs
  for (const LenSpec& s : lens) {
    if (s.skew)
      need_s = std::max(need_s, ((s.L - 1) / 2 - s.p) / 64 + 1);
    else
      need_u = std::max(need_u, (s.L - s.p - 1) / 32 + 1);
  }
  ln->mode = lens.size() > 1 ? 2 : (lens[0].skew ? 0 : 1);
  for (const auto& sl : kSlots) {
    ln->ns = sl[0];
    ln->nu = sl[1];
    if (need_s <= sl[0] && need_u <= sl[1]) break;
  }
  int64_t item = 0;
  int sn = 16, tab = 16;
  for (size_t i = 0; i < lens.size(); i++) {
    WalkLen& e = P.len[i];
    const LenSpec& s = lens[i];
    e.L = s.L;
    e.skew = s.skew;
    e.p = s.p;
    e.k = (s.L - 1) / 2;
    e.c = (s.L + 1) / 2;
    int lo, hi;  // sequence bytes reached: S[-lo] .. S[hi]
    if (s.skew) {
      e.hmax = e.k - s.p;
      const int hpad = 64 * ln->ns - 1;  // distances of the last slots, with and without a neighbour
      e.t1 = (std::max(e.k + 1, hpad + 1) + 3) / 4 * 4;
      e.t2 = 3 * e.t1;
      // T reads S[h +- 2g] for g <= max(k, hmax); the table update S[a +- d] for whole 128-lag turns
      hi = std::max(hpad + 2 * e.k, std::min(2 * e.hmax + e.k, 3 * e.hmax) + 127);
      lo = std::max(2 * e.k, std::min(e.k, 2 * e.hmax) + 127);
    } else {
      e.hmax = s.L - s.p - 1;
      const int mpad = s.p + 32 * ln->nu;  // position of the last slot
      e.t1 = 128 * ((std::max(s.L - 1, 32 * ln->nu - 1)) / 128 + 1);
      e.t2 = e.t1 + (std::max(2 * std::max(s.L + 64, mpad + 1), mpad + s.L + 1) + 3) / 4 * 4;
      hi = std::max(2 * s.L + 127, mpad + s.L);
      lo = std::max(s.L + 127, mpad);
    }
    e.so = (lo + 8) / 4 * 4;  // a realigned word may start three bytes below
    e.sn = (e.so + hi + 8 + 3) / 4 * 4;
    sn = std::max(sn, e.sn);
    tab = std::max(tab, 2 * e.t2);
    e.T_i = s.T_i > 0 ? s.T_i : 4 * (s.L + 1);
    e.E_thr_value = INT32_MAX;
    e.item_begin = item;
    e.walk_begin = s.walk_begin;
    item += s.walks;
  }
  P.n_items = item;
  auto up16 = [](int b) { return (b + 15) & ~15; };
  SlabPlan& sp = P.slab;
  sp.off_ctl = up16(4 * kBitWords);
  sp.off_S = sp.off_ctl + up16((int)sizeof(WalkCtl));
  sp.off_tab = sp.off_S + up16(sn);
  sp.off_bloom = sp.off_tab + up16(tab);
  sp.bytes = sp.off_bloom + up16(std::max(kScratch, (1 << bloom_log2) / 8));
}

// Lets the kernel have its shared memory and sizes the persistent grid.  A block is one SM's walks: as many
// warps as its registers and shared memory hold, fewer when the launch has fewer walks than that per SM (a
// few walks then spread over all SMs instead of filling some).  A batch times that number against fewer (trial_warps).
static int plan_launch(labs_ctx* ctx, const WalkParams& P, int requested_warps, bool biased, Launch* ln) {
  int warps = walk_block_threads(ln->mode, ln->ns, ln->nu) / 32;
  if (requested_warps > 0) {
    warps = requested_warps;
  } else {
    const int64_t per_sm = (P.n_items + ctx->num_sms - 1) / ctx->num_sms;
    warps = (int)std::max<int64_t>(1, std::min<int64_t>(warps, per_sm));
  }
  while (warps > 1 && (size_t)P.slab.bytes * warps > ctx->smem_optin) warps--;
  ln->warps = warps;
  ln->smem = (size_t)P.slab.bytes * warps;
  WalkKernel kern = walk_fn(*ln, biased);
  if (allow_smem(ctx, kern) != cudaSuccess) return LABS_ERR_CUDA;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * warps, ln->smem) != cudaSuccess || per_sm < 1)
    return LABS_ERR_CUDA;
  const long long b = (long long)per_sm * ctx->num_sms, need = (P.n_items + warps - 1) / warps;
  ln->blocks = std::max(1ll, std::min(b, need));
  return LABS_OK;
}

static int run_walks(const WalkParams& P, const Launch& ln, cudaStream_t st) {
  walk_fn(ln, P.bias != nullptr)<<<(unsigned)ln.blocks, 32 * ln.warps, ln.smem, st>>>(P);
  return cuda_status(cudaGetLastError());
}

static int run_init(const WalkParams& P, cudaStream_t st) {
  walk_init_kernel<<<(unsigned)P.n_len, 128, 0, st>>>(P, const_cast<uint64_t*>(P.zpair));
  return cuda_status(cudaGetLastError());
}

static void base_params(WalkParams& P, int R, int bloom_log2, int bloom_k, int p, int n_prefix, int64_t flip_budget,
                        uint64_t seed, int32_t E_target, const uint64_t* prefixes, labs_candidate* out,
                        int64_t* walk_stats, labs_walk_stats* stats, unsigned long long* counter, uint64_t* zpair) {
  P.R = R;
  P.bloom_log2 = bloom_log2;
  P.bloom_k = bloom_k;
  P.prefix_words = p > 0 ? (p + 63) / 64 : 1;
  P.n_prefix = n_prefix;
  P.flip_budget = flip_budget;
  P.seed = seed;
  P.E_target = E_target;
  P.prefixes = prefixes;
  P.out = out;
  P.walk_stats = walk_stats;
  P.stats = stats;
  P.counter = counter;
  P.zpair = zpair;
  P.E_thr_dev = nullptr;
}

// Bytes of the fingerprint changes of a launch's lengths.
static size_t zpair_bytes(size_t n_len) { return sizeof(uint64_t) * kMaxL * n_len; }

}  // namespace

int launch_sample_threshold(labs_ctx* ctx, int L, int skew, int p, const uint64_t* prefixes, int n_prefix,
                            int prefix_words, uint64_t seed, int64_t n_samples, int64_t rank, int32_t* E_thr_out,
                            int32_t* E_samples, cudaStream_t st) {
  int32_t* Es = E_samples;
  if (!Es) {
    Es = static_cast<int32_t*>(ws_get(ctx, kWsThreshSamples, sizeof(int32_t) * (size_t)n_samples));
    if (!Es) return LABS_ERR_NOMEM;
  }
  unsigned* hist = static_cast<unsigned*>(ws_get(ctx, kWsThreshHist, sizeof(unsigned) * 2 * kHistBins + 64));
  if (!hist) return LABS_ERR_NOMEM;
  long long* sel = reinterpret_cast<long long*>(hist + 2 * kHistBins);
  return issue_threshold(ctx->num_sms, L, skew, p, prefixes, n_prefix, prefix_words, seed, n_samples, rank, E_thr_out,
                         Es, hist, sel, st);
}

int launch_skew_search(labs_ctx* ctx, const labs_walk_cfg* cfg, const uint64_t* prefixes, int n_prefix,
                       labs_candidate* out, int64_t* walk_stats, labs_walk_stats* stats, cudaStream_t st) {
  return launch_chunked_search(ctx, cfg, nullptr, 0.f, 0, prefixes, n_prefix, out, walk_stats, stats, nullptr, nullptr,
                               nullptr, st);
}

// ---------------------------------------------------------------------------------------------
// Walks of one length.  Without a network they run in one launch, which also writes the logs of a chunked
// run (chunk > 0): a walk does not depend on the others, so its state at a chunk's beginning is logged as it
// passes it.  With a network the walks run `chunk` accepted flips per launch and are saved in between, and
// the network scores every walk's current state before each chunk.
// ---------------------------------------------------------------------------------------------
int launch_chunked_search(labs_ctx* ctx, const labs_walk_cfg* cfg, labs_policy* policy, float lambda, int chunk,
                          const uint64_t* prefixes, int n_prefix, labs_candidate* out, int64_t* walk_stats,
                          labs_walk_stats* stats, float* logits_log, uint64_t* state_log, int32_t* move_log,
                          cudaStream_t st) {
  std::vector<LenSpec> lens{{cfg->L, cfg->skew, cfg->p, cfg->T_i, cfg->n_walks, cfg->walk_begin}};
  if (!accepted(lens, cfg->tile_m, cfg->lanes_per_walk, cfg->R, cfg->warps_per_cta)) return LABS_ERR_INVALID_ARG;
  std::unique_ptr<WalkParams> P(new (std::nothrow) WalkParams());
  char* w = static_cast<char*>(ws_get(ctx, kWsWalkCounters, 256));
  uint64_t* zpair = static_cast<uint64_t*>(ws_get(ctx, kWsZpair, zpair_bytes(1)));
  if (!P || !w || !zpair) return LABS_ERR_NOMEM;
  unsigned long long* counter = reinterpret_cast<unsigned long long*>(w);
  base_params(*P, cfg->R, cfg->bloom_log2, cfg->bloom_k, cfg->p, n_prefix, cfg->flip_budget, cfg->seed, cfg->E_target,
              prefixes, out, walk_stats, stats, counter, zpair);
  Launch ln;
  fill_params(*P, lens, cfg->bloom_log2, &ln);
  const long long n = cfg->n_walks;
  const int L = cfg->L, W = (L + 63) / 64;
  const long long n_chunks = chunk > 0 ? (cfg->flip_budget + chunk - 1) / chunk : 0;
  unsigned char* state = nullptr;
  uint64_t* seqbuf = nullptr;
  // the kernel logs whole words: a log that is not aligned for them is written in workspace and copied
  uint64_t* log = state_log;
  const size_t log_bytes = 8 * (size_t)n_chunks * (size_t)n * W;
  if (!policy && reinterpret_cast<uintptr_t>(state_log) & 7u) {
    log = static_cast<uint64_t*>(ws_get(ctx, kWsChunkIo, log_bytes));
    if (!log) return LABS_ERR_NOMEM;
  }
  float* logits = nullptr;
  if (policy) {
    P->state_stride = P->slab.bytes + 128 * walk_slots(ln.mode, ln.ns, ln.nu);
    state = static_cast<unsigned char*>(ws_get(ctx, kWsChunkState, (size_t)P->state_stride * (size_t)n));
    char* io = static_cast<char*>(ws_get(ctx, kWsChunkIo, (size_t)n * (8 * W + 4 * L) + 256));
    if (!state || !io) return LABS_ERR_NOMEM;
    seqbuf = reinterpret_cast<uint64_t*>(io);
    logits = reinterpret_cast<float*>(io + (((size_t)n * 8 * W + 255) & ~size_t(255)));
  }
  int32_t* thr = reinterpret_cast<int32_t*>(w + 64);
  int s = LABS_OK;
  if (cfg->E_thr_dev) {
    P->E_thr_dev = cfg->E_thr_dev;
  } else if (cfg->E_thr == LABS_AUTO_THRESHOLD) {
    s = launch_sample_threshold(ctx, cfg->L, cfg->skew, cfg->p, prefixes, n_prefix, P->prefix_words, cfg->seed,
                                cfg->n_thresh_samples, cfg->thresh_rank, thr, nullptr, st);
    P->E_thr_dev = thr;
  } else {
    P->len[0].E_thr_value = cfg->E_thr;
  }
  Launch biased = ln;
  if (s == LABS_OK) s = plan_launch(ctx, *P, cfg->warps_per_cta, false, &ln);
  if (s == LABS_OK && policy) s = plan_launch(ctx, *P, cfg->warps_per_cta, true, &biased);
  if (s == LABS_OK) s = run_init(*P, st);
  if (s != LABS_OK) return s;
  if (!policy) {
    P->log_chunk = state_log || move_log ? chunk : 0;
    P->state_log = log;
    P->move_log = move_log;
    s = n > 0 ? run_walks(*P, ln, st) : LABS_OK;
    if (s == LABS_OK && log != state_log && log_bytes)
      s = cuda_status(cudaMemcpyAsync(state_log, log, log_bytes, cudaMemcpyDeviceToDevice, st));
    return s;
  }
  P->state = state;
  P->seq_out = seqbuf;
  P->chunk = -1;  // set-up launch: every walk's first state
  if (n > 0) s = run_walks(*P, ln, st);
  P->chunk = chunk;
  P->log_chunk = move_log ? chunk : 0;
  P->bias = logits;
  P->lambda = lambda;
  for (long long c = 0; c < n_chunks && s == LABS_OK && n > 0; c++) {
    s = labs_policy_forward(policy, seqbuf, n, logits, st);
    if (s != LABS_OK) break;
    if ((logits_log && cudaMemcpyAsync(logits_log + (size_t)c * n * L, logits, sizeof(float) * (size_t)n * L,
                                       cudaMemcpyDeviceToDevice, st) != cudaSuccess) ||
        (state_log && cudaMemcpyAsync(state_log + (size_t)c * n * W, seqbuf, 8 * (size_t)n * W,
                                      cudaMemcpyDeviceToDevice, st) != cudaSuccess) ||
        cudaMemsetAsync(counter, 0, sizeof(unsigned long long), st) != cudaSuccess) {
      s = LABS_ERR_CUDA;
      break;
    }
    P->move_log = move_log ? move_log + (size_t)c * n * 2 : nullptr;
    s = run_walks(*P, biased, st);
  }
  // the network's tensor-core waits: a failure makes the logits of that chunk invalid
  const int ps = labs_policy_sync_status(policy, st);
  return s == LABS_OK ? ps : s;
}

// ---------------------------------------------------------------------------------------------
// Batched mixed-length search: every length's sieve bound, then one persistent walk launch over all
// (length, walk) items; the sequence is captured once into a CUDA graph and replayed.
// ---------------------------------------------------------------------------------------------
namespace {

uint64_t mix_key(uint64_t h, uint64_t v) { return sm64_at(h ^ v, 0x5EED); }

// Issues the whole batched step on `st`: stream work only (capturable).
int issue_batch(labs_ctx* ctx, const labs_batch_cfg* cfg, const std::vector<LenSpec>& lens, const WalkParams& P,
                const Launch& ln, int32_t* thr, cudaStream_t st) {
  int s = LABS_OK;
  for (size_t i = 0; i < lens.size() && s == LABS_OK; i++)
    s = launch_sample_threshold(ctx, lens[i].L, lens[i].skew, lens[i].p, P.prefixes, P.n_prefix, P.prefix_words,
                                cfg->seed, cfg->n_thresh_samples, cfg->thresh_rank, thr + i, nullptr, st);
  if (s == LABS_OK) s = run_init(P, st);
  if (s == LABS_OK && P.n_items > 0) s = run_walks(P, ln, st);
  return s;
}

// Whether `st` is being captured (or cannot be asked for it now).
bool capturing(cudaStream_t st) {
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &status) == cudaSuccess) return status != cudaStreamCaptureStatusNone;
  cudaGetLastError();
  return true;
}

// Walks per block of a batch by a timed trial: the number that plan_launch chose against the next two multiples of
// four below (an SM has four schedulers), each with a proportional part of the walks that fills its blocks kTrialRounds
// times, for kTrialFlips flips, the sieve closed.  How many walks an SM should hold depends on the lengths in the
// launch: L = 450 .. 527, 42,000 walks x 500 flips: 33.4 ms with 23 (as many as fit), 30.7 with 20, 33.1 with 16; L =
// 500 .. 576: 38.2 with 22, 39.6 and 37.2; L = 64 .. 141: 13.6 with 32, 14.8 with 24.  Slots a lane need no trial: the
// smallest number that holds the lengths is the fastest (one step more: 8 to 100% slower).  Candidates of the trial go
// to `out`, which the search then overwrites.
constexpr int kTrialFlips = 256, kTrialRounds = 3;
int trial_warps(labs_ctx* ctx, const labs_batch_cfg* cfg, const std::vector<LenSpec>& lens, const WalkParams& P,
                const Launch& ln, cudaStream_t st, int* warps) {
  std::unique_ptr<WalkParams> Q(new (std::nothrow) WalkParams(P));
  if (!Q) return LABS_ERR_NOMEM;
  Q->flip_budget = std::min<int64_t>(cfg->flip_budget, kTrialFlips);
  Q->walk_stats = nullptr;
  Q->E_thr_dev = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    return LABS_ERR_CUDA;
  }
  double best = 0;
  int s = LABS_OK;
  for (int turn = -1; turn < 3 && s == LABS_OK; turn++) {  // turn -1: untimed
    const int w = turn < 1 ? ln.warps : (ln.warps - 1) / 4 * 4 - 4 * (turn - 1);
    if (w < 4) break;
    std::vector<LenSpec> part = lens;
    const double share = std::min(1.0, (double)kTrialRounds * w * ctx->num_sms / (double)P.n_items);
    for (LenSpec& e : part) e.walks = e.walks > 0 ? std::max<int64_t>(1, (int64_t)(share * (double)e.walks)) : 0;
    Launch q;
    fill_params(*Q, part, cfg->bloom_log2, &q);
    for (int i = 0; i < Q->n_len; i++) Q->len[i].E_thr_value = INT32_MIN;
    s = plan_launch(ctx, *Q, w, false, &q);
    if (s == LABS_OK) s = run_init(*Q, st);
    if (s == LABS_OK && cudaEventRecord(e0, st) != cudaSuccess) s = LABS_ERR_CUDA;
    if (s == LABS_OK) s = run_walks(*Q, q, st);
    float ms = 0.f;
    if (s == LABS_OK && (cudaEventRecord(e1, st) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
                         cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess))
      s = LABS_ERR_CUDA;
    if (s != LABS_OK || turn < 0) continue;
    const double per_walk = (double)ms / (double)Q->n_items;
    if (turn == 0 || per_walk < 0.98 * best) {  // fewer walks only where that is clearly faster
      best = per_walk;
      *warps = w;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return s;
}

}  // namespace

int launch_batched_search(labs_ctx* ctx, const labs_batch_cfg* cfg, const int32_t* lengths, const int64_t* walks,
                          const uint64_t* prefixes, int n_prefix, labs_candidate* out, int64_t* walk_stats,
                          int32_t* E_thr_out, labs_walk_stats* stats, cudaStream_t st) {
  std::vector<LenSpec> lens;
  for (int i = 0; i < cfg->n_len; i++) {
    const int L = lengths[i];
    const int skew = L & 1;
    lens.push_back({L, skew, skew ? cfg->p : 0, cfg->T_i, walks[i], 0});
  }
  if (!accepted(lens, cfg->tile_m, 0, cfg->R, cfg->warps_per_cta)) return LABS_ERR_INVALID_ARG;
  // workspace first (nothing below may allocate once a capture has begun)
  char* w = static_cast<char*>(ws_get(ctx, kWsWalkCounters, 256));
  int32_t* thr = E_thr_out ? E_thr_out : static_cast<int32_t*>(ws_get(ctx, kWsBatchThresholds, sizeof(int32_t) * kMaxLens));
  uint64_t* zpair = static_cast<uint64_t*>(ws_get(ctx, kWsZpair, zpair_bytes(kMaxLens)));
  std::unique_ptr<WalkParams> P(new (std::nothrow) WalkParams());
  if (!w || !thr || !zpair || !P) return LABS_ERR_NOMEM;
  if (!ws_get(ctx, kWsThreshSamples, sizeof(int32_t) * (size_t)cfg->n_thresh_samples) ||
      !ws_get(ctx, kWsThreshHist, sizeof(unsigned) * 2 * kHistBins + 64))
    return LABS_ERR_NOMEM;
  unsigned long long* counter = reinterpret_cast<unsigned long long*>(w);
  base_params(*P, cfg->R, cfg->bloom_log2, cfg->bloom_k, cfg->p, n_prefix, cfg->flip_budget, cfg->seed, cfg->E_target,
              prefixes, out, walk_stats, stats, counter, zpair);
  Launch ln;
  fill_params(*P, lens, cfg->bloom_log2, &ln);
  P->E_thr_dev = thr;
  // kernel attributes and grid size before any capture
  int s = plan_launch(ctx, *P, cfg->warps_per_cta, false, &ln);
  if (s != LABS_OK) return s;
  // (a search shorter than its trial is left to plan_launch)
  const double trial_flips = 4.0 * kTrialRounds * ln.warps * ctx->num_sms * kTrialFlips;
  if (cfg->warps_per_cta == 0 && ln.warps >= 8 && (double)P->n_items * (double)cfg->flip_budget >= trial_flips &&
      !capturing(st)) {
    uint64_t tkey = mix_key((uint64_t)ctx->num_sms,
                            ((uint64_t)cfg->bloom_log2 << 32) ^ ((uint64_t)cfg->bloom_k << 16) ^ (uint64_t)cfg->R);
    for (const LenSpec& e : lens) tkey = mix_key(tkey, ((uint64_t)e.L << 50) ^ ((uint64_t)e.p << 40) ^ (uint64_t)e.walks);
    int warps = 0;
    for (int i = 0; i < std::min(ctx->n_tuned, kMaxTuned); i++)
      if (ctx->tuned_key[i] == tkey) warps = ctx->tuned_warps[i];
    if (!warps) {
      s = trial_warps(ctx, cfg, lens, *P, ln, st, &warps);
      if (s != LABS_OK) return s;
      ctx->tuned_key[ctx->n_tuned % kMaxTuned] = tkey;
      ctx->tuned_warps[ctx->n_tuned % kMaxTuned] = warps;
      ctx->n_tuned++;
    }
    s = plan_launch(ctx, *P, warps, false, &ln);
    if (s != LABS_OK) return s;
  }
  if (!cfg->use_graph) return issue_batch(ctx, cfg, lens, *P, ln, thr, st);

  // ---- CUDA graph: capture once per (configuration, buffers), replay afterwards
  uint64_t gkey = (uint64_t)ctx->num_sms;
  for (const LenSpec& e : lens) gkey = mix_key(gkey, ((uint64_t)e.L << 40) ^ (uint64_t)e.walks);
  gkey = mix_key(gkey, ((uint64_t)(100 * ln.ns + ln.nu) << 32) ^ ((uint64_t)ln.mode << 16) ^ (uint64_t)ln.warps);
  gkey = mix_key(gkey, (uint64_t)cfg->flip_budget ^ ((uint64_t)cfg->R << 48));
  gkey = mix_key(gkey, cfg->seed);
  gkey = mix_key(gkey, ((uint64_t)cfg->p << 32) ^ ((uint64_t)cfg->bloom_log2 << 16) ^ (uint64_t)cfg->bloom_k);
  gkey = mix_key(gkey, ((uint64_t)cfg->T_i << 32) ^ (uint32_t)cfg->E_target);
  gkey = mix_key(gkey, (uint64_t)cfg->n_thresh_samples ^ ((uint64_t)cfg->thresh_rank << 40));
  const void* bufs[] = {prefixes, out, walk_stats, thr, stats, w, zpair, ctx->ws[kWsThreshSamples], ctx->ws[kWsThreshHist]};
  for (const void* ptr : bufs) gkey = mix_key(gkey, (uint64_t)(uintptr_t)ptr);
  gkey = mix_key(gkey, (uint64_t)n_prefix ^ ((uint64_t)ln.blocks << 32));
  if (!ctx->graph_exec || ctx->graph_key != gkey) {
    if (!ctx->capture_stream && cudaStreamCreateWithFlags(&ctx->capture_stream, cudaStreamNonBlocking) != cudaSuccess)
      return LABS_ERR_CUDA;
    if (cudaStreamBeginCapture(ctx->capture_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
      return LABS_ERR_CUDA;
    s = issue_batch(ctx, cfg, lens, *P, ln, thr, ctx->capture_stream);
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(ctx->capture_stream, &g);
    if (s != LABS_OK) {
      if (g) cudaGraphDestroy(g);
      return s;
    }
    if (e != cudaSuccess) return LABS_ERR_CUDA;
    cudaGraphExec_t ex = nullptr;
    e = cudaGraphInstantiate(&ex, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return LABS_ERR_CUDA;
    if (ctx->graph_exec) cudaGraphExecDestroy(ctx->graph_exec);
    ctx->graph_exec = ex;
    ctx->graph_key = gkey;
  }
  return cuda_status(cudaGraphLaunch(ctx->graph_exec, st));
}

}  // namespace labsg

// ---------------------------------------------------------------------------------------------
// Sieve bound without any allocation (labs_sample_threshold_noalloc).
//
// Some callers cannot allocate device memory while they run this library.  An application whose
// allocator owns every device byte (a framework memory pool, a fixed arena sized at start-up) forbids
// direct cudaMalloc; latency-sensitive callers avoid it because it can synchronise the device; and no
// library context (which grows workspace on demand) may exist at all.  For them this entry point runs the
// same kernels as labs_sample_threshold with its scratch -- the sampled energies, both histograms and the
// selected bin -- in one file-scope device array of fixed size, loaded with the library.
// ---------------------------------------------------------------------------------------------
namespace labsg {
namespace {

constexpr int64_t kNoAllocMaxSamples = int64_t(1) << 20;  // 1,048,576 samples (>= the 10^6 sieve sample)
constexpr size_t kNoAllocSamplesBytes = sizeof(int32_t) * (size_t)kNoAllocMaxSamples;
constexpr size_t kNoAllocHistBytes = sizeof(unsigned) * 2 * kHistBins;
constexpr size_t kNoAllocBytes = kNoAllocSamplesBytes + kNoAllocHistBytes + 256;  // + the selected bin

// Every GPU that loads the library holds these 4.26 MB until the process exits.  All calls share it.
static __device__ __align__(256) unsigned char g_threshold_scratch[kNoAllocBytes];

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_scratch_mu;
void* g_scratch_addr[kNoAllocMaxDevices];  // device address of g_threshold_scratch per device

// Set-up, once per device, with that device current: the host-side name of the array is not a device
// address, so ask the runtime for it.
int threshold_scratch(int device, unsigned char** out) {
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (!g_scratch_addr[device]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_threshold_scratch) != cudaSuccess || !p) return LABS_ERR_CUDA;
    g_scratch_addr[device] = p;
  }
  *out = static_cast<unsigned char*>(g_scratch_addr[device]);
  return LABS_OK;
}

}  // namespace
}  // namespace labsg

extern "C" int labs_sample_threshold_noalloc(int L, int skew, int p, const uint64_t* prefixes, int n_prefix,
                                             uint64_t seed, int64_t n_samples, int64_t rank, int32_t* E_thr_out,
                                             void* stream) {
  using namespace labsg;
  if (check_walk_shape(L, skew, p, n_prefix, prefixes) != LABS_OK) return LABS_ERR_INVALID_ARG;
  if (!E_thr_out || (reinterpret_cast<uintptr_t>(E_thr_out) & 3u)) return LABS_ERR_INVALID_ARG;
  if (n_samples < 1 || rank < 0 || rank >= n_samples) return LABS_ERR_INVALID_ARG;
  if (n_samples > kNoAllocMaxSamples) return LABS_ERR_CAPACITY;  // beyond the fixed scratch
  int device = 0, sms = 0;
  if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= kNoAllocMaxDevices) return LABS_ERR_CUDA;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || sms < 1)
    return LABS_ERR_CUDA;
  unsigned char* base = nullptr;
  int s = threshold_scratch(device, &base);
  if (s != LABS_OK) return s;
  int32_t* Es = reinterpret_cast<int32_t*>(base);
  unsigned* hist = reinterpret_cast<unsigned*>(base + kNoAllocSamplesBytes);
  long long* sel = reinterpret_cast<long long*>(base + kNoAllocSamplesBytes + kNoAllocHistBytes);
  cudaStream_t st = (cudaStream_t)stream;
  const int prefix_words = p > 0 ? (p + 63) / 64 : 1;
  // (the histograms keep the previous call's counts and are cleared first)
  return issue_threshold(sms, L, skew, p, prefixes, n_prefix, prefix_words, seed, n_samples, rank, E_thr_out, Es, hist,
                         sel, st);
}

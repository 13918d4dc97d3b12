// pq_indep.cu -- step 2 with one independent priority queue per candidate (labs_pq_independent): the
// paper's own parallelisation of Algorithm 2 (every candidate refined on its own, Section 3), with the
// queue unbounded as in the listing (nothing is evicted) and B = 1 pops per step.
//
// GB300 mapping.  One warp per candidate; a candidate's state lives in HBM:
//   arena  -- every pushed node as a 16-byte record (E, link, fp); the survivors of one pop are appended
//             as one run, in no particular order;
//   runs   -- a 32-ary heap over the runs keyed by each run's smallest (E, fp): its top is the queue
//             minimum.  A pop takes that node out of its run (the run's last node fills the gap), finds
//             the run's new smallest by one warp-wide rescan (at most L + 2 T_r records) and sifts down, the
//             32 children of a level read and ranked by the warp at once; a new run is one sift-up.  Keys
//             (E, fp) are distinct in a queue (the visited set admits a sequence once), so the pop order is
//             that of the sequential definition;
//   pivots -- the sequence of every popped node (a node is stored as its pivot and column, and is made
//             into a sequence only when popped);
//   H      -- the candidate's visited set (open addressing, cleared per candidate), where it is needed: without
//             rotations every node ever pushed is the seed or a neighbour of a popped pivot, so a neighbour p^i
//             of the pivot p was visited exactly if some earlier pivot differs from p in i and one other
//             position, or in i alone (the seed is the first pivot).  Up to kPairPops pops the pivots
//             themselves are compared -- a few hundred coalesced words a pop instead of L inserts at random
//             places of a set that lies in DRAM.
// A pop forms its correlations and every neighbour's sum from the sequence alone (scan_mma.cuh: some 2,000 warp
// instructions, less than keeping tables per pivot would move); each neighbour is one insert-if-absent into H, a
// survivor being one whose key was absent.  With T_r > 0 the pivot's 2 T_r rotations follow the flips (a
// rotation equal to a flip child or to an earlier rotation finds its key in H and is dropped, as the ordered
// dedup keeps the smaller column).  Memory per resident warp is about max_expansions x (L + 2 T_r) x 16 B, and
// 2^H_log2 x 8 B where H is needed: HBM capacity, not bandwidth, is what this design spends.
#include <algorithm>

#include "labs_internal.h"
#include "scan_mma.cuh"

namespace labsg {
namespace {

constexpr int kIWarps = 4;
constexpr uint64_t kEmpty = ~0ull;
constexpr int kProbeLimit = 1 << 20;
constexpr int kMaxTr = 64;  // rotations per side (the library's bound on T_r)
// Pops up to which the pivots are compared pairwise: n / 2 pivots of 64 bytes a pop against L random 32-byte
// sectors read and written, and a set that is cleared first.
constexpr long long kPairPops = 1024;

struct Node {  // one queue record: 16 bytes
  int32_t E;
  int32_t link;  // pivot * 1024 + column (column < L: flip, else rotation column - L); -1: the seed
  uint64_t fp;
};

struct RunHead {  // heap element: the run's smallest key, where it is, and the run's live range
  int32_t E;
  int32_t cur;  // arena index of the smallest node
  uint64_t fp;
  int32_t end;    // live nodes are [begin, end)
  int32_t begin;
};

struct IndepArgs {
  int L, W, Tr, width, H_log2;
  long long max_exp, T_u;
  long long arena_cap, heap_cap;
  long long n;
  const uint64_t* seeds;
  uint64_t* best_seqs;
  int32_t* best_E;
  labs_pq_stats* stats;
  // per-slot workspaces (slot = resident warp)
  Node* arena;
  RunHead* heap;
  uint64_t* pivots;  // [W][max_exp] a slot
  uint64_t* H;
  const uint64_t* ztab;
  unsigned long long* counter;
};

__device__ __forceinline__ bool kless(int Ea, uint64_t fa, int Eb, uint64_t fb) {
  return Ea < Eb || (Ea == Eb && fa < fb);
}

// Visited set of one slot (open addressing, linear probing); *err set on an exhausted probe sequence.
// The first compare-and-swap of several keys is issued by the caller, all at once, so that their
// latencies overlap; the _from forms continue a key's probe sequence after a first slot that held
// another key.
__device__ __forceinline__ uint64_t hs_home(uint64_t fp, int log2) { return (fp * kGamma) >> (64 - log2); }
__device__ __forceinline__ void hs_insert_from(uint64_t* H, int log2, uint64_t fp, uint64_t s, int* err) {
  const uint64_t mask = (1ull << log2) - 1;
  for (int it = 1; it < kProbeLimit; it++) {
    s = (s + 1) & mask;
    const unsigned long long old =
        atomicCAS(reinterpret_cast<unsigned long long*>(&H[s]), (unsigned long long)kEmpty, fp);
    if (old == kEmpty || old == fp) return;
  }
  *err = 1;
}
__device__ __forceinline__ void hs_insert(uint64_t* H, int log2, uint64_t fp, int* err) {
  const uint64_t s = hs_home(fp, log2);
  const unsigned long long old = atomicCAS(reinterpret_cast<unsigned long long*>(&H[s]), (unsigned long long)kEmpty, fp);
  if (old == kEmpty || old == fp) return;
  hs_insert_from(H, log2, fp, s, err);
}
// Insert-if-absent, continuing after slot s (whose key was another one): true when fp was inserted.
__device__ __forceinline__ bool hs_add_from(uint64_t* H, int log2, uint64_t fp, uint64_t s, int* err) {
  const uint64_t mask = (1ull << log2) - 1;
  for (int it = 1; it < kProbeLimit; it++) {
    s = (s + 1) & mask;
    const unsigned long long old =
        atomicCAS(reinterpret_cast<unsigned long long*>(&H[s]), (unsigned long long)kEmpty, fp);
    if (old == kEmpty) return true;
    if (old == fp) return false;
  }
  *err = 1;
  return false;
}
// Insert-if-absent (the key ~0 by the flag has_empty): true when fp was inserted.
__device__ __forceinline__ bool hs_add(uint64_t* H, int log2, uint64_t fp, bool& has_empty, int* err) {
  if (fp == kEmpty) {
    const bool fresh = !has_empty;
    has_empty = true;
    return fresh;
  }
  const uint64_t s = hs_home(fp, log2);
  const unsigned long long old = atomicCAS(reinterpret_cast<unsigned long long*>(&H[s]), (unsigned long long)kEmpty, fp);
  if (old == kEmpty) return true;
  if (old == fp) return false;
  return hs_add_from(H, log2, fp, s, err);
}

// Left shift of rotation code c: c < Tr moves the first c + 1 elements to the end, c >= Tr the last
// c - Tr + 1 to the start.
__device__ __forceinline__ int rshift(int L, int Tr, int c) {
  const int r = c < Tr ? c + 1 : L - ((c - Tr + 1) % L);
  return r % L;
}

// bits (32-bit words in shared memory) of src with position col + 1 flipped.
__device__ __forceinline__ void flip_bits(const uint32_t* src, int col, uint32_t* dst) {
  const int lane = lane_id();
  if (lane < kBitWords) dst[lane] = src[lane] ^ (lane == (col >> 5) ? 1u << (col & 31) : 0u);
  __syncwarp();
}

template <int NW>
__device__ __forceinline__ void rotate_bits(const uint32_t* src, int L, int r, uint32_t* dst) {
  const uint32_t y = rotated_word<NW>(src, L, r);
  if (lane_id() < kBitWords) dst[lane_id()] = y;
  __syncwarp();
}

// (words of a sequence `stride` apart)
__device__ __forceinline__ void words_to_bits(const uint64_t* src, int L, uint32_t* dst, long long stride = 1) {
  const int lane = lane_id();
  if (lane < kBitWords) {
    const int W32 = (L + 31) >> 5;
    uint32_t v = 0;
    if (lane < W32) {
      const uint64_t x = src[(lane >> 1) * stride];
      v = (lane & 1) ? (uint32_t)(x >> 32) : (uint32_t)x;
      const int rem = L - 32 * lane;
      if (rem < 32) v &= (1u << rem) - 1u;
    }
    dst[lane] = v;
  }
  __syncwarp();
}

__device__ __forceinline__ void bits_to_words(const uint32_t* src, int L, uint64_t* dst, long long stride = 1) {
  const int lane = lane_id();
  if (lane < ((L + 63) >> 6)) dst[lane * stride] = (uint64_t)src[2 * lane] | ((uint64_t)src[2 * lane + 1] << 32);
}

__device__ __forceinline__ uint64_t fp_bits(const uint32_t* bits, int L, const uint64_t* ztab) {
  uint64_t h = 0;
  for (int i = lane_id(); i < L; i += 32)
    if (!((bits[i >> 5] >> (i & 31)) & 1u)) h ^= ztab[i];
  return warp_xor_u64(h);
}

// The warp's smallest (E, fp) over the lanes' candidates (bi >= 0; keys distinct) and its index, on every
// lane.
__device__ __forceinline__ void warp_argmin(int bE, uint64_t bf, int bi, int& E, uint64_t& fp, int& idx) {
  const int mE = __reduce_min_sync(kFull, bE);
  const unsigned mhi = __reduce_min_sync(kFull, bE == mE ? (unsigned)(bf >> 32) : 0xffffffffu);
  const bool on = bE == mE && (unsigned)(bf >> 32) == mhi;
  const unsigned mlo = __reduce_min_sync(kFull, on ? (unsigned)bf : 0xffffffffu);
  const unsigned who = __ballot_sync(kFull, on && (unsigned)bf == mlo && bi >= 0);
  E = mE;
  fp = ((uint64_t)mhi << 32) | mlo;
  idx = __shfl_sync(kFull, bi, __ffs(who) - 1);
}

// Smallest (E, fp) of arena nodes [begin, end) (non-empty, keys distinct) and its index, on every lane; eight
// records a lane in flight.
__device__ __forceinline__ void run_min(const Node* arena, int begin, int end, int& E, uint64_t& fp, int& idx) {
  int bE = INT32_MAX, bi = -1;
  uint64_t bf = ~0ull;
  for (int i0 = begin + lane_id(); i0 - lane_id() < end; i0 += 256) {
    int4 x[8];
#pragma unroll
    for (int j = 0; j < 8; j++)
      x[j] = i0 + 32 * j < end ? reinterpret_cast<const int4*>(arena)[i0 + 32 * j] : make_int4(INT32_MAX, 0, -1, -1);
#pragma unroll
    for (int j = 0; j < 8; j++) {
      const uint64_t f = ((uint64_t)(uint32_t)x[j].w << 32) | (uint32_t)x[j].z;
      if (kless(x[j].x, f, bE, bf)) {
        bE = x[j].x;
        bf = f;
        bi = i0 + 32 * j;
      }
    }
  }
  warp_argmin(bE, bf, bi, E, fp, idx);
}

// Shared memory of one warp, in 32-bit words from its slab's start.
struct IndepPlan {
  ScanMmaPlan mma;
  int q, x, v, words;
};
constexpr int kInP = 0, kInC = 24, kInClass = 48, kInRev = kInClass + 2 * kClassWords, kInTables = kInRev + 2 * kClassWords;

// Seven blocks an SM hold 28 candidates (72 registers a thread, 7.7 KB of slab a warp at L = 451), 4,256 on the chip.
// Beyond 512 positions the slab leaves room for six blocks (80 registers), 3,648 candidates.  V_IN_Q (compiled there): V is formed
// first, where the table of q comes to lie, and a lane keeps its outputs' values in registers, so that seven blocks
// fit again; a pop takes longer (more registers saved).  The 72 registers cost spills (92 bytes a thread at L = 451, 232
// with a visited set, 212 to 400 in the V_IN_Q forms); with six blocks of 80 registers, 4,096 candidates of L = 451 x 256
// pops take 11.3 ms, with seven 10.5 ms.
template <int NW, bool PAIRS, bool V_IN_Q>
__global__ void __launch_bounds__(32 * kIWarps, NW > 16 && !V_IN_Q ? 6 : 7) pq_indep_kernel(IndepArgs a, IndepPlan ip) {
  constexpr int NT = (NW + 3) / 4;
  extern __shared__ __align__(16) uint32_t in_smem[];
  uint32_t* slab = in_smem + (size_t)(threadIdx.x >> 5) * ip.words;
  uint32_t *pbits = slab + kInP, *cbits = slab + kInC, *cw = slab + kInClass, *rw = slab + kInRev;
  uint32_t *qt = slab + ip.q, *xt = slab + ip.x;
  // v[1 .. L]; in q: its elements at distances -(L - 1) .. 0, all of which but q(0) = 0 are written for every pivot
  int16_t* v = V_IN_Q ? reinterpret_cast<int16_t*>(qt) + ip.mma.off - a.L : reinterpret_cast<int16_t*>(slab + ip.v);
  const int lane = lane_id();
  const int slot = blockIdx.x * kIWarps + (threadIdx.x >> 5);
  Node* const arena = a.arena + slot * a.arena_cap;
  RunHead* const heap = a.heap + slot * a.heap_cap;
  uint64_t* const pivots = a.pivots + slot * a.max_exp * a.W;
  uint64_t* const H = PAIRS ? nullptr : a.H + ((long long)slot << a.H_log2);
  const long long hslots = 1ll << a.H_log2;
  const uint32_t* const xs[1] = {xt};
  for (int i = lane; i < ip.words; i += 32) slab[i] = 0u;
  __syncwarp();

  while (true) {
    unsigned long long cand = 0;
    if (lane == 0) cand = atomicAdd(a.counter, 1ull);
    cand = __shfl_sync(kFull, cand, 0);
    if ((long long)cand >= a.n) break;
    int err = 0;
    // ---- reset the visited set, seed the queue
    if (!PAIRS)
      for (long long t = lane; t < hslots / 2; t += 32) reinterpret_cast<ulonglong2*>(H)[t] = make_ulonglong2(kEmpty, kEmpty);
    __threadfence_block();
    __syncwarp();
    words_to_bits(a.seeds + cand * a.W, a.L, pbits);
    int bestE = energy_words<NW>(pbits, a.L);
    uint64_t bestfp = fp_bits(pbits, a.L, a.ztab);
    bool has_empty = bestfp == kEmpty;
    if (lane == 0) {
      if (!PAIRS && !has_empty) hs_insert(H, a.H_log2, bestfp, &err);
      arena[0] = Node{bestE, -1, bestfp};
      heap[0] = RunHead{bestE, 0, bestfp, 1, 0};
    }
    bits_to_words(pbits, a.L, a.best_seqs + cand * a.W);
    __syncwarp();
    // all counts stay below 2^31: at most 2^21 pops of 704 children
    int heap_n = 1, top = 1, exps = 0, u = 0, improvements = 0;
    int stop = 0;
    while (true) {
      if (exps >= a.max_exp) stop = 1;
      else if (heap_n == 0) stop = 2;
      else if (a.T_u > 0 && u >= a.T_u) stop = 3;
      if (stop || err) break;
      // ---- pop: the top run's smallest node; the run's last node fills its place, the run's new
      //      smallest by a rescan, then the sift-down
      RunHead h = heap[0];
      const Node nd = arena[h.cur];
      const Node last = arena[h.end - 1];
      const int pE = nd.E, plink = nd.link;
      const uint64_t pfp = nd.fp;
      __syncwarp();
      if (lane == 0 && h.cur != h.end - 1) arena[h.cur] = last;
      __syncwarp();
      h.end--;
      if (h.end > h.begin) {
        run_min(arena, h.begin, h.end, h.E, h.fp, h.cur);
      } else {
        heap_n--;
        h = heap[heap_n];
      }
      if (heap_n > 0) {
        int i = 0;
        while (true) {
          const int c = 32 * i + 1 + lane;  // the level's children, one a lane
          RunHead ch{INT32_MAX, 0, ~0ull, 0, 0};
          if (c < heap_n) ch = heap[c];
          int E;
          uint64_t fp;
          int who;
          warp_argmin(ch.E, ch.fp, c < heap_n ? lane : -1, E, fp, who);
          if (!(kless(E, fp, h.E, h.fp))) break;
          if (lane == who) heap[i] = ch;
          i = 32 * i + 1 + who;
        }
        __syncwarp();
        if (lane == 0) heap[i] = h;
      }
      // ---- the pivot's sequence: the seed, or the child `col` of an earlier pivot
      if (plink < 0) {
        words_to_bits(a.seeds + cand * a.W, a.L, pbits);
      } else {
        words_to_bits(pivots + (plink >> 10), a.L, cbits, a.max_exp);
        const int col = plink & 1023;
        if (col < a.L)
          flip_bits(cbits, col, pbits);
        else
          rotate_bits<NW>(cbits, a.L, rshift(a.L, a.Tr, col - a.L), pbits);
      }
      bits_to_words(pbits, a.L, pivots + exps, a.max_exp);
      if (PAIRS) {  // cbits: the neighbours visited before
        if (lane < kBitWords) cbits[lane] = 0u;
        __syncwarp();
        constexpr int W = (NW + 1) / 2;
        for (int q0 = 0; q0 < exps; q0 += 64) {
          uint64_t x[2][W];
#pragma unroll
          for (int i = 0; i < 2; i++)
#pragma unroll
            for (int w = 0; w < W; w++) x[i][w] = pivots[w * a.max_exp + min(q0 + 32 * i + lane, exps - 1)];
#pragma unroll
          for (int i = 0; i < 2; i++) {
            int d = 0;
#pragma unroll
            for (int w = 0; w < W; w++) {
              x[i][w] ^= reinterpret_cast<const uint64_t*>(pbits)[w];
              d += __popcll(x[i][w]);
            }
            if (d <= 2) {  // (an earlier pivot differs in one position at least)
#pragma unroll
              for (int w = 0; w < W; w++) {
                if (uint32_t lo = (uint32_t)x[i][w]) atomicOr(&cbits[2 * w], lo);
                if (uint32_t hi = (uint32_t)(x[i][w] >> 32)) atomicOr(&cbits[2 * w + 1], hi);
              }
            }
          }
        }
        __syncwarp();
      }
      // ---- correlations, V and the neighbours' sums
      auto output = [&](int T, int r) { return 128 * T + 32 * (lane & 3) + (lane >> 2) + 16 * (r & 1) + 8 * (r >> 1) + 1; };
      uint32_t vr[V_IN_Q ? 2 * NT : 1];  // V of the lane's outputs, two a word
      if constexpr (V_IN_Q) {
        split_classes(pbits, cw);
        self_convolution<(NW + 1) / 2>(cw, rw, a.L, v);
#pragma unroll
        for (int i = 0; i < 2 * NT; i++) {
          const int m0 = output(i >> 1, 2 * (i & 1)), m1 = output(i >> 1, 2 * (i & 1) + 1);
          vr[i] = (m0 <= a.L ? (uint32_t)(uint16_t)v[m0] : 0u) | (m1 <= a.L ? (uint32_t)(uint16_t)v[m1] << 16 : 0u);
        }
        __syncwarp();
        if (lane == 0) v[a.L] = 0;  // q(0)
      }
      corr_words<NW>(pbits, pbits, a.L, [&](int d, int cd) {
        if (d >= 1 && d < a.L) put_q(qt, ip.mma, d, cd);
      });
      put_x(xt, pbits, a.L);
      if constexpr (!V_IN_Q) {
        split_classes(pbits, cw);
        self_convolution<(NW + 1) / 2>(cw, rw, a.L, v);
      } else {
        __syncwarp();
      }
      float acc[1][NT][4];
      scan_mma<1, NT>(qt, xs, ip.mma, a.L, acc);
      Node* run = arena + top;
      const int link0 = exps << 10;
      int nu = 0;
      int rE = INT32_MAX, ri = -1;  // this lane's smallest survivor (the run's head comes from these)
      uint64_t rf = ~0ull;
      // H: an insert-if-absent of each neighbour into the visited set, the first compare-and-swap of two tiles'
      // in flight at once: a neighbour is a survivor when its key was absent.  Inserting while other
      // neighbours are still tested changes none of their answers: their keys differ, and inserts only fill
      // empty slots, which no probe sequence of a present key crosses.
#pragma unroll
      for (int T0 = 0; T0 < NT; T0 += 2) {
        unsigned long long hv[8];
        uint64_t fv[8];
#pragma unroll
        for (int i = 0; i < 8; i++) {
          const int T = T0 + (i >> 2), m = output(T, i & 3);
          fv[i] = kEmpty;
          hv[i] = kEmpty;
          if (T < NT && m <= a.L) {
            fv[i] = pfp ^ a.ztab[m - 1];
            if (!PAIRS && fv[i] != kEmpty)
              hv[i] = atomicCAS(reinterpret_cast<unsigned long long*>(&H[hs_home(fv[i], a.H_log2)]), (unsigned long long)kEmpty, fv[i]);
          }
        }
#pragma unroll
        for (int i = 0; i < 8; i++) {
          const int T = T0 + (i >> 2);
          if (T >= NT) break;
          const int m = output(T, i & 3), jl = m - 1;
          bool fresh = false;
          if (m <= a.L) {
            if (PAIRS) {
              fresh = !((cbits[jl >> 5] >> (jl & 31)) & 1u);
            } else if (fv[i] == kEmpty) {
              fresh = !has_empty;
              has_empty = true;
            } else if (hv[i] == kEmpty || hv[i] == fv[i]) {
              fresh = hv[i] == kEmpty;
            } else {
              fresh = hs_add_from(H, a.H_log2, fv[i], hs_home(fv[i], a.H_log2), &err);
            }
          }
          const unsigned who = __ballot_sync(kFull, fresh);
          if (fresh) {
            const int tm = (int)acc[0][T][i & 3];
            const int vm = V_IN_Q ? (int)(int16_t)(vr[V_IN_Q ? 2 * T + ((i & 3) >> 1) : 0] >> (16 * (i & 1))) : (int)v[m];
            const int E = pE + 4 * (vm + a.L - 2 - ((pbits[jl >> 5] >> (jl & 31) & 1u) ? tm : -tm));
            const int k = nu + __popc(who & ((1u << lane) - 1u));
            run[k] = Node{E, link0 | jl, fv[i]};
            if (kless(E, fv[i], rE, rf)) {
              rE = E;
              rf = fv[i];
              ri = top + k;
            }
          }
          nu += __popc(who);
        }
      }
      has_empty = __any_sync(kFull, has_empty);
      // ---- the rotations, after the flips: one equal to a flip child or to an earlier rotation finds
      //      its key in the visited set (the same sequence; the smaller column is kept)
      for (int c = 0; c < (PAIRS ? 0 : 2 * a.Tr); c++) {
        rotate_bits<NW>(pbits, a.L, rshift(a.L, a.Tr, c), cbits);
        const int e = energy_words<NW>(cbits, a.L);
        const uint64_t hf = fp_bits(cbits, a.L, a.ztab);
        bool fresh = false;
        if (lane == 0 && hs_add(H, a.H_log2, hf, has_empty, &err)) {
          fresh = true;
          run[nu] = Node{e, link0 | (a.L + c), hf};
          if (kless(e, hf, rE, rf)) {
            rE = e;
            rf = hf;
            ri = top + nu;
          }
        }
        nu += __shfl_sync(kFull, (int)fresh, 0);
      }
      has_empty = __any_sync(kFull, has_empty);
      err = __reduce_or_sync(kFull, err);
      __syncwarp();
      // ---- best, statistics, the new run
      int E0 = INT32_MAX, i0 = 0;
      uint64_t fp0 = 0;
      if (nu > 0) warp_argmin(rE, rf, ri, E0, fp0, i0);
      if (nu > 0 && E0 < bestE) {
        bestE = E0;
        bestfp = fp0;
        const int col = arena[i0].link & 1023;
        if (col < a.L)
          flip_bits(pbits, col, cbits);
        else
          rotate_bits<NW>(pbits, a.L, rshift(a.L, a.Tr, col - a.L), cbits);
        bits_to_words(cbits, a.L, a.best_seqs + cand * a.W);
        improvements++;
        u = 0;
      } else {
        u++;
      }
      if (nu > 0) {  // push the run: sift up
        const RunHead nh{E0, i0, fp0, top + nu, top};
        int i = heap_n;
        while (i > 0) {
          const int pp = (i - 1) >> 5;
          const RunHead par = heap[pp];
          if (!kless(nh.E, nh.fp, par.E, par.fp)) break;
          __syncwarp();
          if (lane == 0) heap[i] = par;
          i = pp;
        }
        if (lane == 0) heap[i] = nh;
        heap_n++;
      }
      top += nu;  // the seed and every survivor: the visited set's size
      exps++;
      __syncwarp();
      if ((long long)top * 4 > hslots * 3) err = 1;  // keep the visited set below 3/4 load
    }
    if (lane == 0) {
      a.best_E[cand] = bestE;
      labs_pq_stats st{};
      st.expansions = exps;
      st.rounds = exps;
      st.survivors = top - 1;
      st.admitted = top - 1;
      st.evicted = 0;
      st.h_size = top;
      st.improvements = improvements;
      st.best_fp = bestfp;
      st.stop_reason = err ? 0 : stop;
      st.status = err ? LABS_ERR_CAPACITY : LABS_OK;
      a.stats[cand] = st;
    }
    __syncwarp();
  }
}

__global__ void indep_ztab_kernel(uint64_t* ztab, int L) {
  const uint64_t zk = stream_key(0, kPurposeZobrist, (uint64_t)L, 0);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < L; i += gridDim.x * blockDim.x) ztab[i] = zobrist(zk, i + 1);
}

}  // namespace

int launch_pq_independent(labs_ctx* ctx, const labs_pq_indep_cfg* cfg, const uint64_t* seeds, int n,
                          uint64_t* best_seqs, int32_t* best_E, labs_pq_stats* stats, cudaStream_t st) {
  if (n == 0) return LABS_OK;
  const int L = cfg->L, W = (L + 63) / 64;
  IndepArgs a{};
  a.L = L;
  a.W = W;
  a.Tr = cfg->T_r;
  a.width = L + 2 * cfg->T_r;
  a.H_log2 = cfg->H_log2;
  a.max_exp = cfg->max_expansions;
  a.T_u = cfg->T_u;
  a.arena_cap = 1 + a.max_exp * a.width;
  a.heap_cap = a.max_exp + 1;
  a.n = n;
  a.seeds = seeds;
  a.best_seqs = best_seqs;
  a.best_E = best_E;
  a.stats = stats;
  // resident warps: as many slots as the memory budget allows, at most one per candidate
  const bool pairs = cfg->T_r == 0 && a.max_exp <= kPairPops;
  const size_t base_slot =
      (size_t)a.arena_cap * sizeof(Node) + (size_t)a.heap_cap * sizeof(RunHead) + (size_t)a.max_exp * W * 8;
  const size_t per_slot = base_slot + (pairs ? 0 : 8ull << a.H_log2);
  // the stated need of one block (records, run heads, pivots with 4 L B of tables each, the visited set) must fit,
  // although less is allocated
  const size_t stated_slot = base_slot + (size_t)a.max_exp * 4 * (size_t)L + (8ull << a.H_log2);
  const size_t budget = cfg->max_workspace_bytes > 0 ? (size_t)cfg->max_workspace_bytes : ((size_t)64 << 30);
  if (cfg->T_r > kMaxTr) return LABS_ERR_INVALID_ARG;
  if (budget / (stated_slot * kIWarps) < 1) return LABS_ERR_NOMEM;
  IndepPlan ip;
  ip.mma = scan_mma_plan(L, 0, L - 1);
  ip.q = kInTables;
  ip.x = ip.q + 2 * ip.mma.q_words;
  ip.v = ip.x + ip.mma.x_words;
  void (*kern)(IndepArgs, IndepPlan) = nullptr;
  size_t smem = 0;
  long long blocks = 0, rounds = 0;
  // the plain form, or with V in q where that lets all candidates run in fewer rounds (4,096 of L = 527, T_r = 4, 64
  // pops: 35 ms in two rounds, 24.4 ms in one; 3,600, one round either way: 20.4 and 22.5 ms)
  for (int v_in_q = 0; v_in_q < 2; v_in_q++) {
    const int words = ip.v + (v_in_q ? 0 : L / 2 + 1);  // v[1 .. L]
    const size_t bytes = sizeof(uint32_t) * (size_t)((words + 3) / 4 * 4) * kIWarps;
    void (*k)(IndepArgs, IndepPlan) = nullptr;
    const int ks = by_words((L + 31) >> 5, [&](auto nw) {
      constexpr int NW = decltype(nw)::value;
      if constexpr (NW > 16)
        if (v_in_q) k = pairs ? pq_indep_kernel<NW, true, true> : pq_indep_kernel<NW, false, true>;
      if (!v_in_q) k = pairs ? pq_indep_kernel<NW, true, false> : pq_indep_kernel<NW, false, false>;
      return k ? cuda_status(allow_smem(ctx, k)) : LABS_OK;
    });
    if (!k && ks == LABS_OK) break;  // compiled in the plain form only
    int per_sm = 0;
    if (ks != LABS_OK || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 32 * kIWarps, bytes) != cudaSuccess ||
        per_sm < 1)
      return LABS_ERR_CUDA;
    long long b = std::min<long long>((long long)per_sm * ctx->num_sms, ((long long)n + kIWarps - 1) / kIWarps);
    b = std::min<long long>(b, (long long)(budget / (per_slot * kIWarps)));
    if (b < 1) return LABS_ERR_NOMEM;
    const long long r = ((long long)n + b * kIWarps - 1) / (b * kIWarps);
    if (kern && r >= rounds) break;
    kern = k;
    smem = bytes;
    blocks = b;
    rounds = r;
    ip.words = (int)(bytes / sizeof(uint32_t)) / kIWarps;
    if (r == 1) break;
  }
  const size_t slots = (size_t)blocks * kIWarps;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t o = off;
    off += (bytes + 255) & ~size_t(255);
    return o;
  };
  const size_t oA = take(slots * (size_t)a.arena_cap * sizeof(Node)), oHp = take(slots * (size_t)a.heap_cap * sizeof(RunHead));
  const size_t oP = take(slots * (size_t)a.max_exp * W * 8), oH = take(pairs ? 0 : slots * (8ull << a.H_log2));
  const size_t oZ = take(8 * (size_t)L), oC = take(8);
  char* base = static_cast<char*>(ws_get(ctx, kWsPqIndep, off));
  if (!base) return LABS_ERR_NOMEM;
  a.arena = reinterpret_cast<Node*>(base + oA);
  a.heap = reinterpret_cast<RunHead*>(base + oHp);
  a.pivots = reinterpret_cast<uint64_t*>(base + oP);
  a.H = reinterpret_cast<uint64_t*>(base + oH);
  a.ztab = reinterpret_cast<uint64_t*>(base + oZ);
  a.counter = reinterpret_cast<unsigned long long*>(base + oC);
  indep_ztab_kernel<<<(L + 255) / 256, 256, 0, st>>>(reinterpret_cast<uint64_t*>(base + oZ), L);
  if (cudaMemsetAsync(a.counter, 0, 8, st) != cudaSuccess) return LABS_ERR_CUDA;
  kern<<<(unsigned)blocks, 32 * kIWarps, smem, st>>>(a, ip);
  return cuda_status(cudaGetLastError());
}

}  // namespace labsg

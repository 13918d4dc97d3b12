// pq.cu -- step 2 of the dual-step search: Algorithm 2's priority-queue refinement over the unrestricted
// space, in batch-synchronous form (labs_pq_refine).
//
// GB300 mapping.  The paper runs one priority queue per candidate in Rust on CPU cores; here one open
// set of the cap smallest (E, fp) keys lives in HBM as an UNORDERED pool of entries (energy,
// fingerprint, sequence) with a free-slot stack, and beside it a histogram of the entries' energies
// (one bin per energy, clamped at both ends of a 2^17-bin window, and a coarse level whose bins each
// cover 256 fine bins).  The B smallest keys, or the cap smallest, are then found without ordering the pool: the
// histogram's prefix sums give the bin where the count is reached, every entry below it is taken, and
// only the entries of that one boundary bin are ranked (by their fingerprints' first bits, counted as they are
// gathered, then among the few that share the boundary's; a clamped bin holding several energies takes a radix
// select on the full key).  A round
//   pop      -- the b = min(B, open, budget left) smallest keys leave the pool (one pass over it): the round's
//               pivots, in any order (a sequence reached from two pivots is the same sequence);
//   expand   -- one warp per pivot: its correlations, every neighbour's sum on the tensor cores (scan_mma.cuh),
//               into a dense [pivot][column] array; one warp more per rotation of a pivot (MAKE_ROTATIONS,
//               T_r > 0: columns L .. L + 2 T_r - 1);
//   dedup    -- a visited-set lookup per child; survivors with equal (E', fp') (the same sequence) are kept once,
//               through a hash table;
//   best     -- strict improvement test on the smallest survivor key;
//   cut      -- the cap smallest of (pool u survivors): entries of the pool above the cut are evicted,
//               survivors below it are admitted into free slots and into the visited set H;
// keeps every result identical to the sequential definition whatever order threads run in.  The seeds
// enter through the same survivor path.
//
// Where counts meet one address (free slots, admissions) a block adds up first, one atomic per 1,024 entries;
// the pool's histogram after a round follows from the cut (bins below it gain the survivors', the boundary bin
// keeps what was taken, bins above are empty), so no entry updates it.
#include <algorithm>
#include <new>

#include "labs_internal.h"
#include "scan_mma.cuh"

namespace labsg {
namespace {

constexpr uint64_t kEmptyKey = ~0ull;  // free slot of the visited set (fp == ~0 is tracked by a flag)
constexpr int kPqWarps = 4;
constexpr int kMaxProbe = 1 << 20;
constexpr int kNB = 1 << 17;        // fine energy bins: bin = clamp(E - E_base, 0, kNB - 1)
constexpr int kCoarse = 256;        // fine bins per coarse bin
constexpr int kNC = kNB / kCoarse;  // coarse bins
constexpr int kMaxB = 8192;         // pops per round
constexpr int kSelThreads = 1024;   // threads of the single-block kernels
constexpr int kFpBins = 1024;       // first bits of the boundary candidates' fingerprints

// Device-side state of one refinement (every round reads and writes it; the host only polls `stop`).
struct PqState {
  long long nP;  // open-set entries
  long long expansions, rounds, survivors, admitted, evicted, h_size, improvements, u;
  unsigned long long best_fp;
  long long free_top;   // free pool slots (the stack holds their ids)
  long long pop_base;   // stack slots the round's pops are freed to
  long long pop_cnt;    // entries gathered for popping this round
  long long cand_cnt;   // boundary-bin candidates gathered
  long long nU;         // unique survivors of the round
  long long n_dense;    // dense survivor entries of the round: b x width, or the seeds
  long long sel_need;   // entries taken from the boundary bin; 0: none; -1: no cut (everything kept)
  long long ev_round;   // evicted this round
  long long adm_round;  // admitted this round
  int b, stop, best_E, error, h_has_empty, E_base;
  int sel_bin;     // boundary fine bin
  int minE_round;  // smallest survivor energy of the round
  int sel_E, pmax_bin;        // pmax_bin: highest occupied bin of the pool after the pops (-1: empty pool)
  unsigned long long sel_fp;  // boundary key: a boundary-bin entry is taken iff (E, fp) <= (sel_E, sel_fp)
  unsigned long long minfp_round;
  long long nU_low;    // survivors in bins <= pmax_bin
  int grp_n, done;     // fingerprints collected by the boundary select, blocks finished with their part
};

struct PqBufs {
  int L, W, B, H_log2;
  int Tr, width;  // rotations per side (MAKE_ROTATIONS) and survivor columns per pivot: L flips + 2 Tr rotations
  long long cap, max_exp, T_u;
  int hs_log2;        // dedup hash table: 2^hs_log2 slots, at least twice the dense survivors
  long long cand_cap; // boundary candidate capacity (cap + dense survivors)
  int n_seeds;
  int32_t* pE;        // pool [cap]: energy, INT32_MAX for a free slot
  uint64_t* pFp;      // pool [cap]: fingerprint
  uint64_t* pSeq;     // pool [cap][W]
  int32_t* freeIds;   // free-slot stack [cap]
  unsigned* hP;       // histogram of the pool's energies: fine [kNB], coarse [kNC]
  unsigned* hP2;
  unsigned* hU;       // histogram of the round's unique survivors
  unsigned* hU2;
  unsigned* hF;       // [kFpBins] first fingerprint bits of the boundary candidates
  int32_t* popId;     // pool ids of the pops [B], with their keys
  int32_t* popE;
  uint64_t* popF;
  uint64_t* pivSeq;   // [B][W]: their sequences
  int32_t* candId;    // boundary candidates: pool id >= 0, or -(u + 1) for survivor u
  int32_t* cE;        // their keys, gathered contiguously
  uint64_t* cF;
  uint64_t* grp;      // fingerprints of the boundary's group
  int32_t* dE;        // dense survivors [pivot][column]: energy, or INT32_MAX (visited, or an equal one is kept)
  uint64_t* dFp;
  uint64_t* hkey;     // dedup hash table: mixed (E, fp) key, 0 = empty
  uint64_t* H;        // visited set (open addressing)
  uint32_t* filter;   // its filter, 2^f_log2 bits
  int f_log2;
  uint64_t* ztab;
  PqState* st;
  uint64_t* best_seq;
  const uint64_t* seeds;
};

// Left shift of rotation code c (MAKE_ROTATIONS): c < Tr moves the first c + 1 elements to the end,
// c >= Tr moves the last c - Tr + 1 elements to the start (a left shift by L - (c - Tr + 1)).
__host__ __device__ __forceinline__ int rot_shift(int L, int Tr, int c) {
  const int r = c < Tr ? c + 1 : L - ((c - Tr + 1) % L);
  return r % L;
}

// Survivor column col of a pivot (src, W words): col < L flips position col + 1, else rotation col - L.
// One thread; dst may be global memory.
__device__ __forceinline__ void pq_child(const uint64_t* src, const PqBufs& b, int col, uint64_t* dst) {
  uint64_t out[LABS_MAX_W];
  if (col < b.L) {
    for (int t = 0; t < b.W; t++) out[t] = src[t] ^ (t == (col >> 6) ? 1ull << (col & 63) : 0ull);
  } else {
    const int r = rot_shift(b.L, b.Tr, col - b.L);  // element i is element i + r (mod L)
    for (int t = 0; t < b.W; t++) {
      const int o = 64 * t + r, ow = o - b.L;
      uint64_t x = 0;
      auto window = [&](int p) {  // 64 bits from bit p on; bits at and above L are zero
        const int w = p >> 6, sh = p & 63;
        return (src[w] >> sh) | (sh && w + 1 < b.W ? src[w + 1] << (64 - sh) : 0ull);
      };
      if (o < b.L) x = window(o);
      if (ow >= 0)  // elements past the end come from the start
        x = window(ow);
      else if (ow > -64)
        x |= src[0] << -ow;
      const int left = b.L - 64 * t;
      out[t] = left < 64 ? x & ((1ull << left) - 1) : x;
    }
  }
  for (int t = 0; t < b.W; t++) dst[t] = out[t];
}

__device__ __forceinline__ uint64_t h_slot(uint64_t fp, int log2) { return (fp * kGamma) >> (64 - log2); }

// Continues the probe sequence of fp after slot s, whose key was another one.
__device__ __forceinline__ bool h_contains_after(const PqBufs& b, uint64_t fp, uint64_t s) {
  const uint64_t mask = (1ull << b.H_log2) - 1;
  for (int it = 1; it < kMaxProbe; it++) {
    s = (s + 1) & mask;
    const uint64_t v = b.H[s];
    if (v == fp) return true;
    if (v == kEmptyKey) return false;
  }
  atomicExch(&b.st->error, 1);  // probe limit: the set is too full (reported as a capacity error)
  return true;
}

// One bit per home slot of H (or per 2^k of them, at most 2^kFilterMax bits, 32 MB): a clear bit means that
// nothing hashed there was inserted, so most lookups of new states end in L2 instead of reading H from DRAM.
// Past kFilterFull insertions, when 63% of the bits are set at most, lookups go to H at once.  L = 451, 4,096 seeds, a
// visited set of 1.8e8 states at the end (10^7 pops): 601 ms with the filter to the end, 619 ms with half of kFilterFull;
// of 4.4e8 states (4 10^7 pops): 3.00 s and, never given up, 3.05 s.
constexpr int kFilterMax = 28;
constexpr long long kFilterFull = 1ll << kFilterMax;
__device__ __forceinline__ bool use_filter(const PqBufs& b) { return b.st->h_size < kFilterFull; }
__device__ __forceinline__ uint32_t filter_bit(const PqBufs& b, uint64_t fp) {
  return (uint32_t)((fp * kGamma) >> (64 - b.f_log2));
}
__device__ __forceinline__ bool filter_hit(const PqBufs& b, uint64_t fp) {
  const uint32_t i = filter_bit(b, fp);
  return (b.filter[i >> 5] >> (i & 31)) & 1u;
}

// Inserts fp; returns 1 when it was not there yet (the caller counts insertions into h_size in bulk).
__device__ __forceinline__ int h_insert(const PqBufs& b, uint64_t fp) {
  if (fp == kEmptyKey) return atomicExch(&b.st->h_has_empty, 1) == 0 ? 1 : 0;
  const uint32_t fi = filter_bit(b, fp);
  atomicOr(&b.filter[fi >> 5], 1u << (fi & 31));
  const uint64_t mask = (1ull << b.H_log2) - 1;
  uint64_t s = h_slot(fp, b.H_log2);
  for (int it = 0; it < kMaxProbe; it++) {
    const unsigned long long old =
        atomicCAS(reinterpret_cast<unsigned long long*>(&b.H[s]), (unsigned long long)kEmptyKey, fp);
    if (old == kEmptyKey) return 1;
    if (old == fp) return 0;
    s = (s + 1) & mask;
  }
  atomicExch(&b.st->error, 1);
  return 0;
}

__device__ __forceinline__ bool key_le(int Ea, uint64_t fa, int Eb, uint64_t fb) {
  return Ea < Eb || (Ea == Eb && fa <= fb);
}

__device__ __forceinline__ int e_bin(int E, int E_base) {
  const int d = E - E_base;
  return d < 0 ? 0 : (d >= kNB ? kNB - 1 : d);
}

// Whether a bin holds one energy only: not the window's end bins.
__device__ __forceinline__ bool one_energy(int bin) { return bin > 0 && bin < kNB - 1; }

// Block-wide sum added to *ctr with one atomic per block (every thread of the block calls it).
__device__ __forceinline__ void block_add(long long* ctr, long long v) {
  __shared__ long long part[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  if (lane_id() == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += part[w];
    if (t) atomicAdd(reinterpret_cast<unsigned long long*>(ctr), (unsigned long long)t);
  }
  __syncthreads();
}

// Block-wide minimum folded into *dst with one atomic per block (every thread calls it).
__device__ __forceinline__ void block_min(int* dst, int v) {
  __shared__ int part[32];
  v = __reduce_min_sync(kFull, v);
  if (lane_id() == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = INT32_MAX;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) t = min(t, part[w]);
    if (t != INT32_MAX) atomicMin(dst, t);
  }
  __syncthreads();
}

// Adds sign times the block's total of n (per thread) to *ctr with one atomic (every thread calls it; two
// barriers) and returns the counter's value before it; *before: the counts of the threads in front.
__device__ __forceinline__ long long block_reserve(long long* ctr, int n, int sign, int* total, int* before) {
  __shared__ int part[32];
  __shared__ long long base;
  int incl = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kFull, incl, o);
    if (lane_id() >= o) incl += v;
  }
  if (lane_id() == 31) part[threadIdx.x >> 5] = incl;
  __syncthreads();
  const int nw = (int)(blockDim.x >> 5);
  int front = 0, all = 0;
  for (int w = 0; w < nw; w++) {
    const int v = part[w];
    if (w < (int)(threadIdx.x >> 5)) front += v;
    all += v;
  }
  if (threadIdx.x == 0)
    base = all ? (long long)atomicAdd(reinterpret_cast<unsigned long long*>(ctr), (unsigned long long)(long long)(sign * all)) : 0;
  __syncthreads();
  *total = all;
  *before = front + incl - n;
  return base;
}

// Survivor histogram of a block: the fine bins are counted one by one in global memory (a round's energies
// spread over some hundred), the coarse ones, few and hot, in shared memory and added once.  The window's two end
// bins hold every energy beyond it, a round's survivors all together where a search has left the window: a thread
// counts those itself (low half: bin 0, high half: the last), and a block adds them once.
struct CoarseCounts {
  unsigned* n;  // [kNC] shared
  unsigned ends;
  __device__ __forceinline__ explicit CoarseCounts(unsigned* shared) : n(shared), ends(0) {
    for (int i = threadIdx.x; i < kNC; i += blockDim.x) n[i] = 0u;
    __syncthreads();
  }
  __device__ __forceinline__ void add(unsigned* fine, int bin) {
    if (one_energy(bin)) {
      atomicAdd(&fine[bin], 1u);
      atomicAdd(&n[bin / kCoarse], 1u);
    } else {
      ends += bin ? 0x10000u : 1u;  // (a thread sees some ten entries a round)
    }
  }
  __device__ __forceinline__ void flush(unsigned* fine, unsigned* coarse) {
    if (__syncthreads_or((int)ends)) {
      __shared__ unsigned both[2];
      if (threadIdx.x < 2) both[threadIdx.x] = 0u;
      __syncthreads();
      const unsigned lo = __reduce_add_sync(kFull, ends & 0xffffu), hi = __reduce_add_sync(kFull, ends >> 16);
      if (lane_id() == 0) {
        if (lo) atomicAdd(&both[0], lo);
        if (hi) atomicAdd(&both[1], hi);
      }
      __syncthreads();
      if (threadIdx.x < 2 && both[threadIdx.x]) {
        atomicAdd(&fine[threadIdx.x ? kNB - 1 : 0], both[threadIdx.x]);
        atomicAdd(&n[threadIdx.x ? kNC - 1 : 0], both[threadIdx.x]);
      }
      __syncthreads();
    }
    for (int i = threadIdx.x; i < kNC; i += blockDim.x)
      if (n[i]) atomicAdd(&coarse[i], n[i]);
  }
};

// Mixed key of (E, fp) for the dedup table; 0 marks an empty slot, so a mixed key of 0 becomes 1.
__device__ __forceinline__ uint64_t dedup_key(int E, uint64_t fp) {
  const uint64_t k = fp ^ ((uint64_t)(uint32_t)E * 0xD6E8FEB86659FD93ull);
  return k ? k : 1ull;
}

// ---------------------------------------------------------------------------------------------
// Set-up kernels
// ---------------------------------------------------------------------------------------------
__global__ void pq_ztab_kernel(uint64_t* ztab, int L) {
  const uint64_t zk = stream_key(0, kPurposeZobrist, (uint64_t)L, 0);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < L; i += gridDim.x * blockDim.x) ztab[i] = zobrist(zk, i + 1);
}

// Every pool slot free (the stack holds them all), the state zeroed.
__global__ void pq_init_kernel(PqBufs b) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < b.cap; i += (long long)gridDim.x * blockDim.x) {
    b.pE[i] = INT32_MAX;
    b.freeIds[i] = (int32_t)(b.cap - 1 - i);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    PqState z{};
    z.free_top = b.cap;
    z.best_E = INT32_MAX;
    z.best_fp = ~0ull;
    z.minE_round = INT32_MAX;
    z.minfp_round = ~0ull;
    z.pmax_bin = -1;
    z.sel_need = -1;
    z.n_dense = b.n_seeds;
    *b.st = z;
  }
}

// One warp per seed: energy over all lags and the fingerprint, into the dense arrays (one column).
__global__ void __launch_bounds__(32 * kPqWarps) pq_seed_kernel(PqBufs b, int n_seeds) {
  __shared__ uint32_t bits_all[kPqWarps][kBitWords];
  uint32_t* bits = bits_all[threadIdx.x >> 5];
  const int lane = lane_id();
  for (int q = blockIdx.x * kPqWarps + (threadIdx.x >> 5); q < n_seeds; q += gridDim.x * kPqWarps) {
    const uint64_t* src = b.seeds + (size_t)q * b.W;
    if (lane < kBitWords) {
      const int W32 = (b.L + 31) >> 5;
      uint32_t v = 0;
      if (lane < W32) {
        uint64_t x = src[lane >> 1];
        v = (lane & 1) ? (uint32_t)(x >> 32) : (uint32_t)x;
        int rem = b.L - 32 * lane;
        if (rem < 32) v &= (1u << rem) - 1u;
      }
      bits[lane] = v;
    }
    __syncwarp();
    int e = 0;
    for (int k = lane + 1; k < b.L; k += 32) {
      const int c = corr_lag(bits, b.L, k);
      e += c * c;
    }
    e = warp_sum_i32(e);
    uint64_t h = 0;
    for (int i = lane + 1; i <= b.L; i += 32)
      if (!((bits[(i - 1) >> 5] >> ((i - 1) & 31)) & 1u)) h ^= b.ztab[i - 1];
    h = warp_xor_u64(h);
    if (lane == 0) {
      b.dE[q] = e;
      b.dFp[q] = h;
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------------------------
// Round kernels.  SEED = true runs the survivor path on the seeds (dense = the seeds, one column each; nothing
// is counted as a survivor or an admission).
// ---------------------------------------------------------------------------------------------

// One block: the fine bin where the count of entries (hP, plus hU when CUT) reaches target > 0, into sel_bin,
// and the entries to take from it, into sel_need.
template <bool CUT>
__device__ __forceinline__ void select_bin(const PqBufs& b, long long target) {
  __shared__ unsigned long long wsum[kSelThreads / 32];
  __shared__ int s_cb;
  __shared__ unsigned long long s_before;
  PqState* st = b.st;
  const int t = threadIdx.x, lane = lane_id();
  auto scan = [&](unsigned long long own) {  // inclusive sum over the threads in front
    unsigned long long c = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long v = __shfl_up_sync(kFull, c, o);
      if (lane >= o) c += v;
    }
    __syncthreads();  // wsum's last readers are done
    if (lane == 31) wsum[t >> 5] = c;
    __syncthreads();
    for (int w = 0; w < t >> 5; w++) c += wsum[w];
    return c;
  };
  const unsigned long long tg = (unsigned long long)target;
  unsigned long long own = 0;
  if (t == 0) {  // a consistent histogram has a crossing bin
    s_cb = 0;
    s_before = 0;
  }
  if (t < kNC) own = (unsigned long long)b.hP2[t] + (CUT ? __ldcg(&b.hU2[t]) : 0u);
  unsigned long long c = scan(own);
  if (own && c >= tg && c - own < tg) {
    s_cb = t;
    s_before = c - own;
  }
  __syncthreads();
  const int cb = s_cb;
  const unsigned long long before = s_before;
  own = 0;
  if (t < kCoarse) own = (unsigned long long)b.hP[cb * kCoarse + t] + (CUT ? __ldcg(&b.hU[cb * kCoarse + t]) : 0u);
  c = before + scan(own);
  if (own && c >= tg && c - own < tg) {
    st->sel_bin = cb * kCoarse + t;
    st->sel_need = target - (long long)(c - own);
  }
  __syncthreads();
}

// The block's list of coarse bins with entries in the pool (or, CUT, among the survivors); returns their number.
template <bool CUT>
__device__ __forceinline__ int occupied_coarse(const PqBufs& b, int* list) {
  __shared__ int n;
  const int t = threadIdx.x;
  if (t == 0) n = 0;
  __syncthreads();
  if (t < kNC && (b.hP2[t] || (CUT && b.hU2[t]))) list[atomicAdd(&n, 1)] = t;
  __syncthreads();
  return n;
}

// Whether the cut needs the survivors above the pool's occupied bins counted: not when the pool's rest and the
// survivors inside those bins reach the cap.
__device__ __forceinline__ bool counts_all(const PqState* st, long long cap) {
  return st->pmax_bin < 0 || st->nP - st->b + st->nU_low < cap;
}

// One block: ends the round (or the seeds): the pool's histogram after the cut, the best (a strict improvement,
// as in Algorithm 2; for the seeds, the smallest seed) and the counters; then begins the next one: its number
// of pops and the bin that holds the last of them.
template <bool SEED>
__global__ void __launch_bounds__(kSelThreads) pq_finish_kernel(PqBufs b) {
  PqState* st = b.st;
  __shared__ int coarse[kNC];
  const int t = threadIdx.x, lane = lane_id();
  if (SEED || st->b > 0) {
    // ---- histogram: a warp per coarse bin that holds anything
    const int nc = occupied_coarse<true>(b, coarse);
    const bool cut = st->sel_need >= 0;
    const int sel = cut ? st->sel_bin : kNB;
    const unsigned need = cut ? (unsigned)st->sel_need : 0u;
    for (int x = t >> 5; x < nc; x += kSelThreads / 32) {
      const int cb = coarse[x];
      unsigned u[kCoarse / 32], h[kCoarse / 32], sum = 0;
#pragma unroll
      for (int i = 0; i < kCoarse / 32; i++) {
        u[i] = b.hU[cb * kCoarse + 32 * i + lane];
        h[i] = b.hP[cb * kCoarse + 32 * i + lane];
      }
#pragma unroll
      for (int i = 0; i < kCoarse / 32; i++) {
        const int bin = cb * kCoarse + 32 * i + lane;
        const unsigned now = bin < sel ? h[i] + u[i] : (bin == sel ? need : 0u);
        if (now != h[i]) b.hP[bin] = now;
        if (u[i]) b.hU[bin] = 0u;
        sum += now;
      }
      sum = (unsigned)warp_sum_i32((int)sum);
      __syncwarp();
      if (lane == 0) {
        b.hP2[cb] = sum;
        b.hU2[cb] = 0u;
      }
    }
    __syncthreads();
    // ---- the best: an improvement's survivor is looked up in the dense array (few rounds improve)
    __shared__ long long s_best;
    const bool improved = st->nU > 0 && (SEED || st->minE_round < st->best_E);
    if (t == 0) s_best = -1;
    __syncthreads();
    if (improved) {
      const int E = st->minE_round;
      const uint64_t fp = st->minfp_round;
      const long long n = st->n_dense, nq = (n + 3) >> 2;
#pragma unroll 4
      for (long long qd = t; qd < nq; qd += kSelThreads) {
        const int4 e4 = reinterpret_cast<const int4*>(b.dE)[qd];
        const int Ev[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
        for (int j = 0; j < 4; j++)
          if (Ev[j] == E && 4 * qd + j < n && b.dFp[4 * qd + j] == fp) s_best = 4 * qd + j;
      }
      __syncthreads();
    }
    if (t == 0) {
      if (!SEED) st->survivors += st->nU;
      if (!SEED && st->pop_cnt != st->b) st->error = 1;
      if (improved) {
        const int E = st->minE_round;
        const uint64_t fp = st->minfp_round;
        const long long i = s_best;
        if (i < 0) {
          st->error = 1;  // cannot happen: the smallest key is a survivor's
        } else {
          st->best_E = E;
          st->best_fp = fp;
          if (SEED) {
            for (int w = 0; w < b.W; w++) b.best_seq[w] = b.seeds[(size_t)i * b.W + w];
          } else {
            pq_child(b.pivSeq + (size_t)(i / b.width) * b.W, b, (int)(i % b.width), b.best_seq);
            st->improvements++;
          }
        }
        if (!SEED) st->u = 0;
      } else if (!SEED) {
        st->u += st->b;
      }
      if (SEED) {
        st->nP = st->adm_round;
      } else {
        st->nP = st->nP - st->b - st->ev_round + st->adm_round;
        st->admitted += st->adm_round;
        st->evicted += st->ev_round;
        st->expansions += st->b;
        st->rounds++;
      }
      const long long slots = 1ll << b.H_log2;
      if (st->h_size * 4 > slots * 3) st->error = 1;
    }
    __syncthreads();
  }
  // ---- the next round
  if (t == 0) {
    if (!st->stop) {
      if (st->error)
        st->stop = 4;
      else if (st->expansions >= b.max_exp)
        st->stop = 1;
      else if (st->nP == 0)
        st->stop = 2;
      else if (b.T_u > 0 && st->u >= b.T_u)
        st->stop = 3;
    }
    st->pop_cnt = 0;
    st->cand_cnt = 0;
    st->nU = 0;
    st->nU_low = 0;
    st->ev_round = 0;
    st->adm_round = 0;
    st->minE_round = INT32_MAX;
    st->minfp_round = ~0ull;
    st->sel_need = 0;
    st->sel_bin = kNB;
    const long long bb = st->stop ? 0 : min(min((long long)b.B, st->nP), b.max_exp - st->expansions);
    st->b = (int)bb;
    st->n_dense = bb * b.width;
  }
  for (int i = t; i < kFpBins; i += kSelThreads) b.hF[i] = 0u;
  __syncthreads();
  if (st->b > 0) select_bin<false>(b, st->b);
}

// Entries of a pool or survivor pass per thread: 16 consecutive ones, four 16-byte loads of their energies in
// flight (the arrays are 256-byte aligned, their sizes rounded to whole quads), so that a pass costs a block one
// or two reservations.
constexpr int kPer = 16;
__device__ __forceinline__ void load_energies(const int32_t* src, long long first, long long n, int (&E)[kPer]) {
#pragma unroll
  for (int v = 0; v < kPer / 4; v++) {
    int4 e4 = make_int4(INT32_MAX, INT32_MAX, INT32_MAX, INT32_MAX);
    if (first + 4 * v < n) e4 = reinterpret_cast<const int4*>(src + first)[v];
    E[4 * v] = e4.x;
    E[4 * v + 1] = first + 4 * v + 1 < n ? e4.y : INT32_MAX;
    E[4 * v + 2] = first + 4 * v + 2 < n ? e4.z : INT32_MAX;
    E[4 * v + 3] = first + 4 * v + 3 < n ? e4.w : INT32_MAX;
  }
}

// Appends a block's boundary candidates: the entries of the thread's mask `is`.
__device__ __forceinline__ void append_candidates(const PqBufs& b, unsigned is, const int (&E)[kPer], long long first,
                                                  bool survivors) {
  if (!__syncthreads_or((int)is)) return;
  const bool grouped = one_energy(b.st->sel_bin);
  int total, before;
  long long o = block_reserve(&b.st->cand_cnt, __popc(is), 1, &total, &before);
  o += before;
#pragma unroll
  for (int e = 0; e < kPer; e++)
    if (is >> e & 1) {
      if (o >= b.cand_cap) {
        b.st->error = 1;  // the histogram bounds the count: only an inconsistent state gets here
      } else {
        const uint64_t fp = survivors ? b.dFp[first + e] : b.pFp[first + e];
        b.candId[o] = survivors ? -(int32_t)(first + e) - 1 : (int32_t)(first + e);
        b.cE[o] = E[e];
        b.cF[o] = fp;
        if (grouped) atomicAdd(&b.hF[fp >> 54], 1u);
      }
      o++;
    }
}

// Pass over the pool by the first pool_blocks blocks.  POP gathers the entries below the boundary bin (popped)
// and those in it (candidates); the cut evicts the entries above it (slot freed) and gathers those in it, and the
// blocks behind gather the boundary bin's survivors.
template <bool POP>
__global__ void __launch_bounds__(256) pq_pool_kernel(PqBufs b, unsigned pool_blocks) {
  PqState* st = b.st;
  if (POP ? st->b == 0 : st->sel_need <= 0) return;
  const int sel = st->sel_bin, Eb = st->E_base;
  if (!POP && blockIdx.x >= pool_blocks) {
    const long long n = st->n_dense;
    const long long stride = (long long)(gridDim.x - pool_blocks) * blockDim.x * kPer;
    for (long long base = (long long)(blockIdx.x - pool_blocks) * blockDim.x * kPer; base < n; base += stride) {
      const long long first = base + (long long)threadIdx.x * kPer;
      int E[kPer];
      load_energies(b.dE, first, n, E);
      unsigned cand = 0;
#pragma unroll
      for (int e = 0; e < kPer; e++)
        if (E[e] != INT32_MAX && e_bin(E[e], Eb) == sel) cand |= 1u << e;
      append_candidates(b, cand, E, first, true);
    }
    return;
  }
  const long long stride = (long long)pool_blocks * blockDim.x * kPer;
  long long freed = 0;
  for (long long base = (long long)blockIdx.x * blockDim.x * kPer; base < b.cap; base += stride) {
    const long long first = base + (long long)threadIdx.x * kPer;
    int E[kPer];
    load_energies(b.pE, first, b.cap, E);
    unsigned take = 0, cand = 0;
#pragma unroll
    for (int e = 0; e < kPer; e++)
      if (E[e] != INT32_MAX) {
        const int bin = e_bin(E[e], Eb);
        if (POP ? bin < sel : bin > sel) take |= 1u << e;
        if (bin == sel) cand |= 1u << e;
      }
    if (__syncthreads_or((int)take)) {
      int total, before;
      long long o = block_reserve(POP ? &st->pop_cnt : &st->free_top, __popc(take), 1, &total, &before);
      o += before;
#pragma unroll
      for (int e = 0; e < kPer; e++)
        if (take >> e & 1) {
          const long long i = first + e;
          if (o >= (POP ? (long long)b.B : b.cap)) {
            st->error = 1;  // the histogram bounds the count
          } else if (POP) {
            b.popId[o] = (int32_t)i;
            b.popE[o] = E[e];
            b.popF[o] = b.pFp[i];
          } else {
            b.freeIds[o] = (int32_t)i;
            b.pE[i] = INT32_MAX;
            freed++;
          }
          o++;
        }
    }
    append_candidates(b, cand, E, first, false);
  }
  if (!POP) block_add(&st->ev_round, freed);
}

// The sel_need smallest (E, fp) keys among the boundary candidates, whose keys are distinct.  A bin that is not
// clamped holds one energy: the counts of the fingerprints' first ten bits give the group that holds the
// boundary; all blocks collect that group's fingerprints (a thousandth of the candidates), and the last one to
// finish ranks them against each other.  Otherwise (a clamped bin, or a group beyond kGroup) the last block narrows
// the 96-bit key down, eleven bits a pass over the candidates, and ranks those that share the boundary's bits as
// soon as they fit in shared memory: one pass and the gathering one where the energies are spread.  Measured on 4
// random seeds of L = 527 (4,000 pops of 64 a round, cap 65,536: 30,000 candidates a select): 10.5 ms in all; 24.3 ms
// with twelve passes of a byte each, one global atomic per survivor of the end bin and one block to apply the cut,
// and 15.7 ms with a full pass per byte until 8,192 were left.
constexpr int kGroup = 4096;
constexpr int kDigit = 11, kStage = 2048;  // bits a pass; candidates ranked in shared memory
template <bool POP>
__global__ void __launch_bounds__(kSelThreads) pq_boundary_kernel(PqBufs b) {
  PqState* st = b.st;
  if (POP ? st->b == 0 : st->sel_need <= 0) return;
  __shared__ uint64_t grp[kGroup];
  __shared__ int s_bin, s_n, s_E, s_last;
  __shared__ long long s_need;
  __shared__ unsigned long long s_fp;
  __shared__ unsigned s_hist[1 << kDigit];
  __shared__ unsigned wsum[kSelThreads / 32];
  const int t = threadIdx.x, lane = lane_id();
  const long long n = min(st->cand_cnt, b.cand_cap);
  const long long need = st->sel_need;
  const int sel = st->sel_bin;
  if (t == 0) {
    s_n = 0;
    s_bin = 0;
    s_need = need;
    s_E = st->E_base + sel;
    s_fp = ~0ull;
  }
  // group of the boundary: inclusive sums of the counts
  const unsigned own = b.hF[t];
  unsigned c = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(kFull, c, o);
    if (lane >= o) c += v;
  }
  if (lane == 31) wsum[t >> 5] = c;
  __syncthreads();
  for (int w = 0; w < t >> 5; w++) c += wsum[w];
  if (own && (long long)c >= need && (long long)(c - own) < need) {
    s_bin = t;
    s_need = need - (long long)(c - own);  // rank inside the group, from 1
  }
  __syncthreads();
  const int gb = s_bin;
  const bool grouped = one_energy(sel) && b.hF[gb] <= (unsigned)kGroup;
  const long long stride = (long long)gridDim.x * kSelThreads;
  if (grouped)
    for (long long i0 = (long long)blockIdx.x * kSelThreads; i0 < n; i0 += 4 * stride) {
      uint64_t f[4];
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const long long i = i0 + e * stride + t;
        f[e] = i < n ? b.cF[i] : 0ull;
      }
#pragma unroll
      for (int e = 0; e < 4; e++)
        if (i0 + e * stride + t < n && (int)(f[e] >> 54) == gb) {
          const int w = atomicAdd(&st->grp_n, 1);
          if (w < kGroup) b.grp[w] = f[e];
        }
    }
  __threadfence();
  __syncthreads();
  if (t == 0) s_last = atomicAdd(&st->done, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (grouped) {
    const int m = min(*reinterpret_cast<volatile int*>(&st->grp_n), kGroup);
    for (int i = t; i < m; i += kSelThreads) grp[i] = *reinterpret_cast<volatile uint64_t*>(&b.grp[i]);
    __syncthreads();
    for (int i = t; i < m; i += kSelThreads) {
      const uint64_t f = grp[i];
      int r = 1;
      for (int j = 0; j < m; j++) r += grp[j] < f ? 1 : 0;
      if (r == (int)s_need) s_fp = f;
    }
    __syncthreads();
  } else {
    // Keys that agree with (preE, preF) in all bits from (sE, sF) up are still in question; the boundary is the k-th
    // of them.  Energies of the lower end bin are at most E_base, all below 2^26.
    uint64_t preF = 0;
    uint32_t preE = one_energy(sel) ? (uint32_t)s_E : 0u;
    int sE = one_energy(sel) ? 0 : (sel == 0 ? 32 - __clz(st->E_base) : 26), sF = 64;
    long long k = need, left = n;
    auto in_question = [&](uint32_t e, uint64_t f) {
      return e >> sE == preE >> sE && (sF == 64 || (f >> sF) == (preF >> sF));
    };
    auto each = [&](auto&& fn) {  // fn(candidate, energy); a thread's quads are loaded four at a time
      const long long nq = (n + 3) >> 2;
#pragma unroll 4
      for (long long q = t; q < nq; q += kSelThreads) {
        const int4 e4 = reinterpret_cast<const int4*>(b.cE)[q];
        const uint32_t e[4] = {(uint32_t)e4.x, (uint32_t)e4.y, (uint32_t)e4.z, (uint32_t)e4.w};
#pragma unroll
        for (int j = 0; j < 4; j++)
          if (4 * q + j < n) fn(4 * q + j, e[j]);
      }
    };
    while (left > kStage && sE + sF > 0) {
      // the next bits: of the energy, then of the fingerprint
      const int nE = sE ? max(sE - kDigit, 0) : 0, nF = sE ? 64 : max(sF - kDigit, 0);
      const bool fp_bits = sE == 0;
      for (int i = t; i < 1 << kDigit; i += kSelThreads) s_hist[i] = 0u;
      __syncthreads();
      each([&](long long i, uint32_t e) {
        const uint64_t f = fp_bits ? b.cF[i] : 0ull;
        if (in_question(e, f)) {
          const unsigned digit = fp_bits ? (unsigned)(f >> nF) : e >> nE;
          atomicAdd(&s_hist[digit & ((1u << kDigit) - 1u)], 1u);
        }
      });
      __syncthreads();
      // the digit where the count reaches k: two bins a thread
      const unsigned own0 = s_hist[2 * t], own1 = s_hist[2 * t + 1];
      unsigned c = own0 + own1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(kFull, c, o);
        if (lane >= o) c += v;
      }
      if (lane == 31) wsum[t >> 5] = c;
      __syncthreads();
      for (int w = 0; w < t >> 5; w++) c += wsum[w];
      const long long before = (long long)c - own0 - own1;
      if (before < k && (long long)c >= k) {
        const bool second = before + own0 < k;
        s_bin = 2 * t + (second ? 1 : 0);
        s_need = k - before - (second ? own0 : 0u);
        s_n = (int)(second ? own1 : own0);
      }
      __syncthreads();
      k = s_need;
      left = s_n;
      if (fp_bits)
        preF |= (uint64_t)s_bin << nF;
      else
        preE |= (uint32_t)s_bin << nE;
      sE = nE;
      sF = nF;
      __syncthreads();
    }
    // the candidates left, ranked against each other (grp: their fingerprints, behind them their energies)
    int* grpE = reinterpret_cast<int*>(grp + kStage);
    if (t == 0) s_n = 0;
    __syncthreads();
    each([&](long long i, uint32_t e) {
      if (e >> sE != preE >> sE) return;
      const uint64_t f = b.cF[i];
      if (in_question(e, f)) {
        const int w = atomicAdd(&s_n, 1);
        if (w < kStage) {
          grp[w] = f;
          grpE[w] = (int)e;
        }
      }
    });
    __syncthreads();
    const int m = min(s_n, kStage);
    for (int i = t; i < m; i += kSelThreads) {
      const uint64_t f = grp[i];
      const int e = grpE[i];
      int r = 0;
      for (int j = 0; j < m; j++) r += key_le(grpE[j], grp[j], e, f) ? 1 : 0;
      if (r == (int)k) {
        s_E = e;
        s_fp = f;
      }
    }
    __syncthreads();
  }
  if (t == 0) {
    st->sel_E = s_E;
    st->sel_fp = s_fp;
    st->grp_n = 0;  // for the next select
    st->done = 0;
  }
}

// The boundary candidates themselves: POP adds those up to the boundary to the pops; the cut evicts the pool's
// beyond it.  Block 0 of POP also takes the pops out of the histogram (all below the boundary bin, sel_need of
// it) and finds the highest occupied bin.
template <bool POP>
__global__ void __launch_bounds__(kSelThreads) pq_boundary_apply_kernel(PqBufs b) {
  PqState* st = b.st;
  if (POP ? st->b == 0 : st->sel_need <= 0) return;
  const int t = threadIdx.x, lane = lane_id();
  const long long n = min(st->cand_cnt, b.cand_cap);
  const int selE = st->sel_E;
  const uint64_t selF = st->sel_fp;
  long long freed = 0;
  for (long long i0 = (long long)blockIdx.x * kSelThreads; i0 < n; i0 += (long long)gridDim.x * kSelThreads) {
    const long long i = i0 + t;
    bool on = false;
    int id = 0, E = 0;
    uint64_t fp = 0;
    if (i < n) {
      id = b.candId[i];
      E = b.cE[i];
      fp = b.cF[i];
      const bool in = key_le(E, fp, selE, selF);
      on = POP ? in : (!in && id >= 0);
    }
    if (!__syncthreads_or(on)) continue;
    int total, before;
    long long o = block_reserve(POP ? &st->pop_cnt : &st->free_top, on ? 1 : 0, 1, &total, &before);
    o += before;
    if (on) {
      if (o >= (POP ? (long long)b.B : b.cap)) {
        st->error = 1;
      } else if (POP) {
        b.popId[o] = id;
        b.popE[o] = E;
        b.popF[o] = fp;
      } else {
        b.freeIds[o] = id;
        b.pE[id] = INT32_MAX;
        freed++;
      }
    }
  }
  if (!POP) {
    block_add(&st->ev_round, freed);
    return;
  }
  if (blockIdx.x != 0) return;
  __shared__ int coarse[kNC];
  __shared__ int s_bin;
  const int sel = st->sel_bin;
  const unsigned need = (unsigned)st->sel_need;
  const int nc = occupied_coarse<false>(b, coarse);
  if (t == 0) s_bin = -1;
  __syncthreads();
  for (int x = t >> 5; x < nc; x += kSelThreads / 32) {
    const int cb = coarse[x];
    unsigned h[kCoarse / 32], left = 0;
    int top = -1;
#pragma unroll
    for (int i = 0; i < kCoarse / 32; i++) h[i] = b.hP[cb * kCoarse + 32 * i + lane];
#pragma unroll
    for (int i = 0; i < kCoarse / 32; i++) {
      const int bin = cb * kCoarse + 32 * i + lane;
      const unsigned now = bin < sel ? 0u : (bin == sel ? h[i] - need : h[i]);
      if (now != h[i]) b.hP[bin] = now;
      left += now;
      if (now) top = bin;
    }
    left = (unsigned)warp_sum_i32((int)left);
    top = warp_max_i32(top);
    if (lane == 0) {
      b.hP2[cb] = left;
      if (top >= 0) atomicMax(&s_bin, top);
    }
  }
  __syncthreads();
  if (t == 0) {
    st->pmax_bin = s_bin;
    st->pop_base = st->free_top;
    st->free_top += st->b;  // filled by the expansion
  }
}

// Shared memory of one expanding warp, in 32-bit words from its slab's start.
struct ExpandPlan {
  ScanMmaPlan mma;
  int q, x, v, words;
};
constexpr int kExpBits = 0, kExpClass = kBitWords, kExpRev = kExpClass + 2 * kClassWords, kExpTables = kExpRev + 2 * kClassWords;

// Work items: pivot q's flips (c = 0) and its rotations (c = 1 .. 2 T_r), one warp each.  The flips' warp also
// takes the pivot's sequence out of the pool and frees its slot.
template <int NW>
__global__ void __launch_bounds__(32 * kPqWarps, NW <= 8 ? 6 : 4) pq_expand_kernel(PqBufs b, ExpandPlan ep) {
  constexpr int NT = (NW + 3) / 4;
  extern __shared__ __align__(16) uint32_t pq_smem[];
  uint32_t* slab = pq_smem + (size_t)(threadIdx.x >> 5) * ep.words;
  uint32_t *bits = slab + kExpBits, *cw = slab + kExpClass, *rw = slab + kExpRev, *qt = slab + ep.q, *xt = slab + ep.x;
  int16_t* v = reinterpret_cast<int16_t*>(slab + ep.v);
  const int lane = lane_id(), L = b.L;
  const PqState* st = b.st;
  const int nb = st->b;
  if (nb == 0 || st->pop_cnt != nb || st->error) return;  // an inconsistent pop ends the search in pq_finish_kernel
  for (int i = lane; i < ep.words; i += 32) slab[i] = 0u;
  __syncwarp();
  const int per = 1 + 2 * b.Tr;
  const uint32_t* const xs[1] = {xt};
  for (int it = blockIdx.x * kPqWarps + (threadIdx.x >> 5); it < nb * per; it += gridDim.x * kPqWarps) {
    // all flips first, so that a tail of short rotation items evens out the blocks
    const int q = it < nb ? it : (it - nb) % nb, rot = it < nb ? 0 : 1 + (it - nb) / nb;
    const int id = b.popId[q], E = b.popE[q];
    const uint64_t* src = b.pSeq + (size_t)id * b.W;
    __syncwarp();
    if (lane < NW) {
      const uint32_t w = reinterpret_cast<const uint32_t*>(src)[lane];
      bits[lane] = lane == NW - 1 ? w & (0xffffffffu >> (32 * NW - L)) : w;
    }
    __syncwarp();
    if (rot) {
      // rotation: element i is element i + r (mod L); its energy and fingerprint from scratch
      const uint32_t y = rotated_word<NW>(bits, L, rot_shift(L, b.Tr, rot - 1));
      if (lane < kBitWords) rw[lane] = y;
      __syncwarp();
      const int e = energy_words<NW>(rw, L);
      uint64_t h = 0;
      for (int i = lane; i < L; i += 32)
        if (!((rw[i >> 5] >> (i & 31)) & 1u)) h ^= b.ztab[i];
      h = warp_xor_u64(h);
      if (lane == 0) {
        const size_t di = (size_t)q * b.width + L + rot - 1;
        b.dE[di] = e;
        b.dFp[di] = h;
      }
      continue;
    }
    if (lane < b.W) b.pivSeq[(size_t)q * b.W + lane] = src[lane];
    if (lane == 0) {
      b.pE[id] = INT32_MAX;
      b.freeIds[st->pop_base + q] = id;
    }
    const uint64_t fp = b.popF[q];
    corr_words<NW>(bits, bits, L, [&](int d, int cd) {
      if (d >= 1 && d < L) put_q(qt, ep.mma, d, cd);
    });
    put_x(xt, bits, L);
    split_classes(bits, cw);
    self_convolution<(NW + 1) / 2>(cw, rw, L, v);
    __syncwarp();
    float acc[1][NT][4];
    scan_mma<1, NT>(qt, xs, ep.mma, L, acc);
    int32_t* oe = b.dE + (size_t)q * b.width;
    uint64_t* of = b.dFp + (size_t)q * b.width;
#pragma unroll
    for (int T = 0; T < NT; T++) {
      const int jl = 128 * T + 32 * (lane & 3) + (lane >> 2);
      const uint32_t own = jl < L ? bits[jl >> 5] >> (lane >> 2) : 0u;
#pragma unroll
      for (int r = 0; r < 4; r++) {
        const int o = 16 * (r & 1) + 8 * (r >> 1), m = jl + o + 1;
        if (m <= L) {
          const int tm = (int)acc[0][T][r];
          oe[m - 1] = E + 4 * ((int)v[m] + L - 2 - ((own >> o & 1u) ? tm : -tm));
          of[m - 1] = fp ^ b.ztab[m - 1];
        }
      }
    }
  }
}

// Visited set and dedup: a child found in H is dropped; every other inserts its (E, fp) key; the first inserter of a key stays the key's survivor, the
// others are dropped from the dense array.  Which one stays does not
// matter: equal keys are the same sequence.  Survivors inside the pool's occupied bins are counted on the way
// (the cut lies there once the pool is full).  Each thread takes four consecutive survivors and keeps their four
// probes in flight together (the pass is bound by the latency of the table's compare-and-swaps).  Six blocks an SM hold
// it to 40 registers and 168 bytes of spills; with four (57 registers, none) 10^6 pops of L = 451 measured 50.4 ms against
// 51.7 ms.
template <bool SEED>
__global__ void __launch_bounds__(256, 6) pq_dedup_kernel(PqBufs b) {
  PqState* st = b.st;
  __shared__ unsigned coarse[kNC];
  const long long n = st->n_dense;
  if (n == 0) return;
  CoarseCounts counts(coarse);
  const bool filter = use_filter(b);
  const long long nq = (n + 3) >> 2;
  const uint64_t mask = (1ull << b.hs_log2) - 1;
  const int Eb = st->E_base, pmax = SEED ? -1 : st->pmax_bin;  // the seeds' energy window is not set yet
  long long kept = 0, low = 0;
  int mE = INT32_MAX;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long base = (long long)blockIdx.x * blockDim.x; base < nq; base += stride) {  // warp-uniform
    const long long qd = base + threadIdx.x;
    int E[4] = {INT32_MAX, INT32_MAX, INT32_MAX, INT32_MAX};
    if (qd < nq) {
      const int4 e4 = reinterpret_cast<const int4*>(b.dE)[qd];
      E[0] = e4.x;
      E[1] = e4.y;
      E[2] = e4.z;
      E[3] = e4.w;
    }
    uint64_t k[4], s[4];
    bool act[4], fresh[4];
    {
      uint64_t fp[4], hv[4];
#pragma unroll
      for (int j = 0; j < 4; j++) {
        act[j] = 4 * qd + j < n;
        fp[j] = act[j] ? b.dFp[4 * qd + j] : kEmptyKey;
      }
      if (!SEED) {
#pragma unroll
        for (int j = 0; j < 4; j++) hv[j] = fp[j] != kEmptyKey && (!filter || filter_hit(b, fp[j])) ? b.H[h_slot(fp[j], b.H_log2)] : kEmptyKey;
#pragma unroll
        for (int j = 0; j < 4; j++) {
          if (!act[j]) continue;
          bool seen;
          if (fp[j] == kEmptyKey)
            seen = st->h_has_empty != 0;
          else if (hv[j] == fp[j] || hv[j] == kEmptyKey)
            seen = hv[j] == fp[j];
          else
            seen = h_contains_after(b, fp[j], h_slot(fp[j], b.H_log2));
          if (seen) {
            b.dE[4 * qd + j] = INT32_MAX;
            act[j] = false;
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 4; j++) {
        fresh[j] = false;
        k[j] = act[j] ? dedup_key(E[j], fp[j]) : 0ull;
        s[j] = (k[j] * kGamma) >> (64 - b.hs_log2);
      }
    }
    for (uint64_t it = 0; it <= mask && (act[0] || act[1] || act[2] || act[3]); it++) {  // at most half full
      unsigned long long old[4];
#pragma unroll
      for (int j = 0; j < 4; j++)
        old[j] = act[j] ? atomicCAS(reinterpret_cast<unsigned long long*>(&b.hkey[s[j]]), 0ull, k[j]) : 0ull;
#pragma unroll
      for (int j = 0; j < 4; j++) {
        if (!act[j]) continue;
        if (old[j] == 0ull) {
          fresh[j] = true;
          act[j] = false;
        } else if (old[j] == k[j]) {
          act[j] = false;
          b.dE[4 * qd + j] = INT32_MAX;
        } else {
          s[j] = (s[j] + 1) & mask;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; j++) {
      if (fresh[j]) {
        kept++;
        mE = min(mE, E[j]);
        const int bin = e_bin(E[j], Eb);
        if (bin <= pmax) {
          low++;
          counts.add(b.hU, bin);
        }
      }
    }
  }
  counts.flush(b.hU, b.hU2);
  block_add(&st->nU, kept);
  block_min(&st->minE_round, mE);
  block_add(&st->nU_low, low);
}

// The survivors above the pool's occupied bins are counted when the cut may lie there or nothing is cut; then the
// last block to finish finds where the cap cuts (pool's rest u survivors), or that everything fits.
__global__ void __launch_bounds__(kSelThreads) pq_cut_kernel(PqBufs b) {
  PqState* st = b.st;
  __shared__ unsigned coarse[kNC];
  __shared__ int s_last;
  if (counts_all(st, b.cap)) {
    CoarseCounts counts(coarse);
    const long long n = st->n_dense;
    const int Eb = st->E_base, pmax = st->pmax_bin;
    const long long stride = (long long)gridDim.x * blockDim.x * kPer;
    for (long long first = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * kPer; first < n; first += stride) {
      int E[kPer];
      load_energies(b.dE, first, n, E);
#pragma unroll
      for (int e = 0; e < kPer; e++)
        if (E[e] != INT32_MAX) {
          const int bin = e_bin(E[e], Eb);
          if (bin > pmax) counts.add(b.hU, bin);
        }
    }
    counts.flush(b.hU, b.hU2);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&st->done, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const bool fits = st->nP - st->b + st->nU <= b.cap;
  __syncthreads();
  if (threadIdx.x == 0) {
    st->done = 0;
    st->cand_cnt = 0;  // the pop's candidates are done with
    st->sel_need = fits ? -1 : 0;
    st->sel_bin = kNB;
  }
  for (int i = threadIdx.x; i < kFpBins; i += kSelThreads) b.hF[i] = 0u;
  __syncthreads();
  if (!fits) select_bin<true>(b, b.cap);
}

// The histogram's energy window, from the smallest seed energy: 65,536 below it and above it.  From sieved seeds a
// search stays inside; from random ones at L = 527 the best is below after some thirty rounds, and from then on most
// entries lie in bin 0 (from constant ones in either end bin).
__global__ void pq_set_window_kernel(PqBufs b) {
  PqState* st = b.st;
  st->E_base = st->minE_round == INT32_MAX ? 0 : max(0, st->minE_round - kNB / 2);
}

// Survivor pass: the survivors inside the cut take a free slot (the sequence built from the pivot, or copied
// from the seed) and enter the visited set; the smallest fingerprint among the smallest energies is noted for
// the best.  Four consecutive survivors per thread: a fingerprint is read only where the cut or the best test
// needs it.
template <bool SEED>
__global__ void __launch_bounds__(256) pq_admit_kernel(PqBufs b) {
  PqState* st = b.st;
  const long long n = st->n_dense;
  if (n == 0) return;
  const long long nq = (n + 3) >> 2;
  const int Eb = st->E_base;
  const bool cut = st->sel_need >= 0;
  const int sel_bin = st->sel_bin, minE = st->minE_round, selE = st->sel_E;
  const uint64_t selF = st->sel_fp;
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long ins = 0, adm = 0;
  uint64_t mf = ~0ull;
  for (long long base = (long long)blockIdx.x * blockDim.x; base < nq; base += stride) {  // block-uniform
    const long long qd = base + threadIdx.x;
    int4 e4 = make_int4(INT32_MAX, INT32_MAX, INT32_MAX, INT32_MAX);
    if (qd < nq) e4 = reinterpret_cast<const int4*>(b.dE)[qd];
    const int E[4] = {e4.x, e4.y, e4.z, e4.w};
    bool in[4];
    uint64_t fp[4];
    int mine = 0;
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const long long u = 4 * qd + j;
      in[j] = false;
      fp[j] = 0;
      if (u < n && E[j] != INT32_MAX) {
        const int bin = e_bin(E[j], Eb);
        if (!cut || bin <= sel_bin || E[j] == minE) {
          fp[j] = b.dFp[u];
          in[j] = !cut || bin < sel_bin || (bin == sel_bin && key_le(E[j], fp[j], selE, selF));
          if (E[j] == minE) mf = min(mf, fp[j]);
        }
      }
      mine += in[j] ? 1 : 0;
    }
    if (!__syncthreads_or(mine)) continue;
    int total, before;
    // free slots come off the top of the stack, the block's share at once
    long long o = block_reserve(&st->free_top, mine, -1, &total, &before);
    o += before - total;
#pragma unroll
    for (int j = 0; j < 4; j++)
      if (in[j]) {
        const long long u = 4 * qd + j;
        if (o < 0) {  // more admissions than free slots: only an inconsistent state gets here
          st->error = 1;
          o++;
          continue;
        }
        const int id = b.freeIds[o++];
        b.pE[id] = E[j];
        b.pFp[id] = fp[j];
        if (SEED) {
          for (int t = 0; t < b.W; t++) b.pSeq[(size_t)id * b.W + t] = b.seeds[(size_t)u * b.W + t];
        } else {
          pq_child(b.pivSeq + (size_t)(u / b.width) * b.W, b, (int)(u % b.width), b.pSeq + (size_t)id * b.W);
        }
        adm++;
        ins += h_insert(b, fp[j]);
      }
  }
  if (mf != ~0ull) atomicMin(reinterpret_cast<unsigned long long*>(&st->minfp_round), (unsigned long long)mf);
  block_add(&st->h_size, ins);
  block_add(&st->adm_round, adm);
}

__global__ void pq_write_stats_kernel(PqBufs b, int32_t* best_E, labs_pq_stats* out) {
  const PqState* st = b.st;
  *best_E = st->best_E;
  out->expansions = st->expansions;
  out->rounds = st->rounds;
  out->survivors = st->survivors;
  out->admitted = st->admitted;
  out->evicted = st->evicted;
  out->h_size = st->h_size;
  out->improvements = st->improvements;
  out->best_fp = st->best_fp;
  out->stop_reason = st->stop == 4 ? 0 : st->stop;
  out->status = st->error ? LABS_ERR_CAPACITY : LABS_OK;
}

}  // namespace

int launch_pq_refine(labs_ctx* ctx, const labs_pq_cfg* cfg, const uint64_t* seeds, int n_seeds, uint64_t* best_seq,
                     int32_t* best_E, labs_pq_stats* stats, cudaStream_t st) {
  const int L = cfg->L, W = (L + 63) / 64;
  if (cfg->B > kMaxB) return LABS_ERR_INVALID_ARG;
  const int width = L + 2 * cfg->T_r;
  const long long n_dense = std::max<long long>((long long)cfg->B * width, n_seeds);
  int hs_log2 = 10;
  while ((1ll << hs_log2) < 2 * n_dense) hs_log2++;
  const long long cap = cfg->cap;
  // workspace layout (one region, 256-byte aligned pieces)
  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t o = off;
    off += (bytes + 255) & ~size_t(255);
    return o;
  };
  const size_t opE = take(4 * ((cap + 3) & ~3ll)), opF = take(8 * cap), opS = take(8 * cap * W), ofree = take(4 * cap);
  const size_t ohP = take(4 * kNB), ohP2 = take(4 * kNC), ohU = take(4 * kNB), ohU2 = take(4 * kNC);
  const size_t ohF = take(4 * kFpBins), opop = take(4 * (size_t)cfg->B);
  const size_t opopE = take(4 * (size_t)cfg->B), opopF = take(8 * (size_t)cfg->B);
  const size_t opivS = take(8 * (size_t)cfg->B * W);
  const size_t ocand = take(4 * (size_t)(cap + n_dense)), ocE = take(4 * (size_t)(cap + n_dense));
  const size_t ocF = take(8 * (size_t)(cap + n_dense)), ogrp = take(8 * (size_t)kGroup);
  const size_t odE = take(4 * ((n_dense + 3) & ~3ll)), odF = take(8 * n_dense);
  const size_t ohk = take(8ull << hs_log2);
  const size_t ozt = take(8 * L), ost = take(sizeof(PqState)), obest = take(8 * W);
  const int f_log2 = std::min(cfg->H_log2, kFilterMax);
  const size_t oH = take(8ull << cfg->H_log2), ofil = take((1ull << f_log2) / 8);
  char* base = static_cast<char*>(ws_get(ctx, kWsPq0, off));
  if (!base) return LABS_ERR_NOMEM;
  PqBufs b{};
  b.L = L;
  b.W = W;
  b.B = cfg->B;
  b.Tr = cfg->T_r;
  b.width = width;
  b.H_log2 = cfg->H_log2;
  b.cap = cap;
  b.max_exp = cfg->max_expansions;
  b.T_u = cfg->T_u;
  b.hs_log2 = hs_log2;
  b.cand_cap = cap + n_dense;
  b.n_seeds = n_seeds;
  b.pE = reinterpret_cast<int32_t*>(base + opE);
  b.pFp = reinterpret_cast<uint64_t*>(base + opF);
  b.pSeq = reinterpret_cast<uint64_t*>(base + opS);
  b.freeIds = reinterpret_cast<int32_t*>(base + ofree);
  b.hP = reinterpret_cast<unsigned*>(base + ohP);
  b.hP2 = reinterpret_cast<unsigned*>(base + ohP2);
  b.hU = reinterpret_cast<unsigned*>(base + ohU);
  b.hU2 = reinterpret_cast<unsigned*>(base + ohU2);
  b.popId = reinterpret_cast<int32_t*>(base + opop);
  b.popE = reinterpret_cast<int32_t*>(base + opopE);
  b.popF = reinterpret_cast<uint64_t*>(base + opopF);
  b.hF = reinterpret_cast<unsigned*>(base + ohF);
  b.pivSeq = reinterpret_cast<uint64_t*>(base + opivS);
  b.candId = reinterpret_cast<int32_t*>(base + ocand);
  b.cE = reinterpret_cast<int32_t*>(base + ocE);
  b.cF = reinterpret_cast<uint64_t*>(base + ocF);
  b.grp = reinterpret_cast<uint64_t*>(base + ogrp);
  b.dE = reinterpret_cast<int32_t*>(base + odE);
  b.dFp = reinterpret_cast<uint64_t*>(base + odF);
  b.hkey = reinterpret_cast<uint64_t*>(base + ohk);
  b.ztab = reinterpret_cast<uint64_t*>(base + ozt);
  b.st = reinterpret_cast<PqState*>(base + ost);
  b.best_seq = reinterpret_cast<uint64_t*>(base + obest);
  b.H = reinterpret_cast<uint64_t*>(base + oH);
  b.filter = reinterpret_cast<uint32_t*>(base + ofil);
  b.f_log2 = f_log2;
  b.seeds = seeds;

  // a thread takes kPer entries of a pool or survivor pass a turn, four in the passes that probe hash tables
  auto pass_blocks = [&](long long n) {
    return (unsigned)std::max(1ll, std::min<long long>((n + 256 * kPer - 1) / (256 * kPer), (long long)ctx->num_sms * 8));
  };
  const unsigned g_pool = pass_blocks(cap), g_cand_dense = pass_blocks(n_dense);
  const unsigned g_dense =
      (unsigned)std::max(1ll, std::min<long long>((n_dense + 1023) / 1024, (long long)ctx->num_sms * 8));

  // boundary candidates: a bin's share of the pool and the survivors, a thousandth or so (collected by g_cand
  // blocks), but all of them where they lie in an end bin of the window (applied by g_apply blocks, a barrier for
  // every 1,024 of them; half as many blocks: 2 to 7% more for a search outside the window, nothing less inside)
  const unsigned g_cand = (unsigned)std::max(1ll, std::min<long long>((cap + n_dense) / 65536, ctx->num_sms / 2));
  const unsigned g_apply = (unsigned)std::max(1ll, std::min<long long>((cap + n_dense) / 4096, ctx->num_sms));

  // The survivor path, shared by the seeds and every round: dedup, cut, eviction, admission, best, and the next
  // round's beginning.
  auto survivor_path = [&](bool seed, cudaStream_t s) {
    if (seed) {
      pq_dedup_kernel<true><<<g_dense, 256, 0, s>>>(b);
      pq_set_window_kernel<<<1, 1, 0, s>>>(b);
    } else {
      pq_dedup_kernel<false><<<g_dense, 256, 0, s>>>(b);
    }
    pq_cut_kernel<<<std::max(1u, g_cand_dense / 4), kSelThreads, 0, s>>>(b);
    pq_pool_kernel<false><<<g_pool + g_cand_dense, 256, 0, s>>>(b, g_pool);
    pq_boundary_kernel<false><<<g_cand, kSelThreads, 0, s>>>(b);
    pq_boundary_apply_kernel<false><<<g_apply, kSelThreads, 0, s>>>(b);
    if (seed) {
      pq_admit_kernel<true><<<g_dense, 256, 0, s>>>(b);
      pq_finish_kernel<true><<<1, kSelThreads, 0, s>>>(b);
    } else {
      pq_admit_kernel<false><<<g_dense, 256, 0, s>>>(b);
      pq_finish_kernel<false><<<1, kSelThreads, 0, s>>>(b);
    }
    cudaMemsetAsync(b.hkey, 0, 8ull << hs_log2, s);  // the dedup table, for the next round
  };

  // ---- set-up: visited set, pool, histograms, dedup table, Zobrist keys; the seeds go through the
  // survivor path into the empty pool (equal seeds kept once, the cap smallest admitted)
  if (cudaMemsetAsync(b.H, 0xff, 8ull << cfg->H_log2, st) != cudaSuccess ||
      cudaMemsetAsync(b.filter, 0, (1ull << f_log2) / 8, st) != cudaSuccess)
    return LABS_ERR_CUDA;
  if (cudaMemsetAsync(b.hP, 0, 4 * kNB, st) != cudaSuccess || cudaMemsetAsync(b.hP2, 0, 4 * kNC, st) != cudaSuccess ||
      cudaMemsetAsync(b.hU, 0, 4 * kNB, st) != cudaSuccess || cudaMemsetAsync(b.hU2, 0, 4 * kNC, st) != cudaSuccess ||
      cudaMemsetAsync(b.hkey, 0, 8ull << hs_log2, st) != cudaSuccess)
    return LABS_ERR_CUDA;
  pq_ztab_kernel<<<(L + 255) / 256, 256, 0, st>>>(b.ztab, L);
  pq_init_kernel<<<g_pool, 256, 0, st>>>(b);
  pq_seed_kernel<<<(unsigned)std::min<long long>((n_seeds + kPqWarps - 1) / kPqWarps, ctx->num_sms * 16), 32 * kPqWarps,
                   0, st>>>(b, n_seeds);
  survivor_path(true, st);
  if (cudaGetLastError() != cudaSuccess) return LABS_ERR_CUDA;

  // ---- rounds
  const long long max_rounds = (cfg->max_expansions + cfg->B - 1) / cfg->B + 1;
  ExpandPlan ep;
  ep.mma = scan_mma_plan(L, 0, L - 1);
  ep.q = kExpTables;
  ep.x = ep.q + 2 * ep.mma.q_words;
  ep.v = ep.x + ep.mma.x_words;
  ep.words = (ep.v + L / 2 + 1 + 3) / 4 * 4;  // v[1 .. L]
  const size_t exp_smem = sizeof(uint32_t) * (size_t)ep.words * kPqWarps;
  void (*expand)(PqBufs, ExpandPlan) = nullptr;
  int per_sm = 0;
  const int es = by_words((L + 31) >> 5, [&](auto nw) {
    expand = pq_expand_kernel<decltype(nw)::value>;
    return cuda_status(allow_smem(ctx, expand));
  });
  if (es != LABS_OK ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, expand, 32 * kPqWarps, exp_smem) != cudaSuccess || per_sm < 1)
    return LABS_ERR_CUDA;
  const long long exp_items = (long long)cfg->B * (1 + 2 * cfg->T_r);
  const unsigned exp_blocks =
      (unsigned)std::max(1ll, std::min<long long>((exp_items + kPqWarps - 1) / kPqWarps, (long long)ctx->num_sms * per_sm));
  // Every round issues the same launches with the same arguments (a round's sizes and stop state live
  // in device memory), so one round is captured as a CUDA graph and replayed.
  if (!ctx->capture_stream && cudaStreamCreateWithFlags(&ctx->capture_stream, cudaStreamNonBlocking) != cudaSuccess)
    return LABS_ERR_CUDA;
  if (cudaStreamBeginCapture(ctx->capture_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return LABS_ERR_CUDA;
  {
    cudaStream_t cs = ctx->capture_stream;
    pq_pool_kernel<true><<<g_pool, 256, 0, cs>>>(b, g_pool);
    pq_boundary_kernel<true><<<g_cand, kSelThreads, 0, cs>>>(b);
    pq_boundary_apply_kernel<true><<<g_apply, kSelThreads, 0, cs>>>(b);
    expand<<<exp_blocks, 32 * kPqWarps, exp_smem, cs>>>(b, ep);
    survivor_path(false, cs);
  }
  cudaGraph_t round_graph = nullptr;
  cudaError_t ce = cudaStreamEndCapture(ctx->capture_stream, &round_graph);
  cudaGraphExec_t round_exec = nullptr;
  if (ce == cudaSuccess) ce = cudaGraphInstantiate(&round_exec, round_graph, 0);
  if (round_graph) cudaGraphDestroy(round_graph);
  if (ce != cudaSuccess) {
    cudaGetLastError();
    return LABS_ERR_CUDA;
  }
  int* hstop = nullptr;
  if (cudaMallocHost(&hstop, sizeof(int)) != cudaSuccess) {
    cudaGraphExecDestroy(round_exec);
    return LABS_ERR_NOMEM;
  }
  int status = LABS_OK;
  for (long long r = 0; r < max_rounds; r++) {
    if (cudaGraphLaunch(round_exec, st) != cudaSuccess) {
      status = LABS_ERR_CUDA;
      break;
    }
    if ((r & 31) == 31 || r + 1 == max_rounds) {  // poll the stop flag
      if (cudaMemcpyAsync(hstop, &b.st->stop, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
          cudaStreamSynchronize(st) != cudaSuccess) {
        status = LABS_ERR_CUDA;
        break;
      }
      if (*hstop) break;
    }
  }
  pq_write_stats_kernel<<<1, 1, 0, st>>>(b, best_E, stats);
  if (cudaMemcpyAsync(best_seq, b.best_seq, 8 * W, cudaMemcpyDeviceToDevice, st) != cudaSuccess) status = LABS_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) status = LABS_ERR_CUDA;
  cudaFreeHost(hstop);
  cudaGraphExecDestroy(round_exec);
  return status;
}

}  // namespace labsg

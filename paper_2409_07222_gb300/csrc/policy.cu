// policy.cu -- the learned flip-proposal network (labs_policy_*): an optional bias for Algorithm 1's
// neighbour choice.  The paper has no learned component; the exact energy scan stays the judge and a
// zero bias is the plain walk.
//
// Network: features x[0][i] = s_{i+1}, x[1][k] = C_k / sqrt(L-k) (x[1][0] = 0); three Conv1d layers
// (2 -> 64 -> 64 -> 64 channels, kernel 9, padding 4, ReLU); Linear(64 L -> 256, ReLU); Linear(256 -> L).
// Weights are stored in BF16 (an FP32 master copy is kept for the optimizer), all sums accumulate in
// FP32.  Training minimises the weighted cross-entropy over each sample's free positions toward the
// flip it took, with Adam.
//
// Inference (labs_policy_forward, the learned walks) runs on the tensor cores (policy_tc.cu): BF16
// channels-last activations, tcgen05 implicit-GEMM convolutions and a tcgen05 GEMM for the 64 L -> 256
// layer; the first convolution and the 256 -> L layer stay on CUDA cores.
// Training (labs_policy_train_step) runs on CUDA cores with FP32 activations: direct convolution tiles
// (64 output channels x 128 positions per block, 8x8 outputs per thread, input and weight chunks staged
// in shared memory) for the forward pass and the data gradient (the same kernel on flipped, transposed
// weights); an outer-product kernel for the weight gradient; a 128x128-tile GEMM with strided operands for
// the two dense layers and their gradients, its K split over blocks where the output has few tiles.  A
// training step on 512 samples of L = 451 takes 3.11 ms (8.56 ms with one shared load an operand and unsplit tiles); the
// FMAs alone, 63 G, take 1.57 ms at one a lane and clock.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <new>

#include "fma2.cuh"
#include "labs_core.cuh"
#include "labs_internal.h"
#include "policy_tc.h"

struct labs_policy {
  labs_ctx* ctx;
  int L;
  long long n_params;
  long long off[11];  // offsets of w1 b1 w2 b2 w3 b3 W4 b4 W5 b5 (and the end)
  float* master;      // FP32 parameters
  __nv_bfloat16* wbf; // BF16 copy used by every forward pass
  __nv_bfloat16* wT2; // conv2 / conv3 weights flipped and transposed (data gradients)
  __nv_bfloat16* wT3;
  float* grad;
  float* m1;
  float* m2;
  long long step;
  // training activations for up to cap_n samples
  long long cap_n;
  float *x, *h1, *h2, *h3, *a, *logits, *d_logits, *da, *dh_a, *dh_b, *wsum, *loss, *lossv, *wpart, *kpart;
  // tensor-core inference: weight images (rebuilt when tc_stale) and activations for up to cap_i samples
  __nv_bfloat16 *img2, *img3, *W4p;
  bool tc_stale;
  int* tc_err;
  long long cap_i;
  float *xi, *ai, *part;
  __nv_bfloat16 *h1b, *h2b, *h3b;
};

namespace labsg {
namespace {

constexpr int kC = 64, kKW = 9, kPad = 4, kHid = 256;

// ---------------------------------------------------------------------------------------------
// Features
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(128) features_kernel(const uint64_t* __restrict__ seqs, int L, long long n,
                                                       float* __restrict__ x) {
  __shared__ uint32_t bits_all[4][kBitWords];
  uint32_t* bits = bits_all[threadIdx.x >> 5];
  const int lane = lane_id();
  const int W = (L + 63) >> 6;
  for (long long q = (long long)blockIdx.x * 4 + (threadIdx.x >> 5); q < n; q += (long long)gridDim.x * 4) {
    if (lane < kBitWords) {
      const int W32 = (L + 31) >> 5;
      uint32_t v = 0;
      if (lane < W32) {
        const uint64_t w = seqs[q * W + (lane >> 1)];
        v = (lane & 1) ? (uint32_t)(w >> 32) : (uint32_t)w;
        const int rem = L - 32 * lane;
        if (rem < 32) v &= (1u << rem) - 1u;
      }
      bits[lane] = v;
    }
    __syncwarp();
    float* xs = x + q * 2 * L;
    for (int i = lane; i < L; i += 32) xs[i] = ((bits[i >> 5] >> (i & 31)) & 1u) ? 1.f : -1.f;
    if (lane == 0) xs[L] = 0.f;
    for (int k = lane + 1; k < L; k += 32) xs[L + k] = (float)corr_lag(bits, L, k) / sqrtf((float)(L - k));
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------------------------
// Direct convolution: out[n][co][i] = bias[co] + sum_{ci,t} w[co][ci][t] in[n][ci][i+t-4] (ReLU), or
// for a data gradient (no bias) times (mask[n][co][i] > 0).  64 output channels, 128 positions a block.
// ---------------------------------------------------------------------------------------------
constexpr int kCT = 8;  // input channels staged at a time

// Bound: FP32 FMA.  A block takes 16 chunks of eight positions (of one or more samples, so that only a sample's last
// chunk is padded) and all 64 output channels, a thread 8 channels x one chunk: its window of sixteen inputs (four
// 16-byte loads a channel) serves all nine taps, and its eight weights of a tap are two 16-byte broadcasts: 22 shared
// loads for 288 two-wide FMAs.  (With 4 positions a thread it is 21 for 144, and the loads' 512 bytes each are the
// bound.)  512 samples of L = 451: 328 us a layer (26 TFMA/s of 40; 488 us before).  The sum runs over channels, then
// taps, as one chain per output.  The windows lie 20 floats apart: eight threads' 16-byte reads fall into different
// banks.  The results go through shared memory to leave in whole lines.
constexpr int kConvThreads = 128, kChunks = 16, kWin = 20;

template <int CIN>
__global__ void __launch_bounds__(kConvThreads, 4)
    conv_kernel(const float* __restrict__ in, const __nv_bfloat16* __restrict__ w, const float* __restrict__ bias,
                const float* __restrict__ mask, float* __restrict__ out, int L, long long chunks, int relu) {
  constexpr int CH = CIN < kCT ? CIN : kCT;
  constexpr int kRow = kC + 4, kOut = 8 * kChunks + 4;
  constexpr int kBuf = CH * kKW * kRow > kC / 2 * kOut ? CH * kKW * kRow : kC / 2 * kOut;
  __shared__ __align__(16) float in_s[CH][kChunks * kWin];
  __shared__ __align__(16) float buf[kBuf];  // weights [channel, tap][output], at the end half of the results
  __shared__ int sample_s[kChunks], pos_s[kChunks];
  const int ty = threadIdx.x >> 4;  // output channels 8ty .. 8ty+7
  const int tx = threadIdx.x & 15;  // chunk
  if (threadIdx.x < kChunks) {
    const int per = (L + 7) >> 3;
    const long long g = (long long)blockIdx.x * kChunks + threadIdx.x;
    sample_s[threadIdx.x] = g < chunks ? (int)(g / per) : -1;
    pos_s[threadIdx.x] = 8 * (int)(g % per);
  }
  uint64_t acc[4][8];  // output channels in pairs x positions
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 8; b++) acc[a][b] = 0ull;
  __syncthreads();
  for (int c0 = 0; c0 < CIN; c0 += CH) {
    for (int e = threadIdx.x; e < CH * kChunks * 16; e += kConvThreads) {
      const int ci = e / (kChunks * 16), c = (e >> 4) & (kChunks - 1), j = e & 15;
      const int s = sample_s[c], pos = pos_s[c] + j - kPad;
      in_s[ci][c * kWin + j] = (s >= 0 && pos >= 0 && pos < L) ? in[((long long)s * CIN + c0 + ci) * L + pos] : 0.f;
    }
    for (int e = threadIdx.x >> 5; e < (kC / 4) * ((CH * kKW + 7) / 8); e += kConvThreads / 32) {
      // a warp stores eight rows of four output channels: 32 different banks
      const int co = 4 * (e & 15) + ((threadIdx.x & 31) >> 3), r = 8 * (e >> 4) + (threadIdx.x & 7);
      if (r < CH * kKW) buf[r * kRow + co] = __bfloat162float(w[((long long)co * CIN + c0) * kKW + r]);
    }
    __syncthreads();
    for (int ci = 0; ci < CH; ci++) {
      uint64_t iv[16];
#pragma unroll
      for (int v = 0; v < 4; v++) {
        const float4 x = *reinterpret_cast<const float4*>(&in_s[ci][tx * kWin + 4 * v]);
        iv[4 * v] = pack2(x.x, x.x);
        iv[4 * v + 1] = pack2(x.y, x.y);
        iv[4 * v + 2] = pack2(x.z, x.z);
        iv[4 * v + 3] = pack2(x.w, x.w);
      }
#pragma unroll
      for (int t = 0; t < kKW; t++) {
        const float* wr = &buf[(ci * kKW + t) * kRow + 8 * ty];
        const ulonglong2 w0 = *reinterpret_cast<const ulonglong2*>(wr);
        const ulonglong2 w1 = *reinterpret_cast<const ulonglong2*>(wr + 4);
        const uint64_t wv[4] = {w0.x, w0.y, w1.x, w1.y};
#pragma unroll
        for (int a = 0; a < 4; a++)
#pragma unroll
          for (int b = 0; b < 8; b++) ffma2(acc[a][b], wv[a], iv[b + t]);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int half = 0; half < 2; half++) {
    if ((ty >> 2) == half) {
#pragma unroll
      for (int a = 0; a < 4; a++) {
        float* o = &buf[(8 * (ty & 3) + 2 * a) * kOut + 8 * tx];
#pragma unroll
        for (int b = 0; b < 8; b++) {
          const float2 pair = unpack2(acc[a][b]);
          o[b] = pair.x;
          o[kOut + b] = pair.y;
        }
      }
    }
    __syncthreads();
    const int s = sample_s[threadIdx.x >> 3], i = pos_s[threadIdx.x >> 3] + (threadIdx.x & 7);
    if (s >= 0 && i < L) {
#pragma unroll 8
      for (int a = 0; a < kC / 2; a++) {
        const int co = half * (kC / 2) + a;
        const long long o = ((long long)s * kC + co) * L + i;
        float v = buf[a * kOut + threadIdx.x] + (bias ? bias[co] : 0.f);
        if (relu) v = fmaxf(v, 0.f);
        if (mask) v = mask[o] > 0.f ? v : 0.f;
        out[o] = v;
      }
    }
    __syncthreads();
  }
}

// Weight gradient of a convolution for a run of tiles (64 positions of a sample) per block:
// part[block][(co * CIN + ci) * 9 + t] = sum_{n, i in the run} dout[n][co][i] in[n][ci][i+t-4] and part[block][64 * CIN * 9 + co] = sum dout[n][co][i];
// wgrad_reduce_kernel adds the blocks in order (deterministic).
// Bound: FP32 FMA.  A thread holds NA output channels x nine taps of one input channel and takes four positions a
// turn, from a window of twelve inputs and its channels' output gradients, which lie by position so that a 16-byte
// load gives four channels of one: 64 input channels: 32 a block, NA = 8, eleven 16-byte loads for 144 two-wide FMAs (375 us on 512 samples of L = 451, 685 us before).
// Two input channels (the features): NA = 2, and four threads share the positions of a tile.  Each sum runs over the
// positions in order (of a quarter: two input channels, and the bias).
constexpr int kWP = 64;  // positions of a tile

template <int CIN>
__global__ void __launch_bounds__(256, 2) conv_wgrad_kernel(const float* __restrict__ in, const float* __restrict__ dout,
                                                            float* __restrict__ part, int L, long long n,
                                                            int per_block) {
  constexpr bool kFew = CIN == 2;
  constexpr int CH = kFew ? 2 : 32, NA = kFew ? 2 : 8;
  constexpr int kSlices = 256 * NA / (kC * CH);  // threads that share a tile's positions: 1, or 4
  __shared__ __align__(16) float do_s[kWP][kC + 4];
  __shared__ __align__(16) float in_s[CH][kWP + 12];  // rows 12 banks apart: eight rows' 16-byte reads do not collide
  __shared__ float red[4][kC];
  const int c0 = blockIdx.y * CH;
  const int ci = threadIdx.x % CH, co0 = NA * (threadIdx.x / CH % (kC / NA)), slice = threadIdx.x / (CH * (kC / NA));
  uint64_t acc[NA / 2][kKW];  // output channels in pairs x taps
#pragma unroll
  for (int a = 0; a < NA / 2; a++)
#pragma unroll
    for (int t = 0; t < kKW; t++) acc[a][t] = 0ull;
  float db = 0.f;  // of output channel threadIdx.x % 64, a quarter of each tile's positions
  const int tiles = (L + kWP - 1) / kWP;
  const long long ub = (long long)blockIdx.x * per_block, ue = min(n * tiles, ub + per_block);
  for (long long u = ub; u < ue; u++) {
    const long long s = u / tiles;
    const int i0 = (int)(u % tiles) * kWP;
    for (int e = threadIdx.x >> 5; e < (kC / 4) * (kWP / 8); e += 8) {
      // a warp stores eight positions of four channels: 32 different banks
      const int co = 4 * (e >> 3) + ((threadIdx.x & 31) >> 3), j = 8 * (e & 7) + (threadIdx.x & 7);
      do_s[j][co] = (i0 + j < L) ? dout[((s * kC) + co) * L + i0 + j] : 0.f;
    }
    for (int e = threadIdx.x; e < CH * (kWP + 8); e += 256) {
      const int c = e / (kWP + 8), j = e % (kWP + 8);
      const int pos = i0 + j - kPad;
      in_s[c][j] = (pos >= 0 && pos < L) ? in[((s * CIN) + c0 + c) * L + pos] : 0.f;
    }
    __syncthreads();
    const int jn = min(kWP, (L - i0 + 3) & ~3);  // the positions beyond are zero
    const int jb = slice * (kWP / kSlices), je = min(jn, jb + kWP / kSlices);
    for (int j = jb; j < je; j += 4) {
      uint64_t iv[12];
#pragma unroll
      for (int v = 0; v < 3; v++) {
        const float4 x = *reinterpret_cast<const float4*>(&in_s[ci][j + 4 * v]);
        iv[4 * v] = pack2(x.x, x.x);
        iv[4 * v + 1] = pack2(x.y, x.y);
        iv[4 * v + 2] = pack2(x.z, x.z);
        iv[4 * v + 3] = pack2(x.w, x.w);
      }
#pragma unroll
      for (int jj = 0; jj < 4; jj++) {
        uint64_t d2[NA / 2];
        if constexpr (kFew) {
          d2[0] = *reinterpret_cast<const uint64_t*>(&do_s[j + jj][co0]);
        } else {
#pragma unroll
          for (int v = 0; v < NA / 4; v++) {
            const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(&do_s[j + jj][co0 + 4 * v]);
            d2[2 * v] = x.x;
            d2[2 * v + 1] = x.y;
          }
        }
#pragma unroll
        for (int a = 0; a < NA / 2; a++)
#pragma unroll
          for (int t = 0; t < kKW; t++) ffma2(acc[a][t], d2[a], iv[jj + t]);
      }
    }
    if (blockIdx.y == 0) {
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < kWP / 4; j++) sum += do_s[(threadIdx.x >> 6) * (kWP / 4) + j][threadIdx.x & 63];
      db += sum;
    }
    __syncthreads();
  }
  float* pb = part + (long long)blockIdx.x * (kC * CIN * kKW + kC);
  if constexpr (kFew) {
    // the slices' sums in order
    __shared__ float acc_s[kSlices][kC * 2 * kKW];
#pragma unroll
    for (int t = 0; t < kKW; t++) {
      const float2 pair = unpack2(acc[0][t]);
      acc_s[slice][(co0 * 2 + ci) * kKW + t] = pair.x;
      acc_s[slice][((co0 + 1) * 2 + ci) * kKW + t] = pair.y;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kC * 2 * kKW; e += 256) {
      float v = 0.f;
#pragma unroll
      for (int q = 0; q < kSlices; q++) v += acc_s[q][e];
      pb[e] = v;
    }
  } else {
#pragma unroll
    for (int a = 0; a < NA; a++)
#pragma unroll
      for (int t = 0; t < kKW; t++) {
        const float2 pair = unpack2(acc[a >> 1][t]);
        pb[((co0 + a) * CIN + c0 + ci) * kKW + t] = a & 1 ? pair.y : pair.x;
      }
  }
  if (blockIdx.y == 0) {
    red[threadIdx.x >> 6][threadIdx.x & 63] = db;
    __syncthreads();
    if (threadIdx.x < kC)
      pb[kC * CIN * kKW + threadIdx.x] =
          red[0][threadIdx.x] + red[1][threadIdx.x] + red[2][threadIdx.x] + red[3][threadIdx.x];
  }
}

// dw[e] += sum over blocks of part[b][e] (e < 64 CIN 9), db likewise, blocks in order.
__global__ void wgrad_reduce_kernel(const float* __restrict__ part, int blocks, int nw, float* __restrict__ dw,
                                    float* __restrict__ db) {
  const int stride = nw + kC;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < stride; e += gridDim.x * blockDim.x) {
    float v = 0.f;
#pragma unroll 16
    for (int b = 0; b < blocks; b++) v += part[(long long)b * stride + e];
    if (e < nw)
      dw[e] += v;
    else
      db[e - nw] += v;
  }
}

// wT[ci][co][t] = w[co][ci][8 - t]: a convolution with wT maps output gradients to input gradients.
__global__ void flip_transpose_kernel(const float* __restrict__ w, __nv_bfloat16* __restrict__ wT, int cout, int cin) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= cout * cin * kKW) return;
  const int co = e / (cin * kKW), r = e % (cin * kKW), ci = r / kKW, t = r % kKW;
  wT[((long long)ci * cout + co) * kKW + (kKW - 1 - t)] = __float2bfloat16_rn(w[e]);
}

// ---------------------------------------------------------------------------------------------
// GEMM with strided operands: C[m][n] (+)= sum_k A(m,k) B(k,n), A(m,k) = A[m*am + k*ak],
// B(k,n) = B[k*bk + n*bn]; epilogue: + bias[n], ReLU, times (mask[m][n] > 0).  Tiles of 128 x 128, 8 deep, 8 x 8
// outputs a thread (four 16-byte shared loads for 64 FMAs), the next tile's operands loaded while this one is
// multiplied, two buffers and one barrier a tile.  An output of few tiles (fc2 and its gradients) gets its K split over blocks, whose partial
// sums splitk_reduce_kernel adds in order (deterministic).  512 samples, L = 451: W4's gradient 172 us, h3's 206 us
// (322 and 439 us in 64 x 64 tiles of 4 x 4 a thread).
// ---------------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ float ld_as_float(const T* p, long long i);
template <>
__device__ __forceinline__ float ld_as_float<float>(const float* p, long long i) {
  return p[i];
}
template <>
__device__ __forceinline__ float ld_as_float<__nv_bfloat16>(const __nv_bfloat16* p, long long i) {
  return __bfloat162float(p[i]);
}

constexpr int kGT = 128, kGK = 8;

template <typename TA, typename TB>
__global__ void __launch_bounds__(256, 2) gemm_kernel(int M, int N, long long K, const TA* __restrict__ A, long long am,
                                                   long long ak, const TB* __restrict__ B, long long bk, long long bn,
                                                   float* __restrict__ C, long long ldc, const float* __restrict__ bias,
                                                   int relu, const float* __restrict__ mask, int accumulate,
                                                   long long k_part, float* __restrict__ part) {
  __shared__ __align__(16) float As[2][kGK][kGT + 4];
  __shared__ __align__(16) float Bs[2][kGK][kGT + 4];
  const int m0 = blockIdx.y * kGT, n0 = blockIdx.x * kGT;
  const long long kb = blockIdx.z * k_part, ke = min(K, kb + k_part);
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  // a thread fetches kE elements of each tile: along k first where the operand is contiguous in k, else along m or n
  constexpr int kE = kGT * kGK / 256;
  const bool ka = ak == 1, kbf = bk == 1;
  const int a_k = ka ? threadIdx.x % kGK : threadIdx.x / kGT, a_m = ka ? threadIdx.x / kGK : threadIdx.x % kGT;
  const int b_k = kbf ? threadIdx.x % kGK : threadIdx.x / kGT, b_n = kbf ? threadIdx.x / kGK : threadIdx.x % kGT;
  const int a_dk = ka ? 0 : 256 / kGT, a_dm = ka ? 256 / kGK : 0;  // from one element to the next
  const int b_dk = kbf ? 0 : 256 / kGT, b_dn = kbf ? 256 / kGK : 0;
  const long long a_step = a_dk * ak + a_dm * am, b_step = b_dk * bk + b_dn * bn;
  float ra[kE], rb[kE];
  auto fetch = [&](long long k0) {
    const int left = (int)min((long long)kGK, ke - k0);
    const long long ao = (m0 + a_m) * am + (k0 + a_k) * ak, bo = (k0 + b_k) * bk + (n0 + b_n) * bn;
#pragma unroll
    for (int i = 0; i < kE; i++) {
      ra[i] = (m0 + a_m + i * a_dm < M && a_k + i * a_dk < left) ? ld_as_float(A, ao + i * a_step) : 0.f;
      rb[i] = (n0 + b_n + i * b_dn < N && b_k + i * b_dk < left) ? ld_as_float(B, bo + i * b_step) : 0.f;
    }
  };
  uint64_t acc[8][4];  // rows x columns in pairs
#pragma unroll
  for (int a = 0; a < 8; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) acc[a][b] = 0ull;
  fetch(kb);
  int buf = 0;
  for (long long k0 = kb; k0 < ke; k0 += kGK, buf ^= 1) {
#pragma unroll
    for (int i = 0; i < kE; i++) {
      As[buf][a_k + i * a_dk][a_m + i * a_dm] = ra[i];
      Bs[buf][b_k + i * b_dk][b_n + i * b_dn] = rb[i];
    }
    __syncthreads();  // the other buffer is not written before every thread is past the next barrier
    if (k0 + kGK < ke) fetch(k0 + kGK);
#pragma unroll
    for (int kk = 0; kk < kGK; kk++) {
      // rows 4 ty .. and 64 + 4 ty .., columns likewise: a quarter warp's 16-byte reads stay on different banks
      const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][kk][4 * ty]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][kk][64 + 4 * ty]);
      const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][4 * tx]);
      const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][64 + 4 * tx]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const uint64_t bv[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
      for (int a = 0; a < 8; a++) {
        const uint64_t aa = pack2(av[a], av[a]);
#pragma unroll
        for (int b = 0; b < 4; b++) ffma2(acc[a][b], aa, bv[b]);
      }
    }
  }
#pragma unroll
  for (int a = 0; a < 8; a++) {
    const int m = m0 + 4 * ty + (a & 3) + 64 * (a >> 2);
    if (m >= M) continue;
#pragma unroll
    for (int b = 0; b < 8; b++) {
      const int nn = n0 + 4 * tx + (b & 3) + 64 * (b >> 2);
      if (nn >= N) continue;
      const float2 pair = unpack2(acc[a][b >> 1]);
      const float x = b & 1 ? pair.y : pair.x;
      if (part) {
        part[((long long)blockIdx.z * M + m) * N + nn] = x;
        continue;
      }
      const long long o = m * ldc + nn;
      float v = x + (bias ? bias[nn] : 0.f);
      if (relu) v = fmaxf(v, 0.f);
      if (mask) v = mask[o] > 0.f ? v : 0.f;
      C[o] = accumulate ? C[o] + v : v;
    }
  }
}

// The epilogue of a split GEMM: the parts added in order.
__global__ void __launch_bounds__(256) splitk_reduce_kernel(const float* __restrict__ part, int parts, int M, int N,
                                                            float* __restrict__ C, long long ldc,
                                                            const float* __restrict__ bias, int relu,
                                                            const float* __restrict__ mask, int accumulate) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)M * N) return;
  const int m = (int)(e / N), nn = (int)(e % N);
  float v = 0.f;
#pragma unroll 8
  for (int p = 0; p < parts; p++) v += part[(long long)p * M * N + e];
  const long long o = m * ldc + nn;
  v += bias ? bias[nn] : 0.f;
  if (relu) v = fmaxf(v, 0.f);
  if (mask) v = mask[o] > 0.f ? v : 0.f;
  C[o] = accumulate ? C[o] + v : v;
}

// Parts that K is split into: none where the tiles fill the chip, else up to two blocks an SM, at least 128 deep.
// Fixed by the shape, so a result does not depend on the machine's load.  Parts x tiles <= kSplitBlocks bounds the
// partial sums of every shape by kPartFloats.
constexpr int kSplitBlocks = 304;
constexpr size_t kPartFloats = (size_t)kSplitBlocks * kGT * kGT;
inline int gemm_parts(int M, int N, long long K) {
  const long long tiles = (long long)((M + kGT - 1) / kGT) * ((N + kGT - 1) / kGT);
  return (int)std::max(1ll, std::min<long long>(kSplitBlocks / tiles, K / 128));
}

// part: scratch for the partial sums (kPartFloats), or null: K in one piece.
template <typename TA, typename TB>
void gemm(cudaStream_t st, int M, int N, long long K, const TA* A, long long am, long long ak, const TB* B, long long bk,
          long long bn, float* C, long long ldc, const float* bias, int relu, const float* mask, int accumulate,
          float* part = nullptr) {
  const int parts = part ? gemm_parts(M, N, K) : 1;
  const long long k_part = ((K + parts - 1) / parts + kGK - 1) / kGK * kGK;
  const dim3 grid((N + kGT - 1) / kGT, (M + kGT - 1) / kGT, (unsigned)((K + k_part - 1) / k_part));
  gemm_kernel<TA, TB><<<grid, 256, 0, st>>>(M, N, K, A, am, ak, B, bk, bn, C, ldc, bias, relu, mask, accumulate, k_part,
                                            grid.z > 1 ? part : nullptr);
  if (grid.z > 1)
    splitk_reduce_kernel<<<(unsigned)(((long long)M * N + 255) / 256), 256, 0, st>>>(part, (int)grid.z, M, N, C, ldc, bias,
                                                                                     relu, mask, accumulate);
}

// a[n][j] = relu(b4[j] + sum_k h3[n][k] W4[j][k]), K = 64 L, each sum one chain over k: its sign is the mask of the
// gradients, so it is not split as the other long sums are.  512 samples have eight 128 x 128 tiles: here a block
// takes 32 samples x 32 outputs, a thread 2 x 4 of them, which is what the FMA pipe needs to be busy in all of an SM
// and what bounds the kernel by its shared reads instead (eight 16-byte reads for 64 FMAs, the weights kept BF16).
// Chunks of 64 k (K is a multiple) through three cp.async buffers.  L = 451: 345 us for 512 samples (3.81 ms in the
// former 64 x 64 tiles), 2.99 ms for 6,112.  gemm_kernel takes 4.47 ms for anything up to one tile an SM (9,728
// samples), where fc1_kernel would take 4.8 ms: the line lies there.
constexpr int kFT = 32, kFK = 64, kFStages = 3;
constexpr int kFc1Samples = 152 * 64;

__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src));
}

__global__ void __launch_bounds__(128) fc1_kernel(const float* __restrict__ h, const __nv_bfloat16* __restrict__ w,
                                                  const float* __restrict__ bias, float* __restrict__ out, int n,
                                                  long long K) {
  __shared__ __align__(16) float A[kFStages][kFT][kFK + 4];
  __shared__ __align__(16) __nv_bfloat16 B[kFStages][kFT][kFK + 8];
  const int j0 = blockIdx.x * kFT, n0 = blockIdx.y * kFT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = 16 * (warp >> 1) + (lane & 7);         // samples n0 + r, + 8
  const int c = 16 * (warp & 1) + (lane >> 3);         // outputs j0 + c, + 4, + 8, + 12
  auto fetch = [&](int stage, long long k0) {
#pragma unroll
    for (int i = 0; i < kFT * kFK * 4 / 16 / 128; i++) {
      const int e = threadIdx.x + 128 * i, row = e >> 4, q = e & 15;
      copy16(&A[stage][row][4 * q], h + (long long)min(n0 + row, n - 1) * K + k0 + 4 * q);
    }
#pragma unroll
    for (int i = 0; i < kFT * kFK * 2 / 16 / 128; i++) {
      const int e = threadIdx.x + 128 * i, row = e >> 3, q = e & 7;
      copy16(&B[stage][row][8 * q], w + (long long)(j0 + row) * K + k0 + 8 * q);
    }
  };
  float acc[2][4];
#pragma unroll
  for (int a = 0; a < 2; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) acc[a][b] = 0.f;
  const int chunks = (int)(K / kFK);
#pragma unroll
  for (int i = 0; i < kFStages; i++) {
    if (i < chunks) fetch(i, (long long)i * kFK);
    asm volatile("cp.async.commit_group;");
  }
  // the operands of eight k, read while the eight before are multiplied
  struct Eight {
    float4 a[2][2];
    uint4 b[4];
  };
  auto load = [&](Eight& o, int stage, int k) {
#pragma unroll
    for (int a = 0; a < 2; a++)
#pragma unroll
      for (int v = 0; v < 2; v++) o.a[a][v] = *reinterpret_cast<const float4*>(&A[stage][r + 8 * a][k + 4 * v]);
#pragma unroll
    for (int b = 0; b < 4; b++) o.b[b] = *reinterpret_cast<const uint4*>(&B[stage][c + 4 * b][k]);
  };
  Eight e[2];
  asm volatile("cp.async.wait_group %0;" ::"n"(kFStages - 1));
  __syncthreads();
  load(e[0], 0, 0);
  int stage = 0;
  for (int ch = 0; ch < chunks; ch++) {
    const int next = stage + 1 == kFStages ? 0 : stage + 1;
#pragma unroll
    for (int g = 0; g < kFK / 8; g++) {
      if (g + 1 < kFK / 8) {
        load(e[(g + 1) & 1], stage, 8 * (g + 1));
      } else if (ch + 1 < chunks) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kFStages - 2));
        __syncthreads();  // chunk ch + 1 is there, and every thread has read the last of chunk ch
        if (ch + kFStages < chunks) fetch(stage, (long long)(ch + kFStages) * kFK);
        asm volatile("cp.async.commit_group;");
        load(e[(g + 1) & 1], next, 0);
      }
      const Eight& x = e[g & 1];
      float av[2][8], bv[4][8];
#pragma unroll
      for (int a = 0; a < 2; a++)
#pragma unroll
        for (int v = 0; v < 2; v++) {
          av[a][4 * v] = x.a[a][v].x;
          av[a][4 * v + 1] = x.a[a][v].y;
          av[a][4 * v + 2] = x.a[a][v].z;
          av[a][4 * v + 3] = x.a[a][v].w;
        }
#pragma unroll
      for (int b = 0; b < 4; b++) {
        const uint32_t w2[4] = {x.b[b].x, x.b[b].y, x.b[b].z, x.b[b].w};
#pragma unroll
        for (int v = 0; v < 4; v++) {  // BF16 to FP32: the bits, moved up
          bv[b][2 * v] = __uint_as_float(w2[v] << 16);
          bv[b][2 * v + 1] = __uint_as_float(w2[v] & 0xFFFF0000u);
        }
      }
#pragma unroll
      for (int i = 0; i < 8; i++)
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
          for (int b = 0; b < 4; b++) acc[a][b] = fmaf(av[a][i], bv[b][i], acc[a][b]);
    }
    stage = next;
  }
#pragma unroll
  for (int a = 0; a < 2; a++) {
    const int m = n0 + r + 8 * a;
    if (m >= n) continue;
#pragma unroll
    for (int b = 0; b < 4; b++) {
      const int j = j0 + c + 4 * b;
      out[(long long)m * kHid + j] = fmaxf(acc[a][b] + bias[j], 0.f);
    }
  }
}

// column sums: out[j] += sum_i d[i][j]; 32 columns a block, eight strands of rows added in order
__global__ void __launch_bounds__(256) colsum_kernel(const float* __restrict__ d, long long rows, int cols,
                                                     float* __restrict__ out) {
  __shared__ float part[8][32];
  const int lane = threadIdx.x & 31, strand = threadIdx.x >> 5;
  const int j = blockIdx.x * 32 + lane;
  float s = 0.f;
  if (j < cols)
#pragma unroll 16
    for (long long i = strand; i < rows; i += 8) s += d[i * cols + j];
  part[strand][lane] = s;
  __syncthreads();
  if (strand == 0 && j < cols) {
    float v = 0.f;
#pragma unroll
    for (int q = 0; q < 8; q++) v += part[q][lane];
    out[j] += v;
  }
}

// ---------------------------------------------------------------------------------------------
// Loss: weighted cross-entropy over the free positions [lo, hi] (0-based) toward target[n].
// ---------------------------------------------------------------------------------------------
__global__ void wsum_kernel(const float* __restrict__ wgt, long long n, float* __restrict__ out) {
  float s = 0.f;
  for (long long i = threadIdx.x; i < n; i += blockDim.x) s += wgt[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
  __shared__ float ws[32];
  if (lane_id() == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int i = 0; i < (int)(blockDim.x >> 5); i++) t += ws[i];
    *out = t;
  }
}

__global__ void __launch_bounds__(128) loss_kernel(const float* __restrict__ logits, int L, long long n, int lo, int hi,
                                                   const int32_t* __restrict__ target, const float* __restrict__ wgt,
                                                   const float* __restrict__ wsum, float* __restrict__ dlogits,
                                                   float* __restrict__ loss) {
  const int lane = lane_id();
  const float inv = 1.f / *wsum;
  for (long long q = (long long)blockIdx.x * 4 + (threadIdx.x >> 5); q < n; q += (long long)gridDim.x * 4) {
    const float* lg = logits + q * L;
    float mx = -INFINITY;
    for (int i = lo + lane; i <= hi; i += 32) mx = fmaxf(mx, lg[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
    float z = 0.f;
    for (int i = lo + lane; i <= hi; i += 32) z += expf(lg[i] - mx);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(kFull, z, o);
    const int t = target[q];
    const float w = wgt[q] * inv;
    for (int i = lane; i < L; i += 32) {
      float d = 0.f;
      if (i >= lo && i <= hi) d = expf(lg[i] - mx) / z;
      if (i == t) d -= 1.f;
      dlogits[q * L + i] = d * w;
    }
    if (lane == 0) loss[q] = w * (mx + logf(z) - lg[t]);  // summed in order by wsum_kernel
  }
}

// ---------------------------------------------------------------------------------------------
// Adam (FP32 master weights), BF16 copy refreshed
// ---------------------------------------------------------------------------------------------
// (bound by HBM: 30 bytes a parameter; four parameters a thread and turn)
__global__ void __launch_bounds__(256) adam_kernel(float* __restrict__ p, const float* __restrict__ g,
                                                   float* __restrict__ m1, float* __restrict__ m2,
                                                   __nv_bfloat16* __restrict__ wbf, long long n, float lr, float b1,
                                                   float b2, float eps, float c1, float c2) {
  auto update = [&](float& pi, float gi, float& ai, float& vi) {
    const float a = b1 * ai + (1.f - b1) * gi;
    const float v = b2 * vi + (1.f - b2) * gi * gi;
    ai = a;
    vi = v;
    pi = pi - lr * (a / c1) / (sqrtf(v / c2) + eps);
    return __float2bfloat16_rn(pi);
  };
  const long long n4 = n >> 2, stride = (long long)gridDim.x * blockDim.x, first = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (long long i = first; i < n4; i += stride) {
    float4 x = reinterpret_cast<float4*>(p)[i], a = reinterpret_cast<float4*>(m1)[i], v = reinterpret_cast<float4*>(m2)[i];
    const float4 d = reinterpret_cast<const float4*>(g)[i];
    __nv_bfloat162 lo, hi;
    lo.x = update(x.x, d.x, a.x, v.x);
    lo.y = update(x.y, d.y, a.y, v.y);
    hi.x = update(x.z, d.z, a.z, v.z);
    hi.y = update(x.w, d.w, a.w, v.w);
    reinterpret_cast<float4*>(p)[i] = x;
    reinterpret_cast<float4*>(m1)[i] = a;
    reinterpret_cast<float4*>(m2)[i] = v;
    reinterpret_cast<__nv_bfloat162*>(wbf)[2 * i] = lo;
    reinterpret_cast<__nv_bfloat162*>(wbf)[2 * i + 1] = hi;
  }
  for (long long i = 4 * n4 + first; i < n; i += stride) wbf[i] = update(p[i], g[i], m1[i], m2[i]);
}

__global__ void to_bf16_kernel(const float* __restrict__ p, __nv_bfloat16* __restrict__ wbf, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    wbf[i] = __float2bfloat16_rn(p[i]);
}

// SplitMix64 uniform in [-lim, lim] for He-uniform initialisation (purpose 4, parameter index i).
__global__ void init_params_kernel(float* __restrict__ p, long long lo, long long hi, float lim, uint64_t key) {
  for (long long i = lo + (long long)blockIdx.x * blockDim.x + threadIdx.x; i < hi;
       i += (long long)gridDim.x * blockDim.x) {
    const uint64_t r = sm64_at(key, (uint64_t)i);
    const float u = (float)(r >> 40) * (1.f / 16777216.f);  // 24 random bits in [0, 1)
    p[i] = (2.f * u - 1.f) * lim;
  }
}

// Blocks of a weight-gradient launch, `slots` of which the chip holds at a time: runs of equal length, whole rounds
// of blocks, and no sum longer than four samples' positions.
struct WgradPlan {
  unsigned blocks;
  int per_block;
};
inline WgradPlan wgrad_plan(long long n, int L, int slots) {
  const long long tiles = (L + kWP - 1) / kWP, units = n * tiles;
  const long long rounds = (units + slots * 4 * tiles - 1) / (slots * 4 * tiles);
  const long long per = (units + slots * rounds - 1) / (slots * rounds);
  return {(unsigned)((units + per - 1) / per), (int)per};
}
constexpr int kWgradSlots64 = 152, kWgradSlots2 = 304;  // two blocks an SM; 64 channels: two halves

int ensure_acts(labs_policy* P, long long n) {
  if (n <= P->cap_n) return LABS_OK;
  float* bufs[] = {P->x, P->h1, P->h2, P->h3, P->a, P->logits, P->d_logits, P->da, P->dh_a, P->dh_b, P->lossv, P->wpart, P->kpart};
  for (float* b : bufs)
    if (b) cudaFree(b);
  const long long L = P->L;
  const size_t sz[] = {(size_t)n * 2 * L, (size_t)n * kC * L, (size_t)n * kC * L, (size_t)n * kC * L,
                       (size_t)n * kHid, (size_t)n * L, (size_t)n * L, (size_t)n * kHid, (size_t)n * kC * L,
                       (size_t)n * kC * L, (size_t)n, (size_t)kWgradSlots64 * (size_t)((n + 4 * kWgradSlots64 - 1) / (4 * kWgradSlots64)) * (kC * kC * kKW + kC),
                       kPartFloats};
  float** dst[] = {&P->x, &P->h1, &P->h2, &P->h3, &P->a, &P->logits, &P->d_logits, &P->da, &P->dh_a, &P->dh_b,
                   &P->lossv, &P->wpart, &P->kpart};
  for (float** d : dst) *d = nullptr;  // none is left dangling where one of the allocations fails
  P->cap_n = 0;
  for (int i = 0; i < 13; i++)
    if (cudaMalloc(dst[i], sizeof(float) * sz[i]) != cudaSuccess) return LABS_ERR_NOMEM;
  P->cap_n = n;
  return LABS_OK;
}

// Forward pass for n samples already featurised in P->x; logits into `logits` (stride L).
void forward(labs_policy* P, long long n, float* logits, cudaStream_t st) {
  const int L = P->L;
  const long long chunks = n * ((L + 7) / 8);
  const unsigned g = (unsigned)((chunks + kChunks - 1) / kChunks);
  const __nv_bfloat16* w = P->wbf;
  const float* m = P->master;
  conv_kernel<2><<<g, kConvThreads, 0, st>>>(P->x, w + P->off[0], m + P->off[1], nullptr, P->h1, L, chunks, 1);
  conv_kernel<64><<<g, kConvThreads, 0, st>>>(P->h1, w + P->off[2], m + P->off[3], nullptr, P->h2, L, chunks, 1);
  conv_kernel<64><<<g, kConvThreads, 0, st>>>(P->h2, w + P->off[4], m + P->off[5], nullptr, P->h3, L, chunks, 1);
  const long long K4 = (long long)kC * L;
  // a[n][j] = relu(b4[j] + sum_k h3[n][k] W4[j][k]): the same chains either way; the larger tiles once they fill
  // the chip
  if (n < kFc1Samples)
    fc1_kernel<<<dim3(kHid / kFT, (unsigned)((n + kFT - 1) / kFT)), 128, 0, st>>>(P->h3, w + P->off[6], m + P->off[7],
                                                                                P->a, (int)n, K4);
  else
    gemm(st, (int)n, kHid, K4, P->h3, K4, 1ll, w + P->off[6], 1ll, K4, P->a, kHid, m + P->off[7], 1,
         (const float*)nullptr, 0);
  // logits[n][i] = b5[i] + sum_j a[n][j] W5[i][j]
  gemm(st, (int)n, L, (long long)kHid, P->a, (long long)kHid, 1ll, w + P->off[8], 1ll, (long long)kHid, logits, L,
       m + P->off[9], 0, (const float*)nullptr, 0, P->kpart);
}

int ensure_inference(labs_policy* P, long long n) {
  if (n <= P->cap_i) return LABS_OK;
  void* bufs[] = {P->xi, P->ai, P->part, P->h1b, P->h2b, P->h3b};
  for (void* b : bufs)
    if (b) cudaFree(b);
  P->xi = P->ai = P->part = nullptr;
  P->h1b = P->h2b = P->h3b = nullptr;
  P->cap_i = 0;
  const size_t L = (size_t)P->L, act = (size_t)n * L * kC * 2;
  const size_t part_rows = (size_t)tc::tc_dense_splits(kC * P->L) * (size_t)n;  // split-K partial sums
  if (cudaMalloc(&P->xi, 4 * (size_t)n * 2 * L) != cudaSuccess || cudaMalloc(&P->ai, 4 * (size_t)n * kHid) != cudaSuccess ||
      cudaMalloc(&P->part, 4 * part_rows * kHid) != cudaSuccess ||
      cudaMalloc(&P->h1b, act) != cudaSuccess || cudaMalloc(&P->h2b, act) != cudaSuccess ||
      cudaMalloc(&P->h3b, act) != cudaSuccess)
    return LABS_ERR_NOMEM;
  P->cap_i = n;
  return LABS_OK;
}

// Inference for n packed sequences: features, conv1 (CUDA cores, BF16 channels-last out), conv2 and
// conv3 (tcgen05), the 64 L -> 256 layer (tcgen05), the 256 -> L layer (CUDA cores).
int forward_tc(labs_policy* P, const uint64_t* seqs, long long n, float* logits, cudaStream_t st) {
  const int L = P->L;
  const float* m = P->master;
  const int sms = P->ctx->num_sms;
  int s = LABS_OK;
  if (P->tc_stale) {
    s = tc::tc_prepare_weights(m + P->off[2], m + P->off[4], m + P->off[6], L, P->img2, P->img3, P->W4p, st);
    if (s != LABS_OK) return s;
    P->tc_stale = false;
  }
  features_kernel<<<(unsigned)std::min<long long>((n + 3) / 4, 4096), 128, 0, st>>>(seqs, L, n, P->xi);
  s = tc::tc_conv1(P->xi, P->wbf + P->off[0], m + P->off[1], P->h1b, L, n, sms, st);
  if (s == LABS_OK) s = tc::tc_conv64(P->h1b, P->img2, m + P->off[3], P->h2b, L, n, sms, P->tc_err, st);
  if (s == LABS_OK) s = tc::tc_conv64(P->h2b, P->img3, m + P->off[5], P->h3b, L, n, sms, P->tc_err, st);
  if (s == LABS_OK) s = tc::tc_dense(P->h3b, P->W4p, m + P->off[7], P->part, P->ai, n, kC * L, sms, P->tc_err, st);
  if (s != LABS_OK) return s;
  gemm(st, (int)n, L, (long long)kHid, P->ai, (long long)kHid, 1ll, P->wbf + P->off[8], 1ll, (long long)kHid, logits, L,
       m + P->off[9], 0, (const float*)nullptr, 0);
  return cuda_status(cudaGetLastError());
}

}  // namespace

int policy_length(const labs_policy* P) { return P->L; }

}  // namespace labsg

using namespace labsg;

extern "C" {

int labs_policy_param_count(int L, int64_t* n_out) {
  if (L < 2 || L > LABS_MAX_L || !n_out) return LABS_ERR_INVALID_ARG;
  *n_out = (int64_t)kC * 2 * kKW + kC + 2 * ((int64_t)kC * kC * kKW + kC) + (int64_t)kHid * kC * L + kHid +
           (int64_t)L * kHid + L;
  return LABS_OK;
}

int labs_policy_create(labs_ctx* ctx, int L, uint64_t seed, labs_policy** out) {
  if (!ctx || !out || L < 2 || L > LABS_MAX_L) return LABS_ERR_INVALID_ARG;
  *out = nullptr;
  if (cudaSetDevice(ctx->device) != cudaSuccess) return LABS_ERR_CUDA;
  labs_policy* P = new (std::nothrow) labs_policy();
  if (!P) return LABS_ERR_NOMEM;
  P->ctx = ctx;
  P->L = L;
  const long long sizes[10] = {(long long)kC * 2 * kKW, kC, (long long)kC * kC * kKW, kC, (long long)kC * kC * kKW,
                               kC, (long long)kHid * kC * L, kHid, (long long)L * kHid, L};
  long long o = 0;
  for (int i = 0; i < 10; i++) {
    P->off[i] = o;
    o += sizes[i];
  }
  P->off[10] = o;
  P->n_params = o;
  const size_t n = (size_t)o;
  if (cudaMalloc(&P->master, 4 * n) != cudaSuccess || cudaMalloc(&P->wbf, 2 * n) != cudaSuccess ||
      cudaMalloc(&P->grad, 4 * n) != cudaSuccess || cudaMalloc(&P->m1, 4 * n) != cudaSuccess ||
      cudaMalloc(&P->m2, 4 * n) != cudaSuccess || cudaMalloc(&P->wT2, 2 * sizes[2]) != cudaSuccess ||
      cudaMalloc(&P->wT3, 2 * sizes[4]) != cudaSuccess || cudaMalloc(&P->wsum, 8) != cudaSuccess ||
      cudaMalloc(&P->loss, 8) != cudaSuccess || cudaMalloc(&P->img2, 2 * sizes[2]) != cudaSuccess ||
      cudaMalloc(&P->img3, 2 * sizes[4]) != cudaSuccess || cudaMalloc(&P->W4p, 2 * sizes[6]) != cudaSuccess ||
      cudaMalloc(&P->tc_err, sizeof(int)) != cudaSuccess) {
    labs_policy_destroy(P);
    return LABS_ERR_NOMEM;
  }
  cudaMemset(P->master, 0, 4 * n);
  cudaMemset(P->tc_err, 0, sizeof(int));
  P->tc_stale = true;
  cudaMemset(P->m1, 0, 4 * n);
  cudaMemset(P->m2, 0, 4 * n);
  // He-uniform weights, zero biases
  const int fan[10] = {2 * kKW, 0, kC * kKW, 0, kC * kKW, 0, kC * L, 0, kHid, 0};
  for (int i = 0; i < 10; i += 2) {
    const float lim = sqrtf(6.f / (float)fan[i]);
    init_params_kernel<<<256, 256>>>(P->master, P->off[i], P->off[i] + sizes[i], lim, stream_key(seed, 4, (uint64_t)i, 0));
  }
  to_bf16_kernel<<<1024, 256>>>(P->master, P->wbf, o);
  if (cudaDeviceSynchronize() != cudaSuccess) {
    labs_policy_destroy(P);
    return LABS_ERR_CUDA;
  }
  *out = P;
  return LABS_OK;
}

void labs_policy_destroy(labs_policy* P) {
  if (!P) return;
  cudaSetDevice(P->ctx->device);
  cudaDeviceSynchronize();
  void* ptrs[] = {P->master, P->wbf, P->grad, P->m1, P->m2, P->wT2, P->wT3, P->wsum, P->loss, P->x, P->h1,
                  P->h2, P->h3, P->a, P->logits, P->d_logits, P->da, P->dh_a, P->dh_b, P->lossv, P->wpart, P->kpart, P->img2, P->img3,
                  P->W4p, P->tc_err, P->xi, P->ai, P->part, P->h1b, P->h2b, P->h3b};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  delete P;
}

int labs_policy_set_params(labs_policy* P, const float* params, void* stream) {
  if (!P || !params) return LABS_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemcpyAsync(P->master, params, 4 * (size_t)P->n_params, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return LABS_ERR_CUDA;
  to_bf16_kernel<<<1024, 256, 0, st>>>(P->master, P->wbf, P->n_params);
  cudaMemsetAsync(P->m1, 0, 4 * (size_t)P->n_params, st);
  cudaMemsetAsync(P->m2, 0, 4 * (size_t)P->n_params, st);
  P->step = 0;
  P->tc_stale = true;
  return cuda_status(cudaGetLastError());
}

int labs_policy_get_params(labs_policy* P, float* params, void* stream) {
  if (!P || !params) return LABS_ERR_INVALID_ARG;
  return cuda_status(cudaMemcpyAsync(params, P->master, 4 * (size_t)P->n_params, cudaMemcpyDeviceToDevice,
                                     (cudaStream_t)stream));
}

int labs_policy_forward(labs_policy* P, const uint64_t* seqs, int64_t n, float* logits, void* stream) {
  LABS_TRACE("labs_policy_forward");
  if (!P || n < 0 || (n > 0 && (!seqs || !logits))) return LABS_ERR_INVALID_ARG;
  if (n == 0) return LABS_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const long long chunk = 8192;
  int s = ensure_inference(P, std::min<long long>(n, chunk));
  if (s != LABS_OK) return s;
  const int W = (P->L + 63) / 64;
  for (long long b = 0; b < n && s == LABS_OK; b += chunk)
    s = forward_tc(P, seqs + b * W, std::min<long long>(chunk, n - b), logits + b * P->L, st);
  return s;
}

int labs_policy_train_step(labs_policy* P, const uint64_t* seqs, const int32_t* target, const float* weight, int64_t n,
                           int free_lo, int free_hi, float lr, float* loss_out, float* grads_out, void* stream) {
  LABS_TRACE("labs_policy_train_step");
  if (!P || n < 1 || !seqs || !target || !weight || free_lo < 0 || free_hi >= P->L || free_lo > free_hi)
    return LABS_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  int s = ensure_acts(P, n);
  if (s != LABS_OK) return s;
  const int L = P->L;
  const long long K4 = (long long)kC * L;
  features_kernel<<<(unsigned)std::min<long long>((n + 3) / 4, 4096), 128, 0, st>>>(seqs, L, n, P->x);
  forward(P, n, P->logits, st);
  cudaMemsetAsync(P->grad, 0, 4 * (size_t)P->off[6], st);  // W4's part is written whole
  cudaMemsetAsync(P->grad + P->off[7], 0, 4 * (size_t)(P->n_params - P->off[7]), st);
  wsum_kernel<<<1, 1024, 0, st>>>(weight, n, P->wsum);
  loss_kernel<<<(unsigned)std::min<long long>((n + 3) / 4, 4096), 128, 0, st>>>(P->logits, L, n, free_lo, free_hi,
                                                                                  target, weight, P->wsum,
                                                                                  P->d_logits, P->lossv);
  wsum_kernel<<<1, 1024, 0, st>>>(P->lossv, n, P->loss);
  float* g = P->grad;
  const __nv_bfloat16* w = P->wbf;
  // fc2: dW5[i][j] = sum_n dl[n][i] a[n][j]; db5; da[n][j] = sum_i dl[n][i] W5[i][j], masked by a > 0
  gemm(st, L, kHid, n, P->d_logits, 1ll, (long long)L, P->a, (long long)kHid, 1ll, g + P->off[8], kHid,
       (const float*)nullptr, 0, (const float*)nullptr, 1, P->kpart);
  colsum_kernel<<<(L + 31) / 32, 256, 0, st>>>(P->d_logits, n, L, g + P->off[9]);
  gemm(st, (int)n, kHid, (long long)L, P->d_logits, (long long)L, 1ll, w + P->off[8], (long long)kHid, 1ll, P->da, kHid,
       (const float*)nullptr, 0, P->a, 0, P->kpart);
  // fc1: dW4[j][k] = sum_n da[n][j] h3[n][k]; db4; dh3[n][k] = sum_j da[n][j] W4[j][k], masked by h3 > 0
  gemm(st, kHid, (int)K4, n, P->da, 1ll, (long long)kHid, P->h3, K4, 1ll, g + P->off[6], K4, (const float*)nullptr, 0,
       (const float*)nullptr, 0);
  colsum_kernel<<<kHid / 32, 256, 0, st>>>(P->da, n, kHid, g + P->off[7]);
  gemm(st, (int)n, (int)K4, (long long)kHid, P->da, (long long)kHid, 1ll, w + P->off[6], K4, 1ll, P->dh_a, K4,
       (const float*)nullptr, 0, P->h3, 0);
  // conv3: weight gradient from (h2, dc3); data gradient into h2's grid, masked by h2 > 0
  const WgradPlan w64 = wgrad_plan(n, L, kWgradSlots64), w2 = wgrad_plan(n, L, kWgradSlots2);
  const int nw64 = kC * kC * kKW, nw2 = kC * 2 * kKW;
  conv_wgrad_kernel<64><<<dim3(w64.blocks, kC / 32), 256, 0, st>>>(P->h2, P->dh_a, P->wpart, L, n, w64.per_block);
  wgrad_reduce_kernel<<<(nw64 + kC + 255) / 256, 256, 0, st>>>(P->wpart, (int)w64.blocks, nw64, g + P->off[4], g + P->off[5]);
  flip_transpose_kernel<<<(kC * kC * kKW + 255) / 256, 256, 0, st>>>(P->master + P->off[4], P->wT3, kC, kC);
  const long long chunks = n * ((L + 7) / 8);
  const unsigned gc = (unsigned)((chunks + kChunks - 1) / kChunks);
  conv_kernel<64><<<gc, kConvThreads, 0, st>>>(P->dh_a, P->wT3, nullptr, P->h2, P->dh_b, L, chunks, 0);
  // conv2
  conv_wgrad_kernel<64><<<dim3(w64.blocks, kC / 32), 256, 0, st>>>(P->h1, P->dh_b, P->wpart, L, n, w64.per_block);
  wgrad_reduce_kernel<<<(nw64 + kC + 255) / 256, 256, 0, st>>>(P->wpart, (int)w64.blocks, nw64, g + P->off[2], g + P->off[3]);
  flip_transpose_kernel<<<(kC * kC * kKW + 255) / 256, 256, 0, st>>>(P->master + P->off[2], P->wT2, kC, kC);
  conv_kernel<64><<<gc, kConvThreads, 0, st>>>(P->dh_b, P->wT2, nullptr, P->h1, P->dh_a, L, chunks, 0);
  // conv1 (input features need no gradient)
  conv_wgrad_kernel<2><<<dim3(w2.blocks, 1), 256, 0, st>>>(P->x, P->dh_a, P->wpart, L, n, w2.per_block);
  wgrad_reduce_kernel<<<(nw2 + kC + 255) / 256, 256, 0, st>>>(P->wpart, (int)w2.blocks, nw2, g + P->off[0], g + P->off[1]);
  if (grads_out && cudaMemcpyAsync(grads_out, g, 4 * (size_t)P->n_params, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return LABS_ERR_CUDA;
  if (loss_out && cudaMemcpyAsync(loss_out, P->loss, 4, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return LABS_ERR_CUDA;
  if (lr != 0.f) {
    P->step++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)P->step), c2 = 1.f - powf(b2, (float)P->step);
    adam_kernel<<<1024, 256, 0, st>>>(P->master, g, P->m1, P->m2, P->wbf, P->n_params, lr, b1, b2, 1e-8f, c1, c2);
    P->tc_stale = true;
  }
  return cuda_status(cudaGetLastError());
}

int labs_policy_sync_status(labs_policy* P, void* stream) {
  if (!P) return LABS_ERR_INVALID_ARG;
  if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return LABS_ERR_CUDA;
  int e = 0;
  if (cudaMemcpy(&e, P->tc_err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return LABS_ERR_CUDA;
  if (e && cudaMemset(P->tc_err, 0, sizeof(int)) != cudaSuccess) return LABS_ERR_CUDA;
  return e ? LABS_ERR_TIMEOUT : LABS_OK;
}

}  // extern "C"

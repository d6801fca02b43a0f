// Learned surrogate network: a 1-D convolutional operator on the moment fields
// of quasi-1-D tubes, with forward, backward and Adam in hand-written kernels.
// The paper has no learned component.
//
// Architecture (fine sequence of L points, L a multiple of R = 4):
//   unshuffle (L, Cin) -> (L/4, 4 Cin)   [a reshape of the position-major layout]
//   lift      conv k=1, 4 Cin -> C, bias
//   B blocks  h <- h + conv5(relu(conv5(relu(h))))   (C -> C, zero padding)
//   head      conv k=1 of relu(h), C -> 4 Cout, bias
//   shuffle   (L/4, 4 Cout) -> (L, Cout)
// Tensors are FP32 in memory, position-major ([position][channel]); every
// contraction runs on the tensor cores with BF16 operands (converted while a
// tile is staged in shared memory) and FP32 accumulation.
//
//   k_block_tc a whole residual block or its input gradient (tcgen05; C = 128)
//   k_dw_tc    all blocks' weight and bias gradients in one launch (tcgen05; C = 128)
//   k_conv1    one-tap layers (mma.sync m16n8k16)
//   k_conv     the other layers and widths (mma.sync):
//              out[q][m] = (sum_{t,j} A[m][t][j] * act(X[q + s (t - c)][j]) + bias)
//              x (mask > 0) + residual; s = +1 forward, s = -1 input gradient
//              (A = W transposed per tap), zero outside each sequence
//   k_conv_dw  dW[o][t][i] += sum_q dY[q][o] * act(X[q + t - c][i])  (split over q)
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "rpk_internal.h"

namespace {

constexpr int BM = 64, BN = 64, BK = 32, kPadK = 8;  // tile sizes; smem row padding
constexpr int kThreads = 128;                        // 4 warps: 2 (m) x 2 (n), 32 x 32 each
constexpr int R = 4, K5 = 5;

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat16 x = __float2bfloat16_rn(a), y = __float2bfloat16_rn(b);
  return (uint32_t)(*reinterpret_cast<const uint16_t*>(&x)) |
         ((uint32_t)(*reinterpret_cast<const uint16_t*>(&y)) << 16);
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4],
                                         const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

struct ConvArgs {
  const __nv_bfloat16* A;  // [M][taps][Kc]
  const float* X;          // [npos][Kc], position-major
  float* out;              // [npos][M]
  const float* bias;       // [M] or null
  const float* res;        // [npos][M] added, or null
  const float* mask;       // [npos][M]: out *= (mask > 0), or null
  const int2* qseq;        // per position (first position, length) of its sequence, or null
  int M, Kc, taps, sgn, relu_in;
  int npos, seq_len;       // seq_len: common sequence length when qseq is null
};

// One warp-tile step: 2 x 4 mma over one k16 slice of the staged tiles.
__device__ __forceinline__ void warp_mma(const uint16_t (*As)[BK + kPadK],
                                         const uint16_t (*Bs)[BK + kPadK], int wm, int wn,
                                         int k16, float (&acc)[2][4][4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  uint32_t a[2][4], b[4][2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = wm * 32 + i * 16 + g;
    a[i][0] = *reinterpret_cast<const uint32_t*>(&As[r][k16 + 2 * t]);
    a[i][1] = *reinterpret_cast<const uint32_t*>(&As[r + 8][k16 + 2 * t]);
    a[i][2] = *reinterpret_cast<const uint32_t*>(&As[r][k16 + 2 * t + 8]);
    a[i][3] = *reinterpret_cast<const uint32_t*>(&As[r + 8][k16 + 2 * t + 8]);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int n = wn * 32 + j * 8 + g;
    b[j][0] = *reinterpret_cast<const uint32_t*>(&Bs[n][k16 + 2 * t]);
    b[j][1] = *reinterpret_cast<const uint32_t*>(&Bs[n][k16 + 2 * t + 8]);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a[i], b[j]);
}

__global__ void __launch_bounds__(kThreads) k_conv(ConvArgs P) {
  __shared__ __align__(16) uint16_t As[BM][BK + kPadK];
  __shared__ __align__(16) uint16_t Bs[BN][BK + kPadK];
  __shared__ int s_lo[BN], s_len[BN];  // sequence of each position of the tile
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  if (threadIdx.x < BN) {
    const int q = n0 + threadIdx.x;
    int lo = 0, len = 0;
    if (q < P.npos) {
      if (P.qseq) {
        const int2 v = P.qseq[q];
        lo = v.x;
        len = v.y;
      } else {
        lo = (q / P.seq_len) * P.seq_len;
        len = P.seq_len;
      }
    }
    s_lo[threadIdx.x] = lo;
    s_len[threadIdx.x] = len;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, wm = warp >> 1, wn = warp & 1;
  const int c = (P.taps - 1) / 2;
  const int K = P.taps * P.Kc;
  float acc[2][4][4] = {};
  for (int k0 = 0; k0 < K; k0 += BK) {
    // stage A (m, k) and B (n, k) as bf16
    for (int e = threadIdx.x; e < BM * BK / 2; e += kThreads) {
      const int mm = e / (BK / 2), kk = 2 * (e % (BK / 2));
      const int m = m0 + mm;
      float v0 = 0.f, v1 = 0.f;
      if (m < P.M) {
        const int ka = k0 + kk, kb = ka + 1;
        if (ka < K) v0 = __bfloat162float(P.A[(int64_t)m * K + ka]);
        if (kb < K) v1 = __bfloat162float(P.A[(int64_t)m * K + kb]);
      }
      *reinterpret_cast<uint32_t*>(&As[mm][kk]) = pack_bf16(v0, v1);
    }
    for (int e = threadIdx.x; e < BN * BK / 2; e += kThreads) {
      const int nn = e / (BK / 2), kk = 2 * (e % (BK / 2));
      const int q = n0 + nn;
      float v[2] = {0.f, 0.f};
      if (q < P.npos) {
        const int lo = s_lo[nn], len = s_len[nn], l = q - lo;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k = k0 + kk + h;
          if (k < K) {
            const int t = k / P.Kc, j = k - t * P.Kc;
            const int l2 = l + P.sgn * (t - c);
            if (l2 >= 0 && l2 < len) {
              float x = P.X[((int64_t)lo + l2) * P.Kc + j];
              v[h] = P.relu_in ? fmaxf(x, 0.f) : x;
            }
          }
        }
      }
      *reinterpret_cast<uint32_t*>(&Bs[nn][kk]) = pack_bf16(v[0], v[1]);
    }
    __syncthreads();
    warp_mma(As, Bs, wm, wn, 0, acc);
    warp_mma(As, Bs, wm, wn, 16, acc);
    __syncthreads();
  }
  // epilogue
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int m = m0 + wm * 32 + i * 16 + g + (h >= 2 ? 8 : 0);
        const int q = n0 + wn * 32 + j * 8 + 2 * t + (h & 1);
        if (m < P.M && q < P.npos) {
          const int64_t o = (int64_t)q * P.M + m;
          float v = acc[i][j][h];
          if (P.bias) v += P.bias[m];
          if (P.mask && !(P.mask[o] > 0.f)) v = 0.f;
          if (P.res) v += P.res[o];
          P.out[o] = v;
        }
      }
}

// k_conv for one tap (lift, head and the head's input gradient), bound by its
// input and output: a warp takes 16 positions, reads their rows straight into
// fragments (32-byte segments, each element once) and all kMT x 16 output channels
// from weights that the block stages once for all its positions, in k_conv's order
// over k. Positions are the rows of the mma and each pair of 8-column tiles holds 16
// channels interleaved by twos, so that a thread has four consecutive channels of a
// position: one 16-byte store (with its bias) instead of four. 606 K positions: lift
// 340 us in 64 x 64 tiles staged element by element, 141 with channels as rows, 79
// now; head 324, 60 and 59.
struct Conv1Args {
  const __nv_bfloat16* A;  // [M][K]
  const float* X;          // [npos][K]
  float* out;              // [npos][M]
  const float* bias;
  const float* mask;
  int M, K, relu_in, npos;
  int quads;               // rows of out (and mask) are whole 16-byte pieces
};
constexpr int kConv1Threads = 256;

template <int kMT>
__global__ void __launch_bounds__(kConv1Threads) k_conv1(Conv1Args P) {
  extern __shared__ __align__(16) uint16_t c1_smem[];
  __shared__ __align__(16) float c1_bias[kMT * 16];
  const int Kp = (P.K + 15) / 16 * 16, ld = Kp + kPadK;
  const int m0 = blockIdx.y * kMT * 16;
  // a warp takes whole rows of weights, a word of two at a time (K is even, so words are
  // aligned); row 8 j + g of a tile pair holds channel 4 (g / 2) + 2 j + g % 2
#pragma unroll 4
  for (int r = threadIdx.x >> 5; r < kMT * 16; r += kConv1Threads / 32) {
    const int m = m0 + (r & ~15) + 4 * ((r & 7) >> 1) + 2 * ((r >> 3) & 1) + (r & 1);
    const uint32_t* src = reinterpret_cast<const uint32_t*>(P.A + (int64_t)m * P.K);
    for (int k = threadIdx.x & 31; k < ld / 2; k += 32)
      reinterpret_cast<uint32_t*>(c1_smem)[r * (ld / 2) + k] = m < P.M && 2 * k < P.K ? src[k] : 0u;
  }
  if (threadIdx.x < kMT * 16) c1_bias[threadIdx.x] = P.bias && m0 + threadIdx.x < P.M ? P.bias[m0 + threadIdx.x] : 0.f;
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int tiles = (P.npos + 15) / 16;
  for (int tile = blockIdx.x * (kConv1Threads / 32) + warp; tile < tiles; tile += gridDim.x * (kConv1Threads / 32)) {
    const int n0 = tile * 16;
    float acc[kMT][2][4] = {};
#pragma unroll 3
    for (int k0 = 0; k0 < Kp; k0 += 16) {
      uint32_t a[4];
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int q = n0 + j * 8 + g, k = k0 + 2 * t + 8 * h;
          float2 x = make_float2(0.f, 0.f);
          if (q < P.npos && k < P.K) x = *reinterpret_cast<const float2*>(P.X + (int64_t)q * P.K + k);
          if (P.relu_in) x.x = fmaxf(x.x, 0.f), x.y = fmaxf(x.y, 0.f);
          a[j + 2 * h] = pack_bf16(x.x, x.y);
        }
#pragma unroll
      for (int i = 0; i < kMT; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const uint16_t* r = c1_smem + (i * 16 + 8 * j + g) * ld + k0 + 2 * t;
          const uint32_t b[2] = {*reinterpret_cast<const uint32_t*>(r), *reinterpret_cast<const uint32_t*>(r + 8)};
          mma_bf16(acc[i][j], a, b);
        }
    }
#pragma unroll
    for (int i = 0; i < kMT; ++i) {
      const int c = i * 16 + 4 * t;  // first of this thread's four channels
      const float4 b = *reinterpret_cast<const float4*>(c1_bias + c);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int q = n0 + 8 * h + g;
        if (q >= P.npos || m0 + c >= P.M) continue;
        const int64_t o = (int64_t)q * P.M + m0 + c;
        float v[4] = {acc[i][0][2 * h] + b.x, acc[i][0][2 * h + 1] + b.y, acc[i][1][2 * h] + b.z,
                      acc[i][1][2 * h + 1] + b.w};
        if (P.quads) {
          if (P.mask) {
            const float4 m = *reinterpret_cast<const float4*>(P.mask + o);
            if (!(m.x > 0.f)) v[0] = 0.f;
            if (!(m.y > 0.f)) v[1] = 0.f;
            if (!(m.z > 0.f)) v[2] = 0.f;
            if (!(m.w > 0.f)) v[3] = 0.f;
          }
          *reinterpret_cast<float4*>(P.out + o) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
          for (int l = 0; l < 4; ++l)
            if (m0 + c + l < P.M) {
              if (P.mask && !(P.mask[o + l] > 0.f)) v[l] = 0.f;
              P.out[o + l] = v[l];
            }
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Tensor-core (tcgen05) path of a residual block, both convolutions (Co = Ci =
// 128, 5 taps) in one kernel; the same kernel runs the block's input gradient:
//   forward:   z = conv(relu(x); W1) + b1,    out = (conv(relu(z); W2) + b2) + x
//   gradient:  z = conv^T(x; W1) (m1 > 0),    out = conv^T(z; W2) (m2 > 0) + x
// (z is stored when zout is given: training needs it.) One persistent CTA per SM
// walks over tiles of 124 output positions of one sequence; the tile's 128 rows
// of z never leave the SM between the two convolutions. Roles:
//   producers (warps 8-15) load tile i's 132 input rows into registers while
//     the MMAs of tile i - 1 still read B1, then store them (activation, BF16);
//   a loader thread (warp 16) keeps a ring of five 16 KB slots filled with half
//     taps of weights, which lie in memory in the operand's own layout: one bulk
//     copy each;
//   an issuing thread (warp 17): 40 MMAs (M 128 positions, N 128 channels, K 16)
//     per convolution in the order conv1(0), conv1(1), conv2(0), conv1(2),
//     conv2(1), ..., so that the tensor cores work on conv1(i + 1) while the
//     epilogue turns conv1(i) into conv2(i)'s operand;
//   the epilogue (warps 0-7; TMEM lane = position, so that a thread holds 64
//     consecutive channels of one position): e1(i) moves the first accumulator
//     through bias, mask and activation into B2 (16-byte BF16 stores), then e2(i - 1)
//     adds bias, mask and residual to the second one. Each warp owns 32 positions x
//     64 channels of the tile: its residual rows were copied into its own staging
//     block (cp.async) a tile earlier, and its output rows leave from there two
//     whole rows an instruction, so no warp waits for another. Staging rows are 16
//     bytes longer than their data: threads reading 16 bytes of 32 rows hit
//     distinct banks.
// The operand of tap t is the staged tile seen from row t (forward) or 4 - t
// (gradient): in the interleaved no-swizzle layout (rows 16 bytes apart inside
// each 8-column chunk) a row shift is a start-address offset. Every element is
// accumulated in the same order as one convolution per launch did.
// Bound: two launches per block moved 2.5 KB a position (z written and read, the
// residual read again) at 3.5-5 TB/s with the epilogue's residual latency in the
// way; one moves 1 KB, and the weights' 320 KB per tile come from L2. What is left
// is shared memory: 8 KB per MMA, 320 KB of weights and the epilogue's rows make
// 1.35 MB a tile, 10.5 k of the tile's 12.5 k cycles at 128 bytes a cycle. 606 K
// positions: 2 x 178 us a block in two launches, 225 us in one; 32 crops of 1024
// points (training, 96 tiles): 2 x 29.9 us -> 18.9 us. Tried: residual rows loaded
// in the epilogue instead of copied ahead, 1715 against 1685 us a forward pass;
// TMEM lane = channel with 2-byte stores into B2 and whole-block staging
// barriers, 1863; CTA pairs (M 256 over two SMs, each with half of the weights), 225 us a
// block as before -- 450 with cluster-scope releases, which wait for the SM's global
// stores -- since the epilogue's 10 k cycles a tile are the next bound; its residual
// and output rows as bulk copies of 256 bytes, 223 alone and 220 with pairs; e1 moved
// to the producers' warps, 260 with pairs.
constexpr int TC_M = 128, TC_N = 128, TC_KC = 128, TC_TAPS = 5;
constexpr int TC_OUT = TC_N - (TC_TAPS - 1);               // 124 output positions per tile
constexpr int TC_ROWS = TC_N + TC_TAPS - 1;                // 132 staged rows
constexpr int TC_K = TC_TAPS * TC_KC;                      // 640
constexpr uint32_t TC_W_LBO = TC_N * 16;                   // bytes between 8-wide k chunks of a tap's weights
// bytes between 8-wide k chunks of B1 and B2: one row more than staged, so that
// the producers' 16-byte stores of one row's consecutive chunks fall in distinct
// shared-memory banks (2128 / 4 = 532 = 20 mod 32)
constexpr uint32_t TC_B_LBO = (TC_ROWS + 1) * 16;
constexpr uint32_t TC_B_BYTES = (TC_KC / 8) * TC_B_LBO;    // 34048
constexpr uint32_t TC_HALF_BYTES = TC_N * TC_KC;           // 16384: half a tap's weights (64 k)
constexpr int TC_RING = 5;
constexpr int TC_WCH = 64;                                 // channels of an epilogue warp's block
constexpr uint32_t TC_S_LD = TC_WCH * 4 + 16;              // bytes between its staged rows
constexpr uint32_t TC_SW_BYTES = 32 * TC_S_LD;             // staging of a warp
constexpr uint32_t TC_W_OFF = 0;
constexpr uint32_t TC_S_OFF = TC_W_OFF + TC_RING * TC_HALF_BYTES;
constexpr uint32_t TC_B1_OFF = TC_S_OFF + 8 * TC_SW_BYTES;
constexpr uint32_t TC_B2_OFF = TC_B1_OFF + TC_B_BYTES;
constexpr uint32_t TC_BAR_OFF = TC_B2_OFF + TC_B_BYTES;
constexpr uint32_t TC_BIAS_OFF = TC_BAR_OFF + 256;         // 17 mbarriers + TMEM address, then both biases
constexpr uint32_t TC_SMEM = TC_BIAS_OFF + 2 * TC_N * 4;
static_assert(TC_SMEM <= 227 * 1024, "tensor-core tiles exceed shared memory");
static_assert(TC_S_OFF % 128 == 0 && TC_B1_OFF % 128 == 0 && TC_BIAS_OFF % 16 == 0, "operand alignment");
constexpr int TC_EPI = 256;                                // epilogue threads (warps 0-7)
constexpr int TC_PROD = 256;                               // producer threads (warps 8-15)
constexpr int TC_THREADS = TC_EPI + TC_PROD + 64;          // + loader and issuing warps
constexpr int TC_COLS = 4 * TC_N;                          // two accumulators per convolution
constexpr long long TC_WAIT_LIMIT = 1ll << 22;             // mbarrier polls before giving up

struct BlockArgs {
  const __nv_bfloat16* w1;  // taps' weights, [5][16 chunks of 8 k][128 channels][8]
  const __nv_bfloat16* w2;
  const float* x;           // [npos][128] input, and the residual
  float* zout;              // [npos][128], or null
  float* out;               // [npos][128]
  const float* b1;          // biases, or null
  const float* b2;
  const float* m1;          // masks (> 0 keeps), or null
  const float* m2;
  const int4* tiles;        // per tile (q0, count, sequence start, sequence length), or null
  int ntiles, seq_len, tiles_per_seq, sgn, relu;
  unsigned* error;          // set to 1 when an mbarrier wait gives up
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// tcgen05 shared-memory matrix descriptor: start, leading (k-chunk) and stride
// (8-row group) byte offsets, descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24.
constexpr uint32_t TC_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TC_N >> 3) << 17) |
                              ((uint32_t)(TC_M >> 4) << 24);

__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
  for (long long it = 0; it < TC_WAIT_LIMIT; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void tc_tile(const BlockArgs& P, int tile, int& q0, int& cnt, int& lo, int& len) {
  if (P.tiles) {
    const int4 d = P.tiles[tile];
    q0 = d.x, cnt = d.y, lo = d.z, len = d.w;
  } else {
    const int sq = tile / P.tiles_per_seq, part = tile - sq * P.tiles_per_seq;
    lo = sq * P.seq_len;
    len = P.seq_len;
    q0 = lo + part * TC_OUT;
    cnt = min(TC_OUT, len - part * TC_OUT);
  }
}

// 16 consecutive accumulator columns of this thread's TMEM lane (32x32b shape)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}

// 32 consecutive accumulator columns
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
}

// Announce the bytes that bulk copies will complete on bar (its one arrival).
__device__ __forceinline__ void bulk_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// Bulk copy of bytes into shared memory, counted on bar.
__device__ __forceinline__ void bulk_load(uint32_t bar, uint32_t dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// mbarriers of k_block_tc
enum {
  kB1Full = 0,   // producers: x tile staged
  kB1Free,       // MMAs of conv1 done with it
  kB2Full,       // epilogue: z tile staged (its TMEM reads done)
  kAcc1,         // + 0, 1: conv1's accumulator ready
  kAcc2 = kAcc1 + 2,  // + 0, 1: conv2's accumulator ready, B2 free
  kWFull = kAcc2 + 2,
  kWFree = kWFull + TC_RING,
  kBars = kWFree + TC_RING
};
static_assert(kBars * 8 + 8 <= 256, "barrier space");

__global__ void __launch_bounds__(TC_THREADS, 1) k_block_tc(BlockArgs P) {
  extern __shared__ __align__(1024) unsigned char tc_smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(tc_smem + TC_BAR_OFF);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tc_smem + TC_BAR_OFF + 8 * kBars);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t base = smem_u32(tc_smem), bar0 = smem_u32(bars);
  auto bar = [&](int k) { return bar0 + 8u * (uint32_t)k; };

  // the next kernel's CTAs may take the SMs this grid leaves free
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(TC_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int k = 0; k < kBars; ++k) {
      const int n = k == kB1Full ? TC_PROD : k == kB2Full ? TC_EPI : 1;
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar(k)), "r"(n) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // parameters (weights and biases) are never written while kernels of one pass
  // follow each other: they are read before the previous kernel has finished
  float* sbias = reinterpret_cast<float*>(tc_smem + TC_BIAS_OFF);
  if (tid < 2 * TC_N) {
    const float* b = tid < TC_N ? P.b1 : P.b2;
    sbias[tid] = b ? b[tid & (TC_N - 1)] : 0.f;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  // tiles of this CTA: blockIdx.x + i gridDim.x, i < n
  const int n = (P.ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  bool ok = true;

  if (warp == 16) {
    if (lane == 0) {
      int r = 0;
      for (int i = 0; i <= n && ok; ++i)
        for (int c = 0; c < 2 && ok; ++c) {
          if (c == 0 ? i == n : i == 0) continue;
          const unsigned char* w = reinterpret_cast<const unsigned char*>(c == 0 ? P.w1 : P.w2);
          for (int t = 0; t < 2 * TC_TAPS && ok; ++t, ++r) {
            const int slot = r % TC_RING;
            if (r >= TC_RING) ok = mbar_wait(bar(kWFree + slot), ((r / TC_RING) - 1) & 1);
            if (ok) {
              bulk_expect(bar(kWFull + slot), TC_HALF_BYTES);
              bulk_load(bar(kWFull + slot), base + TC_W_OFF + slot * TC_HALF_BYTES, w + t * TC_HALF_BYTES, TC_HALF_BYTES);
            }
          }
        }
      if (!ok) atomicOr(P.error, 1u);
      // copies still in flight land before the CTA's shared memory is released
      for (int k = max(0, r - TC_RING); k < r; ++k) mbar_wait(bar(kWFull + k % TC_RING), (k / TC_RING) & 1);
    }
  } else if (warp == 17) {
    // the whole warp runs the loop, so that descriptors stay in uniform
    // registers; one elected lane issues
    uint32_t one;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(one));
    int r = 0;
    auto commit = [&](uint32_t b) {
      asm volatile(
          "{\n .reg .pred e;\n setp.ne.b32 e, %1, 0;\n"
          " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(b),
          "r"(one)
          : "memory");
    };
    auto conv = [&](uint32_t b_base, uint32_t d) {
#pragma unroll 2
      for (int t = 0; t < 2 * TC_TAPS; ++t, ++r) {  // half taps
        const int slot = r % TC_RING;
        if (!mbar_wait(bar(kWFull + slot), (r / TC_RING) & 1)) return false;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int tap = t >> 1, row0 = P.sgn > 0 ? tap : TC_TAPS - 1 - tap;
        const uint64_t ad = tc_desc(b_base + (uint32_t)((t & 1) * 8) * TC_B_LBO + (uint32_t)row0 * 16, TC_B_LBO, 128);
        const uint64_t bd = tc_desc(base + TC_W_OFF + slot * TC_HALF_BYTES, TC_W_LBO, 128);
#pragma unroll
        for (int k = 0; k < TC_KC / 32; ++k) {
          // the address field counts 16 bytes
          asm volatile(
              "{\n .reg .pred p, e;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 e, %5, 0;\n"
              " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
              "l"(ad + (uint64_t)(2 * k * (TC_B_LBO / 16))), "l"(bd + (uint64_t)(2 * k * (TC_W_LBO / 16))),
              "r"(TC_IDESC), "r"((uint32_t)(t | k)), "r"(one)
              : "memory");
        }
        commit(bar(kWFree + slot));
      }
      return true;
    };
    for (int i = 0; i <= n && ok; ++i) {
      if (i < n) {
        // accumulator i % 2 was read by e1(i - 2), before conv2(i - 2) was issued
        ok = mbar_wait(bar(kB1Full), i & 1) && conv(base + TC_B1_OFF, tmem + (uint32_t)((i & 1) * TC_N));
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        commit(bar(kB1Free));
        commit(bar(kAcc1 + (i & 1)));
      }
      if (i >= 1) {
        const int j = i - 1;
        // accumulator j % 2 was read by e2(j - 2), before e1(j) staged B2
        ok = mbar_wait(bar(kB2Full), j & 1) && conv(base + TC_B2_OFF, tmem + (uint32_t)((2 + (j & 1)) * TC_N));
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        commit(bar(kAcc2 + (j & 1)));
      }
    }
    if (!ok && lane == 0) atomicOr(P.error, 1u);
  } else if (tid >= TC_EPI) {
    // producers: 2112 (row, 8-channel chunk) elements, at most 9 per thread;
    // consecutive threads take consecutive 32-byte chunks of a row
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int ptid = tid - TC_EPI;
    constexpr int kElems = TC_ROWS * (TC_KC / 8);
    constexpr int kBatch = (kElems + TC_PROD - 1) / TC_PROD;
    for (int i = 0; i < n && ok; ++i) {
      int q0, cnt, lo, len;
      tc_tile(P, (int)blockIdx.x + i * (int)gridDim.x, q0, cnt, lo, len);
      float4 f[kBatch][2];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int e = ptid + u * TC_PROD;
        const int r = e / (TC_KC / 8), c = e % (TC_KC / 8);
        const int q = q0 - (TC_TAPS - 1) + r;
        f[u][0] = f[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e < kElems && q >= lo && q < lo + len) {
          const float4* src = reinterpret_cast<const float4*>(P.x + (int64_t)q * TC_KC + 8 * c);
          f[u][0] = src[0];
          f[u][1] = src[1];
        }
      }
      if (i >= 1) ok = __all_sync(0xffffffffu, mbar_wait(bar(kB1Free), (i - 1) & 1));
      if (!ok) break;
      unsigned char* sB = tc_smem + TC_B1_OFF;
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int e = ptid + u * TC_PROD;
        if (e >= kElems) break;
        const int r = e / (TC_KC / 8), c = e % (TC_KC / 8);
        float4 f0 = f[u][0], f1 = f[u][1];
        if (P.relu) {
          f0.x = fmaxf(f0.x, 0.f), f0.y = fmaxf(f0.y, 0.f), f0.z = fmaxf(f0.z, 0.f), f0.w = fmaxf(f0.w, 0.f);
          f1.x = fmaxf(f1.x, 0.f), f1.y = fmaxf(f1.y, 0.f), f1.z = fmaxf(f1.z, 0.f), f1.w = fmaxf(f1.w, 0.f);
        }
        *reinterpret_cast<uint4*>(sB + c * TC_B_LBO + r * 16) =
            make_uint4(pack_bf16(f0.x, f0.y), pack_bf16(f0.z, f0.w), pack_bf16(f1.x, f1.y),
                       pack_bf16(f1.z, f1.w));
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(bar(kB1Full));
    }
    if (!ok && lane == 0) atomicOr(P.error, 1u);
  } else {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int quad = warp & 3, c0 = (warp >> 2) * TC_WCH;  // positions 32 quad .., channels c0 ..
    const int row = quad * 32 + lane;
    const uint32_t lanes = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0;
    const uint32_t s_base = base + TC_S_OFF + warp * TC_SW_BYTES;
    float* srow = reinterpret_cast<float*>(tc_smem + TC_S_OFF + warp * TC_SW_BYTES + lane * TC_S_LD);
    // lane's 16-byte piece of a row pair: rows 2 k + (lane / 16), piece lane % 16
    const int prow = lane >> 4, piece = lane & 15;
    // residual rows of tile i, asynchronously
    auto load_residual = [&](int i) {
      int q0, cnt, lo, len;
      tc_tile(P, (int)blockIdx.x + i * (int)gridDim.x, q0, cnt, lo, len);
      const float* src = P.x + (int64_t)(q0 + quad * 32 + prow) * TC_M + c0 + 4 * piece;
      const uint32_t dst = s_base + prow * TC_S_LD + 16 * piece;
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (quad * 32 + 2 * k + prow < cnt)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 2 * k * TC_S_LD),
                       "l"(src + 2 * k * TC_M)
                       : "memory");
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // bit c: channel c0 + c of position q is masked out (q inside its sequence)
    auto masked = [&](const float* mask, int64_t q) {
      uint64_t drop = 0;
      const float4* src = reinterpret_cast<const float4*>(mask + q * TC_M + c0);
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        float4 f[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) f[k] = src[8 * g + k];
        uint32_t bits = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          bits |= ((f[k].x > 0.f ? 0u : 1u) | (f[k].y > 0.f ? 0u : 2u) | (f[k].z > 0.f ? 0u : 4u) |
                   (f[k].w > 0.f ? 0u : 8u))
                  << (4 * k);
        drop |= (uint64_t)bits << (32 * g);
      }
      return drop;
    };
    if (n > 0) load_residual(0);
    for (int i = 0; i <= n && ok; ++i) {
      if (i < n) {
        // e1(i): row q0 - 2 + row of z
        int q0, cnt, lo, len;
        tc_tile(P, (int)blockIdx.x + i * (int)gridDim.x, q0, cnt, lo, len);
        const int q = q0 - 2 + row;
        const bool in = q >= lo && q < lo + len;  // else zero padding of the second convolution
        const uint64_t drop = P.m1 ? masked(P.m1, min(max(q, lo), lo + len - 1)) : 0;
        ok = mbar_wait(bar(kAcc1 + (i & 1)), (i >> 1) & 1);
        // conv2(i - 1) has read B2
        if (ok && i >= 1) ok = mbar_wait(bar(kAcc2 + ((i - 1) & 1)), ((i - 1) >> 1) & 1);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        unsigned char* zb = tc_smem + TC_B2_OFF + (c0 / 8) * TC_B_LBO + row * 16;
        float4* zo = P.zout && row >= 2 && row < 2 + cnt ? reinterpret_cast<float4*>(P.zout + (int64_t)q * TC_M + c0)
                                                         : nullptr;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          uint32_t v[32];
          tmem_ld32(lanes + (uint32_t)((i & 1) * TC_N + g * 32), v);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          const uint32_t d32 = (uint32_t)(drop >> (32 * g));
          const float4* b4 = reinterpret_cast<const float4*>(sbias + c0 + g * 32);
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const float4 b = b4[k];
            float f[4] = {__uint_as_float(v[4 * k]) + b.x, __uint_as_float(v[4 * k + 1]) + b.y,
                          __uint_as_float(v[4 * k + 2]) + b.z, __uint_as_float(v[4 * k + 3]) + b.w};
#pragma unroll
            for (int l = 0; l < 4; ++l)
              if (!in || ((d32 >> (4 * k + l)) & 1u)) f[l] = 0.f;
            if (zo) zo[8 * g + k] = make_float4(f[0], f[1], f[2], f[3]);
            if (P.relu) {
#pragma unroll
              for (int l = 0; l < 4; ++l) f[l] = fmaxf(f[l], 0.f);
            }
            v[2 * k] = pack_bf16(f[0], f[1]);
            v[2 * k + 1] = pack_bf16(f[2], f[3]);
          }
#pragma unroll
          for (int c = 0; c < 4; ++c)
            *reinterpret_cast<uint4*>(zb + (4 * g + c) * TC_B_LBO) =
                make_uint4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        mbar_arrive(bar(kB2Full));
      } else if (n > 0) {
        ok = __all_sync(0xffffffffu, mbar_wait(bar(kAcc2 + ((n - 1) & 1)), ((n - 1) >> 1) & 1));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      }
      if (i >= 1) {
        // e2(i - 1)
        const int j = i - 1;
        int q0, cnt, lo, len;
        tc_tile(P, (int)blockIdx.x + j * (int)gridDim.x, q0, cnt, lo, len);
        const uint64_t drop = P.m2 ? masked(P.m2, min(q0 + row, lo + len - 1)) : 0;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();  // every lane's pieces have landed
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          uint32_t v[32];
          tmem_ld32(lanes + (uint32_t)((2 + (j & 1)) * TC_N + g * 32), v);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          const uint32_t d32 = (uint32_t)(drop >> (32 * g));
          const float4* b4 = reinterpret_cast<const float4*>(sbias + TC_N + c0 + g * 32);
          float4* s4 = reinterpret_cast<float4*>(srow + g * 32);
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const float4 b = b4[k];
            float4 r = s4[k];
            float f[4] = {__uint_as_float(v[4 * k]) + b.x, __uint_as_float(v[4 * k + 1]) + b.y,
                          __uint_as_float(v[4 * k + 2]) + b.z, __uint_as_float(v[4 * k + 3]) + b.w};
#pragma unroll
            for (int l = 0; l < 4; ++l)
              if ((d32 >> (4 * k + l)) & 1u) f[l] = 0.f;
            r.x = f[0] + r.x, r.y = f[1] + r.y, r.z = f[2] + r.z, r.w = f[3] + r.w;
            s4[k] = r;
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        const float4* from = reinterpret_cast<const float4*>(tc_smem + TC_S_OFF + warp * TC_SW_BYTES +
                                                             prow * TC_S_LD + 16 * piece);
        float* to = P.out + (int64_t)(q0 + quad * 32 + prow) * TC_M + c0 + 4 * piece;
#pragma unroll
        for (int k = 0; k < 16; ++k)
          if (quad * 32 + 2 * k + prow < cnt)
            *reinterpret_cast<float4*>(to + 2 * k * TC_M) = from[2 * k * (TC_S_LD / 16)];
        __syncwarp();  // read out before the next residual lands there
        if (i < n) load_residual(i);
      }
    }
    if (!ok && lane == 0) atomicOr(P.error, 1u);
    // residual copies still in flight after a wait that gave up
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_COLS) : "memory");
}

// ---------------------------------------------------------------------------
// Weight and bias gradients of all residual-block convolutions in one launch
// (tcgen05; Co = Ci = 128, 5 taps, ReLU inputs):
//   dW[o][t][i] += sum_q dY[q][o] relu(X[q + t - 2][i]),  db[o] += sum_q dY[q][o].
// The reduction runs over positions, so both operands are MN-major: a tile of
// 128 positions is staged as in k_block_tc (8-channel chunks, rows 16 bytes
// apart), which read with channels as M or N and rows as K is the no-swizzle
// MN-major layout (SBO = chunk stride, LBO = 128 bytes between groups of 8
// rows), and the tap shift is again a start-address offset of 16 bytes a row.
// A CTA owns (layer, half of the input channels, share of the tiles): M 128, N
// 64 per tap, 5 x 64 TMEM columns. All 512 threads stage tile i (loads, ReLU,
// BF16, stores) while the 40 MMAs of tile i - 1 run from the other buffer; the
// accumulators are added to dW once per CTA by 16-byte atomics, and the bias
// gradient is the FP32 column sums of dY on their way to shared memory.
// Bound: reading dY and X (FP32) once per half. One launch after the whole
// input-gradient chain fills the chip where a layer alone gave 10 x 2 x 29 small
// tiles re-staged by every block: 12 launches of 99 us (mma.sync) and 12 of
// 22.5 us (bias) for 32 crops of 1024 points became one of 41 us.
constexpr int DW_N = 64;                                    // input channels per CTA
constexpr int DW_THREADS = 512;
constexpr uint32_t DW_A_STRIDE = (TC_N + 1) * 16;           // dY: bytes between 8-channel chunks
constexpr uint32_t DW_B_STRIDE = (TC_ROWS + 1) * 16;        // X
constexpr uint32_t DW_A_BYTES = (TC_M / 8) * DW_A_STRIDE;   // 33024
constexpr uint32_t DW_B_BYTES = (DW_N / 8) * DW_B_STRIDE;   // 17024
constexpr uint32_t DW_BUF = DW_A_BYTES + DW_B_BYTES;
constexpr uint32_t DW_BAR_OFF = 2 * DW_BUF;
constexpr uint32_t DW_SMEM = DW_BAR_OFF + 64;
constexpr int DW_COLS = 512;                                // 5 x 64 accumulator columns, a power of two
constexpr uint32_t DW_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                              ((uint32_t)(DW_N >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);

struct DwTcArgs {
  const float* dy_even;  // output gradients of even layers: block b's at dy_even + b * dy_stride
  const float* dy_odd;   // and of odd layers
  const float* h;        // even layers' inputs: block b's at h + b * stride
  const float* z;        // odd layers' inputs
  float* g;           // layer l's weight gradient at g + l * gstride, then its bias gradient
  int64_t stride, dy_stride, gstride;
  int ntiles, tiles_per_seq, seq_len, splits;
  unsigned* error;
};

__global__ void __launch_bounds__(DW_THREADS, 1) k_dw_tc(DwTcArgs P) {
  extern __shared__ __align__(1024) unsigned char tc_smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(tc_smem + DW_BAR_OFF);  // MMAs of buffer 0, 1 done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tc_smem + DW_BAR_OFF + 32);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int split = blockIdx.x % P.splits, part = blockIdx.x / P.splits;
  const int half = part & 1, layer = part >> 1;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(DW_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int b = 0; b < 2; ++b)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bars + b)), "r"(1) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot, bar0 = smem_u32(bars), base = smem_u32(tc_smem);
  const float* dY = ((layer & 1) ? P.dy_odd : P.dy_even) + (layer >> 1) * P.dy_stride;
  const float* X = ((layer & 1) ? P.z : P.h) + (layer >> 1) * P.stride + half * DW_N;
  constexpr int kA = TC_N * (TC_M / 8) / DW_THREADS;                              // 4 dY elements per thread
  constexpr int kB = (TC_ROWS * (DW_N / 8) + DW_THREADS - 1) / DW_THREADS;        // 3 X elements
  float bsum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  bool ok = true;
  int n = 0;  // tiles issued
  for (int tile = split; tile < P.ntiles; tile += P.splits, ++n) {
    const int sq = tile / P.tiles_per_seq, part0 = (tile - sq * P.tiles_per_seq) * TC_N;
    const int lo = sq * P.seq_len, q0 = lo + part0, cnt = min(TC_N, P.seq_len - part0);
    float4 a[kA][2], b[kB][2];
#pragma unroll
    for (int u = 0; u < kA; ++u) {
      const int e = tid + u * DW_THREADS, r = e / (TC_M / 8), c = e % (TC_M / 8);
      a[u][0] = a[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < cnt) {
        const float4* src = reinterpret_cast<const float4*>(dY + (int64_t)(q0 + r) * TC_M + 8 * c);
        a[u][0] = src[0];
        a[u][1] = src[1];
      }
    }
#pragma unroll
    for (int u = 0; u < kB; ++u) {
      const int e = tid + u * DW_THREADS, r = e / (DW_N / 8), c = e % (DW_N / 8);
      const int q = q0 - 2 + r;
      b[u][0] = b[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < TC_ROWS && q >= lo && q < lo + P.seq_len) {
        const float4* src = reinterpret_cast<const float4*>(X + (int64_t)q * TC_KC + 8 * c);
        b[u][0] = src[0];
        b[u][1] = src[1];
      }
    }
    const int buf = n & 1;
    if (n >= 2) ok = mbar_wait(bar0 + 8 * buf, ((n >> 1) - 1) & 1);
    ok = __syncthreads_and(ok);
    if (!ok) break;
    unsigned char* sA = tc_smem + buf * DW_BUF;
    unsigned char* sB = sA + DW_A_BYTES;
#pragma unroll
    for (int u = 0; u < kA; ++u) {
      const int e = tid + u * DW_THREADS, r = e / (TC_M / 8), c = e % (TC_M / 8);
      const float4 f = a[u][0], g = a[u][1];
      bsum[0] += f.x, bsum[1] += f.y, bsum[2] += f.z, bsum[3] += f.w;
      bsum[4] += g.x, bsum[5] += g.y, bsum[6] += g.z, bsum[7] += g.w;
      *reinterpret_cast<uint4*>(sA + c * DW_A_STRIDE + r * 16) =
          make_uint4(pack_bf16(f.x, f.y), pack_bf16(f.z, f.w), pack_bf16(g.x, g.y), pack_bf16(g.z, g.w));
    }
#pragma unroll
    for (int u = 0; u < kB; ++u) {
      const int e = tid + u * DW_THREADS, r = e / (DW_N / 8), c = e % (DW_N / 8);
      if (r >= TC_ROWS) break;
      const float4 f = b[u][0], g = b[u][1];
      *reinterpret_cast<uint4*>(sB + c * DW_B_STRIDE + r * 16) =
          make_uint4(pack_bf16(fmaxf(f.x, 0.f), fmaxf(f.y, 0.f)), pack_bf16(fmaxf(f.z, 0.f), fmaxf(f.w, 0.f)),
                     pack_bf16(fmaxf(g.x, 0.f), fmaxf(g.y, 0.f)), pack_bf16(fmaxf(g.z, 0.f), fmaxf(g.w, 0.f)));
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t ab = base + buf * DW_BUF, bb = ab + DW_A_BYTES;
#pragma unroll 1
      for (int t = 0; t < TC_TAPS; ++t)
#pragma unroll
        for (int k = 0; k < TC_N / 16; ++k) {
          const uint64_t ad = tc_desc(ab + (uint32_t)k * 256, 128, DW_A_STRIDE);
          const uint64_t bd = tc_desc(bb + (uint32_t)(16 * k + t) * 16, 128, DW_B_STRIDE);
          const uint32_t accum = (n | k) ? 1u : 0u;
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem + (uint32_t)(t * DW_N)),
              "l"(ad), "l"(bd), "r"(DW_IDESC), "r"(accum)
              : "memory");
        }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar0 + 8 * buf)
                   : "memory");
    }
  }
  // every MMA has completed: the last tile of each buffer
  for (int b = 0; b < 2; ++b)
    if (n > b) ok = mbar_wait(bar0 + 8 * b, (((n - 1 - b) >> 1) & 1)) && ok;
  ok = __syncthreads_and(ok);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!ok && tid == 0) atomicOr(P.error, 1u);
  if (ok && n > 0) {
    // warps w and w + 4, ..: TMEM lanes 32 (w % 4) ..; 20 pieces of 16 columns over 4 warps
    const int m = (warp & 3) * 32 + lane;
    float* dW = P.g + layer * P.gstride + (int64_t)m * TC_K + half * DW_N;
    for (int piece = warp >> 2; piece < TC_TAPS * (DW_N / 16); piece += DW_THREADS / 128) {
      uint32_t v[16];
      tmem_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(piece * 16), v);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      const int t = piece / (DW_N / 16), j = piece % (DW_N / 16) * 16;
#pragma unroll
      for (int k = 0; k < 16; k += 4)
        atomicAdd(reinterpret_cast<float4*>(dW + t * TC_KC + j + k),
                  make_float4(__uint_as_float(v[k]), __uint_as_float(v[k + 1]), __uint_as_float(v[k + 2]),
                              __uint_as_float(v[k + 3])));
    }
    if (half == 0) {
      // column sums of dY: threads of equal tid % 16 hold the same 8 channels
      float* red = reinterpret_cast<float*>(tc_smem);  // [16 warps][128 channels]
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float v = bsum[k] + __shfl_xor_sync(0xffffffffu, bsum[k], 16);
        if (lane < 16) red[warp * TC_M + lane * 8 + k] = v;
      }
    }
  }
  __syncthreads();
  if (ok && n > 0 && half == 0 && tid < TC_M) {
    const float* red = reinterpret_cast<const float*>(tc_smem);
    float v = 0.f;
    for (int w = 0; w < DW_THREADS / 32; ++w) v += red[w * TC_M + tid];
    atomicAdd(P.g + layer * P.gstride + (int64_t)TC_M * TC_K + tid, v);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(DW_COLS) : "memory");
}

struct DwArgs {
  const float* dY;  // [npos][M]
  const float* X;   // [npos][Kc]
  float* dW;        // [M][taps][Kc], accumulated
  int M, Kc, taps, relu_in, npos, seq_len, qchunk;
};

// dW[m][n] += sum_q dY[q][m] act(X[q + t - c][j]), n = t Kc + j; blockIdx.z picks
// a chunk of positions; partial tiles are added with atomics.
__global__ void __launch_bounds__(kThreads) k_conv_dw(DwArgs P) {
  __shared__ __align__(16) uint16_t As[BM][BK + kPadK];
  __shared__ __align__(16) uint16_t Bs[BN][BK + kPadK];
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int q_begin = blockIdx.z * P.qchunk;
  const int q_end = min(P.npos, q_begin + P.qchunk);
  const int warp = threadIdx.x >> 5, wm = warp >> 1, wn = warp & 1;
  const int c = (P.taps - 1) / 2;
  const int N = P.taps * P.Kc;
  float acc[2][4][4] = {};
  for (int k0 = q_begin; k0 < q_end; k0 += BK) {
    for (int e = threadIdx.x; e < BM * BK / 2; e += kThreads) {
      const int mm = e / (BK / 2), kk = 2 * (e % (BK / 2));
      const int m = m0 + mm;
      float v0 = 0.f, v1 = 0.f;
      if (m < P.M) {
        if (k0 + kk < q_end) v0 = P.dY[(int64_t)(k0 + kk) * P.M + m];
        if (k0 + kk + 1 < q_end) v1 = P.dY[(int64_t)(k0 + kk + 1) * P.M + m];
      }
      *reinterpret_cast<uint32_t*>(&As[mm][kk]) = pack_bf16(v0, v1);
    }
    for (int e = threadIdx.x; e < BN * BK / 2; e += kThreads) {
      const int nn = e / (BK / 2), kk = 2 * (e % (BK / 2));
      const int n = n0 + nn;
      float v[2] = {0.f, 0.f};
      if (n < N) {
        const int t = n / P.Kc, j = n - t * P.Kc;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int q = k0 + kk + h;
          if (q < q_end) {
            const int seq = q / P.seq_len, l = q - seq * P.seq_len;
            const int l2 = l + t - c;
            if (l2 >= 0 && l2 < P.seq_len) {
              const float x = P.X[((int64_t)seq * P.seq_len + l2) * P.Kc + j];
              v[h] = P.relu_in ? fmaxf(x, 0.f) : x;
            }
          }
        }
      }
      *reinterpret_cast<uint32_t*>(&Bs[nn][kk]) = pack_bf16(v[0], v[1]);
    }
    __syncthreads();
    warp_mma(As, Bs, wm, wn, 0, acc);
    warp_mma(As, Bs, wm, wn, 16, acc);
    __syncthreads();
  }
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int m = m0 + wm * 32 + i * 16 + g + (h >= 2 ? 8 : 0);
        const int n = n0 + wn * 32 + j * 8 + 2 * t + (h & 1);
        if (m < P.M && n < N) atomicAdd(&P.dW[(int64_t)m * N + n], acc[i][j][h]);
      }
}

// db[m] += sum_q dY[q][m]: a block takes kBiasRows positions, its threads the
// channels (rows read whole), and adds its partial sums.
constexpr int kBiasRows = 32;
__global__ void __launch_bounds__(256) k_bias_grad(const float* __restrict__ dY, int npos, int M, float* __restrict__ db) {
  __shared__ float red[256];
  const int q0 = blockIdx.x * kBiasRows, q1 = min(npos, q0 + kBiasRows);
  const int per = M < 256 ? 256 / M : 1;  // rows read at a time
  for (int m0 = 0; m0 < M; m0 += 256) {
    const int row = M < 256 ? threadIdx.x / M : 0, m = M < 256 ? threadIdx.x - row * M : m0 + threadIdx.x;
    float s = 0.f;
    if (row < per && m < M)
#pragma unroll 8
      for (int q = q0 + row; q < q1; q += per) s += dY[(int64_t)q * M + m];
    red[threadIdx.x] = s;
    __syncthreads();
    if (row == 0 && m < M) {
      for (int r = 1; r < per; ++r) s += red[r * M + m];
      atomicAdd(db + m, s);
    }
    __syncthreads();
  }
}

// Sum of the mask weights, into acc[0] (acc zeroed before).
__global__ void k_mask_sum(const float* __restrict__ mask, int64_t npts, double* __restrict__ acc) {
  double local = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npts;
       i += (int64_t)gridDim.x * blockDim.x)
    local += (double)mask[i];
  __shared__ double red[256];
  red[threadIdx.x] = local;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(acc, red[0]);
}

// Masked MSE with weights w = mask[point] and norm = cout sum(w) (acc[0]):
// loss (acc[1]) = sum w (y - target)^2 / norm, dy = 2 w (y - target) / norm.
__global__ void k_mse(const float* __restrict__ y, const float* __restrict__ target,
                      const float* __restrict__ mask, int64_t npts, int cout,
                      float* __restrict__ dy, double* __restrict__ acc) {
  const double norm = acc[0] * (double)cout;
  const float inv_norm = norm > 0.0 ? (float)(1.0 / norm) : 0.f;
  double local = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npts * cout;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float w = mask[i / cout];
    const float d = y[i] - target[i];
    dy[i] = 2.f * w * d * inv_norm;
    local += (double)w * (double)d * (double)d;
  }
  __shared__ double red[256];
  red[threadIdx.x] = local;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(acc + 1, red[0] * (double)inv_norm);
}

// Adam step on the FP32 master weights, then their BF16 copies.
__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// BF16 copies of every layer's weights W[o][t][i] (blockIdx.y: layer) and of the
// per-tap transposes WT[i][t][o] (the operands of the input-gradient pass). The
// residual blocks' layers of the tensor-core path are laid out as that operand's
// shared-memory image, tap by tap: [t][k / 8][m][k % 8] with (m, k) = (o, i) and (i, o).
struct LayerDev {
  int Co, taps, Ci, image;
  int64_t w_off, wb_off;
};

__global__ void k_weights_bf16(const float* __restrict__ w, const LayerDev* __restrict__ layers,
                               __nv_bfloat16* __restrict__ wb, __nv_bfloat16* __restrict__ wtb) {
  const LayerDev L = layers[blockIdx.y];
  const int n = L.Co * L.taps * L.Ci;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const int i = e % L.Ci, ot = e / L.Ci, t = ot % L.taps, o = ot / L.taps;
    const __nv_bfloat16 b = __float2bfloat16_rn(w[L.w_off + e]);
    if (L.image) {
      wb[L.wb_off + (((t * (L.Ci / 8) + i / 8) * L.Co + o) * 8 + i % 8)] = b;
      wtb[L.wb_off + (((t * (L.Co / 8) + o / 8) * L.Ci + i) * 8 + o % 8)] = b;
    } else {
      wb[L.wb_off + e] = b;
      wtb[L.wb_off + ((int64_t)i * L.taps + t) * L.Co + o] = b;
    }
  }
}

}  // namespace

// ---------------------------------------------------------------------------

struct rpk_net {
  int cin = 0, cout = 0, width = 0, nblocks = 0, device = 0;
  cudaStream_t stream = nullptr;
  struct Layer {
    int Co, taps, Ci;
    int64_t w_off, b_off;      // offsets in the parameter vector
    int64_t wb_off;            // offset in the bf16 weight arrays
  };
  std::vector<Layer> layers;   // lift, (b0 c0, b0 c1, ...), head
  int64_t nparams = 0, nwb = 0;
  float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
  __nv_bfloat16 *wb = nullptr, *wtb = nullptr;
  LayerDev* layers_dev = nullptr;
  int64_t step = 0;
  // activation workspace for up to cap_q coarse positions
  int64_t cap_q = 0;
  float* act = nullptr;   // h_0..h_B (B+1), z0 per block (B): (2B+1) x cap_q x width
  // training workspace for up to cap_t coarse positions
  int64_t cap_t = 0;
  float* work = nullptr;  // output gradients, slots of nq x width (layout: backward)
  int64_t work_floats = 0;
  float* headout = nullptr;
  float* dybuf = nullptr;
  double* loss = nullptr;
  int2* qseq = nullptr;        // ragged sequence table, cap_q entries
  int2* starts = nullptr;      // ragged sequences' first position and tile, cap_seq + 1 entries
  int cap_seq = 0;
  int4* tiles = nullptr;       // ragged tensor-core tiles (q0, count, start, length)
  int ntiles = 0, cap_tiles = 0;
  unsigned* tc_error = nullptr;  // set by the tcgen05 kernels when a wait gives up
  int nsm = 0;
  bool tc = false;             // the tensor-core path serves the block convolutions
};

namespace {

rpk_status net_alloc(void** p, size_t bytes) {
  cudaError_t err = cudaMalloc(p, bytes);
  if (err != cudaSuccess) {
    *p = nullptr;
    cudaGetLastError();
    return rpk::fail(RPK_ERR_OOM, std::string("network allocation failed: ") + cudaGetErrorString(err));
  }
  return RPK_OK;
}

rpk_status ensure_workspace(rpk_net* N, int64_t nq) {
  if (nq <= N->cap_q) return RPK_OK;
  cudaFree(N->act);
  cudaFree(N->qseq);
  N->act = nullptr;
  N->qseq = nullptr;
  N->cap_q = 0;
  const size_t W = N->width;
  rpk_status st = net_alloc((void**)&N->act, sizeof(float) * (2 * N->nblocks + 1) * nq * W);
  if (st == RPK_OK) st = net_alloc((void**)&N->qseq, sizeof(int2) * nq);
  if (st != RPK_OK) return st;
  N->cap_q = nq;
  return RPK_OK;
}

// Output gradients: one slot per layer (2 B + 1) lets one launch take every block's weight
// gradients at the end; where they would take more than this, or do not fit the device,
// two slots serve and each block's weight gradients follow its input gradient, so that
// a batch is never refused for the sake of the slots. Batches that large fill the chip
// with one block's layers: six blocks, a step of 204,800 coarse positions 3.31 ms with
// all slots (1.4 GB) and 3.36 with two, of 768,000 11.37 (5.1 GB) and 11.32.
constexpr int64_t kAllSlotsBytes = 4ll << 30;

int64_t all_slots(const rpk_net* N, int64_t nq) { return (2 * (int64_t)N->nblocks + 1) * nq * N->width; }

rpk_status ensure_training(rpk_net* N, int64_t nq) {
  rpk_status st = ensure_workspace(N, nq);
  if (st != RPK_OK || nq <= N->cap_t) return st;
  cudaFree(N->work);
  cudaFree(N->headout);
  cudaFree(N->dybuf);
  N->work = N->headout = N->dybuf = nullptr;
  N->cap_t = 0;
  st = net_alloc((void**)&N->headout, sizeof(float) * nq * R * N->cout);
  if (st == RPK_OK) st = net_alloc((void**)&N->dybuf, sizeof(float) * nq * R * N->cout);
  if (st != RPK_OK) return st;
  const int64_t two = std::min<int64_t>(2 * nq * N->width, all_slots(N, nq));
  N->work_floats = std::max(two, std::min(all_slots(N, nq), kAllSlotsBytes / (int64_t)sizeof(float)));
  st = net_alloc((void**)&N->work, sizeof(float) * N->work_floats);
  if (st != RPK_OK && N->work_floats > two) {
    N->work_floats = two;
    st = net_alloc((void**)&N->work, sizeof(float) * two);
  }
  if (st != RPK_OK) return st;
  N->cap_t = nq;
  return RPK_OK;
}

// Error word of the tensor-core path (synchronises the stream).
rpk_status tc_status(rpk_net* N) {
  if (!N->tc_error) return RPK_OK;
  unsigned e = 0;
  RPK_CUDA(cudaMemcpyAsync(&e, N->tc_error, sizeof(unsigned), cudaMemcpyDeviceToHost, N->stream));
  RPK_CUDA(cudaStreamSynchronize(N->stream));
  if (e) return rpk::fail(RPK_ERR_CUDA, "tensor-core convolution: an mbarrier wait gave up");
  return RPK_OK;
}

rpk_status refresh_bf16(rpk_net* N) {
  k_weights_bf16<<<dim3(64, (unsigned)N->layers.size()), 256, 0, N->stream>>>(N->w, N->layers_dev, N->wb, N->wtb);
  RPK_CUDA(cudaGetLastError());
  return RPK_OK;
}

rpk_status conv(rpk_net* N, const __nv_bfloat16* A, int M, int taps, int Kc, int sgn,
                const float* X, int relu_in, float* out, const float* bias, const float* res,
                const float* mask, int64_t nq, int seq_len, const int2* qseq = nullptr) {
  // one tap, 8-byte input pairs, weights that fit the default shared memory
  const int mt = M <= 16 ? 1 : 8;
  const size_t smem = (size_t)mt * 16 * ((Kc + 15) / 16 * 16 + kPadK) * 2;
  if (taps == 1 && !res && Kc % 2 == 0 && ((uintptr_t)X & 7) == 0 && smem + mt * 64 <= 48 * 1024) {
    const int quads = M % 4 == 0 && ((uintptr_t)out & 15) == 0 && ((uintptr_t)mask & 15) == 0;
    Conv1Args P{A, X, out, bias, mask, M, Kc, relu_in, (int)nq, quads};
    const int64_t want = (nq + 16 * (kConv1Threads / 32) - 1) / (16 * (kConv1Threads / 32));
    const dim3 grid((unsigned)std::min<int64_t>(want, 4 * (int64_t)std::max(N->nsm, 1)),
                    (unsigned)((M + mt * 16 - 1) / (mt * 16)));
    if (mt == 1)
      k_conv1<1><<<grid, kConv1Threads, smem, N->stream>>>(P);
    else
      k_conv1<8><<<grid, kConv1Threads, smem, N->stream>>>(P);
    RPK_CUDA(cudaGetLastError());
    return RPK_OK;
  }
  ConvArgs P{A, X, out, bias, res, mask, qseq, M, Kc, taps, sgn, relu_in, (int)nq, seq_len};
  const dim3 grid((unsigned)((nq + BN - 1) / BN), (unsigned)((M + BM - 1) / BM));
  k_conv<<<grid, kThreads, 0, N->stream>>>(P);
  RPK_CUDA(cudaGetLastError());
  return RPK_OK;
}

// A residual block (or its input gradient) on the tensor cores. Launched so
// that its CTAs may start where the previous kernel leaves SMs free.
rpk_status block_tc(rpk_net* N, BlockArgs T, int64_t nq, int seq_len, const int2* qseq) {
  T.error = N->tc_error;
  if (qseq) {
    T.tiles = N->tiles;
    T.ntiles = N->ntiles;
  } else {
    T.seq_len = seq_len;
    T.tiles_per_seq = (seq_len + TC_OUT - 1) / TC_OUT;
    T.ntiles = (int)(nq / seq_len) * T.tiles_per_seq;
  }
  cudaLaunchConfig_t c{};
  c.gridDim = dim3((unsigned)std::max(1, std::min(T.ntiles, N->nsm)));
  c.blockDim = dim3(TC_THREADS);
  c.dynamicSmemBytes = TC_SMEM;
  c.stream = N->stream;
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &a;
  c.numAttrs = 1;
  RPK_CUDA(cudaLaunchKernelEx(&c, k_block_tc, T));
  return RPK_OK;
}

rpk_status conv_dw(rpk_net* N, const float* dY, int M, const float* X, int Kc, int taps,
                   int relu_in, float* dW, int64_t nq, int seq_len) {
  // positions per block: enough blocks for about four per SM over the
  // (output x input) tiles, between BK and 2048 positions, a multiple of BK
  const int64_t tiles = (int64_t)((taps * Kc + BN - 1) / BN) * ((M + BM - 1) / BM);
  const int64_t want = std::max<int64_t>(1, 4 * (int64_t)std::max(N->nsm, 1) / std::max<int64_t>(tiles, 1));
  int64_t qc = (nq + want - 1) / want;
  qc = std::min<int64_t>(2048, std::max<int64_t>(BK, (qc + BK - 1) / BK * BK));
  const int qchunk = (int)qc;
  DwArgs P{dY, X, dW, M, Kc, taps, relu_in, (int)nq, seq_len, qchunk};
  const dim3 grid((unsigned)((taps * Kc + BN - 1) / BN), (unsigned)((M + BM - 1) / BM),
                  (unsigned)((nq + qchunk - 1) / qchunk));
  k_conv_dw<<<grid, kThreads, 0, N->stream>>>(P);
  RPK_CUDA(cudaGetLastError());
  return RPK_OK;
}

void bias_grad(rpk_net* N, const float* dY, int64_t nq, int M, float* db) {
  k_bias_grad<<<(unsigned)((nq + kBiasRows - 1) / kBiasRows), 256, 0, N->stream>>>(dY, (int)nq, M, db);
}

// Forward pass over nq coarse positions (sequences of Lq positions each, or the
// sequences described by qseq); keeps the blocks' inputs and, for training, the
// activations between their convolutions.
rpk_status forward(rpk_net* N, const float* x, int64_t nq, int Lq, const int2* qseq, float* y, bool train) {
  rpk_status st = ensure_workspace(N, nq);
  if (st != RPK_OK) return st;
  const int64_t stride = nq * N->width;
  float* h = N->act;  // h_b at act + b * stride; z0_b at act + (B + 1 + b) * stride
  const auto& lift = N->layers[0];
  st = conv(N, N->wb + lift.wb_off, N->width, 1, R * N->cin, +1, x, 0, h, N->w + lift.b_off,
            nullptr, nullptr, nq, Lq, qseq);
  for (int b = 0; b < N->nblocks && st == RPK_OK; ++b) {
    const auto& c0 = N->layers[1 + 2 * b];
    const auto& c1 = N->layers[2 + 2 * b];
    float* hb = N->act + b * stride;
    float* z0 = N->act + (N->nblocks + 1 + b) * stride;
    float* hn = N->act + (b + 1) * stride;
    if (N->tc) {
      st = block_tc(N, BlockArgs{N->wb + c0.wb_off, N->wb + c1.wb_off, hb, train ? z0 : nullptr, hn, N->w + c0.b_off,
                                 N->w + c1.b_off, nullptr, nullptr, nullptr, 0, 0, 0, +1, 1, nullptr},
                    nq, Lq, qseq);
      continue;
    }
    st = conv(N, N->wb + c0.wb_off, N->width, K5, N->width, +1, hb, 1, z0, N->w + c0.b_off,
              nullptr, nullptr, nq, Lq, qseq);
    if (st == RPK_OK)
      st = conv(N, N->wb + c1.wb_off, N->width, K5, N->width, +1, z0, 1, hn, N->w + c1.b_off, hb,
                nullptr, nq, Lq, qseq);
  }
  if (st != RPK_OK) return st;
  const auto& head = N->layers.back();
  return conv(N, N->wb + head.wb_off, R * N->cout, 1, N->width, +1, N->act + N->nblocks * stride,
              1, y, N->w + head.b_off, nullptr, nullptr, nq, Lq, qseq);
}

// qseq[q] = (first position, length) of the sequence holding coarse position q, and
// the sequence's tensor-core tiles (TC_OUT positions each, the first at index .y); one
// block per sequence, starts[s].x .. starts[s + 1].x (coarse positions).
__global__ void k_fill_sequences(const int2* __restrict__ starts, int2* __restrict__ qseq, int4* __restrict__ tiles) {
  const int2 a = starts[blockIdx.x], b = starts[blockIdx.x + 1];
  const int lo = a.x, hi = b.x;
  for (int q = lo + threadIdx.x; q < hi; q += blockDim.x) qseq[q] = make_int2(lo, hi - lo);
  for (int k = threadIdx.x; k < b.y - a.y; k += blockDim.x) {
    const int q = lo + k * TC_OUT;
    tiles[a.y + k] = make_int4(q, min(TC_OUT, hi - q), lo, hi - lo);
  }
}

// Gradients of the weights and biases of blocks b0 .. b0 + nb - 1 from the output
// gradients of their even and odd layers (block b0's first, then dy_stride apart).
rpk_status block_grads(rpk_net* N, int64_t nq, int Lq, int b0, int nb, const float* dy_even, const float* dy_odd,
                       int64_t dy_stride) {
  const int64_t stride = nq * N->width;
  const int nl = 2 * nb, W = N->width;
  if (nl == 0) return RPK_OK;
  const float* h = N->act + b0 * stride;
  const float* z = N->act + (N->nblocks + 1 + b0) * stride;
  const auto& first = N->layers[1 + 2 * b0];
  if (N->tc && (((uintptr_t)(N->g + first.w_off)) & 15) == 0) {
    DwTcArgs P{dy_even, dy_odd, h, z, N->g + first.w_off, stride, dy_stride,
               (int64_t)W * TC_K + W, 0, (Lq + TC_N - 1) / TC_N, Lq, 1, N->tc_error};
    P.ntiles = (int)(nq / Lq) * P.tiles_per_seq;
    // one CTA per SM: as many shares of the tiles as the SMs hold (layer, half) pairs
    P.splits = std::max(1, std::min(P.ntiles, N->nsm / (2 * nl)));
    k_dw_tc<<<2 * nl * P.splits, DW_THREADS, DW_SMEM, N->stream>>>(P);
    RPK_CUDA(cudaGetLastError());
    return RPK_OK;
  }
  for (int l = 0; l < nl; ++l) {
    const float* X = ((l & 1) ? z : h) + (l >> 1) * stride;
    const float* dY = ((l & 1) ? dy_odd : dy_even) + (l >> 1) * dy_stride;
    const auto& L = N->layers[1 + 2 * b0 + l];
    rpk_status st = conv_dw(N, dY, W, X, W, K5, 1, N->g + L.w_off, nq, Lq);
    if (st != RPK_OK) return st;
    bias_grad(N, dY, nq, W, N->g + L.b_off);
  }
  RPK_CUDA(cudaGetLastError());
  return RPK_OK;
}

// Backward pass from dy (fine layout == coarse layout), gradients into N->g. With
// a slot of N->work per layer the chain of input gradients comes first (slot 0 the
// lift's, slot l + 1 block layer l's output gradient) and the blocks' weight gradients
// together after it. With two slots a block's weight gradients follow its input
// gradient, whose output goes where an output gradient is no longer needed: slot 0
// and the last block's output h_B in turn (h_B serves only the head).
rpk_status backward(rpk_net* N, const float* x, const float* dy, int nseq, int L) {
  const int64_t nq = (int64_t)nseq * (L / R);
  const int Lq = L / R;
  const int64_t stride = nq * N->width;
  RPK_CUDA(cudaMemsetAsync(N->g, 0, sizeof(float) * N->nparams, N->stream));
  const bool all = all_slots(N, nq) <= N->work_floats;
  auto slot = [&](int k) { return N->work + k * stride; };
  const int W = N->width;
  const auto& head = N->layers.back();
  float* hB = N->act + N->nblocks * stride;
  rpk_status st = conv_dw(N, dy, R * N->cout, hB, W, 1, 1, N->g + head.w_off, nq, Lq);
  bias_grad(N, dy, nq, R * N->cout, N->g + head.b_off);
  // d relu(h_B) = W_head^T dy, then mask by h_B > 0
  float* dh = all ? slot(2 * N->nblocks) : slot(0);
  float* spare = hB;
  if (st == RPK_OK)
    st = conv(N, N->wtb + head.wb_off, W, 1, R * N->cout, -1, dy, 0, dh, nullptr, nullptr, hB, nq, Lq);
  for (int b = N->nblocks - 1; b >= 0 && st == RPK_OK; --b) {
    const auto& c0 = N->layers[1 + 2 * b];
    const auto& c1 = N->layers[2 + 2 * b];
    const float* hb = N->act + b * stride;
    const float* z0 = N->act + (N->nblocks + 1 + b) * stride;
    // z1 = conv(relu(z0)): d z1 = dh; z0 = conv(relu(h_b)): d z0 = dz; d h_b = dp
    float* dz = all ? slot(2 * b + 1) : slot(1);
    float* dp = all ? slot(2 * b) : spare;
    if (N->tc) {
      st = block_tc(N, BlockArgs{N->wtb + c1.wb_off, N->wtb + c0.wb_off, dh, dz, dp, nullptr, nullptr, z0, hb,
                                 nullptr, 0, 0, 0, -1, 0, nullptr},
                    nq, Lq, nullptr);
    } else {
      st = conv(N, N->wtb + c1.wb_off, W, K5, W, -1, dh, 0, dz, nullptr, nullptr, z0, nq, Lq);
      // d h_b = dh + (W0^T dz) masked by h_b > 0
      if (st == RPK_OK)
        st = conv(N, N->wtb + c0.wb_off, W, K5, W, -1, dz, 0, dp, nullptr, dh, hb, nq, Lq);
    }
    if (!all && st == RPK_OK) st = block_grads(N, nq, Lq, b, 1, dz, dh, 0);
    spare = dh;
    dh = dp;
  }
  if (all && st == RPK_OK) st = block_grads(N, nq, Lq, 0, N->nblocks, slot(1), slot(2), 2 * stride);
  if (st != RPK_OK) return st;
  const auto& lift = N->layers[0];
  st = conv_dw(N, dh, W, x, R * N->cin, 1, 0, N->g + lift.w_off, nq, Lq);
  bias_grad(N, dh, nq, W, N->g + lift.b_off);
  RPK_CUDA(cudaGetLastError());
  return st;
}

}  // namespace

extern "C" {

rpk_status rpk_net_create(int cin, int cout, int width, int nblocks, uint64_t seed,
                          void* cuda_stream, rpk_net** out) {
  if (!out) return rpk::fail(RPK_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (cin < 1 || cout < 1 || width < 16 || width % 16 || nblocks < 0 || nblocks > 64)
    return rpk::fail(RPK_ERR_ARG, "cin, cout >= 1; width a multiple of 16; 0 <= nblocks <= 64");
  rpk_net* N = new (std::nothrow) rpk_net();
  if (!N) return rpk::fail(RPK_ERR_OOM, "host allocation failed");
  N->cin = cin;
  N->cout = cout;
  N->width = width;
  N->nblocks = nblocks;
  N->stream = static_cast<cudaStream_t>(cuda_stream);
  cudaGetDevice(&N->device);
  auto add = [&](int Co, int taps, int Ci) {
    rpk_net::Layer L{Co, taps, Ci, N->nparams, N->nparams + (int64_t)Co * taps * Ci, N->nwb};
    N->nparams += (int64_t)Co * taps * Ci + Co;
    N->nwb += (int64_t)Co * taps * Ci;
    N->layers.push_back(L);
  };
  add(width, 1, R * cin);
  for (int b = 0; b < nblocks; ++b) {
    add(width, K5, width);
    add(width, K5, width);
  }
  add(R * cout, 1, width);
  // He-style initialisation drawn on the host; biases zero
  std::vector<float> w(N->nparams, 0.f);
  std::mt19937_64 rng(seed);
  for (size_t li = 0; li < N->layers.size(); ++li) {
    const auto& L = N->layers[li];
    const bool head = li + 1 == N->layers.size();
    const double sd = std::sqrt((head ? 1.0 : 2.0) / (L.taps * L.Ci));
    std::normal_distribution<double> nd(0.0, sd);
    for (int64_t i = 0; i < (int64_t)L.Co * L.taps * L.Ci; ++i) w[L.w_off + i] = (float)nd(rng);
  }
  rpk_status st = net_alloc((void**)&N->w, sizeof(float) * N->nparams);
  if (st == RPK_OK) st = net_alloc((void**)&N->g, sizeof(float) * N->nparams);
  if (st == RPK_OK) st = net_alloc((void**)&N->m, sizeof(float) * N->nparams);
  if (st == RPK_OK) st = net_alloc((void**)&N->v, sizeof(float) * N->nparams);
  if (st == RPK_OK) st = net_alloc((void**)&N->wb, sizeof(__nv_bfloat16) * N->nwb);
  if (st == RPK_OK) st = net_alloc((void**)&N->wtb, sizeof(__nv_bfloat16) * N->nwb);
  if (st == RPK_OK) st = net_alloc((void**)&N->loss, 2 * sizeof(double));
  if (st == RPK_OK) st = net_alloc((void**)&N->tc_error, sizeof(unsigned));
  if (st == RPK_OK) st = net_alloc((void**)&N->layers_dev, sizeof(LayerDev) * N->layers.size());
  if (st == RPK_OK) {
    cudaDeviceGetAttribute(&N->nsm, cudaDevAttrMultiProcessorCount, N->device);
    N->tc = width == TC_M &&
            cudaFuncSetAttribute(k_block_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM) ==
                cudaSuccess &&
            cudaFuncSetAttribute(k_dw_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DW_SMEM) == cudaSuccess;
    cudaGetLastError();
  }
  std::vector<LayerDev> ld;
  for (const auto& L : N->layers) ld.push_back({L.Co, L.taps, L.Ci, N->tc && L.taps == TC_TAPS, L.w_off, L.wb_off});
  cudaError_t err = cudaSuccess;
  if (st == RPK_OK)
    err = cudaMemcpyAsync(N->layers_dev, ld.data(), sizeof(LayerDev) * ld.size(), cudaMemcpyHostToDevice, N->stream);
  if (st == RPK_OK && err == cudaSuccess)
    err = cudaMemcpyAsync(N->w, w.data(), sizeof(float) * N->nparams, cudaMemcpyHostToDevice, N->stream);
  if (st == RPK_OK && err == cudaSuccess) err = cudaMemsetAsync(N->m, 0, sizeof(float) * N->nparams, N->stream);
  if (st == RPK_OK && err == cudaSuccess) err = cudaMemsetAsync(N->v, 0, sizeof(float) * N->nparams, N->stream);
  if (st == RPK_OK && err == cudaSuccess) err = cudaMemsetAsync(N->tc_error, 0, sizeof(unsigned), N->stream);
  if (st == RPK_OK && err == cudaSuccess) st = refresh_bf16(N);
  if (st == RPK_OK && err == cudaSuccess) err = cudaStreamSynchronize(N->stream);
  if (st != RPK_OK || err != cudaSuccess) {
    if (st == RPK_OK) st = rpk::cuda_fail(err, "rpk_net_create");
    rpk_net_destroy(N);
    return st;
  }
  *out = N;
  return RPK_OK;
}

void rpk_net_destroy(rpk_net* N) {
  if (!N) return;
  cudaStreamSynchronize(N->stream);
  void* p[] = {N->w,    N->g,       N->m,     N->v,    N->wb,     N->wtb,  N->act,
               N->work, N->headout, N->dybuf, N->loss, N->qseq, N->starts, N->tiles, N->tc_error,
               N->layers_dev};
  for (void* q : p)
    if (q) cudaFree(q);
  delete N;
}

int64_t rpk_net_num_params(const rpk_net* N) { return N ? N->nparams : 0; }

rpk_status rpk_net_get_params(rpk_net* N, float* host, int which) {
  if (!N || !host) return rpk::fail(RPK_ERR_ARG, "NULL argument");
  const float* src = which == 1 ? N->g : N->w;
  RPK_CUDA(cudaMemcpyAsync(host, src, sizeof(float) * N->nparams, cudaMemcpyDeviceToHost, N->stream));
  RPK_CUDA(cudaStreamSynchronize(N->stream));
  return RPK_OK;
}

rpk_status rpk_net_set_params(rpk_net* N, const float* host) {
  if (!N || !host) return rpk::fail(RPK_ERR_ARG, "NULL argument");
  RPK_CUDA(cudaMemcpyAsync(N->w, host, sizeof(float) * N->nparams, cudaMemcpyHostToDevice, N->stream));
  rpk_status st = refresh_bf16(N);
  if (st != RPK_OK) return st;
  RPK_CUDA(cudaStreamSynchronize(N->stream));
  return RPK_OK;
}

rpk_status rpk_net_forward(rpk_net* N, const float* x, int nseq, int len, float* y) {
  if (!N || !x || !y) return rpk::fail(RPK_ERR_ARG, "NULL argument");
  if (nseq < 1 || len < R || len % R) return rpk::fail(RPK_ERR_ARG, "len must be a positive multiple of 4");
  RPK_CUDA(cudaSetDevice(N->device));
  return forward(N, x, (int64_t)nseq * (len / R), len / R, nullptr, y, false);
}

rpk_status rpk_net_forward_ragged(rpk_net* N, const float* x, int nseq, const int* lens, float* y) {
  if (!N || !x || !y || !lens) return rpk::fail(RPK_ERR_ARG, "NULL argument");
  if (nseq < 1) return rpk::fail(RPK_ERR_ARG, "nseq must be >= 1");
  std::vector<int2> starts(nseq + 1, make_int2(0, 0));  // first position, first tile
  for (int s = 0; s < nseq; ++s) {
    if (lens[s] < R || lens[s] % R)
      return rpk::fail(RPK_ERR_ARG, "every length must be a positive multiple of 4");
    const int len = lens[s] / R;
    if ((int64_t)starts[s].x + len > INT32_MAX / 2)
      return rpk::fail(RPK_ERR_ARG, "too many positions");
    starts[s + 1] = make_int2(starts[s].x + len, starts[s].y + (len + TC_OUT - 1) / TC_OUT);
  }
  RPK_CUDA(cudaSetDevice(N->device));
  const int64_t nq = starts[nseq].x;
  rpk_status st = ensure_workspace(N, nq);
  if (st != RPK_OK) return st;
  if (nseq > N->cap_seq) {
    cudaFree(N->starts);
    N->starts = nullptr;
    N->cap_seq = 0;
    st = net_alloc((void**)&N->starts, sizeof(int2) * (nseq + 1));
    if (st != RPK_OK) return st;
    N->cap_seq = nseq;
  }
  N->ntiles = starts[nseq].y;
  if (N->ntiles > N->cap_tiles) {
    cudaFree(N->tiles);
    N->tiles = nullptr;
    N->cap_tiles = 0;
    st = net_alloc((void**)&N->tiles, sizeof(int4) * N->ntiles);
    if (st != RPK_OK) return st;
    N->cap_tiles = N->ntiles;
  }
  RPK_CUDA(cudaMemcpyAsync(N->starts, starts.data(), sizeof(int2) * (nseq + 1), cudaMemcpyHostToDevice, N->stream));
  k_fill_sequences<<<nseq, 256, 0, N->stream>>>(N->starts, N->qseq, N->tiles);
  cudaError_t err = cudaGetLastError();
  if (err == cudaSuccess) st = forward(N, x, nq, 0, N->qseq, y, false);
  // the table is read before it goes away, also after an error
  if (err == cudaSuccess && st == RPK_OK) return tc_status(N);
  cudaStreamSynchronize(N->stream);
  return st != RPK_OK ? st : rpk::cuda_fail(err, "rpk_net_forward_ragged");
}

rpk_status rpk_net_loss_grad(rpk_net* N, const float* x, const float* target, const float* mask,
                             int nseq, int len, double* loss) {
  if (!N || !x || !target || !mask || !loss) return rpk::fail(RPK_ERR_ARG, "NULL argument");
  if (nseq < 1 || len < R || len % R) return rpk::fail(RPK_ERR_ARG, "len must be a positive multiple of 4");
  RPK_CUDA(cudaSetDevice(N->device));
  const int64_t nq = (int64_t)nseq * (len / R);
  rpk_status st = ensure_training(N, nq);
  if (st != RPK_OK) return st;
  float* y = N->headout;
  st = forward(N, x, nq, len / R, nullptr, y, true);
  if (st != RPK_OK) return st;
  RPK_CUDA(cudaMemsetAsync(N->loss, 0, 2 * sizeof(double), N->stream));
  const int64_t npts = (int64_t)nseq * len;
  k_mask_sum<<<256, 256, 0, N->stream>>>(mask, npts, N->loss);
  k_mse<<<512, 256, 0, N->stream>>>(y, target, mask, npts, N->cout, N->dybuf, N->loss);
  cudaError_t err = cudaGetLastError();
  if (err == cudaSuccess) st = backward(N, x, N->dybuf, nseq, len);
  if (err == cudaSuccess && st == RPK_OK)
    err = cudaMemcpyAsync(loss, N->loss + 1, sizeof(double), cudaMemcpyDeviceToHost, N->stream);
  if (err == cudaSuccess && st == RPK_OK) err = cudaStreamSynchronize(N->stream);
  if (st != RPK_OK) return st;
  if (err != cudaSuccess) return rpk::cuda_fail(err, "rpk_net_loss_grad");
  return tc_status(N);
}

rpk_status rpk_net_adam(rpk_net* N, float lr, float beta1, float beta2, float eps) {
  if (!N) return rpk::fail(RPK_ERR_ARG, "NULL network");
  RPK_CUDA(cudaSetDevice(N->device));
  N->step += 1;
  const float c1 = 1.f - (float)std::pow((double)beta1, (double)N->step);
  const float c2 = 1.f - (float)std::pow((double)beta2, (double)N->step);
  k_adam<<<1024, 256, 0, N->stream>>>(N->w, N->g, N->m, N->v, N->nparams, lr, beta1, beta2, eps, c1, c2);
  RPK_CUDA(cudaGetLastError());
  return refresh_bf16(N);
}

}  // extern "C"

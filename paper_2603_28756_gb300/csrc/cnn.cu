// Learned warm start: a four-layer 3x3 convolutional refiner (1 -> 32 -> 32 -> 32 -> 1, ReLU
// after the first three layers, zero padding) applied to the normalised FBP start, with its
// own training kernels.  The paper has no learned component; this refiner is an addition.
//
// Precision: FP32 master weights, BF16 activations and weight copies, FP32 accumulation.
// The two 32 -> 32 layers are implicit GEMMs on the 5th-generation tensor cores (tcgen05.mma,
// BF16 operands in shared memory, FP32 accumulators in TMEM): M = 128 pixels of an image row,
// N = 32 output channels, K = 9 taps x 32 channels.
// Their data gradient is the same kernel run on the flipped, transposed weights, and their weight
// gradients are GEMMs over the pixels on the same tensor cores.  The first and last layers (32 MACs
// per tap) run on the CUDA cores.  Weight gradients are reduced over a fixed set of blocks in a fixed
// order (deterministic).
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <random>
#include <vector>

#include "internal.h"
#include "tc05.cuh"

namespace tmbir {

constexpr int kC = 32;                          // channels of the hidden layers
constexpr int kW0 = kC * 9, kB0 = kC;           // layer 0: [co][tap], bias
constexpr int kW1 = kC * kC * 9, kB1 = kC;      // layers 1, 2: [co][ci][tap] (oracle layout)
constexpr int kW3 = kC * 9, kB3 = 1;            // layer 3: [ci][tap]
constexpr int kOff0 = 0, kOffB0 = kW0;
constexpr int kOff1 = kOffB0 + kB0, kOffB1 = kOff1 + kW1;
constexpr int kOff2 = kOffB1 + kB1, kOffB2 = kOff2 + kW1;
constexpr int kOff3 = kOffB2 + kB1, kOffB3 = kOff3 + kW3;
constexpr int kParams = kOffB3 + kB3;  // 19105
constexpr int kTM = 128;               // pixels of one tensor-core tile (MMA M): a run of one image row
constexpr int kTX = kTM + 2;           // staged pixels of a row: x0 - 1 .. x0 + kTM
constexpr int kChunkB = kTX * 16;      // bytes of one staged (row, 8-channel chunk) array
constexpr int kRows = 4;                          // output rows of one tile (independent accumulators)
constexpr int kStageA = (kRows + 2) * 4 * kChunkB;  // staged rows x four chunks
constexpr int kStageAPad = (kStageA + 127) / 128 * 128;
constexpr int kWElems = 9 * 4 * kC * 8;           // packed 32 -> 32 weights [tap][chunk][n][8]
constexpr int kConvSmem = kStageAPad + kWElems * 2;  // staged rows + weights
constexpr uint32_t kMmaPolls = 1u << 22;          // bound of every wait on an MMA completion
constexpr int kWgradBlocks = 304;      // most blocks of the weight-gradient reductions: two per SM
constexpr int kPartRow = kW1 + kB1;    // one block's partial sums

struct CnnNet {
  cudaStream_t stream;
  int max_batch, H, W;
  float* master;        // [kParams] FP32 weights (oracle layout)
  float* grad;          // [kParams]
  float* adam_m;        // [kParams]
  float* adam_v;        // [kParams]
  __nv_bfloat16* wg1;   // layer 1 as the MMA's B operand: [tap][k chunk][co][8], k = ci
  __nv_bfloat16* wg2;   // layer 2
  __nv_bfloat16* wt1;   // flipped transpose of layer 1 for the data gradient: [tap][k chunk][ci][8], k = co
  __nv_bfloat16* wt2;
  int* err;             // set when a bounded wait on the tensor core gives up
  __nv_bfloat16* a0;    // activations NHWC [B][H][W][32]
  __nv_bfloat16* a1;
  __nv_bfloat16* a2;
  __nv_bfloat16* g1;    // gradients NHWC
  __nv_bfloat16* g2;
  float* xin;           // [B][H][W] normalised input
  float* out;           // [B][H][W] network output
  float* gout;          // [B][H][W]
  float* sig;           // [B] per-image scale
  float* wpart;         // [kWgradBlocks][kPartRow] weight-gradient partials
  double* dpart;        // scalar partials
  int step;
};

// ---------------------------------------------------------------- weight layouts
// Weights of the two 32 -> 32 layers in the layout of the MMA's B operand (no swizzle,
// K-major): element (tap, k chunk j, row n, e) = W[n][k = 8 j + e][tap] for the forward pass and
// the flipped transpose W[co = 8 j + e][ci = n][8 - tap] for the data gradient.
__global__ void k_cnn_pack(const float* __restrict__ master, __nv_bfloat16* wg1, __nv_bfloat16* wg2,
                           __nv_bfloat16* wt1, __nv_bfloat16* wt2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kWElems; i += gridDim.x * blockDim.x) {
    const int e = i % 8, n = (i / 8) % kC, j = (i / (8 * kC)) % 4, tap = i / (32 * kC);
    const int k = 8 * j + e;
    wg1[i] = __float2bfloat16_rn(master[kOff1 + (n * kC + k) * 9 + tap]);
    wg2[i] = __float2bfloat16_rn(master[kOff2 + (n * kC + k) * 9 + tap]);
    wt1[i] = __float2bfloat16_rn(master[kOff1 + (k * kC + n) * 9 + (8 - tap)]);
    wt2[i] = __float2bfloat16_rn(master[kOff2 + (k * kC + n) * 9 + (8 - tap)]);
  }
}

// ---------------------------------------------------------------- tensor-core 32 -> 32 convolution
// out[p][n] = sum_{tap, c} w[tap][n][c] in[p + tap][c] (+ bias, ReLU), as an implicit GEMM on the
// 5th-generation tensor cores.  A tile is kRows image rows x 128 pixels; each of its rows is an
// MMA with M = 128 pixels and N = 32 output channels, and each of the nine taps is one K = 32
// step (two K = 16 MMAs).  The kRows accumulators (32 TMEM columns each) are independent, and
// the MMAs are issued tap-major across them so consecutive MMAs do not wait on one another.
// The input rows y0-1 .. y0+kRows (pixels x0-1..x0+128, zero outside the image) are staged
// once per tile as 8-channel chunks, [row][chunk][pixel][8], which is the no-swizzle K-major
// operand layout; tap (dy, dx) of output row r is staged row r + dy started dx pixels (16
// bytes) later.  Each warp moves its 32 pixels of every row out with tcgen05.ld.
// MASK (data gradient): the result is multiplied by (mask[p][n] > 0).
// Bound by the latency of staging, products and stores in turn (three blocks per SM; tensor pipe 17 %,
// DRAM 30 % of their rates).  8 x 1024^2, forward: 466 us with 16-byte copies and stores a row chunk
// at a time, 408 with whole pixels staged and rows stored in bulk; asking L2 for the next tile's rows
// gains nothing (424).
template <bool BIAS_RELU, bool MASK>
__global__ void __launch_bounds__(128, 3) k_conv32(const __nv_bfloat16* __restrict__ in, int B, int H, int W,
                                                const __nv_bfloat16* __restrict__ wpk, const float* __restrict__ bias,
                                                const __nv_bfloat16* __restrict__ mask, __nv_bfloat16* __restrict__ out,
                                                int* err) {
  namespace tc = tc05;
  extern __shared__ __align__(128) unsigned char smraw[];
  unsigned char* sa = smraw;
  unsigned char* sw = smraw + kStageAPad;
  __shared__ uint64_t bar;
  __shared__ uint32_t tmem_base;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr uint32_t IDESC = tc::idesc_bf16_f32<kTM, kC>();
  const unsigned char* wsrc = reinterpret_cast<const unsigned char*>(wpk);
  for (int i = threadIdx.x; i < kWElems * 2 / 16; i += blockDim.x) tc::cp_async16(sw + 16 * i, wsrc + 16 * i, true);
  if (warp == 0) tc::tmem_alloc<kRows * kC>(&tmem_base);
  if (threadIdx.x == 0) {
    tc::mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_base;
  const uint32_t a_base = tc::smem_addr(sa), w_base = tc::smem_addr(sw);
  const uint64_t a_desc = tc::smem_desc(a_base, kChunkB, 128), w_desc = tc::smem_desc(w_base, kC * 16, 128);
  float bias_r[kC];
#pragma unroll
  for (int c = 0; c < kC; ++c) bias_r[c] = BIAS_RELU ? __ldg(bias + c) : 0.f;
  const int tiles_x = (W + kTM - 1) / kTM, tiles_y = (H + kRows - 1) / kRows;
  const int ntiles = B * tiles_y * tiles_x;
  uint32_t parity = 0;
  bool failed = false;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int tx = tile % tiles_x, ty = (tile / tiles_x) % tiles_y, b = tile / (tiles_x * tiles_y);
    const int y0 = ty * kRows, x0 = tx * kTM;
    // four neighbouring threads copy the four chunks of a staged pixel (whole sectors of 64 bytes)
    for (int i = threadIdx.x; i < kTX * 4; i += blockDim.x) {
      const int px = i >> 2, j = i & 3, gx = x0 - 1 + px;
      const bool vx = gx >= 0 && gx < W;
#pragma unroll
      for (int sr = 0; sr < kRows + 2; ++sr) {
        const int gy = y0 + sr - 1;
        const bool v = vx && gy >= 0 && gy < H;
        tc::cp_async16(sa + (sr * 4 + j) * kChunkB + px * 16, v ? in + (((size_t)b * H + gy) * W + gx) * kC + 8 * j : in, v);
      }
    }
    tc::cp_async_wait_all();  // this tile's rows (and, the first time, the weights)
    tc::fence_async_shared();
    __syncthreads();
    if (threadIdx.x == 0) {
      tc::fence_after_sync();
      // every operand start is a fixed byte offset from the staging / weight bases, added to the
      // descriptors' start-address field (bytes >> 4; the offsets stay inside the 14-bit field)
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        const int dy = tap / 3, dx = tap % 3;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const uint64_t bd = w_desc + (uint64_t)(((tap * 4 + 2 * s) * (kC * 16)) >> 4);
#pragma unroll
          for (int r = 0; r < kRows; ++r) {
            const uint64_t ad = a_desc + (uint64_t)((((r + dy) * 4 + 2 * s) * kChunkB + dx * 16) >> 4);
            tc::mma_bf16(tmem + r * kC, ad, bd, IDESC, (tap | s) ? 1u : 0u);
          }
        }
      }
      tc::mma_commit(&bar);
    }
    const bool ok = tc::mbar_wait(&bar, parity, kMmaPolls);
    parity ^= 1u;
    if (__syncthreads_or(!ok)) {
      failed = true;
      break;
    }
    tc::fence_after_sync();
    const int gx = x0 + warp * 32 + lane;
    // the warp's 32 pixels of every row, gathered over the staged rows (the MMAs have read them) and
    // written out as one bulk copy per row: a thread's 64 bytes of one pixel are half sectors otherwise
    unsigned char* so = sa + warp * kRows * 2048;
#pragma unroll 1
    for (int r = 0; r < kRows; ++r) {
      float v[32];
      tc::tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + r * kC, v);
      const int gy = y0 + r;
      if (gx >= W || gy >= H) continue;
      const size_t pbase = (((size_t)b * H + gy) * W + gx) * kC;
      if constexpr (BIAS_RELU) {
#pragma unroll
        for (int c = 0; c < kC; ++c) v[c] = fmaxf(v[c] + bias_r[c], 0.f);
      }
      if constexpr (MASK) {
        const uint4* mk = reinterpret_cast<const uint4*>(mask + pbase);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint4 m = mk[q];
          const __nv_bfloat162* mb = reinterpret_cast<const __nv_bfloat162*>(&m);
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const float2 f = __bfloat1622float2(mb[h]);
            if (!(f.x > 0.f)) v[8 * q + 2 * h] = 0.f;
            if (!(f.y > 0.f)) v[8 * q + 2 * h + 1] = 0.f;
          }
        }
      }
      uint4* dst = reinterpret_cast<uint4*>(so + r * 2048 + lane * 64);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint4 o;
        __nv_bfloat162* ob = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
        for (int h = 0; h < 4; ++h) ob[h] = __floats2bfloat162_rn(v[8 * q + 2 * h], v[8 * q + 2 * h + 1]);
        dst[q] = o;
      }
    }
    tc::fence_async_shared();
    __syncwarp();
    const int npx = min(32, W - (x0 + warp * 32));
    if (lane < kRows && npx > 0 && y0 + lane < H) {
      tc::bulk_store(out + (((size_t)b * H + y0 + lane) * W + x0 + warp * 32) * kC, so + lane * 2048, npx * 64);
      tc::bulk_commit();
      tc::bulk_wait_read();
    }
    // TMEM and the staged rows are reused by the next tile
    tc::fence_before_sync();
    __syncthreads();
  }
  tc::bulk_wait_all();
  if (failed) {
    // give the outstanding MMAs a second bounded chance to finish before freeing their TMEM
    tc::mbar_wait(&bar, parity ^ 1u, kMmaPolls);
    if (threadIdx.x == 0) atomicExch(err, 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc<kRows * kC>(tmem);
}

// ---------------------------------------------------------------- first and last layers (CUDA cores)
// a0[p][co] = relu(b0[co] + sum_tap w0[co][tap] x[p + tap]).  A block stages an 8 x 32 tile of
// x with a one-pixel halo; thread t owns output channels 4 (t % 8) .. +3 (weights in
// registers) for the pixels t / 8 + 32 k, so the eight threads of a pixel write its 64 bytes.
constexpr int kFH = 8, kFW = 32;
__global__ void __launch_bounds__(256) k_conv_first(const float* __restrict__ x, int B, int H, int W,
                                                    const float* __restrict__ master, __nv_bfloat16* __restrict__ a0) {
  __shared__ float xt[kFH + 2][kFW + 2];
  const int cg = threadIdx.x & 7, ps = threadIdx.x >> 3;
  float2 wr[2][9], br[2];  // channel pairs
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const float* w = master + kOff0 + (4 * cg + 2 * c) * 9;
#pragma unroll
    for (int t = 0; t < 9; ++t) wr[c][t] = make_float2(w[t], w[9 + t]);
    br[c] = make_float2(master[kOff0 + kW0 + 4 * cg + 2 * c], master[kOff0 + kW0 + 4 * cg + 2 * c + 1]);
  }
  const int tiles_x = (W + kFW - 1) / kFW, tiles_y = (H + kFH - 1) / kFH;
  const int tpi = tiles_x * tiles_y;
  for (int tile = blockIdx.x; tile < B * tpi; tile += gridDim.x) {
    const int b = tile / tpi, ty = (tile % tpi) / tiles_x, tx = tile % tiles_x;
    const int y0 = ty * kFH, x0 = tx * kFW;
    __syncthreads();
    for (int q = threadIdx.x; q < (kFH + 2) * (kFW + 2); q += blockDim.x) {
      const int gy = y0 - 1 + q / (kFW + 2), gx = x0 - 1 + q % (kFW + 2);
      xt[q / (kFW + 2)][q % (kFW + 2)] =
          (gy >= 0 && gy < H && gx >= 0 && gx < W) ? x[((size_t)b * H + gy) * W + gx] : 0.f;
    }
    __syncthreads();
    // the 3 x 3 window slides down the rows: three shared loads per pixel
    float2 nb[9];
#pragma unroll
    for (int t = 0; t < 6; ++t) nb[t + 3] = make_float2(xt[t / 3][ps + t % 3], xt[t / 3][ps + t % 3]);
#pragma unroll
    for (int ly = 0; ly < kFH; ++ly) {
#pragma unroll
      for (int t = 0; t < 6; ++t) nb[t] = nb[t + 3];
#pragma unroll
      for (int t = 0; t < 3; ++t) nb[6 + t] = make_float2(xt[ly + 2][ps + t], xt[ly + 2][ps + t]);
      const int gy = y0 + ly, gx = x0 + ps;
      if (gy >= H || gx >= W) continue;
      float2 v[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float2 acc = br[c];
#pragma unroll
        for (int t = 0; t < 9; ++t) acc = __ffma2_rn(wr[c][t], nb[t], acc);
        v[c] = make_float2(fmaxf(acc.x, 0.f), fmaxf(acc.y, 0.f));
      }
      uint2 o;
      reinterpret_cast<__nv_bfloat162*>(&o)[0] = __floats2bfloat162_rn(v[0].x, v[0].y);
      reinterpret_cast<__nv_bfloat162*>(&o)[1] = __floats2bfloat162_rn(v[1].x, v[1].y);
      *reinterpret_cast<uint2*>(a0 + (((size_t)b * H + gy) * W + gx) * kC + 4 * cg) = o;
    }
  }
}

// out[p] = b3 + sum_{tap, ci} w3[ci][tap] a2[p + tap][ci], as out[p] = b3 + sum_tap T[p + tap][tap]
// with T[q][tap] = sum_ci w3[ci][tap] a2[q][ci]: a block computes T once per pixel of its 16 x 32
// tile plus a one-pixel halo (each activation vector read once) and sums the nine shifted
// entries from shared memory.  Four lanes share a pixel, eight channels each (one 16-byte load, whole
// lines per warp) with their 72 weights in registers as channel pairs; their nine partial sums are
// added by exchanging halves, so that a lane ends with two or three of the nine.  Bound by FP32 issue
// and by the activation stream (64 B per pixel, 79 us at 8 x 1024^2).  The loads of four pixels are
// issued before their sums: with one or two in flight the warps waited for memory (8 x 1024^2: 412 us,
// with four 305).
// DGRAD: the data gradient of layer 0, gin[p] = sum_{tap, co} w0[co][tap] g0[p - tap][co]: the same
// sums with layer 0's weights, the taps flipped and no bias.
constexpr int kLH = 16, kLW = 32;
template <bool DGRAD>
__global__ void __launch_bounds__(256, 2) k_conv_last(const __nv_bfloat16* __restrict__ a2, int B, int H, int W,
                                                      const float* __restrict__ master, float* __restrict__ out) {
  constexpr int PX = (kLH + 2) * (kLW + 2);
  __shared__ float T[PX][9];
  const int q = threadIdx.x & 3;  // channels 8 q .. 8 q + 7
  const bool b0 = q & 1, b1 = q & 2;
  float2 w[4][9];
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const float* m = master + (DGRAD ? kOff0 : kOff3) + (8 * q + 2 * c) * 9 + (DGRAD ? 8 - t : t);
      w[c][t] = make_float2(m[0], m[9]);
    }
  const float b3 = DGRAD ? 0.f : master[kOff3 + kW3];
  const int tiles_x = (W + kLW - 1) / kLW, tiles_y = (H + kLH - 1) / kLH;
  const int tpi = tiles_x * tiles_y;
  for (int tile = blockIdx.x; tile < B * tpi; tile += gridDim.x) {
    const int b = tile / tpi, ty = (tile % tpi) / tiles_x, tx = tile % tiles_x;
    const int y0 = ty * kLH, x0 = tx * kLW;
    __syncthreads();  // T of the previous tile consumed
    // several pixels per lane quad and step, their loads issued first
    constexpr int BATCH = 4;
#pragma unroll 1
    for (int i0 = threadIdx.x >> 2; (i0 & ~7) < PX; i0 += BATCH * 64) {
      uint4 ub[BATCH];
#pragma unroll
      for (int k = 0; k < BATCH; ++k) {
        const int i = i0 + 64 * k, gy = y0 - 1 + i / (kLW + 2), gx = x0 - 1 + i % (kLW + 2);
        ub[k] = make_uint4(0, 0, 0, 0);
        if (i < PX && gy >= 0 && gy < H && gx >= 0 && gx < W)
          ub[k] = __ldg(reinterpret_cast<const uint4*>(a2 + (((size_t)b * H + gy) * W + gx) * kC) + q);
      }
#pragma unroll
      for (int k = 0; k < BATCH; ++k) {
        const int i = i0 + 64 * k;
        if ((i & ~7) >= PX) break;  // the same for the whole warp, which holds eight consecutive pixels
        const uint4 u = ub[k];
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
        float2 s[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) s[t] = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float2 a = __bfloat1622float2(h[c]);
#pragma unroll
          for (int t = 0; t < 9; ++t) s[t] = __ffma2_rn(w[c][t], a, s[t]);
        }
        float t[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) t[k] = s[k].x + s[k].y;
        // lanes differing in bit 0 share taps 0-3 / 4-7, then in bit 1 the pairs; tap 8 by all
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float give = b0 ? t[k] : t[k + 4];
          t[k] = (b0 ? t[k + 4] : t[k]) + __shfl_xor_sync(0xffffffffu, give, 1);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float give = b1 ? t[k] : t[k + 2];
          t[k] = (b1 ? t[k + 2] : t[k]) + __shfl_xor_sync(0xffffffffu, give, 2);
        }
        t[8] += __shfl_xor_sync(0xffffffffu, t[8], 1);
        t[8] += __shfl_xor_sync(0xffffffffu, t[8], 2);
        if (i < PX) {
          float* d = T[i] + (b0 ? 4 : 0) + (b1 ? 2 : 0);
          d[0] = t[0];
          d[1] = t[1];
          if (q == 0) T[i][8] = t[8];
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kLH / 8; ++r) {
      const int ly = threadIdx.x / kLW + 8 * r, lx = threadIdx.x % kLW;
      const int gy = y0 + ly, gx = x0 + lx;
      if (gy < H && gx < W) {
        float s = b3;
#pragma unroll
        for (int k = 0; k < 9; ++k) s += T[(ly + k / 3) * (kLW + 2) + lx + k % 3][k];
        out[((size_t)b * H + gy) * W + gx] = s;
      }
    }
  }
}

// g2[p][ci] = (a2[p][ci] > 0) * sum_tap w3[ci][tap] gout[p - tap].  A block stages a 16 x 32 tile of
// gout with a one-pixel halo; four lanes share a pixel, eight channels each with their weights in
// registers, so the mask is read and the result written in whole lines.  Four masks are loaded before
// their pixels are computed (8 x 1024^2: 397 -> 319 us).
__global__ void __launch_bounds__(256, 2) k_last_dgrad(const float* __restrict__ gout, const __nv_bfloat16* __restrict__ a2,
                                                       int B, int H, int W, const float* __restrict__ master,
                                                       __nv_bfloat16* __restrict__ g2) {
  __shared__ float gt[kLH + 2][kLW + 2];
  const int q = threadIdx.x & 3;
  float2 w[4][9];
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const float* m = master + kOff3 + (8 * q + 2 * c) * 9 + t;
      w[c][t] = make_float2(m[0], m[9]);
    }
  const int tiles_x = (W + kLW - 1) / kLW, tiles_y = (H + kLH - 1) / kLH;
  const int tpi = tiles_x * tiles_y;
  for (int tile = blockIdx.x; tile < B * tpi; tile += gridDim.x) {
    const int b = tile / tpi, ty = (tile % tpi) / tiles_x, tx = tile % tiles_x;
    const int y0 = ty * kLH, x0 = tx * kLW;
    __syncthreads();
    for (int i = threadIdx.x; i < (kLH + 2) * (kLW + 2); i += blockDim.x) {
      const int gy = y0 - 1 + i / (kLW + 2), gx = x0 - 1 + i % (kLW + 2);
      gt[i / (kLW + 2)][i % (kLW + 2)] =
          (gy >= 0 && gy < H && gx >= 0 && gx < W) ? __ldg(gout + ((size_t)b * H + gy) * W + gx) : 0.f;
    }
    __syncthreads();
    constexpr int BATCH = 4;
#pragma unroll 1
    for (int i0 = threadIdx.x >> 2; i0 < kLH * kLW; i0 += BATCH * 64) {
      uint4 mb[BATCH];
#pragma unroll
      for (int k = 0; k < BATCH; ++k) {
        const int i = i0 + 64 * k, gy = y0 + i / kLW, gx = x0 + i % kLW;
        mb[k] = make_uint4(0, 0, 0, 0);
        if (gy < H && gx < W) mb[k] = __ldg(reinterpret_cast<const uint4*>(a2 + (((size_t)b * H + gy) * W + gx) * kC + 8 * q));
      }
#pragma unroll
      for (int k = 0; k < BATCH; ++k) {
        const int i = i0 + 64 * k, ly = i / kLW, lx = i % kLW, gy = y0 + ly, gx = x0 + lx;
        if (gy >= H || gx >= W) continue;
        const __nv_bfloat162* mh = reinterpret_cast<const __nv_bfloat162*>(&mb[k]);
        float2 s[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) s[c] = make_float2(0.f, 0.f);
#pragma unroll
        for (int t = 0; t < 9; ++t) {
          const float gv = gt[ly + 2 - t / 3][lx + 2 - t % 3];
#pragma unroll
          for (int c = 0; c < 4; ++c) s[c] = __ffma2_rn(w[c][t], make_float2(gv, gv), s[c]);
        }
        uint4 o;
        __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float2 a = __bfloat1622float2(mh[c]);
          oh[c] = __floats2bfloat162_rn(a.x > 0.f ? s[c].x : 0.f, a.y > 0.f ? s[c].y : 0.f);
        }
        *reinterpret_cast<uint4*>(g2 + (((size_t)b * H + gy) * W + gx) * kC + 8 * q) = o;
      }
    }
  }
}

// ---------------------------------------------------------------- weight gradients (fixed-order block partials)
// Layers 1, 2: dW[co][ci][tap] = sum_p g[p][co] in[p + tap][ci] and db[co] = sum_p g[p][co], as a
// GEMM over the pixels on the tensor cores.  The images' channel-last layout makes the channels of a
// pixel contiguous and the pixels the contraction index, which is the MMA's MN-major operand layout
// with the staging of the forward convolution ([row][8-channel chunk][pixel][8]):
//   A (M = 128): the 32 channels of four consecutive rows of g, rows y - 1 .. y + 2 against input
//      row y: three of the four are the taps dy = +1, 0, -1 (the fourth is not used);
//   B (N = 32):  input row y shifted by dx pixels (16 bytes), one MMA per dx; the centre one takes
//      N = 48 with 16 further columns of ones, whose products are the bias gradient.
// A tile is kGRows input rows x 128 pixels (8 K-steps of 16 pixels per row), accumulated in TMEM and
// then added to FP32 registers, thread = (dy, co), 96 sums: the tensor core's accumulator is not
// rounded to nearest, so its chains are kept to 32 K-steps, which leaves the sums nearer to 64 bits
// than one FP32 chain per thread over all pixels.
// Bound by the operand reads from shared memory (4 KB of A per MMA) and by the two activation
// streams (128 B per pixel); the CUDA-core form this replaced read every pixel's nine neighbours
// in every thread: 76 ms at 8 x 1024^2, now 0.55.
constexpr int kGRows = 4;
constexpr int kGRowB = 4 * kTM * 16;               // bytes of one staged row of g
constexpr int kGInB = 6 * kChunkB;                 // one staged input row: four chunks, ones, zeros
constexpr int kGSmemG = (kGRows + 3) * kGRowB;     // rows y0 - 1 .. y0 + kGRows + 1 (the last stays zero)
constexpr int kGradSmem = kGSmemG + kGRows * kGInB;


__global__ void __launch_bounds__(128, 2) k_wgrad32(const __nv_bfloat16* __restrict__ g, const __nv_bfloat16* __restrict__ in,
                                                 int B, int H, int W, float* __restrict__ part, int* err) {
  namespace tc = tc05;
  extern __shared__ __align__(128) unsigned char smraw[];
  unsigned char* sg = smraw;
  unsigned char* si = smraw + kGSmemG;
  __shared__ uint64_t bar;
  __shared__ uint32_t tmem_base;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0) tc::tmem_alloc<128>(&tmem_base);
  if (threadIdx.x == 0) {
    tc::mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the parts that staging never writes: the ones and zeros of every input row, the last row of g
  for (int i = threadIdx.x; i < kGRows * 2 * kTX; i += blockDim.x) {
    const int r = i / (2 * kTX), c = (i / kTX) & 1, px = i % kTX;
    const uint32_t one2 = 0x3f803f80u;
    const uint4 v = c == 0 ? make_uint4(one2, one2, one2, one2) : make_uint4(0, 0, 0, 0);
    *reinterpret_cast<uint4*>(si + r * kGInB + (4 + c) * kChunkB + px * 16) = v;
  }
  for (int i = threadIdx.x; i < kGRowB / 16; i += blockDim.x)
    *reinterpret_cast<uint4*>(sg + (kGRows + 2) * kGRowB + i * 16) = make_uint4(0, 0, 0, 0);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_base;
  // MN-major: M (N) chunks of 8 channels lie sbo apart, groups of 8 pixels lbo = 128 bytes apart
  const uint64_t a_desc = tc::smem_desc(tc::smem_addr(sg), 128, kTM * 16);
  const uint64_t b_desc = tc::smem_desc(tc::smem_addr(si), 128, kChunkB);
  constexpr uint32_t ID32 = tc::idesc_bf16_f32_mn<128, 32>(), ID48 = tc::idesc_bf16_f32_mn<128, 48>();
  const int tiles_x = (W + kTM - 1) / kTM, tiles_y = (H + kGRows - 1) / kGRows;
  const int ntiles = B * tiles_y * tiles_x;
  float acc[3 * kC], accb = 0.f;
#pragma unroll
  for (int i = 0; i < 3 * kC; ++i) acc[i] = 0.f;
  uint32_t parity = 0;
  bool failed = false;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int tx = tile % tiles_x, ty = (tile / tiles_x) % tiles_y, b = tile / (tiles_x * tiles_y);
    const int y0 = ty * kGRows, x0 = tx * kTM;
    // four neighbouring threads copy the four chunks of a staged pixel
    for (int i = threadIdx.x; i < kTX * 4; i += blockDim.x) {
      const int px = i >> 2, j = i & 3;
      if (px < kTM) {
        const int gx = x0 + px;
#pragma unroll
        for (int r = 0; r < kGRows + 2; ++r) {
          const int gy = y0 - 1 + r;
          const bool v = gx < W && gy >= 0 && gy < H;
          tc::cp_async16(sg + r * kGRowB + j * (kTM * 16) + px * 16, v ? g + (((size_t)b * H + gy) * W + gx) * kC + 8 * j : g, v);
        }
      }
      const int gx = x0 - 1 + px;
#pragma unroll
      for (int r = 0; r < kGRows; ++r) {
        const int gy = y0 + r;
        const bool v = gx >= 0 && gx < W && gy < H;
        tc::cp_async16(si + r * kGInB + j * kChunkB + px * 16, v ? in + (((size_t)b * H + gy) * W + gx) * kC + 8 * j : in, v);
      }
    }
    tc::cp_async_wait_all();
    tc::fence_async_shared();
    __syncthreads();
    if (threadIdx.x == 0) {
      tc::fence_after_sync();
#pragma unroll 1
      for (int r = 0; r < kGRows; ++r) {
#pragma unroll
        for (int s = 0; s < kTM / 16; ++s) {
          const uint64_t ad = a_desc + (uint64_t)((r * kGRowB + s * 256) >> 4);
          const uint64_t bd = b_desc + (uint64_t)((r * kGInB + s * 256) >> 4);
          const uint32_t more = (r | s) ? 1u : 0u;
          tc::mma_bf16(tmem, ad, bd, ID32, more);
          tc::mma_bf16(tmem + 32, ad, bd + 1, ID48, more);
          tc::mma_bf16(tmem + 80, ad, bd + 2, ID32, more);
        }
      }
      tc::mma_commit(&bar);
    }
    const bool ok = tc::mbar_wait(&bar, parity, kMmaPolls);
    parity ^= 1u;
    if (__syncthreads_or(!ok)) {
      failed = true;
      break;
    }
    tc::fence_after_sync();
    if (warp < 3) {  // warp = row of g relative to the input row: tap row 2 - warp
      const uint32_t base = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll
      for (int dx = 0; dx < 3; ++dx) {
        float v[32];
        tc::tmem_ld32(base + (dx == 2 ? 80 : 32 * dx), v);
#pragma unroll
        for (int c = 0; c < kC; ++c) acc[dx * kC + c] += v[c];
      }
      if (warp == 1) accb += tc::tmem_ld1(base + 64);
    }
    tc::fence_before_sync();
    __syncthreads();  // TMEM and the staged rows are reused by the next tile
  }
  if (failed) {
    // give the outstanding MMAs a second bounded chance to finish before freeing their TMEM
    tc::mbar_wait(&bar, parity ^ 1u, kMmaPolls);
    if (threadIdx.x == 0) atomicExch(err, 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc<128>(tmem);
  float* o = part + (size_t)blockIdx.x * kPartRow;
  if (warp < 3) {
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
      for (int c = 0; c < kC; ++c) o[(lane * kC + c) * 9 + (2 - warp) * 3 + dx] = acc[dx * kC + c];
    if (warp == 1) o[kW1 + lane] = accb;
  }
}

// Layers 0 and 3, FP32 on the CUDA cores: dW[c][tap] = sum_q h[q][c] f[q + s tap] with 32 BF16
// channels h and one FP32 image f.  FIRST: h = g0, f = xin, s = +1, bias db[c] = sum_q h[q][c];
// otherwise h = a2, f = gout, s = -1 (dW3[ci][tap] = sum_p gout[p] a2[p + tap][ci]) and
// db = sum_q f[q].  A block takes tiles of 8 rows x 128 pixels, one row per warp; a lane owns a
// channel pair (packed FP32 FMAs), the two half-warps walk the two halves of the row, and the nine
// values of f slide along x, so a step costs one 4-byte load of h and three shared loads of f for
// 18 sums.  Partial row layout: [0, 288) dW, then the bias.  The form this replaced read h once
// per tap and pixel from 64 to 128 threads a block: 23.5 ms (first) and 36.9 ms (last)
// at 8 x 1024^2, now 0.23 and 0.23.
constexpr int kEH = 8, kEW = 128;
template <bool FIRST>
__global__ void __launch_bounds__(256) k_wgrad_edge(const __nv_bfloat16* __restrict__ h, const float* __restrict__ f,
                                                    int B, int H, int W, float* __restrict__ part) {
  __shared__ float ft[kEH + 2][kEW + 2];
  __shared__ float2 red[8][10][16];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, half = lane >> 4, cp = lane & 15;
  float2 acc[9], accb = make_float2(0.f, 0.f);
#pragma unroll
  for (int t = 0; t < 9; ++t) acc[t] = make_float2(0.f, 0.f);
  const int tiles_x = (W + kEW - 1) / kEW, tiles_y = (H + kEH - 1) / kEH;
  const int ntiles = B * tiles_x * tiles_y;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int tx = tile % tiles_x, ty = (tile / tiles_x) % tiles_y, b = tile / (tiles_x * tiles_y);
    const int y0 = ty * kEH, x0 = tx * kEW;
    __syncthreads();
    for (int q = threadIdx.x; q < (kEH + 2) * (kEW + 2); q += blockDim.x) {
      const int gy = y0 - 1 + q / (kEW + 2), gx = x0 - 1 + q % (kEW + 2);
      ft[q / (kEW + 2)][q % (kEW + 2)] =
          (gy >= 0 && gy < H && gx >= 0 && gx < W) ? __ldg(f + ((size_t)b * H + gy) * W + gx) : 0.f;
    }
    __syncthreads();
    const int y = y0 + warp;
    if (y < H) {
      const int xs = half * (kEW / 2);
      const __nv_bfloat162* hp = reinterpret_cast<const __nv_bfloat162*>(h) + (((size_t)b * H + y) * W + x0 + xs) * (kC / 2) + cp;
      const int n = min(kEW / 2, W - x0 - xs);  // this half's pixels (may be <= 0)
      const float* fr = &ft[warp][xs];
      // window win[i][j] = f at row y + i - 1, column x + j - 1
      float win[3][3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        win[i][0] = 0.f;
        win[i][1] = fr[i * (kEW + 2)];
        win[i][2] = fr[i * (kEW + 2) + 1];
      }
#pragma unroll 8
      for (int k = 0; k < kEW / 2; ++k) {
        __nv_bfloat162 hv = __floats2bfloat162_rn(0.f, 0.f);
        if (k < n) hv = hp[(size_t)k * (kC / 2)];
        const float2 v = __bfloat1622float2(hv);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          win[i][0] = win[i][1];
          win[i][1] = win[i][2];
          win[i][2] = fr[i * (kEW + 2) + k + 2];
        }
#pragma unroll
        for (int t = 0; t < 9; ++t) {
          const float fv = FIRST ? win[t / 3][t % 3] : win[2 - t / 3][2 - t % 3];
          acc[t] = __ffma2_rn(v, make_float2(fv, fv), acc[t]);
        }
        if constexpr (FIRST)
          accb = __fadd2_rn(accb, v);
        else if (k < n)
          accb.x += win[1][1];  // every lane of the half holds the half's sum
      }
    }
  }
  // the two halves, then the eight warps in order
#pragma unroll
  for (int t = 0; t < 10; ++t) {
    float2 v = t < 9 ? acc[t < 9 ? t : 0] : accb;
    v.x += __shfl_down_sync(0xffffffffu, v.x, 16);
    v.y += __shfl_down_sync(0xffffffffu, v.y, 16);
    if (half == 0) red[warp][t][cp] = v;
  }
  __syncthreads();
  float* o = part + (size_t)blockIdx.x * kPartRow;
  for (int q = threadIdx.x; q < 160; q += blockDim.x) {
    const int t = q / 16, c = q % 16;
    float2 s = make_float2(0.f, 0.f);
    for (int w = 0; w < 8; ++w) {
      s.x += red[w][t][c].x;
      s.y += red[w][t][c].y;
    }
    if (t < 9) {
      o[(2 * c) * 9 + t] = s.x;
      o[(2 * c + 1) * 9 + t] = s.y;
    } else if (FIRST) {
      o[288 + 2 * c] = s.x;
      o[288 + 2 * c + 1] = s.y;
    } else if (c == 0) {
      o[288] = s.x;
    }
  }
}
enum class Layer { First, Hidden, Last };

// One block's share of weight i's sum in k_wgrad32 (Hidden: h = g) or k_wgrad_edge, product by product
// and without those outside the image.
template <Layer L>
__device__ __noinline__ float wgrad_inside(const __nv_bfloat16* h, const void* other, int B, int H, int W, int block,
                                           int nblocks, int i) {
  constexpr int TH = L == Layer::Hidden ? kGRows : kEH, TW = L == Layer::Hidden ? kTM : kEW;
  const int tap = i % 9, dy = tap / 3 - 1, dx = tap % 3 - 1, ci = i / 9 % kC, c = L == Layer::Hidden ? i / (9 * kC) : ci;
  const int tiles_x = (W + TW - 1) / TW, tiles_y = (H + TH - 1) / TH;
  float s = 0.f;
  for (int tile = block; tile < B * tiles_y * tiles_x; tile += nblocks) {
    const int x0 = tile % tiles_x * TW, y0 = tile / tiles_x % tiles_y * TH;
    const size_t plane = (size_t)(tile / (tiles_x * tiles_y)) * H;
    for (int q = 0; q < TH * TW; ++q) {
      const int y = y0 + q / TW, hx = x0 + q % TW;  // Hidden: y is the row of the layer's input
      const int hy = L == Layer::Hidden ? y - dy : y, oy = L == Layer::Hidden ? y : (L == Layer::First ? y + dy : y - dy);
      const int ox = L == Layer::Last ? hx - dx : hx + dx;
      if (hy < 0 || hy >= H || hx >= W || oy < 0 || oy >= H || ox < 0 || ox >= W) continue;
      const size_t o = (plane + oy) * W + ox;
      const float f = L == Layer::Hidden ? __bfloat162float(static_cast<const __nv_bfloat16*>(other)[o * kC + ci])
                                         : static_cast<const float*>(other)[o];
      s = fmaf(__bfloat162float(h[((plane + hy) * W + hx) * kC + c]), f, s);
    }
  }
  return s;
}

// dst[i] += sum over blocks of part[b][i], i < n, in FP64: eight threads per element take every
// eighth block, then their sums in order.  The blocks multiply infinities and NaN beside the border by
// the zeros staged outside the image, which makes NaN of sums that such a value is not part of: where
// a weight's sum is not finite, its blocks' shares are formed again without those products.
template <Layer L>
__global__ void __launch_bounds__(256) k_reduce_parts(const float* __restrict__ part, int nblocks, int n,
                                                      float* __restrict__ dst, const __nv_bfloat16* h, const void* other,
                                                      int B, int H, int W) {
  __shared__ double sh[8][32];
  const int i = blockIdx.x * 32 + (threadIdx.x & 31), r = threadIdx.x >> 5;
  double s = 0.0;
  if (i < n)
    for (int b = r; b < nblocks; b += 8) s += part[(size_t)b * kPartRow + i];
  if (i < (L == Layer::Hidden ? kW1 : kW0) && !isfinite(s)) {
    s = 0.0;
    for (int b = r; b < nblocks; b += 8) {
      const float v = part[(size_t)b * kPartRow + i];
      s += isfinite(v) ? v : wgrad_inside<L>(h, other, B, H, W, b, nblocks, i);
    }
  }
  sh[r][threadIdx.x & 31] = s;
  __syncthreads();
  if (r == 0 && i < n) {
#pragma unroll
    for (int k = 1; k < 8; ++k) s += sh[k][threadIdx.x];
    dst[i] += (float)s;
  }
}

// ---------------------------------------------------------------- normalisation, loss, optimiser
// per image: sig = sqrt(mean x^2) (1 if zero); xin = x / sig.  kNormBlocks blocks per image
// each reduce a strided share in FP64, then one block per image adds the shares in order.
constexpr int kNormBlocks = 64;
__global__ void k_norm_partial(const float* __restrict__ x, int HW, double* __restrict__ part) {
  __shared__ double sh[256];
  const int b = blockIdx.y;
  const float* xb = x + (size_t)b * HW;
  double s = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < HW; i += kNormBlocks * blockDim.x) s += (double)xb[i] * xb[i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[(size_t)b * kNormBlocks + blockIdx.x] = sh[0];
}
__global__ void k_norm_stats(const double* __restrict__ part, int HW, float* __restrict__ sig) {
  if (threadIdx.x != 0) return;
  double s = 0.0;
  for (int k = 0; k < kNormBlocks; ++k) s += part[(size_t)blockIdx.x * kNormBlocks + k];
  const double r = sqrt(s / HW);
  sig[blockIdx.x] = r > 0 ? (float)r : 1.f;
}
__global__ void k_scale_in(const float* __restrict__ x, int HW, size_t total, const float* __restrict__ sig,
                           float* __restrict__ xin) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x)
    xin[i] = x[i] / sig[i / HW];
}
// refined = x + sig * net
__global__ void k_residual_out(const float* __restrict__ x, const float* __restrict__ net, int HW, size_t total,
                               const float* __restrict__ sig, float* __restrict__ y) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x)
    y[i] = x[i] + sig[i / HW] * net[i];
}
// loss = mean (net - (t - x)/sig)^2; gout = 2 (net - r) / P; per-block FP64 partials
__global__ void k_loss(const float* __restrict__ net, const float* __restrict__ x, const float* __restrict__ t, int HW,
                       size_t total, const float* __restrict__ sig, float* __restrict__ gout, double* __restrict__ part) {
  __shared__ double sh[256];
  double s = 0.0;
  const float inv = 1.0f / (float)total;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const float r = (t[i] - x[i]) / sig[i / HW];
    const float d = net[i] - r;
    gout[i] = 2.0f * d * inv;
    s += (double)d * d;
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}
__global__ void k_sum_d(const double* __restrict__ part, int n, double scale, double* __restrict__ out) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < n; ++i) s += part[i];
    *out = s * scale;
  }
}
// Adam (Kingma & Ba 2015) on the FP32 master weights
__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       int n, float lr, float b1, float b2, float eps, float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// ---------------------------------------------------------------- host sequences
static size_t cnn_bytes(int B, int H, int W, size_t* offs) {
  size_t off = 0;
  auto take = [&](size_t b) {
    off = (off + 255) / 256 * 256;
    size_t o = off;
    off += b;
    return o;
  };
  const size_t P = (size_t)B * H * W;
  offs[0] = take(kParams * 4);                         // master
  offs[1] = take(kParams * 4);                         // grad
  offs[2] = take(kParams * 4);                         // m
  offs[3] = take(kParams * 4);                         // v
  for (int i = 0; i < 4; ++i) offs[4 + i] = take((size_t)kWElems * 2);  // wg1 wg2 wt1 wt2
  for (int i = 0; i < 5; ++i) offs[8 + i] = take(P * kC * 2);           // a0 a1 a2 g1 g2
  for (int i = 0; i < 3; ++i) offs[13 + i] = take(P * 4);               // xin out gout
  offs[16] = take((size_t)B * 4);                                        // sig
  offs[17] = take((size_t)kWgradBlocks * kPartRow * 4);                  // wpart
  offs[18] = take(std::max<size_t>(4096, (size_t)B * kNormBlocks) * 8);  // dpart (loss / norm partials)
  offs[19] = take(256);                                                  // err
  return (off + 255) / 256 * 256;
}

static int conv32(CnnNet& n, const __nv_bfloat16* in, int B, const __nv_bfloat16* w, const float* bias,
                  const __nv_bfloat16* mask, __nv_bfloat16* out, bool relu) {
  static bool attr = false;
  if (!attr) {
    TMBIR_CUDA(cudaFuncSetAttribute(k_conv32<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kConvSmem));
    TMBIR_CUDA(cudaFuncSetAttribute(k_conv32<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kConvSmem));
    attr = true;
  }
  const int tiles = B * ((n.H + kRows - 1) / kRows) * ((n.W + kTM - 1) / kTM);
  const int blocks = std::min(tiles, 152 * 3);
  if (relu)
    k_conv32<true, false><<<blocks, 128, kConvSmem, n.stream>>>(in, B, n.H, n.W, w, bias, nullptr, out, n.err);
  else
    k_conv32<false, true><<<blocks, 128, kConvSmem, n.stream>>>(in, B, n.H, n.W, w, bias, mask, out, n.err);
  TMBIR_CHECK_LAUNCH();
  return TMBIR_OK;
}
// TMBIR_ERR_TIMEOUT (and the flag cleared) when a convolution gave up waiting on the tensor core;
// reads the flag after the stream has drained up to here
static int check_tc(CnnNet& n) {
  int flag = 0;
  TMBIR_CUDA(cudaMemcpyAsync(&flag, n.err, sizeof(int), cudaMemcpyDeviceToHost, n.stream));
  TMBIR_CUDA(cudaStreamSynchronize(n.stream));
  if (flag) {
    TMBIR_CUDA(cudaMemsetAsync(n.err, 0, sizeof(int), n.stream));
    return set_error(TMBIR_ERR_TIMEOUT, "cnn: a tensor-core convolution timed out waiting for its MMAs");
  }
  return TMBIR_OK;
}

static int net_forward(CnnNet& n, int B) {
  const size_t P = (size_t)B * n.H * n.W;
  const int blocks = (int)std::min<size_t>((P + 255) / 256, 152 * 16);
  k_conv_first<<<blocks, 256, 0, n.stream>>>(n.xin, B, n.H, n.W, n.master, n.a0);
  TMBIR_CHECK_LAUNCH();
  if (int e = conv32(n, n.a0, B, n.wg1, n.master + kOffB1, nullptr, n.a1, true)) return e;
  if (int e = conv32(n, n.a1, B, n.wg2, n.master + kOffB2, nullptr, n.a2, true)) return e;
  k_conv_last<false><<<blocks, 256, 0, n.stream>>>(n.a2, B, n.H, n.W, n.master, n.out);
  TMBIR_CHECK_LAUNCH();
  return TMBIR_OK;
}

// dW and db of a 32 -> 32 layer into n.grad at `off` (weights, then the bias)
static int wgrad32(CnnNet& n, int B, const __nv_bfloat16* g, const __nv_bfloat16* in, int off) {
  static bool attr = false;
  if (!attr) {
    TMBIR_CUDA(cudaFuncSetAttribute(k_wgrad32, cudaFuncAttributeMaxDynamicSharedMemorySize, kGradSmem));
    attr = true;
  }
  const int tiles = B * ((n.H + kGRows - 1) / kGRows) * ((n.W + kTM - 1) / kTM);
  const int blocks = std::min(tiles, kWgradBlocks);
  k_wgrad32<<<blocks, 128, kGradSmem, n.stream>>>(g, in, B, n.H, n.W, n.wpart, n.err);
  TMBIR_CHECK_LAUNCH();
  k_reduce_parts<Layer::Hidden><<<(kPartRow + 31) / 32, 256, 0, n.stream>>>(n.wpart, blocks, kPartRow, n.grad + off, g, in,
                                                                            B, n.H, n.W);
  TMBIR_CHECK_LAUNCH();
  return TMBIR_OK;
}

// gradients of sum(gout * net(xin)) added into n.grad; gin (optional, FP32) receives d/dxin
static int net_backward(CnnNet& n, int B, float* gin) {
  const size_t P = (size_t)B * n.H * n.W;
  const int blocks = (int)std::min<size_t>((P + 255) / 256, 152 * 16);
  const int etiles = B * ((n.H + kEH - 1) / kEH) * ((n.W + kEW - 1) / kEW);
  const int eblocks = std::min(etiles, kWgradBlocks);
  // layer 3
  k_wgrad_edge<false><<<eblocks, 256, 0, n.stream>>>(n.a2, n.gout, B, n.H, n.W, n.wpart);
  TMBIR_CHECK_LAUNCH();
  k_reduce_parts<Layer::Last><<<(kW3 + kB3 + 31) / 32, 256, 0, n.stream>>>(n.wpart, eblocks, kW3 + kB3, n.grad + kOff3, n.a2,
                                                                           n.gout, B, n.H, n.W);
  TMBIR_CHECK_LAUNCH();
  k_last_dgrad<<<blocks, 256, 0, n.stream>>>(n.gout, n.a2, B, n.H, n.W, n.master, n.g2);
  TMBIR_CHECK_LAUNCH();
  // layer 2: weights from (g2, a1), then g1 = mask(a1) conv(g2, W2 flipped transposed)
  if (int e = wgrad32(n, B, n.g2, n.a1, kOff2)) return e;
  if (int e = conv32(n, n.g2, B, n.wt2, nullptr, n.a1, n.g1, false)) return e;
  // layer 1: weights from (g1, a0), then g0 = mask(a0) conv(g1, W1 flipped transposed) into g2's buffer
  if (int e = wgrad32(n, B, n.g1, n.a0, kOff1)) return e;
  __nv_bfloat16* g0 = n.g2;
  if (int e = conv32(n, n.g1, B, n.wt1, nullptr, n.a0, g0, false)) return e;
  // layer 0
  k_wgrad_edge<true><<<eblocks, 256, 0, n.stream>>>(g0, n.xin, B, n.H, n.W, n.wpart);
  TMBIR_CHECK_LAUNCH();
  k_reduce_parts<Layer::First><<<(kW0 + kB0 + 31) / 32, 256, 0, n.stream>>>(n.wpart, eblocks, kW0 + kB0, n.grad + kOff0, g0,
                                                                            n.xin, B, n.H, n.W);
  TMBIR_CHECK_LAUNCH();
  if (gin) {
    k_conv_last<true><<<blocks, 256, 0, n.stream>>>(g0, B, n.H, n.W, n.master, gin);
    TMBIR_CHECK_LAUNCH();
  }
  return TMBIR_OK;
}

static int pack(CnnNet& n) {
  k_cnn_pack<<<(kWElems + 255) / 256, 256, 0, n.stream>>>(n.master, n.wg1, n.wg2, n.wt1, n.wt2);
  TMBIR_CHECK_LAUNCH();
  return TMBIR_OK;
}

static int normalise(CnnNet& n, const float* x, int B) {
  const int HW = n.H * n.W;
  const size_t P = (size_t)B * HW;
  k_norm_partial<<<dim3(kNormBlocks, B), 256, 0, n.stream>>>(x, HW, n.dpart);
  TMBIR_CHECK_LAUNCH();
  k_norm_stats<<<B, 32, 0, n.stream>>>(n.dpart, HW, n.sig);
  TMBIR_CHECK_LAUNCH();
  k_scale_in<<<(int)std::min<size_t>((P + 255) / 256, 152 * 16), 256, 0, n.stream>>>(x, HW, P, n.sig, n.xin);
  TMBIR_CHECK_LAUNCH();
  return TMBIR_OK;
}

}  // namespace tmbir

using namespace tmbir;

struct tmbir_cnn {
  CnnNet n;
  size_t offs[20];
};

#define CNN_REQUIRE(cond, code, msg) \
  do {                               \
    if (!(cond)) return set_error(code, msg); \
  } while (0)

static bool al16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

extern "C" {

int tmbir_cnn_param_count(void) { return kParams; }

int tmbir_cnn_workspace_size(int max_batch, int H, int W, size_t* bytes) {
  CNN_REQUIRE(bytes && max_batch >= 1 && H >= 1 && W >= 1 && (size_t)max_batch * H * W < ((size_t)1 << 31),
              TMBIR_ERR_ARG, "cnn_workspace_size: bad sizes");
  size_t offs[20];
  *bytes = cnn_bytes(max_batch, H, W, offs);
  return TMBIR_OK;
}

int tmbir_cnn_create(tmbir_cnn** out, void* stream, int max_batch, int H, int W, void* d_ws, size_t bytes) {
  CNN_REQUIRE(out && d_ws && ((uintptr_t)d_ws & 255u) == 0, TMBIR_ERR_ARG,
              "cnn_create: NULL argument or workspace not 256-byte aligned");
  size_t need = 0;
  if (int e = tmbir_cnn_workspace_size(max_batch, H, W, &need)) return e;
  CNN_REQUIRE(bytes >= need, TMBIR_ERR_WORKSPACE, "cnn_create: workspace too small");
  tmbir_cnn* c = new tmbir_cnn();
  cnn_bytes(max_batch, H, W, c->offs);
  char* ws = static_cast<char*>(d_ws);
  CnnNet& n = c->n;
  n.stream = (cudaStream_t)stream;
  n.max_batch = max_batch;
  n.H = H;
  n.W = W;
  n.master = reinterpret_cast<float*>(ws + c->offs[0]);
  n.grad = reinterpret_cast<float*>(ws + c->offs[1]);
  n.adam_m = reinterpret_cast<float*>(ws + c->offs[2]);
  n.adam_v = reinterpret_cast<float*>(ws + c->offs[3]);
  n.wg1 = reinterpret_cast<__nv_bfloat16*>(ws + c->offs[4]);
  n.wg2 = reinterpret_cast<__nv_bfloat16*>(ws + c->offs[5]);
  n.wt1 = reinterpret_cast<__nv_bfloat16*>(ws + c->offs[6]);
  n.wt2 = reinterpret_cast<__nv_bfloat16*>(ws + c->offs[7]);
  n.a0 = reinterpret_cast<__nv_bfloat16*>(ws + c->offs[8]);
  n.a1 = reinterpret_cast<__nv_bfloat16*>(ws + c->offs[9]);
  n.a2 = reinterpret_cast<__nv_bfloat16*>(ws + c->offs[10]);
  n.g1 = reinterpret_cast<__nv_bfloat16*>(ws + c->offs[11]);
  n.g2 = reinterpret_cast<__nv_bfloat16*>(ws + c->offs[12]);
  n.xin = reinterpret_cast<float*>(ws + c->offs[13]);
  n.out = reinterpret_cast<float*>(ws + c->offs[14]);
  n.gout = reinterpret_cast<float*>(ws + c->offs[15]);
  n.sig = reinterpret_cast<float*>(ws + c->offs[16]);
  n.wpart = reinterpret_cast<float*>(ws + c->offs[17]);
  n.dpart = reinterpret_cast<double*>(ws + c->offs[18]);
  n.err = reinterpret_cast<int*>(ws + c->offs[19]);
  if (cudaMemsetAsync(n.err, 0, sizeof(int), n.stream) != cudaSuccess) {
    delete c;
    return set_error(TMBIR_ERR_CUDA, "cnn_create: cudaMemsetAsync failed");
  }
  n.step = 0;
  *out = c;
  return TMBIR_OK;
}

int tmbir_cnn_destroy(tmbir_cnn* net) {
  delete net;
  return TMBIR_OK;
}

int tmbir_cnn_set_weights(tmbir_cnn* net, const float* h_params) {
  CNN_REQUIRE(net && h_params, TMBIR_ERR_ARG, "cnn_set_weights: NULL argument");
  CnnNet& n = net->n;
  TMBIR_CUDA(cudaMemcpyAsync(n.master, h_params, kParams * sizeof(float), cudaMemcpyHostToDevice, n.stream));
  TMBIR_CUDA(cudaMemsetAsync(n.adam_m, 0, kParams * sizeof(float), n.stream));
  TMBIR_CUDA(cudaMemsetAsync(n.adam_v, 0, kParams * sizeof(float), n.stream));
  n.step = 0;
  if (int e = pack(n)) return e;
  TMBIR_CUDA(cudaStreamSynchronize(n.stream));
  return TMBIR_OK;
}

int tmbir_cnn_get_weights(tmbir_cnn* net, float* h_params) {
  CNN_REQUIRE(net && h_params, TMBIR_ERR_ARG, "cnn_get_weights: NULL argument");
  CnnNet& n = net->n;
  TMBIR_CUDA(cudaMemcpyAsync(h_params, n.master, kParams * sizeof(float), cudaMemcpyDeviceToHost, n.stream));
  TMBIR_CUDA(cudaStreamSynchronize(n.stream));
  return TMBIR_OK;
}

int tmbir_cnn_init(tmbir_cnn* net, unsigned long long seed) {
  CNN_REQUIRE(net, TMBIR_ERR_ARG, "cnn_init: NULL argument");
  std::mt19937_64 rng(seed);
  std::vector<float> p(kParams, 0.f);
  auto fill = [&](int off, int count, int fan_in, float gain) {
    std::normal_distribution<double> nd(0.0, gain * std::sqrt(2.0 / fan_in));
    for (int i = 0; i < count; ++i) p[off + i] = (float)nd(rng);
  };
  fill(kOff0, kW0, 9, 1.f);
  fill(kOff1, kW1, 9 * kC, 1.f);
  fill(kOff2, kW1, 9 * kC, 1.f);
  fill(kOff3, kW3, 9 * kC, 0.1f);  // small last layer: the refiner starts close to the identity
  return tmbir_cnn_set_weights(net, p.data());
}

int tmbir_cnn_net_forward(tmbir_cnn* net, const float* d_in, int batch, float* d_out) {
  TMBIR_TRACE("tmbir_cnn_net_forward");
  CNN_REQUIRE(net && d_in && d_out && al16(d_in) && al16(d_out), TMBIR_ERR_ARG, "cnn_net_forward: bad buffers");
  CnnNet& n = net->n;
  CNN_REQUIRE(batch >= 1 && batch <= n.max_batch, TMBIR_ERR_ARG, "cnn_net_forward: batch out of range");
  const size_t P = (size_t)batch * n.H * n.W;
  TMBIR_CUDA(cudaMemcpyAsync(n.xin, d_in, P * sizeof(float), cudaMemcpyDeviceToDevice, n.stream));
  if (int e = net_forward(n, batch)) return e;
  TMBIR_CUDA(cudaMemcpyAsync(d_out, n.out, P * sizeof(float), cudaMemcpyDeviceToDevice, n.stream));
  return TMBIR_OK;
}

int tmbir_cnn_net_backward(tmbir_cnn* net, const float* d_in, const float* d_gout, int batch, float* h_gparams,
                           float* d_gin) {
  TMBIR_TRACE("tmbir_cnn_net_backward");
  CNN_REQUIRE(net && d_in && d_gout && h_gparams && al16(d_in) && al16(d_gout) && (!d_gin || al16(d_gin)),
              TMBIR_ERR_ARG, "cnn_net_backward: bad buffers");
  CnnNet& n = net->n;
  CNN_REQUIRE(batch >= 1 && batch <= n.max_batch, TMBIR_ERR_ARG, "cnn_net_backward: batch out of range");
  const size_t P = (size_t)batch * n.H * n.W;
  TMBIR_CUDA(cudaMemcpyAsync(n.xin, d_in, P * sizeof(float), cudaMemcpyDeviceToDevice, n.stream));
  if (int e = net_forward(n, batch)) return e;
  TMBIR_CUDA(cudaMemcpyAsync(n.gout, d_gout, P * sizeof(float), cudaMemcpyDeviceToDevice, n.stream));
  TMBIR_CUDA(cudaMemsetAsync(n.grad, 0, kParams * sizeof(float), n.stream));
  if (int e = net_backward(n, batch, d_gin)) return e;
  TMBIR_CUDA(cudaMemcpyAsync(h_gparams, n.grad, kParams * sizeof(float), cudaMemcpyDeviceToHost, n.stream));
  return check_tc(n);
}

int tmbir_cnn_apply(tmbir_cnn* net, const float* d_x, int batch, float* d_y) {
  TMBIR_TRACE("tmbir_cnn_apply");
  CNN_REQUIRE(net && d_x && d_y && al16(d_x) && al16(d_y), TMBIR_ERR_ARG, "cnn_apply: bad buffers");
  CnnNet& n = net->n;
  CNN_REQUIRE(batch >= 1 && batch <= n.max_batch, TMBIR_ERR_ARG, "cnn_apply: batch out of range");
  const size_t P = (size_t)batch * n.H * n.W;
  if (int e = normalise(n, d_x, batch)) return e;
  if (int e = net_forward(n, batch)) return e;
  k_residual_out<<<(int)std::min<size_t>((P + 255) / 256, 152 * 16), 256, 0, n.stream>>>(d_x, n.out, n.H * n.W, P,
                                                                                        n.sig, d_y);
  TMBIR_CHECK_LAUNCH();
  return TMBIR_OK;
}

int tmbir_cnn_train_step(tmbir_cnn* net, const float* d_x, const float* d_target, int batch, float lr, double* h_loss) {
  TMBIR_TRACE("tmbir_cnn_train_step");
  CNN_REQUIRE(net && d_x && d_target && al16(d_x) && al16(d_target), TMBIR_ERR_ARG, "cnn_train_step: bad buffers");
  CnnNet& n = net->n;
  CNN_REQUIRE(batch >= 1 && batch <= n.max_batch && lr > 0.f, TMBIR_ERR_ARG, "cnn_train_step: bad batch or rate");
  const size_t P = (size_t)batch * n.H * n.W;
  if (int e = normalise(n, d_x, batch)) return e;
  if (int e = net_forward(n, batch)) return e;
  const int lb = 1024;
  k_loss<<<lb, 256, 0, n.stream>>>(n.out, d_x, d_target, n.H * n.W, P, n.sig, n.gout, n.dpart);
  TMBIR_CHECK_LAUNCH();
  k_sum_d<<<1, 32, 0, n.stream>>>(n.dpart, lb, 1.0 / (double)P, n.dpart + lb);
  TMBIR_CHECK_LAUNCH();
  TMBIR_CUDA(cudaMemsetAsync(n.grad, 0, kParams * sizeof(float), n.stream));
  if (int e = net_backward(n, batch, nullptr)) return e;
  n.step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)n.step), c2 = 1.f - std::pow(b2, (float)n.step);
  k_adam<<<(kParams + 255) / 256, 256, 0, n.stream>>>(n.master, n.grad, n.adam_m, n.adam_v, kParams, lr, b1, b2, 1e-8f,
                                                      c1, c2);
  TMBIR_CHECK_LAUNCH();
  if (int e = pack(n)) return e;
  if (h_loss) {
    TMBIR_CUDA(cudaMemcpyAsync(h_loss, n.dpart + lb, sizeof(double), cudaMemcpyDeviceToHost, n.stream));
    return check_tc(n);
  }
  return TMBIR_OK;
}

int tmbir_warm_start(tmbir_ctx* ctx, tmbir_cnn* net, const float* d_fbp, const float* d_atg, const tmbir_params* prm,
                     float* d_x0, int* h_used_cnn) {
  TMBIR_TRACE("tmbir_warm_start");
  CNN_REQUIRE(ctx && net && d_fbp && d_atg && prm && d_x0 && al16(d_fbp) && al16(d_x0), TMBIR_ERR_ARG,
              "warm_start: bad arguments");
  CNN_REQUIRE(d_x0 != d_fbp, TMBIR_ERR_ARG, "warm_start: output must not alias the FBP start");
  Ctx& c = ctx->c;
  CnnNet& n = net->n;
  CNN_REQUIRE(c.groups.size() == 1 && c.groups[0].N == n.H && n.H == n.W, TMBIR_ERR_SHAPE,
              "warm_start: needs one geometry group whose N equals the network's image size");
  const int S = c.groups[0].n_slices;
  const size_t HW = (size_t)n.H * n.W;
  // the network runs on its own stream: it starts after the context's pending work and the
  // objectives below start after it
  cudaEvent_t ev[2] = {nullptr, nullptr};
  if (n.stream != c.stream) {
    TMBIR_CUDA(cudaEventCreateWithFlags(&ev[0], cudaEventDisableTiming));
    if (cudaEventCreateWithFlags(&ev[1], cudaEventDisableTiming) != cudaSuccess) {
      cudaEventDestroy(ev[0]);
      return set_error(TMBIR_ERR_CUDA, "warm_start: cudaEventCreate failed");
    }
  }
  auto release = [&](int e) {
    for (cudaEvent_t x : ev)
      if (x) cudaEventDestroy(x);
    return e;
  };
  if (ev[0]) {
    if (cudaEventRecord(ev[0], c.stream) != cudaSuccess || cudaStreamWaitEvent(n.stream, ev[0], 0) != cudaSuccess)
      return release(set_error(TMBIR_ERR_CUDA, "warm_start: stream ordering failed"));
  }
  for (int s0 = 0; s0 < S; s0 += n.max_batch) {
    const int b = std::min(n.max_batch, S - s0);
    if (int e = tmbir_cnn_apply(net, d_fbp + s0 * HW, b, d_x0 + s0 * HW)) return release(e);
  }
  if (ev[1]) {
    if (cudaEventRecord(ev[1], n.stream) != cudaSuccess || cudaStreamWaitEvent(c.stream, ev[1], 0) != cudaSuccess)
      return release(set_error(TMBIR_ERR_CUDA, "warm_start: stream ordering failed"));
  }
  release(0);
  double F_cnn = 0.0, F_fbp = 0.0;
  if (int e = tmbir_objective(ctx, d_x0, d_atg, prm, &F_cnn)) return e;
  if (int e = tmbir_objective(ctx, d_fbp, d_atg, prm, &F_fbp)) return e;
  const int use = F_cnn < F_fbp ? 1 : 0;
  if (!use) TMBIR_CUDA(cudaMemcpyAsync(d_x0, d_fbp, S * HW * sizeof(float), cudaMemcpyDeviceToDevice, c.stream));
  if (h_used_cnn) *h_used_cnn = use;
  return check_tc(n);
}

}  // extern "C"

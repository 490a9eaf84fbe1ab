// The per-iteration hot path: R*R y as a zero-padded 2N x 2N FFT convolution with the
// point-spread kernel (Sec. 2.1, Eq. 9), fused with -R*g (Eq. 11), the qGGMRF prior
// gradient over the 26-neighbourhood (Eq. 5, Sec. 2.4) and the fast-gradient update with
// restart (Sec. 2, Eq. 6).
//
// Four launches per iteration, each over every slice of a group:
//   pass 1  rows:    y = x_k + beta (x_k - x_{k-1}); real FFT of length 2N of each row (the
//                    upper N entries are the zero padding), written column-major
//                    spec[v][r], v = 0..N (half spectrum), r = 0..N-1 (nonzero rows only).
//   pass 2  columns: per column v, FFT of length 2N of the N nonzero rows, multiply by the
//                    real kernel spectrum, inverse FFT, keep the first N rows (the crop).
//                    The length-2N transforms are split into their even and odd halves, two
//                    length-N transforms each (above 1024 into 2N/512 of 512 points), so the
//                    zero padding and the crop cost nothing.
//   pass 3a rows:    inverse real FFT of each row, keep the first N columns -> K (*) y.
//   pass 3b stencil: per voxel G = K(*)y - R*g + lambda grad Phi(y) (each neighbour pair of the
//                    26-neighbourhood evaluated once), x_{k+1} = y - G/L, and the partial sums
//                    the optimiser needs (compensated FP32 per thread, FP64 per block).
// A finalize kernel (one block) reduces the partials in a fixed order and advances the
// device-resident momentum state, so a whole run needs no host round trip.
//
// The intermediate spectrum is stored as FP32 complex, or (BF = true) as BF16 pairs with all
// arithmetic still in FP32: the storage halves and every transform accumulates in FP32.
#pragma once
#include <cuda_bf16.h>

#include "fft.cuh"
#include "internal.h"
#include "tc05.cuh"

namespace tmbir {

// ---------------------------------------------------------------- spectrum storage
template <bool BF>
struct SpecIO;
template <>
struct SpecIO<false> {
  using T = float2;
  __device__ __forceinline__ static float2 ld(const T* p, size_t i) { return p[i]; }
  __device__ __forceinline__ static void st(T* p, size_t i, float2 v) { p[i] = v; }
};
template <>
struct SpecIO<true> {
  using T = __nv_bfloat162;
  __device__ __forceinline__ static float2 ld(const T* p, size_t i) { return __bfloat1622float2(p[i]); }
  __device__ __forceinline__ static void st(T* p, size_t i, float2 v) { p[i] = __float22bfloat162_rn(v); }
};
// In Iterate mode every pass checks the run's current storage phase and leaves when it is
// not its own, so the BF16 and FP32 variants can be enqueued back to back.
template <bool BF>
__device__ __forceinline__ bool skip_iter(const IterState* st) {
  return st->done || (st->bf16 != 0) != BF;
}

// Copies count elements, e = threadIdx.x + k * NT, from ld(e) to st(e, v) in batches of B whose
// loads are all issued before their stores, so that a thread keeps B global loads in flight
// instead of waiting out each load's latency before the next.
template <int NT, int B, class Ld, class St>
__device__ __forceinline__ void batched_copy(int count, Ld&& ld, St&& st) {
  for (int e0 = threadIdx.x; e0 < count; e0 += B * NT) {
    float2 v[B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int e = e0 + b * NT;
      v[b] = e < count ? ld(e) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int e = e0 + b * NT;
      if (e < count) st(e, v[b]);
    }
  }
}

// ---------------------------------------------------------------- launch geometry
template <int N, int Wp = 4>
struct Geo {
  using F = typename FFTShape<N>::type;
  static constexpr int T = F::T, P = F::P, G = 32 / T;
  static constexpr int W = Wp;          // warps per block
  static constexpr int THREADS = 32 * W;
  static constexpr int RB = W * G;      // rows per block in passes 1 and 3
  static constexpr int NB = N / RB;     // row blocks per slice
  static constexpr int LD = N + 4;      // row stride (complex) of the row-major staging buffer
  static constexpr int UNITS = W * G;   // (column, half) units per block in pass 2
  static constexpr int CPB = UNITS / 2; // columns per block in pass 2
  static constexpr size_t SM_FFT = (size_t)W * G * F::SMEM * sizeof(float2);
  static constexpr size_t SM_TB = (size_t)RB * LD * sizeof(float2);
  static constexpr size_t cmax(size_t a, size_t b) { return a > b ? a : b; }
  static constexpr size_t SM1 = cmax(SM_FFT, SM_TB);
  static constexpr size_t SM2 = SM_FFT;
};

// Launch shapes of pass 3a and pass 2 at N = 1024, chosen by measurement on GB300 (64 slices,
// 256 angles; ms per launch):
//   pass 3a: eight warps per block gather 8-row (64-byte) segments of the column-major
//            spectrum instead of 4-row (32-byte) ones; with at most 128 registers (two blocks
//            per SM) 0.211 ms against 0.262 with four warps (0.252 with eight warps at the
//            compiler's register choice, 0.278 at three blocks per SM).  Eight warps do not
//            help pass 1 (0.234 against 0.230), which keeps four.
//   pass 2:  at most 170 registers (three blocks per SM), 0.401 ms against 0.407 (128
//            registers: 0.588, spills).
// The other image sides keep four warps and the compiler's register choice.
#if defined(TMBIR_N) && TMBIR_N == 1024
#define TMBIR_P3A_BOUNDS(T) __launch_bounds__(T, 2)
#define TMBIR_P2_BOUNDS(T) __launch_bounds__(T, 3)
#else
#define TMBIR_P3A_BOUNDS(T) __launch_bounds__(T)
#define TMBIR_P2_BOUNDS(T) __launch_bounds__(T)
#endif
template <int N>
constexpr int pass3a_warps() {
  return N == 1024 ? 8 : 4;
}
template <int N>
using Geo3a = Geo<N, pass3a_warps<N>()>;

// ---------------------------------------------------------------- special-function unit helpers
__device__ __forceinline__ float ex2a(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2a(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcpa(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Packed FP32 pairs: one instruction computes both lanes of a float2 (sm_100 and later).
__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }
// the largest of three values, NaN if one of them is
__device__ __forceinline__ float max_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 f2mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 f2add(float2 a, float2 b) { return __fadd2_rn(a, b); }

// the row passes' rotations keep the remainder of 1/sqrt(2) (twmul), except beside BF16 spectra, whose
// rounding is 2^15 times larger
template <int DIR, bool BF>
constexpr int kRowDir = BF ? DIR : 2 * DIR;
// and pass 2's at 1536, whose columns rotate by odd multiples of pi/4 more often than in the four radix
// stages that the 512-point split replaced: without it R*R's error there is 2.63e-7 (4 slices of noise, 64
// angles), with it 2.53e-7, with the stages 2.58e-7.  8 x 1536^2: 143 -> 148 us
template <int DIR, int N, bool BF>
constexpr int kColDir = !BF && N == 1536 ? 2 * DIR : DIR;

// ---------------------------------------------------------------- pass 1: rows, forward
template <int N, bool BF>
__global__ void __launch_bounds__(Geo<N>::THREADS) k_pass1(const __grid_constant__ GroupSet gs, StepArgs a) {
  using Gm = Geo<N>;
  using F = typename Gm::F;
  constexpr int T = Gm::T, P = Gm::P, G = Gm::G, RB = Gm::RB, LD = Gm::LD;
  extern __shared__ float2 sm[];
  int bid_;
  const int gi_ = gs.pick(bid_);
  const GroupDev& g = gs.g[gi_];
  const float *x, *xp;
  float beta;
  if (a.st) {
    if (skip_iter<BF>(a.st)) return;
    int cur = a.st->cur;
    // selects rather than an indexed parameter array, which would be copied to local memory
    x = cur == 0 ? a.xb[0] : (cur == 1 ? a.xb[1] : a.xb[2]);
    xp = cur == 0 ? a.xb[2] : (cur == 1 ? a.xb[0] : a.xb[1]);
    beta = (float)(a.gm + gi_)->beta;
  } else {
    x = a.x;
    xp = a.xprev;
    beta = a.beta;
  }
  const int s = bid_ / Gm::NB, rb = bid_ % Gm::NB;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane / T, t = lane % T;
  const int rl = warp * G + grp;
  const int r = rb * RB + rl;
  const size_t base = g.img_off + ((size_t)s * N + r) * N;

  // packed real row: z[n] = y[2n] + i y[2n+1], nonzero for n < N/2 (the rest is padding)
  float2 v[P];
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    if constexpr (i < P / 2) {
      const int n = t + T * i;
      float2 xv = __ldg(reinterpret_cast<const float2*>(x + base) + n);
      float2 pv = __ldg(reinterpret_cast<const float2*>(xp + base) + n);
      v[i] = make_float2(fmaf(beta, xv.x - pv.x, xv.x), fmaf(beta, xv.y - pv.y, xv.y));
    } else {
      v[i] = make_float2(0.f, 0.f);
    }
  });
  F::template run<kRowDir<-1, BF>>(v, sm + (warp * G + grp) * F::SMEM, g.twN, t);

  // split the packed transform: Y[v] = E[v] + w^v O[v], needs Z[v] and Z[N - v]
  float2 y[P];
  const int partner = (T - t) % T;
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    float2 zo = v[P - 1 - i];
    float2 zs;
    zs.x = __shfl_sync(0xffffffffu, zo.x, partner, T);
    zs.y = __shfl_sync(0xffffffffu, zo.y, partner, T);
    if (t == 0) zs = v[(P - i) % P];
    float2 z = v[i];
    float2 e = make_float2(0.5f * (z.x + zs.x), 0.5f * (z.y - zs.y));
    float2 o = make_float2(0.5f * (z.y + zs.y), -0.5f * (z.x - zs.x));
    float2 w = __ldg(&g.twM[t + T * i]);
    y[i] = cadd(e, cmul(w, o));
  });
  const float nyq = v[0].x - v[0].y;
  __syncthreads();
  float2* tb = sm;
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    tb[rl * LD + t + T * i] = y[i];
  });
  if (t == 0) tb[rl * LD + N] = make_float2(nyq, 0.f);
  __syncthreads();
  using IO = SpecIO<BF>;
  typename IO::T* out = reinterpret_cast<typename IO::T*>(g.spec) + (size_t)s * (N + 1) * N + rb * RB;
  for (int e = threadIdx.x; e < (N + 1) * RB; e += Gm::THREADS) {
    const int vv = e / RB, rr = e - vv * RB;
    IO::st(out, (size_t)vv * N + rr, tb[rr * LD + vv]);
  }
}

// ---------------------------------------------------------------- pass 2: columns
// Column order of pass 2: chunks of kColChunk slices, and within a chunk the slices fastest, so
// that consecutive blocks share a column of the kernel spectrum (L2 reuse) while the blocks in
// flight stay within a few hundred MB of the spectrum instead of spreading over every slice of
// a large volume (TLB reach).  Column index -> (kernel column vcol, slice s).
constexpr int kColChunk = 16;
__device__ __forceinline__ void column_of(int col, int S, int ncol, int& vcol, int& s) {
  const int chunk = col / (kColChunk * ncol);
  const int within = col - chunk * kColChunk * ncol;
  const int rem = min(kColChunk, S - chunk * kColChunk);
  vcol = within / rem;
  s = chunk * kColChunk + (within - vcol * rem);
}

template <int N, bool BF>
__global__ void TMBIR_P2_BOUNDS(Geo<N>::THREADS) k_pass2(const __grid_constant__ GroupSet gs, const IterState* st) {
  using Gm = Geo<N>;
  using F = typename Gm::F;
  constexpr int T = Gm::T, P = Gm::P, G = Gm::G;
  extern __shared__ float2 sm[];
  int bid_;
  const int gi_ = gs.pick(bid_);
  const GroupDev& g = gs.g[gi_];
  if (st && skip_iter<BF>(st)) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane / T, t = lane % T;
  const int unit = warp * G + grp, h = unit & 1;
  const int col = bid_ * Gm::CPB + (unit >> 1);
  const int ncols = g.S * (N + 1);
  const bool active = col < ncols;
  int vcol = 0, s = 0;
  if (active) column_of(col, g.S, N + 1, vcol, s);
  using IO = SpecIO<BF>;
  typename IO::T* p = reinterpret_cast<typename IO::T*>(g.spec) + ((size_t)s * (N + 1) + vcol) * N;
  float2 v[P];
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    const int rr = t + T * i;
    float2 w = active ? IO::ld(p, rr) : make_float2(0.f, 0.f);
    if (h) w = cmul(w, __ldg(&g.twM[rr]));  // odd half: w[r] * exp(-2 pi i r / 2N)
    v[i] = w;
  });
  float2* xs = sm + unit * F::SMEM;
  F::template run<-1>(v, xs, g.twN, t);
  const float* cc = g.chat + ((size_t)vcol * 2 + h) * N;
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    const float c = __ldg(&cc[t + T * i]);
    v[i] = make_float2(v[i].x * c, v[i].y * c);
  });
  F::template run<1>(v, xs, g.twN, t);
  if (h) {
    SFor<0, P>::run([&](auto i_) {
      constexpr int i = decltype(i_)::value;
      v[i] = cmulc(v[i], __ldg(&g.twM[t + T * i]));
    });
  }
  // even and odd units can share a warp (N <= 512): every lane reaches this barrier
  __syncwarp();
  if (h) {
    SFor<0, P>::run([&](auto i_) {
      constexpr int i = decltype(i_)::value;
      xs[t + T * i] = v[i];
    });
  }
  __syncthreads();
  if (!h && active) {
    const float2* os = sm + (unit + 1) * F::SMEM;
    SFor<0, P>::run([&](auto i_) {
      constexpr int i = decltype(i_)::value;
      const int rr = t + T * i;
      IO::st(p, rr, cadd(v[i], os[rr]));
    });
  }
}

// ---------------------------------------------------------------- pass 3a: rows, inverse
// Inverse packed real row transform of every row (one row group per warp, RB rows per block,
// the layout of pass 1), crop to the first N columns: K (*) y written row-major as FP32.
template <int N, bool BF>
__global__ void TMBIR_P3A_BOUNDS(Geo3a<N>::THREADS) k_pass3a(const __grid_constant__ GroupSet gs, const IterState* st, float* apply_out) {
  using Gm = Geo3a<N>;
  using F = typename Gm::F;
  constexpr int T = Gm::T, P = Gm::P, G = Gm::G, RB = Gm::RB, LD = Gm::LD;
  extern __shared__ float2 sm[];
  int bid_;
  const int gi_ = gs.pick(bid_);
  const GroupDev& g = gs.g[gi_];
  float* kz = apply_out ? apply_out + g.img_off : g.kz;
  if (st && skip_iter<BF>(st)) return;
  const int s = bid_ / Gm::NB, rb = bid_ % Gm::NB;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane / T, t = lane % T;
  const int rl = warp * G + grp;
  const int r0 = rb * RB;
  float2* tb = sm;
  {
    using IO = SpecIO<BF>;
    const typename IO::T* sp = reinterpret_cast<const typename IO::T*>(g.spec) + (size_t)s * (N + 1) * N + r0;
    if constexpr (!BF) {
      // RB-row segments of the column-major spectrum, gathered by asynchronous 8-byte copies so
      // that every thread has all of its loads in flight at once
      for (int e = threadIdx.x; e < (N + 1) * RB; e += Gm::THREADS) {
        const int vv = e / RB, rr = e - vv * RB;
        tc05::cp_async8(&tb[rr * LD + vv], sp + (size_t)vv * N + rr);
      }
      tc05::cp_async_wait_all();
    } else {
      batched_copy<Gm::THREADS, 8>(
          (N + 1) * RB, [&](int e) { return IO::ld(sp, (size_t)(e / RB) * N + e % RB); },
          [&](int e, float2 v) { tb[(e % RB) * LD + e / RB] = v; });
    }
  }
  __syncthreads();
  // the length-2N real inverse as a length-N complex inverse of Z[v] = E[v] + i O[v]
  float2 q[P];
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    const int vp = t + T * i;
    const float2 zv = tb[rl * LD + vp];
    const float2 zr = tb[rl * LD + N - vp];
    const float2 e = make_float2(zv.x + zr.x, zv.y - zr.y);
    const float2 d = make_float2(zv.x - zr.x, zv.y + zr.y);
    const float2 o = cmulc(d, __ldg(&g.twM[vp]));
    q[i] = make_float2(e.x - o.y, e.y + o.x);
  });
  __syncthreads();
  F::template run<kRowDir<1, BF>>(q, sm + (warp * G + grp) * F::SMEM, g.twN, t);
  // the first N/2 packed outputs are the N kept columns
  float2* out = reinterpret_cast<float2*>(kz + ((size_t)s * N + r0 + rl) * N);
  SFor<0, P / 2>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    out[t + T * i] = q[i];
  });
}

// ---------------------------------------------------------------- passes 1, 2, 3a for 1536, 2048 and 2560
// N = 512 J (J = 3, 4, 5): every transform is split into transforms of 512 points, one register group
// FFT (16 threads x 32 values) each, by a J-point DFT and a twiddle in registers before (forward) or
// after (inverse) it, which is also where the zero padding and the crop are pruned.  Layouts, scaling
// and the packed-real split are those of the other passes (w = exp(-2 pi i / N), W = exp(-2 pi i / 2N)):
//   pass 1: the packed row z has N/2 nonzero values,
//           Z[J k + j] = DFT_512(w^(jm) sum_q z[m + 512 q] exp(-2 pi i j q / J))[k];
//   pass 2: the column c has N nonzero values of 2N,
//           X[2J k + j] = DFT_512(W^(jm) sum_q c[m + 512 q] exp(-2 pi i j q / 2J))[k], the even and odd j
//           as two J-point DFTs; after the kernel multiply the kept rows m + 512 q are
//           sum_j W^(-jm) exp(2 pi i j q / 2J) u_j[m], u_j the inverse 512-point transforms;
//   pass 3a: z[m + 512 q] = sum_j w^(-jm) exp(2 pi i j q / J) u_j[m], u_j of Z[J k + j].
// A shared-memory round trip carries the values between the J-point DFTs (threads along m) and the
// group FFTs (one per j), and one more is inside each group FFT.
//
// Bound by the shared-memory / L1 data pipe (72, 69 and 50 % busy in passes 1, 2 and 3a at 2048; 3a, one
// block per SM, also waits for its gather), so its wavefronts are what the
// layouts save: twiddles come from tables that are contiguous in m (W^m, W^2m, W^4m, W^8m; the others
// are one product of two of these), the kernel spectrum is stored per j, and for J = 4 a staged row
// keeps the four residues of v apart (stride-4 accesses would meet in four banks).  Measured per
// launch, pass 1 / 2 / 3a: 6 x 2560^2 177 / 369 / 179 us, 8 x 1536^2 92 / 148 / 96 us (632 / 1215 /
// 570 and 188 / 448 / 212 us with the four-stage block-wide Stockham transform, five round trips with a
// block barrier each, that this replaced); 32 x 2048^2 540 / 932 / 582 us (707 / 1026 / 690 us with
// 1024-point transforms of one warp).
template <int N, int RBp = 4>
struct GeoH {
  static constexpr int H = 512, J = N / H, J2 = 2 * J;
  using F = GroupFFT<16, 32>;
  static constexpr int RB = RBp;                          // rows per block of passes 1 and 3a
  static constexpr int NB = N / RB;
  static constexpr int UNITS = RB * J;                    // group FFTs per block in passes 1 and 3a
  static constexpr int THREADS = 16 * UNITS;
  // staged rows (complex): place of v = J k + j in a row, row stride.  The half-warps of the split
  // take four rows x four consecutive v, those of the group FFTs 16 consecutive k.
  static constexpr bool PLANES = J == 4;
  static constexpr int HP = H + 4;
  static constexpr int LDZ = PLANES ? J * HP + 1 : N + 4;
  __device__ __forceinline__ static int place(int v) { return PLANES ? (v % J) * HP + v / J : v; }
  __device__ __forceinline__ static int place(int k, int j) { return PLANES ? j * HP + k : J * k + j; }
  static constexpr int THREADS2 = 16 * J2;                // pass 2: one column per block
  static constexpr size_t SM_ROWS = (size_t)(RB * LDZ > UNITS * F::SMEM ? RB * LDZ : UNITS * F::SMEM) * sizeof(float2);
  static constexpr size_t SM_COL = (size_t)J2 * F::SMEM * sizeof(float2);
  static_assert(N % H == 0 && THREADS % 32 == 0 && THREADS2 % 32 == 0, "split");
};

// Pass 3a gathers eight rows (64-byte segments of the column-major spectrum, half the load
// wavefronts of four): 582 against 647 us at 32 x 2048^2, 96 against 112 us at 8 x 1536^2.  Not at 2560:
// 40 group FFTs are a block of 640 threads and 169 KB, the only one of its SM, which measured 190 us
// against 179 with two blocks of 320 threads and four rows (at 2048 eight rows are one block of 512 threads
// as well, and still win).  Pass 1, whose stores need no registers while they are in flight, keeps four
// rows and three blocks per SM (540 against 636 us at 2048).
template <int N>
using GeoH3 = GeoH<N, N == 2560 ? 4 : 8>;

// w[j] = W^(2^L j m) for j < J: the powers of two from the side's tables (twM[m] = W^m,
// twN[512 l + m] = W^(2^l m)), the others as one product of two of them (7 = 4 + 3: two products)
template <int L, int J>
__device__ __forceinline__ void tw_powers(const GroupDev& g, int m, float2 (&w)[J]) {
  SFor<1, J>::run([&](auto j_) {
    constexpr int j = decltype(j_)::value;
    constexpr int l = j >= 8 ? 3 : (j >= 4 ? 2 : (j >= 2 ? 1 : 0));
    if constexpr (j == 1 << l)
      w[j] = __ldg(L + l == 0 ? &g.twM[m] : &g.twN[512 * (L + l) + m]);
    else
      w[j] = cmul(w[1 << l], w[j - (1 << l)]);
  });
}

template <int N, bool BF>
__global__ void __launch_bounds__(GeoH<N>::THREADS) k_pass1_h(const __grid_constant__ GroupSet gs, StepArgs a) {
  using Q = GeoH<N>;
  using F = typename Q::F;
  constexpr int J = Q::J, H = Q::H, RB = Q::RB, LDZ = Q::LDZ, T = F::T, P = F::P;
  extern __shared__ float2 sm[];
  int bid_;
  const int gi_ = gs.pick(bid_);
  const GroupDev& g = gs.g[gi_];
  const float *x, *xp;
  float beta;
  if (a.st) {
    if (skip_iter<BF>(a.st)) return;
    const int cur = a.st->cur;
    // selects rather than an indexed parameter array, which would be copied to local memory
    x = cur == 0 ? a.xb[0] : (cur == 1 ? a.xb[1] : a.xb[2]);
    xp = cur == 0 ? a.xb[2] : (cur == 1 ? a.xb[0] : a.xb[1]);
    beta = (float)(a.gm + gi_)->beta;
  } else {
    x = a.x;
    xp = a.xprev;
    beta = a.beta;
  }
  const int s = bid_ / Q::NB, rb = bid_ % Q::NB;
  const size_t base = g.img_off + ((size_t)s * N + rb * RB) * N;
  // packed rows z[m] = y[2m] + i y[2m+1], m < N/2, through the J-point DFTs into the units' buffers
#pragma unroll 2
  for (int e = threadIdx.x; e < RB * H; e += Q::THREADS) {
    const int rr = e / H, m = e % H;
    const float2* xr = reinterpret_cast<const float2*>(x + base + (size_t)rr * N);
    const float2* pr = reinterpret_cast<const float2*>(xp + base + (size_t)rr * N);
    float2 c[J], w[J];
    SFor<0, J>::run([&](auto q_) {
      constexpr int q = decltype(q_)::value;
      c[q] = make_float2(0.f, 0.f);
      if constexpr (q * H < N / 2) {
        if ((q + 1) * H <= N / 2 || m < N / 2 - q * H) {
          const float2 xv = __ldg(xr + m + q * H), pv = __ldg(pr + m + q * H);
          c[q] = make_float2(fmaf(beta, xv.x - pv.x, xv.x), fmaf(beta, xv.y - pv.y, xv.y));
        }
      }
    });
    tw_powers<1>(g, m, w);
    reg_dft<J, -1, float2>(c);
    float2* b = sm + rr * J * F::SMEM + m;
    SFor<0, J>::run([&](auto j_) {
      constexpr int j = decltype(j_)::value;
      b[j * F::SMEM] = j ? cmul(c[j], w[j]) : c[j];
    });
  }
  __syncthreads();
  const int unit = threadIdx.x / T, t = threadIdx.x % T, rl = unit / J, j = unit - rl * J;
  float2* xs = sm + unit * F::SMEM;
  float2 v[P];
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    v[i] = xs[t + T * i];
  });
  F::template run<kRowDir<-1, BF>>(v, xs, g.twN, t);
  __syncthreads();  // every exchange buffer is free: the staged rows alias them
  float2* zrow = sm + rl * LDZ;
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    zrow[Q::place(t + T * i, j)] = v[i];
  });
  __syncthreads();
  // split Y[v] = E[v] + W^v O[v] with E = (Z[v] + conj Z[N - v]) / 2, O = (Z[v] - conj Z[N - v]) / 2i,
  // two mirrored outputs at a time: E[N - v] = conj E[v], O[N - v] = conj O[v] and
  // W^(N - v) = -conj W^v give Y[N - v] = conj(E[v] - W^v O[v]) (v = 0: Y[N] = Re Z[0] - Im Z[0]);
  // written column-major (RB-row segments)
  using IO = SpecIO<BF>;
  typename IO::T* out = reinterpret_cast<typename IO::T*>(g.spec) + (size_t)s * (N + 1) * N + rb * RB;
#pragma unroll 2
  for (int e = threadIdx.x; e < (N / 2 + 1) * RB; e += Q::THREADS) {
    const int vv = e / RB, rr = e - vv * RB;
    const float2* zr = sm + rr * LDZ;
    const float2 z = zr[Q::place(vv)], zs = zr[Q::place(vv ? N - vv : 0)];
    const float2 ev = make_float2(0.5f * (z.x + zs.x), 0.5f * (z.y - zs.y));
    const float2 od = make_float2(0.5f * (z.y + zs.y), -0.5f * (z.x - zs.x));
    const float2 wo = cmul(__ldg(&g.twM[vv]), od);
    IO::st(out, (size_t)vv * N + rr, cadd(ev, wo));
    if (vv != N / 2) IO::st(out, (size_t)(N - vv) * N + rr, make_float2(ev.x - wo.x, wo.y - ev.y));
  }
}

template <int N, bool BF>
__global__ void __launch_bounds__(GeoH<N>::THREADS2) k_pass2_h(const __grid_constant__ GroupSet gs, const IterState* st) {
  using Q = GeoH<N>;
  using F = typename Q::F;
  constexpr int J = Q::J, J2 = Q::J2, H = Q::H, T = F::T, P = F::P, NT = Q::THREADS2;
  extern __shared__ float2 sm[];
  int bid_;
  const int gi_ = gs.pick(bid_);
  const GroupDev& g = gs.g[gi_];
  if (st && skip_iter<BF>(st)) return;
  int vcol, s;
  column_of(bid_, g.S, N + 1, vcol, s);
  using IO = SpecIO<BF>;
  typename IO::T* p = reinterpret_cast<typename IO::T*>(g.spec) + ((size_t)s * (N + 1) + vcol) * N;
  // the J values of each m through the two J-point DFTs into the units' buffers
  constexpr int IT = (H + NT - 1) / NT;
  float2 c[IT][J];
  SFor<0, IT>::run([&](auto k_) {
    constexpr int k = decltype(k_)::value;
    const int m = threadIdx.x + k * NT;
    SFor<0, J>::run([&](auto q_) {
      constexpr int q = decltype(q_)::value;
      c[k][q] = m < H ? IO::ld(p, m + q * H) : make_float2(0.f, 0.f);
    });
  });
  SFor<0, IT>::run([&](auto k_) {
    constexpr int k = decltype(k_)::value;
    const int m = threadIdx.x + k * NT;
    if (m < H) {
      float2 w[J2], o[J];
      tw_powers<0>(g, m, w);
      SFor<0, J>::run([&](auto q_) {
        constexpr int q = decltype(q_)::value;
        o[q] = twmul<q, J2, kColDir<-1, N, BF>>(c[k][q]);
      });
      reg_dft<J, kColDir<-1, N, BF>, float2>(c[k]);
      reg_dft<J, kColDir<-1, N, BF>, float2>(o);
      SFor<0, J>::run([&](auto i_) {
        constexpr int i = decltype(i_)::value;
        sm[2 * i * F::SMEM + m] = i ? cmul(c[k][i], w[2 * i]) : c[k][i];
        sm[(2 * i + 1) * F::SMEM + m] = cmul(o[i], w[2 * i + 1]);
      });
    }
  });
  __syncthreads();
  const int j = threadIdx.x / T, t = threadIdx.x % T;
  float2* xs = sm + j * F::SMEM;
  float2 v[P];
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    v[i] = xs[t + T * i];
  });
  F::template run<kColDir<-1, N, BF>>(v, xs, g.twN, t);
  // v[i] = X[2J k + j], k = t + 16 i
  const float* cc = g.chat + (size_t)vcol * 2 * N + j * H;
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    const float f = __ldg(&cc[t + T * i]);
    v[i] = make_float2(v[i].x * f, v[i].y * f);
  });
  F::template run<kColDir<1, N, BF>>(v, xs, g.twN, t);
  __syncwarp();  // the transform's last exchange reads are done
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    xs[t + T * i] = v[i];
  });
  __syncthreads();
  for (int m = threadIdx.x; m < H; m += NT) {
    float2 w[J2], e[J], o[J];
    tw_powers<0>(g, m, w);
    SFor<0, J>::run([&](auto i_) {
      constexpr int i = decltype(i_)::value;
      e[i] = sm[2 * i * F::SMEM + m];
      if constexpr (i > 0) e[i] = cmulc(e[i], w[2 * i]);
      o[i] = cmulc(sm[(2 * i + 1) * F::SMEM + m], w[2 * i + 1]);
    });
    reg_dft<J, kColDir<1, N, BF>, float2>(e);
    reg_dft<J, kColDir<1, N, BF>, float2>(o);
    SFor<0, J>::run([&](auto q_) {
      constexpr int q = decltype(q_)::value;
      IO::st(p, m + q * H, cadd(e[q], twmul<q, J2, kColDir<1, N, BF>>(o[q])));
    });
  }
}

template <int N, bool BF>
__global__ void __launch_bounds__(GeoH3<N>::THREADS) k_pass3a_h(const __grid_constant__ GroupSet gs, const IterState* st, float* apply_out) {
  using Q = GeoH3<N>;
  using F = typename Q::F;
  constexpr int J = Q::J, H = Q::H, RB = Q::RB, LDZ = Q::LDZ, T = F::T, P = F::P;
  extern __shared__ float2 sm[];
  int bid_;
  const int gi_ = gs.pick(bid_);
  const GroupDev& g = gs.g[gi_];
  float* kz = apply_out ? apply_out + g.img_off : g.kz;
  if (st && skip_iter<BF>(st)) return;
  const int s = bid_ / Q::NB, rb = bid_ % Q::NB;
  const int r0 = rb * RB;
  {
    // the length-2N real inverse as a length-N complex inverse of Z[v] = E[v] + i O[v], two mirrored
    // values at a time: with e, o of v, Z[N - v] = conj(e) + i conj(o)
    using IO = SpecIO<BF>;
    const typename IO::T* sp = reinterpret_cast<const typename IO::T*>(g.spec) + (size_t)s * (N + 1) * N + r0;
    constexpr int B = 4, COUNT = (N / 2 + 1) * RB;
    for (int e0 = threadIdx.x; e0 < COUNT; e0 += B * Q::THREADS) {
      float2 zv[B], zr[B], w[B];
#pragma unroll
      for (int b = 0; b < B; ++b) {
        const int e = e0 + b * Q::THREADS, vv = e / RB, rr = e - vv * RB;
        if (e < COUNT) {
          zv[b] = IO::ld(sp, (size_t)vv * N + rr);
          zr[b] = IO::ld(sp, (size_t)(N - vv) * N + rr);
          w[b] = __ldg(&g.twM[vv]);
        }
      }
#pragma unroll
      for (int b = 0; b < B; ++b) {
        const int e = e0 + b * Q::THREADS, vv = e / RB, rr = e - vv * RB;
        if (e < COUNT) {
          const float2 ev = make_float2(zv[b].x + zr[b].x, zv[b].y - zr[b].y);
          const float2 d = make_float2(zv[b].x - zr[b].x, zv[b].y + zr[b].y);
          const float2 o = cmulc(d, w[b]);
          sm[rr * LDZ + Q::place(vv)] = make_float2(ev.x - o.y, ev.y + o.x);
          sm[rr * LDZ + Q::place(N - vv)] = make_float2(ev.x + o.y, o.x - ev.y);  // (Z[N] is not used)
        }
      }
    }
  }
  __syncthreads();
  const int unit = threadIdx.x / T, t = threadIdx.x % T, rl = unit / J, j = unit - rl * J;
  const float2* zrow = sm + rl * LDZ;
  float2 v[P];
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    v[i] = zrow[Q::place(t + T * i, j)];
  });
  __syncthreads();  // the staged rows are read: the exchange buffers alias them
  float2* xs = sm + unit * F::SMEM;
  F::template run<kRowDir<1, BF>>(v, xs, g.twN, t);
  __syncwarp();
  SFor<0, P>::run([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    xs[t + T * i] = v[i];
  });
  __syncthreads();
  // the kept N/2 packed outputs
#pragma unroll 2
  for (int e = threadIdx.x; e < RB * H; e += Q::THREADS) {
    const int rr = e / H, m = e % H;
    float2 c[J], w[J];
    tw_powers<1>(g, m, w);
    const float2* b = sm + rr * J * F::SMEM + m;
    SFor<0, J>::run([&](auto j_) {
      constexpr int jj = decltype(j_)::value;
      c[jj] = b[jj * F::SMEM];
      if constexpr (jj > 0) c[jj] = cmulc(c[jj], w[jj]);
    });
    reg_dft<J, 1, float2>(c);
    float2* out = reinterpret_cast<float2*>(kz + ((size_t)s * N + r0 + rr) * N);
    SFor<0, J>::run([&](auto q_) {
      constexpr int q = decltype(q_)::value;
      if constexpr (q * H < N / 2)
        if ((q + 1) * H <= N / 2 || m < N / 2 - q * H) out[m + q * H] = c[q];
    });
  }
}

// ---------------------------------------------------------------- pass 3b: gradient and update
// The prior gradient of Eq. 5 at voxel v is sum_o w_o rho'(y_v - y_{v+o}) over the 26
// neighbours; rho' is odd, so the pair (v, v+o) adds +f to v and -f to v+o.  Every unordered
// pair is evaluated once, from its lexicographically smaller end (13 forward offsets), and
// the value is handed to the other end instead of being recomputed there.
//
// A block owns two bands of R rows by BC columns of one group, one below the other, and marches
// through a chunk of its slices.  A lane owns one column; the two lanes of its packed FP32 pairs
// are the rows r0 + t and r0 + R + t, so every neighbour offset is the same for both halves: the
// ring in shared memory interleaves the two bands (float2 per column) and a neighbour pair is one
// aligned 8-byte load at any column offset, without shifted copies and without exchanges between
// the halves.  (With two neighbouring columns in a pair, as this kernel was first built, the
// offsets dx = +-1 need a copy shifted by one column and scalar hand-overs between the halves.)
//
// Rows are walked by the target row u: the pairs that end in row u of slice zs (from rows u - 1 and
// u) and in row u of slice zs + 1 (from rows u - 1, u, u + 1).  A target row's contributions are
// then complete after one step, its loads are used at once, and what stays in registers between
// steps is three centre values and two gradient rows: 6 shared loads per voxel pair and row
// instead of 14.  The walk is a loop, not unrolled: the unrolled bodies of the four boundary
// variants are 130 KB of instructions and measured slower (1.50 against 1.29 ms at 32 x 2048^2).
// The shares of the pairs with dx = +-1 go to the neighbouring lanes by shuffle once per row.
// Across a warp's outer columns the pairs within a slice are evaluated once more by the receiving
// warp (three per row, one evaluation for all rows), and those into slice zs + 1 are handed over
// through shared memory.  The halo rows -1 and R are sources or targets only.  Slice zs is the
// source of the pairs into slice zs + 1, whose contributions wait in shared memory (one entry per
// thread and row) for the next step.  A chunk starting at z0 > 0 first evaluates the pairs between
// slices z0 - 1 and z0 (evaluated twice, once per chunk).  x and x_prev of slice z + 2 arrive by
// asynchronous copies while slice z is worked on; K (*) y, R*g and x_k of a row are loaded into
// registers one row ahead of their use.  A neighbour outside the volume is masked to d = 0.
//
// What bounds it: the special-function unit, then FP32 issue.  Per packed pair the unit spends 16
// cycles of an SM quarter on two log2, 8 on two exp2 and 8 on one reciprocal (measured rates: 16
// log2, 32 exp2 and 16 reciprocals per clock and SM), the FMA pipe about 25.  The two halves share
// one reciprocal (r_x = e_y / (e_x e_y)); with one each the kernel ran at the unit's rate (40 cycles a
// pair).  Measured at 32 x 2048^2: 1.64 ms with neighbouring columns in a pair, 1.36 with the two
// bands, 1.30 with the shared reciprocal and eight-row bands; at 64 x 1024^2 0.87, 0.77 and 0.70 ms.
// At 8 x 2048^2 62 % of the issue slots, the FMA pipe 47 % and the unit 58 % (32 cycles per packed pair).
template <int N>
struct GeoP {
  static_assert(N % 64 == 0, "a warp owns 32 columns, a block at least two warps");
  static constexpr int R = pass3_band(N);                 // rows of a band
  static constexpr int ROWS = 2 * R;                      // rows of a block
  static constexpr int WPB = pass3_warps(N);              // warps per block
  static constexpr int THREADS = 32 * WPB;
  static constexpr int BC = 32 * WPB;                     // columns of a block
  static constexpr int CB = N / BC;                       // column blocks per band pair
  static constexpr int NB = N / ROWS;                     // band pairs per slice
  static constexpr int LDR = BC + 8;                      // row stride of ring and staging: columns c0 - 4 .. c0 + BC + 3
  static constexpr int RING = (R + 2) * LDR;              // float2 entries of one slice
  static constexpr int STG = (ROWS + 2) * LDR;            // floats of one staged array
  static constexpr int EDGE = 4 * R;                      // a warp's outer sums: left, right, outside the block, zeros
  static constexpr int XCH = 2 * (WPB + 2) * R;           // shares handed from warp to warp (one parity)
  // ring (2 slices) | carry | warps' outer sums | warp-to-warp shares (2 parities) | staged x, x_prev
  static constexpr size_t SM = (size_t)(2 * RING + R * THREADS + WPB * EDGE + 2 * XCH) * 8 + (size_t)2 * STG * 4;
  static_assert(3 * R <= 32 && WPB >= 2, "outer pairs of a warp in one evaluation per target slice");
  static_assert(N % BC == 0 && N % ROWS == 0, "blocks");
};

// y = x + beta (x - x_prev) of one slice into a ring slot: ring row i, column q of the float4
// grid, holds rows r0 - 1 + i (first halves) and r0 - 1 + i + R (second halves) at columns
// c0 - 4 + 4 q .. + 3.  ld(row index 0 .. 2R + 1, q, which) gives the float4 of x (0) or x_prev (1).
// A thread keeps its column and takes every fourth row; the two halo columns of all rows go to the
// first threads.  Returns the largest |y| of the thread's values, NaN if one of them is.
template <int N, class Ld>
__device__ __forceinline__ float fill_ring(float2* slot, float beta, Ld&& ld) {
  using GP = GeoP<N>;
  constexpr int QB = GP::BC / 4;
  float top = 0.f;
  auto see = [&](float2 y) { top = max_nan(top, fabsf(y.x), fabsf(y.y)); };
  const float2 b2 = f2(beta);
  auto yv = [&](float2 x, float2 p) { return f2fma(b2, make_float2(x.x - p.x, x.y - p.y), x); };
  auto put = [&](int i, int q) {
    const float4 xa = ld(i, q, 0), pa = ld(i, q, 1), xb = ld(i + GP::R, q, 0), pb = ld(i + GP::R, q, 1);
    const float2 y0 = yv(make_float2(xa.x, xb.x), make_float2(pa.x, pb.x));
    const float2 y1 = yv(make_float2(xa.y, xb.y), make_float2(pa.y, pb.y));
    const float2 y2 = yv(make_float2(xa.z, xb.z), make_float2(pa.z, pb.z));
    const float2 y3 = yv(make_float2(xa.w, xb.w), make_float2(pa.w, pb.w));
    float4* d = reinterpret_cast<float4*>(slot + i * GP::LDR + 4 * q);
    d[0] = make_float4(y0.x, y0.y, y1.x, y1.y);
    d[1] = make_float4(y2.x, y2.y, y3.x, y3.y);
    see(y0);
    see(y1);
    see(y2);
    see(y3);
  };
  const int q = threadIdx.x % QB + 1, i0 = threadIdx.x / QB;
#pragma unroll
  for (int h = 0; h < (GP::R + 2 + 3) / 4; ++h)
    if (i0 + 4 * h < GP::R + 2) put(i0 + 4 * h, q);
  // (from the other end of the block, whose threads have fewer rows)
  const int e = GP::THREADS - 1 - threadIdx.x;
  if (e < 2 * (GP::R + 2)) put(e >> 1, (e & 1) * (QB + 1));
  return top;
}
// from global memory (zero outside the image)
template <int N>
__device__ __forceinline__ float load_ring_p(float2* slot, const float* x, const float* xp, float beta,
                                             size_t off_slice, int r0, int c0) {
  return fill_ring<N>(slot, beta, [&](int i, int q, int which) {
    const int rr = r0 - 1 + i, cc = c0 - 4 + 4 * q;
    if (rr < 0 || rr >= N || cc < 0 || cc >= N) return make_float4(0.f, 0.f, 0.f, 0.f);
    return __ldg(reinterpret_cast<const float4*>((which ? xp : x) + off_slice + (size_t)rr * N + cc));
  });
}
// x and x_prev of one slice (rows r0 - 1 .. r0 + 2R, the ring's columns) into the staging area by
// asynchronous 16-byte copies, zero-filled outside the image.  A thread copies one array and one
// column, every second row, from one pointer at fixed offsets; the halo columns go to the first
// threads.
template <int N>
struct Stager {
  using GP = GeoP<N>;
  static constexpr int QB = GP::BC / 4, ITEMS = (GP::ROWS + 2) / 2;
  static_assert(4 * (GP::ROWS + 2) <= GP::THREADS, "halo items");
  const float* src;    // first item in slice 0
  const float* hsrc;   // halo item in slice 0
  float *dst, *hdst;
  bool first, last, halo, hok;
  __device__ __forceinline__ Stager(float* stg, const float* x, const float* xp, int r0, int c0) {
    const int q = threadIdx.x % QB, arr = (threadIdx.x / QB) & 1, row = threadIdx.x / (2 * QB);
    src = (arr ? xp : x) + (ptrdiff_t)(r0 - 1 + row) * N + c0 + 4 * q;
    dst = stg + arr * GP::STG + row * GP::LDR + 4 * (q + 1);
    first = row > 0 || r0 > 0;
    last = row == 0 || r0 + GP::ROWS < N;
    const int hr = threadIdx.x >> 2, ha = (threadIdx.x >> 1) & 1, side = threadIdx.x & 1;
    halo = threadIdx.x < 4 * (GP::ROWS + 2);
    hok = r0 - 1 + hr >= 0 && r0 - 1 + hr < N && (side ? c0 + GP::BC < N : c0 > 0);
    hsrc = (ha ? xp : x) + (ptrdiff_t)(r0 - 1 + hr) * N + (side ? c0 + GP::BC : c0 - 4);
    hdst = stg + ha * GP::STG + hr * GP::LDR + side * (GP::BC + 4);
  }
  __device__ __forceinline__ void issue(size_t off_slice) const {
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      const bool ok = i == 0 ? first : (i == ITEMS - 1 ? last : true);
      tc05::cp_async16(dst + 2 * i * GP::LDR, ok ? src + off_slice + 2 * i * N : src + off_slice + 2 * N, ok);
    }
    if (halo) tc05::cp_async16(hdst, hok ? hsrc + off_slice : src + off_slice + 2 * N, hok);
  }
};
template <int N>
__device__ __forceinline__ float stage_to_ring(float2* slot, const float* stg, float beta) {
  using GP = GeoP<N>;
  return fill_ring<N>(slot, beta, [&](int i, int q, int which) {
    return reinterpret_cast<const float4*>(stg + which * GP::STG + i * GP::LDR)[q];
  });
}

// Keeps a loop constant in its registers: the compiler otherwise rebuilds the two halves of every
// packed constant with moves at each use (six of the 22 instructions of a pair).
__device__ __forceinline__ float2 pin(float2 v) {
  asm volatile("" : "+f"(v.x), "+f"(v.y));
  return v;
}
// Constants of the packed pair term.
struct PairK {
  float2 half_qp, qp_l2, p, qmp, one;
  float2 half_q2, q2_l2;  // q != 2 only
};
template <bool Q2>
__device__ __forceinline__ PairK pair_k(const PriorC& c) {
  PairK k;
  // q = p: any positive exponent this small gives 1 for every difference but 0, whose term vanishes
  k.half_qp = pin(f2(fmaxf(0.5f * c.qp, 1.5e-38f)));
  k.qp_l2 = pin(f2(c.qp_l2_inv_csig));
  k.p = pin(f2(c.p));
  k.qmp = pin(f2(c.qp));
  k.one = pin(f2(1.f));
  if constexpr (!Q2) {
    k.half_q2 = f2(0.5f * (c.q - 2.0f));
    k.q2_l2 = f2((c.q - 2.0f) * c.l2_inv_sig);
  }
  return k;
}
// Unweighted pair value v = sigma^2 rho'(nb - y) of two pairs at once from n = -y, with the identity
//   sigma^2 rho'(d) = d |d/sigma|^(q-2) r (p + (q - p) r), r = 1 / (1 + |d/(c sigma)|^(q-p)).
// With PH, ph += sigma^2 rho(d) = d^2 |d/sigma|^(q-2) r (unweighted).  MX, MY: the first / second
// half counts only when okx / oky.  For q = 2 the two halves share one reciprocal, which needs the
// product of the two e to be finite; WIDE gives each its own, for slices with values past
// PriorC::pair_lim (or not finite, which would spread from one half to the other).  The values are
// looked at when they enter the ring: limiting the exponents here instead took two minima a pair (0.704
// against 0.698 ms at 64 x 1024^2, 1.307 against 1.303 at 32 x 2048^2; a launch at 1 x 128^2 is 0.2 us
// faster with them) and gave wrong gradients past the limit.  log2 0 = -inf
// gives r = 1, and d = 0 ends both terms; WIDE takes 2 log2 |d|, whose range d^2 does not have.  For
// q != 2 the logarithm is kept finite, since the second exponential would meet it with a negative factor.
template <bool Q2, bool PH, bool MX, bool MY, bool WIDE>
__device__ __forceinline__ float2 pairv(float2 n, float2 nb, const PairK& k, bool okx, bool oky, float2& ph) {
  float2 d = f2add(nb, n);
  if constexpr (MX) d.x = okx ? d.x : 0.f;
  if constexpr (MY) d.y = oky ? d.y : 0.f;
  float2 la;
  if constexpr (Q2 && WIDE) {
    la = f2mul(make_float2(lg2a(fabsf(d.x)), lg2a(fabsf(d.y))), f2(2.f));
  } else {
    const float2 sq = Q2 ? f2mul(d, d) : f2fma(d, d, f2(1e-30f));
    la = make_float2(lg2a(sq.x), lg2a(sq.y));
  }
  const float2 s = f2fma(k.half_qp, la, k.qp_l2);
  const float2 e = f2add(make_float2(ex2a(s.x), ex2a(s.y)), k.one);
  float2 r;
  if constexpr (Q2 && !WIDE) {
    const float ri = rcpa(e.x * e.y);
    r = make_float2(ri * e.y, ri * e.x);
  } else {
    r = make_float2(rcpa(e.x), rcpa(e.y));
  }
  float2 dr = f2mul(d, r);
  if constexpr (!Q2) {
    const float2 s2 = f2fma(k.half_q2, la, k.q2_l2);
    dr = f2mul(dr, make_float2(ex2a(s2.x), ex2a(s2.y)));
  }
  if constexpr (PH) ph = f2fma(d, dr, ph);
  return f2mul(dr, f2fma(k.qmp, r, k.p));
}

// hi + lo += v with the rounding error of the addition kept in lo (Knuth's TwoSum): the
// per-slice partial sums stay in FP32, whose pipe is wide, instead of FP64, whose is not
__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float v) {
  const float s = hi + v;
  const float bp = s - hi;
  lo += (hi - (s - bp)) + (v - bp);
  hi = s;
}

// Block reduction of compensated FP32 sums (hi + lo per thread) to partials[block]: TwoSum
// across each warp, FP64 across the warps, in a fixed order.
template <int W>
__device__ __forceinline__ void block_partials_f(float (&hi)[kParts], float (&lo)[kParts], double* red,
                                                 double* out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < kParts; ++j) {
    float h = hi[j], l = lo[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float h2 = __shfl_down_sync(0xffffffffu, h, o), l2 = __shfl_down_sync(0xffffffffu, l, o);
      l += l2;
      two_sum_add(h, l, h2);
    }
    if (lane == 0) red[warp * kParts + j] = (double)h + (double)l;
  }
  __syncthreads();
  if (threadIdx.x < kParts) {
    double sum = 0.0;
    for (int w = 0; w < W; ++w) sum += red[w * kParts + threadIdx.x];
    out[threadIdx.x] = sum;
  }
}

// What the boundary tests know about the block and the lane.
struct BandB {
  bool okT, okB;  // image row r0 - 1 (above the first band) and r0 + 2R (below the second) exist
  bool okL, okR;  // this lane's columns c - 1 and c + 1 exist
};
// The pairs across the warp's outer columns that a lane evaluates, into target row u = lane % R:
//   zs: the warp's first column from the column before it, rows u (lanes 0 .. R - 1) and u - 1
//       (R .. 2R - 1), and its last column from the column after it, row u - 1 (2R .. 3R - 1);
//   zs + 1, the block's first and last warp only, whose neighbours belong to other blocks: that
//       side's column from rows u - 1, u, u + 1 of zs.
// The other pairs into slice zs + 1 across a warp's columns are handed over by the neighbouring
// warp, which has a barrier's time for it.
struct OuterItem {
  int src, tgt;  // ring places of the source and the target
  float w;       // class weight
  bool on, okx, oky;
};
template <int N>
__device__ __forceinline__ OuterItem outer_item(bool cross, const float2 (&w)[3], const BandB& bb, int warp, int c0w) {
  using GP = GeoP<N>;
  constexpr int R = GP::R;
  const int lane = threadIdx.x & 31, kd = lane / R, u = lane - kd * R;
  OuterItem it;
  const bool left = cross ? warp == 0 : kd < 2;
  const int sr = cross ? kd - 1 : (kd == 0 ? 0 : -1);
  it.on = kd < 3 && (!cross || warp == 0 || warp == GP::WPB - 1) && (left ? c0w > 0 : c0w + 32 < N);
  const int tc = 32 * warp + 4 + (left ? 0 : 31);
  it.tgt = it.on ? (u + 1) * GP::LDR + tc : 0;
  it.src = it.on ? (u + sr + 1) * GP::LDR + (left ? tc - 1 : tc + 1) : 0;
  it.w = cross ? (sr != 0 ? w[2].x : w[1].x) : (kd == 0 ? w[0].x : w[1].x);
  it.okx = u + sr >= 0 || bb.okT;
  it.oky = u + sr < R || bb.okB;
  return it;
}
// the weighted value of the lane's outer pair, and its sums over the lanes of the same row
template <int N, bool Q2, bool ROWE, bool WIDE>
__device__ __forceinline__ void outer_sums(const float2* S0, const float2* T, const OuterItem& it, const PairK& k,
                                           float2& v, float2& v2, float2& v3) {
  constexpr int R = GeoP<N>::R;
  float2 unused = f2(0.f);
  const float2 sv = S0[it.src];
  v = pairv<Q2, false, true, true, WIDE>(make_float2(-sv.x, -sv.y), T[it.tgt], k, it.on && (!ROWE || it.okx),
                                         it.on && (!ROWE || it.oky), unused);
  v = f2mul(f2(it.w), v);
  float2 a, b;
  a.x = __shfl_down_sync(0xffffffffu, v.x, R);
  a.y = __shfl_down_sync(0xffffffffu, v.y, R);
  b.x = __shfl_down_sync(0xffffffffu, v.x, 2 * R);
  b.y = __shfl_down_sync(0xffffffffu, v.y, 2 * R);
  v2 = f2add(v, a);
  v3 = f2add(v, f2add(a, b));
}

// One slice step of a block's two bands: every pair with an end in the owned rows whose source
// voxel lies in slice zs (ring slot S0) and whose other end lies in zs or zs + 1 (slot S1, when
// have1).  The carried contributions of slice zs (cr, this thread's entries, one per row, and the
// neighbouring warps' shares xin) start the sums of the rows and are replaced by those of slice
// zs + 1 (cr and the shares xout for the neighbouring warps).  PRE: only the pairs into slice
// zs + 1 (a chunk start); otherwise pre(u) is called a row ahead and fin(u, h, -y) once row u is
// complete, with h = -(the prior gradient) and ph the unweighted sigma^2 rho sums by class of the
// pairs whose target row the band owns.  w: class weights w / sigma^2 (face, edge, corner).  ROWE:
// the block holds the image's first or last rows; COLE: the warp holds its first or last columns.
// Elsewhere every neighbour lies inside the image and the boundary tests drop out.  WIDE: see pairv.
template <int N, bool Q2, bool PHI, bool PRE, bool ROWE, bool COLE, bool WIDE, class Pre, class Fin>
__device__ __forceinline__ void band_step(const float2* S0, const float2* S1, bool have1, const BandB& bb,
                                          const OuterItem& it, const OuterItem& itx, int ic, float2* cr, float2* edge,
                                          const float2* xin, float2* xout, const PairK& k, const float2 (&w)[3],
                                          float2 (&ph)[3], Pre&& pre, Fin&& fin) {
  using GP = GeoP<N>;
  constexpr int R = GP::R, LDR = GP::LDR, CRS = GP::THREADS;
  constexpr bool PH = PHI && !PRE;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float2 zero = f2(0.f);
  auto neg = [](float2 v) { return make_float2(-v.x, -v.y); };
  auto sub = [](float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); };

  // ---- the pairs across the warp's outer columns (OuterItem), summed per target row
  {
    float2 v, v2, v3;
    if constexpr (!PRE) {
      outer_sums<N, Q2, ROWE, WIDE>(S0, S0, it, k, v, v2, v3);
      if (lane < R) edge[lane] = v2;
      if (lane >= 2 * R && lane < 3 * R) edge[lane - R] = v;
    }
    if (have1 && (warp == 0 || warp == GP::WPB - 1)) {
      outer_sums<N, Q2, ROWE, WIDE>(S0, S1, itx, k, v, v2, v3);
      if (lane < R) edge[2 * R + lane] = v3;
    }
  }
  __syncwarp();
  // lane 0 starts its rows from the left sums, lane 31 from the right ones, the others from zero; into
  // slice zs + 1 only the block's outer lanes
  const float2* es = edge + (lane == 0 ? 0 : (lane == 31 ? R : 3 * R));
  const float2* ex =
      edge + ((lane == 0 && warp == 0) || (lane == 31 && warp == GP::WPB - 1) ? 2 * R : 3 * R);
  // the share of lane 31's pairs belongs to the next warp's first column, lane 0's to the last of the one before
  float2* xo = xout + (lane == 31 ? (warp + 2) * R : (GP::WPB + 2) * R + warp * R);
  const float2* xi = xin + (lane == 31 ? (GP::WPB + 2) * R : 0) + (lane == 0 || lane == 31 ? (warp + 1) * R : 0);

  // the neighbouring lanes' shares (dx = +-1) added to a target row's sum
  const bool inL = lane > 0, inR = lane < 31;
  auto receive = [&](float2 c, float2 sR, float2 sL) {
    float2 a, b;
    a.x = __shfl_up_sync(0xffffffffu, sR.x, 1);
    a.y = __shfl_up_sync(0xffffffffu, sR.y, 1);
    b.x = __shfl_down_sync(0xffffffffu, sL.x, 1);
    b.y = __shfl_down_sync(0xffffffffu, sL.y, 1);
    a = make_float2(inL ? a.x : 0.f, inL ? a.y : 0.f);
    b = make_float2(inR ? b.x : 0.f, inR ? b.y : 0.f);
    return f2add(c, f2add(a, b));
  };
  // carried sums of a row: the thread's own and, at the warp's ends, the neighbouring warp's
  auto carried = [&](int u) { return sub(neg(cr[u * CRS]), xi[u]); };
  // a pair at column offset DX; mx, my: the first / second half's row exists (ROWE only)
  auto pair = [&](auto DX_, auto PH_, float2 n, float2 nb, bool mx, bool my, float2& p) {
    constexpr int DX = decltype(DX_)::value;
    constexpr bool C = COLE && DX != 0;
    const bool okc = DX < 0 ? bb.okL : bb.okR;
    return pairv<Q2, decltype(PH_)::value, ROWE || C, ROWE || C, WIDE>(n, nb, k, (!ROWE || mx) && (!C || okc),
                                                                       (!ROWE || my) && (!C || okc), p);
  };
  using Lf = std::integral_constant<int, -1>;
  using Ce = std::integral_constant<int, 0>;
  using Ri = std::integral_constant<int, 1>;
  using No = std::false_type;
  using Ph = std::integral_constant<bool, PH>;
  float2 unused = zero;

  // ---- the row walk
  const float2* p0 = S0 + ic;       // row u - 1 of slice zs while row u is the target
  const float2* p1 = S1 + LDR + ic; // row u of slice zs + 1
  float2 nm = neg(p0[0]), n0 = neg(p0[LDR]);  // -y of rows u - 1, u
  float2 hm = zero, h0 = PRE ? zero : carried(0);  // their sums
  if (!PRE && have1) {  // u = -1: source row 0
    h0 = f2fma(w[2], pair(Lf{}, No{}, n0, p1[-LDR - 1], bb.okT, true, unused), h0);
    h0 = f2fma(w[1], pair(Ce{}, No{}, n0, p1[-LDR], bb.okT, true, unused), h0);
    h0 = f2fma(w[2], pair(Ri{}, No{}, n0, p1[-LDR + 1], bb.okT, true, unused), h0);
  }
#pragma unroll 1
  for (int u = 0; u < R; ++u) {
    const bool mT = u > 0 || bb.okT, mB = u + 1 < R || bb.okB;  // rows u - 1 / u + 1 exist in both halves
    const float2 np = neg(p0[2 * LDR]);
    float2 hp = PRE || u + 1 >= R ? zero : carried(u + 1);
    if constexpr (!PRE) {
      pre(u);
      const float2 L = p0[LDR - 1], C = p0[LDR], Rr = p0[LDR + 1];
      float2 c = es[u], sR, sL;
      // from row u - 1: (0, +1, -1 / 0 / +1)
      float2 v = pair(Lf{}, Ph{}, nm, L, mT, true, ph[1]);
      hm = f2fma(w[1], v, hm);
      sL = f2mul(w[1], v);
      v = pair(Ce{}, Ph{}, nm, C, mT, true, ph[0]);
      hm = f2fma(w[0], v, hm);
      c = f2fma(w[0], v, c);
      v = pair(Ri{}, Ph{}, nm, Rr, mT, true, ph[1]);
      hm = f2fma(w[1], v, hm);
      sR = f2mul(w[1], v);
      // (0, 0, +1), then the row's total
      v = pair(Ri{}, Ph{}, n0, Rr, true, true, ph[0]);
      h0 = f2fma(w[0], v, h0);
      sR = f2fma(w[0], v, sR);
      h0 = sub(h0, receive(c, sR, sL));
    }
    if (have1) {
      const float2 L = p1[-1], C = p1[0], Rr = p1[1];
      float2 c = ex[u], sR = zero, sL = zero;
      // the three pairs from one source row
      auto three = [&](auto CS_, float2 n, float2& h, bool mx, bool my) {
        constexpr int CS = decltype(CS_)::value, C0 = CS - 1;
        float2 v = pair(Lf{}, Ph{}, n, L, mx, my, ph[CS]);
        h = f2fma(w[CS], v, h);
        sL = f2fma(w[CS], v, sL);
        v = pair(Ce{}, Ph{}, n, C, mx, my, ph[C0]);
        h = f2fma(w[C0], v, h);
        c = f2fma(w[C0], v, c);
        v = pair(Ri{}, Ph{}, n, Rr, mx, my, ph[CS]);
        h = f2fma(w[CS], v, h);
        sR = f2fma(w[CS], v, sR);
      };
      using Diag = std::integral_constant<int, 2>;
      three(Diag{}, nm, hm, mT, true);
      three(std::integral_constant<int, 1>{}, n0, h0, true, true);
      three(Diag{}, np, hp, true, mB);
      cr[u * CRS] = receive(c, sR, sL);
      if (!inL) xo[u] = sL;
      if (!inR) xo[u] = sR;
    }
    if constexpr (!PRE)
      if (u >= 1) fin(u - 1, hm, nm);
    // slide the windows down one row
    nm = n0;
    n0 = np;
    hm = h0;
    h0 = hp;
    p0 += LDR;
    p1 += LDR;
  }
  if constexpr (!PRE) {  // u = R: source row R - 1
    hm = f2fma(w[1], pair(Lf{}, No{}, nm, p0[LDR - 1], true, bb.okB, unused), hm);
    hm = f2fma(w[0], pair(Ce{}, No{}, nm, p0[LDR], true, bb.okB, unused), hm);
    hm = f2fma(w[1], pair(Ri{}, No{}, nm, p0[LDR + 1], true, bb.okB, unused), hm);
    if (have1) {
      hm = f2fma(w[2], pair(Lf{}, No{}, nm, p1[-1], true, bb.okB, unused), hm);
      hm = f2fma(w[1], pair(Ce{}, No{}, nm, p1[0], true, bb.okB, unused), hm);
      hm = f2fma(w[2], pair(Ri{}, No{}, nm, p1[1], true, bb.okB, unused), hm);
    }
    fin(R - 1, hm, nm);
  }
}

// kz: K (*) y of the group from pass 3a ([slice][row][col]); phase: in Iterate mode, the storage
// phase this launch belongs to (0 FP32, 1 BF16), checked like the other passes.
template <int N, int MODE, bool Q2, bool MULTI>
__global__ void __launch_bounds__(GeoP<N>::THREADS, 512 / GeoP<N>::THREADS)
    k_pass3(const __grid_constant__ GroupSet gs, StepArgs a, PriorC pc, const float* apply_out, int phase,
            double* partials, int block_offset) {
  using GP = GeoP<N>;
  constexpr int R = GP::R;
  constexpr bool PRIOR = MODE != (int)Pass3Mode::Apply;
  constexpr bool PHI = MODE == (int)Pass3Mode::Step || MODE == (int)Pass3Mode::Iterate ||
                       MODE == (int)Pass3Mode::Objective;
  constexpr bool UPDATE = MODE == (int)Pass3Mode::Step || MODE == (int)Pass3Mode::Iterate;
  extern __shared__ float2 sm[];
  __shared__ double red[GP::WPB * kParts];
  __shared__ std::conditional_t<GP::WPB == 2, uint16_t, uint32_t> past_lim[2];  // a byte per warp and ring slot
  static_assert(GP::WPB == 2 || GP::WPB == 4, "a byte per warp");
  int bid_;
  const int gi_ = gs.template pick<MULTI>(bid_);
  const GroupDev& g = gs.g[MULTI ? gi_ : 0];
  const float* __restrict__ kz = apply_out ? apply_out + g.img_off : g.kz;
  const int zc = g.zc;  // resolved by the launcher
  const float *x, *xp;
  float* out;
  float beta, invL;
  if constexpr (MODE == (int)Pass3Mode::Iterate) {
    if (a.st->done || a.st->bf16 != phase) return;
    const int cur = a.st->cur;
    x = cur == 0 ? a.xb[0] : (cur == 1 ? a.xb[1] : a.xb[2]);
    xp = cur == 0 ? a.xb[2] : (cur == 1 ? a.xb[0] : a.xb[1]);
    out = cur == 0 ? a.xb[1] : (cur == 1 ? a.xb[2] : a.xb[0]);
    beta = (float)(a.gm + gi_)->beta;
    invL = (float)(a.gm + gi_)->invL;
  } else {
    x = a.x;
    xp = a.xprev;
    out = a.out;
    beta = a.beta;
    invL = a.invL;
  }
  // the group's slices as the origin of every image pointer
  const size_t go = g.img_off;
  const int S = g.S;
  x += go;
  xp += go;
  out += go;
  const float* __restrict__ atg = a.atg + go;
  const int band = bid_ % GP::NB;
  const int cb = (bid_ / GP::NB) % GP::CB;
  const int chunk = bid_ / (GP::NB * GP::CB);
  const int z0 = g.zlo + chunk * zc, z1 = min(g.zlo + (g.zn > 0 ? g.zn : S), z0 + zc);
  const int r0 = band * GP::ROWS, c0 = cb * GP::BC;
  const int warp = threadIdx.x >> 5;
  const int col = c0 + threadIdx.x;  // this lane's column
  const int ic = threadIdx.x + 4;    // and its place in a ring row
  const size_t N2 = (size_t)N * N;

  float hi[kParts], lo[kParts];  // compensated FP32 sums of the block's slices
#pragma unroll
  for (int j = 0; j < kParts; ++j) hi[j] = lo[j] = 0.f;

  if constexpr (!PRIOR) {
    // Apply: pass 3a wrote K (*) x to the output itself; only the partial sums remain
    for (int z = z0; z < z1; ++z) {
      float acc0 = 0.f, acc5 = 0.f;
#pragma unroll
      for (int t = 0; t < GP::ROWS; ++t) {
        const size_t o = (size_t)z * N2 + (size_t)(r0 + t) * N + col;
        const float zd = __ldg(kz + o), xv = __ldg(x + o);
        acc0 = fmaf(xv, zd, acc0);
        acc5 = fmaf(zd, zd, acc5);
      }
      two_sum_add(hi[0], lo[0], acc0);
      two_sum_add(hi[5], lo[5], acc5);
    }
  } else {
    const PairK pk = pair_k<Q2>(pc);
    const float2 w[3] = {pin(f2(pc.wf * pc.inv_sig2)), pin(f2(pc.we * pc.inv_sig2)), pin(f2(pc.wc * pc.inv_sig2))};
    const float2 mlam = f2(-pc.lam);
    BandB bb;
    bb.okT = r0 > 0;
    bb.okB = r0 + GP::ROWS < N;
    const int c0w = c0 + 32 * warp;
    bb.okL = col > 0;
    bb.okR = col + 1 < N;
    const OuterItem it = outer_item<N>(false, w, bb, warp, c0w), itx = outer_item<N>(true, w, bb, warp, c0w);
    float2* ring = sm;
    float2* cr = ring + 2 * GP::RING + threadIdx.x;
    float2* edge = ring + 2 * GP::RING + R * GP::THREADS + warp * GP::EDGE;
    float2* xch = ring + 2 * GP::RING + R * GP::THREADS + GP::WPB * GP::EDGE;
    float* stg = reinterpret_cast<float*>(xch + 2 * GP::XCH);
    if ((threadIdx.x & 31) < R) edge[3 * R + (threadIdx.x & 31)] = f2(0.f);
    // shares[parity]: [side][warp + 1][row]; the places beyond the block's warps stay zero
    for (int i = threadIdx.x; i < 2 * GP::XCH; i += GP::THREADS) xch[i] = f2(0.f);
    float2 ph[3] = {f2(0.f), f2(0.f), f2(0.f)};
    // every warp notes whether its part of a ring slot holds values past the limit of the shared
    // reciprocal; the block's answer is the same wherever the slice is held, in any division into chunks
    auto note = [&](int z, float top) {
      if constexpr (Q2) {
        const bool past = __any_sync(0xffffffffu, !(top <= pc.pair_lim));
        if ((threadIdx.x & 31) == 0) reinterpret_cast<bool*>(&past_lim[z & 1])[warp] = past;
      }
    };
    note(z0, load_ring_p<N>(ring + (z0 & 1) * GP::RING, x, xp, beta, (size_t)z0 * N2, r0, c0));
    if (z0 > 0) {
      note(z0 - 1, load_ring_p<N>(ring + ((z0 - 1) & 1) * GP::RING, x, xp, beta, (size_t)(z0 - 1) * N2, r0, c0));
    } else {
#pragma unroll
      for (int t = 0; t < R; ++t) cr[t * GP::THREADS] = f2(0.f);
    }
    const Stager<N> stager(stg, x, xp, r0, c0);
    if (z0 + 1 < S) stager.issue((size_t)(z0 + 1) * N2);
    __syncthreads();
    // boundary tests only where the warp's neighbourhoods leave the image
    const bool rowe = !(bb.okT && bb.okB), cole = !(c0w > 0 && c0w + 32 < N);
    auto none = [](int) {};
    if (z0 > 0) {
      auto fin0 = [](int, float2, float2) {};
      const float2* s0 = ring + ((z0 - 1) & 1) * GP::RING;
      const float2* s1 = ring + (z0 & 1) * GP::RING;
      float2* xo0 = xch + (z0 & 1) * GP::XCH;
      const float2* xi0 = xo0;  // not read
      if (Q2 && (past_lim[0] | past_lim[1]))
        band_step<N, Q2, PHI, true, true, true, true>(s0, s1, true, bb, it, itx, ic, cr, edge, xi0, xo0, pk, w, ph, none, fin0);
      else if (rowe || cole)
        band_step<N, Q2, PHI, true, true, true, false>(s0, s1, true, bb, it, itx, ic, cr, edge, xi0, xo0, pk, w, ph, none, fin0);
      else
        band_step<N, Q2, PHI, true, false, false, false>(s0, s1, true, bb, it, itx, ic, cr, edge, xi0, xo0, pk, w, ph, none, fin0);
    }
    for (int z = z0; z < z1; ++z) {
      // every thread has finished slice z - 1, so its ring slot takes slice z + 1 from the
      // staging area; then the staging area takes slice z + 2 while slice z is worked on
      tc05::cp_async_wait_all();
      __syncthreads();
      if (z + 1 < S) {
        note(z + 1, stage_to_ring<N>(ring + ((z + 1) & 1) * GP::RING, stg, beta));
        __syncthreads();
      }
      if (z + 1 < z1 && z + 2 < S) stager.issue((size_t)(z + 2) * N2);
      float2 acc[kParts];
#pragma unroll
      for (int j = 0; j < kParts; ++j) acc[j] = f2(0.f);
      const size_t img = (size_t)z * N2 + (size_t)r0 * N + col;
      const float *kzp = kz + img, *atp = atg + img, *xkp = x + img;
      float* op = out + img;
      // K (*) y, R*g and x_k of row u, loaded while the rows u - 1 and u are worked on
      float2 zd, at, xv, zdn, atn, xvn;
      zd = at = xv = zdn = atn = xvn = f2(0.f);
      auto pre = [&](int u) {
        zd = zdn;
        at = atn;
        zdn = make_float2(__ldg(kzp + u * N), __ldg(kzp + (u + R) * N));
        atn = make_float2(__ldg(atp + u * N), __ldg(atp + (u + R) * N));
        if constexpr (UPDATE) {
          xv = xvn;
          xvn = make_float2(__ldg(xkp + u * N), __ldg(xkp + (u + R) * N));
        }
      };
      auto fin = [&](int u, float2 h, float2 n) {
        if (u == R - 1) {  // the last row was not followed by another
          zd = zdn;
          at = atn;
          xv = xvn;
        }
        const float2 yv = make_float2(-n.x, -n.y);
        const float2 Gv = f2fma(mlam, h, make_float2(zd.x - at.x, zd.y - at.y));
        acc[0] = f2fma(yv, zd, acc[0]);
        acc[1] = f2fma(yv, at, acc[1]);
        acc[4] = f2fma(Gv, Gv, acc[4]);
        if constexpr (MODE == (int)Pass3Mode::Gradient) {
          op[u * N] = Gv.x;
          op[(u + R) * N] = Gv.y;
        } else if constexpr (UPDATE) {
          float2 xn = f2fma(f2(-invL), Gv, yv);
          if (pc.nonneg) xn = make_float2(fmaxf(xn.x, 0.f), fmaxf(xn.y, 0.f));
          op[u * N] = xn.x;
          op[(u + R) * N] = xn.y;
          acc[3] = f2fma(Gv, make_float2(xn.x - xv.x, xn.y - xv.y), acc[3]);
        }
      };
      const float2* s0 = ring + (z & 1) * GP::RING;
      const float2* s1 = ring + ((z + 1) & 1) * GP::RING;
      const float2* xi = xch + (z & 1) * GP::XCH;        // what slice z - 1 handed over
      float2* xo = xch + ((z + 1) & 1) * GP::XCH;
      if (Q2 && (past_lim[z & 1] | (z + 1 < S ? past_lim[(z + 1) & 1] : 0)))
        band_step<N, Q2, PHI, false, true, true, true>(s0, s1, z + 1 < S, bb, it, itx, ic, cr, edge, xi, xo, pk, w, ph, pre, fin);
      else if (rowe || cole)
        band_step<N, Q2, PHI, false, true, true, false>(s0, s1, z + 1 < S, bb, it, itx, ic, cr, edge, xi, xo, pk, w, ph, pre, fin);
      else
        band_step<N, Q2, PHI, false, false, false, false>(s0, s1, z + 1 < S, bb, it, itx, ic, cr, edge, xi, xo, pk, w, ph, pre, fin);
      if constexpr (PHI) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          acc[2] = f2fma(w[j], ph[j], acc[2]);
          ph[j] = f2(0.f);
        }
      }
#pragma unroll
      for (int j = 0; j < 5; ++j) two_sum_add(hi[j], lo[j], acc[j].x + acc[j].y);
    }
  }
  block_partials_f<GP::WPB>(hi, lo, red, partials + (size_t)(block_offset + blockIdx.x) * kParts);
}

// ---------------------------------------------------------------- host launchers
template <int N>
static int set_smem_limits() {
  using Gm = Geo<N>;
  using Gr = Geo3a<N>;
  static bool done = false;
  if (done) return TMBIR_OK;
  if constexpr (is_split_side<N>()) {
    using Q = GeoH<N>;
    TMBIR_CUDA(cudaFuncSetAttribute(k_pass1_h<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Q::SM_ROWS));
    TMBIR_CUDA(cudaFuncSetAttribute(k_pass1_h<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Q::SM_ROWS));
    TMBIR_CUDA(cudaFuncSetAttribute(k_pass2_h<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Q::SM_COL));
    TMBIR_CUDA(cudaFuncSetAttribute(k_pass2_h<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Q::SM_COL));
    TMBIR_CUDA(cudaFuncSetAttribute(k_pass3a_h<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GeoH3<N>::SM_ROWS));
    TMBIR_CUDA(cudaFuncSetAttribute(k_pass3a_h<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GeoH3<N>::SM_ROWS));
  } else {
    TMBIR_CUDA(cudaFuncSetAttribute(k_pass1<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gm::SM1));
    TMBIR_CUDA(cudaFuncSetAttribute(k_pass1<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gm::SM1));
    TMBIR_CUDA(cudaFuncSetAttribute(k_pass2<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gm::SM2));
    TMBIR_CUDA(cudaFuncSetAttribute(k_pass2<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gm::SM2));
    TMBIR_CUDA(cudaFuncSetAttribute(k_pass3a<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gr::SM1));
    TMBIR_CUDA(cudaFuncSetAttribute(k_pass3a<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gr::SM1));
  }
#define TMBIR_P3ATTR(M, Q)                                                                           \
  TMBIR_CUDA(cudaFuncSetAttribute(k_pass3<N, M, Q, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                  (int)GeoP<N>::SM));
  TMBIR_P3ATTR(0, true) TMBIR_P3ATTR(1, true) TMBIR_P3ATTR(2, true) TMBIR_P3ATTR(3, true) TMBIR_P3ATTR(4, true)
  TMBIR_P3ATTR(0, false) TMBIR_P3ATTR(1, false) TMBIR_P3ATTR(2, false) TMBIR_P3ATTR(3, false) TMBIR_P3ATTR(4, false)
#undef TMBIR_P3ATTR
  TMBIR_CUDA(cudaFuncSetAttribute(k_pass3<N, 3, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)GeoP<N>::SM));
  TMBIR_CUDA(cudaFuncSetAttribute(k_pass3<N, 3, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)GeoP<N>::SM));
  done = true;
  return TMBIR_OK;
}

// A group set of n groups, with each group's share of the launch's blocks.
template <class BlocksOf>
static GroupSet make_set(const GroupDev* gs, int n, BlocksOf&& blocks_of) {
  static_assert(sizeof(GroupSet) <= 4000, "group set exceeds the kernel parameter space");
  GroupSet set{};
  set.n = n;
  for (int i = 0; i < n; ++i) {
    set.g[i] = gs[i];
    set.boff[i + 1] = set.boff[i] + blocks_of(gs[i]);
  }
  return set;
}

template <int N>
static int pass1_n(const GroupDev* gs, int n, const StepArgs& a, bool bf16, cudaStream_t s) {
  using Gm = Geo<N>;
  if (int e = set_smem_limits<N>()) return e;
  if constexpr (is_split_side<N>()) {
    using Q = GeoH<N>;
    const GroupSet set = make_set(gs, n, [](const GroupDev& g) { return g.S * Q::NB; });
    if (bf16)
      k_pass1_h<N, true><<<set.boff[n], Q::THREADS, Q::SM_ROWS, s>>>(set, a);
    else
      k_pass1_h<N, false><<<set.boff[n], Q::THREADS, Q::SM_ROWS, s>>>(set, a);
  } else {
    const GroupSet set = make_set(gs, n, [](const GroupDev& g) { return g.S * Gm::NB; });
    if (bf16)
      k_pass1<N, true><<<set.boff[n], Gm::THREADS, Gm::SM1, s>>>(set, a);
    else
      k_pass1<N, false><<<set.boff[n], Gm::THREADS, Gm::SM1, s>>>(set, a);
  }
  TMBIR_CHECK_LAUNCH();
  return TMBIR_OK;
}
template <int N>
static int pass2_n(const GroupDev* gs, int n, const IterState* st, bool bf16, cudaStream_t s) {
  using Gm = Geo<N>;
  if (int e = set_smem_limits<N>()) return e;
  if constexpr (is_split_side<N>()) {
    using Q = GeoH<N>;
    const GroupSet set = make_set(gs, n, [](const GroupDev& g) { return g.S * (N + 1); });
    if (bf16)
      k_pass2_h<N, true><<<set.boff[n], Q::THREADS2, Q::SM_COL, s>>>(set, st);
    else
      k_pass2_h<N, false><<<set.boff[n], Q::THREADS2, Q::SM_COL, s>>>(set, st);
  } else {
    const GroupSet set =
        make_set(gs, n, [](const GroupDev& g) { return (g.S * (N + 1) + Gm::CPB - 1) / Gm::CPB; });
    if (bf16)
      k_pass2<N, true><<<set.boff[n], Gm::THREADS, Gm::SM2, s>>>(set, st);
    else
      k_pass2<N, false><<<set.boff[n], Gm::THREADS, Gm::SM2, s>>>(set, st);
  }
  TMBIR_CHECK_LAUNCH();
  return TMBIR_OK;
}
template <int N, int MODE>
static int pass3_nm(const GroupDev* gs, int n, const StepArgs& a, const PriorC& pc, const float* apply_out,
                    int phase, double* partials, int off, cudaStream_t s) {
  using GP = GeoP<N>;
  static_assert(GP::NB * GP::CB == pass3_row_blocks(N), "pass-3b block count");
  // each group's slices per block resolved (tuned value or the default rule)
  GroupDev rz[kMergeMax];
  for (int i = 0; i < n; ++i) {
    rz[i] = gs[i];
    rz[i].zc = pass3_zc(gs[i], GP::NB * GP::CB);
  }
  const GroupSet set =
      make_set(rz, n, [](const GroupDev& g) { return GP::NB * GP::CB * ((pass3_slices(g) + g.zc - 1) / g.zc); });
  // a set of several groups only in Iterate mode (the other modes run one group per launch)
  if constexpr (MODE == 3) {
    if (n > 1) {
      if (pc.q_is_2)
        k_pass3<N, 3, true, true><<<set.boff[n], GP::THREADS, GP::SM, s>>>(set, a, pc, apply_out, phase, partials, off);
      else
        k_pass3<N, 3, false, true><<<set.boff[n], GP::THREADS, GP::SM, s>>>(set, a, pc, apply_out, phase, partials,
                                                                           off);
      TMBIR_CHECK_LAUNCH();
      return TMBIR_OK;
    }
  }
  if (n != 1) return set_error(TMBIR_ERR_ARG, "pass 3b takes several groups in Iterate mode only");
  if (pc.q_is_2 || MODE == 0)
    k_pass3<N, MODE, true, false><<<set.boff[n], GP::THREADS, GP::SM, s>>>(set, a, pc, apply_out, phase, partials, off);
  else
    k_pass3<N, MODE, false, false><<<set.boff[n], GP::THREADS, GP::SM, s>>>(set, a, pc, apply_out, phase, partials,
                                                                            off);
  TMBIR_CHECK_LAUNCH();
  return TMBIR_OK;
}
// part: 1 pass 3a only, 2 pass 3b only, 3 both
template <int N>
static int pass3_n(const GroupDev* gs, int n, const StepArgs& a, Pass3Mode m, const PriorC& pc, double* partials,
                   int off, bool bf16, int part, cudaStream_t s) {
  using Gm = Geo3a<N>;
  if (int e = set_smem_limits<N>()) return e;
  if (n < 1 || n > kMergeMax) return set_error(TMBIR_ERR_ARG, "group set size");
  if (bf16 && m != Pass3Mode::Iterate) return set_error(TMBIR_ERR_ARG, "BF16 spectra are an iteration option only");
  // Apply writes K (*) x straight into the output; every other mode into the group's buffer
  float* apply_out = m == Pass3Mode::Apply ? a.out : nullptr;
  const IterState* st = m == Pass3Mode::Iterate ? a.st : nullptr;
  if (part & 1) {
    if constexpr (is_split_side<N>()) {
      using Q = GeoH3<N>;
      const GroupSet set = make_set(gs, n, [](const GroupDev& g) { return g.S * Q::NB; });
      if (bf16)
        k_pass3a_h<N, true><<<set.boff[n], Q::THREADS, Q::SM_ROWS, s>>>(set, st, apply_out);
      else
        k_pass3a_h<N, false><<<set.boff[n], Q::THREADS, Q::SM_ROWS, s>>>(set, st, apply_out);
    } else {
      const GroupSet set = make_set(gs, n, [](const GroupDev& g) { return g.S * Gm::NB; });
      if (bf16)
        k_pass3a<N, true><<<set.boff[n], Gm::THREADS, Gm::SM1, s>>>(set, st, apply_out);
      else
        k_pass3a<N, false><<<set.boff[n], Gm::THREADS, Gm::SM1, s>>>(set, st, apply_out);
    }
    TMBIR_CHECK_LAUNCH();
  }
  if (!(part & 2)) return TMBIR_OK;
  const int phase = bf16 ? 1 : 0;
  switch (m) {
    case Pass3Mode::Apply: return pass3_nm<N, 0>(gs, n, a, pc, apply_out, phase, partials, off, s);
    case Pass3Mode::Gradient: return pass3_nm<N, 1>(gs, n, a, pc, apply_out, phase, partials, off, s);
    case Pass3Mode::Step: return pass3_nm<N, 2>(gs, n, a, pc, apply_out, phase, partials, off, s);
    case Pass3Mode::Iterate: return pass3_nm<N, 3>(gs, n, a, pc, apply_out, phase, partials, off, s);
    default: return pass3_nm<N, 4>(gs, n, a, pc, apply_out, phase, partials, off, s);
  }
}

}  // namespace tmbir

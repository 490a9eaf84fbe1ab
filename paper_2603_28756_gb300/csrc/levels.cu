// Level transfer of the hierarchical reconstruction (Sec. 2.3): the x2 Lanczos-3 upsampler
// (Eqs. 16-17) and the coarse projections obtained by subsampling the detector.
#include "internal.h"

namespace tmbir {

// Lanczos kernel L(x) = sinc(x) sinc(x/3) at the half-integer offsets 2.5, 1.5, 0.5, -0.5,
// -1.5, -2.5 (the printed Eq. 16 is garbled; this is the standard windowed sinc), normalised to
// sum 1.  Filled on the host in FP64 and passed by value.
struct Lz3 {
  float w[6];
};

static Lz3 lanczos3_half_weights() {
  Lz3 z{};
  double w[6], s = 0.0;
  for (int t = 0; t < 6; ++t) {
    const double x = 2.5 - t;
    w[t] = 3.0 * std::sin(M_PI * x) * std::sin(M_PI * x / 3.0) / (M_PI * M_PI * x * x);
    s += w[t];
  }
  for (int t = 0; t < 6; ++t) z.w[t] = (float)(w[t] / s);
  return z;
}

// Separable x2 upsampling: fine sample 2i copies coarse sample i; fine sample 2i+1 =
// sum_t w[t] coarse[i-2+t], along x and then along y.
// Bound by memory (each coarse pixel read once, four fine pixels written).  A thread owns two
// coarse columns (four fine ones) and walks down `rows` coarse rows: the six coarse rows that the
// y taps need stay in registers, already upsampled along x, so a row is read and upsampled once
// per walk plus five rows of overlap, there is no shared memory and every store is 16 bytes.  The
// eight coarse values of the x taps come as four 8-byte loads (neighbouring threads share them in
// L1).  Measured at 32 x 1024^2 (671 MB): 133 us, 5.0 TB/s; the shared-memory form with one output
// per thread and step took 1099 us.  VEC: Nc even, so that rows start on the vector boundaries; odd sides use scalar accesses.
template <bool VEC>
__global__ void __launch_bounds__(128) k_upsample(const float* __restrict__ in, int Nc, int xblocks, int yblocks, int rows,
                                                  float* __restrict__ out, Lz3 z) {
  const int xb = blockIdx.x % xblocks;
  const int s = blockIdx.x / (xblocks * yblocks), yb = (blockIdx.x / xblocks) % yblocks;
  const int c = 2 * (xb * 128 + threadIdx.x);
  if (c >= Nc) return;
  const int Nf = 2 * Nc, r0 = yb * rows, r1 = min(Nc, r0 + rows);
  const float* src = in + (size_t)s * Nc * Nc;
  float* dst = out + (size_t)s * Nf * Nf + 2 * (size_t)c;
  // coarse row r upsampled along x at the thread's four fine columns (zero outside the image)
  auto xrow = [&](int r) {
    if (r < 0 || r >= Nc) return make_float4(0.f, 0.f, 0.f, 0.f);
    const float* row = src + (size_t)r * Nc;
    float v[8];  // coarse columns c - 2 .. c + 5
    if constexpr (VEC) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int cc = c - 2 + 2 * q;
        const float2 p = cc >= 0 && cc < Nc ? __ldg(reinterpret_cast<const float2*>(row + cc)) : make_float2(0.f, 0.f);
        v[2 * q] = p.x;
        v[2 * q + 1] = p.y;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int cc = c - 2 + q;
        v[q] = cc >= 0 && cc < Nc ? __ldg(row + cc) : 0.f;
      }
    }
    float a = 0.f, b = 0.f;
#pragma unroll
    for (int t = 0; t < 6; ++t) {
      a = fmaf(z.w[t], v[t], a);
      b = fmaf(z.w[t], v[t + 1], b);
    }
    return make_float4(v[2], a, v[3], b);
  };
  auto put = [&](int fr, float4 v) {
    float* p = dst + (size_t)fr * Nf;
    if constexpr (VEC) {
      *reinterpret_cast<float4*>(p) = v;
    } else {
      p[0] = v.x;
      p[1] = v.y;
      if (c + 1 < Nc) {
        p[2] = v.z;
        p[3] = v.w;
      }
    }
  };
  float4 w[6];  // rows r - 2 .. r + 3
#pragma unroll
  for (int q = 0; q < 5; ++q) w[q] = xrow(r0 - 2 + q);
#pragma unroll 4
  for (int r = r0; r < r1; ++r) {
    w[5] = xrow(r + 3);
    put(2 * r, w[2]);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int t = 0; t < 6; ++t) {
      v.x = fmaf(z.w[t], w[t].x, v.x);
      v.y = fmaf(z.w[t], w[t].y, v.y);
      v.z = fmaf(z.w[t], w[t].z, v.z);
      v.w = fmaf(z.w[t], w[t].w, v.w);
    }
    put(2 * r + 1, v);
#pragma unroll
    for (int q = 0; q < 5; ++q) w[q] = w[q + 1];
  }
}

int launch_upsample_lanczos3(const float* in, int S, int Nc, float* out, cudaStream_t s) {
  const Lz3 z = lanczos3_half_weights();
  if (Nc > 1969) return set_error(TMBIR_ERR_SHAPE, "upsample: coarse grid too wide");
  // long walks (5 rows of overlap in 37) while they leave four blocks per SM, short ones for small volumes
  const int xblocks = (Nc + 255) / 256;
  const int rows = (long long)S * xblocks * ((Nc + 31) / 32) >= 152 * 4 ? 32 : 8;
  const int yblocks = (Nc + rows - 1) / rows;
  const int blocks = S * xblocks * yblocks;
  if (Nc % 2 == 0)
    k_upsample<true><<<blocks, 128, 0, s>>>(in, Nc, xblocks, yblocks, rows, out, z);
  else
    k_upsample<false><<<blocks, 128, 0, s>>>(in, Nc, xblocks, yblocks, rows, out, z);
  TMBIR_CHECK_LAUNCH();
  return TMBIR_OK;
}

__global__ void k_downsample(const float* __restrict__ in, size_t rows, int nd, int f, float* __restrict__ out) {
  const int ndc = nd / f;
  const float inv = 1.0f / (float)f;
  const size_t total = rows * ndc;
  for (size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x; id < total; id += (size_t)gridDim.x * blockDim.x) {
    const size_t row = id / ndc;
    const int m = (int)(id % ndc);
    out[id] = in[row * nd + (size_t)f * m] * inv;
  }
}

int launch_downsample_sino(const float* in, int S, int na, int nd, int f, float* out, cudaStream_t s) {
  const size_t rows = (size_t)S * na;
  const size_t total = rows * (nd / f);
  const int blocks = (int)std::min<size_t>((total + 255) / 256, 152 * 32);
  k_downsample<<<blocks, 256, 0, s>>>(in, rows, nd, f, out);
  TMBIR_CHECK_LAUNCH();
  return TMBIR_OK;
}

}  // namespace tmbir

// mlp.cu -- the learned warm start: a small MLP maps (E/N, 1/L, J1..J4) to ln g(E)/N and seeds every
// walker's ln g before plain Wang-Landau refines it (the paper has no learned part; Wang-Landau
// still runs every stage, so the network only saves ln f reductions).
//
// Network: 6 inputs (shifted and scaled by fixed per-input constants), 3 hidden layers of 128 SiLU
// units, 1 linear output.  Weights and biases are used in BF16 (rounded from an FP32 master copy
// that Adam updates); activations and every accumulation are FP32.
// Parameter layout (FP32 master, BF16 copy; W stored transposed, WT[k][j] = weight from input k
// to unit j): WT1 [6][128] | b1 [128] | WT2 [128][128] | b2 [128] | WT3 [128][128] | b3 [128] |
// WT4 [128] | b4 [1].
// Loss: per-run centred mean square error, L = (1/M) sum_runs sum_bins (r - mean_run r)^2 with
// r = y - ln g/N, since ln g of a run is only defined up to a constant.
//
// The 128 x 128 contractions run on tensor cores (m16n8k16, BF16 operands, FP32 accumulation): the weights
// are BF16 already, and an FP32 activation is the exact sum of three BF16 numbers (8 + 8 + 8 bits), so
// three products per weight give the FP32 product exactly; products of two FP32 numbers take the six of
// nine partial products above 2^-24.  Each block of 16 terms starts from zero and is then added to the
// FP32 accumulator with a rounded addition, which keeps the error below that of a chain of FP32 FMAs
// (a tensor core's own accumulation truncates).  The accumulator fragments of one layer are, element by
// element, the operand fragments of the next, so a tile of 16 samples stays in one warp's registers
// through the whole network; that is why these are warp-level instructions rather than the CTA-level
// ones with their accumulators in tensor memory: no activation passes through shared memory.
//
// Measured on GB300 (51 840 samples, one Adam step): 1.49 -> 0.25 ms in kernels (forward 0.27 -> 0.043, backward
// with the weight gradients 1.14 -> 0.18) against one CTA of 128 threads per SM with FP32 FMAs; the gradient's
// error against 64 bits 1.9e-7 -> 1.0e-7, the output's 4e-7 -> 2e-7.  Tensor instructions keep the SM 32-41 % busy
// (a loop of nothing else reaches 607 TFLOP/s); the rest is the elementwise part, which two warps per scheduler overlap only
// partly.  (Elementwise work fused between the tensor instructions of the next columns ran slower: the code then
// exceeds the instruction cache.)
//
// Kernels:
//   mlp_fwd_kernel    -- a warp per tile of 16 samples, weights in shared memory;
//   mlp_loss_kernel   -- one CTA per run: centred residual, loss, dL/dy;
//   mlp_bwd_kernel    -- a warp per tile: forward again, back to dL/dZ of every layer; activations and dL/dZ
//                        of a chunk of samples go to a scratch buffer that fits the L2;
//   mlp_dw_kernel     -- weight gradients of the chunk: split over the samples, one partial row per CTA,
//                        in a fixed order;
//   mlp_reduce_kernel -- sum of the partial rows in CTA order (deterministic), loss of the step, and Adam on
//                        the FP32 master with the BF16 copy refreshed.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <random>
#include <string>
#include <vector>

#include "../../include/rewl.h"
#include "device_math.cuh"
#include "jobs.h"
#include "walker.h"

namespace rewl {
namespace mlp {

constexpr int kIn = 6, kH = 128, kT = 16;      // inputs, units of a hidden layer, samples of a warp's tile
constexpr int kWs = kH + 8;                      // padded BF16 row: eight rows of 16 bytes fall into different banks
constexpr int kWarps = 8, kThreads = 32 * kWarps;
constexpr int oW1 = 0, ob1 = oW1 + kIn * kH, oW2 = ob1 + kH, ob2 = oW2 + kH * kH, oW3 = ob2 + kH,
              ob3 = oW3 + kH * kH, oW4 = ob3 + kH, ob4 = oW4 + kH, kParams = ob4 + 1;
constexpr int kRow = (kParams + 7) / 8 * 8;       // partial row, aligned
constexpr int kNt = kH / 8, kKs = kH / 16;       // n-tiles of a layer's output, k-steps of its input

// Weights of a CTA in shared memory: WT1 padded to 16 inputs, WT2, WT3 (rows = inputs), FP32 biases and W4.
struct Weights {
  alignas(16) __nv_bfloat16 w1[16 * kWs];
  __nv_bfloat16 w23[2][kH * kWs];
  alignas(16) float b[3][kH];
  float w4[kH];
  float b4;
};

struct Net {
  const __nv_bfloat16* p;    // BF16 parameters
  float shift[kIn], scale[kIn];
};

// 1 / (1 + e^-z).  Below z = -88, where e^-z would overflow, the value there (6e-39 or 0) stands for it.
__device__ __forceinline__ float sigmoid(float z) { return reciprocal(1.0f + expf(-fmaxf(z, -88.0f))); }

__device__ void stage_weights(Weights& s, const __nv_bfloat16* __restrict__ p) {
  for (int i = threadIdx.x; i < 16 * kH; i += blockDim.x)
    s.w1[(i / kH) * kWs + i % kH] = i < kIn * kH ? p[oW1 + i] : __float2bfloat16_rn(0.0f);
  // rows of 128 BF16 in pieces of 16 bytes (oW2 and oW3 are multiples of 8, the parameter block is aligned)
  static_assert(oW2 % 8 == 0 && oW3 % 8 == 0, "16-byte loads of the weights");
  for (int i = threadIdx.x; i < 2 * kH * kH / 8; i += blockDim.x) {
    const int l = i / (kH * kH / 8), e = (i % (kH * kH / 8)) * 8;
    *reinterpret_cast<uint4*>(&s.w23[l][(e / kH) * kWs + e % kH]) =
        *reinterpret_cast<const uint4*>(p + (l == 0 ? oW2 : oW3) + e);
  }
  for (int i = threadIdx.x; i < kH; i += blockDim.x) {
    s.b[0][i] = __bfloat162float(p[ob1 + i]);
    s.b[1][i] = __bfloat162float(p[ob2 + i]);
    s.b[2][i] = __bfloat162float(p[ob3 + i]);
    s.w4[i] = __bfloat162float(p[oW4 + i]);
  }
  if (threadIdx.x == 0) s.b4 = __bfloat162float(p[ob4]);
}

// D = A B + C on one 16 x 8 tile, K = 16.  Lane = 4 g + t holds rows g and g + 8, columns 2t and 2t + 1 of C
// and D, and the pairs of A's columns 2t, 2t + 8 in those rows.
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, float c0,
                                         float c1, float c2, float c3) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%10, %11, %12, %13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}

template <bool kTrans>
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], const __nv_bfloat16* p) {
  const uint32_t addr = (uint32_t)__cvta_generic_to_shared(p);
  if constexpr (kTrans)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

// (x, y) = hi + mid + lo, each a pair of BF16 (x in the low half): the top 16 bits of an FP32 number are a
// BF16 number, and so are those of the rest, twice; the last rest has at most 8 significant bits.  Exact.
__device__ __forceinline__ void split3(float x, float y, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  auto top = [](float v) { return __uint_as_float(__float_as_uint(v) & 0xffff0000u); };
  auto pack = [](float u, float v) { return __byte_perm(__float_as_uint(u), __float_as_uint(v), 0x7632); };
  hi = pack(x, y);
  const float rx = x - top(x), ry = y - top(y);
  mid = pack(rx, ry);
  lo = pack(rx - top(rx), ry - top(ry));
}

// A warp's 16 x 128 operand: the three parts of k-step i's fragment.
struct Operand {
  uint32_t hi[kKs][4], mid[kKs][4], lo[kKs][4];
  // elements of n-tile nt of a 16 x 128 accumulator: (row g: c0, c1), (row g + 8: c2, c3)
  __device__ __forceinline__ void set(int nt, float c0, float c1, float c2, float c3) {
    const int i = nt / 2, h = 2 * (nt & 1);
    split3(c0, c1, hi[i][h], mid[i][h], lo[i][h]);
    split3(c2, c3, hi[i][h + 1], mid[i][h + 1], lo[i][h + 1]);
  }
};

// The tensor core cuts a block's sum towards zero to 24 bits, which loses 4.3e-8 of it on average (half a unit in
// the last place).  Over five contractions in a row that adds up to a gradient 1.5e-7 too small, so three
// blocks of eight are scaled by 1 + 2^-23 when they are added, 4.5e-8 on average.
__device__ __forceinline__ float block_scale(int k) { return (0x92 >> (k & 7)) & 1 ? 1.0f + 0x1.0p-23f : 1.0f; }

// acc += A W (kTrans: W rows = inputs, the forward pass) or A W^T (the backward pass); W in shared memory.
template <bool kTrans, int kSteps>
__device__ __forceinline__ void contract(float (&acc)[kNt][4], const Operand& A, const __nv_bfloat16* W) {
  const int lane = threadIdx.x & 31;
  const int r = kTrans ? (lane & 15) : (lane & 7) + ((lane >> 4) << 3);
  const int c = kTrans ? (lane >> 4) * 8 : ((lane >> 3) & 1) * 8;
  const __nv_bfloat16* w = W + r * kWs + c;
  constexpr int kG = kSteps < 2 ? kSteps : 2;    // k-steps at a time: 2 kG independent chains of three
#pragma unroll
  for (int np = 0; np < kNt / 2; ++np)
#pragma unroll
    for (int k0 = 0; k0 < kSteps; k0 += kG) {
      uint32_t b[kG][4];
      float t[kG][2][4], u[kG][2][4];
#pragma unroll
      for (int i = 0; i < kG; ++i)
        ldmatrix4<kTrans>(b[i], kTrans ? w + (k0 + i) * 16 * kWs + np * 16 : w + np * 16 * kWs + (k0 + i) * 16);
#pragma unroll
      for (int i = 0; i < kG; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          mma16816(t[i][h], A.lo[k0 + i], b[i][2 * h], b[i][2 * h + 1], 0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
      for (int i = 0; i < kG; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          mma16816(u[i][h], A.mid[k0 + i], b[i][2 * h], b[i][2 * h + 1], t[i][h][0], t[i][h][1], t[i][h][2],
                   t[i][h][3]);
#pragma unroll
      for (int i = 0; i < kG; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          mma16816(t[i][h], A.hi[k0 + i], b[i][2 * h], b[i][2 * h + 1], u[i][h][0], u[i][h][1], u[i][h][2],
                   u[i][h][3]);
#pragma unroll
      for (int i = 0; i < kG; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[2 * np + h][q] = fmaf(t[i][h][q], block_scale(k0 + i), acc[2 * np + h][q]);
    }
}

__device__ __forceinline__ void set_bias(float (&acc)[kNt][4], const float* b) {
  const int t = threadIdx.x & 3;
#pragma unroll
  for (int nt = 0; nt < kNt; ++nt) {
    const float2 v = *reinterpret_cast<const float2*>(b + nt * 8 + 2 * t);
    acc[nt][0] = acc[nt][2] = v.x;
    acc[nt][1] = acc[nt][3] = v.y;
  }
}

// (x - shift) * scale with one rounding (the difference's own rounding error is carried along: 1/L - 0.19, times
// 20, would lose three bits).
__device__ __forceinline__ float normalise(float x, float shift, float scale) {
  const float s = x - shift, b = s - x;
  const float e = (x - (s - b)) - (shift + b);
  return fmaf(s, scale, e * scale);
}

// Normalised inputs of the tile's rows (zero beyond n_t samples) as the first k-step of A, and the first
// layer's Z.
__device__ __forceinline__ void first_layer(const Net& net, const Weights& s, const float* __restrict__ x, int n_t,
                                            Operand& A, float (&z)[kNt][4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  float v[2][2] = {};
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int k = 2 * t + e, row = g + 8 * h;
      if (k < kIn && row < n_t) {
        float sh = net.shift[0], sc = net.scale[0];
#pragma unroll
        for (int q = 1; q < kIn; ++q) {
          sh = k == q ? net.shift[q] : sh;
          sc = k == q ? net.scale[q] : sc;
        }
        v[h][e] = normalise(x[(size_t)row * kIn + k], sh, sc);
      }
    }
  A.set(0, v[0][0], v[0][1], v[1][0], v[1][1]);
  A.set(1, 0.0f, 0.0f, 0.0f, 0.0f);
  set_bias(z, s.b[0]);
  contract<true, 1>(z, A, s.w1);
}

__global__ void __launch_bounds__(kThreads, 1) mlp_fwd_kernel(const Net net, const float* __restrict__ x, long long n,
                                                              float* __restrict__ y) {
  extern __shared__ __align__(16) unsigned char raw[];
  Weights& s = *reinterpret_cast<Weights*>(raw);
  stage_weights(s, net.p);
  __syncthreads();
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const long long n_tiles = (n + kT - 1) / kT;
  // neighbouring tiles go to different CTAs, so that a short batch still spreads over the SMs
  for (long long tile = (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; tile < n_tiles;
       tile += (long long)kWarps * gridDim.x) {
    const long long s0 = tile * kT;
    const int n_t = (int)std::min<long long>(kT, n - s0);
    Operand A;
    float z[kNt][4];
    first_layer(net, s, x + s0 * kIn, n_t, A, z);
#pragma unroll 1
    for (int l = 0; l < 2; ++l) {
#pragma unroll
      for (int nt = 0; nt < kNt; ++nt)
        A.set(nt, z[nt][0] * sigmoid(z[nt][0]), z[nt][1] * sigmoid(z[nt][1]), z[nt][2] * sigmoid(z[nt][2]),
              z[nt][3] * sigmoid(z[nt][3]));
      set_bias(z, s.b[l + 1]);
      contract<true, kKs>(z, A, s.w23[l]);
    }
    float y0 = 0.0f, y1 = 0.0f;
#pragma unroll
    for (int nt = 0; nt < kNt; ++nt) {
      const float2 w = *reinterpret_cast<const float2*>(s.w4 + nt * 8 + 2 * t);
      y0 = fmaf(w.x, z[nt][0] * sigmoid(z[nt][0]), fmaf(w.y, z[nt][1] * sigmoid(z[nt][1]), y0));
      y1 = fmaf(w.x, z[nt][2] * sigmoid(z[nt][2]), fmaf(w.y, z[nt][3] * sigmoid(z[nt][3]), y1));
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      y0 += __shfl_xor_sync(0xffffffffu, y0, o);
      y1 += __shfl_xor_sync(0xffffffffu, y1, o);
    }
    if (t == 0) {
      if (g < n_t) y[s0 + g] = s.b4 + y0;
      if (g + 8 < n_t) y[s0 + g + 8] = s.b4 + y1;
    }
  }
}

// One CTA per run g (samples seg[g] .. seg[g+1]-1): residual r = y - t, its mean, the loss part
// sum (r - mean)^2 (FP64) and dy = 2 (r - mean) / M.
__global__ void mlp_loss_kernel(const float* __restrict__ y, const float* __restrict__ t, const int* __restrict__ seg,
                                double m, float* __restrict__ dy, double* __restrict__ loss_part) {
  const int g = blockIdx.x;
  const int a = seg[g], b = seg[g + 1];
  __shared__ double red[32];
  double sr = 0.0;
  for (int i = a + threadIdx.x; i < b; i += blockDim.x) sr += (double)y[i] - (double)t[i];
  for (int o = 16; o > 0; o >>= 1) sr += __shfl_xor_sync(0xffffffffu, sr, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sr;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[w];
    red[31] = b > a ? v / (double)(b - a) : 0.0;
  }
  __syncthreads();
  const double mean = red[31];
  __syncthreads();
  double sl = 0.0;
  for (int i = a + threadIdx.x; i < b; i += blockDim.x) {
    const double r = ((double)y[i] - (double)t[i]) - mean;
    sl += r * r;
    dy[i] = (float)(2.0 * r / m);
  }
  for (int o = 16; o > 0; o >>= 1) sl += __shfl_xor_sync(0xffffffffu, sl, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sl;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[w];
    loss_part[g] = v;
  }
}

// Activations A1, A2 and dL/dZ of the three hidden layers for one chunk of samples, [samples][128] each.
struct Chunk {
  float* a[2];
  float* dz[3];
  static Chunk of(float* p, long long chunk) {
    Chunk c;
    for (int l = 0; l < 2; ++l) c.a[l] = p + l * chunk * kH;
    for (int l = 0; l < 3; ++l) c.dz[l] = p + (2 + l) * chunk * kH;
    return c;
  }
};

struct BwdSmem {
  Weights w;
  alignas(16) float4 d[kWarps][2][kNt][32];    // silu'(Z1), silu'(Z2): every thread's own elements
  float g4[kWarps][kH], gb4[kWarps];
};
static_assert(sizeof(BwdSmem) <= 227 * 1024, "backward pass does not fit in shared memory");

// silu(z) = z s and silu'(z) = s (1 + z (1 - s)) with s = 1 / (1 + e), 1 - s = e s (no cancellation), e = e^-z
__device__ __forceinline__ float silu(float z, float& d) {
  const float e = expf(-fmaxf(z, -88.0f)), sg = reciprocal(1.0f + e);
  d = sg * fmaf(z, e * sg, 1.0f);
  return z * sg;
}

__device__ __forceinline__ void put_rows(float* out, int n_t, int nt, float c0, float c1, float c2, float c3) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  float* p = out + (size_t)g * kH + nt * 8 + 2 * t;
  if (g < n_t) *reinterpret_cast<float2*>(p) = make_float2(c0, c1);
  if (g + 8 < n_t) *reinterpret_cast<float2*>(p + 8 * kH) = make_float2(c2, c3);
}

// One chunk of n samples: forward again, then dL/dZ of every layer; the output layer's gradient into row
// blockIdx.x of partial (first: set, else added).
// What bounds it: the tensor-core instructions and the elementwise part about equally (per tile of 16 samples
// and layer 384 of the former and 64 elements a thread of the latter).
__global__ void __launch_bounds__(kThreads, 1) mlp_bwd_kernel(const Net net, const float* __restrict__ x,
                                                              const float* __restrict__ dy, int n, const Chunk c,
                                                              float* __restrict__ partial, int first) {
  extern __shared__ __align__(16) unsigned char raw[];
  BwdSmem& s = *reinterpret_cast<BwdSmem*>(raw);
  stage_weights(s.w, net.p);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  float g4[4] = {0.0f, 0.0f, 0.0f, 0.0f}, gb4 = 0.0f;
  const int n_tiles = (n + kT - 1) / kT;
  for (int tile = warp * gridDim.x + blockIdx.x; tile < n_tiles; tile += kWarps * gridDim.x) {
    const int s0 = tile * kT;
    const int n_t = min(kT, n - s0);
    Operand A;
    float z[kNt][4];
    first_layer(net, s.w, x + (size_t)s0 * kIn, n_t, A, z);
#pragma unroll 1
    for (int l = 0; l < 2; ++l) {
      float* out = (l == 0 ? c.a[0] : c.a[1]) + (size_t)s0 * kH;
#pragma unroll
      for (int nt = 0; nt < kNt; ++nt) {
        float4 d;
        const float a0 = silu(z[nt][0], d.x), a1 = silu(z[nt][1], d.y), a2 = silu(z[nt][2], d.z),
                    a3 = silu(z[nt][3], d.w);
        s.d[warp][l][nt][lane] = d;
        put_rows(out, n_t, nt, a0, a1, a2, a3);
        A.set(nt, a0, a1, a2, a3);
      }
      set_bias(z, s.w.b[l + 1]);
      contract<true, kKs>(z, A, s.w.w23[l]);
    }
    const float dy0 = g < n_t ? dy[s0 + g] : 0.0f, dy1 = g + 8 < n_t ? dy[s0 + g + 8] : 0.0f;
    // output layer: y = b4 + sum_k W4[k] A3[k]; its gradient's sums over the tile's rows: the lanes of a
    // column group (same t) halve the columns they hold at every exchange, so 28 of them do
    float p4[2 * kNt];
#pragma unroll
    for (int nt = 0; nt < kNt; ++nt) {
      float4 d;
      const float a0 = silu(z[nt][0], d.x), a1 = silu(z[nt][1], d.y), a2 = silu(z[nt][2], d.z),
                  a3 = silu(z[nt][3], d.w);
      p4[2 * nt] = fmaf(a0, dy0, a2 * dy1);
      p4[2 * nt + 1] = fmaf(a1, dy0, a3 * dy1);
      const float2 w = *reinterpret_cast<const float2*>(s.w.w4 + nt * 8 + 2 * t);
      const float e0 = w.x * dy0 * d.x, e1 = w.y * dy0 * d.y, e2 = w.x * dy1 * d.z, e3 = w.y * dy1 * d.w;
      put_rows(c.dz[2] + (size_t)s0 * kH, n_t, nt, e0, e1, e2, e3);
      A.set(nt, e0, e1, e2, e3);
    }
#pragma unroll
    for (int o = 0; o < 3; ++o) {
      const int half = kNt >> o, bit = 16 >> o;          // values kept: 16, 8, 4
      const bool up = (lane & bit) != 0;
#pragma unroll
      for (int q = 0; q < half; ++q) {
        const float keep = up ? p4[half + q] : p4[q], give = up ? p4[q] : p4[half + q];
        p4[q] = keep + __shfl_xor_sync(0xffffffffu, give, bit);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) g4[q] += p4[q];
    gb4 += t == 0 ? dy0 + dy1 : 0.0f;
    // hidden layers 3 and 2: dA = dZ W^T, dZ below = dA silu'
#pragma unroll 1
    for (int l = 1; l >= 0; --l) {
#pragma unroll
      for (int nt = 0; nt < kNt; ++nt) z[nt][0] = z[nt][1] = z[nt][2] = z[nt][3] = 0.0f;
      contract<false, kKs>(z, A, s.w.w23[l]);
      float* out = (l == 0 ? c.dz[0] : c.dz[1]) + (size_t)s0 * kH;
#pragma unroll
      for (int nt = 0; nt < kNt; ++nt) {
        const float4 d = s.d[warp][l][nt][lane];
        const float e0 = z[nt][0] * d.x, e1 = z[nt][1] * d.y, e2 = z[nt][2] * d.z, e3 = z[nt][3] * d.w;
        put_rows(out, n_t, nt, e0, e1, e2, e3);
        A.set(nt, e0, e1, e2, e3);
      }
    }
  }
  // column of value q of this lane: the three exchanges took the upper half for lane bits 16, 8, 4
  const int v0 = ((lane >> 4) & 1) * 16 + ((lane >> 3) & 1) * 8 + ((lane >> 2) & 1) * 4;
#pragma unroll
  for (int q = 0; q < 4; ++q) s.g4[warp][((v0 + q) >> 1) * 8 + 2 * t + ((v0 + q) & 1)] = g4[q];
  for (int o = 16; o > 0; o >>= 1) gb4 += __shfl_xor_sync(0xffffffffu, gb4, o);
  if (lane == 0) s.gb4[warp] = gb4;
  __syncthreads();
  float* row = partial + (size_t)blockIdx.x * kRow;
  if (threadIdx.x <= kH) {
    const bool bias = threadIdx.x == kH;
    float v = 0.0f;
    for (int w = 0; w < kWarps; ++w) v += bias ? s.gb4[w] : s.g4[w][threadIdx.x];
    float* o = row + (bias ? ob4 : oW4 + threadIdx.x);
    *o = first ? v : *o + v;
  }
}

constexpr int kDwT = 64;                         // samples of a tile of the weight-gradient kernel

// Three BF16 parts of a tile of A (or of the inputs, in 16 columns) and of dZ, rows = samples; two tiles, one
// in use and one being filled.
struct DwSmem {
  struct Tile {
    alignas(16) __nv_bfloat16 a[3][kDwT * kWs];
    alignas(16) __nv_bfloat16 z[3][kDwT * kWs];
  } tile[2];
  alignas(16) float4 bias[3][kWarps][32];
};
static_assert(sizeof(DwSmem) <= 227 * 1024, "weight-gradient tiles do not fit in shared memory");

// This thread's part of a [64][128] tile: columns 4 lane .. 4 lane + 3 of rows warp, warp + 8, ...; rows beyond
// n_r are zero.
__device__ __forceinline__ void fetch_tile(float4 (&v)[kDwT / kWarps], const float* __restrict__ in, int n_r) {
#pragma unroll
  for (int i = 0; i < kDwT / kWarps; ++i) {
    const int r = (threadIdx.x >> 5) + kWarps * i;
    v[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (r < n_r) v[i] = *reinterpret_cast<const float4*>(in + (size_t)r * kH + (threadIdx.x & 31) * 4);
  }
}

__device__ __forceinline__ void store_tile(__nv_bfloat16 (&out)[3][kDwT * kWs], const float4 (&v)[kDwT / kWarps]) {
  const int col = (threadIdx.x & 31) * 4;
#pragma unroll
  for (int i = 0; i < kDwT / kWarps; ++i) {
    const int r = (threadIdx.x >> 5) + kWarps * i;
    uint2 hi, mid, lo;
    split3(v[i].x, v[i].y, hi.x, mid.x, lo.x);
    split3(v[i].z, v[i].w, hi.y, mid.y, lo.y);
    *reinterpret_cast<uint2*>(&out[0][r * kWs + col]) = hi;
    *reinterpret_cast<uint2*>(&out[1][r * kWs + col]) = mid;
    *reinterpret_cast<uint2*>(&out[2][r * kWs + col]) = lo;
  }
}

// acc[mt][n .. n + 1] += the products of FP32 operands given by their three parts: the six partial products that
// reach FP32 precision, smallest first, 2 kMt independent chains.
template <int kMt>
__device__ __forceinline__ void mma_fp32(float (&acc)[2][8][4], int n, const uint32_t (&a)[kMt][3][4],
                                         const uint32_t (&b)[3][4], float scale) {
  constexpr int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
  float t[kMt][2][4] = {};
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float (&d)[4] = t[mt][h];
        mma16816(d, a[mt][pa[i]], b[pb[i]][2 * h], b[pb[i]][2 * h + 1], d[0], d[1], d[2], d[3]);
      }
#pragma unroll
  for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[mt][n + h][q] = fmaf(t[mt][h][q], scale, acc[mt][n + h][q]);
}

// Weight and bias gradients of a chunk: CTA i does layers 3, 2, 1 for the i-th share of its samples, into row i
// of partial (first: set, else added).  Warp w holds rows 32 (w / 2) .., columns 64 (w % 2) .. of the
// 128 x 128 gradient.  The next tile is loaded while the present one is multiplied.
// What bounds it: the tensor-core instructions (6 x 128 per 16 samples and layer).
__global__ void __launch_bounds__(kThreads, 1) mlp_dw_kernel(const Net net, const float* __restrict__ x, int n,
                                                             const Chunk c, float* __restrict__ partial, int first) {
  extern __shared__ __align__(16) unsigned char raw[];
  DwSmem& s = *reinterpret_cast<DwSmem*>(raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int share = ((n + (int)gridDim.x - 1) / (int)gridDim.x + kT - 1) / kT * kT;
  const int s_begin = min(n, (int)blockIdx.x * share), s_end = min(n, s_begin + share);
  const int tiles = max(1, (s_end - s_begin + kDwT - 1) / kDwT);
  float* row = partial + (size_t)blockIdx.x * kRow;
  const int ra = (lane & 7) + ((lane >> 4) << 3), ca = ((lane >> 3) & 1) * 8;   // A: ldmatrix row, column
  const int rb = lane & 15, cb = (lane >> 4) * 8;                                // B
  const int m0 = 32 * (warp >> 1), n0 = 64 * (warp & 1);
  auto put = [&](float* o, float v) { *o = first ? v : *o + v; };
  // step q: layer 2 - q / tiles (operand and dZ: 2: A2, dZ3; 1: A1, dZ2; 0: inputs, dZ1), tile q % tiles
  float4 vz[kDwT / kWarps], va[kDwT / kWarps];
  float2 vx[2];
  float4 sum[3] = {};                        // column sums of dZ, by layer
  auto fetch = [&](int l, int k) {
    const int s0 = s_begin + k * kDwT, n_r = max(0, min(kDwT, s_end - s0));
    fetch_tile(vz, (l == 2 ? c.dz[2] : (l == 1 ? c.dz[1] : c.dz[0])) + (size_t)s0 * kH, n_r);
    if (l > 0) {
      fetch_tile(va, (l == 2 ? c.a[1] : c.a[0]) + (size_t)s0 * kH, n_r);
    } else {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int e = threadIdx.x + i * kThreads, r = e >> 3, k2 = (e & 7) * 2;
        float v[2] = {0.0f, 0.0f};
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int j = 0; j < kIn; ++j)
            if (k2 + h == j && r < n_r) v[h] = normalise(x[(size_t)(s0 + r) * kIn + j], net.shift[j], net.scale[j]);
        vx[i] = make_float2(v[0], v[1]);
      }
    }
  };
  auto store = [&](int l, DwSmem::Tile& b) {
#pragma unroll
    for (int j = 0; j < 3; ++j)
      if (l == j) {
#pragma unroll
        for (int i = 0; i < kDwT / kWarps; ++i) {
          sum[j].x += vz[i].x;
          sum[j].y += vz[i].y;
          sum[j].z += vz[i].z;
          sum[j].w += vz[i].w;
        }
      }
    store_tile(b.z, vz);
    if (l > 0) {
      store_tile(b.a, va);
    } else {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int e = threadIdx.x + i * kThreads, r = e >> 3, k2 = (e & 7) * 2;
        uint32_t hi, mid, lo;
        split3(vx[i].x, vx[i].y, hi, mid, lo);
        *reinterpret_cast<uint32_t*>(&b.a[0][r * kWs + k2]) = hi;
        *reinterpret_cast<uint32_t*>(&b.a[1][r * kWs + k2]) = mid;
        *reinterpret_cast<uint32_t*>(&b.a[2][r * kWs + k2]) = lo;
      }
    }
  };
  static_assert(kDwT * 8 == 2 * kThreads, "two input pairs per thread");
  // Two warps share a scheduler: while one multiplies the present tile, the other splits and stores its part of the
  // next (fetched a tile ahead), then they change over.
  const bool store_first = (warp & 4) != 0;
  const int n_steps = 3 * tiles;
  fetch(2, 0);
  store(2, s.tile[0]);
  if (tiles > 1)
    fetch(2, 1);
  else
    fetch(1, 0);
  __syncthreads();
  float acc[2][8][4] = {};
  int l = 2, k = 0;
#pragma unroll 1
  for (int q = 0; q < n_steps; ++q) {
    const int l1 = k + 1 < tiles ? l : l - 1, k1 = k + 1 < tiles ? k + 1 : 0;        // the next step
    const int l2 = k1 + 1 < tiles ? l1 : l1 - 1, k2 = k1 + 1 < tiles ? k1 + 1 : 0;   // the one after it
    const DwSmem::Tile& b = s.tile[q & 1];
    auto hand_on = [&]() {
      if (q + 1 < n_steps) store(l1, s.tile[(q & 1) ^ 1]);
      if (q + 2 < n_steps) fetch(l2, k2);
    };
    if (store_first) hand_on();
    const int steps = (max(0, min(kDwT, s_end - s_begin - k * kDwT)) + kT - 1) / kT;
    if (l > 0) {
#pragma unroll 1
      for (int ks = 0; ks < steps; ++ks) {
        const float scale = block_scale(4 * k + ks + (int)blockIdx.x);
        uint32_t a[2][3][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
          for (int p = 0; p < 3; ++p)
            ldmatrix4<true>(a[mt][p], &b.a[p][(ks * kT + ra) * kWs + m0 + mt * 16 + ca]);
#pragma unroll
        for (int np = 0; np < 4; ++np) {
          uint32_t b4[3][4];
#pragma unroll
          for (int p = 0; p < 3; ++p) ldmatrix4<true>(b4[p], &b.z[p][(ks * kT + rb) * kWs + n0 + np * 16 + cb]);
          mma_fp32<2>(acc, 2 * np, a, b4, scale);
        }
      }
    } else {
#pragma unroll 1
      for (int ks = 0; ks < steps; ++ks) {
        const float scale = block_scale(4 * k + ks + (int)blockIdx.x);
        uint32_t a[1][3][4], b4[3][4];
#pragma unroll
        for (int p = 0; p < 3; ++p) {
          ldmatrix4<true>(a[0][p], &b.a[p][(ks * kT + ra) * kWs + ca]);
          ldmatrix4<true>(b4[p], &b.z[p][(ks * kT + rb) * kWs + warp * 16 + cb]);
        }
        mma_fp32<1>(acc, 0, a, b4, scale);
      }
    }
    if (k + 1 == tiles) {                    // the layer's weights
      if (l > 0) {
        // the reads of an earlier chunk's sums all go out before the first write (a write would hold
        // back the reads after it)
        float* gw = row + (l == 2 ? oW3 : oW2) + (m0 + g) * kH + n0 + 2 * t;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
          float2 old[8][2] = {};
          if (!first) {
#pragma unroll
            for (int nt = 0; nt < 8; ++nt)
#pragma unroll
              for (int e = 0; e < 2; ++e)
                old[nt][e] = *reinterpret_cast<const float2*>(gw + (mt * 16 + e * 8) * kH + nt * 8);
          }
#pragma unroll
          for (int nt = 0; nt < 8; ++nt)
#pragma unroll
            for (int e = 0; e < 2; ++e)
              *reinterpret_cast<float2*>(gw + (mt * 16 + e * 8) * kH + nt * 8) =
                  make_float2(old[nt][e].x + acc[mt][nt][2 * e], old[nt][e].y + acc[mt][nt][2 * e + 1]);
        }
      } else if (g < kIn) {
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int e = 0; e < 2; ++e)
            put(row + oW1 + g * kH + warp * 16 + nt * 8 + 2 * t + e, acc[0][nt][e]);
      }
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 8; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[mt][nt][e] = 0.0f;
    }
    if (!store_first) hand_on();
    __syncthreads();
    l = l1;
    k = k1;
  }
  // biases: the eight row groups' column sums
  s.bias[0][warp][lane] = sum[0];
  s.bias[1][warp][lane] = sum[1];
  s.bias[2][warp][lane] = sum[2];
  __syncthreads();
  for (int i = threadIdx.x; i < 3 * kH; i += kThreads) {
    const int bl = i / kH, col = i % kH;
    const float* bs = reinterpret_cast<const float*>(s.bias[bl]);
    float v = 0.0f;
    for (int w = 0; w < kWarps; ++w) v += bs[w * kH + col];
    put(row + (bl == 2 ? ob3 : (bl == 1 ? ob2 : ob1)) + col, v);
  }
}

struct AdamArgs {
  float lr, b1, b2, eps, c1, c2;   // c1 = 1 - b1^t, c2 = 1 - b2^t
};

// grad[p] = sum of the partial rows in row order; with w, one Adam step of parameter p.  The last CTA sums
// the runs' loss parts (over the n samples) into *loss when given.
__global__ void mlp_reduce_kernel(const float* __restrict__ partial, int n_rows, float* __restrict__ grad,
                                  const double* __restrict__ loss_part, int n_runs, double n, double* loss,
                                  float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                                  __nv_bfloat16* __restrict__ wb, const AdamArgs a) {
  if (blockIdx.x == gridDim.x - 1) {
    if (loss && threadIdx.x < 32) {
      double t = 0.0;
      for (int r = threadIdx.x; r < n_runs; r += 32) t += loss_part[r];
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (threadIdx.x == 0) *loss = t / n;
    }
    return;
  }
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kParams) return;
  // the rounding error of every addition is kept (two-sum) and added at the end: 152 plain additions would
  // lose 2e-7, more than everything before them
  float gr = 0.0f, lost = 0.0f;
#pragma unroll 8
  for (int r = 0; r < n_rows; ++r) {
    const float v = partial[(size_t)r * kRow + p];
    const float t = gr + v, b = t - gr;
    lost += (gr - (t - b)) + (v - b);
    gr = t;
  }
  gr += lost;
  grad[p] = gr;
  if (!w) return;
  const float mm = a.b1 * m[p] + (1.0f - a.b1) * gr;
  const float vv = a.b2 * v[p] + (1.0f - a.b2) * gr * gr;
  m[p] = mm;
  v[p] = vv;
  const float mh = mm / a.c1, vh = vv / a.c2;
  const float nw = w[p] - a.lr * mh / (sqrtf(vh) + a.eps);
  w[p] = nw;
  wb[p] = __float2bfloat16_rn(nw);
}

__global__ void to_bf16_kernel(const float* __restrict__ w, __nv_bfloat16* __restrict__ wb) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < kParams) wb[p] = __float2bfloat16_rn(w[p]);
}

}  // namespace mlp
}  // namespace rewl

using namespace rewl;
using namespace rewl::mlp;

struct rewl_mlp {
  Net net{};
  cudaStream_t stream = nullptr;
  float* d_w = nullptr;          // FP32 master
  __nv_bfloat16* d_wb = nullptr;  // BF16 copy used by the kernels
  float* d_grad = nullptr;
  float* d_m = nullptr;
  float* d_v = nullptr;
  float* d_partial = nullptr;
  float* d_chunk = nullptr;      // activations and dL/dZ of one chunk of samples, allocated by the first gradient
  long long chunk_rows = 0;      // samples that d_chunk holds
  int grid = 0;                  // CTAs of a pass over the samples (= rows of d_partial)
  long long adam_t = 0;
  std::vector<void*> allocations;
  bool broken = false;
};

namespace {

rewl_status mfail(rewl_mlp* m, rewl_status s, const std::string& msg) {
  if (m && s == REWL_ECUDA) m->broken = true;
  set_handleless_error("mlp: " + msg);
  return s;
}

#define MCUDA(m, call)                                                                                  \
  do {                                                                                                  \
    cudaError_t e_ = (call);                                                                            \
    if (e_ != cudaSuccess) return mfail((m), REWL_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

template <class T>
rewl_status malloc_dev(rewl_mlp* m, T** p, size_t count) {
  void* q = nullptr;
  const cudaError_t e = cudaMalloc(&q, std::max<size_t>(count, 1) * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();          // (the model stays usable: the next launch's check must not find this)
    return mfail(m, REWL_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  }
  m->allocations.push_back(q);
  *p = static_cast<T*>(q);
  return REWL_OK;
}

// device scratch of one call, freed on return in the order of the model's stream
struct Scratch {
  cudaStream_t stream;
  std::vector<void*> ptrs;
  explicit Scratch(rewl_mlp* m) : stream(m->stream) {}
  ~Scratch() {
    for (void* p : ptrs) pool_free(p, stream);
  }
  template <class T>
  cudaError_t get(T** p, size_t count) {
    void* q = nullptr;
    const cudaError_t e = pool_alloc(&q, std::max<size_t>(count, 1) * sizeof(T), stream);
    if (e == cudaSuccess) {
      ptrs.push_back(q);
      *p = static_cast<T*>(q);
    }
    return e;
  }
};

rewl_status check_mlp(rewl_mlp* m) {
  if (!m) return mfail(nullptr, REWL_EINVAL, "null model");
  if (m->broken) return mfail(m, REWL_ESTATE, "model saw a CUDA error; destroy it");
  return REWL_OK;
}

int fwd_grid(const rewl_mlp* m, long long n) {
  const long long ctas = (n + kWarps * kT - 1) / (kWarps * kT);
  return (int)std::max<long long>(1, std::min<long long>(ctas, m->grid));
}

rewl_status check_segments(const int32_t* seg, int n_segs, long long n) {
  if (!seg || n_segs < 1) return mfail(nullptr, REWL_EINVAL, "no runs");
  if (seg[0] != 0 || seg[n_segs] != n) return mfail(nullptr, REWL_EINVAL, "run offsets must start at 0 and end at n");
  for (int g = 0; g < n_segs; ++g)
    if (seg[g + 1] <= seg[g]) return mfail(nullptr, REWL_EINVAL, "run offsets must increase");
  return REWL_OK;
}

// Room in d_chunk for `rows` samples, of `most` that are ever needed at once.  It grows by half at least, so that
// larger and larger corpora seldom allocate; from the pool, as a new model's first gradient pays for it (500 samples:
// 475 us, 590 with a cudaMalloc of its own).
rewl_status reserve_chunk(rewl_mlp* m, long long rows, long long most) {
  if (rows <= m->chunk_rows) return REWL_OK;
  rows = std::min(most, std::max(rows, m->chunk_rows + m->chunk_rows / 2));
  pool_free(m->d_chunk, m->stream);
  m->d_chunk = nullptr;
  m->chunk_rows = 0;
  void* p = nullptr;
  const cudaError_t e = pool_alloc(&p, 5 * (size_t)rows * kH * sizeof(float), m->stream);
  if (e != cudaSuccess) return mfail(m, REWL_ENOMEM, std::string("backward scratch: ") + cudaGetErrorString(e));
  m->d_chunk = static_cast<float*>(p);
  m->chunk_rows = rows;
  return REWL_OK;
}

// Loss and gradient of the full batch into m->d_grad, the loss (FP32) into *d_loss when given; with adam,
// one step of the parameters too.  Stream-ordered.
rewl_status loss_and_grad(rewl_mlp* m, const float* dx, const float* dt, const int* dseg, int n_segs, long long n,
                          float* dy_buf, float* dydy, double* dloss, double* d_loss, const AdamArgs* adam) {
  const long long chunk = 2LL * m->grid * kWarps * kT;   // two rounds of the backward pass: about 100 MB, in the L2
  const rewl_status s = reserve_chunk(m, std::min(n, chunk), chunk);
  if (s != REWL_OK) return s;
  mlp_fwd_kernel<<<fwd_grid(m, n), kThreads, sizeof(Weights), m->stream>>>(m->net, dx, n, dy_buf);
  MCUDA(m, cudaGetLastError());
  mlp_loss_kernel<<<n_segs, 256, 0, m->stream>>>(dy_buf, dt, dseg, (double)n, dydy, dloss);
  MCUDA(m, cudaGetLastError());
  const Chunk c = Chunk::of(m->d_chunk, m->chunk_rows);
  for (long long s0 = 0; s0 < n; s0 += chunk) {
    const int n_c = (int)std::min<long long>(chunk, n - s0);
    const int first = s0 == 0 ? 1 : 0;
    mlp_bwd_kernel<<<m->grid, kThreads, sizeof(BwdSmem), m->stream>>>(m->net, dx + s0 * kIn, dydy + s0, n_c, c,
                                                                       m->d_partial, first);
    MCUDA(m, cudaGetLastError());
    mlp_dw_kernel<<<m->grid, kThreads, sizeof(DwSmem), m->stream>>>(m->net, dx + s0 * kIn, n_c, c,
                                                                              m->d_partial, first);
    MCUDA(m, cudaGetLastError());
  }
  AdamArgs a{};
  if (adam) a = *adam;
  mlp_reduce_kernel<<<(kParams + 255) / 256 + 1, 256, 0, m->stream>>>(m->d_partial, m->grid, m->d_grad, dloss, n_segs,
                                                                     (double)n, d_loss, adam ? m->d_w : nullptr,
                                                                     m->d_m, m->d_v, m->d_wb, a);
  MCUDA(m, cudaGetLastError());
  return REWL_OK;
}

struct Corpus {
  Scratch sc;
  explicit Corpus(rewl_mlp* m) : sc(m) {}
  float *x = nullptr, *t = nullptr, *y = nullptr, *dy = nullptr;
  int* seg = nullptr;
  double* loss = nullptr;
};

rewl_status upload_corpus(rewl_mlp* m, Corpus& c, const float* x, const float* t, const int32_t* seg, int n_segs) {
  const long long n = seg[n_segs];
  MCUDA(m, c.sc.get(&c.x, (size_t)n * kIn));
  MCUDA(m, c.sc.get(&c.t, (size_t)n));
  MCUDA(m, c.sc.get(&c.y, (size_t)n));
  MCUDA(m, c.sc.get(&c.dy, (size_t)n));
  MCUDA(m, c.sc.get(&c.seg, (size_t)n_segs + 1));
  MCUDA(m, c.sc.get(&c.loss, (size_t)n_segs));
  MCUDA(m, cudaMemcpyAsync(c.x, x, sizeof(float) * (size_t)n * kIn, cudaMemcpyHostToDevice, m->stream));
  MCUDA(m, cudaMemcpyAsync(c.t, t, sizeof(float) * (size_t)n, cudaMemcpyHostToDevice, m->stream));
  MCUDA(m, cudaMemcpyAsync(c.seg, seg, sizeof(int) * ((size_t)n_segs + 1), cudaMemcpyHostToDevice, m->stream));
  return REWL_OK;
}

}  // namespace

extern "C" int64_t rewl_mlp_param_count(void) { return kParams; }

extern "C" rewl_status rewl_mlp_create(const float* in_shift, const float* in_scale, uint64_t seed, void* cuda_stream,
                                       rewl_mlp** out) {
  if (!out) return mfail(nullptr, REWL_EINVAL, "NULL out");
  *out = nullptr;
  if (!in_shift || !in_scale) return mfail(nullptr, REWL_EINVAL, "NULL input normalisation");
  for (int k = 0; k < kIn; ++k)
    if (!std::isfinite(in_shift[k]) || !std::isfinite(in_scale[k]) || in_scale[k] == 0.0f)
      return mfail(nullptr, REWL_EINVAL, "input normalisation must be finite with nonzero scales");
  auto* m = new rewl_mlp();
  pool_retain();
  for (int k = 0; k < kIn; ++k) {
    m->net.shift[k] = in_shift[k];
    m->net.scale[k] = in_scale[k];
  }
  m->stream = static_cast<cudaStream_t>(cuda_stream);
  int dev = 0, n_sms = 0;
  cudaError_t ce = cudaGetDevice(&dev);
  if (ce == cudaSuccess) ce = cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev);
  if (ce == cudaSuccess)
    ce = cudaFuncSetAttribute(mlp_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Weights));
  if (ce == cudaSuccess)
    ce = cudaFuncSetAttribute(mlp_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BwdSmem));
  if (ce == cudaSuccess)
    ce = cudaFuncSetAttribute(mlp_dw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DwSmem));
  if (ce != cudaSuccess) {
    pool_release();
    delete m;
    return mfail(nullptr, REWL_ECUDA, std::string("CUDA set-up: ") + cudaGetErrorString(ce));
  }
  m->grid = std::max(1, n_sms);
  rewl_status s = malloc_dev(m, &m->d_w, kParams);
  if (s == REWL_OK) s = malloc_dev(m, &m->d_wb, kParams);
  if (s == REWL_OK) s = malloc_dev(m, &m->d_grad, kParams);
  if (s == REWL_OK) s = malloc_dev(m, &m->d_m, kParams);
  if (s == REWL_OK) s = malloc_dev(m, &m->d_v, kParams);
  if (s == REWL_OK) s = malloc_dev(m, &m->d_partial, (size_t)m->grid * kRow);
  if (s != REWL_OK) {
    rewl_mlp_destroy(m);
    return s;
  }
  m->net.p = m->d_wb;
  // uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) weights, zero biases, from a seeded generator
  std::vector<float> w(kParams, 0.0f);
  std::mt19937_64 gen(seed);
  auto fill = [&](int off, int count, int fan_in) {
    std::uniform_real_distribution<float> d(-1.0f / std::sqrt((float)fan_in), 1.0f / std::sqrt((float)fan_in));
    for (int i = 0; i < count; ++i) w[off + i] = d(gen);
  };
  fill(oW1, kIn * kH, kIn);
  fill(oW2, kH * kH, kH);
  fill(oW3, kH * kH, kH);
  fill(oW4, kH, kH);
  s = rewl_mlp_set_params(m, w.data());
  if (s != REWL_OK) {
    rewl_mlp_destroy(m);
    return s;
  }
  *out = m;
  return REWL_OK;
}

extern "C" rewl_status rewl_mlp_set_params(rewl_mlp* m, const float* params) {
  rewl_status s = check_mlp(m);
  if (s != REWL_OK) return s;
  if (!params) return mfail(m, REWL_EINVAL, "NULL params");
  MCUDA(m, cudaMemcpyAsync(m->d_w, params, sizeof(float) * kParams, cudaMemcpyHostToDevice, m->stream));
  to_bf16_kernel<<<(kParams + 255) / 256, 256, 0, m->stream>>>(m->d_w, m->d_wb);
  MCUDA(m, cudaGetLastError());
  MCUDA(m, cudaMemsetAsync(m->d_m, 0, sizeof(float) * kParams, m->stream));
  MCUDA(m, cudaMemsetAsync(m->d_v, 0, sizeof(float) * kParams, m->stream));
  MCUDA(m, cudaStreamSynchronize(m->stream));
  m->adam_t = 0;
  return REWL_OK;
}

extern "C" rewl_status rewl_mlp_get_params(rewl_mlp* m, float* params, uint16_t* params_bf16) {
  rewl_status s = check_mlp(m);
  if (s != REWL_OK) return s;
  if (params)
    MCUDA(m, cudaMemcpyAsync(params, m->d_w, sizeof(float) * kParams, cudaMemcpyDeviceToHost, m->stream));
  if (params_bf16)
    MCUDA(m, cudaMemcpyAsync(params_bf16, m->d_wb, sizeof(uint16_t) * kParams, cudaMemcpyDeviceToHost, m->stream));
  MCUDA(m, cudaStreamSynchronize(m->stream));
  return REWL_OK;
}

extern "C" rewl_status rewl_mlp_forward(rewl_mlp* m, const float* x, int64_t n, float* y) {
  rewl_status s = check_mlp(m);
  if (s != REWL_OK) return s;
  if (!x || !y || n < 1) return mfail(m, REWL_EINVAL, "bad forward arguments");
  Corpus c(m);
  MCUDA(m, c.sc.get(&c.x, (size_t)n * kIn));
  MCUDA(m, c.sc.get(&c.y, (size_t)n));
  MCUDA(m, cudaMemcpyAsync(c.x, x, sizeof(float) * (size_t)n * kIn, cudaMemcpyHostToDevice, m->stream));
  mlp_fwd_kernel<<<fwd_grid(m, n), kThreads, sizeof(Weights), m->stream>>>(m->net, c.x, n, c.y);
  MCUDA(m, cudaGetLastError());
  MCUDA(m, cudaMemcpyAsync(y, c.y, sizeof(float) * (size_t)n, cudaMemcpyDeviceToHost, m->stream));
  MCUDA(m, cudaStreamSynchronize(m->stream));
  return REWL_OK;
}

extern "C" rewl_status rewl_mlp_gradient(rewl_mlp* m, const float* x, const float* target, const int32_t* run_offsets,
                                         int n_runs, double* loss, float* grad) {
  rewl_status s = check_mlp(m);
  if (s != REWL_OK) return s;
  if (!x || !target) return mfail(m, REWL_EINVAL, "NULL corpus");
  s = check_segments(run_offsets, n_runs, run_offsets ? run_offsets[n_runs] : 0);
  if (s != REWL_OK) return s;
  Corpus c(m);
  s = upload_corpus(m, c, x, target, run_offsets, n_runs);
  if (s != REWL_OK) return s;
  double* d_loss = nullptr;
  MCUDA(m, c.sc.get(&d_loss, 1));
  s = loss_and_grad(m, c.x, c.t, c.seg, n_runs, run_offsets[n_runs], c.y, c.dy, c.loss, d_loss, nullptr);
  if (s != REWL_OK) return s;
  if (loss) MCUDA(m, cudaMemcpyAsync(loss, d_loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
  if (grad) MCUDA(m, cudaMemcpyAsync(grad, m->d_grad, sizeof(float) * kParams, cudaMemcpyDeviceToHost, m->stream));
  MCUDA(m, cudaStreamSynchronize(m->stream));
  return REWL_OK;
}

extern "C" rewl_status rewl_mlp_train(rewl_mlp* m, const float* x, const float* target, const int32_t* run_offsets,
                                      int n_runs, int steps, float lr, float* loss_history) {
  rewl_status s = check_mlp(m);
  if (s != REWL_OK) return s;
  if (!x || !target || steps < 1 || !(lr > 0.0f)) return mfail(m, REWL_EINVAL, "bad training arguments");
  s = check_segments(run_offsets, n_runs, run_offsets ? run_offsets[n_runs] : 0);
  if (s != REWL_OK) return s;
  const long long n = run_offsets[n_runs];
  Corpus c(m);
  s = upload_corpus(m, c, x, target, run_offsets, n_runs);
  if (s != REWL_OK) return s;
  std::vector<double> loss;
  try {
    if (loss_history) loss.resize((size_t)steps);
  } catch (const std::bad_alloc&) {
    return mfail(m, REWL_ENOMEM, "no host memory for the loss history");
  }
  double* d_loss = nullptr;      // loss before each step
  if (loss_history) MCUDA(m, c.sc.get(&d_loss, (size_t)steps));
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  for (int it = 0; it < steps; ++it) {
    const long long step = m->adam_t + 1;
    AdamArgs a{};
    a.lr = lr;
    a.b1 = b1;
    a.b2 = b2;
    a.eps = eps;
    a.c1 = 1.0f - std::pow(b1, (float)step);
    a.c2 = 1.0f - std::pow(b2, (float)step);
    s = loss_and_grad(m, c.x, c.t, c.seg, n_runs, n, c.y, c.dy, c.loss, d_loss ? d_loss + it : nullptr, &a);
    if (s != REWL_OK) return s;
    m->adam_t = step;
  }
  if (loss_history) {
    MCUDA(m, cudaMemcpyAsync(loss.data(), d_loss, sizeof(double) * (size_t)steps, cudaMemcpyDeviceToHost, m->stream));
    MCUDA(m, cudaStreamSynchronize(m->stream));
    for (int it = 0; it < steps; ++it) loss_history[it] = (float)loss[it];
  }
  MCUDA(m, cudaStreamSynchronize(m->stream));
  return REWL_OK;
}

extern "C" rewl_status rewl_mlp_features(const rewl_handle* h, const double* lng, float* x_out, float* t_out) {
  if (!h || !x_out) return mfail(nullptr, REWL_EINVAL, "NULL argument");
  if (t_out && !lng) return mfail(nullptr, REWL_EINVAL, "targets need ln g");
  JobView v;
  job_view(h, &v);
  if (v.kind != REWL_LATTICE_BCC) return mfail(nullptr, REWL_EINVAL, "features are defined for bcc jobs");
  double Jsh[4] = {0, 0, 0, 0}, e_min = 0, dE = 0;
  job_couplings(h, Jsh, &e_min, &dE);
  const int B = job_bins(h);
  for (int b = 0; b < B; ++b) {
    const double e = (e_min + (b + 0.5) * dE) / (double)v.N;
    float* r = x_out + (size_t)b * kIn;
    r[0] = (float)e;
    r[1] = (float)(1.0 / (double)v.L);
    for (int s = 0; s < 4; ++s) r[2 + s] = (float)Jsh[s];
    if (t_out) t_out[b] = (float)(lng[b] / (double)v.N);
  }
  return REWL_OK;
}

extern "C" rewl_status rewl_mlp_warm_start(rewl_mlp* m, rewl_handle* h, double lnf0, double* lng_out) {
  rewl_status s = check_mlp(m);
  if (s != REWL_OK) return s;
  if (!h || !(lnf0 > 0.0)) return mfail(m, REWL_EINVAL, "bad warm-start arguments");
  const int B = job_bins(h);
  JobView v;
  job_view(h, &v);
  std::vector<float> x((size_t)B * kIn), y(B);
  s = rewl_mlp_features(h, nullptr, x.data(), nullptr);
  if (s != REWL_OK) return s;
  s = rewl_mlp_forward(m, x.data(), B, y.data());
  if (s != REWL_OK) return s;
  std::vector<double> lng(B);
  for (int b = 0; b < B; ++b) lng[b] = (double)y[b] * (double)v.N;
  if (lng_out) std::copy(lng.begin(), lng.end(), lng_out);
  s = rewl_set_initial_lng(h, lng.data(), lnf0);
  if (s != REWL_OK) return mfail(m, s, std::string("set_initial_lng: ") + rewl_last_error(h));
  return REWL_OK;
}

extern "C" void rewl_mlp_destroy(rewl_mlp* m) {
  if (!m) return;
  if (!m->broken) cudaStreamSynchronize(m->stream);
  for (void* p : m->allocations) cudaFree(p);   // (waits for the device)
  cudaFree(m->d_chunk);
  pool_release();
  delete m;
}

// lsas_dn.cu -- learned refinement of the LS channel estimate (Sec. II-C's
// LS is the input, the fallback and the yardstick).
//
// Per antenna row of N subcarriers: normalise H_LS by its RMS, run a residual
// 1-D convolutional network over subcarriers (2 -> 32 -> 32 -> 32 -> 2
// channels, kernel 5, ReLU, output added to the input), denormalise.  The
// same kernels train it: forward with stored ReLU outputs, mean squared
// error against the normalised true channel, backward (data gradients as
// forward convolutions with transposed, flipped weights and ReLU masks;
// weight gradients as fixed-order block reductions) and Adam.  Inference can
// read bf16 weights; every sum is fp32.
//
// Layouts: activations [R][C][N] float; parameters one float vector
// W1[32][2][5] b1[32] W2[32][32][5] b2[32] W3[32][32][5] b3[32] W4[2][32][5]
// b4[2] (10978 values).
#include <cuda_bf16.h>

#include "lsas.h"
#include "lsas_kernels.cuh"

namespace lsas {

constexpr int kDnK = 5;
constexpr int kDnPos = 128;   // subcarriers per block of the conv kernels
constexpr int kDnParams = 10978;
constexpr int kOffW1 = 0, kOffB1 = 320, kOffW2 = 352, kOffB2 = 5472, kOffW3 = 5504,
              kOffB3 = 10624, kOffW4 = 10656, kOffB4 = 10976;

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }

// FP32 network: the two 32 -> 32 layers on the tensor cores in split precision,
// the rest on the CUDA cores.  Activations are stored after their ReLU
// (r > 0 is the backward's mask), [R][C][N]; every kernel works on tiles of
// kDnPos positions of one row.
//
// Weights as the kernels read them (dn_setup_kernel), so that the outputs a
// thread keeps lie next to each other: forward layers 1 to 3 [in][k][out],
// layer 4 [in][out][k]; data gradients W'[out][in][k] = W[in][out][4 - k] of
// layers 4, 3 and 2 as forward convolutions, [in][k][out].
constexpr int kFw1 = 0, kFw2 = kFw1 + 320, kFw3 = kFw2 + 5120, kFw4 = kFw3 + 5120;
constexpr int kBw4 = kFw4 + 320, kBw3 = kBw4 + 320, kBw2 = kBw3 + 5120;
constexpr int kBias = kBw2 + 5120, kWtFloats = kBias + 100;   // b1, b2, b3, b4 (two, two unused)

template <typename WT>
__device__ __forceinline__ void fp32_weights(const WT* __restrict__ P, float* __restrict__ wt,
                                             int first, int step) {
  for (int e = first; e < kWtFloats; e += step) {
    int src;
    if (e < kFw2) {                                  // [j][k][o]
      src = kOffW1 + ((e % 32) * 2 + e / 160) * kDnK + (e / 32) % kDnK;
    } else if (e < kFw4) {                           // [c][k][o]
      const int f = (e - kFw2) % 5120;
      src = (e < kFw3 ? kOffW2 : kOffW3) + ((f % 32) * 32 + f / 160) * kDnK + (f / 32) % kDnK;
    } else if (e < kBw4) {                           // [c][j][k]
      const int f = e - kFw4;
      src = kOffW4 + (((f / kDnK) % 2) * 32 + f / 10) * kDnK + f % kDnK;
    } else if (e < kBw3) {                           // [j][k][c]
      const int f = e - kBw4;
      src = kOffW4 + ((f / 160) * 32 + f % 32) * kDnK + 4 - (f / 32) % kDnK;
    } else if (e < kBias) {                          // [o][k][c]
      const int f = (e - kBw3) % 5120;
      src = (e < kBw2 ? kOffW3 : kOffW2) + ((f / 160) * 32 + f % 32) * kDnK + 4 - (f / 32) % kDnK;
    } else {
      const int f = e - kBias, l = f / 32;
      src = (l == 0 ? kOffB1 : l == 1 ? kOffB2 : l == 2 ? kOffB3 : kOffB4) + (f % 32) % (l < 3 ? 32 : 2);
    }
    wt[e] = to_f(P[src]);
  }
}

// positions q - 2 .. q + 5 of a row (q a multiple of 4), zero outside [0, N)
__device__ __forceinline__ void window8(const float* __restrict__ row, int q, int N, float (&w)[8]) {
  const float4 c = *reinterpret_cast<const float4*>(row + q);
  const float2 a = q > 0 ? *reinterpret_cast<const float2*>(row + q - 2) : make_float2(0.f, 0.f);
  const float2 d = q + 4 < N ? *reinterpret_cast<const float2*>(row + q + 4) : make_float2(0.f, 0.f);
  w[0] = a.x; w[1] = a.y;
  w[2] = c.x; w[3] = c.y; w[4] = c.z; w[5] = c.w;
  w[6] = d.x; w[7] = d.y;
}

__device__ __forceinline__ void cp_async(uint32_t dst, const void* src, bool on, int bytes) {
  // bytes is 4 or 8; zero-fills when off
  if (bytes == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(on ? 4 : 0)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(on ? 8 : 0)
                 : "memory");
}

__device__ __forceinline__ float4 relu4(float4 v) {
  return make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
}
// v where m > 0, else 0
__device__ __forceinline__ float4 mask4(float4 v, float4 m) {
  return make_float4(m.x > 0.f ? v.x : 0.f, m.y > 0.f ? v.y : 0.f, m.z > 0.f ? v.z : 0.f,
                     m.w > 0.f ? v.w : 0.f);
}

// 2 -> 32 channels: layer 1 (bias and ReLU) or the data gradient of layer 4
// (masked by the stored layer output).  Bound by writing the 32 channels: a
// warp takes four of them and a lane four positions, inputs and outputs in
// 16-byte pieces.  256 rows of 1024: 9 us against 19.6 us for one position a
// thread with scalar shared-memory operands.
template <bool BWD>
__global__ void __launch_bounds__(256) dn_conv_in_kernel(const float* __restrict__ in,
                                                         const float* __restrict__ wt,
                                                         const float* __restrict__ bias,
                                                         const float* __restrict__ mask,
                                                         float* __restrict__ out, int N) {
  pdl_wait();
  __shared__ __align__(16) float ws[320];
  const int tiles_row = N / kDnPos;
  const int r = blockIdx.x / tiles_row;
  const int lane = threadIdx.x & 31, ch = (threadIdx.x >> 5) * 4;
  const int q = (blockIdx.x % tiles_row) * kDnPos + 4 * lane;
  for (int i = threadIdx.x; i < 320; i += 256) ws[i] = wt[i];
  float w[2][8];
  window8(in + static_cast<size_t>(r) * 2 * N, q, N, w[0]);
  window8(in + (static_cast<size_t>(r) * 2 + 1) * N, q, N, w[1]);
  float acc[4][4];   // [channel][position]
#pragma unroll
  for (int o = 0; o < 4; ++o)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[o][i] = BWD ? 0.f : bias[ch + o];
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int k = 0; k < kDnK; ++k) {
      const float4 v = *reinterpret_cast<const float4*>(ws + (j * kDnK + k) * 32 + ch);
      const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[o][i] = fmaf(vv[o], w[j][i + k], acc[o][i]);
    }
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    const size_t at = (static_cast<size_t>(r) * 32 + ch + o) * N + q;
    float4 v = make_float4(acc[o][0], acc[o][1], acc[o][2], acc[o][3]);
    v = BWD ? mask4(v, *reinterpret_cast<const float4*>(mask + at)) : relu4(v);
    *reinterpret_cast<float4*>(out + at) = v;
  }
}

// 32 -> 32 channels in FP32 on tcgen05: layers 2 and 3 (bias and ReLU) or their
// data gradients (masked).  The FMA pipe would need 33 us for 256 rows of 1024
// (5120 FMAs a position), so the products go to the tensor cores.  Their FP32
// additions truncate: a sum of plain bf16 terms is always too small, and weight
// gradients, which add many outputs, keep that (1.2 times their error).  So the
// leading terms are small integers: x0 is the value rounded to a grid 2^-8 of
// the power of two above the largest of its position's 32 channels (at most 256
// steps, exact in bf16), w0 likewise with the 32 weights of an output and tap.
// A tap's 32 products x0 w0 are then multiples of one step, at most 2^21 of
// them, and their sum is exact in any order.  The remainder is exact too and
// goes into three more bf16 terms, nearest even, which hold all of it.  Products
// of terms are exact in FP32; those beside x0 w0 share three sums by order (x0
// w1 + x1 w0; x0 w2 + x1 w1 + x2 w0; the four of the third), 2^-8 of the largest
// product and less, where truncation does not count; the rest is below 2^-34 of
// it.  Channels are scaled by powers of two so that each one's largest weight is
// 1 to 2, which keeps a channel of small values and large weights as exact as
// the others.  The CUDA cores add the taps' and the small sums, rounding to
// nearest.  Relative error (norm) against 64 bits, geometric means over 80 sets
// of 8 x 128 to 500 x 512 and 256 x 1024 rows: output 0.87 and gradients 0.67 of
// the same layers as FMAs (tests/test_gpu_split_conv_rounding.py).
//
// Layout: positions as rows 16 bytes (eight channels) apart, so that the
// operand of tap k is the same buffer k rows on; the weights' terms one after
// the other as N, so that x0 meets w1, w2 and w3 in one MMA of N = 96.  A block
// fetches the next tile under a tile's MMAs; two blocks an SM fill each
// other's gaps.  A tile with a scaled value outside 2^-100 .. 2^60 (but zero),
// whose last term may be no normal number or whose products may overflow on the
// way, and, after a wait that gave up, every further tile is summed by FMAs
// (cv_fma_tile).  Bound by
// the 50 MMAs of a tile (4 KB of shared memory each whatever their N; tensor
// pipe 55 to 60 % busy) and the splitting between them.  256 rows of 1024: 36
// us, 36 masked (10 and 15 to read and write HBM), against 51 us for packed FMAs
// from registers (8 outputs x 4 positions a thread) and 27 with three plain
// bf16 terms, whose sums shrink by 1.6e-8.
constexpr int kCvRows = kDnPos + kDnK - 1;           // row j holds position q0 - 2 + j
constexpr int kCvLbo = kCvRows * 16;                 // bytes between channel chunks
constexpr int kCvPlane = 4 * kCvLbo;                 // one term of a tile's input
constexpr int kCvTerms = 4;
constexpr int kCvTap = kCvTerms * 32 * 64;           // one tap's weights: four terms x 32 outputs
constexpr int kCvX = kDnK * kCvTap;
constexpr int kCvMax = kCvX + kCvTerms * kCvPlane;   // [2][128]: largest of half a position's channels
constexpr int kCvScale = kCvMax + 2 * kDnPos * 4;    // [32]: a channel's power of two
constexpr int kCvBar = kCvScale + 32 * 4;
constexpr int kCvSmem = kCvBar + 16;
constexpr int kCvThreads = 256;
constexpr int kCvSmall = 32 * kDnK, kCvCols = 256;   // TMEM: a sum per tap, then three of small products
static_assert(kCvX % 16 == 0 && kCvBar % 16 == 0, "16-byte operand alignment");

// Whether a value is outside the range of the split: zero, and 2^-100 (whose
// last term is a normal bf16 still) up to 2^60 (whose products' sums stay finite).
__device__ __forceinline__ bool cv_off(float x) {
  constexpr uint32_t kLo = (127u - 100u) << 23, kHi = (127u + 60u) << 23;
  const uint32_t u = __float_as_uint(x) & 0x7fffffffu;
  return u - kLo >= kHi - kLo && u != 0;
}
// The number whose addition and subtraction round a value to the grid of a
// group with this largest magnitude: 1.5 * 2^16 times its power of two, so that
// one unit in the last place of the sum is 2^-7 of that power.
__device__ __forceinline__ float cv_grid(float most) {
  return 1.5f * __uint_as_float((__float_as_uint(most) & 0x7f800000u) + (16u << 23));
}
// Eight values as four bf16 terms each whose sum is the value: the multiple of
// the grid, then the remainder's three (nearest even; every remainder is exact).
__device__ __forceinline__ void cv_split8(const float (&x)[8], float grid, uint4 (&out)[kCvTerms]) {
  uint32_t w[kCvTerms][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float a = x[2 * i], b = x[2 * i + 1];
#pragma unroll
    for (int s = 0; s < kCvTerms; ++s) {
      const __nv_bfloat162 h =
          s == 0 ? __floats2bfloat162_rn(__fsub_rn(__fadd_rn(a, grid), grid), __fsub_rn(__fadd_rn(b, grid), grid))
                 : __floats2bfloat162_rn(a, b);
      w[s][i] = *reinterpret_cast<const uint32_t*>(&h);
      a -= __low2float(h);
      b -= __high2float(h);
    }
  }
#pragma unroll
  for (int s = 0; s < kCvTerms; ++s) out[s] = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

// A tile's sums as FMAs, for values that the split does not take: the inputs
// through `raw` ([32][kCvRows], the place of their terms), a warp four outputs
// and a lane four positions.  A layer of 256 rows of 1024 whose tiles all go
// this way takes 90 us, against 305 with every warp reading its operands of each
// FMA from memory; the main path's launches take 1 to 2 us more beside it.
template <bool BWD>
__device__ __noinline__ void cv_fma_tile(const float* __restrict__ in, const float* __restrict__ wt,
                                         const float* __restrict__ bias, const float* __restrict__ mask,
                                         float* __restrict__ out, int r, int q0, int N, float* raw) {
  const int lane = threadIdx.x & 31, o0 = 4 * (threadIdx.x >> 5);
  const float* row = in + static_cast<size_t>(r) * 32 * N;
#pragma unroll 4
  for (int i = threadIdx.x; i < 32 * kCvRows; i += kCvThreads) {
    const int c = i / kCvRows, q = q0 - 2 + i % kCvRows;
    raw[i] = q >= 0 && q < N ? row[static_cast<size_t>(c) * N + q] : 0.f;
  }
  __syncthreads();
  float acc[4][4];   // [output][position]
#pragma unroll
  for (int o = 0; o < 4; ++o)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[o][i] = BWD ? 0.f : bias[o0 + o];
#pragma unroll 2
  for (int c = 0; c < 32; ++c) {
    const float4 lo = *reinterpret_cast<const float4*>(raw + c * kCvRows + 4 * lane);
    const float4 hi = *reinterpret_cast<const float4*>(raw + c * kCvRows + 4 * lane + 4);
    const float x[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
    for (int k = 0; k < kDnK; ++k) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(wt + (c * kDnK + k) * 32 + o0));
      const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[o][i] = fmaf(w[o], x[i + k], acc[o][i]);
    }
  }
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    const size_t at = (static_cast<size_t>(r) * 32 + o0 + o) * N + q0 + 4 * lane;
    const float4 v = make_float4(acc[o][0], acc[o][1], acc[o][2], acc[o][3]);
    *reinterpret_cast<float4*>(out + at) = BWD ? mask4(v, *reinterpret_cast<const float4*>(mask + at)) : relu4(v);
  }
  __syncthreads();   // read before the next tile's terms
}

template <bool BWD>
__global__ void __launch_bounds__(kCvThreads, 2) dn_conv32_kernel(const float* __restrict__ in,
                                                                  const float* __restrict__ wt,
                                                                  const float* __restrict__ bias,
                                                                  const float* __restrict__ mask,
                                                                  float* __restrict__ out, int R, int N) {
  pdl_wait();
  extern __shared__ __align__(128) unsigned char smem[];
  float* most = reinterpret_cast<float*>(smem + kCvMax);
  float* scale = reinterpret_cast<float*>(smem + kCvScale);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + kCvBar);
  uint32_t* tbase = reinterpret_cast<uint32_t*>(bar + 1);
  const int tiles_row = N / kDnPos, tiles = R * tiles_row;
  const int t = threadIdx.x, u = t & 127, half = t >> 7;
  const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);
  if (t == 0) {
    mbar_init(smem_u32(bar), 1);
    fence_mbar_init();
  }
  __syncwarp();
  if (warp == 0) tmem_alloc(smem_u32(tbase), kCvCols);
  // a thread's inputs of a tile, fetched one tile ahead: buffer row u of
  // channel chunks 2 half and 2 half + 1, and, threads 0 to 15, chunk t / 4 of
  // row 128 + t % 4
  float xa[2][8], xb[8];
  auto fetch = [&](int tile) {
    if (tile >= tiles) return;
    const int r = tile / tiles_row, q0 = (tile % tiles_row) * kDnPos;
    const float* row = in + static_cast<size_t>(r) * 32 * N;
    const int qa = q0 - 2 + u, qb = q0 + 126 + (t & 3);
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int i = 0; i < 8; ++i)
        xa[j][i] = qa >= 0 ? row[static_cast<size_t>((2 * half + j) * 8 + i) * N + qa] : 0.f;
    if (t < 16) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        xb[i] = qb < N ? row[static_cast<size_t>((t >> 2) * 8 + i) * N + qb] : 0.f;
    }
  };
  fetch(blockIdx.x);
  // the weights, a thread a tap k and output o
  bool off = false;
  float w[4][8];
  if (t < 32) reinterpret_cast<uint32_t*>(scale)[t] = 0u;
  __syncthreads();
  if (t < kDnK * 32) {
    const int k = t / 32, o = t % 32;
#pragma unroll
    for (int c = 0; c < 32; ++c) w[c / 8][c % 8] = wt[(c * kDnK + k) * 32 + o];
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      const uint32_t big =
          __reduce_max_sync(0xffffffffu, __float_as_uint(w[c / 8][c % 8]) & 0x7fffffffu);
      if (o == 0) atomicMax(reinterpret_cast<uint32_t*>(scale) + c, big);
    }
  }
  __syncthreads();
  // a channel's largest weight becomes 1 to 2, its inputs are scaled inversely
  if (t < 32) {
    const float big = scale[t];
    off |= cv_off(big);
    scale[t] = big > 0.f ? __uint_as_float(__float_as_uint(big) & 0x7f800000u) : 1.f;
  }
  __syncthreads();
  // the weights' terms: rows o, 32 + o, 64 + o, 96 + o
  if (t < kDnK * 32) {
    const int k = t / 32, o = t % 32;
    float big = 0.f;
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      float& v = w[c / 8][c % 8];
      v *= __uint_as_float((254u << 23) - __float_as_uint(scale[c]));   // its inverse
      off |= cv_off(v);
      big = fmaxf(big, fabsf(v));
    }
    const float grid = cv_grid(big);
    uint4 s[kCvTerms];
#pragma unroll
    for (int kc = 0; kc < 4; ++kc) {
      cv_split8(w[kc], grid, s);
#pragma unroll
      for (int p = 0; p < kCvTerms; ++p)
        *reinterpret_cast<uint4*>(smem + k * kCvTap + (4 * p + (o >> 3)) * 512 + kc * 128 + (o & 7) * 16) = s[p];
    }
  }
  tmem_fence_before();
  bool plain = __syncthreads_or(off);   // this block's tiles on the CUDA cores
  tmem_fence_after();
  const uint32_t tmm = *tbase;
  const uint32_t tm = tmm + (static_cast<uint32_t>(32 * (warp & 3)) << 16) + 16 * half;
  const uint64_t dx = umma_desc(smem_u32(smem + kCvX), kCvLbo, 128);
  const uint64_t dw = umma_desc(smem_u32(smem), 128, 512);
  bool ok = true;
  uint32_t phase = 0;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int r = tile / tiles_row, q0 = (tile % tiles_row) * kDnPos;
    const size_t at0 = (static_cast<size_t>(r) * 32 + 16 * half) * N + q0 + u;   // output 16 half
    off = !ok;
    // the largest of the position's channels: this thread's sixteen, the other
    // half's from the warp that holds them
    float big = 0.f;
    auto scaled = [&](float (&x)[8], int chunk) {
      const float4 lo = *reinterpret_cast<const float4*>(scale + 8 * chunk);
      const float4 hi = *reinterpret_cast<const float4*>(scale + 8 * chunk + 4);
      const float f[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        x[i] *= f[i];
        off |= cv_off(x[i]);
        big = fmaxf(big, fabsf(x[i]));
      }
    };
    scaled(xa[0], 2 * half);
    scaled(xa[1], 2 * half + 1);
    most[half * kDnPos + u] = big;
    named_sync(1 + (warp & 3), 64);
    float grid = cv_grid(fmaxf(big, most[(half ^ 1) * kDnPos + u]));
    unsigned char* xs = smem + kCvX;
    uint4 s[kCvTerms];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      cv_split8(xa[j], grid, s);
#pragma unroll
      for (int p = 0; p < kCvTerms; ++p)
        *reinterpret_cast<uint4*>(xs + p * kCvPlane + (2 * half + j) * kCvLbo + u * 16) = s[p];
    }
    if (t < 16) {
      big = 0.f;
      scaled(xb, t >> 2);
      big = fmaxf(big, __shfl_xor_sync(0xffffu, big, 4));
      grid = cv_grid(fmaxf(big, __shfl_xor_sync(0xffffu, big, 8)));
      cv_split8(xb, grid, s);
#pragma unroll
      for (int p = 0; p < kCvTerms; ++p)
        *reinterpret_cast<uint4*>(xs + p * kCvPlane + (t >> 2) * kCvLbo + (128 + (t & 3)) * 16) = s[p];
    }
    fence_proxy_async();
    tmem_fence_before();
    const bool cores = __syncthreads_or(off || plain);
    tmem_fence_after();
    if (t == 0 && !cores) {
#pragma unroll
      for (int k = 0; k < kDnK; ++k)
#pragma unroll
        for (int kh = 0; kh < 2; ++kh) {
          const uint64_t a = dx + ((k * 16 + kh * 2 * kCvLbo) >> 4);
          const uint64_t b = dw + ((k * kCvTap + kh * 256) >> 4);
          const uint32_t more = k + kh > 0 ? 1u : 0u;
          umma_f16(tmm + 32 * k, a, b, umma_idesc(32, true), kh);
          umma_f16(tmm + kCvSmall, a, b + (4 * 512 >> 4), umma_idesc(96, true), more);
          umma_f16(tmm + kCvSmall, a + (kCvPlane >> 4), b, umma_idesc(96, true), 1u);
          umma_f16(tmm + kCvSmall + 32, a + (2 * kCvPlane >> 4), b, umma_idesc(64, true), 1u);
          umma_f16(tmm + kCvSmall + 64, a + (3 * kCvPlane >> 4), b, umma_idesc(32, true), 1u);
        }
      umma_commit(smem_u32(bar));
    }
    fetch(tile + gridDim.x);
    float m[16];
    if (BWD) {
#pragma unroll
      for (int o = 0; o < 16; ++o) m[o] = mask[at0 + static_cast<size_t>(o) * N];
    }
    float y[16];
    if (!cores) {
      ok = __all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(bar), phase));
      phase ^= 1;
    }
    if (!cores && ok) {
      tmem_fence_after();
      float a[16], b[16];
      // the small sums first, then the taps
      Tmem<16>::ld(tm + kCvSmall, y);
      Tmem<16>::ld(tm + kCvSmall + 32, a);
      Tmem<16>::ld(tm + kCvSmall + 64, b);
      tmem_wait_ld();
#pragma unroll
      for (int o = 0; o < 16; ++o) y[o] += a[o] + b[o];
      Tmem<16>::ld(tm, a);
      Tmem<16>::ld(tm + 32, b);
      tmem_wait_ld();
#pragma unroll
      for (int o = 0; o < 16; ++o) y[o] += a[o] + b[o];
      Tmem<16>::ld(tm + 64, a);
      Tmem<16>::ld(tm + 96, b);
      tmem_wait_ld();
#pragma unroll
      for (int o = 0; o < 16; ++o) y[o] += a[o] + b[o];
      Tmem<16>::ld(tm + 128, a);
      tmem_wait_ld();
#pragma unroll
      for (int o = 0; o < 16; ++o) y[o] += BWD ? a[o] : a[o] + bias[16 * half + o];
    } else if (cores) {
      cv_fma_tile<BWD>(in, wt, bias, mask, out, r, q0, N, reinterpret_cast<float*>(xs));
      continue;
    } else {
      // the wait gave up: the same sums as FMAs, in the warps that saw it
#pragma unroll
      for (int o = 0; o < 16; ++o) y[o] = BWD ? 0.f : bias[16 * half + o];
#pragma unroll 1
      for (int ck = 0; ck < 32 * kDnK; ++ck) {
        const int q = q0 + u + ck % kDnK - 2;
        const float x = q >= 0 && q < N ? in[(static_cast<size_t>(r) * 32 + ck / kDnK) * N + q] : 0.f;
#pragma unroll
        for (int o = 0; o < 16; ++o) y[o] = fmaf(wt[ck * 32 + 16 * half + o], x, y[o]);
      }
    }
#pragma unroll
    for (int o = 0; o < 16; ++o)
      out[at0 + static_cast<size_t>(o) * N] = BWD ? (m[o] > 0.f ? y[o] : 0.f) : fmaxf(y[o], 0.f);
  }
  // a wait that gave up: its products get a second bounded chance to finish
  if (!ok) (void)mbar_wait_bounded(smem_u32(bar), phase ^ 1);
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  if (warp == 0) tmem_dealloc(tmm, kCvCols);
}
template <bool BWD>
static cudaError_t conv32(const float* in, const float* wt, const float* bias, const float* mask,
                          float* out, int R, int N, int sms, cudaStream_t st) {
  const cudaError_t e = cudaFuncSetAttribute(dn_conv32_kernel<BWD>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, kCvSmem);
  if (e != cudaSuccess) return e;
  const int tiles = R * (N / kDnPos);
  pdl_launch(dn_conv32_kernel<BWD>, dim3(tiles < 2 * sms ? tiles : 2 * sms), kCvThreads, kCvSmem, st, in,
             wt, bias, mask, out, R, N);
  return cudaSuccess;
}

// 32 -> 2 channels (layer 4) with the network's output: y = x0 + conv, then
// TRAIN: dy = 2 (y - t) / n and the tile's sum of (y - t)^2, else
// Hout = (y[0] + j y[1]) rms.  Bound by reading the 32 channels: a warp takes
// four of them and a lane four positions; the eight warps' sums meet in shared
// memory, added in warp order.  256 rows of 1024: 11 us; before, 23 us and
// a launch of 6 us for the loss.
struct DnOutArgs {
  const float* in;     // r3 [R][32][N]
  const float* wt;     // [c][j][k]
  const float* bias;   // two
  const float* x0;     // [R][2][N]
  const float* tt;     // TRAIN: [R][2][N]
  float* dy;           // TRAIN: [R][2][N]
  float* part;         // TRAIN: one per tile
  float inv_n;         // TRAIN: 2 / n
  const float* rms;    // else
  float2* Hout;        // else
  int N;
};
template <bool TRAIN>
__global__ void __launch_bounds__(256) dn_conv_out_kernel(const DnOutArgs a) {
  pdl_wait();
  __shared__ float ws[320];
  __shared__ __align__(16) float red[8][2][kDnPos];
  __shared__ float se[8];
  const int N = a.N, tiles_row = N / kDnPos;
  const int r = blockIdx.x / tiles_row, q0 = (blockIdx.x % tiles_row) * kDnPos;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int i = t; i < 320; i += 256) ws[i] = a.wt[i];
  __syncthreads();
  float acc[2][4];
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[j][i] = 0.f;
#pragma unroll
  for (int cc = 0; cc < 4; ++cc) {
    const int c = 4 * warp + cc;
    float w[8];
    window8(a.in + (static_cast<size_t>(r) * 32 + c) * N, q0 + 4 * lane, N, w);
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int k = 0; k < kDnK; ++k) {
        const float v = ws[c * 10 + j * kDnK + k];
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[j][i] = fmaf(v, w[i + k], acc[j][i]);
      }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j)
    *reinterpret_cast<float4*>(&red[warp][j][4 * lane]) =
        make_float4(acc[j][0], acc[j][1], acc[j][2], acc[j][3]);
  __syncthreads();
  const int j = t >> 7, p = t & 127;
  float y = a.bias[j];
#pragma unroll
  for (int w = 0; w < 8; ++w) y += red[w][j][p];
  const size_t at = (static_cast<size_t>(r) * 2 + j) * N + q0 + p;
  y += a.x0[at];
  if (TRAIN) {
    const float d = y - a.tt[at];
    a.dy[at] = d * a.inv_n;
    float e = d * d;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) e += __shfl_xor_sync(0xffffffffu, e, off);
    if (lane == 0) se[warp] = e;
    __syncthreads();
    if (t == 0) {
      float sum = se[0];
#pragma unroll
      for (int w = 1; w < 8; ++w) sum += se[w];
      a.part[blockIdx.x] = sum;
    }
  } else {
    reinterpret_cast<float*>(a.Hout)[2 * (static_cast<size_t>(r) * N + q0 + p) + j] = y * a.rms[r];
  }
}

// Weight gradient of a 32 -> 32 layer, FP32: dW[o][c][k] = sum_p G[o][p]
// A[c][p + k - 2] and db[o] = sum_p G[o][p], as a product with the positions
// as the inner dimension.  Bound by the FMA pipe (5120 FMAs a position).  A
// tile's G and A rows come to shared memory by asynchronous copies, one tile
// ahead, G with the values of two outputs side by side (4-byte copies: the
// copies' 16-byte pieces would need a transpose); a thread keeps 2 output pairs
// x 2 inputs x 5 taps and takes the tile four positions at a time: six 16-byte
// loads (A slides in registers, each value in both halves of a pair) for 160
// FMAs, issued as 80 packed ones.  The two halves of a block take the tile's
// halves.  Blocks walk the tiles (two blocks fit on an SM) and write one row of
// partial sums each.  256 rows of 1024: 53 us a layer, FMA pipe 67 % busy
// (scalar FMAs: 58, issue 75 %; packed over even and odd positions, whose
// operand pairs share no register from one to the next: 71; on the tensor cores
// with operands split as above, their sums read out every 32 positions for
// FP32 accuracy: 117); one block per (o, c) that re-read both tensors took
// about 1900 us.
constexpr int kFwThreads = 256;
constexpr int kFwRow = kDnPos + 4;                     // floats of a row of A; rows 4 banks apart
constexpr int kFwGRow = 2 * kDnPos + 4;                // of two rows of G, output pairs side by side
constexpr int kFwG = 16 * kFwGRow * 4;                 // bytes of G, then A
constexpr int kFwStage = kFwG + 32 * kFwRow * 4;
constexpr int kFwSmem = 2 * kFwStage;
constexpr int kWgPart = 5 * 32 * 32 + 32;              // one block's partials (floats)
static_assert(kFwSmem >= 128 * 40 * 4, "the halves meet in the stages");

__global__ void __launch_bounds__(kFwThreads, 2) dn_wgrad32_kernel(const float* __restrict__ G,
                                                                   const float* __restrict__ A, int R,
                                                                   int N, float* __restrict__ part) {
  pdl_wait();
  extern __shared__ __align__(128) unsigned char smem[];
  const int t = threadIdx.x, lane = t & 31;
  const int half = t >> 7, u = t & 127;
  const int og = u & 7, cg = u >> 3;                   // o = 2 (og + 8 i) + {0, 1}, c = cg + 16 j
  const int tiles_row = N / kDnPos, tiles = R * tiles_row;
  auto fetch = [&](int tile, int b) {
    if (tile < tiles) {
      const int r = tile / tiles_row, q0 = (tile % tiles_row) * kDnPos;
      const uint32_t g = smem_u32(smem + b * kFwStage), x = g + kFwG;
#pragma unroll 4
      for (int i = t; i < 32 * kDnPos; i += kFwThreads) {
        const int o = i / kDnPos, p = i % kDnPos;
        cp_async(g + ((o >> 1) * kFwGRow + 2 * p + (o & 1)) * 4,
                 G + (static_cast<size_t>(r) * 32 + o) * N + q0 + p, true, 4);
      }
      constexpr int kHalf = (kDnPos + 4) / 2;
      for (int i = t; i < 32 * kHalf; i += kFwThreads) {
        const int c = i / kHalf, jj = 2 * (i % kHalf), p = q0 + jj - 2;
        const bool on = p >= 0 && p < N;
        cp_async(x + (c * kFwRow + jj) * 4, A + (static_cast<size_t>(r) * 32 + c) * N + (on ? p : 0), on, 8);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float2 acc[2][2][kDnK];   // [output pair][input][tap]
  float2 bacc = make_float2(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int k = 0; k < kDnK; ++k) acc[i][j][k] = make_float2(0.f, 0.f);
  fetch(blockIdx.x, 0);
  int b = 0;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, b ^= 1) {
    fetch(tile + gridDim.x, b ^ 1);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const float* g = reinterpret_cast<const float*>(smem + b * kFwStage);
    const float* x = g + kFwG / 4;
    {   // bias: sixteen threads an output pair, 8 positions each
      const float4* gb = reinterpret_cast<const float4*>(g + (t >> 4) * kFwGRow) + (t & 15);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 v = gb[16 * i];
        bacc = __fadd2_rn(bacc, __fadd2_rn(make_float2(v.x, v.y), make_float2(v.z, v.w)));
      }
    }
    const float* gt = g + og * kFwGRow + 128 * half;
    const float* xt = x + cg * kFwRow + 64 * half;
    float2 lo[2][4];   // {x, x} of the window's first four positions
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float4 v = *reinterpret_cast<const float4*>(xt + 16 * j * kFwRow);
      lo[j][0] = make_float2(v.x, v.x);
      lo[j][1] = make_float2(v.y, v.y);
      lo[j][2] = make_float2(v.z, v.z);
      lo[j][3] = make_float2(v.w, v.w);
    }
#pragma unroll 2
    for (int p = 0; p < 64; p += 4) {
      float2 gv[2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 v = *reinterpret_cast<const float4*>(gt + 8 * i * kFwGRow + 2 * p + 4 * h);
          gv[i][2 * h] = make_float2(v.x, v.y);
          gv[i][2 * h + 1] = make_float2(v.z, v.w);
        }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float4 hi = *reinterpret_cast<const float4*>(xt + 16 * j * kFwRow + p + 4);
        const float2 w[8] = {lo[j][0], lo[j][1], lo[j][2], lo[j][3],
                             make_float2(hi.x, hi.x), make_float2(hi.y, hi.y),
                             make_float2(hi.z, hi.z), make_float2(hi.w, hi.w)};
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int k = 0; k < kDnK; ++k)
#pragma unroll
            for (int i = 0; i < 2; ++i) acc[i][j][k] = __ffma2_rn(gv[i][q], w[k + q], acc[i][j][k]);
#pragma unroll
        for (int q = 0; q < 4; ++q) lo[j][q] = w[4 + q];
      }
    }
    __syncthreads();   // the stage is consumed before the next copies into it
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // the halves' sums meet, the first half writes
  float* out = part + static_cast<size_t>(blockIdx.x) * kWgPart;
  float* comb = reinterpret_cast<float*>(smem);
  float2* comb2 = reinterpret_cast<float2*>(comb);
  if (half == 1) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int k = 0; k < kDnK; ++k)
          comb2[((i * 2 + j) * kDnK + k) * 128 + u] = acc[i][j][k];
  }
  __syncthreads();
  if (half == 0) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int k = 0; k < kDnK; ++k)
          *reinterpret_cast<float2*>(out + (k * 32 + cg + 16 * j) * 32 + 2 * (og + 8 * i)) =
              __fadd2_rn(acc[i][j][k], comb2[((i * 2 + j) * kDnK + k) * 128 + u]);
  }
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) {
    bacc.x += __shfl_xor_sync(0xffffffffu, bacc.x, off);
    bacc.y += __shfl_xor_sync(0xffffffffu, bacc.y, off);
  }
  if ((lane & 15) == 0) *reinterpret_cast<float2*>(out + 5120 + 2 * (t >> 4)) = bacc;
}

// Weight gradients of the layers with a two-channel side, FP32, in one launch
// (blockIdx.y 0: layer 4 with T = dy, B = r3; 1: layer 1 with T = x0, B = g1):
//   layer 4: dW[j][c][k] = sum_q B[c][q] T[j][q + 2 - k], db[j] = sum_q T[j][q]
//   layer 1: dW[c][j][k] = sum_q B[c][q] T[j][q + k - 2], db[c] = sum_q B[c][q]
// Bound by one pass over B.  A warp takes four channels and a lane four
// positions of each tile, 40 sums in registers; blocks walk the tiles and
// write one row of partial sums each ([j][k][c], then the biases).  256 rows of
// 1024: 20 us with one block of each layer an SM (23 with two, whose second
// wave starts and sums anew; 30 without the loads one tile ahead).
constexpr int kSdPart = 320 + 32;
__global__ void __launch_bounds__(256, 2) dn_side32_kernel(const float* __restrict__ dy,
                                                        const float* __restrict__ r3,
                                                        const float* __restrict__ x0,
                                                        const float* __restrict__ g1, int R, int N,
                                                        float* __restrict__ part4,
                                                        float* __restrict__ part1) {
  pdl_wait();
  const bool layer4 = blockIdx.y == 0;
  const float* __restrict__ T = layer4 ? dy : x0;
  const float* __restrict__ B = layer4 ? r3 : g1;
  const int lane = threadIdx.x & 31, ch = (threadIdx.x >> 5) * 4;
  const int tiles_row = N / kDnPos, tiles = R * tiles_row;
  float acc[4][2][kDnK], bacc[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    bacc[c] = 0.f;
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int k = 0; k < kDnK; ++k) acc[c][j][k] = 0.f;
  }
  float wn[2][8];
  float4 bn[4];
  auto fetch = [&](int tile) {   // one tile's loads, a tile ahead of their use
    const int r = tile / tiles_row, q = (tile % tiles_row) * kDnPos + 4 * lane;
#pragma unroll
    for (int j = 0; j < 2; ++j) window8(T + (static_cast<size_t>(r) * 2 + j) * N, q, N, wn[j]);
#pragma unroll
    for (int c = 0; c < 4; ++c)
      bn[c] = *reinterpret_cast<const float4*>(B + (static_cast<size_t>(r) * 32 + ch + c) * N + q);
  };
  if (blockIdx.x < tiles) fetch(blockIdx.x);
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    float w[2][8];
    float4 bv[4];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int i = 0; i < 8; ++i) w[j][i] = wn[j][i];
#pragma unroll
    for (int c = 0; c < 4; ++c) bv[c] = bn[c];
    if (tile + static_cast<int>(gridDim.x) < tiles) fetch(tile + gridDim.x);
    if (layer4) {
#pragma unroll
      for (int j = 0; j < 2; ++j) bacc[j] += (w[j][2] + w[j][3]) + (w[j][4] + w[j][5]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float x[4] = {bv[c].x, bv[c].y, bv[c].z, bv[c].w};
      if (!layer4) bacc[c] += (x[0] + x[1]) + (x[2] + x[3]);
      // kk walks the window upwards: tap 4 - kk for layer 4, kk for layer 1
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int kk = 0; kk < kDnK; ++kk)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[c][j][kk] = fmaf(x[i], w[j][i + kk], acc[c][j][kk]);
    }
  }
  auto lanes = [&](float v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
  };
  float* out = (layer4 ? part4 : part1) + static_cast<size_t>(blockIdx.x) * kSdPart;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int kk = 0; kk < kDnK; ++kk) {
        const float v = lanes(acc[c][j][kk]);
        if (lane == 0) out[(j * kDnK + (layer4 ? 4 - kk : kk)) * 32 + ch + c] = v;
      }
    const float v = lanes(bacc[c]);
    if (lane == 0) {
      if (!layer4) out[320 + ch + c] = v;
      else if (ch == 0 && c < 2) out[320 + c] = v;
    }
  }
}

// x0 = [Re H, Im H] / rms and, when Ht is given, t = [Re Ht, Im Ht] / rms;
// rms over the row of H.  Bound by latency: one block of 256 threads per row
// holds the row in registers (N <= 2048), all loads in flight at once, and the
// tree over the threads ends in one warp.  256 rows of 1024 with the weights:
// 3.6 us (5.8 with the rows read twice and a barrier per level).
__device__ __forceinline__ void prepare_row(const float2* H, const float2* Ht, int r, int N,
                                            float* x0, float* tt, float* rms) {
  __shared__ float red[256];
  const int t = threadIdx.x;
  const float2* h = H + static_cast<size_t>(r) * N;
  const float2* g = Ht ? Ht + static_cast<size_t>(r) * N : h;
  float2 hv[8], gv[8];
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = t + 256 * i;
    if (k < N) {
      hv[i] = h[k];
      gv[i] = g[k];
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (t + 256 * i < N) s = fmaf(hv[i].x, hv[i].x, fmaf(hv[i].y, hv[i].y, s));
  red[t] = s;
  __syncthreads();
  for (int w = 128; w > 32; w >>= 1) {
    if (t < w) red[t] += red[t + w];
    __syncthreads();
  }
  if (t < 32) {   // the tree's last levels
    s = red[t] + red[t + 32];
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) s += __shfl_down_sync(0xffffffffu, s, w);
    if (t == 0) red[0] = s;
  }
  __syncthreads();
  const float rr = sqrtf(red[0] / N);
  const float inv = rr > 0.f ? 1.0f / rr : 0.f;
  if (t == 0) rms[r] = rr;
  float* x = x0 + static_cast<size_t>(r) * 2 * N;
  float* y = Ht ? tt + static_cast<size_t>(r) * 2 * N : nullptr;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = t + 256 * i;
    if (k < N) {
      x[k] = hv[i].x * inv;
      x[N + k] = hv[i].y * inv;
      if (y) {
        y[k] = gv[i].x * inv;
        y[N + k] = gv[i].y * inv;
      }
    }
  }
}

// The FP32 kernels' weights (the first kSetupBlocks blocks) and the
// normalised rows (a block each), in one launch.
constexpr int kSetupBlocks = 32;
template <typename WT>
__global__ void __launch_bounds__(256) dn_setup_kernel(const WT* __restrict__ P, float* wt,
                                                       const float2* H, const float2* Ht, int N,
                                                       float* x0, float* tt, float* rms) {
  pdl_wait();
  if (blockIdx.x < kSetupBlocks)
    fp32_weights(P, wt, blockIdx.x * 256 + threadIdx.x, kSetupBlocks * 256);
  else
    prepare_row(H, Ht, blockIdx.x - kSetupBlocks, N, x0, tt, rms);
}

__global__ void dn_adam_kernel(float* p, const float* g, float* m, float* v, int n, float lr,
                               float b1, float b2, float eps, float c1, float c2) {
  pdl_wait();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

__global__ void dn_bf16_kernel(const float* p, __nv_bfloat16* q, int n) {
  pdl_wait();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    q[i] = __float2bfloat16_rn(p[i]);
}

// ------------------------------------------------------ tensor-core inference
//
// All four layers on tcgen05 (kind::f16, bf16 operands, fp32 accumulators in
// TMEM); the CUDA cores only split the input, apply ReLU, round to bf16
// and write the output.  Each block of 512 threads runs four tile
// slots of 128 threads that share one weight image; a slot walks tiles of
// (row, 116 output subcarriers).  Layers 2 and 3 work in place on the slot's
// one activation buffer: the epilogue writes only after the MMAs that read
// the buffer have completed.
//
// Every layer reads activation rows m .. m + 4 for MMA row m and writes row
// m + 2, with position rows at a uniform 16-byte stride, so the operand of
// tap k is the same buffer shifted by k rows (no im2col):
//  * layer 1 (2 -> 32): the input row holds x0 split into three bf16 terms
//    (hi, mid, lo of the real and imaginary parts; fp32-exact products) in
//    one 8-element K chunk; with the K-chunk stride set to one row, one
//    K = 16 MMA covers two taps: 3 MMAs (the sixth tap's weights are zero);
//  * layers 2, 3 (32 -> 32): activations as [channel chunk of 8][row][8];
//    5 taps x 2 K-halves, N = 32: 10 MMAs each;
//  * layer 4 (32 -> 2): the same operands, N = 16 with 14 zero outputs.
// Biases enter each layer as one more K = 16 MMA of a constant operand (a
// one in the first K slot of every row) against a B holding the bias in its
// first K slot, so the epilogue is a TMEM load and one relu-and-round
// conversion per channel pair.  Buffer rows 0, 1, 130, 131 are zero halos,
// so each layer's output is exact on two fewer MMA rows per side: 116 valid
// outputs of 128.  Activations at positions outside [0, N) are zero, as
// every layer's zero padding asks.
constexpr int kTcValid = 116;                    // final outputs per tile
constexpr int kTcFirst = 6;                      // first valid MMA row
constexpr int kTcRows = 132;                     // buffer rows (2-row halos)
constexpr int kTcLbo = kTcRows * 16;             // bytes between channel chunks
constexpr int kTcActBytes = 4 * kTcLbo;          // one activation buffer (32 ch)
constexpr int kTcXBytes = (kTcRows + 1) * 16;    // split input rows (+1 zero row)
// weight image: B operands of layer 1 (3 x 1 KB), layers 2 and 3 (5 taps x
// 2 KB each), layer 4 (5 taps x 1 KB), the four bias operands (1 KB each),
// then the constant A operand of the bias MMAs (129 rows of [1, 0 x 7])
constexpr int kTcL1 = 0, kTcL2 = 3072, kTcL3 = kTcL2 + 10240, kTcL4 = kTcL3 + 10240;
constexpr int kTcBias = kTcL4 + 5120;
constexpr int kTcOnes = kTcBias + 4 * 1024;
constexpr int kTcImgBytes = kTcOnes + 129 * 16;
constexpr int kTcImgFloats = kTcImgBytes / 4;
constexpr int kTcSlots = 4;                      // tiles in flight per block
constexpr int kTcSlotBytes = kTcXBytes + kTcActBytes;
constexpr int kTcSmem = kTcImgBytes + kTcSlots * kTcSlotBytes + kTcSlots * 8 + 16;
static_assert(kTcImgBytes % 16 == 0 && kTcSlotBytes % 16 == 0, "16-byte operand alignment");

__device__ __forceinline__ __nv_bfloat16 to_b(float v) { return __float2bfloat16_rn(v); }
__device__ __forceinline__ __nv_bfloat16 to_b(__nv_bfloat16 v) { return v; }

// elements first, first + step, ... of the image, from bf16 parameters or from
// fp32 ones rounded to bf16
template <typename PT>
__device__ __forceinline__ void tc_image(const PT* __restrict__ P, float* __restrict__ img, int first,
                                         int step) {
  unsigned char* b = reinterpret_cast<unsigned char*>(img);
  const __nv_bfloat16 zero = __float2bfloat16_rn(0.f);
  for (int e = first; e < kTcImgBytes / 2; e += step) {
    if (e < 1536) {                                   // layer 1: MMA j covers taps 2j, 2j + 1
      const int j = e / 512, o = (e / 16) % 32, kk = e % 16;
      const int tap = 2 * j + (kk >> 3), term = kk & 7;   // term: hi re, hi im, mid re, ...
      const __nv_bfloat16 w = (tap <= 4 && term < 6) ? to_b(P[kOffW1 + (o * 2 + (term & 1)) * 5 + tap]) : zero;
      *reinterpret_cast<__nv_bfloat16*>(b + kTcL1 + j * 1024 + (o >> 3) * 256 + (kk >> 3) * 128 +
                                        (o & 7) * 16 + (kk & 7) * 2) = w;
    } else if (e < 1536 + 10240) {                    // layers 2, 3: tap k, element (o, c)
      const int f = e - 1536;
      const int l = f / 5120, k = (f / 1024) % 5, o = (f / 32) % 32, c = f % 32;
      const __nv_bfloat16 w = to_b(P[(l == 0 ? kOffW2 : kOffW3) + (o * 32 + c) * 5 + k]);
      *reinterpret_cast<__nv_bfloat16*>(b + kTcL2 + l * 10240 + k * 2048 + (o >> 3) * 512 +
                                        (c >> 3) * 128 + (o & 7) * 16 + (c & 7) * 2) = w;
    } else if (e < kTcBias / 2) {                     // layer 4: tap k, element (o < 16, c)
      const int f = e - 1536 - 10240;
      const int k = f / 512, o = (f / 32) % 16, c = f % 32;
      const __nv_bfloat16 w = o < 2 ? to_b(P[kOffW4 + (o * 32 + c) * 5 + k]) : zero;
      *reinterpret_cast<__nv_bfloat16*>(b + kTcL4 + k * 1024 + (o >> 3) * 512 + (c >> 3) * 128 +
                                        (o & 7) * 16 + (c & 7) * 2) = w;
    } else if (e < kTcBias / 2 + 2048) {              // bias operand of layer l: (o, k = 0)
      const int f = e - kTcBias / 2;
      const int l = f / 512, o = (f / 16) % 32, k = f % 16;
      const int src = l == 0 ? kOffB1 : l == 1 ? kOffB2 : l == 2 ? kOffB3 : kOffB4;
      const __nv_bfloat16 w = (k == 0 && (l < 3 || o < 2)) ? to_b(P[src + o]) : zero;
      *reinterpret_cast<__nv_bfloat16*>(b + kTcBias + l * 1024 + (o >> 3) * 256 + (k >> 3) * 128 +
                                        (o & 7) * 16 + (k & 7) * 2) = w;
    } else {                                          // the constant operand: rows [1, 0 x 7]
      const int f = e - kTcBias / 2 - 2048;
      *reinterpret_cast<__nv_bfloat16*>(b + kTcOnes + 2 * f) = __float2bfloat16_rn((f & 7) == 0 ? 1.f : 0.f);
    }
  }
}

// ReLU and round to bf16 (nearest even) a pair of channels: o in the low half
__device__ __forceinline__ uint32_t relu_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
// layer output of MMA row m (bias included) -> buffer row m + 2; zero outside [0, N)
__device__ __forceinline__ void tc_epilogue(const float* d, bool inside, unsigned char* out, int m) {
  if (inside) {
#pragma unroll
    for (int kc = 0; kc < 4; ++kc)
      *reinterpret_cast<uint4*>(out + kc * kTcLbo + (m + 2) * 16) =
          make_uint4(relu_bf16x2(d[8 * kc], d[8 * kc + 1]), relu_bf16x2(d[8 * kc + 2], d[8 * kc + 3]),
                     relu_bf16x2(d[8 * kc + 4], d[8 * kc + 5]), relu_bf16x2(d[8 * kc + 6], d[8 * kc + 7]));
  } else {
#pragma unroll
    for (int kc = 0; kc < 4; ++kc)
      *reinterpret_cast<uint4*>(out + kc * kTcLbo + (m + 2) * 16) = make_uint4(0u, 0u, 0u, 0u);
  }
}

// x -> three bf16 terms whose sum is x to float32 precision
__device__ __forceinline__ void split3(float x, __nv_bfloat16& hi, __nv_bfloat16& mid, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(x);
  const float r1 = x - __bfloat162float(hi);
  mid = __float2bfloat16_rn(r1);
  lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
}
__device__ __forceinline__ uint4 x_row(float re, float im) {
  __nv_bfloat16 h[8];
  split3(re, h[0], h[2], h[4]);
  split3(im, h[1], h[3], h[5]);
  h[6] = h[7] = __float2bfloat16_rn(0.f);
  return *reinterpret_cast<const uint4*>(h);
}

__global__ void __launch_bounds__(128 * kTcSlots, 2) dn_tc_kernel(const float* __restrict__ img_g,
                                                       const float* __restrict__ x0,
                                                       const float* __restrict__ rms, int R, int N,
                                                       float2* __restrict__ Hout, int* status) {
  pdl_wait();
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* wimg = smem;
  const int t = threadIdx.x;
  const int slot = t >> 7, u = t & 127, warp = t >> 5;
  unsigned char* xb = smem + kTcImgBytes + slot * kTcSlotBytes;           // split input rows
  unsigned char* act = xb + kTcXBytes;                                     // layers 1-3 out
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kTcImgBytes + kTcSlots * kTcSlotBytes);
  uint32_t* tbase = reinterpret_cast<uint32_t*>(bars + kTcSlots);
  uint64_t* bar = &bars[slot];
  if (t == 0) {
    for (int g = 0; g < kTcSlots; ++g) mbar_init(smem_u32(&bars[g]), 1);
    fence_mbar_init();
    mbar_expect_tx(smem_u32(&bars[0]), kTcImgBytes);        // phase 0 of slot 0's barrier
    bulk_load(smem_u32(wimg), img_g, kTcImgBytes, smem_u32(&bars[0]), evict_last_policy());
  }
  __syncwarp();
  if (warp == 0) tmem_alloc(smem_u32(tbase), 32 * kTcSlots);
  // halo rows of both activation buffers stay zero
  if (u < 16) {                                     // 4 chunks x rows 0, 1, 130, 131
    const int kc = u >> 2, row = (u & 3) < 2 ? (u & 3) : kTcRows - 4 + (u & 3);
    *reinterpret_cast<uint4*>(act + kc * kTcLbo + row * 16) = make_uint4(0u, 0u, 0u, 0u);
  }
  const int tiles_row = (N + kTcValid - 1) / kTcValid;
  const int tiles = R * tiles_row;
  const int stride = gridDim.x * kTcSlots;
  // x0 of a tile for this thread: rows u and 128 + u (u < 4) of the split
  // input, and the residual at MMA row u; fetched one tile ahead
  float xa0 = 0.f, xa1 = 0.f, xb0 = 0.f, xb1 = 0.f, xr0 = 0.f, xr1 = 0.f;
  auto fetch = [&](int tile) {
    xa0 = xa1 = xb0 = xb1 = xr0 = xr1 = 0.f;
    if (tile >= tiles) return;
    const int r = tile / tiles_row, s0 = (tile % tiles_row) * kTcValid - kTcFirst;
    const float* re = x0 + static_cast<size_t>(r) * 2 * N;
    const float* im = re + N;
    const int qa = s0 - 2 + u, qb = s0 + 126 + u, qr = s0 + u;
    if (qa >= 0 && qa < N) { xa0 = re[qa]; xa1 = im[qa]; }
    if (u < 4 && qb >= 0 && qb < N) { xb0 = re[qb]; xb1 = im[qb]; }
    if (qr >= 0 && qr < N) { xr0 = re[qr]; xr1 = im[qr]; }
  };
  int tile = blockIdx.x * kTcSlots + slot;
  fetch(tile);
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  const uint32_t tm = *tbase + 32 * slot + (static_cast<uint32_t>(32 * (warp & 3)) << 16);
  const uint32_t tm_mma = *tbase + 32 * slot;
  const uint32_t id32 = umma_idesc(32, true), id16 = umma_idesc(16, true);
  // descriptors at offset 0; an offset o (bytes, 16-aligned) adds o >> 4
  const uint64_t dx = umma_desc(smem_u32(xb), 16, 128);
  const uint64_t da = umma_desc(smem_u32(act), kTcLbo, 128);
  const uint64_t dw1 = umma_desc(smem_u32(wimg), 128, 256);
  const uint64_t dw = umma_desc(smem_u32(wimg), 128, 512);
  const uint64_t dones = umma_desc(smem_u32(wimg + kTcOnes), 16, 128);
  // every thread waits for the image (phase 0 of slot 0's barrier)
  bool ok = mbar_wait_bounded(smem_u32(&bars[0]), 0);
  if (!ok) latch(status, kStTimeout);
  uint32_t phase = slot == 0 ? 1u : 0u;
  auto issue_wait = [&](int layer) {
    fence_proxy_async();
    tmem_fence_before();
    named_sync(1 + slot, 128);
    tmem_fence_after();
    if (u == 0) {
      umma_f16(tm_mma, dones, dw1 + ((kTcBias + 1024 * (layer - 1)) >> 4), layer == 4 ? id16 : id32, 0u);
      if (layer == 1) {
#pragma unroll
        for (int j = 0; j < 3; ++j)
          umma_f16(tm_mma, dx + 2 * j, dw1 + ((kTcL1 + 1024 * j) >> 4), id32, 1u);
      } else {
        const int boff = layer == 2 ? kTcL2 : layer == 3 ? kTcL3 : kTcL4;
        const int tapb = layer == 4 ? 1024 : 2048;
        const uint32_t idesc = layer == 4 ? id16 : id32;
#pragma unroll
        for (int k = 0; k < 5; ++k)
#pragma unroll
          for (int kh = 0; kh < 2; ++kh)
            umma_f16(tm_mma, da + ((k * 16 + kh * 2 * kTcLbo) >> 4),
                     dw + ((boff + k * tapb + kh * 256) >> 4), idesc, 1u);
      }
      umma_commit(smem_u32(bar));
      // the issuing thread alone waits; the others sleep in the barrier
      if (ok && !mbar_wait_bounded(smem_u32(bar), phase)) {
        ok = false;
        latch(status, kStTimeout);
      }
    }
    phase ^= 1;
    tmem_fence_before();
    named_sync(1 + slot, 128);
    tmem_fence_after();
  };
  for (; tile < tiles; tile += stride) {
    const int r = tile / tiles_row;
    const int s0 = (tile % tiles_row) * kTcValid - kTcFirst;   // position of MMA row 0
    const float xres0 = xr0, xres1 = xr1;
    // split input: row b <-> position s0 - 2 + b; row 132 stays zero
    *reinterpret_cast<uint4*>(xb + u * 16) = x_row(xa0, xa1);
    if (u < 4) *reinterpret_cast<uint4*>(xb + (128 + u) * 16) = x_row(xb0, xb1);
    if (u == 4) *reinterpret_cast<uint4*>(xb + kTcRows * 16) = make_uint4(0u, 0u, 0u, 0u);
    fetch(tile + stride);                                     // next tile's x0, in flight
    const int q = s0 + u;                                     // position of MMA row u
    const bool inside = q >= 0 && q < N;
    float d[32];
    issue_wait(1);
    Tmem<32>::ld(tm, d);
    tmem_wait_ld();
    tc_epilogue(d, inside, act, u);
    issue_wait(2);
    Tmem<32>::ld(tm, d);
    tmem_wait_ld();
    tc_epilogue(d, inside, act, u);
    issue_wait(3);
    Tmem<32>::ld(tm, d);
    tmem_wait_ld();
    tc_epilogue(d, inside, act, u);
    issue_wait(4);
    float y[2];
    Tmem<2>::ld(tm, y);
    tmem_wait_ld();
    if (u >= kTcFirst && u < kTcFirst + kTcValid && q < N) {
      const float rr = rms[r];
      Hout[static_cast<size_t>(r) * N + q] =
          make_float2((xres0 + y[0]) * rr, (xres1 + y[1]) * rr);
    }
  }
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  if (warp == 0) tmem_dealloc(*tbase, 32 * kTcSlots);
}

// ------------------------------------------------------ tensor-core training
//
// BF16 training on tcgen05 with fp32 master weights (rounded to bf16 for
// every step) and fp32 Adam.  Three passes per step:
//  * forward (dn_tc_train_kernel<false>): the inference tile loop of
//    dn_tc_kernel, which also stores each ReLU output r1, r2, r3 exactly as
//    the next layer consumed it (bf16) and, at the network output,
//    dy = 2 (y - t) / n and the tile's sum of (y - t)^2;
//  * data gradients (dn_tc_train_kernel<true>): the same tile loop over
//    three convolutions with transposed, flipped weights (g3 = conv(dy; W4'),
//    g2 = conv(g3; W3'), g1 = conv(g2; W2'), W'[c][o][k] = W[o][c][4 - k}),
//    each output masked by its layer's ReLU (r > 0) instead of a ReLU, no
//    bias; dy enters split into three bf16 terms like x0, and g3, g2, g1 are
//    stored in bf16;
//  * weight gradients (dn_tc_wgrad_kernel): the two 32 -> 32 layers as
//    tensor-core reductions over positions, the two layers with two-channel
//    sides (1 and 4) and the biases on the CUDA cores from the same bf16
//    tensors; per-block partial sums are added in block order.
// A stored tensor is [R][4][N + 4][8] bf16: four planes of eight channels per
// row, so that the threads of a warp (consecutive positions) write and read
// consecutive 16-byte pieces, with two zero positions at either end of a
// plane (the convolutions' zero padding).
constexpr int kTrPad = 2;    // zero positions at either end of a plane
__host__ __device__ __forceinline__ size_t tr_plane(int R, int N) {   // elements of one tensor
  return static_cast<size_t>(R) * 32 * (N + 2 * kTrPad);
}
// element offset of position q of channel chunk 0 of row r; chunk kc adds kc * tr_chunk(N)
__device__ __forceinline__ size_t tr_at(int r, int N, int q) {
  return (static_cast<size_t>(r) * 4 * (N + 2 * kTrPad) + q + kTrPad) * 8;
}
__device__ __forceinline__ size_t tr_chunk(int N) { return static_cast<size_t>(N + 2 * kTrPad) * 8; }

// Backward weight image: layer-1 slot = W4' (2 -> 32), layer-2 slot = W3',
// layer-3 slot = W2', zero biases and layer-4 slot, the constant operand.
__device__ __forceinline__ void tc_bimage(const float* __restrict__ P, float* __restrict__ img, int first,
                                          int step) {
  unsigned char* b = reinterpret_cast<unsigned char*>(img);
  const __nv_bfloat16 zero = __float2bfloat16_rn(0.f);
  for (int e = first; e < kTcImgBytes / 2; e += step) {
    if (e < 1536) {                                   // W4': out c, in o = term & 1
      const int j = e / 512, c = (e / 16) % 32, kk = e % 16;
      const int tap = 2 * j + (kk >> 3), term = kk & 7;
      const __nv_bfloat16 w =
          (tap <= 4 && term < 6) ? to_b(P[kOffW4 + ((term & 1) * 32 + c) * 5 + (4 - tap)]) : zero;
      *reinterpret_cast<__nv_bfloat16*>(b + kTcL1 + j * 1024 + (c >> 3) * 256 + (kk >> 3) * 128 +
                                        (c & 7) * 16 + (kk & 7) * 2) = w;
    } else if (e < 1536 + 10240) {                    // W3' then W2': tap k, element (out c, in o)
      const int f = e - 1536;
      const int l = f / 5120, k = (f / 1024) % 5, c = (f / 32) % 32, o = f % 32;
      const __nv_bfloat16 w = to_b(P[(l == 0 ? kOffW3 : kOffW2) + (o * 32 + c) * 5 + (4 - k)]);
      *reinterpret_cast<__nv_bfloat16*>(b + kTcL2 + l * 10240 + k * 2048 + (c >> 3) * 512 +
                                        (o >> 3) * 128 + (c & 7) * 16 + (o & 7) * 2) = w;
    } else if (e < kTcOnes / 2) {                     // layer-4 slot and the biases: zero
      *reinterpret_cast<__nv_bfloat16*>(b + 2 * e) = zero;
    } else {                                          // the constant operand: rows [1, 0 x 7]
      const int f = e - kTcOnes / 2;
      *reinterpret_cast<__nv_bfloat16*>(b + kTcOnes + 2 * f) = __float2bfloat16_rn((f & 7) == 0 ? 1.f : 0.f);
    }
  }
}

// Everything a pass needs before its first tile, in one launch of 256-thread
// blocks: the weight images (the first kSetupBlocks blocks an image; bimg
// null: forward image only) and the normalised rows (a block each).  The four
// launches it replaces took 10.3 us at 256 rows of 1024 and their gaps.
template <typename PT>
__global__ void __launch_bounds__(256) dn_tc_setup_kernel(const PT* __restrict__ P, float* img,
                                                          float* bimg, const float2* H,
                                                          const float2* Ht, int N, float* x0,
                                                          float* tt, float* rms) {
  pdl_wait();
  int b = blockIdx.x;
  if (b < kSetupBlocks) {
    tc_image(P, img, b * 256 + threadIdx.x, kSetupBlocks * 256);
    return;
  }
  b -= kSetupBlocks;
  if constexpr (sizeof(PT) == 4) {
    if (bimg) {
      if (b < kSetupBlocks) {
        tc_bimage(P, bimg, b * 256 + threadIdx.x, kSetupBlocks * 256);
        return;
      }
      b -= kSetupBlocks;
    }
  }
  prepare_row(H, Ht, b, N, x0, tt, rms);
}

// pack two floats to bf16 (nearest even), first in the low half
__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
// keep the bf16 halves of v where the halves of mask are nonzero
__device__ __forceinline__ uint32_t mask_bf16x2(uint32_t v, uint32_t mask) {
  const uint32_t keep = ((mask & 0xFFFFu) ? 0xFFFFu : 0u) | ((mask & 0xFFFF0000u) ? 0xFFFF0000u : 0u);
  return v & keep;
}

template <bool BWD>
__global__ void __launch_bounds__(128 * kTcSlots, 2) dn_tc_train_kernel(
    const float* __restrict__ img_g, const float* __restrict__ in0, const float* __restrict__ tt,
    int R, int N, float inv_n, __nv_bfloat16* __restrict__ acts, __nv_bfloat16* __restrict__ grads,
    float* __restrict__ dy, float* __restrict__ part, int* status) {
  pdl_wait();
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* wimg = smem;
  const int t = threadIdx.x;
  const int slot = t >> 7, u = t & 127, warp = t >> 5, lane = t & 31;
  unsigned char* xb = smem + kTcImgBytes + slot * kTcSlotBytes;
  unsigned char* act = xb + kTcXBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kTcImgBytes + kTcSlots * kTcSlotBytes);
  uint32_t* tbase = reinterpret_cast<uint32_t*>(bars + kTcSlots);
  float* red = reinterpret_cast<float*>(tbase + 4);           // [slot][4 warps]
  uint64_t* bar = &bars[slot];
  if (t == 0) {
    for (int g = 0; g < kTcSlots; ++g) mbar_init(smem_u32(&bars[g]), 1);
    fence_mbar_init();
    mbar_expect_tx(smem_u32(&bars[0]), kTcImgBytes);
    bulk_load(smem_u32(wimg), img_g, kTcImgBytes, smem_u32(&bars[0]), evict_last_policy());
  }
  __syncwarp();
  if (warp == 0) tmem_alloc(smem_u32(tbase), 32 * kTcSlots);
  if (u < 16) {
    const int kc = u >> 2, row = (u & 3) < 2 ? (u & 3) : kTcRows - 4 + (u & 3);
    *reinterpret_cast<uint4*>(act + kc * kTcLbo + row * 16) = make_uint4(0u, 0u, 0u, 0u);
  }
  const int tiles_row = (N + kTcValid - 1) / kTcValid;
  const int tiles = R * tiles_row;
  const int stride = gridDim.x * kTcSlots;
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  const uint32_t tm = *tbase + 32 * slot + (static_cast<uint32_t>(32 * (warp & 3)) << 16);
  const uint32_t tm_mma = *tbase + 32 * slot;
  const uint32_t id32 = umma_idesc(32, true), id16 = umma_idesc(16, true);
  const uint64_t dx = umma_desc(smem_u32(xb), 16, 128);
  const uint64_t da = umma_desc(smem_u32(act), kTcLbo, 128);
  const uint64_t dw1 = umma_desc(smem_u32(wimg), 128, 256);
  const uint64_t dw = umma_desc(smem_u32(wimg), 128, 512);
  const uint64_t dones = umma_desc(smem_u32(wimg + kTcOnes), 16, 128);
  bool ok = mbar_wait_bounded(smem_u32(&bars[0]), 0);
  if (!ok) latch(status, kStTimeout);
  uint32_t phase = slot == 0 ? 1u : 0u;
  const size_t plane = tr_plane(R, N);   // one stored tensor (elements)
  const size_t chunk = tr_chunk(N);
  for (int tile = blockIdx.x * kTcSlots + slot; tile < tiles; tile += stride) {
    const int r = tile / tiles_row;
    const int s0 = (tile % tiles_row) * kTcValid - kTcFirst;   // position of MMA row 0
    const float* re = in0 + static_cast<size_t>(r) * 2 * N;
    const float* im = re + N;
    // split input rows: row b <-> position s0 - 2 + b; row 132 stays zero
    {
      const int qa = s0 - 2 + u, qb = s0 + 126 + u;
      float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f;
      if (qa >= 0 && qa < N) { a0 = re[qa]; a1 = im[qa]; }
      if (u < 4 && qb >= 0 && qb < N) { b0 = re[qb]; b1 = im[qb]; }
      *reinterpret_cast<uint4*>(xb + u * 16) = x_row(a0, a1);
      if (u < 4) *reinterpret_cast<uint4*>(xb + (128 + u) * 16) = x_row(b0, b1);
      if (u == 4) *reinterpret_cast<uint4*>(xb + kTcRows * 16) = make_uint4(0u, 0u, 0u, 0u);
    }
    const int q = s0 + u;                                     // position of MMA row u
    const bool inside = q >= 0 && q < N;
    const bool mine = u >= kTcFirst && u < kTcFirst + kTcValid && inside;   // stored by this tile
    const size_t rowoff = tr_at(r, N, q);
    auto issue_wait = [&](int layer) {
      fence_proxy_async();
      tmem_fence_before();
      named_sync(1 + slot, 128);
      tmem_fence_after();
      if (u == 0) {
        umma_f16(tm_mma, dones, dw1 + ((kTcBias + 1024 * (layer - 1)) >> 4), layer == 4 ? id16 : id32, 0u);
        if (layer == 1) {
#pragma unroll
          for (int j = 0; j < 3; ++j)
            umma_f16(tm_mma, dx + 2 * j, dw1 + ((kTcL1 + 1024 * j) >> 4), id32, 1u);
        } else {
          const int boff = layer == 2 ? kTcL2 : layer == 3 ? kTcL3 : kTcL4;
          const int tapb = layer == 4 ? 1024 : 2048;
          const uint32_t idesc = layer == 4 ? id16 : id32;
#pragma unroll
          for (int k = 0; k < 5; ++k)
#pragma unroll
            for (int kh = 0; kh < 2; ++kh)
              umma_f16(tm_mma, da + ((k * 16 + kh * 2 * kTcLbo) >> 4),
                       dw + ((boff + k * tapb + kh * 256) >> 4), idesc, 1u);
        }
        umma_commit(smem_u32(bar));
        if (ok && !mbar_wait_bounded(smem_u32(bar), phase)) {
          ok = false;
          latch(status, kStTimeout);
        }
      }
      phase ^= 1;
      tmem_fence_before();
      named_sync(1 + slot, 128);
      tmem_fence_after();
    };
    // one layer's epilogue: activation (or masked gradient) of MMA row u to
    // buffer row u + 2, and to the stored tensor `out` where this tile owns q
    auto epilogue = [&](const float* d, const __nv_bfloat16* mask_src, __nv_bfloat16* out) {
      uint4 w[4];
      if (inside) {
        uint4 mk[4];
        if (BWD) {
#pragma unroll
          for (int kc = 0; kc < 4; ++kc) mk[kc] = *reinterpret_cast<const uint4*>(mask_src + rowoff + kc * chunk);
        }
#pragma unroll
        for (int kc = 0; kc < 4; ++kc) {
          const float* e = d + 8 * kc;
          if (BWD) {
            w[kc] = make_uint4(mask_bf16x2(bf16x2(e[0], e[1]), mk[kc].x), mask_bf16x2(bf16x2(e[2], e[3]), mk[kc].y),
                               mask_bf16x2(bf16x2(e[4], e[5]), mk[kc].z), mask_bf16x2(bf16x2(e[6], e[7]), mk[kc].w));
          } else {
            w[kc] = make_uint4(relu_bf16x2(e[0], e[1]), relu_bf16x2(e[2], e[3]),
                               relu_bf16x2(e[4], e[5]), relu_bf16x2(e[6], e[7]));
          }
        }
      } else {
#pragma unroll
        for (int kc = 0; kc < 4; ++kc) w[kc] = make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int kc = 0; kc < 4; ++kc) *reinterpret_cast<uint4*>(act + kc * kTcLbo + (u + 2) * 16) = w[kc];
      if (mine) {
#pragma unroll
        for (int kc = 0; kc < 4; ++kc) *reinterpret_cast<uint4*>(out + rowoff + kc * chunk) = w[kc];
        // the row's first and last position also write its zero pads
        if (q == 0 || q == N - 1) {
          const long pad = q == 0 ? -16 : 8;
#pragma unroll
          for (int kc = 0; kc < 4; ++kc) {
            uint4* z = reinterpret_cast<uint4*>(out + rowoff + kc * chunk + pad);
            z[0] = z[1] = make_uint4(0u, 0u, 0u, 0u);
          }
        }
      }
    };
    float d[32];
    issue_wait(1);
    Tmem<32>::ld(tm, d);
    tmem_wait_ld();
    // forward: r1 -> acts[0]; backward: g3 = conv(dy; W4') masked by r3 -> grads[0]
    epilogue(d, acts + 2 * plane, BWD ? grads : acts);
    issue_wait(2);
    Tmem<32>::ld(tm, d);
    tmem_wait_ld();
    epilogue(d, acts + plane, BWD ? grads + plane : acts + plane);
    issue_wait(3);
    Tmem<32>::ld(tm, d);
    tmem_wait_ld();
    epilogue(d, acts, BWD ? grads + 2 * plane : acts + 2 * plane);
    if (!BWD) {
      // network output y = x0 + a4, dy = 2 (y - t) / n, the tile's squared error
      issue_wait(4);
      float y[2];
      Tmem<2>::ld(tm, y);
      tmem_wait_ld();
      float se = 0.f;
      if (mine) {
        const size_t o = static_cast<size_t>(r) * 2 * N + q;
        const float e0 = re[q] + y[0] - tt[o], e1 = im[q] + y[1] - tt[o + N];
        dy[o] = e0 * inv_n;
        dy[o + N] = e1 * inv_n;
        se = fmaf(e0, e0, e1 * e1);
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) se += __shfl_xor_sync(0xffffffffu, se, off);
      if (lane == 0) red[slot * 4 + (warp & 3)] = se;
      named_sync(1 + slot, 128);
      if (u == 0) part[tile] = ((red[slot * 4] + red[slot * 4 + 1]) + red[slot * 4 + 2]) + red[slot * 4 + 3];
      named_sync(1 + slot, 128);
    }
  }
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  if (warp == 0) tmem_dealloc(*tbase, 32 * kTcSlots);
}

constexpr int kTrSmem = kTcSmem + 64;   // + per-slot loss partials of four warps

// All weight gradients of the BF16 training step in one launch, one block per
// SM, three kinds of warps side by side; every block writes one row of partial
// sums per layer, which dn_reduce_kernel adds in block order.
//
// The two 32 -> 32 layers on tcgen05: dW[o][c][k] = sum_q A[c][q + k - 2]
// G[o][q] with positions as K, for layer 3 (A = r2, G = g3) and layer 2 (A =
// r1, G = g2) together.  Bound by operand reads from shared memory (M = 128
// needs 4 KB of A per 16 positions whatever N is), so the layout makes every
// MMA carry two layers and two taps: per 128-position tile the A operand is
// [r2 | r1 | r2' | r1'] (MN-major, eight-channel chunks 2112 bytes apart, '
// shifted by one position) and B is [g3 | g2], N = 64.  Starting A t positions
// later (16 t bytes: a position is one 16-byte row) gives taps t and t + 1, so
// t = 0, 2, 4 covers the five taps; of D only the r2 x g3 and r1 x g2 quarters
// are kept.  A producer warp brings a tile's 24 pieces by bulk copies into a
// ring of four stages, an MMA thread consumes them, and the four warps that
// later read the accumulators sum G for the biases meanwhile.
//
// Layers 1 and 4 (a two-channel side) on the CUDA cores by eight more warps:
// see side_grad.
//
// 256 rows of 1024: 31 us, against 61 us for one launch per layer that staged
// five shifted copies of A through registers, plus 18 us for layers 1 and 4.
// What is left is memory traffic: the stored tensors (100 MB there) outgrow
// L2, so this launch reads them back from HBM while the passes' dirty lines
// drain (36 us without the evict-first hint; dropping the shifted copies or
// most MMAs changes nothing).
constexpr int kWgRows = 132;                               // positions -2 .. 129 of a tile
constexpr int kWgChunk = kWgRows * 16;                     // one channel chunk of A
constexpr int kWgGChunk = 128 * 16;                        // one channel chunk of G
constexpr int kWgA = 0, kWgG = 16 * kWgChunk;              // of a stage
constexpr int kWgStage = kWgG + 8 * kWgGChunk;
constexpr int kWgStages = 4;
constexpr int kWgBars = kWgStages * kWgStage;              // full, empty, done
constexpr int kWgSmem = kWgBars + (2 * kWgStages + 1) * 8 + 8;
// warp 0 copies, 1 MMAs, 2 and 3 bias sums, 4-11 layers 1 and 4, 12 the loss: up
// to 16 warps leave 128 registers a thread, which the loads one tile ahead need
constexpr int kWgSideWarp = 4;
constexpr int kWgLossWarp = kWgSideWarp + 8;
constexpr int kWgThreads = 32 * (kWgLossWarp + 1);
static_assert(kWgSmem <= 232448, "shared memory of one block");

// Weight gradient of a layer with a two-channel side, by eight warps:
// layer 4 (T = dy fp32 [R][2][N], B = r3) or layer 1 (T = x0, B = g1), B a
// stored bf16 tensor:
//   layer 4: dW[j][c][k] = sum_q B[c][q] T[j][q + 2 - k], db[j] = sum_q T[j][q]
//   layer 1: dW[c][j][k] = sum_q B[c][q] T[j][q + k - 2], db[c] = sum_q B[c][q]
// Bound by the FMA pipe (320 FMAs a position) and one pass over B.  A warp
// takes one 8-channel chunk and one j; a lane keeps their 40 sums in registers
// over four consecutive positions of each 128-position tile, so a position's 8
// channels come in one 16-byte load (the two warps of a chunk share it in L1)
// and its 5 shifted T values from an 8-value register window.  (One block per
// channel pair with 2-byte strided loads took 749 + 659 us at 256 rows of
// 1024; both j in one warp spill registers beside the other roles.)
template <bool LAYER4>
__device__ __forceinline__ void side_grad(const float* __restrict__ T,
                                          const __nv_bfloat16* __restrict__ B, int R, int N,
                                          float* __restrict__ out, int warp, int lane) {
  const int kc = warp & 3, j = warp >> 2;
  const int tiles_row = N / 128, tiles = R * tiles_row;
  float2 acc[kDnK][4], bacc[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    bacc[i] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < kDnK; ++k) acc[k][i] = make_float2(0.f, 0.f);
  }
  // one tile's loads: the window of T (positions q - 2 .. q + 5, zero outside
  // the row) and four positions of B; issued a tile ahead
  float4 c;
  float2 a, d;
  uint4 bn[4];
  auto fetch = [&](int tile) {
    const int r = tile / tiles_row, q = (tile % tiles_row) * 128 + 4 * lane;
    const float* t = T + (static_cast<size_t>(r) * 2 + j) * N + q;
    c = *reinterpret_cast<const float4*>(t);
    a = q > 0 ? *reinterpret_cast<const float2*>(t - 2) : make_float2(0.f, 0.f);
    d = q + 4 < N ? *reinterpret_cast<const float2*>(t + 4) : make_float2(0.f, 0.f);
    const uint4* b = reinterpret_cast<const uint4*>(B + tr_at(r, N, q) + kc * tr_chunk(N));
#pragma unroll
    for (int i = 0; i < 4; ++i) bn[i] = b[i];
  };
  if (blockIdx.x < tiles) fetch(blockIdx.x);
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const float w[8] = {a.x, a.y, c.x, c.y, c.z, c.w, d.x, d.y};
    const uint4 bv[4] = {bn[0], bn[1], bn[2], bn[3]};
    if (tile + static_cast<int>(gridDim.x) < tiles) fetch(tile + gridDim.x);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t u[4] = {bv[i].x, bv[i].y, bv[i].z, bv[i].w};
      float2 x[4];
#pragma unroll
      for (int e = 0; e < 4; ++e)
        x[e] = make_float2(__uint_as_float(u[e] << 16), __uint_as_float(u[e] & 0xFFFF0000u));
      if (LAYER4) {
        bacc[0].x += w[2 + i];
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) bacc[e] = cadd(bacc[e], x[e]);
      }
      // kk walks the window upwards: tap 4 - kk for layer 4, kk for layer 1
#pragma unroll
      for (int kk = 0; kk < kDnK; ++kk) {
        const float2 tv = make_float2(w[i + kk], w[i + kk]);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[kk][e] = __ffma2_rn(x[e], tv, acc[kk][e]);
      }
    }
  }
  auto lanes = [&](float v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
  };
#pragma unroll
  for (int kk = 0; kk < kDnK; ++kk) {
    float2* o = reinterpret_cast<float2*>(out + (j * kDnK + (LAYER4 ? 4 - kk : kk)) * 32 + 8 * kc);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 v = make_float2(lanes(acc[kk][e].x), lanes(acc[kk][e].y));
      if (lane == 0) o[e] = v;
    }
  }
  if (LAYER4) {
    const float v = lanes(bacc[0].x);
    if (lane == 0 && kc == 0) out[320 + j] = v;
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 v = make_float2(lanes(bacc[e].x), lanes(bacc[e].y));
      if (lane == 0 && j == 0) reinterpret_cast<float2*>(out + 320 + 8 * kc)[e] = v;
    }
  }
}

struct DnWgradArgs {
  const __nv_bfloat16* acts;    // r1, r2, r3, one tr_plane each
  const __nv_bfloat16* grads;   // g3, g2, g1
  const float* x0;
  const float* dy;
  int R, N;
  float *part3, *part2, *part4, *part1;   // one row per block: kWgPart, kSdPart floats
  const float* loss_part;                 // the forward pass's sums of (y - t)^2, one per tile
  int loss_n;
  size_t n;
  float* loss;
  int* status;
};
__global__ void __launch_bounds__(kWgThreads, 1) dn_tc_wgrad_kernel(const DnWgradArgs a) {
  pdl_wait();
  extern __shared__ __align__(128) unsigned char smem[];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kWgBars);
  uint64_t* empty = full + kWgStages;
  uint64_t* done = empty + kWgStages;
  uint32_t* tbase = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tbase + 1);
  const int N = a.N, R = a.R;
  const size_t plane = tr_plane(R, N);
  if (t == 0) {
    *abort_flag = 0;
    for (int s = 0; s < kWgStages; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 3);   // the MMAs' commit and two summing warps
    }
    mbar_init(smem_u32(done), 1);
    fence_mbar_init();
  }
  if (warp == 1) tmem_alloc(smem_u32(tbase), 256);
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  float* part3 = a.part3 + static_cast<size_t>(blockIdx.x) * kWgPart;
  float* part2 = a.part2 + static_cast<size_t>(blockIdx.x) * kWgPart;
  const uint32_t tD = *tbase;   // three accumulators (taps 0/1, 2/3, 4) of 64 columns
  const int tiles_row = N / 128, tiles = R * tiles_row;
  // a bounded wait that gave up stops every role's loop; waits end at once then
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (*abort_flag) return false;
    if (mbar_wait_bounded(smem_u32(bar), parity)) return true;
    *abort_flag = 1;
    latch(a.status, kStTimeout);
    return false;
  };
  if (warp == kWgLossWarp) {
    // the loss, by one thread: the forward pass's partials added in tile order
    // (the order it has always had, so the same bits), loads 64 values ahead
    if (blockIdx.x == gridDim.x - 1 && lane == 0) {
      const float4* part = reinterpret_cast<const float4*>(a.loss_part);
      const int n4 = a.loss_n / 4;
      float4 v[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = i < n4 ? part[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      float s = 0.f;
      for (int i0 = 0; i0 < n4; i0 += 16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {   // (a sum of squares plus zero is itself)
          s += v[i].x;
          s += v[i].y;
          s += v[i].z;
          s += v[i].w;
          v[i] = i0 + 16 + i < n4 ? part[i0 + 16 + i] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      for (int i = 4 * n4; i < a.loss_n; ++i) s += a.loss_part[i];
      *a.loss = s / static_cast<float>(a.n);
    }
    __syncwarp();
  } else if (warp >= kWgSideWarp) {
    side_grad<true>(a.dy, a.acts + 2 * plane, R, N,
                    a.part4 + static_cast<size_t>(blockIdx.x) * kSdPart, warp - kWgSideWarp, lane);
    side_grad<false>(a.x0, a.grads + 2 * plane, R, N,
                     a.part1 + static_cast<size_t>(blockIdx.x) * kSdPart, warp - kWgSideWarp, lane);
  } else if (warp == 0) {
    // copies: lanes 0-7 the chunks of r2 and r1, 8-15 the same one position
    // later (131 rows: the shifted copy's last row is not used), 16-23 G
    const uint64_t pol = evict_first_policy();
    uint32_t it = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++it) {
      const int r = tile / tiles_row, q0 = (tile % tiles_row) * 128;
      const int s = it % kWgStages;
      unsigned char* st = smem + s * kWgStage;
      if (it >= kWgStages && !wait(&empty[s], ((it / kWgStages) & 1) ^ 1)) break;
      const uint32_t bar = smem_u32(&full[s]);
      if (lane == 0) mbar_expect_tx(bar, 8 * kWgChunk + 8 * (kWgChunk - 16) + 8 * kWgGChunk);
      __syncwarp();
      const int kc = lane & 3, layer2 = (lane >> 2) & 1;
      if (lane < 16) {
        const int later = lane >> 3;
        bulk_load(smem_u32(st + kWgA + lane * kWgChunk),
                  a.acts + (layer2 ? 0 : plane) + tr_at(r, N, q0 - 2 + later) + kc * tr_chunk(N),
                  kWgChunk - 16 * later, bar, pol);
      } else if (lane < 24) {
        bulk_load(smem_u32(st + kWgG + (lane - 16) * kWgGChunk),
                  a.grads + (layer2 ? plane : 0) + tr_at(r, N, q0) + kc * tr_chunk(N), kWgGChunk,
                  bar, pol);
      }
    }
    // no copy is left in flight when the block ends
    const uint32_t n = it;
    for (uint32_t i = n < kWgStages ? 0 : n - kWgStages; i < n; ++i)
      (void)mbar_wait_bounded(smem_u32(&full[i % kWgStages]), (i / kWgStages) & 1);
  } else if (warp == 1) {
    if (lane == 0) {
      // MN-major: K groups of 8 positions 128 bytes apart, channel chunks
      // kWgChunk (A) or kWgGChunk (B) apart; bf16, M = 128, N = 64
      const uint32_t idesc = umma_idesc(64, true) | (1u << 15) | (1u << 16);
      uint32_t it = 0;
      for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++it) {
        const int s = it % kWgStages;
        if (!wait(&full[s], (it / kWgStages) & 1)) break;
        tmem_fence_after();
        const uint64_t da = umma_desc(smem_u32(smem + s * kWgStage + kWgA), 128, kWgChunk);
        const uint64_t db = umma_desc(smem_u32(smem + s * kWgStage + kWgG), 128, kWgGChunk);
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
#pragma unroll
          for (int tp = 0; tp < 3; ++tp)
            umma_f16(tD + 64 * tp, da + ks * 16 + 2 * tp, db + ks * 16, idesc,
                     (it == 0 && ks == 0) ? 0u : 1u);
        umma_commit(smem_u32(&empty[s]));
      }
      umma_commit(smem_u32(done));
    }
    __syncwarp();
  } else {
    // bias sums: thread u takes chunk u / 8 of [g3 | g2], positions u % 8 + 8 i
    const int u = t - 64;
    float bacc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) bacc[e] = 0.f;
    uint32_t it = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++it) {
      const int s = it % kWgStages;
      if (!wait(&full[s], (it / kWgStages) & 1)) break;
      const unsigned char* g = smem + s * kWgStage + kWgG + (u >> 3) * kWgGChunk + (u & 7) * 16;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const uint4 v = *reinterpret_cast<const uint4*>(g + i * 128);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          bacc[2 * e] += __uint_as_float(w[e] << 16);
          bacc[2 * e + 1] += __uint_as_float(w[e] & 0xFFFF0000u);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&empty[s]));
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) bacc[e] += __shfl_xor_sync(0xffffffffu, bacc[e], off);
    }
    if ((u & 7) == 0) {
      float* b = ((u >> 3) < 4 ? part3 : part2) + 5120 + 8 * ((u >> 3) & 3);
#pragma unroll
      for (int e = 0; e < 8; ++e) b[e] = bacc[e];
    }
  }
  if (warp < kWgSideWarp) {
    __syncwarp();
    // warp w holds D rows of tap 2 tp + w / 2: r2 (w even, columns of g3) or
    // r1 (w odd, columns of g2)
    if (!mbar_wait_bounded(smem_u32(done), 0)) latch(a.status, kStTimeout);
    tmem_fence_after();
    float* part = (warp & 1) ? part2 : part3;
#pragma unroll
    for (int tp = 0; tp < 3; ++tp) {
      const int k = 2 * tp + (warp >> 1);
      float v[32];
      Tmem<32>::ld(tD + 64 * tp + 32 * (warp & 1) + (static_cast<uint32_t>(32 * warp) << 16), v);
      tmem_wait_ld();
      if (k < kDnK) {
        float4* w = reinterpret_cast<float4*>(part + (k * 32 + lane) * 32);
#pragma unroll
        for (int o = 0; o < 8; ++o) w[o] = make_float4(v[4 * o], v[4 * o + 1], v[4 * o + 2], v[4 * o + 3]);
      }
    }
  }
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  if (warp == 1) tmem_dealloc(tD, 256);
}

// Sums the blocks' partial rows of every weight gradient and (FP32) the loss
// partials, in a fixed order, in one launch.  A block takes 32 columns of one
// layer's rows: 16 slices of consecutive rows are added side by side (rows / 16
// coalesced loads each, ten at a time as a tree), then the slices as a tree: the
// blocks' sums are of one sign where a gradient is large, so additions one
// after the other at nearly its full size would set its error (1.26 times as
// large against 64 bits, geometric mean of 80 FP32 gradients of 8 x 128 to 500 x
// 512 and 256 x 1024 rows).  (One thread
// per column over 1024 rows took 78 us a layer and one thread over every tile
// 32 us for the loss; this launch takes 3.2 us at 152 rows and 5.1 at 304; 8.7 with the
// rows past the last ten of a slice one after the other.)
struct DnReduceLayer {
  const float* part;   // [rows][stride]
  int rows, stride;
  float* dW;
  float* db;
};
struct DnReduceArgs {
  DnReduceLayer l[4];   // layers 3 and 2 (32 -> 32: [k][c][o], then [o]), 4 and 1 ([j][k][c], bias)
  const float* loss_part;
  int loss_n;
  size_t n;
  float* loss;
};
constexpr int kRdSlices = 16, kRdThreads = 32 * kRdSlices;
constexpr int kRdBig = (5120 + 32) / 32, kRdSide = kSdPart / 32;
constexpr int kRdBlocks = 2 * kRdBig + 2 * kRdSide + 1;
__global__ void __launch_bounds__(kRdThreads) dn_reduce_kernel(const DnReduceArgs a) {
  pdl_wait();
  __shared__ float red[kRdSlices][33];
  const int t = threadIdx.x, col32 = t & 31, slice = t >> 5;
  int b = blockIdx.x;
  if (b == kRdBlocks - 1) {   // the loss (when asked for): strided sums, then a tree
    if (!a.loss) return;
    __shared__ float ls[kRdThreads];
    float s = 0.f;
    for (int i = t; i < a.loss_n; i += kRdThreads) s += a.loss_part[i];
    ls[t] = s;
    __syncthreads();
    for (int w = kRdThreads / 2; w > 0; w >>= 1) {
      if (t < w) ls[t] += ls[t + w];
      __syncthreads();
    }
    if (t == 0) *a.loss = ls[0] / static_cast<float>(a.n);
    return;
  }
  int layer;
  if (b < 2 * kRdBig) {
    layer = b / kRdBig;
    b %= kRdBig;
  } else {
    b -= 2 * kRdBig;
    layer = 2 + b / kRdSide;
    b %= kRdSide;
  }
  const DnReduceLayer l = a.l[layer];
  const int col = b * 32 + col32;
  const int per = (l.rows + kRdSlices - 1) / kRdSlices;
  const int lo = slice * per, hi = min(l.rows, lo + per);
  float s = 0.f;
  // ten rows in flight, the last ones too, added as a tree
  for (int i = lo; i < hi; i += 10) {
    float v[10];
#pragma unroll
    for (int j = 0; j < 10; ++j)
      v[j] = i + j < hi ? l.part[static_cast<size_t>(i + j) * l.stride + col] : 0.f;
    s += (((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]))) + (v[8] + v[9]);
  }
  red[slice][col32] = s;
  __syncthreads();
  if (slice != 0) return;
  float q[kRdSlices];
#pragma unroll
  for (int i = 0; i < kRdSlices; ++i) q[i] = red[i][col32];
#pragma unroll
  for (int w = kRdSlices / 2; w > 0; w /= 2)
#pragma unroll
    for (int i = 0; i < w; ++i) q[i] += q[i + w];
  s = q[0];
  if (layer < 2) {
    if (col < 5120) {
      const int k = col / 1024, c = (col / 32) % 32, o = col % 32;
      l.dW[(o * 32 + c) * kDnK + k] = s;
    } else {
      l.db[col - 5120] = s;
    }
  } else if (col < 320) {
    const int j = col / 160, k = (col / 32) % 5, c = col % 32;
    l.dW[(layer == 2 ? j * 32 + c : c * 2 + j) * kDnK + k] = s;
  } else if (layer == 3 || col < 322) {
    l.db[col - 320] = s;
  }
}

// ------------------------------------------- LS estimate fused with the refinement
//
// For N = 1024 and sc16 input: the LS channel estimate of each antenna row
// goes straight into the network's input form.  dn_ls_rows_kernel (a warp per
// row) transforms the row's pilot symbol (radix 32 x 32 in registers, as the
// fused receiver), forms H = Y conj(X)/|X|^2 (Sec. II-C), the row RMS and
// x0 = H / rms, and writes x0 as split bf16 input rows, 16 bytes a position,
// with zero halo rows on both sides (17 KB a row, read back from L2).
// dn_xtc_kernel then runs the refinement's tiles as dn_tc_kernel does, a
// tile's 133 input rows brought by one bulk copy a tile ahead.
// Both run at the GPU's full width: one kernel that kept a row's 17 KB in
// shared memory had room for four rows per SM and left three of a slot's
// four warps idle during its transform (87 us at 16 frames of 64 antennas,
// against 10 + 54 us).  The first blocks build the weight image.
constexpr int kLsN = 1024;
constexpr int kLsHalo = 8;
constexpr int kLsXRows = kLsN + 5 * kLsHalo;               // 1064 rows of 16 bytes
constexpr int kLsWarps = 4;
constexpr int kLsEx = (kLsN + kLsN / 32) * 8;              // a warp's exchange
constexpr int kLsSmem = kLsN * 8 + kLsWarps * kLsEx;       // pass twiddles, exchanges

constexpr int kLsImgBlocks = 64;                           // blocks that build the weight image

__global__ void __launch_bounds__(32 * kLsWarps) dn_ls_rows_kernel(const KParams p, int R,
                                                                   const __nv_bfloat16* __restrict__ P,
                                                                   float* __restrict__ img,
                                                                   unsigned char* __restrict__ xrows,
                                                                   float* __restrict__ rms) {
  pdl_wait();
  constexpr int N = kLsN;
  if (blockIdx.x < kLsImgBlocks) {
    tc_image(P, img, blockIdx.x * 32 * kLsWarps + threadIdx.x, kLsImgBlocks * 32 * kLsWarps);
    return;
  }
  extern __shared__ __align__(128) unsigned char smem[];
  float2* tws = reinterpret_cast<float2*>(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* ex = reinterpret_cast<float2*>(smem + N * 8 + warp * kLsEx);
  for (int i = threadIdx.x; i < N; i += 32 * kLsWarps) tws[i] = __ldg(p.twP + i);
  __syncthreads();
  const int r = (blockIdx.x - kLsImgBlocks) * kLsWarps + warp;
  if (r >= R) return;
  const int f = r / p.M, m = r % p.M;
  float2 v[32];
  load_row<10, false>(v, row_ptr<10, false>(p, f, m, p.pilot_idx), lane, true);
  dft<32>(v, p);
  final_exchange_write<10>(v, ex, lane);
  __syncwarp();
  final_exchange_read<10>(v, ex, lane, tws);
  final_dft<10>(v, p);
  float e2 = 0.f;
#pragma unroll
  for (int e = 0; e < 32; ++e) {
    v[e] = cmul(v[e], __ldg(p.xinv + lane + 32 * e));   // bin lane + 32 e
    e2 = fmaf(v[e].x, v[e].x, fmaf(v[e].y, v[e].y, e2));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e2 += __shfl_xor_sync(0xffffffffu, e2, o);
  const float rr = sqrtf(e2 / N);
  const float inv = rr > 0.f ? 1.0f / rr : 0.f;
  if (lane == 0) rms[r] = rr;
  unsigned char* x = xrows + static_cast<size_t>(r) * kLsXRows * 16;
#pragma unroll
  for (int e = 0; e < 32; ++e)
    *reinterpret_cast<uint4*>(x + (kLsHalo + lane + 32 * e) * 16) = x_row(v[e].x * inv, v[e].y * inv);
  // halo rows (positions < 0 and >= N) are zero
  for (int j = lane; j < kLsXRows - N; j += 32)
    *reinterpret_cast<uint4*>(x + (j < kLsHalo ? j : N + j) * 16) = make_uint4(0u, 0u, 0u, 0u);
}

constexpr int kXtBytes = (kTcRows + 1) * 16;               // a tile's input rows
constexpr int kXtSlotBytes = 2 * kXtBytes + kTcActBytes;   // two tiles' inputs, activations
constexpr int kXtSmem = kTcImgBytes + kTcSlots * kXtSlotBytes + 3 * kTcSlots * 8 + 16;
static_assert(kXtSlotBytes % 16 == 0, "16-byte operand alignment");

__global__ void __launch_bounds__(128 * kTcSlots, 2) dn_xtc_kernel(const float* __restrict__ img_g,
                                                        const unsigned char* __restrict__ xrows,
                                                        const float* __restrict__ rms, int R,
                                                        float2* __restrict__ Hout, int* status, int fault) {
  pdl_wait();
  constexpr int N = kLsN;
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* wimg = smem;
  const int t = threadIdx.x;
  const int slot = t >> 7, u = t & 127, warp = t >> 5;
  unsigned char* xbuf = smem + kTcImgBytes + slot * kXtSlotBytes;
  unsigned char* act = xbuf + 2 * kXtBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kTcImgBytes + kTcSlots * kXtSlotBytes);
  uint64_t* xbars = bars + kTcSlots + 2 * slot;              // the slot's two input buffers
  uint32_t* tbase = reinterpret_cast<uint32_t*>(bars + 3 * kTcSlots);
  uint64_t* bar = &bars[slot];
  if (t == 0) {
    for (int g = 0; g < 3 * kTcSlots; ++g) mbar_init(smem_u32(&bars[g]), 1);
    fence_mbar_init();
    mbar_expect_tx(smem_u32(&bars[0]), kTcImgBytes);        // phase 0 of slot 0's barrier
    bulk_load(smem_u32(wimg), img_g, kTcImgBytes, smem_u32(&bars[0]), evict_last_policy());
  }
  __syncwarp();
  if (warp == 0) tmem_alloc(smem_u32(tbase), 32 * kTcSlots);
  // halo rows of the activation buffer stay zero
  if (u < 16) {                                     // 4 chunks x rows 0, 1, 130, 131
    const int kc = u >> 2, row = (u & 3) < 2 ? (u & 3) : kTcRows - 4 + (u & 3);
    *reinterpret_cast<uint4*>(act + kc * kTcLbo + row * 16) = make_uint4(0u, 0u, 0u, 0u);
  }
  constexpr int tiles_row = (N + kTcValid - 1) / kTcValid;
  const int tiles = R * tiles_row;
  const int stride = gridDim.x * kTcSlots;
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  const uint64_t pol = evict_first_policy();
  // a tile's input rows, from position s0 - 2 (s0: MMA row 0), into buffer b
  int fetched = 0;
  auto fetch = [&](int tile) {
    const int b = fetched++ & 1;
    const uint32_t xb = smem_u32(&xbars[b]);
    mbar_expect_tx(xb, kXtBytes);
    bulk_load(smem_u32(xbuf + b * kXtBytes),
              xrows + (static_cast<size_t>(tile / tiles_row) * kLsXRows + (tile % tiles_row) * kTcValid -
                       kTcFirst - 2 + kLsHalo) * 16,
              kXtBytes, xb, pol);
  };
  int tile = blockIdx.x * kTcSlots + slot;
  if (u == 0 && tile < tiles) {
    fetch(tile);
    // test hook: block 0's first input rows also wait for 16 bytes that no copy
    // delivers, so that the bounded wait runs out
    if (fault == 1 && blockIdx.x == 0 && slot == 0) mbar_expect_tx_only(smem_u32(&xbars[0]), 16);
  }
  const uint32_t tm = *tbase + 32 * slot + (static_cast<uint32_t>(32 * (warp & 3)) << 16);
  const uint32_t tm_mma = *tbase + 32 * slot;
  const uint32_t id32 = umma_idesc(32, true), id16 = umma_idesc(16, true);
  const uint64_t dx0 = umma_desc(smem_u32(xbuf), 16, 128);
  const uint64_t da = umma_desc(smem_u32(act), kTcLbo, 128);
  const uint64_t dw1 = umma_desc(smem_u32(wimg), 128, 256);
  const uint64_t dw = umma_desc(smem_u32(wimg), 128, 512);
  const uint64_t dones = umma_desc(smem_u32(wimg + kTcOnes), 16, 128);
  bool ok = mbar_wait_bounded(smem_u32(&bars[0]), 0);
  if (!ok) latch(status, kStTimeout);
  uint32_t phase = slot == 0 ? 1u : 0u;
  int n = 0;                                                 // tiles of this slot so far
  for (; tile < tiles; tile += stride, ++n) {
    const int b = n & 1;
    const int r = tile / tiles_row;
    const int s0 = (tile % tiles_row) * kTcValid - kTcFirst;   // position of MMA row 0
    const uint64_t dx = dx0 + (b ? kXtBytes >> 4 : 0);
    const int q = s0 + u;                                      // position of MMA row u
    const bool inside = q >= 0 && q < N;
    auto issue_wait = [&](int layer) {
      fence_proxy_async();
      tmem_fence_before();
      named_sync(1 + slot, 128);
      tmem_fence_after();
      if (u == 0) {
        if (layer == 1) {
          // this tile's rows are here; the other buffer's last reader (the
          // previous tile's output) is behind the barrier above
          if (ok && !mbar_wait_bounded(smem_u32(&xbars[b]), (n >> 1) & 1)) {
            ok = false;
            latch(status, kStTimeout);
          }
          // (after a wait that gave up its buffer may still be in flight, and
          // its barrier takes no further phase)
          if (ok && tile + stride < tiles) fetch(tile + stride);
        }
        umma_f16(tm_mma, dones, dw1 + ((kTcBias + 1024 * (layer - 1)) >> 4),
                 layer == 4 ? id16 : id32, 0u);
        if (layer == 1) {
#pragma unroll
          for (int j = 0; j < 3; ++j)
            umma_f16(tm_mma, dx + 2 * j, dw1 + ((kTcL1 + 1024 * j) >> 4), id32, 1u);
        } else {
          const int boff = layer == 2 ? kTcL2 : layer == 3 ? kTcL3 : kTcL4;
          const int tapb = layer == 4 ? 1024 : 2048;
          const uint32_t idesc = layer == 4 ? id16 : id32;
#pragma unroll
          for (int k = 0; k < 5; ++k)
#pragma unroll
            for (int kh = 0; kh < 2; ++kh)
              umma_f16(tm_mma, da + ((k * 16 + kh * 2 * kTcLbo) >> 4),
                       dw + ((boff + k * tapb + kh * 256) >> 4), idesc, 1u);
        }
        umma_commit(smem_u32(bar));
        if (ok && !mbar_wait_bounded(smem_u32(bar), phase)) {
          ok = false;
          latch(status, kStTimeout);
        }
      }
      phase ^= 1;
      tmem_fence_before();
      named_sync(1 + slot, 128);
      tmem_fence_after();
    };
    float d[32];
    issue_wait(1);
    Tmem<32>::ld(tm, d);
    tmem_wait_ld();
    tc_epilogue(d, inside, act, u);
    issue_wait(2);
    Tmem<32>::ld(tm, d);
    tmem_wait_ld();
    tc_epilogue(d, inside, act, u);
    issue_wait(3);
    Tmem<32>::ld(tm, d);
    tmem_wait_ld();
    tc_epilogue(d, inside, act, u);
    issue_wait(4);
    float y[2];
    Tmem<2>::ld(tm, y);
    tmem_wait_ld();
    if (u >= kTcFirst && u < kTcFirst + kTcValid && q < N) {
      // residual: x0 from its three bf16 terms (exact to float32); the tile's
      // row for position q is u + 2
      const __nv_bfloat16* xr = reinterpret_cast<const __nv_bfloat16*>(xbuf + b * kXtBytes + (u + 2) * 16);
      const float x_re = __bfloat162float(xr[0]) + __bfloat162float(xr[2]) + __bfloat162float(xr[4]);
      const float x_im = __bfloat162float(xr[1]) + __bfloat162float(xr[3]) + __bfloat162float(xr[5]);
      const float rr = rms[r];
      Hout[static_cast<size_t>(r) * N + q] = make_float2((x_re + y[0]) * rr, (x_im + y[1]) * rr);
    }
  }
  if (u == 0 && !ok) {
    // a wait gave up: the last copy into each buffer gets a bounded chance to land
    for (int i = fetched > 2 ? fetched - 2 : 0; i < fetched; ++i)
      (void)mbar_wait_bounded(smem_u32(&xbars[i & 1]), (i >> 1) & 1);
  }
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  if (warp == 0) tmem_dealloc(*tbase, 32 * kTcSlots);
}

// ------------------------------------------------------------- host side

// Work buffer (floats): the tensor-core weight images, forward and backward
// [kTcImgFloats each] (first, so that they keep the buffer's alignment), whose
// place the FP32 kernels' weights take in their passes; the block partials of
// the weight gradients (wp: two 32 -> 32 layers, then the two with
// two-channel sides); x0, t, y, dy [R][2][N]; a1, a2, a3, g1, g2 [R][32][N];
// rms [R].  The tensor-core training pass stores its bf16 tensors r1..r3 from
// a1 on and g3, g2, g1 from g1 on (tr_plane elements each, three to a pair of
// fp32 regions: 192 of the pair's 256 R N bytes plus the pads' 768 R).  The
// loss partials, one per tile, go to y.
struct DnWork {
  float *img, *bimg, *wt, *wp, *x0, *tt, *y, *dy, *a1, *a2, *a3, *g1, *g2, *rms;
};
constexpr int kHeadFloats = (2 * kTcImgFloats > kWtFloats ? 2 * kTcImgFloats : kWtFloats);
static_assert(kHeadFloats % 4 == 0, "16-byte alignment of what follows");
// partial rows of each weight gradient: one per block
constexpr int kMaxParts = 512;
static int wg_blocks(int R, int N) {
  const long t = static_cast<long>(R) * (N / 128);
  return t < kMaxParts ? static_cast<int>(t) : kMaxParts;
}
static size_t part_floats(int R, int N) {
  return 2 * static_cast<size_t>(wg_blocks(R, N)) * (kWgPart + kSdPart);
}
size_t dn_work_floats(int R, int N) {
  // three more than the layout takes: a buffer that is not 16-byte aligned
  // (the FP32 passes accept one) is used from its first aligned float on
  return kHeadFloats + part_floats(R, N) + static_cast<size_t>(R) * N * (4 * 2 + 5 * 32) + R + 3;
}
static DnWork dn_work(float* w, int R, int N) {
  w = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(w) + 15) & ~static_cast<uintptr_t>(15));
  DnWork d;
  const size_t s2 = static_cast<size_t>(R) * 2 * N, s32 = static_cast<size_t>(R) * 32 * N;
  d.img = w; d.bimg = w + kTcImgFloats; d.wt = w;
  d.wp = w + kHeadFloats; d.x0 = d.wp + part_floats(R, N);
  d.tt = d.x0 + s2; d.y = d.tt + s2; d.dy = d.y + s2;
  d.a1 = d.dy + s2; d.a2 = d.a1 + s32; d.a3 = d.a2 + s32; d.g1 = d.a3 + s32; d.g2 = d.g1 + s32;
  d.rms = d.g2 + s32;
  return d;
}

// Raises a kernel's dynamic shared memory limit on the current device, once for
// each device; done: the kernel's flags, one a device (past 64 every call).
template <typename K>
static cudaError_t raise_smem(K* kernel, int bytes, bool (&done)[64]) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || (dev < 64 && done[dev])) return e;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && dev < 64) done[dev] = true;
  return e;
}

// layers 1 to 3 (biases b1, b2, b3 in fp32)
static cudaError_t forward(const float* b, const DnWork& d, int R, int N, int sms, cudaStream_t st) {
  pdl_launch(dn_conv_in_kernel<false>, dim3(R * (N / kDnPos)), 256, 0, st, d.x0, d.wt + kFw1, b,
             nullptr, d.a1, N);
  cudaError_t e = conv32<false>(d.a1, d.wt + kFw2, b + 32, nullptr, d.a2, R, N, sms, st);
  if (e == cudaSuccess) e = conv32<false>(d.a2, d.wt + kFw3, b + 64, nullptr, d.a3, R, N, sms, st);
  return e;
}

cudaError_t dn_apply(const void* params, bool bf16, const float2* H, int R, int N, float* work,
                     float2* Hout, int sms, cudaStream_t st) {
  const DnWork d = dn_work(work, R, N);
  if (bf16)
    pdl_launch(dn_setup_kernel<__nv_bfloat16>, dim3(kSetupBlocks + R), 256, 0, st,
               static_cast<const __nv_bfloat16*>(params), d.wt, H, nullptr, N, d.x0, nullptr, d.rms);
  else
    pdl_launch(dn_setup_kernel<float>, dim3(kSetupBlocks + R), 256, 0, st,
               static_cast<const float*>(params), d.wt, H, nullptr, N, d.x0, nullptr, d.rms);
  const float* b = d.wt + kBias;
  const cudaError_t e = forward(b, d, R, N, sms, st);
  if (e != cudaSuccess) return e;
  DnOutArgs a{};
  a.in = d.a3;
  a.wt = d.wt + kFw4;
  a.bias = b + 96;
  a.x0 = d.x0;
  a.rms = d.rms;
  a.Hout = Hout;
  a.N = N;
  pdl_launch(dn_conv_out_kernel<false>, dim3(R * (N / kDnPos)), 256, 0, st, a);
  return cudaGetLastError();
}

cudaError_t dn_apply_tc(const void* params_bf16, const float2* H, int R, int N, float* work,
                        float2* Hout, int* status, int sms, cudaStream_t st) {
  const DnWork d = dn_work(work, R, N);
  static bool done[64] = {};
  const cudaError_t e = raise_smem(dn_tc_kernel, kTcSmem, done);
  if (e != cudaSuccess) return e;
  const auto* P = static_cast<const __nv_bfloat16*>(params_bf16);
  pdl_launch(dn_tc_setup_kernel<__nv_bfloat16>, dim3(kSetupBlocks + R), 256, 0, st, P, d.img,
             nullptr, H, nullptr, N, d.x0, nullptr, d.rms);
  // two blocks fit per SM (shared memory and the launch bounds' register cap)
  const int tiles = R * ((N + kTcValid - 1) / kTcValid);
  const int want = (tiles + kTcSlots - 1) / kTcSlots;
  const int grid = want < sms * 2 ? want : sms * 2;
  pdl_launch(dn_tc_kernel, dim3(grid), 128 * kTcSlots, kTcSmem, st, d.img, d.x0, d.rms, R, N, Hout,
             status);
  return cudaGetLastError();
}

// LS estimate of every antenna row from the pilot symbol, refined on the
// tensor cores, for N = 1024 sc16 frames (k: the plan's parameters with the
// input set); rows = n_frames * k.M.  The split input rows take the places of
// x0, t and y in the work buffer.
cudaError_t dn_ls_tc(const KParams& k, const void* params_bf16, int n_frames, float* work,
                     float2* Hout, int* status, int sms, cudaStream_t st) {
  static_assert(kLsXRows * 4 <= 4 * 2 * kLsN, "the input rows fit x0 to dy");
  const int R = n_frames * k.M;
  const DnWork d = dn_work(work, R, kLsN);
  static bool done[2][64] = {};
  cudaError_t e = raise_smem(dn_xtc_kernel, kXtSmem, done[0]);
  if (e == cudaSuccess) e = raise_smem(dn_ls_rows_kernel, kLsSmem, done[1]);
  if (e != cudaSuccess) return e;
  const auto* P = static_cast<const __nv_bfloat16*>(params_bf16);
  auto* xrows = reinterpret_cast<unsigned char*>(d.x0);
  pdl_launch(dn_ls_rows_kernel, dim3(kLsImgBlocks + (R + kLsWarps - 1) / kLsWarps), 32 * kLsWarps,
             kLsSmem, st, k, R, P, d.img, xrows, d.rms);
  const int tiles = R * ((kLsN + kTcValid - 1) / kTcValid);
  const int want = (tiles + kTcSlots - 1) / kTcSlots;
  const int grid = want < sms * 2 ? want : sms * 2;
  pdl_launch(dn_xtc_kernel, dim3(grid), 128 * kTcSlots, kXtSmem, st, d.img, xrows, d.rms, R, Hout,
             status, k.fault);
  return cudaGetLastError();
}

cudaError_t dn_grad(const float* P, const float2* Hls, const float2* Ht, int R, int N, float* work,
                    float* grad, float* loss, int sms, cudaStream_t st) {
  const DnWork d = dn_work(work, R, N);
  cudaError_t e =
      cudaFuncSetAttribute(dn_wgrad32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwSmem);
  if (e != cudaSuccess) return e;
  pdl_launch(dn_setup_kernel<float>, dim3(kSetupBlocks + R), 256, 0, st, P, d.wt, Hls, Ht, N, d.x0,
             d.tt, d.rms);
  const float* b = d.wt + kBias;
  e = forward(b, d, R, N, sms, st);
  if (e != cudaSuccess) return e;
  const size_t n = static_cast<size_t>(R) * 2 * N;
  const int tiles = R * (N / kDnPos);
  DnOutArgs o{};
  o.in = d.a3;
  o.wt = d.wt + kFw4;
  o.bias = b + 96;
  o.x0 = d.x0;
  o.tt = d.tt;
  o.dy = d.dy;
  o.part = d.y;
  o.inv_n = 2.0f / static_cast<float>(n);
  o.N = N;
  pdl_launch(dn_conv_out_kernel<true>, dim3(tiles), 256, 0, st, o);
  // two blocks per SM: of one 32 -> 32 layer, or one of each of the other two
  const int parts = wg_blocks(R, N);
  const int wgb = 2 * sms < parts ? 2 * sms : parts, sdb = sms < parts ? sms : parts;
  float* wp3 = d.wp;
  float* wp2 = wp3 + static_cast<size_t>(parts) * kWgPart;
  float* sp4 = wp2 + static_cast<size_t>(parts) * kWgPart;
  float* sp1 = sp4 + static_cast<size_t>(parts) * kSdPart;
  // layer 3: g3 = conv(dy; W4') masked -> g1; layer 2: g2 -> g2; layer 1: g1 -> g1
  pdl_launch(dn_conv_in_kernel<true>, dim3(tiles), 256, 0, st, d.dy, d.wt + kBw4, nullptr, d.a3,
             d.g1, N);
  pdl_launch(dn_wgrad32_kernel, dim3(wgb), kFwThreads, kFwSmem, st, d.g1, d.a2, R, N, wp3);
  e = conv32<true>(d.g1, d.wt + kBw3, nullptr, d.a2, d.g2, R, N, sms, st);
  if (e != cudaSuccess) return e;
  pdl_launch(dn_wgrad32_kernel, dim3(wgb), kFwThreads, kFwSmem, st, d.g2, d.a1, R, N, wp2);
  e = conv32<true>(d.g2, d.wt + kBw2, nullptr, d.a1, d.g1, R, N, sms, st);
  if (e != cudaSuccess) return e;
  pdl_launch(dn_side32_kernel, dim3(sdb, 2), 256, 0, st, d.dy, d.a3, d.x0, d.g1, R, N, sp4, sp1);
  DnReduceArgs a{};
  a.l[0] = {wp3, wgb, kWgPart, grad + kOffW3, grad + kOffB3};
  a.l[1] = {wp2, wgb, kWgPart, grad + kOffW2, grad + kOffB2};
  a.l[2] = {sp4, sdb, kSdPart, grad + kOffW4, grad + kOffB4};
  a.l[3] = {sp1, sdb, kSdPart, grad + kOffW1, grad + kOffB1};
  a.loss_part = d.y;
  a.loss_n = tiles;
  a.n = n;
  a.loss = loss;
  pdl_launch(dn_reduce_kernel, dim3(kRdBlocks), kRdThreads, 0, st, a);
  return cudaGetLastError();
}

// Gradient of the MSE on tcgen05 (bf16 operands and stored tensors, fp32
// sums): see "tensor-core training" above.
cudaError_t dn_grad_tc(const float* P32, const float2* Hls, const float2* Ht, int R, int N,
                       float* work, float* grad, float* loss, int* status, int sms, cudaStream_t st) {
  const DnWork d = dn_work(work, R, N);
  static bool done[3][64] = {};
  cudaError_t e = raise_smem(dn_tc_train_kernel<false>, kTrSmem, done[0]);
  if (e == cudaSuccess) e = raise_smem(dn_tc_train_kernel<true>, kTrSmem, done[1]);
  if (e == cudaSuccess) e = raise_smem(dn_tc_wgrad_kernel, kWgSmem, done[2]);
  if (e != cudaSuccess) return e;
  pdl_launch(dn_tc_setup_kernel<float>, dim3(2 * kSetupBlocks + R), 256, 0, st, P32, d.img, d.bimg,
             Hls, Ht, N, d.x0, d.tt, d.rms);
  const size_t n = static_cast<size_t>(R) * 2 * N;
  const int tiles = R * ((N + kTcValid - 1) / kTcValid);
  const int want = (tiles + kTcSlots - 1) / kTcSlots;
  const int grid = want < sms * 2 ? want : sms * 2;
  auto* acts = reinterpret_cast<__nv_bfloat16*>(d.a1);
  auto* grads = reinterpret_cast<__nv_bfloat16*>(d.g1);
  const size_t plane = tr_plane(R, N);
  pdl_launch(dn_tc_train_kernel<false>, dim3(grid), 128 * kTcSlots, kTrSmem, st, d.img, d.x0, d.tt,
             R, N, 2.0f / static_cast<float>(n), acts, nullptr, d.dy, d.y, status);
  pdl_launch(dn_tc_train_kernel<true>, dim3(grid), 128 * kTcSlots, kTrSmem, st, d.bimg, d.dy,
             nullptr, R, N, 0.f, acts, grads, nullptr, nullptr, status);
  const int parts = wg_blocks(R, N);
  float* wp3 = d.wp;
  float* wp2 = wp3 + static_cast<size_t>(parts) * kWgPart;
  float* sp4 = wp2 + static_cast<size_t>(parts) * kWgPart;
  float* sp1 = sp4 + static_cast<size_t>(parts) * kSdPart;
  const int wgb = sms < parts ? sms : parts;
  DnWgradArgs w;
  w.acts = acts;
  w.grads = grads;
  w.x0 = d.x0;
  w.dy = d.dy;
  w.R = R;
  w.N = N;
  w.part3 = wp3;
  w.part2 = wp2;
  w.part4 = sp4;
  w.part1 = sp1;
  w.status = status;
  w.loss_part = d.y;
  w.loss_n = tiles;
  w.n = n;
  w.loss = loss;
  pdl_launch(dn_tc_wgrad_kernel, dim3(wgb), kWgThreads, kWgSmem, st, w);
  DnReduceArgs a{};
  a.l[0] = {wp3, wgb, kWgPart, grad + kOffW3, grad + kOffB3};
  a.l[1] = {wp2, wgb, kWgPart, grad + kOffW2, grad + kOffB2};
  a.l[2] = {sp4, wgb, kSdPart, grad + kOffW4, grad + kOffB4};
  a.l[3] = {sp1, wgb, kSdPart, grad + kOffW1, grad + kOffB1};
  a.loss = nullptr;   // written by the launch above
  pdl_launch(dn_reduce_kernel, dim3(kRdBlocks), kRdThreads, 0, st, a);
  return cudaGetLastError();
}

cudaError_t dn_adam(float* p, const float* g, float* m, float* v, int step, float lr, float b1,
                    float b2, float eps, cudaStream_t st) {
  const float c1 = 1.f - powf(b1, static_cast<float>(step));
  const float c2 = 1.f - powf(b2, static_cast<float>(step));
  pdl_launch(dn_adam_kernel, dim3(44), 256, 0, st, p, g, m, v, kDnParams, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

cudaError_t dn_to_bf16(const float* p, void* q, cudaStream_t st) {
  pdl_launch(dn_bf16_kernel, dim3(44), 256, 0, st, p, static_cast<__nv_bfloat16*>(q), kDnParams);
  return cudaGetLastError();
}

}  // namespace lsas

namespace {
lsas_status dn_check(int R, int N) {
  if (R < 1 || N < 128 || N > 2048 || N % 128 != 0) return LSAS_ERR_INVALID_ARG;
  return LSAS_OK;
}
int dn_sms() {   // of the current device
  int dev = 0, sms = 1;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 1;
  return sms;
}
}  // namespace

extern "C" {

lsas_status lsas_dn_work_size(int R, int N, size_t* floats) {
  if (!floats) return LSAS_ERR_INVALID_ARG;
  const lsas_status s = dn_check(R, N);
  if (s != LSAS_OK) return s;
  *floats = lsas::dn_work_floats(R, N);
  return LSAS_OK;
}

lsas_status lsas_dn_apply(const void* d_params, int bf16, const float* d_H, int R, int N,
                          float* d_work, float* d_Hout, void* stream) {
  const lsas_status s = dn_check(R, N);
  if (s != LSAS_OK) return s;
  if (!d_params || !d_H || !d_work || !d_Hout) return LSAS_ERR_INVALID_ARG;
  if (lsas::dn_apply(d_params, bf16 != 0, reinterpret_cast<const float2*>(d_H), R, N, d_work,
                     reinterpret_cast<float2*>(d_Hout), dn_sms(),
                     static_cast<cudaStream_t>(stream)) != cudaSuccess)
    return LSAS_ERR_CUDA;
  return LSAS_OK;
}

lsas_status lsas_dn_grad(const float* d_params, const float* d_Hls, const float* d_Htrue, int R,
                         int N, float* d_work, float* d_grad, float* d_loss, void* stream) {
  const lsas_status s = dn_check(R, N);
  if (s != LSAS_OK) return s;
  if (!d_params || !d_Hls || !d_Htrue || !d_work || !d_grad || !d_loss) return LSAS_ERR_INVALID_ARG;
  if (lsas::dn_grad(d_params, reinterpret_cast<const float2*>(d_Hls),
                    reinterpret_cast<const float2*>(d_Htrue), R, N, d_work, d_grad, d_loss, dn_sms(),
                    static_cast<cudaStream_t>(stream)) != cudaSuccess)
    return LSAS_ERR_CUDA;
  return LSAS_OK;
}

lsas_status lsas_dn_adam(float* d_params, const float* d_grad, float* d_m, float* d_v, int step,
                         float lr, void* stream) {
  if (!d_params || !d_grad || !d_m || !d_v || step < 1 || !(lr > 0.f)) return LSAS_ERR_INVALID_ARG;
  if (lsas::dn_adam(d_params, d_grad, d_m, d_v, step, lr, 0.9f, 0.999f, 1e-8f,
                    static_cast<cudaStream_t>(stream)) != cudaSuccess)
    return LSAS_ERR_CUDA;
  return LSAS_OK;
}

lsas_status lsas_dn_apply_tc(const uint16_t* d_params_bf16, const float* d_H, int R, int N,
                             float* d_work, float* d_Hout, int* d_status, void* stream) {
  const lsas_status s = dn_check(R, N);
  if (s != LSAS_OK) return s;
  if (!d_params_bf16 || !d_H || !d_work || !d_Hout || !d_status) return LSAS_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(d_work) % 16 != 0) return LSAS_ERR_INVALID_ARG;
  if (lsas::dn_apply_tc(d_params_bf16, reinterpret_cast<const float2*>(d_H), R, N, d_work,
                        reinterpret_cast<float2*>(d_Hout), d_status, dn_sms(),
                        static_cast<cudaStream_t>(stream)) != cudaSuccess)
    return LSAS_ERR_CUDA;
  return LSAS_OK;
}

lsas_status lsas_dn_grad_tc(const float* d_params, const float* d_Hls, const float* d_Htrue, int R,
                            int N, float* d_work, float* d_grad, float* d_loss, int* d_status,
                            void* stream) {
  const lsas_status s = dn_check(R, N);
  if (s != LSAS_OK) return s;
  if (!d_params || !d_Hls || !d_Htrue || !d_work || !d_grad || !d_loss || !d_status)
    return LSAS_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(d_work) % 16 != 0) return LSAS_ERR_INVALID_ARG;
  if (lsas::dn_grad_tc(d_params, reinterpret_cast<const float2*>(d_Hls),
                       reinterpret_cast<const float2*>(d_Htrue), R, N, d_work, d_grad, d_loss,
                       d_status, dn_sms(), static_cast<cudaStream_t>(stream)) != cudaSuccess)
    return LSAS_ERR_CUDA;
  return LSAS_OK;
}

lsas_status lsas_dn_to_bf16(const float* d_params, uint16_t* d_params_bf16, void* stream) {
  if (!d_params || !d_params_bf16) return LSAS_ERR_INVALID_ARG;
  if (lsas::dn_to_bf16(d_params, d_params_bf16, static_cast<cudaStream_t>(stream)) != cudaSuccess)
    return LSAS_ERR_CUDA;
  return LSAS_OK;
}

}  // extern "C"

// lsas_combine.cu -- combine step of the antenna-split receiver.
//
// Sec. IV proposes distributing the receiver when one server cannot take the
// data of every antenna.  MRC splits cleanly by antenna: each shard of
// antennas forms, per subcarrier, its partial sums sum conj(H) Y (every data
// symbol) and sum |H|^2 (frame_kernel in kModePartial).  This kernel adds the
// partials of G shards in shard order g = 0 .. G-1 (a fixed order, so the
// result does not depend on scheduling), forms z = P / E and finishes as the
// fused kernel does: Gray slicer, packed bits, optional z.
#include <cfloat>

#include <type_traits>

#include "lsas_kernels.cuh"

namespace lsas {

// small blocks: a single frame's 13 x 1024 / 2 threads spread over 52 SMs
constexpr int kCombineThreads = 128;

// One thread per two consecutive points (data symbol d, subcarriers k0, k0 +
// 1) of one frame: 16 bytes of partial sums and 8 of energies per shard, so a
// warp reads and writes consecutive pieces; four neighbouring threads' codes
// make the q bytes their 8 points pack into.  Bound by memory, and for one
// frame by latency: the shards' loads are all in flight, and the launch
// overlaps the shard pass's end (pdl_launch).  60 frames of N = 2048
// in 2 shards with z: 13.6 -> 11 us; one frame of N = 1024 in 8: 5.2 -> 3.6, and
// the pair of launches 19.5 -> 14.3.
// (Before, a thread took 8 points, its 64-byte pieces apart from its
// neighbours'.)
__global__ void __launch_bounds__(kCombineThreads) combine_kernel(const KParams p) {
  const size_t per_frame = static_cast<size_t>(p.D) * p.N / 2;   // a multiple of 32
  const size_t t = static_cast<size_t>(blockIdx.x) * kCombineThreads + threadIdx.x;
  pdl_wait();
  if (t >= per_frame * static_cast<size_t>(p.nframes)) return;   // whole warps
  const int f = static_cast<int>(t / per_frame);
  const size_t r = t % per_frame;   // points 2r, 2r + 1 of the frame's d*N + k
  const int k0 = static_cast<int>((r * 2) % p.N);
  const size_t dn = static_cast<size_t>(p.D) * p.N;
  const float4* Pg = reinterpret_cast<const float4*>(p.P_in + f * dn) + r;
  const float2* Eg = reinterpret_cast<const float2*>(p.E_in + static_cast<size_t>(f) * p.N + k0);
  const size_t ps = static_cast<size_t>(p.nframes) * dn / 2, es = static_cast<size_t>(p.nframes) * p.N / 2;
  float4 P = make_float4(0.f, 0.f, 0.f, 0.f);
  float2 E = make_float2(0.f, 0.f);
  // unrolled so that several shards' loads are in flight at once (the sums
  // still run in shard order)
  // (units: the blocks that touched the frame)
  const int shards = p.units ? (f * p.upf + p.upf - 1) / p.units - f * p.upf / p.units + 1 : p.shards;
#pragma unroll 8
  for (int g = 0; g < shards; ++g) {
    const float4 v = __ldcs(Pg + g * ps);
    const float2 e = __ldg(Eg + g * es);
    P.x += v.x;
    P.y += v.y;
    P.z += v.z;
    P.w += v.w;
    E.x += e.x;
    E.y += e.y;
  }
  // zero or non-finite energy: z = 0 and the frame is flagged
  auto over = [&](float x, float y, float e) {
    const bool ok = (e > 0.f) && (e <= FLT_MAX);
    if (!ok) latch(p.status, kStDevice);
    const float ie = ok ? 1.0f / e : 0.f;
    return ok ? make_float2(x * ie, y * ie) : make_float2(0.f, 0.f);
  };
  const float2 z0 = over(P.x, P.y, E.x), z1 = over(P.z, P.w, E.y);
  if (p.eq) {
    float2* z = p.eq + f * dn + 2 * r;
    if ((reinterpret_cast<uintptr_t>(p.eq) & 15) == 0) {
      *reinterpret_cast<float4*>(z) = make_float4(z0.x, z0.y, z1.x, z1.y);
    } else {
      z[0] = z0;
      z[1] = z1;
    }
  }
  // one copy of the slicing per constellation, so that it has no branches
  auto codes_of = [&](auto tcount) {
    constexpr int T = decltype(tcount)::value;
    auto code = [&](float2 z) {
      uint32_t c = gray(count_ge<T>(z.x, p.thr));
      if (p.axes == 2) c = (c << p.wbits) | gray(count_ge<T>(z.y, p.thr));
      return c;
    };
    return (code(z0) << p.q) | code(z1);
  };
  uint32_t c2;
  switch (p.nthr) {
    case 1: c2 = codes_of(std::integral_constant<int, 1>{}); break;
    case 3: c2 = codes_of(std::integral_constant<int, 3>{}); break;
    case 7: c2 = codes_of(std::integral_constant<int, 7>{}); break;
    default: c2 = codes_of(std::integral_constant<int, kMaxThresholds>{}); break;
  }
  const int j = threadIdx.x & 3;   // of the four threads of 8 points
  uint64_t acc = static_cast<uint64_t>(c2) << ((3 - j) * 2 * p.q);
  acc |= __shfl_xor_sync(0xffffffffu, acc, 1);
  acc |= __shfl_xor_sync(0xffffffffu, acc, 2);
  uint8_t* dst = p.bits + f * (dn * p.q / 8) + (r / 4) * p.q;
  for (int i = j; i < p.q; i += 4) dst[i] = static_cast<uint8_t>(acc >> (8 * (p.q - 1 - i)));
}

cudaError_t launch_combine(const KParams& p, cudaStream_t st) {
  const size_t n = static_cast<size_t>(p.nframes) * p.D * p.N / 2;
  return pdl_launch(combine_kernel, dim3(static_cast<unsigned>((n + kCombineThreads - 1) / kCombineThreads)),
                    kCombineThreads, 0, st, p);
}

}  // namespace lsas

// lsas_sync.cu -- packet detection and output reordering around the receiver.
//
// Sec. II-B: the received baseband is correlated with the maximum-length PN
// sequence that precedes each frame to find where the packet begins.  Here
// every antenna's capture is correlated with the PN chips and the powers are
// summed over antennas; the earliest lag of the largest sum is the preamble
// start, and the frame follows the preamble.  Sec. II-C: fftshift reorders
// the subcarriers so that the zero-frequency bin sits in the middle.
#include <cooperative_groups.h>

#include <type_traits>

#include "lsas_kernels.cuh"

namespace lsas {

namespace cg = cooperative_groups;

constexpr int kPnThreads = 256;
constexpr int kPnLags = 8;     // consecutive lags per thread
constexpr int kPnSeg = 256;    // chips per staged segment
constexpr int kPnMaxCluster = 8;

// Staged samples: two float2 of padding after every eight, so that the
// threads of a quarter-warp, eight samples apart, read 16-byte pieces from
// distinct banks and every group of eight stays 16-byte aligned.
__host__ __device__ constexpr int pn_pad(int i) { return i + 2 * (i >> 3); }
__host__ __device__ constexpr int pn_lags(int ap) { return kPnLags * (kPnThreads / ap); }
__host__ __device__ constexpr int pn_row(int ap) { return pn_pad(pn_lags(ap) + kPnSeg); }
__host__ __device__ constexpr int pn_smem(int ap) {
  const int stage = ap * pn_row(ap) * 8, sums = kPnThreads * kPnLags * 8;
  return (stage > sums ? stage : sums) + kPnSeg * 8;
}

// Packet detection.  Bound by the FMA pipe: one packed FMA per (antenna, lag,
// chip).  A thread correlates one antenna at eight consecutive lags: per eight
// chips it loads eight new samples (its window of sixteen slides in registers)
// and eight chips, for 64 packed FMAs.  A block takes AP antennas side by side
// at 8 * 256 / AP lags, in rounds over the antennas; after a round the
// correlations go through shared memory and one thread per lag adds their
// powers in antenna order, so the sums are those of a single loop over
// antennas and chips.  The blocks of a cluster share a frame's lags and reduce
// (power, lag) over distributed shared memory: the largest power, the smallest
// lag on ties.  32 frames of 64 antennas, 512 lags: 39 us; one block per frame
// and one shared-memory operand pair per FMA took 425 us.
template <bool FC32, int AP>
__global__ void __launch_bounds__(kPnThreads, 2) pn_kernel(const KParams p) {
  pdl_wait();
  constexpr int LAGS = pn_lags(AP), ROW = pn_row(AP);
  static_assert(LAGS <= kPnThreads, "one thread per lag adds the powers");
  extern __shared__ __align__(128) unsigned char smem[];
  float2* chips = reinterpret_cast<float2*>(smem);            // {w, w} per chip of a segment
  float2* stage = chips + kPnSeg;                             // [AP][ROW]
  float2* sums = stage;                                       // [AP][LAGS], after a round
  __shared__ float rv[kPnThreads / 32];
  __shared__ int rt[kPnThreads / 32];
  __shared__ float cv[kPnMaxCluster];
  __shared__ int ct[kPnMaxCluster];
  const int blocks = p.grid_y;                                // of the frame's cluster
  const int f = blockIdx.x / blocks, rank = blockIdx.x % blocks;
  const int tid = threadIdx.x;
  const int ant = tid / (kPnThreads / AP), lg = tid % (kPnThreads / AP);
  cg::cluster_group cluster = cg::this_cluster();
  cluster.sync();   // every block of the cluster runs before its memory is written
  float best = -1.f;
  int best_tau = 0;
  for (int tau0 = rank * LAGS; tau0 < p.window; tau0 += blocks * LAGS) {
    float acc = 0.f;                                          // power at lag tau0 + tid
    for (int m0 = 0; m0 < p.M; m0 += AP) {
      float2 c[kPnLags];
#pragma unroll
      for (int l = 0; l < kPnLags; ++l) c[l] = make_float2(0.f, 0.f);
      const int na = min(AP, p.M - m0);
      for (int s0 = 0; s0 < p.pn_len; s0 += kPnSeg) {
        const int len = min(kPnSeg, p.pn_len - s0);
        __syncthreads();   // the previous segment or round is consumed
        for (int i = tid; i < len; i += kPnThreads) chips[i] = make_float2(p.pn[s0 + i], p.pn[s0 + i]);
        // samples tau0 + s0 .. of each antenna, zero past the capture
        const int span = LAGS + len - 1;
        // (a row's loads all in flight before its stores)
        for (int a = tid >> 5; a < na; a += kPnThreads / 32) {
          using Raw = typename std::conditional<FC32, float2, uint32_t>::type;
          constexpr int IT = (LAGS + kPnSeg - 1 + 31) / 32;
          const Raw* row = static_cast<const Raw*>(p.in) +
                           (static_cast<size_t>(f) * p.M + m0 + a) * p.cap_len + tau0 + s0;
          const int valid = min(span, p.cap_len - tau0 - s0);
          Raw v[IT];
#pragma unroll
          for (int i = 0; i < IT; ++i) {
            const int at = (tid & 31) + 32 * i;
            v[i] = Raw{};
            if (at < valid) v[i] = __ldg(row + at);
          }
#pragma unroll
          for (int i = 0; i < IT; ++i) {
            const int at = (tid & 31) + 32 * i;
            if (at < span) {
              if constexpr (FC32) stage[a * ROW + pn_pad(at)] = v[i];
              else stage[a * ROW + pn_pad(at)] = sc16_to_float2(v[i]);
            }
          }
        }
        __syncthreads();
        if (ant < na) {
          const float2* y = stage + ant * ROW + pn_pad(kPnLags * lg);
          float2 w[2 * kPnLags];
          auto load8 = [&](float2* d, int n) {   // samples n .. n + 7 of the thread's window
            const float4* q = reinterpret_cast<const float4*>(y + pn_pad(n));
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float4 v = q[i];
              d[2 * i] = make_float2(v.x, v.y);
              d[2 * i + 1] = make_float2(v.z, v.w);
            }
          };
          load8(w, 0);
          for (int n = 0; n < len; n += 8) {
            load8(w + 8, n + 8);
            const float4* ch = reinterpret_cast<const float4*>(chips + n);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float4 v = ch[i];   // chips n + 2 i, n + 2 i + 1
              if (n + 2 * i < len) {
#pragma unroll
                for (int l = 0; l < kPnLags; ++l)
                  c[l] = __ffma2_rn(make_float2(v.x, v.y), w[2 * i + l], c[l]);
              }
              if (n + 2 * i + 1 < len) {
#pragma unroll
                for (int l = 0; l < kPnLags; ++l)
                  c[l] = __ffma2_rn(make_float2(v.z, v.w), w[2 * i + 1 + l], c[l]);
              }
            }
#pragma unroll
            for (int l = 0; l < kPnLags; ++l) w[l] = w[8 + l];
          }
        }
      }
      __syncthreads();   // the samples are consumed
      if (ant < na) {
#pragma unroll
        for (int l = 0; l < kPnLags; l += 2)
          *reinterpret_cast<float4*>(sums + ant * LAGS + kPnLags * lg + l) =
              make_float4(c[l].x, c[l].y, c[l + 1].x, c[l + 1].y);
      }
      __syncthreads();
      if (tid < LAGS) {
        for (int a = 0; a < na; ++a) {
          const float2 v = sums[a * LAGS + tid];
          acc = fmaf(v.x, v.x, fmaf(v.y, v.y, acc));
        }
      }
    }
    const int tau = tau0 + tid;
    if (tid < LAGS && tau < p.window && acc > best) {   // lags grow: the earliest wins a tie
      best = acc;
      best_tau = tau;
    }
  }
  // reduction of (power, lag): warp, block, cluster
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, best, o);
    const int ot = __shfl_xor_sync(0xffffffffu, best_tau, o);
    if (ov > best || (ov == best && ot < best_tau)) {
      best = ov;
      best_tau = ot;
    }
  }
  if ((tid & 31) == 0) {
    rv[tid >> 5] = best;
    rt[tid >> 5] = best_tau;
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < kPnThreads / 32; ++w)
      if (rv[w] > best || (rv[w] == best && rt[w] < best_tau)) {
        best = rv[w];
        best_tau = rt[w];
      }
    cluster.map_shared_rank(cv, 0)[rank] = best;
    cluster.map_shared_rank(ct, 0)[rank] = best_tau;
  }
  cluster.sync();
  if (rank == 0 && tid == 0) {
    for (int w = 1; w < blocks; ++w)
      if (cv[w] > best || (cv[w] == best && ct[w] < best_tau)) {
        best = cv[w];
        best_tau = ct[w];
      }
    p.offsets[f] = best_tau;
    if (p.peaks) p.peaks[f] = best;
  }
}

// One row of blocks per (frame, antenna): copy the frame's S (N + CP) samples
// from offset + pn_len - backoff of the capture row into the contiguous frame
// layout.  A start outside the capture zero-fills the row and latches
// LSAS_ERR_DEVICE.  Bound by memory: each output moves as 16 bytes put
// together from the two aligned 16-byte pieces of the capture that hold it
// (the second comes from L1); pieces that reach past the capture buffer and
// rows that do not start on 16 bytes go word by word.  32 frames of 64
// antennas, N = 1024: 46 us (264 MB; floor 39), against 78 us with one sample
// per load.
template <bool FC32>
__global__ void __launch_bounds__(256) extract_kernel(const KParams p) {
  pdl_wait();
  constexpr int WPS = FC32 ? 2 : 1;   // 32-bit words per sample
  const int fm = blockIdx.x;
  const int f = fm / p.M;
  const int T = p.S * (p.N + p.cp);
  const int words = T * WPS;
  const long start = static_cast<long>(p.offsets_in[f]) + p.pn_len - p.backoff;
  uint32_t* dst = reinterpret_cast<uint32_t*>(p.Y_out) + static_cast<size_t>(fm) * words;
  const int t0 = blockIdx.y * blockDim.x + threadIdx.x, step = gridDim.y * blockDim.x;
  if (start < 0 || start + T > p.cap_len) {
    if (t0 == 0) latch(p.status, kStDevice);
    for (int i = t0; i < words; i += step) dst[i] = 0u;
    return;
  }
  const uint32_t* base = static_cast<const uint32_t*>(p.in);
  const uint32_t* end = base + static_cast<size_t>(p.nframes) * p.M * p.cap_len * WPS;
  const uint32_t* src = base + (static_cast<size_t>(fm) * p.cap_len + start) * WPS;
  int done = 0;
  if ((reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
    const int vecs = words / 4;
    const int sh = static_cast<int>((reinterpret_cast<uintptr_t>(src) >> 2) & 3);   // words past 16 bytes
    const uint32_t* s0 = src - sh;                                                 // aligned
#pragma unroll 4
    for (int i = t0; i < vecs; i += step) {
      const uint32_t* s = s0 + 4 * i;
      uint4 o;
      if (s >= base && s + 8 <= end) {
        const uint4 a = __ldg(reinterpret_cast<const uint4*>(s));
        const uint4 b = sh ? __ldg(reinterpret_cast<const uint4*>(s + 4)) : a;
        o = sh == 0 ? a
            : sh == 1 ? make_uint4(a.y, a.z, a.w, b.x)
            : sh == 2 ? make_uint4(a.z, a.w, b.x, b.y)
                      : make_uint4(a.w, b.x, b.y, b.z);
      } else {
        s += sh;
        o = make_uint4(s[0], s[1], s[2], s[3]);
      }
      reinterpret_cast<uint4*>(dst)[i] = o;
    }
    done = vecs * 4;
  }
  for (int i = done + t0; i < words; i += step) dst[i] = src[i];
}

// fftshift of complex rows of N (swap the halves of every row).
__global__ void shift_c64_kernel(float2* buf, size_t rows, int N) {
  pdl_wait();
  const size_t half = static_cast<size_t>(N / 2);
  const size_t n = rows * half;
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t r = i / half, k = i % half;
    float2* a = buf + r * N + k;
    const float2 t = a[0];
    a[0] = a[half];
    a[half] = t;
  }
}

// fftshift of packed bit rows (one data symbol = N q bits): swap the halves.
__global__ void shift_bytes_kernel(uint8_t* buf, size_t rows, int rowbytes) {
  pdl_wait();
  const size_t half = static_cast<size_t>(rowbytes / 2);
  const size_t n = rows * half;
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t r = i / half, k = i % half;
    uint8_t* a = buf + r * rowbytes + k;
    const uint8_t t = a[0];
    a[0] = a[half];
    a[half] = t;
  }
}

template <bool FC32, int AP>
static cudaError_t launch_pn_t(KParams p, int n_frames, int sms, cudaStream_t st) {
  // blocks per frame: a cluster that shares the lags, as long as the blocks
  // fit two an SM and each has lags of its own
  const int chunks = (p.window + pn_lags(AP) - 1) / pn_lags(AP);
  int blocks = 1;
  while (blocks < kPnMaxCluster && blocks * 2 <= chunks &&
         static_cast<long>(n_frames) * blocks < 2L * sms)
    blocks *= 2;
  p.grid_y = blocks;
  const cudaError_t e = cudaFuncSetAttribute(pn_kernel<FC32, AP>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, pn_smem(AP));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(n_frames) * blocks);
  cfg.blockDim = dim3(kPnThreads);
  cfg.dynamicSmemBytes = pn_smem(AP);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim = {static_cast<unsigned>(blocks), 1, 1};
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // as pdl_launch
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, pn_kernel<FC32, AP>, p);
}

template <bool FC32>
static cudaError_t launch_pn_f(const KParams& p, int n_frames, int sms, cudaStream_t st) {
  // antennas side by side: as many as there are, 8 to 32 (fewer antennas leave
  // room for more lags in the block)
  if (p.M > 16) return launch_pn_t<FC32, 32>(p, n_frames, sms, st);
  if (p.M > 8) return launch_pn_t<FC32, 16>(p, n_frames, sms, st);
  return launch_pn_t<FC32, 8>(p, n_frames, sms, st);
}

cudaError_t launch_pn(const KParams& p, bool fc32, int n_frames, int sms, cudaStream_t st) {
  return fc32 ? launch_pn_f<true>(p, n_frames, sms, st) : launch_pn_f<false>(p, n_frames, sms, st);
}

cudaError_t launch_extract(const KParams& p, bool fc32, int n_frames, int sms, cudaStream_t st) {
  // enough blocks to fill the GPU when there are few rows
  const int rows = n_frames * p.M;
  const int vecs = p.S * (p.N + p.cp) * (fc32 ? 2 : 1) / 4;
  int split = 1;
  while (static_cast<long>(rows) * split < 8L * sms && split * 2 * 256 <= vecs) split *= 2;
  if (fc32) pdl_launch(extract_kernel<true>, dim3(rows, split), 256, 0, st, p);
  else pdl_launch(extract_kernel<false>, dim3(rows, split), 256, 0, st, p);
  return cudaGetLastError();
}

cudaError_t launch_shift(void* buf, int kind, size_t rows, int N, int rowbytes, int sms,
                         cudaStream_t st) {
  const int grid = sms * 4;
  if (kind == 0) pdl_launch(shift_c64_kernel, dim3(grid), 256, 0, st, static_cast<float2*>(buf),
                            rows, N);
  else pdl_launch(shift_bytes_kernel, dim3(grid), 256, 0, st, static_cast<uint8_t*>(buf), rows,
                  rowbytes);
  return cudaGetLastError();
}

}  // namespace lsas

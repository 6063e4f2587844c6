// lsas_inst.cuh -- launch wrapper of one FFT length; each lsas_inst_n*.cu
// includes it once so that the six lengths compile in parallel.
#pragma once
#include "lsas_kernels.cuh"
#include "lsas_warp.cuh"
#include "lsas_hyb.cuh"
#include "lsas_pair.cuh"
#include "lsas_twin.cuh"
#include "lsas_twinpair.cuh"

namespace lsas {

// warp_kernel: the largest number of data symbols and pilots any warp of a
// block transforms for nd data symbols of `chunks` antenna chunks, with its
// pairs cut evenly over the warps (share) or as whole chunks.
inline int warp_steps_as(int chunks, int nd, bool share) {
  constexpr int NW = wgeo_warps(4);
  int most = 0;
  for (int w = 0; w < NW; ++w) {
    const int lo = w * chunks * nd / NW, hi = (w + 1) * chunks * nd / NW;
    const int whole = w < chunks ? (chunks - 1 - w) / NW + 1 : 0;
    const int n = share ? (hi > lo ? hi - lo + (hi - 1) / nd - lo / nd + 1 : 0) : whole * (nd + 1);
    most = n > most ? n : most;
  }
  return most;
}
// Cut evenly only where the chunks leave warps idle (no warp then holds two
// chunks' sums of one symbol) and it saves steps.
inline int warp_share(int chunks, int nd) {
  return chunks < wgeo_warps(4) && warp_steps_as(chunks, nd, true) < warp_steps_as(chunks, nd, false) ? 1 : 0;
}

// Forms of the two-symbol kernels: the channel given or estimated, and, at
// N <= 1024, whole frames or partial sums.  Compile-time, since these kernels
// are sensitive to what else they carry: with the grid layers' arithmetic in
// the whole-frame kernel the scale workload took 1524 us instead of 1519.  (At
// N = 2048 the opposite: 3566 us with the partial form in the same kernel,
// 3658 without.)
inline int two_symbol_form(const KParams& p) {
  return (p.H_in ? 1 : 0) + (p.mode == kModePartial ? 2 : 0);
}
template <int LOG2N, bool FC32>
static auto two_symbol_kernel(const KParams& p) -> void (*)(const KParams) {
  if constexpr (LOG2N == 11) {
    void (*const k[4])(const KParams) = {
        twinpair_kernel<LOG2N, false, FC32, false>, twinpair_kernel<LOG2N, true, FC32, false>,
        twinpair_kernel<LOG2N, false, FC32, true>, twinpair_kernel<LOG2N, true, FC32, true>};
    return k[two_symbol_form(p)];
  } else {
    void (*const k[4])(const KParams) = {twin_kernel<LOG2N, false, false>, twin_kernel<LOG2N, true, false>,
                                         twin_kernel<LOG2N, false, true>, twin_kernel<LOG2N, true, true>};
    return k[two_symbol_form(p)];
  }
}

template <int LOG2N, bool FC32>
static cudaError_t launch_t(int kind, const KParams& p, int grid, int smem, cudaStream_t st) {
  void (*fn)(const KParams) = nullptr;
  int threads = Geo<LOG2N>::TW;
  int slot = kind;   // entry of the shared-memory attribute cache below
  bool warp = false;   // warp_kernel
  if (kind == kKindFrame) {
    // fused receiver (the two-symbol kernels in a form of their own for a
    // given channel: 200 frames of 64 antennas at N = 1024 demodulate in 355 us
    // there and split, 499 in the one-symbol kernel; 16 frames 50 against 250):
    // two symbols per step, from aligned sc16 rows, for N = 1024 (and N = 256,
    // 512 with enough antennas; per-warp pipelines) and, from aligned rows of
    // either format, for N = 2048 (pipelines of warp pairs), or, opt-in at
    // N = 1024, the second FFT pass on the tensor cores; otherwise one symbol
    // per step: per-warp pipelines up to N = 1024, pipelines of warp pairs for
    // N = 2048 from sc16 rows and the warp-specialised producer/consumer kernel
    // for N = 2048 from fc32 rows
    if constexpr (LOG2N == 10 && !FC32) {
      if (p.hybrid && p.use_tma == 1) {
        fn = hyb_kernel<false>;
        threads = kHyThreads;
        smem = kHySmem;
        slot = 3;
      } else if (p.twin && p.use_tma == 1) {
        fn = two_symbol_kernel<LOG2N, FC32>(p);
        slot = 4 + two_symbol_form(p);
        threads = kTwThreads;
        smem = make_twlayout().total;
      } else {
        warp = true;
        threads = 32 * wgeo_warps(4);
      }
    } else if constexpr ((LOG2N == 8 || LOG2N == 9) && !FC32) {
      // p.twin is set by the plan only with enough antennas at these sizes
      if (p.twin && p.use_tma == 1) {
        fn = two_symbol_kernel<LOG2N, FC32>(p);
        slot = 4 + two_symbol_form(p);
        threads = kTwThreads;
        smem = make_twlayout().total;
      } else {
        warp = true;
        threads = 32 * wgeo_warps(4);
      }
    } else if constexpr (LOG2N <= 10) {
      warp = true;
      threads = 32 * wgeo_warps(FC32 ? 8 : 4);
    } else {
      if (p.twin && p.use_tma == 1) {
        fn = two_symbol_kernel<LOG2N, FC32>(p);
        threads = kTpThreads;
        smem = make_tplayout().total;
        slot = 4 + two_symbol_form(p);
      } else if constexpr (FC32) {
        fn = frame_kernel<LOG2N, FC32>;
        threads = Geo<LOG2N>::T;
      } else {
        fn = pair_kernel<LOG2N>;
        threads = kPThreads;
      }
    }
  } else {
    // symbol rows to memory: two rows at once where the bulk copies can bring
    // them (aligned sc16 rows), at most one block per SM
    bool two_rows = false;
    if constexpr (LOG2N >= 7 && LOG2N <= 10 && !FC32) two_rows = p.use_tma == 1;
    if constexpr (LOG2N >= 7 && LOG2N <= 10 && !FC32) {
      if (two_rows) {
        fn = kind == kKindEstimate ? twin_rows_kernel<LOG2N, true> : twin_rows_kernel<LOG2N, false>;
        slot = kind == kKindEstimate ? 8 : 9;
        threads = kTwThreads;
        smem = make_twlayout().total;
        grid = p.rows_grid;
      }
    }
    if (!two_rows)
      fn = kind == kKindEstimate ? estimate_kernel<LOG2N, FC32> : fft_kernel<LOG2N, FC32>;
  }
  // rows staged from the boundary before them: the per-warp kernel only
  KParams q = p;
  if (!q.units) q.nf = grid;
  q.full = grid;
  q.zsplit = 1;
  if constexpr (LOG2N <= 10) {
    if (q.use_tma == 2 && !warp) q.use_tma = 0;
    if (warp) {
      // (not an antenna shard in several data-symbol groups: twice the warps
      // then read its channel back in each; 4 antennas of float rows at N = 1024
      // 41.2 us shared, 39.8 as whole chunks)
      if (q.mode != kModePartial || q.group_z || q.D <= q.dg)
        q.share = warp_share(q.chunks, q.dg < q.D ? q.dg : q.D);
      if (q.mode == kModeRun || q.mode == kModeDemod) {
        // symbol-split the frames after the last whole wave where the parts
        // fit one data-symbol group and fewer steps a warp
        const int tail = q.nf % q.sms;
        int best = warp_steps_as(q.chunks, q.D, q.share != 0);
        for (int z = 2; z <= q.D && static_cast<long>(tail) * z <= q.sms; ++z) {
          const int part = (q.D + z - 1) / z;
          const int steps = warp_steps_as(q.chunks, part, q.share != 0);
          if (tail == 0 || part > q.dg || steps >= best) continue;
          best = steps;
          q.zsplit = z;
        }
        if (q.zsplit > 1) {
          q.full = q.nf - tail;
          grid = q.full + tail * q.zsplit;
        }
      }
      if (q.share || q.zsplit > 1 || q.use_tma == 2) {
        fn = warp_kernel<LOG2N, FC32, true>;
        slot = 10;
      } else {
        fn = warp_kernel<LOG2N, FC32, false>;
      }
    }
  } else {
    if (q.use_tma == 2) q.use_tma = 0;
    if (kind == kKindFrame && slot >= 4) q.chunks = q.M;   // an antenna a step
  }
  // raise the kernel's dynamic shared memory limit once per device
  static int limit[11][64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || smem > limit[slot][dev]) {
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) limit[slot][dev] = smem;
  }
  const int gz = q.group_z > 0 ? q.group_z : 1, gy = p.grid_y > 1 ? p.grid_y : 1;
  q.big_first = static_cast<long>(grid) * gy * gz > q.sms ? 1 : 0;
  pdl_launch(fn, dim3(grid, gy, gz), threads, smem, st, q);
  return cudaGetLastError();
}

template <int LOG2N>
cudaError_t launch_n(int kind, bool fc32, const KParams& p, int grid, int smem,
                     cudaStream_t st) {
  return fc32 ? launch_t<LOG2N, true>(kind, p, grid, smem, st)
              : launch_t<LOG2N, false>(kind, p, grid, smem, st);
}

}  // namespace lsas

// lsas_warp.cuh -- per-warp fused receiver kernel for N <= 1024.
//
// One block per frame, NW warps, each an independent pipeline over whole
// antenna-symbol rows.  Warp w takes antenna chunks w, w + NW, ... (A =
// 32/L antennas per chunk; L = N/32 lanes form one antenna's FFT team).  Per
// step a warp
//   * waits for its staging slot (bulk asynchronous copy of the CP-stripped
//     rows, the CP removal of Sec. II-B done as addressing) and refills it
//     K steps ahead,
//   * runs the radix-32 pass in registers, transposes through its own
//     padded exchange region (only __syncwarp), applies the pass twiddles
//     and runs the radix-L pass,
//   * pilot: LS estimate H = Y conj(X) / |X|^2 (Sec. II-C), written out and
//     kept in registers, and |H|^2 added to the channel energy;
//     data symbol: conj(H) Y (Sec. II-C), summed over the chunk's antennas
//     with shuffles,
//   * accumulates per subcarrier in the warp's own tensor-memory columns.
// A warp's work is a list of (chunk, data symbol) pairs.  With at least as many
// chunks as warps they are whole chunks, w, w + NW, ....  With fewer (p.share),
// the chunk-major list of all pairs is cut into NW even pieces: a warp then
// transforms the pilot of each chunk it touches and takes only its own data
// symbols, and the warp with a chunk's first data symbol alone writes its H
// and adds its energy.  No warp holds two chunks' sums of one symbol then, so
// the sums over antennas are those of one chunk per warp, bit for bit.  16
// frames of 8 antennas at N = 64, 15 symbols (one chunk): 25.2 -> 9.4 us.
// The frames after the last whole wave may run as p.zsplit blocks each, with an
// even part of the data symbols (p.full whole frames come first in the grid);
// every block transforms the pilots itself, the first writes H, and the
// results are the same bits again.  Together with the even pieces: 200 frames
// of 24 antennas, N = 256, CP 18: 75.7 -> 57.4 us.
// Rows that do not start on 16 bytes (p.use_tma = 2) are staged from the
// 16-byte boundary before them and read at their own offset.
// Warps never wait for each other inside a data-symbol group.  At a group's
// end the block adds the warps' partial sums in warp order through shared
// memory (the staging rings are idle then), forms z = P / E and demaps
// (Sec. II-B), or writes the block's partial sums (antenna split).
#pragma once

#include <type_traits>

#include "lsas_kernels.cuh"

namespace lsas {

// How a plan's rows (N samples of bps bytes behind a prefix of cp) reach shared
// memory from an input at address `at` (KParams::use_tma): 1, bulk copies, where
// every row starts on 16 bytes; 2, bulk copies from the boundary before each
// row, where the samples are aligned to themselves and that boundary lies
// within what the call may read; 0, plain loads, otherwise.  It lies there
// behind a prefix of three samples (the longest step back is 12 bytes of sc16
// or 8 of fc32), and for an aligned input read whole; the first row of an
// antenna shard (`shard`) with a shorter prefix would reach into the antenna
// before.
inline int row_staging(uintptr_t at, int N, int cp, int bps, bool shard) {
  if (at % 16 == 0 && ((N + cp) * bps) % 16 == 0 && (cp * bps) % 16 == 0) return 1;
  if (at % bps != 0) return 0;
  return cp >= 3 || (at % 16 == 0 && !shard) ? 2 : 0;
}

// Bytes that a copy from the boundary `mis` bytes before a row of `row` bytes
// takes: 16 more than the row, so that it ends in the next one.  The last row
// of a frame's antennas (the shard's, in a split launch) is staged without
// that piece, which the call may not read; its last samples come from memory.
__host__ __device__ constexpr int staged_bytes(int row, int mis, bool last) {
  return mis != 0 && !last ? row + 16 : row;
}
// Whether row s of antenna m of the M that the block takes is that last row.
__host__ __device__ constexpr bool last_row(int M, int S, int m, int s) {
  return m == M - 1 && s == S - 1;
}

#ifdef __CUDACC__


// Issue the bulk copies of one warp step (antennas of chunk c, symbol s)
// into a slot: lane 0 registers the byte count, lane a copies row a.
template <int LOG2N, bool FC32, bool DIV>
__device__ __forceinline__ void wissue(const KParams& p, int f, int c, int s,
                                       unsigned char* slot, int team_stage, uint32_t bar,
                                       uint64_t pol, int lane) {
  constexpr int N = 1 << LOG2N, A = wgeo_A(N);
  constexpr uint32_t bytes = N * (FC32 ? 8 : 4);
  const int nvalid = min(A, p.M - c * A);
  if (DIV && p.use_tma == 2) {
    // from the boundary before each row (staged_bytes)
    static_assert(A <= 32, "one row a lane");
    const unsigned char* src = row_ptr<LOG2N, FC32>(p, f, c * A + lane, s);
    const uint32_t mis = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(src) & 15);
    const uint32_t n = lane >= nvalid ? 0u : staged_bytes(bytes, mis, last_row(p.M, p.S, c * A + lane, s));
    const uint32_t total = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) mbar_expect_tx(bar, total);
    __syncwarp();
    if (n) bulk_load(smem_u32(slot + lane * team_stage), src - mis, n, bar, pol);
    return;
  }
  if (lane == 0) mbar_expect_tx(bar, bytes * nvalid);
  for (int a = lane; a < nvalid; a += 32)
    bulk_load(smem_u32(slot + a * team_stage), row_ptr<LOG2N, FC32>(p, f, c * A + a, s), bytes,
              bar, pol);
}

// Pass-1 inputs of a row staged from the 16-byte boundary before it: sample n
// sits (row mod 16) bytes further on.  A last row's last samples, which were
// not staged, come from memory.
template <int LOG2N, bool FC32>
__device__ __forceinline__ void wload_shifted(float2 (&v)[32], const unsigned char* staged,
                                              const unsigned char* row, bool last, int jt) {
  constexpr int N = 1 << LOG2N, L = N / 32, bps = FC32 ? 8 : 4;
  const int mis = static_cast<int>(reinterpret_cast<uintptr_t>(row) & 15);
  load_row<LOG2N, FC32>(v, staged + mis, jt, false);
  if (last) {
#pragma unroll
    for (int r = 0; r < 32; ++r) {
      const int n = jt + r * L;
      if ((r + 1) * L > N - 4 && (n + 1) * bps + mis > N * bps) {
        if constexpr (FC32) v[r] = __ldg(reinterpret_cast<const float2*>(row) + n);
        else v[r] = sc16_to_float2(__ldg(reinterpret_cast<const uint32_t*>(row) + n));
      }
    }
  }
}

// Symbol index of item `it` of a chunk in a data-symbol group starting at
// data symbol d0 (the pilot first when the group transforms it).
__device__ __forceinline__ int witem_symbol(const KParams& p, bool pilot_here, int d0, int it) {
  if (pilot_here) {
    if (it == 0) return p.pilot_idx;
    --it;
  }
  const int d = d0 + it;
  return d < p.pilot_idx ? d : d + 1;
}

// Load the inputs of the last FFT pass times its twiddles, held in shared
// memory as {w, -j w} pairs (two packed instructions per product).
template <int LOG2N>
__device__ __forceinline__ void wfinal_exchange_read(float2 (&v)[32], const float2* ex, int jt,
                                                     const float4* tw) {
  constexpr int L = (1 << LOG2N) / 32;
#pragma unroll
  for (int i = 0; i < 32 / L; ++i) {
    const int j = jt + i * L;
#pragma unroll
    for (int r = 0; r < L; ++r) {
      const float2 u = ex[xpad(j + 32 * r)];
      if (r == 0) {
        v[i * L + r] = u;
      } else {
        const float4 t = tw[r * 32 + j];
        v[i * L + r] = cmulw(u, make_float2(t.x, t.y), make_float2(t.z, t.w));
      }
    }
  }
}

// DIV: the form that divides a frame (p.share, p.zsplit) and takes shifted rows
// (p.use_tma = 2).  A form of its own, because its address arithmetic in every
// step costs whole frames: 760 float frames of 64 antennas at N = 1024 take 1288
// us without it and 1400 with it.
template <int LOG2N, bool FC32, bool DIV>
__global__ void __launch_bounds__(32 * wgeo_warps(FC32 ? 8 : 4), 1) warp_kernel(const KParams p) {
  pdl_wait();
  constexpr int N = 1 << LOG2N;
  constexpr int NW = wgeo_warps(FC32 ? 8 : 4);   // warps of the block
  constexpr int NT = 32 * NW;
  constexpr int TMW = wgeo_tmem_warp(NW);         // TMEM columns per warp
  constexpr int A = wgeo_A(N), OWN = wgeo_OWN(N), XS = wgeo_XS(N);
  static_assert(N <= 1024, "the per-warp kernel covers N <= 1024");
  using TmP = Tmem<2 * OWN>;   // one data symbol of partial sums (complex)
  using TmE = Tmem<OWN>;       // channel energy
  extern __shared__ __align__(128) unsigned char smem[];
  // whole frames first, then the symbol-split ones, p.zsplit blocks each
  const int bx = blockIdx.x, sx = DIV ? bx - p.full : -1;
  const int f = sx < 0 ? bx : p.full + sx / p.zsplit;
  const int tid = threadIdx.x;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // known uniform: see twinpair_kernel
  const int lane = tid & 31;
  const int alpha = lane % A;   // antenna of the chunk
  const int jt = lane / A;      // FFT team thread
  const int K = p.nslots;
  const WLayout lay = make_wlayout(N, FC32 ? 8 : 4, K, p.dg);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem) + warp * kMaxSlots;
  uint32_t* tmem_base = reinterpret_cast<uint32_t*>(smem + kWTmemAddr);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kWAbort);
  float4* tws = reinterpret_cast<float4*>(smem + lay.tw_off);
  float* ie_s = reinterpret_cast<float*>(smem + lay.ie_off);
  uint8_t* codes = smem + lay.codes_off;
  unsigned char* stage = smem + lay.warp_off + warp * lay.warp_bytes;
  float2* ex = reinterpret_cast<float2*>(stage + lay.stage_bytes) + alpha * XS;
  const int slot_bytes = A * lay.team_stage;

  for (int i = tid; i < N; i += NT) {
    const float2 w = __ldg(p.twP + i);
    tws[i] = make_float4(w.x, w.y, -w.y, w.x);
  }
  if (tid == 0) *abort_flag = 0;
  if (lane == 0 && p.use_tma) {
    for (int s = 0; s < K; ++s) mbar_init(smem_u32(&bars[s]), 1);
    fence_mbar_init();
  }
  if (warp == 0) tmem_alloc(smem_u32(tmem_base), kWTmemCols);
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  // this warp's columns: TMW columns of its lane quarter
  const uint32_t tE = *tmem_base + (static_cast<uint32_t>(32 * (warp & 3)) << 16) +
                      static_cast<uint32_t>((warp >> 2) * TMW);
  const uint32_t tP = tE + OWN;   // data symbol dl at tP + 2 OWN dl
  uint64_t pol = 0;
  if (p.use_tma) {
    if (lane == 0) pol = evict_first_policy();
    pol = __shfl_sync(0xffffffffu, pol, 0);
  }
  // zero-fill of accumulator columns, 16 (or fewer) at a time
  constexpr int ZC = OWN < 16 ? OWN : 16;
  float zero[ZC];
#pragma unroll
  for (int i = 0; i < ZC; ++i) zero[i] = 0.f;

  // start the warps of the upper half a little later, so that the two warps
  // sharing a scheduler tend to be in different phases of their steps
  // (not in a short launch, whose time it would lengthen)
  if (warp >= 4 && p.chunks >= NW) __nanosleep(1400);
  int step = 0;    // this warp's step counter over the whole frame
  int issued = 0;  // steps whose copies this warp has issued
  int slot = 0;    // ring slot of the next step to consume (step % K) ...
  int phase = 0;   // ... and its mbarrier phase ((step / K) & 1)
  // the block's data symbols: all, or an even part (per grid z index in partial
  // mode for small batches, or in a symbol split); every block transforms
  // the pilots itself, and the one with data symbol 0 writes H (and, in
  // partial mode, the channel energy)
  int d_begin = 0, d_end = p.D;
  if (p.group_z) {
    const int z = grid_layer(p);
    d_begin = z * p.D / p.group_z;
    d_end = (z + 1) * p.D / p.group_z;
  } else if (sx >= 0) {
    const int z = sx % p.zsplit;
    d_begin = z * p.D / p.zsplit;
    d_end = (z + 1) * p.D / p.zsplit;
  }
  for (int d0 = d_begin; d0 < d_end; d0 += p.dg) {
    const int nd = min(p.dg, d_end - d0);
    const bool first = d0 == d_begin;
    const bool pilot_here = fft_pilot(p) && first;
    const int pil = pilot_here ? 1 : 0;
    // this warp's pairs (chunk-major), whole chunks warp, warp + NW, ... unless shared
    const bool share = DIV && p.share;
    const int lo = warp * p.chunks * nd / NW, hi = (warp + 1) * p.chunks * nd / NW;
    const int nch = share ? (hi > lo ? (hi - 1) / nd - lo / nd + 1 : 0)
                            : (warp < p.chunks ? (p.chunks - 1 - warp) / NW + 1 : 0);
    // local chunk lc: its number, and its first and past-the-last data symbol of the group
    auto chunk_of = [&](int lc) { return share ? lo / nd + lc : warp + lc * NW; };
    auto sym_lo = [&](int lc) { return share && lc == 0 ? lo % nd : 0; };
    auto sym_hi = [&](int lc) { return share ? min(nd, hi - (lo / nd + lc) * nd) : nd; };
    if (first) {
#pragma unroll
      for (int q0 = 0; q0 < OWN; q0 += ZC) Tmem<ZC>::st(tE + q0, zero);
    }
    for (int dl = 0; dl < nd; ++dl) {
#pragma unroll
      for (int q0 = 0; q0 < 2 * OWN; q0 += ZC) Tmem<ZC>::st(tP + 2 * OWN * dl + q0, zero);
    }
    // issue cursor: local chunk and item of the next step to stage, and how
    // many steps of this group are still to be staged
    int ic = 0, iit = 0;
    int ia = sym_lo(0), iitems = sym_hi(0) - ia + pil;   // of chunk ic
    int to_issue = share ? hi - lo + nch * pil : nch * (nd + pil);
    auto advance = [&]() {
      if (++iit == iitems) {
        iit = 0;
        ++ic;
        ia = sym_lo(ic);
        iitems = sym_hi(ic) - ia + pil;
      }
    };
    if (p.use_tma && !*abort_flag) {
      // the ring held generic data (last group's reduction): order it before
      // the copies, then fill the first K slots of this group
      fence_proxy_async();
      int is = slot;
      for (int s = 0; s < K && to_issue > 0; ++s, --to_issue) {
        wissue<LOG2N, FC32, DIV>(p, f, chunk_of(ic), witem_symbol(p, pilot_here, d0 + ia, iit),
                            stage + is * slot_bytes, lay.team_stage, smem_u32(&bars[is]), pol,
                            lane);
        // test hook: the first staging phase of block 0 also waits for 16
        // bytes that no copy delivers, so its bounded wait runs out
        if (p.fault == 1 && blockIdx.x == 0 && warp == 0 && d0 == 0 && s == 0 && lane == 0)
          mbar_expect_tx_only(smem_u32(&bars[is]), 16);
        ++issued;
        is = (is + 1 == K) ? 0 : is + 1;
        advance();
      }
    }
    for (int lc = 0; lc < nch; ++lc) {
      const int c = chunk_of(lc);
      const int sa = sym_lo(lc), items = sym_hi(lc) - sa + pil;
      const bool lead = sa == 0;   // writes the chunk's H and adds its energy
      const int m = c * A + alpha;
      const bool valid = m < p.M;
      const size_t hrow = (static_cast<size_t>(f) * p.Mtot + p.m0 + blockIdx.y * p.shard_y + m) * N;
      float2 h[32];
      if (!pilot_here) {
        // channel from memory: given (demodulate) or written in the first group
        const float2* Hs = fft_pilot(p) ? p.H_out : p.H_in;
#pragma unroll
        for (int e = 0; e < 32; ++e)
          h[e] = valid ? Hs[hrow + bin_of<LOG2N>(jt, e)] : make_float2(0.f, 0.f);
        if (first && lead) {
          float2 e2[32];
#pragma unroll
          for (int e = 0; e < 32; ++e) e2[e] = make_float2(h[e].x * h[e].x + h[e].y * h[e].y, 0.f);
          reduce_scatter<A, 16>(e2, alpha);
          float acc[OWN];
          tmem_wait_st();
          TmE::ld(tE, acc);
          tmem_wait_ld();
#pragma unroll
          for (int cc = 0; cc < OWN; ++cc) acc[cc] += e2[cc].x;
          TmE::st(tE, acc);
        }
      }
      for (int it = 0; it < items; ++it, ++step) {
        float2 v[32];
        if (p.use_tma) {
          wait_slot(smem_u32(&bars[slot]), phase, abort_flag, p.status);
          if (valid) {
            const unsigned char* row = stage + slot * slot_bytes + alpha * lay.team_stage;
            if (DIV && p.use_tma == 2) {
              const int sym = witem_symbol(p, pilot_here, d0 + sa, it);
              wload_shifted<LOG2N, FC32>(v, row, row_ptr<LOG2N, FC32>(p, f, m, sym),
                                         last_row(p.M, p.S, m, sym), jt);
            } else {
              load_row<LOG2N, FC32>(v, row, jt, false);
            }
          } else {
#pragma unroll
            for (int r = 0; r < 32; ++r) v[r] = make_float2(0.f, 0.f);
          }
        } else {
          if (valid) {
            load_row<LOG2N, FC32>(v, row_ptr<LOG2N, FC32>(p, f, m, witem_symbol(p, pilot_here, d0 + sa, it)),
                                  jt, true);
          } else {
#pragma unroll
            for (int r = 0; r < 32; ++r) v[r] = make_float2(0.f, 0.f);
          }
        }
        // every lane is done with the slot (and with the exchange of the
        // previous step): refill the slot K steps ahead
        __syncwarp();
        if (p.use_tma && to_issue > 0 && !*abort_flag) {
          ++issued;
          fence_proxy_async();
          wissue<LOG2N, FC32, DIV>(p, f, chunk_of(ic), witem_symbol(p, pilot_here, d0 + ia, iit),
                              stage + slot * slot_bytes, lay.team_stage, smem_u32(&bars[slot]),
                              pol, lane);
          --to_issue;
          advance();
        }
        if (++slot == K) {
          slot = 0;
          phase ^= 1;
        }
        dft<32, true>(v, p);
        final_exchange_write<LOG2N>(v, ex, jt);
        __syncwarp();
        wfinal_exchange_read<LOG2N>(v, ex, jt, tws);
        final_dft<LOG2N, true>(v, p);
        if (pilot_here && it == 0) {
          // LS estimate H = Y conj(X) / |X|^2 (1/sqrt(N) folded into xinv)
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            const int k = bin_of<LOG2N>(jt, e);
            const float2 hv = cmul(v[e], __ldg(p.xinv + k));
            h[e] = valid ? hv : make_float2(0.f, 0.f);
            if (valid && lead && d0 == 0) p.H_out[hrow + k] = hv;
            v[e] = make_float2(h[e].x * h[e].x + h[e].y * h[e].y, 0.f);
          }
          if (lead) {
            reduce_scatter<A, 16>(v, alpha);
            float acc[OWN];
            tmem_wait_st();
            TmE::ld(tE, acc);
            tmem_wait_ld();
#pragma unroll
            for (int cc = 0; cc < OWN; ++cc) acc[cc] += v[cc].x;
            TmE::st(tE, acc);
          }
        } else {
          // MRC numerator: conj(H) Y summed over the chunk's antennas
          const int dl = sa + it - pil;
          const uint32_t tp = tP + 2 * OWN * dl;
          if constexpr (A == 1) {
            // one antenna per step: fuse the product into the accumulation,
            // P += conj(H) Y as four FMAs per subcarrier
            tmem_wait_st();
#pragma unroll
            for (int q0 = 0; q0 < 64; q0 += 32) {
              float acc[32];
              Tmem<32>::ld(tp + q0, acc);
              tmem_wait_ld();
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const float2 hh = h[q0 / 2 + i], y = v[q0 / 2 + i];
                acc[2 * i] = fmaf(hh.x, y.x, fmaf(hh.y, y.y, acc[2 * i]));
                acc[2 * i + 1] = fmaf(hh.x, y.y, fmaf(-hh.y, y.x, acc[2 * i + 1]));
              }
              Tmem<32>::st(tp + q0, acc);
            }
          } else {
            // several antennas per step: sum them with shuffles first
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] = cmulc(h[e], v[e]);
            reduce_scatter<A, 16>(v, alpha);
            tmem_wait_st();
#pragma unroll
            for (int q0 = 0; q0 < 2 * OWN; q0 += (2 * OWN < 16 ? 2 * OWN : 16)) {
              constexpr int QC = 2 * OWN < 16 ? 2 * OWN : 16;
              float acc[QC];
              Tmem<QC>::ld(tp + q0, acc);
              tmem_wait_ld();
#pragma unroll
              for (int i = 0; i < QC / 2; ++i) {
                acc[2 * i] += v[q0 / 2 + i].x;
                acc[2 * i + 1] += v[q0 / 2 + i].y;
              }
              Tmem<QC>::st(tp + q0, acc);
            }
          }
        }
      }
    }
    tmem_wait_st();
    // ---- group end: every warp's steps are done, every copy of the group
    // has landed; the per-warp regions are free for the reduction
    __syncthreads();
    if (first && (d0 == 0 || p.mode != kModePartial)) {
      float* RE = reinterpret_cast<float*>(smem + lay.warp_off);   // [NW][N]
      float e[OWN];
      TmE::ld(tE, e);
      tmem_wait_ld();
#pragma unroll
      for (int cc = 0; cc < OWN; ++cc) RE[warp * N + bin_of<LOG2N>(jt, alpha * OWN + cc)] = e[cc];
      __syncthreads();
      for (int k = tid; k < N; k += NT) {
        float E = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) E += RE[w * N + k];
        if (p.mode == kModePartial) {
          p.E_out[(static_cast<size_t>(blockIdx.y) * gridDim.x + f) * N + k] = E;
        } else {
          // zero or non-finite energy flags the frame; z = 0 there
          const bool ok = (E > 0.f) && (E <= 3.4028234663852886e38f);
          if (!ok) latch(p.status, kStDevice);
          ie_s[k] = ok ? (1.0f / E) * p.inv_sqrtN : 0.f;
        }
      }
      __syncthreads();
    }
    float2* RP = reinterpret_cast<float2*>(smem + lay.warp_off);   // [NW][dlc][N]
    const int dlc = min(nd, lay.warp_bytes / (N * 8));
    for (int dl0 = 0; dl0 < nd; dl0 += dlc) {
      const int n = min(dlc, nd - dl0);
      for (int j = 0; j < n; ++j) {
        float acc[2 * OWN];
        TmP::ld(tP + 2 * OWN * (dl0 + j), acc);
        tmem_wait_ld();
        float2* dst = RP + static_cast<size_t>(warp * dlc + j) * N;
#pragma unroll
        for (int cc = 0; cc < OWN; ++cc)
          dst[bin_of<LOG2N>(jt, alpha * OWN + cc)] = make_float2(acc[2 * cc], acc[2 * cc + 1]);
      }
      __syncthreads();
      // four items per thread at a time (their shared-memory sums all loaded
      // before the first is demapped), one copy of the loop per constellation,
      // so that the slicer inside it has no branches
      auto demap_items = [&](auto tcount) {
        constexpr int TC = decltype(tcount)::value;
        for (int idx0 = tid; idx0 < n * N; idx0 += 4 * NT) {
          float2 sv[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int idx = min(idx0 + u * NT, n * N - 1);
            const int j = idx >> LOG2N;
            const int k = idx & (N - 1);
            sv[u] = make_float2(0.f, 0.f);
#pragma unroll
            for (int w = 0; w < NW; ++w) sv[u] = cadd(sv[u], RP[static_cast<size_t>(w * dlc + j) * N + k]);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int idx = idx0 + u * NT;
            if (idx >= n * N) break;
            const int j = idx >> LOG2N;
            const int k = idx & (N - 1);
            const float2 s = sv[u];
            const int dl = dl0 + j;
            if (p.mode == kModePartial) {
              p.P_out[((static_cast<size_t>(blockIdx.y) * gridDim.x + f) * p.D + d0 + dl) * N + k] =
                  make_float2(s.x * p.inv_sqrtN, s.y * p.inv_sqrtN);
            } else {
              const float ie = ie_s[k];
              const float2 z = (ie != 0.f) ? make_float2(s.x * ie, s.y * ie) : make_float2(0.f, 0.f);
              if (p.eq) p.eq[(static_cast<size_t>(f) * p.D + d0 + dl) * N + k] = z;
              uint32_t code = gray(count_ge<TC>(z.x, p.thr));
              if (p.axes == 2) code = (code << p.wbits) | gray(count_ge<TC>(z.y, p.thr));
              codes[dl * N + k] = static_cast<uint8_t>(code);
            }
          }
        }
      };
      switch (p.nthr) {
        case 1: demap_items(std::integral_constant<int, 1>{}); break;
        case 3: demap_items(std::integral_constant<int, 3>{}); break;
        case 7: demap_items(std::integral_constant<int, 7>{}); break;
        default: demap_items(std::integral_constant<int, kMaxThresholds>{}); break;
      }
      __syncthreads();
    }
    if (p.mode != kModePartial) {
      // pack: 8 consecutive subcarriers -> q bytes
      const int items8 = nd * (N / 8);
      const size_t frame_bytes = static_cast<size_t>(p.D) * N * p.q / 8;
      for (int it = tid; it < items8; it += NT) {
        const int dl = it / (N / 8);
        const int k0 = (it % (N / 8)) * 8;
        uint64_t acc = 0;
#pragma unroll
        for (int bb = 0; bb < 8; ++bb) acc = (acc << p.q) | codes[dl * N + k0 + bb];
        uint8_t* dst = p.bits + f * frame_bytes + (static_cast<size_t>(d0 + dl) * N + k0) * p.q / 8;
        for (int jb = 0; jb < p.q; ++jb) dst[jb] = static_cast<uint8_t>(acc >> (8 * (p.q - 1 - jb)));
      }
      __syncthreads();   // codes consumed before the next group writes them
    }
  }
  if (lane == 0 && p.use_tma && *abort_flag) {
    // a wait gave up: give any copy of this warp still in flight a bounded
    // chance to land before the block's shared memory is released (copies
    // stop being issued after the abort: only the issued steps count)
    for (int s = 0; s < K && s < issued; ++s) {
      const int last = issued - 1 - ((issued - 1 - s) % K);
      (void)mbar_wait_bounded(smem_u32(&bars[last % K]), (last / K) & 1);
    }
  }
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  if (warp == 0) tmem_dealloc(*tmem_base, kWTmemCols);
}

#endif  // __CUDACC__

}  // namespace lsas

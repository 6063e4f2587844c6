"""The bytes that the per-warp kernel's row copies read, for every alignment:
inside the call's input, and, for an antenna shard (lsas_mrc_partial), inside
the shard's own rows, as the C interface promises.

A host program includes the kernel's header and goes through the rule, the
copies (from the 16-byte boundary before a row, with the piece after it but for
the last row) and the loads of what was not staged, over input addresses,
prefixes, formats and shards.  Copies must also start and end on 16 bytes.
"""

import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "lsas_warp.cuh"
using namespace lsas;
int main() {
  const int M = 3, F = 2;
  long modes[3] = {0, 0, 0}, bad = 0;
  for (int bps : {4, 8})
    for (int N : {64, 128, 1024})
      for (int S : {2, 3})
        for (int cp = 0; cp <= 9; ++cp)
          for (long at = 4096; at < 4096 + 16; at += 4)
            for (int begin = 0; begin < M; ++begin)
              for (int count = 1; begin + count <= M; ++count) {
                const long row_b = long(N + cp) * bps, ant_b = S * row_b;
                const int mode = row_staging(at, N, cp, bps, count < M);
                ++modes[mode];
                for (int f = 0; f < F; ++f)
                  for (int m = 0; m < count; ++m)
                    for (int s = 0; s < S; ++s) {
                      // what the call may read: the shard's rows of this frame (all
                      // frames' where it is whole)
                      const long frame = at + f * M * ant_b;
                      const long lo = count < M ? frame + begin * ant_b : at;
                      const long hi = count < M ? lo + count * ant_b : at + F * M * ant_b;
                      const long row = frame + (begin + m) * ant_b + s * row_b + cp * bps;
                      const int bytes = N * bps;
                      if (mode == 0) continue;
                      const int mis = mode == 2 ? int(row & 15) : 0;
                      const int n = mode == 2 ? staged_bytes(bytes, mis, last_row(count, S, m, s)) : bytes;
                      const long from = row - mis, to = from + n;
                      // every sample is staged or, in the last row, read by itself
                      const bool all = to >= row + bytes || last_row(count, S, m, s);
                      if (from < lo || to > hi || from % 16 || n % 16 || !all) ++bad;
                    }
              }
  std::printf("%ld %ld %ld %ld\n", bad, modes[0], modes[1], modes[2]);
  return 0;
}
"""


def test_copies_stay_within_the_call_s_rows(tmp_path):
    from paper_1901_07499_gb300.build import CSRC, INCLUDE, nvcc
    src = tmp_path / "staging.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "staging")
    subprocess.run([nvcc(), "-std=c++17", "-I", INCLUDE, "-I", CSRC, "-gencode",
                    "arch=compute_103a,code=sm_103a", str(src), "-o", exe], check=True)
    bad, plain, rows, shifted = map(int, subprocess.run([exe], check=True, capture_output=True,
                                                        text=True).stdout.split())
    assert plain and rows and shifted
    assert bad == 0

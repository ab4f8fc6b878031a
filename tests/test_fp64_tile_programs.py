"""Every tile that the FP64 schedules make fits the program that runs it: the
splits of fixed-size batches (fp64_tile_split) and any extent that the work
lists of grouped and chain plans may use (fp64_tile_ok), with every remainder
that an instance can leave of it. Host code only, from the library's headers."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "bgemm_internal.h"
using namespace bg;
int main() {
  long bad = 0, seen = 0;
  auto check = [&](bg_dtype dt, int mb, int nb) {
    const int per = dt == BG_C128 ? tile_program_c128(mb * nb) : tile_program_r64(mb * nb);
    ++seen;
    if (mb * nb > per * kFp64Threads) ++bad;
  };
  for (int t = 0; t < 2; ++t) {
    const bg_dtype dt = t ? BG_C128 : BG_R64;
    for (int tm = 1; tm <= 65; ++tm)
      for (int tn = 1; tn <= 65; ++tn) {
        if (!fp64_tile_ok(dt, tm, tn)) continue;
        for (int mb = 1; mb <= tm; ++mb)
          for (int nb = 1; nb <= tn; ++nb) check(dt, mb, nb);
      }
    for (int m = 1; m <= 1100; m += m < 130 ? 1 : 37)
      for (int n = 1; n <= 1100; n += n < 130 ? 1 : 37)
        for (int batch = 1; batch <= 300; batch = batch * 3 + 1) {
          int tm = 0, tn = 0;
          fp64_tile_split(dt, m, n, n, batch, 152, &tm, &tn);
          if (!fp64_tile_ok(dt, tm, tn)) ++bad;
          check(dt, (m - 1) % tm + 1, (n - 1) % tn + 1);
          check(dt, m < tm ? m : tm, n < tn ? n : tn);
        }
  }
  printf("%ld %ld\n", bad, seen);
}
"""


def test_tiles_fit_their_programs(bglib, tmp_path):
    from paper_2203_09353_gb300 import build
    src, exe = tmp_path / "tiles.cu", tmp_path / "tiles"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), "-std=c++17", f"-I{build.INCLUDE}", f"-I{build.CSRC}", str(src),
                    "-o", str(exe), build.LIB, "-Xlinker", f"-rpath={build.HERE}"], check=True)
    bad, seen = subprocess.run([str(exe)], check=True, capture_output=True,
                               text=True).stdout.split()
    assert int(bad) == 0 and int(seen) > 10 ** 6

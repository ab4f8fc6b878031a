"""The shape of the entropy's reduction (tri_shape) and the panel memory that it
asks for agree, whatever number of CTAs per walker the device allows: a plan
keeps both, and the launch takes them from the plan. Here the device cannot be
asked, as when its query fails, which gives one CTA per walker; a shape that
needs panel vectors in device memory says so itself. Host code only."""
import subprocess

import paper_2203_09353_gb300.build as build

SOURCE = r"""
#include <cstdio>
#include "bgemm_internal.h"
int main() {
  int bad = 0;
  for (int n = 2; n <= 1024; n *= 2)
    for (long walkers : {0L, 1L, 4L, 16L, 76L, 65535L}) {
      bg::TriShape s;
      bg::tri_shape(walkers, n, 152, &s);
      const bool device_panel = n > 96 && (s.cl > 1 || !s.vws);
      bad += (s.panel > 0) != device_panel || s.panel % 16 != 0;
      bad += s.warps < 4 || s.smem == 0 || s.smem > 227 * 1024 || s.cl < 1 || s.cl > 8;
      bad += n > 96 && (long)s.own * s.cl < n;
    }
  printf("%d\n", bad);
}
"""


def test_shape_and_panel_memory_agree(bglib, tmp_path):
    src, exe = tmp_path / "shape.cu", tmp_path / "shape"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), "-std=c++17", f"-I{build.INCLUDE}", f"-I{build.CSRC}", str(src),
                    "-o", str(exe), build.LIB, "-Xlinker", f"-rpath={build.HERE}"], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert out.strip() == "0"

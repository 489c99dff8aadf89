"""Cutting right-hand sides into blocks, on the host. The persistent batch launch: every item an operator
is cut into runs a body whose buffers fit in what the launch is sized by, for any number of right-hand
sides. FP64 blocks: every width chosen has a kernel instance, and no other computes less."""
import os
import subprocess

import pytest

from paper_1809_10573_gb300 import build as B

PROGRAM = r"""
#include <cstdio>
#include "batch_items.cuh"
#include "node_launch.h"
using namespace idbf;
template <class P>
int check(const char* name) {
  int bad = 0;
  const int shapes[][5] = {{16, 20, 9, 12, 15}, {63, 64, 30, 41, 57}, {200, 210, 100, 150, 180}, {7, 9, 3, 5, 4}};
  for (const auto& s : shapes)
    for (int kind = KIND_V; kind <= KIND_U; ++kind) {
      LevelInfo li;
      li.kind = kind;
      li.max_in = s[0]; li.max_out = s[1]; li.max_rows = s[2]; li.max_cols = s[3]; li.max_rows_pair = s[4];
      for (int rb : {1, 4, 8, 16, 32}) {
        if (rb > bat::max_rb<P>()) continue;
        for (int64_t R = 1; R <= 200; ++R) {
          const int width = node::even_block(R, rb);
          const size_t have = bat::items_smem<P>(li, R, width);
          for (int64_t r0 = 0; r0 < R; r0 += width) {
            const int n = (int)std::min<int64_t>(width, R - r0), pw = bat::pass_width<P>(n);
            size_t need = 0;
            int held = 0;
            bat::at_width<P>(pw, [&](auto w, auto, auto) {
              held = decltype(w)::value;
              need = node::fwd_smem<P, decltype(w)::value>(li.max_in, li.max_out, li.max_rows, li.max_cols, li.max_rows_pair,
                                                           kind == KIND_U);
            });
            if (held < pw || need > have) {
              if (!bad++) printf("%s kind %d rb %d R %d item of %d: needs %zu, has %zu\n", name, kind, rb, (int)R, n, need, have);
            }
          }
        }
      }
    }
  return bad;
}
int widths() {  // FP64 blocks: of the widths that have an instance, and none of 3 to 8 computes less
  int bad = 0;
  for (int64_t R = 1; R <= 5000; ++R) {
    const int w = node::fitting_block(R);
    int64_t least = (R + w - 1) / w * w;
    for (int v = 3; v <= 8; ++v) least = std::min(least, (R + v - 1) / v * v);
    const bool instance = w == 1 || w == 2 || w == 3 || w == 4 || w == 5 || w == 7;
    if ((!instance || (R + w - 1) / w * w != least) && !bad++) printf("R %d: width %d\n", (int)R, w);
  }
  return bad;
}
int main() { return check<FP32P>("fp32") + check<DF64P>("df64") + check<FP64P>("fp64") + widths() ? 1 : 0; }
"""


def test_every_item_fits_in_the_shared_memory_its_launch_is_sized_by(tmp_path):
    nvcc = B._nvcc()
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "items.cu", tmp_path / "items"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, *B.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", B.INCLUDE, "-I", B.CSRC, str(src), "-o",
                    str(exe)], check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

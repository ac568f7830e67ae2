"""Where the forward query's dropped reads fall: a sample outside a grid reads the eight corners
of a cell at the start of the staged nodes, with the strides of that grid's box."""
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2308_02494_gb300" / "csrc"
PROGRAM = r"""
#include <cstdio>
#include "fwd_box.cuh"
using namespace srn;

// Group [lo, hi] and a grid that scales and moves each axis: the last byte of the dropped read.
template <int K, int C, bool F32>
int check() {
  const int smem = fwd_smem(233472, K, F32);   // an SM has 228 KB
  const uint32_t pool = (uint32_t)(smem - FwdLay<K, C, F32, true>::POOL) / (4 * C) * (4 * C);
  int bad = 0;
  for (int R = 2; R <= 64; ++R)
    for (int miss = 0; miss < 8; ++miss)
      for (int part = 0; part < 2; ++part) {   // the whole domain, or a thin slab
        const float lo[3] = {-1.f, -1.f, part ? -0.06f : -1.f}, hi[3] = {1.f, 1.f, part ? 0.06f : 1.f};
        float g[12];   // column pairs of the x and y rows, then the z row
        for (int k = 0; k < 4; ++k)
          for (int d = 0; d < 3; ++d) {
            const float v = k == 3 ? (miss >> d & 1 ? 3.5f : 0.f) : k == d ? 1.f : 0.f;
            if (d < 2) g[2 * k + d] = v; else g[8 + k] = v;
          }
        uint32_t blo = 0xabcdefu, bn = 0x404040u;
        const bool any = sample_box(lo, hi, g, R, blo, bn);
        if (any != (miss == 0)) { std::printf("R %d miss %d: any %d\n", R, miss, any); ++bad; }
        if (any) continue;   // staged where it fits; else its corners come from the grid
        const FwdBox q = fwd_box<C>(blo, bn, 0u);
        const uint32_t last = q.oz + q.oy + 2 * 4 * C;   // bytes from the first staged node on
        if (last > pool) {
          std::printf("K %d C %d f32 %d R %d miss %d: reads %u of %u bytes\n", K, C, F32, R, miss, last, pool);
          ++bad;
        }
      }
  return bad;
}
template <int K>
int widths() {
  return check<K, 1, false>() + check<K, 2, false>() + check<K, 1, true>() + check<K, 2, true>();
}
int main() { return widths<16>() + widths<32>() + widths<64>() + widths<128>() != 0; }
"""


def test_dropped_reads_stay_in_the_staged_nodes(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not Path(nvcc).exists():
        pytest.skip("no nvcc")
    src = tmp_path / "boxes.cu"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                    f"-I{CSRC}", "-o", str(tmp_path / "boxes"), str(src)], check=True)
    r = subprocess.run([str(tmp_path / "boxes")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[:2000]

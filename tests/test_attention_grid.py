"""The attention kernels' blocks, compiled for the host: every (tile, sequence, head) once, tiles slowest, and no limit
below the one on rows."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2608_18469_b200", "csrc")
PROGRAM = r"""
#define __host__
#define __device__
#include "attention_grid.cuh"
#include <cstdio>
using namespace erase;
int main() {
  const int cases[][3] = {{1, 1, 1}, {5, 7, 2}, {12, 8, 8}, {1, 3, 70000}, {3, 70000, 1}};
  for (auto& c : cases) {
    unsigned block = 0;
    for (int tile = 0; tile < c[2]; tile++)
      for (int seq = 0; seq < c[1]; seq++)
        for (int head = 0; head < c[0]; head++, block++) {
          const AttnPlace p = attn_place(block, c[0], c[1]);
          if (p.tile != tile || p.seq != seq || p.head != head) return 1;
        }
    if (block != attn_blocks(c[0], c[1], c[2])) return 2;
  }
  // the most rows a model may have, as one sequence: 2^30 positions, 16 heads
  const AttnPlace last = attn_place((unsigned)(attn_blocks(16, 1, 1 << 23) - 1), 16, 1);
  if (attn_blocks(16, 1, 1 << 23) > ATTN_MAX_BLOCKS || last.tile != (1 << 23) - 1 || last.head != 15) return 3;
  return 0;
}
"""


def test_blocks_cover_every_tile_once(tmp_path):
    src, exe = tmp_path / "grid.cpp", tmp_path / "grid"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_kernels_take_their_place_from_it():
    text = open(os.path.join(CSRC, "attention_tc.cu")).read()
    assert text.count("attn_place(blockIdx.x,") == 3 and "blockIdx.y" not in text and "blockIdx.z" not in text

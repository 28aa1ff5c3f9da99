"""The staging of SMO-2 block inverses in the FP64 sweep (csrc/blocks.cuh), compiled for the host:
every copy of every legal block shape fits the stage that its level gives it, starts on 16 bytes and
stays inside the block's padded rows."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "blocks.cuh"
#include <initializer_list>
#include <cstdio>
using namespace ccm::dev;
int main() {
  long bad = 0;
  for (int core = 8; core <= 128; ++core) for (int over = 0; over <= 64; ++over) {
    const int ext = core + 2 * over;                    // the most a level's blocks can have
    const size_t stage = block_stage_bytes(ext, core, 8, true);
    for (int ne = 1; ne <= ext; ++ne) for (int nc : {1, 7, core}) {
      if (nc > ne || nc > core) continue;
      const int e0 = block_split(ne);
      const long room = ((long)ne * nc + 3) & ~3L;      // values of a block with its padding
      const size_t a = block_copy_bytes(e0, nc, 8), b = block_copy_bytes(ne - e0, nc, 8);
      const bool ok = e0 >= 0 && e0 <= ne && a <= stage && b <= stage && (long)e0 * nc * 8 % (e0 < ne ? 16 : 1) == 0 &&
                      a <= room * 8 && (long)e0 * nc * 8 + (long)b <= room * 8;
      if (!ok && bad++ < 5) printf("core %d overlap %d rows %d columns %d: %zu + %zu of %zu\n", core, over, ne, nc, a, b, stage);
    }
    if (block_stage_bytes(ext, core, 4, false) < block_copy_bytes(ext, core, 4)) ++bad;
  }
  printf("%ld\n", bad);
}
'''


def test_every_part_fits_its_stage(tmp_path):
    (tmp_path / "h.cpp").write_text(SRC)
    inc = os.path.join(ROOT, "paper_2504_00724_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", inc, str(tmp_path / "h.cpp"), "-o", str(tmp_path / "h")], check=True)
    out = subprocess.run([str(tmp_path / "h")], capture_output=True, text=True, check=True).stdout.split("\n")
    assert out[-2] == "0", out

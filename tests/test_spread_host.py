"""How many blocks of a transform an SM may hold: csrc/wino_spread.h compiled for the host."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include <cstdlib>
#include "wino_spread.h"
using namespace wino;
// SM's shared memory 228 KB, of which a block takes 1 KB more than it asks for
static int fit(size_t smem) { return (int)(228 * 1024 / (smem + 1024)); }
int main(int argc, char** argv) {
  if (argc == 5) { std::printf("%d", out_blocks_per_sm(atol(argv[1]), atol(argv[2]), atoi(argv[3]), atoi(argv[4]))); return 0; }
  long bad = 0;
  for (int per = 2; per <= 8; ++per) bad += fit(spread_smem(100, per)) != per;
  bad += spread_smem(5000, 0) != 5000 || spread_smem(200000, 3) != 200000;
  // whatever the choice, no block has to wait for another's place
  for (int sms : {1, 132, 148}) for (long units = 1; units < 3000; ++units) {
    for (int K : {64, 128}) for (long sums : {0l, 2200000l, 2200001l}) {
      const int in = in_blocks_per_sm(units, K, sums, sms);
      const bool limit = units > sms && units <= 8l * sms && (K == 64 || sums <= 2200000l);
      bad += limit ? in < 2 || in > 8 || (long)in * sms < units : in != 0;
    }
    for (long items = 0; items < 700; items += 3) for (int C : {64, 128, 144, 512}) {
      const int out = out_blocks_per_sm(units, items, C, sms);
      bad += out != 0 && (out < 2 || out > 8 || (long)out * sms < units);
    }
  }
  std::printf("%ld", bad);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("spread")
    (d / "spread.cpp").write_text(PROGRAM)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-I",
                           os.path.join(ROOT, "paper_2002_10711_b200", "csrc"), str(d / "spread.cpp"), "-o", str(d / "spread")])
    return lambda *args: int(subprocess.check_output([str(d / "spread"), *map(str, args)]))


def test_all_blocks_find_a_place(program):
    assert program() == 0


# blocks of the output transform, work items and channels of the GEMM in front of it, SMs -> blocks per SM
@pytest.mark.parametrize("units,items,C,want", [
    (64, 128, 512, 2), (128, 128, 512, 2), (144, 128, 384, 2),     # 20 free SMs, which a whole grid would fill
    (100, 144, 64, 3),
    (144, 64, 256, 0), (40, 128, 512, 0),                          # room for all of them
    (296, 72, 128, 3), (256, 36, 128, 3), (256, 72, 192, 2),       # two behind a short GEMM
    (600, 108, 256, 5), (1200, 108, 256, 0),
    (400, 216, 128, 0), (600, 288, 128, 5),                        # uneven and even GEMMs
    (400, 0, 64, 0),                                               # no tensor-core GEMM
])
def test_output_blocks_per_sm(program, units, items, C, want):
    assert program(units, items, C, 148) == want

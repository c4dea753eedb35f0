"""Host check of the particle kernels' walk over a share of slots, up to the end
of the slot range (counts are below 2^31)."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1906_06306_gb300", "csrc")

# Prints, for a share [a, b): the first and last slot taken, how many slots the
# block's threads take in all, and the number of batches; gives up after 2^24.
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "pic_slots.h"
using namespace pic;
int main(int argc, char** argv) {
  const long long a = atoll(argv[1]), b = atoll(argv[2]);
  const int threads = atoi(argv[3]), line = atoi(argv[4]), quad = atoi(argv[5]);
  long long first = -1, last = -1, taken = 0, batches = 0;
  for (SlotWalk w = slot_walk((int)a, (int)b, threads, line, quad); w.more(); w.next(threads)) {
    if (++batches > 1 << 24) break;
    for (int t = 0; t < threads; ++t) {
      const slot_t p = w.slot(t);
      if (!w.mine(p)) continue;
      if (first < 0) first = p;
      if (last >= 0 && (long long)p != last + 1) return 2;
      last = p;
      ++taken;
    }
  }
  printf("%lld %lld %lld %lld\n", first, last, taken, batches);
}
"""
TOP = 2 ** 31 - 1


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    d = tmp_path_factory.mktemp("slots")
    (d / "walk.cpp").write_text(PROGRAM)
    exe = str(d / "walk")
    subprocess.run(["g++", "-std=c++17", "-O1", f"-I{CSRC}", str(d / "walk.cpp"), "-o", exe], check=True)

    def run(*args):
        r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, check=True, timeout=60)
        return tuple(map(int, r.stdout.split()))

    return run


@pytest.mark.parametrize("line,quad", [(0, 0), (1, 0), (0, 1)])
@pytest.mark.parametrize("a,b", [(0, 1), (0, 256), (0, 257), (5, 5), (31, 32), (33, 289), (100, 1000),
                                 (TOP - 1, TOP), (TOP - 255, TOP), (TOP - 256, TOP), (TOP - 257, TOP),
                                 (TOP - 100_000, TOP), (TOP - 1000, TOP - 256), (TOP, TOP)])
def test_every_slot_of_a_share_once(walk, a, b, line, quad):
    first, last, taken, batches = walk(a, b, 256, line, quad)
    plain = -(-(b - a) // 256)
    assert taken == b - a
    assert (first, last) == ((a, b - 1) if b > a else (-1, -1))
    assert plain <= batches <= plain + quad  # a line start takes no batch more

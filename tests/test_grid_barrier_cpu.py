"""The rules of the persistent kernel's grid barrier (csrc/barrier_count.h), run on the CPU: blocks
that arrive and poll in random order, over the point where the 32-bit counter wraps."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_08728_gb300", "csrc")


def _run(tmp_path, source, *args):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(source)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    return subprocess.run([str(exe), *map(str, args)], stdout=subprocess.PIPE, check=True, text=True).stdout.split()


WRAP = r"""
#include "barrier_count.h"
#include <cstdio>
#include <cstdlib>
#include <vector>
int main(int, char** v) {
  const unsigned blocks = atoi(v[1]), gen0 = 0xffffffffu / blocks - 3;
  std::vector<unsigned> gen(blocks, gen0);       // barriers that each block has passed
  std::vector<char> waits(blocks, 0);
  unsigned count = gen0 * blocks, rng = 12345, steps = 0;
  long early = 0, passed = 0, arrived = 0;
  while (passed < (long)blocks * 8 && ++steps < 50000000u) {
    rng = rng * 1664525u + 1013904223u;
    const unsigned b = (rng >> 8) % blocks;
    if (!waits[b]) {
      if (gen[b] == gen0 + 8) continue;
      ++count, ++arrived, waits[b] = 1;
    } else if (kcmg::count_reached(count, (gen[b] + 1) * blocks)) {
      early += arrived < (long)blocks * (gen[b] - gen0 + 1);
      waits[b] = 0, ++gen[b], ++passed;
    }
  }
  printf("%ld %ld\n", early, passed);
}
"""


@pytest.mark.parametrize("blocks", [2, 19, 152])
def test_nobody_passes_early_or_stays_when_the_counter_wraps(tmp_path, blocks):
    early, passed = _run(tmp_path, WRAP, blocks)
    assert (int(early), int(passed)) == (0, 8 * blocks)


LIMIT = r"""
#include "barrier_count.h"
#include <cstdio>
#include <cstdlib>
int main(int, char** v) {   // polls until a block gives up, with a step of block 0 every so many polls
  const unsigned every = atoi(v[1]);
  unsigned polls = 0, seen = 0, n = 0;
  while (n < (1u << 27)) {
    ++n;
    if ((++polls & 1023) == 0 && kcmg::give_up(polls, seen, every ? n / every : 7)) break;
  }
  printf("%u\n", n);
}
"""


@pytest.mark.parametrize("every", [0, 1, 1 << 16, 1 << 22])
def test_a_block_waits_as_long_as_block_0_reports_progress(tmp_path, every):
    n = int(_run(tmp_path, LIMIT, every)[0])
    assert n == 1 << 27 if every else 1 << 23 < n <= (1 << 23) + 2048

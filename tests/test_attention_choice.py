"""The host's choice among the attention kernels on CTA pairs (csrc/attention_choice.h) on its own, compiled without CUDA."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "attention_choice.h"

// resident[1..4] items keys most -> ranges; keys items pairs -> whether pairs pay; prefix -> row, keys of its blocks
int main(int argc, char** argv) {
  if (argc == 8) {
    const int resident[5] = {0, atoi(argv[1]), atoi(argv[2]), atoi(argv[3]), atoi(argv[4])};
    printf("%d\n", phyai::choose_pair_ranges(resident, atoi(argv[5]), atoi(argv[6]), atoi(argv[7])));
  } else if (argc == 4) {
    printf("%d\n", phyai::pairs_pay(atoi(argv[1]), atoi(argv[2]), atoi(argv[3])) ? 1 : 0);
  } else {
    const int P = atoi(argv[1]);
    for (int sb = 0; sb < (P + 63) / 64; ++sb) {
      const phyai::PrefixBlock k = phyai::prefix_block(P, sb);
      printf("%d %llx\n", k.row, (unsigned long long)k.keys);
    }
  }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("attention_choice")
    src, exe = d / "t.cpp", d / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-I", os.path.join(ROOT, "paper_2608_03682_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    return lambda *a: subprocess.run([str(exe), *map(str, a)], capture_output=True, text=True, check=True, timeout=60).stdout.split()


@pytest.mark.parametrize("resident,items,keys,most,ranges", [
    ((74, 36, 22, 15), 8, 867, 4, 4), ((74, 36, 22, 15), 16, 867, 4, 3), ((74, 36, 22, 15), 16, 867, 2, 2), ((74, 36, 22, 15), 128, 1019, 4, 1),
    # a device (or a part of one) that holds no cluster of some sizes, of all but one, of none
    ((-1, 36, 22, 15), 128, 1019, 4, 2), ((-1, 36, 0, 0), 128, 1019, 4, 2), ((-1, -1, -1, -1), 8, 867, 4, 0), ((0, 0, 0, 15), 8, 867, 3, 0)])
def test_key_ranges(program, resident, items, keys, most, ranges):
    cost = lambda c: -(-items // resident[c - 1]) * ((5.5 if c > 1 else 4.0) + -(-keys // (128 * c)))
    options = [c for c in range(1, most + 1) if resident[c - 1] > 0]
    assert ranges == (min(options, key=cost) if options else 0)
    assert program(*resident, items, keys, most) == [str(ranges)]


@pytest.mark.parametrize("keys,items,pays", [(60, 38, 0), (64, 40, 0), (60, 56, 0), (0, 60, 0), (64, 72, 1), (65, 36, 0), (65, 38, 1), (255, 37, 1),
                                              (255, 36, 0), (256, 2, 1), (968, 2, 1)])
def test_small_caches_take_the_pairs_where_they_are_faster(program, keys, items, pays):
    assert program(keys, items, 74) == [str(pays)]


@pytest.mark.parametrize("prefix", [*range(0, 200), 255, 256, 257, 816, 967, 968])
def test_blocks_of_a_prefix(program, prefix):
    """Every key is in one block; the 64 rows of a block end in the prefix, and begin there unless it has fewer."""
    v = program(prefix)
    blocks = [(int(row), int(keys, 16)) for row, keys in zip(v[::2], v[1::2])]
    assert [row + c for row, keys in blocks for c in range(64) if keys >> c & 1] == list(range(prefix))
    for row, keys in blocks:
        assert keys and row + 64 <= prefix and (row >= 0 or prefix < 64)

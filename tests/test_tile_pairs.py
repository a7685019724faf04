"""The values of the tuning knob "ntt_shape" name the same tile pairs in every
version (a saved tuning keeps its pair), and the default is one of them."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2006_10091_gb300", "csrc")
# (column pass bits, rows per tile, row pass bits, rows per tile) of values 0, 1, 2
PAIRS = {12: [(6, 5, 6, 5), (5, 6, 7, 4), (3, 8, 9, 2)], 13: [(7, 4, 6, 5), (6, 5, 7, 4), (4, 7, 9, 2)],
         14: [(7, 4, 7, 4), (8, 3, 6, 5), (5, 6, 9, 2)], 15: [(8, 4, 7, 4), (7, 4, 8, 3), (6, 5, 9, 2)],
         16: [(8, 4, 8, 3), (7, 4, 9, 2), (6, 5, 10, 1)]}
DEFAULT = {11: 0, 12: 0, 13: 0, 14: 2, 15: 1, 16: 2}
SOURCE = """
#include <cstdio>
#include "tile_pairs.h"
template <int L> void row() {
  for (int s = 0; s < 3; ++s)
    he::with_pair<L>(s, [&](auto p) { return std::printf("%d %d %d %d %d %d\\n", L, s, p.m1, p.k1, p.m2, p.k2); });
  std::printf("%d %d\\n", L, he::default_pair(L));
}
int main() { row<12>(); row<13>(); row<14>(); row<15>(); row<16>(); }
"""


def test_a_value_keeps_its_pair(tmp_path):
    (tmp_path / "pairs.cpp").write_text(SOURCE)
    exe = str(tmp_path / "pairs")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", exe, str(tmp_path / "pairs.cpp")], check=True)
    want = []
    for log_n, pairs in PAIRS.items():
        want += [[log_n, s, *p] for s, p in enumerate(pairs)] + [[log_n, DEFAULT[log_n]]]
    got = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    assert [[int(x) for x in line.split()] for line in got.splitlines()] == want


@pytest.mark.gpu
def test_default_value_per_ring_size():
    import paper_2006_10091_gb300 as he
    for log_n, value in DEFAULT.items():
        ctx = he.Context(log_n, 2, 40, 1, 60, 2.0 ** 30, seed=1)
        assert he.he_get_tuning(ctx, "ntt_shape") == value
        ctx.close()

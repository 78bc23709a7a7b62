"""Who takes an odd last row tile (csrc/row_tiles.h), for every number of row tiles and of SMs: each side of a pair of launches has
CTAs, two launches that run at the same time have SMs of their own, and no whole CTA group is lost to the rounding."""
import os
import subprocess

import pytest

from paper_2603_08088_b200.build import CSRC

PROGRAM = """
#include <cstdio>
#include "row_tiles.h"
int main() {
  for (int d = 64; d <= 128; d += 64)
    for (int sms = 1; sms <= 160; ++sms)
      for (int n = 1; n <= 256; ++n) {
        const tv::OddRowTile o = tv::odd_row_tile(sms, n, d);
        std::printf("%d %d %d %d %d %d %d %d\\n", d, sms, n, o.beside_groups, o.odd_groups, o.behind_groups, o.split_from, o.behind_from);
      }
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    at = tmp_path_factory.mktemp("row_tiles")
    (at / "plans.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(at / "plans.cpp"), "-o", str(at / "plans")], check=True)
    lines = subprocess.run([str(at / "plans")], check=True, capture_output=True, text=True).stdout.splitlines()
    return [tuple(map(int, line.split())) for line in lines]


def test_both_sides_of_an_odd_row_tile_have_their_sms(plans):
    assert len(plans) == 2 * 160 * 256
    for d, sms, n, beside, odd, behind, split_from, behind_from in plans:
        pairs, at = n // 2, (d, sms, n)
        if n % 2 == 0 or pairs == 0 or pairs > sms:
            assert (beside, odd, behind) == (0, 0, 0), at
            continue
        assert behind == sms // pairs >= 1, at
        if split_from < behind_from:
            assert beside >= 1 and odd >= 1 and beside * pairs + odd == sms, at
            assert sms // (pairs + 1) < beside <= behind, at             # more groups than one launch with the odd row tile has
        else:
            assert (beside, odd) == (0, 0) and 0 < split_from == behind_from, at


def test_shares_of_a_whole_gpu(plans):
    """148 SMs: narrow head groups beside each other, and all 148 SMs for the pairs of wide ones, where a share of them would lose a
    group of 74, or leave one CTA for the last row tile."""
    at = {(d, n): rest for d, sms, n, *rest in plans if sms == 148}
    assert at[128, 3] == [84, 64, 148, 12, 100] and at[64, 3] == [94, 54, 148, 12, 60] and at[64, 7] == [40, 28, 49, 12, 60]
    wide = {d: [n for n in range(15, 256, 2) if at[d, n][0]] for d in (64, 128)}
    assert all(at[d, n][0] for d in (64, 128) for n in range(3, 15, 2)) and wide == {64: [29, 49], 128: [29]}
    assert at[128, 149] == [0, 0, 2, 60, 60] and at[64, 99] == [0, 0, 3, 60, 60] and at[128, 75] == [0, 0, 4, 60, 60]

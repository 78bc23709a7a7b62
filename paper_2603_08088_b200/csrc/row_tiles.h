// tree_verify_attn, an odd number of row tiles of 128 rows: who takes the last one.
#pragma once

namespace tv {

// From split_from key tiles per SM on (by the lengths on the device) the last row tile has a launch of its own, up to behind_from
// beside the other one: beside_groups CTA groups of row_tiles / 2 CTAs take the pairs of row tiles, and at the same time odd_groups CTAs on
// SMs of their own the last row tile.  From behind_from on one launch runs behind the other, both on all SMs: behind_groups
// groups and sms CTAs.  Below split_from, and always with behind_groups = 0, one launch does it all, in which the last CTA of
// every group has one row tile only.
struct OddRowTile {
  int beside_groups, odd_groups, behind_groups, split_from, behind_from;
};

// Beside: the SMs are shared out by what a key tile costs in either launch (two row tiles 1.3 times as much as one, with 64-wide
// heads, whose keys two warpgroups share there, 1.7 times, and 1.4 beside three to six pairs).  With many row tiles whole groups are
// lost or won by the rounding: from 15 on only where the front launch has a tenth more groups than one launch for all row tiles and
// does not wait for the few CTAs beside it (three were too few at 59 row tiles).  Behind: both launches have all SMs, but a second fill
// and tail, hence longer work.  What beside gains goes with the work, too: the launches that follow one another should find their
// SMs as the ones in front have left them, and a vocabulary scan in between does not leave them so.  us for 8 sequences, 8 KV heads,
// with such a scan, behind / beside: 65 nodes, 64-wide heads, 63 key tiles per SM 202 / 210, 126 407 / 440, 252 804 / 869, 129 nodes 347 / 371,
// 672 / 736, 1315 / 1453; 128-wide heads, 65 nodes 304 / 300, 586 / 591, 1188 / 1208, 129 nodes 484 / 484, 946 / 956, 1846 / 1893; one layer of 19
// per SM (one launch / beside) 64-wide 93 / 83 and 128 / 120, 128-wide 110 / 102 and 160 / 153.
// us a call without a scan, one launch / behind / beside, 16 units of 13.5 and of 65 key tiles per SM (in brackets where beside is never
// taken):
//    64-wide heads,   3 row tiles:  68 /   89 /   62      218 /  202 /   180    128-wide:    65 /   99 /   69      277 /  299 /   283
//                     9            119 /  128 /  114      532 /  496 /   500                143 /  167 /  139      676 /  680 /   639
//                    13            158 /  172 /  153      727 /  714 /   695                200 /  233 /  195      932 /  953 /   885
//                    15            181 /  189 / (189)     827 /  785 /  (863)               226 /  251 / (236)    1049 / 1039 / (1109)
//                    17            203 /  213 / (225)     912 /  889 / (1038)               252 /  279 / (295)    1176 / 1194 / (1369)
//                    29            350 /  348 /  317     1677 / 1575 /  1498                445 /  454 /  402     2102 / 2041 /  1852
//                    59            781 /  653 / (666)       - / 2982 / (3105)               939 /  788 /   -         - / 3771 / (4878)
//                    75           1038 /  804 / (1026)   4788 / 3648 / (4779)              1242 /  963 / (1203)   6050 / 4611 / (5982)
//                   149           3046 / 1569 / (3063)  14278 / 7249 / (14342)             3235 / 1787 / (3098)  14473 / 9290 / (14627)
constexpr OddRowTile odd_row_tile(int sms, int row_tiles, int d) {
  const int pairs = row_tiles / 2;
  if (row_tiles % 2 == 0 || pairs < 1 || pairs > sms) return {0, 0, 0, 0, 0};
  const bool narrow = row_tiles <= 13;
  const int one = d == 64 && narrow && pairs >= 3 ? 12 : 10, two = d == 64 ? 17 : 13, whole = sms / (pairs + 1);
  const int groups = (sms - sms * one / (one + two * pairs)) / pairs, rest = sms - groups * pairs;
  if (rest > 0 && groups > whole && (narrow || (rest > 3 && groups * 10 >= whole * 11 && groups * one <= rest * two)))
    return {groups, rest, sms / pairs, 12, d == 64 ? 60 : 100};
  return {0, 0, sms / pairs, 60, 60};
}

}  // namespace tv

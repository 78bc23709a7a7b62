// tree_verify_attn, an odd number of row tiles of 128 rows: who takes the last one.
#pragma once

namespace tv {

// front_groups CTA groups of row_tiles / 2 CTAs take the pairs of row tiles, odd_groups CTAs the last row tile: at the same time,
// on SMs of their own (beside), or on all SMs, one launch behind the other.  From tiles_per_sm key tiles per SM on; below, and
// always with front_groups = 0, one launch does it all, in which the last CTA of every group has one row tile only.
struct OddRowTile {
  int front_groups, odd_groups, tiles_per_sm;
  bool beside;
};

// Beside: the SMs are shared out by what a key tile costs in either launch (two row tiles 1.3 times as much as one, with 64-wide
// heads, whose keys two warpgroups share there, 1.7 times, and 1.4 beside three to six pairs).  With many row tiles whole groups are
// lost or won by the rounding: from 15 on only where the front launch has a tenth more groups than one launch for all row tiles and
// does not wait for the few CTAs beside it (three were too few at 59 row tiles).  Behind: both launches have all SMs, but a second fill
// and tail, hence longer work.
// us a call, one launch / behind / beside, 16 units of 13.5 and of 65 key tiles per SM (beside in brackets where it is not taken):
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
  if (row_tiles % 2 == 0 || pairs < 1 || pairs > sms) return {0, 0, 0, false};
  const bool narrow = row_tiles <= 13;
  const int one = d == 64 && narrow && pairs >= 3 ? 12 : 10, two = d == 64 ? 17 : 13, whole = sms / (pairs + 1);
  const int groups = (sms - sms * one / (one + two * pairs)) / pairs, rest = sms - groups * pairs;
  if (rest > 0 && groups > whole && (narrow || (rest > 3 && groups * 10 >= whole * 11 && groups * one <= rest * two)))
    return {groups, rest, 12, true};
  return {sms / pairs, sms, 60, false};
}

}  // namespace tv

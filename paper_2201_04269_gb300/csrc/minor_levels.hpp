// minor_levels.hpp - the factor tree's minors by shared Laplace steps (internal, host side).
//
// The minors of one flavour, det M[R, C] for the tree's (R, C) pairs, follow level by level from
// the matrix entries: each column set C keeps one of its columns c to expand along, and
//   det M[R, C] = sum_i (-1)^(i + q) M[r_i, c] det M[R \ r_i, C \ c]   (q: position of c in C)
// needs only minors one level down, which many pairs share.
#pragma once
#include <cstdint>
#include <vector>

#include "plan.hpp"

namespace mbc {

struct MinorLevels {
    int n = 0;
    // level k = 2..n: entries of k + 1 words; word i = (row of the child in level k - 1) << 8 |
    // (r_i * 12 + c); last word = (row of the result in its own level) << 1 | (q odd).  Level 1 is
    // the 144 matrix entries, row r * 12 + c; rows of level n are the tree's minors.
    std::vector<uint32_t> words[7];
    int64_t rows[7] = {};                       // rows of each level
    int64_t extra_rows = 0;                     // rows below level n
    double cfma = 0;                            // complex multiply-adds of one site
};

// n in 2..6; rows[m], cols[m]: the minors.
MinorLevels build_minor_levels(int n, const std::vector<Mask>& rows, const std::vector<Mask>& cols);

}  // namespace mbc

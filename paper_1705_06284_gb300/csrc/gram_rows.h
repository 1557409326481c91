// Row layouts of the shared-operand tensor-core contraction (host code).
#pragma once

#include <array>
#include <vector>

namespace fbs {

// The operand rows of one CTA group and the (A row, B row) slot of every item.
// A row is a product of two bins (x, y), a single bin (x, -1) or empty
// (-1, -1).  Operand A is rows 0..63, operand B the 8 nbch rows from 8 jb0 on
// (jb0 a multiple of 4, so that it starts on a 64-row swizzle atom of hi and
// lo rows); the two may overlap, so a product used on both sides is formed
// once.  The number of rows is a multiple of 16.
struct GramRows {
    std::vector<std::array<int, 2>> rows;
    int jb0 = 0, nbch = 0;
    std::vector<std::array<int, 3>> items;  // (A row, B row relative to 8 jb0, index of the item), ascending
};

constexpr int kGramARows = 64;    // M = 128 holds their hi and lo parts
constexpr int kGramBRows = 256;   // two accumulator tiles of N = 256 (hi and lo)

// Triplets (a, b, c, -1) and quadruplets (a, b, c, d) over one set of rows: an
// item sits where the products of two of its parts meet (pair x pair, or pair
// x single).  False when 64 A rows and 128 B rows do not hold them all.
bool gram_rows_shared(int nb, const std::vector<std::array<int, 4>> &items, GramRows &out);

// Triplets with at most 64 covering pairs (cover: the pair key of each, from
// cover_triplet_pairs) as operand A and the single bins as operand B.  False
// when there are more.
bool gram_rows_pairs(int nb, const std::vector<std::array<int, 3>> &trip, const std::vector<int> &cover,
                     GramRows &out);

// Triplets with the single bins (at most 64) as operand A and the covering
// pairs as operand B, at most 256 to a group.  False for more bins.
bool gram_rows_wide(int nb, const std::vector<std::array<int, 3>> &trip, const std::vector<int> &cover,
                    std::vector<GramRows> &out);

}  // namespace fbs

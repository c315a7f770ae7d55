// minor_levels.cpp - see minor_levels.hpp.
#include "minor_levels.hpp"

#include <algorithm>

namespace mbc {

namespace {
constexpr int kAll = 12, kSets = 1 << kAll;

// The needed (C, R) pairs of a level: per column set present, the row of every needed R (column
// sets, then row sets, ascending), -1 elsewhere.
struct Level {
    std::vector<std::vector<int32_t>> at = std::vector<std::vector<int32_t>>(kSets);
    int64_t n = 0;
    void need(Mask c, Mask r) {
        if (at[c].empty()) at[c].assign(kSets, -1);
        at[c][r] = 0;
    }
    void number() {
        for (auto& v : at)
            for (int32_t& x : v)
                if (x >= 0) x = (int32_t)n++;
    }
};
}  // namespace

MinorLevels build_minor_levels(int n, const std::vector<Mask>& rows, const std::vector<Mask>& cols) {
    MinorLevels out;
    out.n = n;
    std::vector<Level> lev(n + 1);
    for (size_t m = 0; m < rows.size(); ++m) lev[n].need(cols[m], rows[m]);
    std::vector<std::vector<int8_t>> split(n + 1, std::vector<int8_t>(kSets, -1));
    for (int k = n; k >= 2; --k) {
        // the column whose removal leaves the set that most column sets of the level share
        // (ties: the largest column), as in the e-graph's extraction
        std::vector<int> parents(kSets, 0);
        for (int c = 0; c < kSets; ++c)
            for (int i = 0; i < kAll && !lev[k].at[c].empty(); ++i)
                if (c >> i & 1) ++parents[c & ~(1 << i)];
        for (int c = 0; c < kSets; ++c) {
            if (lev[k].at[c].empty()) continue;
            int top = -1;
            for (int i = 0; i < kAll; ++i)
                if ((c >> i & 1) && parents[c & ~(1 << i)] >= top) {
                    top = parents[c & ~(1 << i)];
                    split[k][c] = (int8_t)i;
                }
            if (k == 2) continue;
            const Mask cc = (Mask)(c & ~(1 << split[k][c]));
            for (int r = 0; r < kSets; ++r)
                for (int i = 0; i < kAll && lev[k].at[c][r] >= 0; ++i)
                    if (r >> i & 1) lev[k - 1].need(cc, (Mask)(r & ~(1 << i)));
        }
        lev[k].number();
    }
    out.rows[1] = 144;
    for (int k = 2; k <= n; ++k) {
        out.rows[k] = k == n ? (int64_t)rows.size() : lev[k].n;
        out.cfma += (double)lev[k].n * k;
    }
    for (int k = 1; k < n; ++k) out.extra_rows += out.rows[k];
    // the minor of each (C, R) of level n (a repeated pair: one entry per minor)
    std::vector<int32_t> minor(lev[n].n, -1), same(rows.size(), -1);
    for (size_t m = rows.size(); m-- > 0;) {
        int32_t& first = minor[lev[n].at[cols[m]][rows[m]]];
        same[m] = first;
        first = (int32_t)m;
    }
    for (int k = 2; k <= n; ++k)
        for (int c = 0; c < kSets; ++c) {
            if (lev[k].at[c].empty()) continue;
            const int col = split[k][c];
            const Mask cc = (Mask)(c & ~(1 << col));
            const uint32_t q = __builtin_popcount((unsigned)(c & ((1 << col) - 1))) & 1;
            for (int r = 0; r < kSets; ++r) {
                const int32_t row = lev[k].at[c][r];
                if (row < 0) continue;
                for (int32_t to = k == n ? minor[row] : row; to >= 0; to = k == n ? same[to] : -1) {
                    for (int i = 0; i < kAll; ++i) {
                        if (!(r >> i & 1)) continue;
                        const int rest = r & ~(1 << i);
                        const uint32_t child = k == 2 ? (uint32_t)(__builtin_ctz((unsigned)rest) * 12 +
                                                                   __builtin_ctz((unsigned)cc))
                                                      : (uint32_t)lev[k - 1].at[cc][rest];
                        out.words[k].push_back(child << 8 | (uint32_t)(i * 12 + col));
                    }
                    out.words[k].push_back((uint32_t)to << 1 | q);
                }
            }
        }
    return out;
}

}  // namespace mbc

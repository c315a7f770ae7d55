// Host check of the factor tree's Laplace levels (csrc/minor_levels.cpp): the levels' words are
// replayed in complex double on a random 12 x 12 matrix, every index is checked against the level
// it refers to, and every minor must equal its determinant by elimination.  Dense row and column
// families, scattered pairs and repeated pairs, 2 to 6 rows.  Built and run by
// tests/test_minor_levels_cpu.py; prints "OK <count>" or the first failure.
#include "minor_levels.hpp"

#include <cmath>
#include <cstdio>

using namespace mbc;

static uint32_t g_seed = 7u;
static uint32_t rnd() { g_seed = g_seed * 1664525u + 1013904223u; return g_seed >> 8; }

static Mask random_set(int n) {
    Mask m = 0;
    while (mask_size(m) < n) m |= (Mask)(1u << (rnd() % 12));
    return m;
}

static cplx det(const cplx* M, Mask R, Mask C) {
    int8_t r[12], c[12];
    mask_list(R, r);
    mask_list(C, c);
    const int n = mask_size(R);
    std::vector<cplx> a((size_t)n * n);
    for (int i = 0; i < n; ++i) for (int k = 0; k < n; ++k) a[i * n + k] = M[r[i] * 12 + c[k]];
    cplx d = 1.0;
    for (int k = 0; k < n; ++k) {
        int p = k;
        for (int i = k + 1; i < n; ++i) if (std::abs(a[i * n + k]) > std::abs(a[p * n + k])) p = i;
        if (p != k) { for (int q = 0; q < n; ++q) std::swap(a[k * n + q], a[p * n + q]); d = -d; }
        d *= a[k * n + k];
        for (int i = k + 1; i < n; ++i) {
            const cplx f = a[i * n + k] / a[k * n + k];
            for (int q = k; q < n; ++q) a[i * n + q] -= f * a[k * n + q];
        }
    }
    return d;
}

static bool check(int n, const std::vector<Mask>& rows, const std::vector<Mask>& cols) {
    cplx M[144];
    for (auto& x : M) x = cplx((double)rnd() / (1 << 24) - 0.5, (double)rnd() / (1 << 24) - 0.5);
    const MinorLevels l = build_minor_levels(n, rows, cols);
    std::vector<cplx> below(M, M + 144), out;
    if (l.n != n || l.rows[1] != 144 || l.rows[n] != (int64_t)rows.size()) return false;
    int64_t extra = 144;
    for (int k = 2; k <= n; ++k) {
        const int64_t cnt = l.rows[k];
        if ((int64_t)l.words[k].size() != cnt * (k + 1)) return false;
        if (k < n) extra += cnt;
        out.assign(cnt, cplx(NAN, NAN));
        std::vector<int> written(cnt, 0);
        for (int64_t e = 0; e < cnt; ++e) {
            const uint32_t* w = &l.words[k][e * (k + 1)];
            cplx v = 0.0;
            for (int i = 0; i < k; ++i) {
                if ((w[i] & 0xFF) >= 144 || (w[i] >> 8) >= below.size()) return false;
                v += (i & 1 ? -1.0 : 1.0) * M[w[i] & 0xFF] * below[w[i] >> 8];
            }
            const uint32_t to = w[k] >> 1;
            if ((int64_t)to >= cnt || written[to]++) return false;
            out[to] = (w[k] & 1) ? -v : v;
        }
        below = out;
    }
    if (extra != l.extra_rows) return false;
    for (size_t m = 0; m < rows.size(); ++m)
        if (!(std::abs(below[m] - det(M, rows[m], cols[m])) <= 1e-13)) return false;
    return true;
}

int main() {
    int done = 0;
    for (int n = 2; n <= 6; ++n)
        for (int kind = 0; kind < 4; ++kind) {
            std::vector<Mask> rows, cols;
            if (kind == 0) {                              // one minor
                rows.push_back(random_set(n));
                cols.push_back(random_set(n));
            } else if (kind == 1) {                       // scattered, with repeats
                for (int i = 0; i < 50; ++i) { rows.push_back(random_set(n)); cols.push_back(random_set(n)); }
                for (int i = 0; i < 10; ++i) { rows.push_back(rows[i * 3]); cols.push_back(cols[i * 3]); }
            } else {                                      // families: every pair, or half of them
                std::vector<Mask> a, b;
                for (int i = 0; i < 40; ++i) { a.push_back(random_set(n)); b.push_back(random_set(n)); }
                for (Mask r : a) for (Mask c : b) if (kind == 2 || rnd() % 2) { rows.push_back(r); cols.push_back(c); }
            }
            if (!check(n, rows, cols)) { printf("FAIL n %d kind %d\n", n, kind); return 1; }
            ++done;
        }
    printf("OK %d\n", done);
    return 0;
}

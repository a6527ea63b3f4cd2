// Host check of an open plan's zero rows (no GPU): a random boundary on the
// support the sweep leaves is joined with a dense matrix and crossed layer by
// layer; every row that the join's blocks or a crossing leave out, and every
// input row that a crossing does not read, must be exactly zero. Usage:
//   late_skip_check n d k seed; prints the fraction of rows visited.
#include <cstdio>
#include <cstdlib>
#include <complex>
#include <random>
#include <set>
#include <vector>
#include "tb_plan.h"
using namespace tb;
using cd = std::complex<double>;
static cd C(float2 z) { return cd(z.x, z.y); }

int main(int argc, char** argv) {
    if (argc < 5) return 1;
    const int n = atoi(argv[1]), d = atoi(argv[2]), k = atoi(argv[3]), seed = atoi(argv[4]);
    std::mt19937 rng(seed);
    std::vector<uint8_t> cliff((d + 1) * n), tm(d * n), x(n);
    for (auto& v : cliff) v = seed == 0 ? 0 : rng() % 24;  // seed 0: identity circuit
    for (auto& v : tm) v = (rng() % 10) == 0;
    for (auto& v : x) v = rng() & 1;
    Plan P;
    P.open_k = k;
    std::string err;
    if (plan_build(P, n, d, cliff.data(), tm.data(), nullptr, 0, nullptr, nullptr, err) != TB_OK) {
        printf("plan: %s\n", err.c_str());
        return 1;
    }
    const int h = P.h;
    std::vector<cd> B((size_t)1 << h);
    for (size_t s = 0; s < B.size(); ++s) {
        const size_t sl = s & (((size_t)1 << P.k) - 1), sm = (s >> P.k) & (((size_t)1 << P.m) - 1), st = s >> (P.k + P.m);
        const size_t bk = (s >> (P.k - 1)) & 1, bm = P.m ? (sm >> (P.m - 1)) & 1 : bk;
        B[s] = C(P.init_low[sl]) * C(P.init_mid[(bk << P.m) + sm]) * C(P.init_top[((x[0] * 2 + bm) << P.top) + st]);
    }
    for (size_t q = 0; q < P.steps.size(); ++q) {
        const int t = P.step_tgt[q], c = P.step_ctl[q];
        const float2* g = P.steps[q].g[P.step_xq[q] >= 0 ? x[P.step_xq[q]] : 0];
        for (size_t i = 0; i < B.size(); ++i) {
            if (i >> t & 1) continue;
            const size_t j = i | ((size_t)1 << t);
            const int cv = c < 0 ? 0 : (int)((i >> c) & 1);
            const cd a = B[i], b = B[j];
            B[i] = C(g[cv * 4 + 0]) * a + C(g[cv * 4 + 1]) * b;
            B[j] = C(g[cv * 4 + 2]) * a + C(g[cv * 4 + 3]) * b;
        }
    }
    // which rows (address bits k..h-1) are not zero
    std::vector<char> live((size_t)1 << (h - k), 0);
    for (size_t i = 0; i < B.size(); ++i)
        if (B[i] != 0.0) live[i >> k] = 1;
    {
        std::set<uint32_t> blocks;
        for (uint32_t u = 0; u < ((uint32_t)1 << (h - k - 7 - P.join_skip.n)); ++u) blocks.insert(tile_of(P.join_skip, u));
        for (size_t r = 0; r < live.size(); ++r)
            if (live[r] && !blocks.count((uint32_t)(r >> 7))) { printf("join leaves out row %zu\n", r); return 2; }
    }
    double visited = 0, total = 0;
    for (size_t i = 0; i + 1 < P.open_seg.size(); ++i) {
        const LateSkip& ls = P.late_skip[i];
        std::vector<char> out(live.size() / 2, 0);
        for (size_t r = 0; r < out.size(); ++r) out[r] = live[2 * r] | live[2 * r + 1];
        std::set<size_t> rows;
        for (size_t u = 0; u < (out.size() >> ls.out.n); ++u) rows.insert(tile_of(ls.out, (uint32_t)u));
        visited += (double)rows.size();
        total += (double)out.size();
        for (size_t r = 0; r < out.size(); ++r) {
            if (out[r] && !rows.count(r)) { printf("crossing %zu leaves out row %zu\n", i, r); return 2; }
            if (ls.both || !rows.count(r)) continue;
            const int pick = __builtin_parity((uint32_t)r & ls.mask) ^ (int)ls.fix;
            if (live[2 * r + (1 - pick)]) { printf("crossing %zu does not read row %zu\n", i, 2 * r + (1 - pick)); return 2; }
        }
        live = out;
    }
    printf("visited=%.3f\n", visited / total);
    return 0;
}

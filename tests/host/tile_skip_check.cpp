// Host check of the planner's zero tiles (no GPU): the row-0 boundary and every
// paired step applied one by one to a full boundary; before each pass, every
// tile the pass leaves out must be exactly zero and the visited tile numbers
// must be distinct tiles. Usage:
//   tile_skip_check n d seed precision odd_gates [window bottom top]
// odd_gates: every odd_gates-th one-qubit gate is replaced by a dense one (0:
// none). Prints the fraction of tiles visited; exit 0 when every check holds.
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
    if (argc < 6) return 1;
    const int n = atoi(argv[1]), d = atoi(argv[2]), seed = atoi(argv[3]), odd = atoi(argv[5]);
    std::mt19937 rng(seed);
    std::vector<uint8_t> cliff((d + 1) * n), tm(d * n), x(n);
    for (auto& v : cliff) v = seed == 0 ? 0 : rng() % 24;  // seed 0: identity circuit
    for (auto& v : tm) v = (rng() % 10) == 0;
    for (auto& v : x) v = rng() & 1;
    std::vector<tb_gate1q> extra;
    if (odd)
        for (int i = 0; i < (d + 1) * n; i += odd) {
            const double a = 0.1 + 0.37 * (rng() % 8);
            extra.push_back(tb_gate1q{i % n, i / n, {std::cos(a), 0, -std::sin(a), 0, std::sin(a), 0, std::cos(a), 0}});
        }
    tb_opts o{};
    o.precision = atoi(argv[4]);
    if (argc > 8) { o.window_bits = atoi(argv[6]); o.bottom_bits = atoi(argv[7]); o.top_bits = atoi(argv[8]); }
    Plan P;
    std::string err;
    if (plan_build(P, n, d, cliff.data(), tm.data(), extra.data(), (int)extra.size(), nullptr, &o, err) != TB_OK) {
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
    int done = 0;
    auto advance = [&](int end) {
        for (; done < end; ++done) {
            const int t = P.step_tgt[done], c = P.step_ctl[done];
            const float2* g = P.steps[done].g[P.step_xq[done] >= 0 ? x[P.step_xq[done]] : 0];
            for (size_t i = 0; i < B.size(); ++i) {
                if (i >> t & 1) continue;
                const size_t j = i | ((size_t)1 << t);
                const int cv = c < 0 ? 0 : (int)((i >> c) & 1);
                const cd a = B[i], b = B[j];
                B[i] = C(g[cv * 4 + 0]) * a + C(g[cv * 4 + 1]) * b;
                B[j] = C(g[cv * 4 + 2]) * a + C(g[cv * 4 + 3]) * b;
            }
        }
    };
    double visited = 0, total = 0;
    auto check = [&](int step0, const std::vector<int>& tile, const TileSkip& k) {
        advance(step0);
        std::vector<int> outside;
        for (int b = 0; b < h; ++b) {
            bool in = false;
            for (int t : tile) in |= t == b;
            if (!in) outside.push_back(b);
        }
        std::set<uint32_t> seen;
        for (uint32_t u = 0; u < ((uint32_t)1 << ((int)outside.size() - k.n)); ++u) {
            const uint32_t t = tile_of(k, u);
            if (t >> outside.size() || !seen.insert(t).second) { printf("tile %u of %u: not a new tile\n", u, t); return false; }
        }
        visited += (double)seen.size();
        total += std::ldexp(1.0, (int)outside.size());
        for (size_t i = 0; i < B.size(); ++i) {
            if (B[i] == 0.0) continue;
            uint32_t t = 0;
            for (size_t j = 0; j < outside.size(); ++j) t |= (uint32_t)((i >> outside[j]) & 1) << j;
            if (!seen.count(t)) { printf("pass at step %d leaves out entry %zu, which is not zero\n", step0, i); return false; }
        }
        return true;
    };
    for (const PassDesc& p : P.passes) {
        const bool bottom = bottom_type(p.type);
        std::vector<int> tile;
        for (int b = 0; b < (bottom ? bot_chunk_bits(p.M) : high_low_bits(p.M)); ++b) tile.push_back(b);
        if (!bottom)
            for (int b = 0; b < p.M; ++b) tile.push_back(p.lo + b);
        if (!check(p.step0, tile, p.skip)) return 2;
        // warps with nothing to do: the entries with these low address bits are zero
        const int wn = warp_addr_bits(p.type, p.M);
        for (size_t i = 0; i < B.size() && wn; ++i) {
            if (B[i] == 0.0) continue;
            const uint32_t w = (uint32_t)(i >> warp_low_bit(p.M)) & ((1u << wn) - 1u);
            const uint32_t t = (uint32_t)((i >> 4 & (((size_t)1 << (p.lo - 4)) - 1)) | (i >> (p.lo + p.M) << (p.lo - 4)));
            for (int e = 0; e < p.warps.n; ++e)
                if ((__builtin_parity(t & p.warps.out[e]) ^ __builtin_parity(w & p.warps.warp[e] & 7u)) != (int)(p.warps.warp[e] >> 3)) {
                    printf("pass at step %d: warp %u leaves out entry %zu, which is not zero\n", p.step0, w, i);
                    return 2;
                }
        }
        if (p.skip.n > h - TILE_BITS) {
            printf("pass at step %d visits less than one tile\n", p.step0);
            return 2;
        }
    }
    for (const TcPass& p : P.tc_passes) {
        std::vector<int> tile;
        for (int b = 0; b < P.tc_wb; ++b) tile.push_back(p.lo + b);
        for (int b = 0, low = 0; low < TC_VEC_BITS; ++b)
            if (b < p.lo || b >= p.lo + P.tc_wb) { tile.push_back(b); ++low; }
        if (!check(p.step0, tile, p.skip)) return 2;
    }
    {  // the chunks of the last-row reduction
        std::vector<int> low;
        for (int b = 0; b < P.k; ++b) low.push_back(b);
        if (!check((int)P.steps.size(), low, P.red_skip)) return 2;
    }
    printf("visited=%.3f\n", visited / total);
    return 0;
}

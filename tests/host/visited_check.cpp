// Host check (no GPU): plan_visited counts what the passes do. Every visited tile is
// expanded and, where its warps hold address bits, each of its 8 warps tested against
// the pass's WarpSkip as the kernel does. Usage: visited_check n d seed [window bottom top]
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "tb_plan.h"
using namespace tb;

int main(int argc, char** argv) {
    if (argc < 4) return 1;
    const int n = atoi(argv[1]), d = atoi(argv[2]);
    std::mt19937 rng(atoi(argv[3]));
    std::vector<uint8_t> cliff((d + 1) * n), tm(d * n);
    for (auto& v : cliff) v = rng() % 24;
    for (auto& v : tm) v = (rng() % 10) == 0;
    tb_opts o{};
    if (argc > 6) { o.window_bits = atoi(argv[4]); o.bottom_bits = atoi(argv[5]); o.top_bits = atoi(argv[6]); }
    Plan P;
    std::string err;
    if (plan_build(P, n, d, cliff.data(), tm.data(), nullptr, 0, nullptr, &o, err) != TB_OK) {
        printf("plan: %s\n", err.c_str());
        return 1;
    }
    double entries = 0.0, madds = 0.0, e = 0.0, m = 0.0;
    for (const PassDesc& p : P.passes) {
        const int chl = pass_chunk_log2(p.type, p.M), wn = warp_addr_bits(p.type, p.M);
        const double per = 8 * p.nsteps + (pass_blk(p.type, p.M) >= 0 ? 8 : 0);
        for (uint32_t t = 0; t < ((uint32_t)1 << (P.h - TILE_BITS - p.skip.n)); ++t)
            for (uint32_t w = 0; w < 8; ++w) {
                const uint32_t chunk = w >> 2 & 1u;  // 8-bit windows: two chunks, the highest warp bit
                const uint32_t ti = tile_of(p.skip, (t << chl) | (chl == 1 ? chunk : 0u));
                bool idle = false;
                for (int i = 0; i < p.warps.n && wn; ++i)
                    idle |= (__builtin_parity(ti & p.warps.out[i]) ^ __builtin_parity(w & p.warps.warp[i] & 7u) ^
                             (int)(p.warps.warp[i] >> 3)) != 0;
                entries += 1024.0;
                if (!idle) madds += 1024.0 * per;
            }
    }
    plan_visited(P, &e, &m);
    printf("entries %.0f %.0f madds %.0f %.0f\n", entries, e, madds, m);
    return entries == e && madds == m ? 0 : 2;
}

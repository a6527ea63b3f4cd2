// Host check of an open plan's out-of-place buffers (no GPU): the join and every late
// crossing write only the rows they visit, so each crossing may read only rows that
// the stage before it wrote, and the output, row 0 of the last crossing, is written.
// Usage: late_written_check n d k seed; prints the rows read.
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "tb_plan.h"
using namespace tb;

int main(int argc, char** argv) {
    if (argc < 5) return 1;
    const int n = atoi(argv[1]), d = atoi(argv[2]), k = atoi(argv[3]), seed = atoi(argv[4]);
    std::mt19937 rng(seed);
    std::vector<uint8_t> cliff((d + 1) * n), tm(d * n);
    for (auto& v : cliff) v = seed == 0 ? 0 : rng() % 24;  // seed 0: identity circuit
    for (auto& v : tm) v = (rng() % 10) == 0;
    Plan P;
    P.open_k = k;
    std::string err;
    if (plan_build(P, n, d, cliff.data(), tm.data(), nullptr, 0, nullptr, nullptr, err) != TB_OK) {
        printf("plan: %s\n", err.c_str());
        return 1;
    }
    const int h = P.h;
    std::vector<char> written((size_t)1 << (h - k), k < JOIN_TC_MIN_K);  // the FP32 join writes every row
    if (k >= JOIN_TC_MIN_K)
        for (uint32_t u = 0; u < ((uint32_t)1 << (h - k - 7 - P.join_skip.n)); ++u)
            for (uint32_t r = 0; r < 128; ++r) written[(size_t)tile_of(P.join_skip, u) * 128 + r] = 1;
    long reads = 0;
    for (size_t i = 0; i + 1 < P.open_seg.size(); ++i) {
        const LateSkip& ls = P.late_skip[i];
        std::vector<char> out(written.size() / 2, 0);
        for (int64_t u = 0; u < P.late_rows(i) >> ls.out.n; ++u) {
            const uint32_t r = tile_of(ls.out, (uint32_t)u);
            if (r >= out.size()) { printf("crossing %zu: row %u of %zu\n", i, r, out.size()); return 2; }
            const int pick = __builtin_parity(r & ls.mask) ^ (int)ls.fix;
            for (int s = 0; s < 2; ++s) {
                if (!ls.both && s != pick) continue;
                ++reads;
                if (!written[2 * (size_t)r + s]) {
                    printf("crossing %zu (of %zu) reads row %zu, which nothing wrote\n", i, P.open_seg.size() - 1, 2 * (size_t)r + s);
                    return 2;
                }
            }
            out[r] = 1;
        }
        written = out;
    }
    if (!written[0]) { printf("the output row is not written\n"); return 2; }
    printf("read=%ld\n", reads);
    return 0;
}

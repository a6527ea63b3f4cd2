// Host check (no GPU): an output bit selects a variant only in the steps that
// output_step names; the pass kernels take the coefficients of others from
// variant 0. Also checks that both variants of every other step are the same.
// Usage: output_step_check n d seed [window bottom top]
#include <cstdio>
#include <cstdlib>
#include <cstring>
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
    int selected = 0, steps = 0;
    for (const PassDesc& p : P.passes) {
        for (int j = 0; j < 2; ++j) {
            if (p.xs_step[j] < 0) continue;
            ++selected;
            const int i = p.xs_step[j] == XM_HIGH_BIT ? pass_xm(p.type, p.M) : p.xs_step[j];
            if (!output_step(p.type, p.M, i)) {
                printf("type %d M=%d: step %d depends on an output bit\n", p.type, p.M, i);
                return 2;
            }
        }
        for (int i = 0; i < p.nsteps; ++i) {
            if (i == pass_blk(p.type, p.M) || output_step(p.type, p.M, i)) continue;
            const StepG& g = P.pass_steps[p.pstep0 + pass_entry(p.type, p.M, i)];
            ++steps;
            if (std::memcmp(g.g[0], g.g[1], sizeof(g.g[0])) != 0) {
                printf("type %d M=%d: the variants of step %d differ\n", p.type, p.M, i);
                return 2;
            }
        }
    }
    printf("selected=%d steps=%d\n", selected, steps);
    return selected > 0 && steps > 0 ? 0 : 2;
}

// Host check (no GPU): what a plan leaves out as exactly zero when one-qubit gates
// carry a given factor. Identity circuit otherwise, where almost everything is zero.
// Usage: finite_guard_check n d open_k precision [qubit slot factor]...
// Prints the number of address bits that passes, warps, join, crossings and
// reduction find determined.
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "tb_plan.h"
using namespace tb;

int main(int argc, char** argv) {
    if (argc < 5) return 1;
    const int n = atoi(argv[1]), d = atoi(argv[2]);
    std::vector<tb_gate1q> extra;
    for (int i = 5; i + 2 < argc; i += 3) {
        const double f = strtod(argv[i + 2], nullptr);  // "inf" and "nan" included
        extra.push_back(tb_gate1q{atoi(argv[i]), atoi(argv[i + 1]), {f, 0, 0, 0, 0, 0, f, 0}});
    }
    tb_opts o{};
    o.precision = atoi(argv[4]);
    Plan P;
    P.open_k = atoi(argv[3]);
    std::string err;
    if (plan_build(P, n, d, nullptr, nullptr, extra.data(), (int)extra.size(), nullptr, &o, err) != TB_OK) {
        printf("plan: %s\n", err.c_str());
        return 1;
    }
    int bits = P.red_skip.n + P.join_skip.n;
    for (const PassDesc& p : P.passes) bits += p.skip.n + p.warps.n;
    for (const TcPass& p : P.tc_passes) bits += p.skip.n;
    for (const LateSkip& l : P.late_skip) bits += l.out.n + (l.both ? 0 : 1);
    printf("determined=%d\n", bits);
    return 0;
}

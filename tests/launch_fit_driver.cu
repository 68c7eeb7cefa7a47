// Prints what umi::fit_launch makes of launches read from standard input: lines of
// "W positions curves" give lines of "G R minb threads rule_chain chain smem".
#include <cstdio>

#include "umi_internal.h"

int main()
{
    int W;
    long long positions, curves;
    int nv = 0;
    const umi::Variant *t = umi::variant_table(&nv);
    while (scanf("%d %lld %lld", &W, &positions, &curves) == 3) {
        umi::Plan p;
        if (umi::make_plan(W, positions, &p) != UMI_OK) return 1;
        const int rule = p.chain;
        umi::fit_launch(positions, curves, &p);
        printf("%d %d %d %d %d %d %zu\n", p.G, p.R, t[p.variant].minb, p.threads, rule, p.chain, p.smem_bytes());
    }
    return 0;
}

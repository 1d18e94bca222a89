// Plans read from stdin (test infrastructure: compiled and run by tests/test_batch_plan.py).
// Per line: n_sm per_sm may_alone n, then per item levels flops N cap n_x line; prints
// each item's CTAs and whether it runs one direction per CTA beside the others.
#include <cstdio>

#include "../paper_2201_00241_gb300/csrc/batch_plan.h"

int main() {
    int n_sm, per_sm, may_alone, n;
    while (std::scanf("%d %d %d %d", &n_sm, &per_sm, &may_alone, &n) == 4) {
        rh::BatchItem b[rh::kMaxBatch];
        for (int k = 0; k < n; k++) {
            int line;
            if (std::scanf("%lf %lf %d %d %d %d", &b[k].levels, &b[k].flops, &b[k].N, &b[k].cap, &b[k].n_x, &line) != 6)
                return 1;
            b[k].line = line != 0;
        }
        rh::BatchPlan P;
        rh::BatchPlanner(b, n, n_sm, per_sm, may_alone != 0).plan(P);
        for (int k = 0; k < n; k++) std::printf("%d %d ", P.G[k], P.alone[k] ? 1 : 0);
        std::printf("\n");
    }
    return 0;
}

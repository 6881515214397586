// Host-only driver of the rule that evens out a plain call's CTAs
// (even_threads in gen_kernels.cuh).  Input: lines of "kind fmt groups per_cta
// sectors realigned tail"; output: the CTA size of each, 0 for the shape's own.
#include <cinttypes>
#include <cstdio>

#include "gen_kernels.cuh"

int main()
{
    int kind = 0, fmt = 0, sectors = 0, realigned = 0, tail = 0;
    uint64_t groups = 0, per_cta = 0;
    while (std::scanf("%d %d %" SCNu64 " %" SCNu64 " %d %d %d", &kind, &fmt, &groups, &per_cta,
                      &sectors, &realigned, &tail) == 7)
        std::printf("%d\n", gbrng::even_threads(kind, fmt, groups, per_cta, sectors != 0,
                                                realigned != 0, tail != 0));
    return 0;
}

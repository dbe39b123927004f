// How the intervals of a plan without pair lists are cut (range_split): input "nint M pairs", output, for free
// memory from 300 GB down to none, lines "free part nparts slab".
#include <cstdio>

#include "internal.h"

int main() {
    int nint;
    long long M, pairs;
    if (std::scanf("%d %lld %lld", &nint, &M, &pairs) != 3) return 1;
    for (double f : {3e11, 1e11, 2e10, 4e9, 5e8, 1e7, 1e5, 0.0}) {
        const wave1d::RangeSplit r = wave1d::range_split(nint, M, pairs, (size_t)f);
        std::printf("%.0f %d %d %d\n", f, r.part, r.nparts, r.slab);
    }
    return 0;
}

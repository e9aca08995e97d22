// Host harness of the ACA scratch plan (csrc/hbi_internal.h): for a free memory and the largest block of
// every class, in the order the build plans them.  Prints "<free doubles> <side> <class> <jobs>
// <resident> <want> <grid> <slot>" per class.
#include <cstdio>

#include "../paper_2110_12165_gb300/csrc/hbi_internal.h"

using namespace hbi;

int main() {
    for (int64_t free_b : {(int64_t)1 << 20, (int64_t)64 << 20, (int64_t)700 << 20, (int64_t)3 << 30, (int64_t)270 << 30})
        for (int side : {129, 600, 10000, 60000, 1000000}) {
            int64_t left = free_b / (int64_t)sizeof(double) / ACA_SCRATCH_SHARE;
            for (int c = ACA_CLASSES - 1; c >= 0; --c) {
                const int n = c == 0 ? side : (c == 1 ? 128 : (c == 2 ? 64 : 40)), jobs = 300 * (c + 1), resident = 152 * (c + 1);
                const int64_t want = c == 3 ? (int64_t)6 * n * n : 32LL * 7 * n + n / 2;
                const AcaScratch s = aca_scratch(c, jobs, resident, want, left);
                printf("%lld %d %d %d %d %lld %d %lld\n", (long long)(free_b / 8), side, c, jobs, resident, (long long)want,
                       s.grid, (long long)s.slot);
            }
        }
    return 0;
}

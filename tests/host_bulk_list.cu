// Host check (no GPU) of bulk_list_blocks: the blocks of a bulk launch over a
// work list stay within ctas_per_sm on every SM, by the launch's size or by
// what an SM holds, start no more items than there are, and leave no SM idle
// that has an item. Prints one line and returns 0 when all hold.
#include <algorithm>
#include <cstdio>

#include "flbm_host.cuh"

using namespace flbm;

int main()
{
    int failed = 0, cases = 0;
    for (int nsm : {1, 4, 148, 152})
        for (int ctas = 1; ctas <= 8; ++ctas)
            for (int nitems : {1, 3, 151, 152, 153, 608, 1000000}) {
                const int resident = 4, loop = 2;
                const int b = bulk_list_blocks(nitems, ctas, resident, loop, nsm);
                const bool all = b == nitems, bounded = b <= ctas * nsm;
                failed += b < std::min(nitems, nsm) || b > nitems;
                failed += !(bounded || (all && ctas >= resident));
                failed += ctas >= resident && !all;
                ++cases;
            }
    std::printf("cases %d failed %d\n", cases, failed);
    return failed == 0 ? 0 : 1;
}

// CPU test of the rule that picks how a time-slowest cube's block is gathered:
// series by series only while two of them fit the block, whose steps are then
// few, for every length of the time axis.
#include "cta_emu.h"
#include "../../paper_1503_00638_gb300/csrc/shuffle_cta.cuh"
#include <initializer_list>
using namespace bsg;

int main()
{
    for (uint32_t n : {4u, 16u, 512u, 1024u, 4096u, 8192u})
        for (uint64_t T : std::initializer_list<uint64_t>{1ull, 2ull, n / 2ull, n / 2ull + 1, (uint64_t)n, 1ull << 20, (1ull << 31) - 1, 1ull << 31,
                           (1ull << 31) + 1, (1ull << 31) + n / 4, (1ull << 31) + n / 2, (1ull << 32) - 1})
            if (cta_gather_single((uint32_t)T, n) != (2 * T > n)) {
                fprintf(stderr, "T %llu, %u samples a block\n", (unsigned long long)T, n);
                return 1;
            }
    return 0;
}

// Entry points to the pieces of cr_split.cuh for the tests that compare them
// with exact integer and rational arithmetic.
#include "cr_split.cuh"

using namespace crs;

// split_value of seven digit sums over ks K-steps, on the host.
extern "C" double split_value_host(int ks, const int *sums) {
    int s[kSplitDigits];
    for (int d = 0; d < kSplitDigits; ++d) s[d] = ks == 1 ? (int)((unsigned)sums[d] + (unsigned)kSplitMagic) : sums[d];
    switch (ks) {
        case 1: return split_value<1>(s);
        case 2: return split_value<2>(s);
        case 4: return split_value<4>(s);
        case 8: return split_value<8>(s);
        default: return split_value<16>(s);
    }
}

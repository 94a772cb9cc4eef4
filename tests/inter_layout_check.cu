// Test-only host program (compiled and run by tests/test_kernel_resources_default.py,
// no GPU needed): the slot map of the interleaved spectrum layout covers a row
// of a group exactly once, and the gather's step to the next bin agrees with it.
#include <cstdio>
#include <vector>

#include "bst_inter.cuh"

template <int M, int P> static bool check() {
    std::vector<int> seen((size_t)M * P, 0);
    for (int k = 0; k < M / 2; ++k)
        for (int s = 0; s < 2; ++s)
            for (int p = 0; p < P; ++p) {
                const int at = bst::inter_slot<P>(k, s) + p;
                if (at < 0 || at >= M * P || seen[at]++) {
                    std::printf("FAIL M=%d P=%d k=%d s=%d p=%d slot=%d\n", M, P, k, s, p, at);
                    return false;
                }
                // 16-byte pieces: two pairs side by side, the next bin up1 pieces on
                const int up1 = P == 2 ? ((k & 1) ? 3 : 1) : P;
                if (at % 2 != p % 2 || (k + 1 < M / 2 && bst::inter_slot<P>(k + 1, s) + p != at + 2 * up1)) {
                    std::printf("FAIL step M=%d P=%d k=%d s=%d\n", M, P, k, s);
                    return false;
                }
            }
    return true;
}

int main() {
    static_assert(bst::inter_pairs<32>() == 8 && bst::inter_pairs<512>() == 8 && bst::inter_pairs<768>() == 4 &&
                      bst::inter_pairs<1024>() == 4 && bst::inter_pairs<1536>() == 2 && bst::inter_pairs<4096>() == 2 &&
                      bst::inter_pairs<16>() == 1, "groups of each length");
    if (!(check<32, 8>() && check<48, 8>() && check<512, 8>() && check<768, 4>() && check<1024, 4>() &&
          check<1536, 2>() && check<4096, 2>()))
        return 1;
    std::printf("OK\n");
    return 0;
}

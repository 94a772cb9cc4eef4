// Test-only host program (compiled and run by tests/test_workspace_rules.py, no
// GPU needed): how many slice pairs the workspaces of a plan are sized for.
#include <cstdio>

#include "bst_internal.h"

static int bad = 0;
#define CHECK(c)                                                    \
    do {                                                            \
        if (!(c)) {                                                 \
            std::printf("FAIL line %d: %s\n", __LINE__, #c);        \
            ++bad;                                                  \
        }                                                           \
    } while (0)

constexpr size_t GiB = (size_t)1 << 30;

static bst_plan_s plan(int N, int V, int alpha, size_t free_bytes) {
    bst_plan_s p;
    p.N = N;
    p.V = V;
    p.alpha = alpha;
    p.M = alpha * N;
    p.ws_most = bsth::workspace_most(free_bytes);
    p.chunk_default = p.chunk_pairs = bsth::default_chunk(p.M, bsth::fwd_bytes_per_pair(&p), p.ws_most);
    return p;
}

// The forward workspace of a large call: two lanes of a chunk each.
static void forward() {
    const int N[] = {8, 16, 48, 256, 512, 1024, 1536, 2048, 4096}, V[] = {2, 64, 2048, 20000};
    const size_t free_bytes[] = {GiB / 4, GiB, 8 * GiB, 270 * GiB};
    for (int n : N)
        for (int v : V)
            for (int alpha = 1; alpha <= 2; ++alpha)
                for (size_t f : free_bytes) {
                    if (alpha * n > 4096 || !bsth::supported_fft_length(alpha * n)) continue;
                    const bst_plan_s p = plan(n, v, alpha, f);
                    const size_t per = bsth::fwd_bytes_per_pair(&p), ws = 2 * p.chunk_pairs * per;
                    CHECK(p.chunk_pairs >= 1 && p.chunk_pairs <= 256);
                    CHECK(p.chunk_pairs == 1 || (ws <= 4 * GiB && ws <= f / 16));
                }
    // plenty of memory: at least 8 pairs up to 4096 rays, one pair of 4096 rays and 20000 angles costs 0.8 GB
    CHECK(plan(2048, 2048, 2, 270 * GiB).chunk_pairs == 8);
    CHECK(plan(4096, 4096, 1, 270 * GiB).chunk_pairs == 8);
    CHECK(plan(4096, 20000, 1, 270 * GiB).chunk_pairs == 2);
    CHECK(plan(256, 256, 2, 270 * GiB).chunk_pairs == 32);
    // little of it: one pair a lane, a quarter of a GiB at 2048 rays
    CHECK(plan(2048, 2048, 2, 4 * GiB).chunk_pairs == 1);
}

int main() {
    forward();
    if (!bad) std::printf("OK\n");
    return bad != 0;
}

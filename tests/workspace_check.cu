// Test-only host program (compiled and run by tests/test_workspace_rules.py, no
// GPU needed): how many slice pairs the workspaces of a plan are sized for, and the
// rules that ask for the device's number of SMs.
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

// What the autotuner allocates: the rays, the volume and the largest workspace.
static void autotuner() {
    struct { int N, V, alpha; size_t room; } cases[] = {
        {2048, 2048, 2, 135 * GiB}, {2048, 2048, 2, 3 * GiB}, {2048, 2048, 2, GiB}, {4096, 20000, 1, 135 * GiB},
        {4096, 20000, 1, 20 * GiB}, {4096, 20000, 1, 4 * GiB}, {512, 512, 2, 135 * GiB}, {64, 64, 2, GiB / 2},
        {8, 8, 2, GiB}};
    for (const auto& c : cases)
        for (int kind : {BST_GRID_BILINEAR, BST_GRID_KAISER_BESSEL})
            for (int slices : {4, 64, 4096})
                for (int lanes : {1, 2}) {
                    bst_plan_s p = plan(c.N, c.V, c.alpha, 2 * c.room);
                    p.grid_kind = kind;
                    p.max_lanes = lanes;
                    const bsth::TuneRun r = bsth::tune_run(&p, slices, c.room);
                    CHECK(!r.shapes.empty() && r.slices >= 2);
                    size_t ws = 0;
                    int most = 0;
                    for (const bst_fwd_config_t& s : r.shapes) {
                        CHECK(s.chunk_pairs >= 1 && s.chunk_pairs <= 256);
                        most = std::max(most, s.chunk_pairs);
                        ws = std::max(ws, bsth::fwd_ws_bytes(&p, r.slices, s.chunk_pairs));
                    }
                    CHECK(ws == r.ws);
                    CHECK(r.ws + ((size_t)c.V * c.N + (size_t)c.N * c.N) * sizeof(float) * r.slices <= c.room);
                    if (c.room > 100 * GiB && slices < 4096) {   // everything fits: all candidates, the slices asked for
                        CHECK(most == std::min(256, 2 * p.chunk_default));
                        CHECK(r.slices == std::max(slices, 4 * most));
                    }
                }
}

// The adjoint: a pair alone, or what stays within the bound.
static void adjoint() {
    const int N[] = {8, 48, 512, 1024, 1536, 2048}, V[] = {2, 64, 2048, 20000};
    const size_t free_bytes[] = {GiB / 4, GiB, 4 * GiB, 270 * GiB};
    for (int n : N)
        for (int v : V)
            for (size_t f : free_bytes)
                for (int pairs : {1, 2, 3, 5, 64, 1000}) {
                    const bst_plan_s p = plan(n, v, 2, f);
                    const int c = bsth::adj_chunk(&p, pairs);
                    CHECK(c >= 1 && c <= pairs);
                    CHECK(c == 1 || c * bsth::adj_bytes_per_pair(&p) <= f / 16);
                }
    const bst_plan_s p = plan(1024, 1024, 2, 270 * GiB), q = plan(2048, 2048, 2, 270 * GiB);
    CHECK(bsth::adj_chunk(&p, 64) == 8 && bsth::adj_chunk(&p, 3) == 3 && bsth::adj_chunk(&q, 64) == 2);
}

// Shapes by the blocks per SM: the same number of blocks an SM gives the same shape.
static void per_sm() {
    auto is = [](bsth::SsShape s, int h, int r) { return s.h == h && s.r == r; };
    CHECK(is(bsth::ss_shape(512, 16, 152), 2, 4) && is(bsth::ss_shape(512, 20, 152), 1, 4));
    CHECK(is(bsth::ss_shape(512, 8, 152), 1, 4) && is(bsth::ss_shape(192, 16, 152), 1, 2));
    CHECK(is(bsth::ss_shape(64, 1, 152), 1, 1) && is(bsth::ss_shape(64, 1, 16), 1, 2));
    CHECK(is(bsth::ss_shape(512, 16, 8), 2, 4) && is(bsth::ss_shape(192, 16, 19), 2, 4));
    CHECK(is(bsth::ss_shape(512, 16, 1520), 1, 2) && is(bsth::ss_shape(192, 16, 1520), 1, 1));
    bst_plan_s p = plan(1024, 1024, 2, 270 * GiB);
    for (int sms : {8, 148, 152}) {
        p.sms = sms;
        CHECK(bsth::adj_fg_blocks(&p, 8) == (2 * sms + 7) / 8 && bsth::adj_fg_blocks(&p, 1000) == 1);
    }
}

int main() {
    per_sm();
    forward();
    adjoint();
    autotuner();
    if (!bad) std::printf("OK\n");
    return bad != 0;
}

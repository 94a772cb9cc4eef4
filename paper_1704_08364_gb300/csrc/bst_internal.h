// bst_internal.h -- plan object and host-side helpers shared by the
// translation units of libbst (not part of the public ABI).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "../../include/bst.h"
#include "bst_geo.cuh"

struct bst_plan_s {
    int N = 0, V = 0, M = 0, alpha = 0;
    int device = 0;
    int sms = 0;                    // multiprocessors of the device
    std::vector<double> theta;      // angles as given (float32 widened exactly)
    // device tables owned by the plan
    float2* tw = nullptr;           // [M] exp(-2 pi i m / M)
    float4* dir = nullptr;          // [V+2] angle directions, double-float
    float* invdth = nullptr;        // [V+1]
    int* lut = nullptr;             // [L]
    int L = 0;
    float lut_scale = 0.f;
    int uniform = 0;                // evenly spaced angles (bracket estimate by arithmetic)
    float th0 = 0.f, inv_step = 0.f;
    double2* cs64 = nullptr;        // [V] (cos, sin) in double, slant-stack tile origins
    float2* cs32 = nullptr;         // [V] (cos, sin) in float, slant-stack tile offsets
    float* wq = nullptr;            // [V] trapezoid weights of Eq. 2
    int* err = nullptr;             // sticky device error word
    // gridding geometry of the half grid c' in [0, M/2), [M/2][M], built at plan
    // creation: (bracket J << 16) | floor(rho) (J = -2: the point is zero) and
    // (angle fraction, radius fraction)
    int* geo_J = nullptr;
    float2* geo_f = nullptr;
    // P5 gridding kernel (BST_GRID_BILINEAR or BST_GRID_KAISER_BESSEL) and the
    // KB tables: kernel table, deapodization 1/C per output index, per-strip
    // sample lists and work items (built by bst_plan_set_gridding)
    int grid_kind = 0;
    int kb_w = 0;
    float kb_poly[13] = {0};        // phi as a degree-12 polynomial in t = 2 (2x/W)^2 - 1
    float* kb_dk = nullptr;         // [N]
    int* kb_start = nullptr;        // [kb_nstrips + 1] first item of each strip
    int* kb_list = nullptr;         // [kb_n] sample ids
    int4* kb_items = nullptr;       // (band, first entry, end entry, 1 if the band has others)
    size_t kb_n = 0;
    int kb_nstrips = 0;
    int chunk_pairs = 1;            // slice pairs per chunk of the forward path
    int chunk_default = 1;          // the chunk that the plan started with (bsth::default_chunk)
    size_t ws_most = 0;             // bytes of a workspace with more than one pair in flight
    int maxr = 16;                  // FFT radix schedule of the forward path (16 or 8)
    int fwd_layout = 0;             // a bst_layout_t (interleaved at creation; autotuned)
    int pair_fast = 0;              // gridding blocks ordered pair-fastest (autotuned)
    int max_lanes = 2;              // streams alternating chunks (1 or 2)
    int grid_xchg = 0;              // register-fed paired gridding (0 or 1)
    // two plan-owned streams that alternate chunks of the forward path (fork
    // from and join back to the caller's stream with events), created on first use
    cudaStream_t lane[3] = {nullptr, nullptr, nullptr};
    cudaEvent_t ev_fork = nullptr;
    cudaEvent_t ev_join[3] = {nullptr, nullptr, nullptr};
    // bst_fbp_host: upload and download streams and their events, created on first use
    cudaStream_t hs[2] = {nullptr, nullptr};
    cudaEvent_t hev[7] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    // gridding cell lists for the adjoint, built on first use
    int* cell_start = nullptr;      // [(V+1) M + 1]
    int* cell_pts = nullptr;        // [n] index c * M + r of each Cartesian point
    float2* cell_w = nullptr;       // [n] (fth, frac) of each point
    int cell_n = 0;
    bool cells_built = false;
    // optional per-stage timing: an event after every launch (see bst_plan_set_timing)
    bool timing = false;
    std::vector<cudaEvent_t> ev_pool;
    std::vector<int> ev_stage;     // stage that ended at each recorded event (-1: start mark)
    size_t ev_used = 0;
    double stage_ms[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    long long stage_launches[8] = {0, 0, 0, 0, 0, 0, 0, 0};

    bst::Geo geo() const {
        bst::Geo g;
        g.dir = dir;
        g.invdth = invdth;
        g.lut = lut;
        g.V = V;
        g.M = M;
        g.L = L;
        g.lut_scale = lut_scale;
        g.uniform = uniform;
        g.th0 = th0;
        g.inv_step = inv_step;
        return g;
    }
};

namespace bsth {

// chunks of the forward path in flight at once, each on its own stream with its
// own workspace (a third one measured no faster than two at 2048^3)
constexpr int kMaxLanes = 2;
static_assert(kMaxLanes <= (int)(sizeof(bst_plan_s::lane) / sizeof(cudaStream_t)) &&
                  kMaxLanes <= (int)(sizeof(bst_plan_s::ev_join) / sizeof(cudaEvent_t)),
              "the plan holds a stream and a join event per lane");

// A plan's tables live on the device that was current at its creation; the
// calls that launch work or build tables for it check that it is current.
inline bool on_plan_device(const bst_plan_s* p) {
    int dev = -1;
    return cudaGetDevice(&dev) == cudaSuccess && dev == p->device;
}

// The opt-in to more than 48 KB of dynamic shared memory is an attribute of a
// kernel on one device.  A launch site keeps one bit per device in `done` and
// runs `set` (which sets its kernels' attributes on the current device) the
// first time it launches on that device; on devices beyond 63 it runs `set`
// every time.
template <class F>
inline bool once_per_device(std::atomic<unsigned long long>& done, F&& set) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    const unsigned long long bit = (dev >= 0 && dev < 64) ? 1ull << dev : 0ull;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return true;
    if (!set()) return false;
    if (bit) done.fetch_or(bit, std::memory_order_release);
    return true;
}

inline bool supported_fft_length(int M) {
    int m = M;
    if (m % 3 == 0) m /= 3;
    if (m < 16 || (m & (m - 1)) != 0) return false;
    return M >= 16 && M <= 4096;
}

inline bool check_cuda(cudaError_t e) { return e == cudaSuccess; }

// byte sizes of the per-pair workspace of the forward path (one lane)
inline size_t fwd_bytes_per_pair(const bst_plan_s* p) {
    const size_t rows_t = (size_t)((p->N + 3) / 4) * 4;
    return ((size_t)p->V * p->M + rows_t * p->M) * sizeof(float2);
}

// Slice pairs of a group of the interleaved layout for FFT length M (1: the
// length has none): 256 / (threads per line), at most 8 and a multiple of the
// rows that a half-warp covers (bst_inter.cuh).
__host__ __device__ constexpr int inter_pairs_of(int M) {
    const int tpl = M % 3 == 0 ? M / 12 : M / 16;
    const int c = 256 / tpl > 8 ? 8 : tpl >= 256 ? 2 : 256 / tpl;
    return c > 0 && tpl % (16 / c) == 0 ? c : 1;
}

// Bytes that a workspace of a plan may take with more than one slice pair in flight (a
// lane, on the forward path): 4 GiB, less where little device memory is free at the plan's creation.
inline size_t workspace_most(size_t free_bytes) { return std::min<size_t>((size_t)4 << 30, free_bytes / 16); }

// Slice pairs per chunk that a plan starts with: 64 MiB of workspace, but at least 8
// pairs (whole groups), which fill several waves of blocks at every length; fewer,
// down to one, where two lanes of them would take more than `most` bytes.  Chunks
// of 2, 4, 8, 16 pairs: 64 x 2048 x 2048 4421, 4354, 4299, 4258 us; 512 x 512 x 512
// 2360, 1751, 1656, 1651 us.  8 pairs of 2048 x 2048 at pad factor 2 take 2 GiB.
inline int default_chunk(int M, size_t per_pair, size_t most) {
    const size_t fit = std::min<size_t>(256, ((size_t)64 << 20) / per_pair);
    const size_t want = std::max<size_t>(8, fit & ~(size_t)7), cap = most / (kMaxLanes * per_pair);
    if (cap >= want) return (int)want;
    const size_t g = (size_t)inter_pairs_of(M);
    return (int)std::max<size_t>(1, cap >= g ? cap / g * g : cap);
}

// Slice pairs per chunk for a call of `pairs` pairs with at most `most` a chunk.
// A call that would be one chunk is split over the two lanes, in whole groups,
// where the halves still fill the GPU: one half's gridding then overlaps the
// other's FFTs.  The line, pairs M^2 >= 2^23, is a call of about 80 us: below it a
// half's kernels are shorter than their launches.
inline int fwd_chunk(const bst_plan_s* p, int pairs, int most) {
    const int c = std::min(pairs, most);
    if (p->max_lanes < 2 || c < pairs || pairs < 2 || (long long)pairs * p->M * p->M < (1ll << 23)) return c;
    const int g = inter_pairs_of(p->M), h = (pairs + 1) / 2;
    return std::min(pairs, (h + g - 1) / g * g);
}

// bytes of the per-call tables of bst_fbp_prep (weight times phase of every
// bin, window), behind the lanes of the workspace
inline size_t prep_table_bytes(const bst_plan_s* p) {
    return ((size_t)p->M * sizeof(float2) + (size_t)p->N * sizeof(float) + 255) & ~(size_t)255;
}

// bytes of the forward workspace for `slices` slices in chunks of at most `most` pairs
inline size_t fwd_ws_bytes(const bst_plan_s* p, int slices, int most) {
    const int pairs = (slices + 1) / 2;
    const int chunk = fwd_chunk(p, pairs, most);
    const int nchunks = (pairs + chunk - 1) / chunk;
    const int lanes = std::min(std::min(nchunks, kMaxLanes), std::max(p->max_lanes, 1));   // chunks in flight
    return (size_t)lanes * chunk * fwd_bytes_per_pair(p) + prep_table_bytes(p);
}

// rows of T of a slice pair; bytes of a slice pair of the adjoint and the filter gradient
inline size_t adj_rows_t(const bst_plan_s* p) { return (size_t)((p->N + 3) / 4) * 4; }
inline size_t adj_bytes_per_pair(const bst_plan_s* p) {
    return (std::max(adj_rows_t(p), (size_t)p->V) * p->M + (size_t)p->M * p->M) * sizeof(float2);
}

// Slice pairs that the adjoint has in flight: as many as fit in 512 MiB, whole groups
// of four where there are more, and at least the pairs that the polar kernel takes
// together; fewer, down to one, where that exceeds the plan's bound.
inline int adj_chunk(const bst_plan_s* p, int pairs) {
    const size_t per = adj_bytes_per_pair(p), group = p->M >= 3072 ? 2 : 4;
    size_t c = std::max(std::min(group, p->ws_most / per), std::min<size_t>((size_t)512 << 20, p->ws_most) / per);
    if (c > 4) c &= ~(size_t)3;
    else if (c == 3 && group == 4) c = 2;   // three take the space of four
    return (int)std::min<size_t>((size_t)pairs, std::max<size_t>(c, 1));
}

// Angle blocks per pair of the filter gradient: two blocks an SM over the chunk's pairs.
inline int adj_fg_blocks(const bst_plan_s* p, int chunk) {
    const int tpl = (p->M % 3 == 0) ? p->M / 12 : p->M / 16;
    const int lpc = std::max(1, 256 / tpl);
    return std::max(1, std::min((p->V + lpc - 1) / lpc, (2 * p->sms + chunk - 1) / chunk));
}

// Slant stack: 4 h slices and r pixels a thread, by the blocks per SM that each shape
// gives.  Eight slices (four pixels) read a window for twice the slices, but a block
// takes 7/4 of the time of one of four slices, and below three blocks an SM its longer
// chain shows.  With four slices, more pixels a thread do less work in all, and
// fewer have the shorter chain.  300 angles, us with one, two, four pixels: 64 x 64
// 57, 61, 77; 16 slices of 192 x 192 130, 89, 91; 5 of 384 x 384 228, 165, 126;
// four and eight slices: 20 of 512 x 512 467, 494; 40 904, 754.
struct SsShape {
    int h, r;
};
inline SsShape ss_shape(int N, int slices, int sms) {
    const auto blocks = [&](int h, int r) {
        return (long long)((N + 31) / 32) * ((N + 4 * r - 1) / (4 * r)) * ((slices + 4 * h - 1) / (4 * h));
    };
    const long long b4 = blocks(1, 4), c4 = (b4 + sms - 1) / sms, c8 = (blocks(2, 4) + sms - 1) / sms;
    if (c8 >= 3 && 7 * c8 < 4 * c4) return {2, 4};
    if (5 * b4 > 12 * sms) return {1, 4};
    return {1, blocks(1, 1) > sms ? 2 : 1};
}

// The candidate launch shapes of the autotuner, largest chunk first: for bilinear
// plans the interleaved layout (where the length has it) and the paired one; twice
// the default chunk, the default and half of it (a larger chunk fills more waves of
// blocks, a smaller one keeps the intermediates in L2); either block order.  The
// lane count stays the plan's.  Radix 8 (never fewer passes), the packed layout
// and the paired gather through shared memory measured slower at every length
// and are left to bst_plan_set_forward_config.
inline std::vector<bst_fwd_config_t> tune_candidates(const bst_plan_s* p) {
    std::vector<bst_fwd_config_t> out;
    std::vector<int> layouts;
    if (p->grid_kind != BST_GRID_BILINEAR) {
        layouts = {BST_LAYOUT_PACKED};
    } else {
        if (inter_pairs_of(p->M) > 1) layouts.push_back(BST_LAYOUT_INTERLEAVED);
        layouts.push_back(BST_LAYOUT_PAIRED);
    }
    int last = 0;
    for (int ch : {std::min(256, 2 * p->chunk_default), p->chunk_default, std::max(1, p->chunk_default / 2)}) {
        if (ch == last) continue;
        last = ch;
        for (int l : layouts)
            for (int pf : {0, 1}) out.push_back(bst_fwd_config_t{16, l, ch, pf, p->max_lanes, 1});
    }
    return out;
}

// What the autotuner runs, within `room` bytes where it can: every candidate on
// `slices` slices, but at least one chunk of the largest on each lane.  Where that
// is too much, fewer slices, then without the largest chunks, and with the smallest
// chunk alone as few slices as one pair.
struct TuneRun {
    std::vector<bst_fwd_config_t> shapes;
    int slices = 0;
    size_t ws = 0;      // workspace of the largest candidate
};
inline TuneRun tune_run(const bst_plan_s* p, int slices, size_t room) {
    const size_t per_slice = ((size_t)p->V * p->N + (size_t)p->N * p->N) * sizeof(float);
    TuneRun r;
    r.shapes = tune_candidates(p);
    for (;;) {
        const int most = r.shapes.front().chunk_pairs;
        const bool last = r.shapes.back().chunk_pairs == most;
        const int least = last ? 2 : 2 * kMaxLanes * most;
        for (r.slices = std::max(slices, 2 * kMaxLanes * most);; r.slices = std::max(least, r.slices / 2)) {
            r.ws = 0;
            for (const bst_fwd_config_t& c : r.shapes) r.ws = std::max(r.ws, fwd_ws_bytes(p, r.slices, c.chunk_pairs));
            if (r.ws + r.slices * per_slice <= room) return r;
            if (r.slices == least) break;
        }
        if (last) return r;
        r.shapes.erase(std::remove_if(r.shapes.begin(), r.shapes.end(),
                                      [&](const bst_fwd_config_t& c) { return c.chunk_pairs == most; }),
                       r.shapes.end());
    }
}

}  // namespace bsth

// Record a timing mark on `st` after a launch of `stage` (or a start mark
// with stage -1).  No-op unless timing is enabled on the plan.
void bst_timing_mark(bst_plan_s* p, cudaStream_t st, int stage);

// launchers (one dispatch on M each), defined in the kernel translation units
bst_status_t bst_launch_forward(bst_plan_s* p, const float* sino, int slices, int mode, const float* g,
                                float* vol, void* ws, size_t ws_bytes, cudaStream_t st);
// as bst_launch_forward, with at most max_chunk slice pairs per chunk of the
// workspace and up to `lanes` (1 or 2) streams alternating the chunks
bst_status_t bst_launch_forward_chunked(bst_plan_s* p, const float* sino, int slices, int mode, const float* g,
                                        float* vol, void* ws, cudaStream_t st, int max_chunk, int lanes);
namespace bst {
struct PrepArgs;
}
// the forward path for pad factor 1 or 2 (fbp_pad1.cu, fbp_pad2.cu); prep may be null
bst_status_t bst_forward_pad1(bst_plan_s* p, const float* sino, int slices, int mode, const float* g, float* vol,
                              void* ws, cudaStream_t st, int max_chunk, int lanes, const bst::PrepArgs* prep);
bst_status_t bst_forward_pad2(bst_plan_s* p, const float* sino, int slices, int mode, const float* g, float* vol,
                              void* ws, cudaStream_t st, int max_chunk, int lanes, const bst::PrepArgs* prep);
// create the plan's two chunk streams and their events (false on failure)
bool bst_ensure_lanes(bst_plan_s* p);
bst_status_t bst_launch_adjoint(bst_plan_s* p, int mode, const float* g, const float* vol, int slices,
                                float* sino, void* ws, size_t ws_bytes, cudaStream_t st);
bst_status_t bst_launch_filter_grad(bst_plan_s* p, const float* sino, const float* gvol, int slices,
                                    float* grad_g, void* ws, size_t ws_bytes, cudaStream_t st);
bst_status_t bst_launch_backward(bst_plan_s* p, const float* sino, const float* gvol, int slices, const float* g,
                                 float* grad_sino, float* grad_g, void* ws, cudaStream_t st);
bst_status_t bst_launch_brute(bst_plan_s* p, const float* sino, int slices, const float* g, float* vol,
                              void* ws, size_t ws_bytes, cudaStream_t st);
bst_status_t bst_build_cells(bst_plan_s* p, cudaStream_t st);
bst_status_t bst_build_geo_table(bst_plan_s* p);
// KB gridding + column inverse FFT of np pairs (kb.cu)
bst_status_t bst_launch_kb_col(bst_plan_s* p, const float2* Z, float2* T, int np, cudaStream_t st);
void bst_free_kb(bst_plan_s* p);
double bst_bessel_i0(double x);
// look up (and cache) the device address of bst_fbp_noalloc's scratch array
// on the current device (noalloc.cu); called by bst_plan_create
bst_status_t bst_noalloc_setup_current_device();
size_t bst_adjoint_ws(const bst_plan_s* p, int slices);
size_t bst_brute_ws(const bst_plan_s* p, int slices, int filtered);

// mode values shared by the launchers
enum { BSTK_FILTER = 0, BSTK_BACKPROJECT = 1, BSTK_RAW = 2 };
// flag or-ed into the ray-stage mode: also multiply by the polar cell area
// |k| (1/4 at k = 0) for KB gridding
enum { BSTK_KBW = 8 };
// flag or-ed into the ray-stage mode: write the spectrum in the paired
// (Z[k], Z[-k]) layout read by the paired bilinear gridding kernel
enum { BSTK_PAIRED = 16 };

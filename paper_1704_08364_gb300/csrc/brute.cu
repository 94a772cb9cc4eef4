// brute.cu -- slant-stack backprojection (brute_backproject), the O(N^3)
// per-slice comparator of Sec. 2, with an optional ramp-type prefilter.
//
//   k_ss_filter  per angle and slice pair: zero-pad to M, FFT along t,
//                multiply by h_k / M (h_k = |sigma_k| g[k], h_0 = dsigma/4 g[0],
//                h_{M/2} = 0), inverse FFT, crop to N samples.
//   k_ss_bp      Eq. 2 as a Riemann sum: b[r][c] = sum_j w_j y_j(i_f) with
//                i_f = (c - N/2) cos t_j + (r - N/2) sin t_j + N/2 and linear
//                interpolation (zero outside [0, N-1]).  A tile of 32 columns
//                and 4 or 16 rows and 4 or 8 slices per block (the slices share
//                the geometry, as the paper's blocks of Q sinograms do); batches
//                of angles are staged in shared memory with zero fill, so the
//                inner loop has no bounds tests.  The tile centre's detector
//                coordinate is computed in double precision, the per-pixel
//                offset from it (< 18 samples) in float.
#include <cuda_runtime.h>

#include <algorithm>

#include "bst_fft.cuh"
#include "bst_internal.h"

namespace bst {

template <int M> __host__ __device__ constexpr int brute_tpl() { return (M % 3 == 0) ? M / 12 : M / 16; }

struct SsRaySrc {
    const float* ya;
    const float* yb;
    int N, M;
    bool live;
    static constexpr bool kSmem = false;
    __device__ __forceinline__ float2 load(int m) const {
        int i = m + (N >> 1);
        if (i >= M) i -= M;
        if (!live || i >= N) return make_float2(0.f, 0.f);
        return make_float2(__ldg(ya + i), yb ? __ldg(yb + i) : 0.f);
    }
};

// multiply the spectrum by h_k / M while storing it back into shared memory
struct RampSmem {
    float2* p;
    const float* g;
    int M;
    float dsig;
    static constexpr bool kSmem = true;
    __device__ __forceinline__ void store(int k, float2 v) const {
        const int ak = k <= (M >> 1) ? k : M - k;
        float h;
        if (ak == (M >> 1)) h = 0.f;
        else {
            const float gk = g ? __ldg(g + ak) : 1.f;
            h = (ak == 0 ? 0.25f * dsig : (float)ak * dsig) * gk;
        }
        h = h / (float)M;
        p[k + (k >> 4)] = make_float2(v.x * h, v.y * h);
    }
    __device__ __forceinline__ float2 load(int i) const { return p[i + (i >> 4)]; }
};

struct CropDst {
    float* qa;
    float* qb;
    int N, M;
    bool live;
    static constexpr bool kSmem = false;
    __device__ __forceinline__ void store(int m, float2 v) const {
        if (!live) return;
        const int i = signed_freq(m, M) + (N >> 1);
        if (i < 0 || i >= N) return;
        qa[i] = v.x;
        if (qb) qb[i] = v.y;
    }
};

template <int M, int TPL, int LPC>
__global__ void __launch_bounds__(TPL * LPC)
    k_ss_filter(const float* __restrict__ sino, int slices, int N, int V, const float* __restrict__ g, float dsig,
                float* __restrict__ q, const float2* __restrict__ tw) {
    extern __shared__ float2 smem[];
    const int line = threadIdx.x / TPL, t = threadIdx.x % TPL;
    const int j = blockIdx.x * LPC + line;
    const int sa = 2 * blockIdx.y, sb = sa + 1;
    const bool live = j < V;
    const int jj = live ? j : 0;
    SsRaySrc src{sino + ((size_t)sa * V + jj) * N, sb < slices ? sino + ((size_t)sb * V + jj) * N : nullptr, N, M,
                 live};
    float2* base = smem + line * smem_line_len(M);
    RampSmem mid{base, g, M, dsig};
    SmemLine sm{base};
    fft_line<M, TPL, false>(t, src, mid, sm, tw);
    __syncthreads();
    CropDst dst{q + ((size_t)sa * V + jj) * N, sb < slices ? q + ((size_t)sb * V + jj) * N : nullptr, N, M, live};
    fft_line<M, TPL, true>(t, sm, dst, sm, tw);
}

constexpr int SS_TX = 32;      // pixels of a tile along x (a warp's lanes)
constexpr int SS_WARPS = 4;    // warps a block; warp w covers rows w R .. w R + R - 1 of the tile
constexpr int SS_AB = 12;      // angles per staged batch

// staged samples per angle and slice: 31 |cos| + (4 R - 1) sin + the window
template <int R> __host__ __device__ constexpr int ss_w() { return R > 1 ? 40 : 36; }

// acc += w * z for the 4 H slices, with packed FP32 multiply-adds (one issue
// slot for two)
template <int H>
__device__ __forceinline__ void fma_slices(float2 (&acc)[H][2], float w, const float4 (&z)[H]) {
    const float2 ww = make_float2(w, w);
#pragma unroll
    for (int h = 0; h < H; ++h) {
        acc[h][0] = __ffma2_rn(ww, make_float2(z[h].x, z[h].y), acc[h][0]);
        acc[h][1] = __ffma2_rn(ww, make_float2(z[h].z, z[h].w), acc[h][1]);
    }
}

// A thread holds R vertically adjacent pixels of 4 H slices.  Their detector
// coordinates v_p = v_0 + p sin t (0 <= sin t <= 1) lie in
// [floor(v_0), floor(v_0) + p + 1), so the samples floor(v_0) .. floor(v_0) + R
// serve all R of them: sample k weighs max(0, 1 - |v_p - k|), which is linear
// interpolation, and is zero for k > p + 1.  Each sample is read once per R
// pixels, four slices to a 16-byte load (lanes along x read consecutive
// 16-byte words: no bank conflicts): per pixel, angle and 8 slices 8.6
// shared-memory wavefronts on average with R = 4 against 16 for two reads per
// pixel and slice.  A batch of angles with a value that is not finite reads the
// two samples of each pixel instead (a zero weight would not hide it).  What
// bounds it: FP32 issue (64 to 70 %) and the shared-memory wavefronts (61 to 71 %),
// about alike, and with few blocks the chain of a batch: staging loads, barrier, sums.  The loads of a
// warp for a whole batch are issued together, and the next batch's geometry with
// them (six blocks of eight slices an SM leave the registers): 512 x 512, 512 angles, 16
// slices 632 -> 555 us (this kernel alone), 64 x 64, 300 angles, one slice 75 -> 57 us.  The form with
// one pixel a thread, two 4-byte loads a slice and 103 warp instructions per 32
// pixels, angle and 8 slices took 1033 us for the former.
template <int H, int R>
__global__ void __launch_bounds__(32 * SS_WARPS, H > 1 ? 6 : R > 1 ? 7 : 8)
    k_ss_bp(const float* __restrict__ y, int S, int V, int N, const double2* __restrict__ cs64,
            const float2* __restrict__ cs32, const float* __restrict__ wq, float* __restrict__ vol) {
    constexpr int W = ss_w<R>();
    constexpr int TY = SS_WARPS * R;
    __shared__ float4 seg[SS_AB][H][W];
    // per angle of the batch (double-buffered): cos, sin, fraction of the tile
    // centre's coordinate, weight; staged index of its integer part (low half)
    // and the last sample after floor(v_0) that a pixel can reach (high half),
    // first staged sample
    __shared__ float4 ang[2][SS_AB];
    __shared__ int2 pos[2][SS_AB];
    // the sums over the batches so far: a batch's sum starts at zero and is
    // added once, so that rounding does not grow with the number of angles
    __shared__ float4 total[R * H][32 * SS_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c0 = blockIdx.x * SS_TX, r0 = blockIdx.y * TY;
    const int s0 = blockIdx.z * (4 * H);
    // a batch's geometry by its first SS_AB threads: the loads, and what follows them
    double2 cs;
    float2 cf;
    float wj;
    auto geometry_load = [&](int jb) {
        const int j = jb + threadIdx.x;
        const bool in = threadIdx.x < SS_AB && j < V;
        cs = in ? cs64[j] : make_double2(0.0, 0.0);
        cf = in ? cs32[j] : make_float2(0.f, 0.f);
        wj = in ? wq[j] : 0.f;
    };
    auto geometry = [&](int buf, int jb) {
        if (threadIdx.x < SS_AB && jb + (int)threadIdx.x < V) {
            const double fc = (double)(c0 + SS_TX / 2 - N / 2) * cs.x + (double)(r0 + TY / 2 - N / 2) * cs.y +
                              (double)(N / 2);
            const double mn = fc - (SS_TX / 2) * cs.x - (TY / 2) * cs.y + fmin(0.0, (SS_TX - 1) * cs.x);
            const int lo = (int)floor(mn) - 1, ic = (int)floor(fc);
            ang[buf][threadIdx.x] = make_float4(cf.x, cf.y, (float)(fc - (double)ic), wj);
            // pixel R - 1 lies below 1 + (R - 1) sin t; one more for its second sample
            const int top = R == 1 ? 1 : 2 + (int)((float)(R - 1) * cf.y);
            pos[buf][threadIdx.x] = make_int2((ic - lo) | (top << 16), lo);
        }
    };
    const float fx = (float)(lane - SS_TX / 2), fy = (float)(warp * R - TY / 2);
    geometry_load(0);
    geometry(0, 0);
    for (int jb = 0, buf = 0; jb < V; jb += SS_AB, buf ^= 1) {
        __syncthreads();   // this batch's geometry is there, the previous batch's samples are done with
        const int na = min(SS_AB, V - jb);
        bool odd = false;   // a staged value is not finite
        geometry_load(jb + SS_AB);
        // all of the warp's loads of the batch are issued before the first is used
        constexpr int NU = SS_AB / SS_WARPS, NI = (H * W + 31) / 32;
        float v[NU][NI][4];
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const int a = warp + u * SS_WARPS;
            const float* yj = y + (size_t)(jb + a) * N;
            const int lo = a < na ? pos[buf][a].y : N;
#pragma unroll
            for (int n = 0; n < NI; ++n) {
                const int it = lane + 32 * n, h = it >= W, g = lo + it - h * W;
                const bool in = it < H * W && g >= 0 && g < N;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int s = s0 + 4 * h + q;
                    v[u][n][q] = in && s < S ? __ldg(yj + (size_t)s * V * N + g) : 0.f;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const int a = warp + u * SS_WARPS;
            if (a >= na) break;
            const float w = ang[buf][a].w;
#pragma unroll
            for (int n = 0; n < NI; ++n) {
                const int it = lane + 32 * n, h = it >= W, i = it - h * W;
                if (it < H * W) {
                    const float4 z = make_float4(v[u][n][0] * w, v[u][n][1] * w, v[u][n][2] * w, v[u][n][3] * w);
                    seg[a][h][i] = z;
                    odd |= !(fabsf(z.x) + fabsf(z.y) + fabsf(z.z) + fabsf(z.w) < INFINITY);
                }
            }
        }
        geometry(buf ^ 1, jb + SS_AB);
        odd = __syncthreads_or(odd);
        float2 acc[R][H][2];
#pragma unroll
        for (int p = 0; p < R; ++p)
#pragma unroll
            for (int h = 0; h < H; ++h) acc[p][h][0] = acc[p][h][1] = make_float2(0.f, 0.f);
        if (R > 1 && odd) {
#pragma unroll 1
            for (int a = 0; a < na; ++a) {
                const float4 an = ang[buf][a];
                const float vx = fmaf(fx, an.x, an.z);
#pragma unroll
                for (int p = 0; p < R; ++p) {
                    const float v = fmaf(fy + (float)p, an.y, vx), fl = floorf(v);
                    const float4* base = &seg[a][0][(int)fl + (pos[buf][a].x & 0xffff)];
                    float4 z0[H], z1[H];
#pragma unroll
                    for (int h = 0; h < H; ++h) {
                        z0[h] = base[h * W];
                        z1[h] = base[h * W + 1];
                    }
                    fma_slices<H>(acc[p], 1.f - (v - fl), z0);
                    fma_slices<H>(acc[p], v - fl, z1);
                }
            }
        } else {
            for (int a = 0; a < na; ++a) {
                const float4 an = ang[buf][a];
                const int ps = pos[buf][a].x;
                const float vx = fmaf(fx, an.x, an.z);
                const float v0 = fmaf(fy, an.y, vx);
                const float fl = floorf(v0);
                const float4* base = &seg[a][0][(int)fl + (ps & 0xffff)];
                float d[R];   // coordinates from sample floor(v_0)
                d[0] = v0 - fl;
#pragma unroll
                for (int p = 1; p < R; ++p) d[p] = fmaf(fy + (float)p, an.y, vx) - fl;
#pragma unroll
                for (int k = 0; k <= R; ++k) {
                    if (k > 2 && k > ps >> 16) break;   // the same for the whole block
                    float4 z[H];
#pragma unroll
                    for (int h = 0; h < H; ++h) z[h] = base[h * W + k];
#pragma unroll
                    for (int p = k > 1 ? k - 1 : 0; p < R; ++p)
                        fma_slices<H>(acc[p],
                                      k == 0 ? __saturatef(1.f - d[p]) : __saturatef(1.f - fabsf(d[p] - (float)k)), z);
                }
            }
        }
#pragma unroll
        for (int p = 0; p < R; ++p)
#pragma unroll
            for (int h = 0; h < H; ++h) {
                float4& t = total[p * H + h][threadIdx.x];   // this thread's own
                const float2 lo = acc[p][h][0], hi = acc[p][h][1];
                const float4 o = jb ? t : make_float4(0.f, 0.f, 0.f, 0.f);
                t = make_float4(o.x + lo.x, o.y + lo.y, o.z + hi.x, o.w + hi.y);
            }
    }
    const int c = c0 + lane;
#pragma unroll
    for (int p = 0; p < R; ++p) {
        const int r = r0 + warp * R + p;
        if (r < N && c < N) {
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const float4 t = total[p * H + h][threadIdx.x];
                const float v[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int s = s0 + 4 * h + q;
                    if (s < S) vol[((size_t)s * N + r) * N + c] = v[q];
                }
            }
        }
    }
}

template <int H, int R>
static void launch_ss_bp(const bst_plan_s* p, const float* y, int slices, float* vol, cudaStream_t st) {
    const int N = p->N;
    const dim3 grid((N + SS_TX - 1) / SS_TX, (N + SS_WARPS * R - 1) / (SS_WARPS * R), (slices + 4 * H - 1) / (4 * H));
    k_ss_bp<H, R><<<grid, 32 * SS_WARPS, 0, st>>>(y, slices, p->V, N, p->cs64, p->cs32, p->wq, vol);
}

template <int M>
bst_status_t launch_ss_filter_M(bst_plan_s* p, const float* sino, int slices, const float* g, float* q,
                                cudaStream_t st) {
    constexpr int TPL = brute_tpl<M>();
    constexpr int LPC = (256 / TPL) > 1 ? 256 / TPL : 1;
    constexpr size_t S = (size_t)LPC * smem_line_len(M) * sizeof(float2);
    static std::atomic<unsigned long long> attr_done{0};
    if (!bsth::once_per_device(attr_done, [] {
            return S <= 48 * 1024 || cudaFuncSetAttribute(k_ss_filter<M, TPL, LPC>,
                                                          cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                          (int)S) == cudaSuccess;
        }))
        return BST_ERR_CUDA;
    const int pairs = (slices + 1) / 2;
    const float dsig = (float)((double)p->N / (2.0 * (double)M));
    bst_timing_mark(p, st, -1);
    k_ss_filter<M, TPL, LPC><<<dim3((p->V + LPC - 1) / LPC, pairs), TPL * LPC, S, st>>>(sino, slices, p->N, p->V, g,
                                                                                        dsig, q, p->tw);
    bst_timing_mark(p, st, 3);
    return BST_OK;
}

}  // namespace bst

size_t bst_brute_ws(const bst_plan_s* p, int slices, int filtered) {
    if (!filtered) return 0;
    return (size_t)slices * p->V * p->N * sizeof(float);
}

#define BST_FOR_EACH_M(X) \
    X(16) X(32) X(64) X(128) X(256) X(512) X(1024) X(2048) X(4096) X(48) X(96) X(192) X(384) X(768) X(1536) X(3072)

bst_status_t bst_launch_brute(bst_plan_s* p, const float* sino, int slices, const float* g, float* vol, void* ws,
                              size_t /*ws_bytes*/, cudaStream_t st) {
    const float* y = sino;
    if (g) {
        float* q = (float*)ws;
        bst_status_t s = BST_ERR_UNSUPPORTED_SIZE;
        switch (p->M) {
#define BST_CASE(m) \
    case m: s = bst::launch_ss_filter_M<m>(p, sino, slices, g, q, st); break;
            BST_FOR_EACH_M(BST_CASE)
#undef BST_CASE
        }
        if (s != BST_OK) return s;
        y = q;
    }
    const bsth::SsShape sh = bsth::ss_shape(p->N, slices, p->sms);
    bst_timing_mark(p, st, -1);
    if (sh.h == 2) bst::launch_ss_bp<2, 4>(p, y, slices, vol, st);
    else if (sh.r == 4) bst::launch_ss_bp<1, 4>(p, y, slices, vol, st);
    else if (sh.r == 2) bst::launch_ss_bp<1, 2>(p, y, slices, vol, st);
    else bst::launch_ss_bp<1, 1>(p, y, slices, vol, st);
    bst_timing_mark(p, st, 4);
    return cudaGetLastError() == cudaSuccess ? BST_OK : BST_ERR_CUDA;
}

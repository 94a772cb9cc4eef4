// fbp.cu -- plan-level entry points of the BST forward path: the plan's
// geometry table, the dispatch of bst_fbp / bst_backproject / bst_fbp_prep on
// the FFT length and the pad factor (the kernels are in bst_forward.cuh,
// instantiated by fbp_pad1.cu and fbp_pad2.cu), and bst_fbp_prep.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "bst_launch.cuh"

namespace bst {

// Plan set-up: the angular part of the geometry of every point (q, r') of the
// half grid q in [0, M/2) (the mirror half shares it), bracket -2 for points
// that are zero (outside the band, or the origin, which takes the DC mean).
__global__ void k_geo_table(Geo geo, int M, int* __restrict__ gJ, float2* __restrict__ gF) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)(M / 2) * M) return;
    const int q = (int)(idx / M), ridx = (int)(idx % M);
    const int ry = signed_freq(ridx, M);
    Polar P;
    int jk = (int)(-2 * 65536);
    float2 f = make_float2(0.f, 0.f);
    if (!(q == 0 && ry == 0) && polar_of(q, ry, geo, P)) {
        jk = P.J * 65536 + P.k0;
        f = make_float2(P.fth, P.frac);
    }
    gJ[idx] = jk;
    gF[idx] = f;
}

// The tables of the pre-reconstruction stages: cw[k] = weight(k) exp(+2 pi i k
// shift / M) and, with win, the window at the measured samples (evaluated in
// double; which samples lie inside it is decided in float).
__global__ void k_prep_tables(int M, int N, int mode, const float* __restrict__ g, float two_alpha, float shift,
                              float beta, float half, float2* __restrict__ cw, float* __restrict__ win) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < M) {
        double s, c;
        sincospi(2.0 * (double)signed_freq(i, M) * (double)shift / (double)M, &s, &c);
        const double w = (double)bin_weight(i, M, mode, g, two_alpha);
        cw[i] = make_float2((float)(w * c), (float)(w * s));
    }
    if (win && i < N) {
        const float uf = ((float)(i - (N >> 1)) - shift) * (2.f / (float)N) * (1.f / half);
        const double u = ((double)(i - (N >> 1)) - (double)shift) * (2.0 / (double)N) / (double)half;
        win[i] = fabsf(uf) <= 1.f ? (float)(cyl_bessel_i0((double)beta * sqrt(fmax(1.0 - u * u, 0.0))) /
                                            cyl_bessel_i0((double)beta))
                                  : 0.f;
    }
}

}  // namespace bst

static bst_status_t forward_dispatch(bst_plan_s* p, const float* sino, int slices, int mode, const float* g,
                                     float* vol, void* ws, cudaStream_t st, int max_chunk, int lanes,
                                     const bst::PrepArgs* prep) {
    return p->alpha == 2 ? bst_forward_pad2(p, sino, slices, mode, g, vol, ws, st, max_chunk, lanes, prep)
                         : bst_forward_pad1(p, sino, slices, mode, g, vol, ws, st, max_chunk, lanes, prep);
}

bst_status_t bst_launch_forward_chunked(bst_plan_s* p, const float* sino, int slices, int mode, const float* g,
                                        float* vol, void* ws, cudaStream_t st, int max_chunk, int lanes) {
    return forward_dispatch(p, sino, slices, mode, g, vol, ws, st, max_chunk, lanes, nullptr);
}

bst_status_t bst_launch_forward(bst_plan_s* p, const float* sino, int slices, int mode, const float* g, float* vol,
                                void* ws, size_t ws_bytes, cudaStream_t st) {
    const int pairs = (slices + 1) / 2;
    const int chunk = bsth::fwd_chunk(p, pairs, p->chunk_pairs);
    const int lanes = (int)std::min<size_t>(bsth::kMaxLanes, ws_bytes / ((size_t)chunk * bsth::fwd_bytes_per_pair(p)));
    return bst_launch_forward_chunked(p, sino, slices, mode, g, vol, ws, st, p->chunk_pairs, lanes);
}

bst_status_t bst_build_geo_table(bst_plan_s* p) {
    const size_t n = (size_t)(p->M / 2) * p->M;
    if (cudaMalloc((void**)&p->geo_J, n * sizeof(int)) != cudaSuccess) return BST_ERR_OUT_OF_MEMORY;
    if (cudaMalloc((void**)&p->geo_f, n * sizeof(float2)) != cudaSuccess) return BST_ERR_OUT_OF_MEMORY;
    bst::k_geo_table<<<(unsigned)((n + 255) / 256), 256>>>(p->geo(), p->M, p->geo_J, p->geo_f);
    if (cudaGetLastError() != cudaSuccess) return BST_ERR_CUDA;
    return cudaDeviceSynchronize() == cudaSuccess ? BST_OK : BST_ERR_CUDA;
}

extern "C" bst_status_t bst_fbp_prep(bst_plan_t p, const float* d_sino, int slices, const float* d_dark,
                                     const float* d_flat, float shift, float kb_beta, float kb_halfwidth,
                                     const float* d_g, float* d_volume, void* d_ws, size_t ws_bytes,
                                     bst_stream_t stream) {
    if (!p || !d_sino || !d_volume || slices <= 0) return BST_ERR_INVALID_ARGUMENT;
    if (!bsth::on_plan_device(p)) return BST_ERR_INVALID_ARGUMENT;
    if (d_dark && !d_flat) return BST_ERR_INVALID_ARGUMENT;
    if (!std::isfinite(shift) || std::fabs(shift) >= (float)p->N) return BST_ERR_INVALID_ARGUMENT;
    if (!(kb_beta >= 0.f) || !std::isfinite(kb_beta) || (kb_beta > 0.f && !(kb_halfwidth > 0.f)))
        return BST_ERR_INVALID_ARGUMENT;
    const size_t ns = (size_t)slices * p->V * p->N * sizeof(float), nv = (size_t)slices * p->N * p->N * sizeof(float);
    const uintptr_t a0 = (uintptr_t)d_sino, b0 = (uintptr_t)d_volume;
    if (a0 < b0 + nv && b0 < a0 + ns) return BST_ERR_INVALID_ARGUMENT;
    if (!d_ws || ws_bytes < bst_workspace_bytes(p, slices)) return BST_ERR_WORKSPACE_TOO_SMALL;
    const int chunk = bsth::fwd_chunk(p, (slices + 1) / 2, p->chunk_pairs);
    const size_t lane = (size_t)chunk * bsth::fwd_bytes_per_pair(p);
    const int lanes = (int)std::min<size_t>(bsth::kMaxLanes, (ws_bytes - bsth::prep_table_bytes(p)) / lane);
    float2* cw = (float2*)((char*)d_ws + lanes * lane);
    float* win = kb_beta > 0.f ? (float*)(cw + p->M) : nullptr;
    const cudaStream_t st = (cudaStream_t)stream;
    bst::k_prep_tables<<<(std::max(p->M, p->N) + 127) / 128, 128, 0, st>>>(
        p->M, p->N, BSTK_FILTER | (p->grid_kind == BST_GRID_KAISER_BESSEL ? BSTK_KBW : 0), d_g, (float)(2 * p->alpha),
        shift, kb_beta, kb_halfwidth, cw, win);
    const bst::PrepArgs pa{d_dark, d_flat, win, cw};
    return forward_dispatch(p, d_sino, slices, BSTK_FILTER, d_g, d_volume, d_ws, st, p->chunk_pairs, lanes, &pa);
}


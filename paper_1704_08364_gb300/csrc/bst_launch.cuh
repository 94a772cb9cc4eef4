// bst_launch.cuh -- host launcher of the BST forward path (the kernels are
// in bst_forward.cuh): per chunk of slice pairs, the ray, gridding and row
// kernels on one of up to two plan-owned streams, with the plan's launch
// shape (radix schedule, spectrum layout, chunk, block order, lanes).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>

#include "bst_forward.cuh"
#include "bst_inter.cuh"

namespace bst {

// ---------------------------------------------------------------------------
// host launcher

template <class K>
static bool set_smem(K kernel, size_t bytes) {
    if (bytes <= 48 * 1024) return true;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

// kernel<<<grid, block, smem, st>>>(args...); `chain`: with programmatic stream
// serialization, for kernels that start with chain_begin()
template <class... P, class... A>
static void launch(bool chain, void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = chain ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

template <int M> struct FwdCfg {
    static constexpr int TPL = tpl_of<M>();
    // ray kernel: 256 threads a block, or, for lengths whose line takes 256
    // threads, two interleaved angle rows in 512 (whole lines of the paired
    // layout per warp store)
    static constexpr bool ILV1 = TPL >= 256;
    static constexpr int LPC1 = ILV1 ? 2 : ((256 / TPL) > 1 ? 256 / TPL : 1);
    static constexpr int CPC = (128 / TPL) > 1 ? 128 / TPL : 1;
    static constexpr int TPC = (128 / (4 * TPL)) > 1 ? 128 / (4 * TPL) : 1;
    static constexpr size_t S1 = (size_t)LPC1 * ray_line_stride<M, ILV1>() * sizeof(float2);
    static constexpr size_t S2 = (size_t)CPC * smem_line_len(M) * sizeof(float2);
    static constexpr int CPCP = paired_cpc<M>();
    static constexpr size_t S2P = (size_t)2 * CPCP * smem_line_len(M) * sizeof(float2);
    // the register-fed gridding kernel: half-warps of 16 consecutive threads of a column
    static constexpr bool XCHG_OK = TPL % 16 == 0;
    static constexpr size_t S2X = (size_t)2 * smem_line_len(M) * sizeof(float2);
    static constexpr size_t S3 = (size_t)4 * TPC * row_line_stride<M>() * sizeof(float2);
};

// the shared-memory opt-in of the register-fed gridding kernel, where it exists
template <int M, int MAXR, int NC>
static bool set_smem_xchg() {
    using C = FwdCfg<M>;
    if constexpr (C::XCHG_OK) return set_smem(k_grid_col_xchg<M, C::TPL, MAXR, NC>, C::S2X);
    return true;
}

// shared memory of the interleaved kernels, and their opt-in, for the lengths
// that have them
template <int M> struct InterCfg {
    static constexpr int P = inter_pairs<M>(), LP = inter_lanes<P>(), TPL = tpl_of<M>();
    static constexpr bool OK = P > 1;
    static constexpr size_t S1 = (size_t)inter_ray_rows<M>() * LP * inter_stride<M>(LP) * sizeof(float2);
    static constexpr size_t S2 = (size_t)2 * P * inter_stride<M>(P) * sizeof(float2);
    static constexpr size_t S3 = (size_t)4 * inter_row_tiles<M>() * row_line_stride<M>() * sizeof(float2);
};
template <int M, int MAXR, int NC>
static bool set_smem_inter() {
    using I = InterCfg<M>;
    if constexpr (I::OK)
        return set_smem(k_ray_inter<M, MAXR, NC, false>, I::S1) && set_smem(k_ray_inter<M, MAXR, NC, true>, I::S1) &&
               set_smem(k_grid_inter<M, MAXR, NC>, I::S2) && set_smem(k_row_inter<M, MAXR, NC>, I::S3);
    return true;
}

template <int M, int MAXR, int NC>
bst_status_t launch_forward_M(bst_plan_s* p, const float* sino, int slices, int mode, const float* g, float* vol,
                              void* ws, cudaStream_t st, int max_chunk, int lanes, const PrepArgs* prep) {
    using C = FwdCfg<M>;
    static std::atomic<unsigned long long> attr_done{0};
    if (!bsth::once_per_device(attr_done, [] {
            return set_smem(k_ray_fft<M, C::TPL, C::LPC1, MAXR, NC, C::ILV1>, C::S1) &&
                   set_smem(k_ray_fft_prep<M, C::TPL, C::LPC1, MAXR, NC, C::ILV1>, C::S1) &&
                   set_smem(k_grid_col<M, C::TPL, C::CPC, MAXR, NC>, C::S2) &&
                   set_smem(k_grid_col_paired<M, C::TPL, C::CPCP, MAXR, NC>, C::S2P) &&
                   set_smem_xchg<M, MAXR, NC>() && set_smem_inter<M, MAXR, NC>() &&
                   set_smem(k_row_ifft<M, C::TPL, C::TPC, MAXR, NC>, C::S3);
        }))
        return BST_ERR_CUDA;
    const int N = p->N, V = p->V;
    const int pairs = (slices + 1) / 2;
    const int chunk = lanes > 1 ? bsth::fwd_chunk(p, pairs, max_chunk) : std::min(pairs, max_chunk);
    const int nchunks = (pairs + chunk - 1) / chunk;
    // chunks rotate over up to kMaxLanes streams (each with its own part of the
    // workspace) so that one chunk's gridding overlaps the next chunk's FFTs;
    // per-stage timing keeps everything on the caller's stream
    int nl = std::min(std::min(std::min(lanes, nchunks), bsth::kMaxLanes), std::max(p->max_lanes, 1));
    if (nl < 2 || p->timing || !bst_ensure_lanes(p)) nl = 1;
    const size_t lane_elems = (size_t)chunk * (V + (size_t)((N + 3) / 4) * 4) * M;
    const float scale = (float)((double)N / (2.0 * (double)M * (double)M));
    const float two_alpha = (float)(2 * p->alpha);
    const int row_tiles = (N + 3) / 4;
    const bool kbg = p->grid_kind == BST_GRID_KAISER_BESSEL;
    if (kbg) mode |= BSTK_KBW;
    // The paired and interleaved layouts serve the bilinear gridding only; their
    // kernels read the workspace 16 bytes at a time, so a workspace that is not
    // so aligned takes the packed layout.  Groups of inter_pairs<M>() slice
    // pairs are interleaved; what remains of a chunk is paired.  A call with pairs
    // left over is paired altogether below pairs M (V + N) = 2^23: three more launches
    // cost it more than the groups save (12 pairs of 64 x 64 22.2 against 13.4 us, 6 of
    // 512 x 512 59.5 against 50.8; 9 of 512 x 512, just above, 68.8 against 80.5).
    const bool wide = !kbg && ((uintptr_t)ws & 15) == 0;
    const bool paired = wide && p->fwd_layout != BST_LAYOUT_PACKED;
    const bool inter = wide && p->fwd_layout == BST_LAYOUT_INTERLEAVED && InterCfg<M>::OK &&
                       (pairs % bsth::inter_pairs_of(M) == 0 || (long long)pairs * M * (V + N) >= 1 << 23);
    const int base_mode = mode;
    if (paired) mode |= BSTK_PAIRED;
    const int pf = p->pair_fast ? 1 : 0;
    const float* dk = kbg ? p->kb_dk : nullptr;
    if (nl > 1) {
        if (cudaEventRecord(p->ev_fork, st) != cudaSuccess) return BST_ERR_CUDA;
        for (int l = 0; l < nl; ++l)
            if (cudaStreamWaitEvent(p->lane[l], p->ev_fork, 0) != cudaSuccess) return BST_ERR_CUDA;
    }
    // The kernels of a call of one chunk are chained (their set-up overlaps the
    // previous kernel's end): one 256 x 256 slice takes 12.9 us on the device
    // against 19.4 us.  With two lanes the other lane's blocks fill that end, and
    // blocks that only wait would keep them out; with many small chunks on one
    // stream the dearer launches (about 1 us each) bound the call.
    const bool chain = chainable(M) && nchunks == 1 && !p->timing;
    // the three stages of np pairs from pair p0 on stream s, groups interleaved
    auto run_inter = [&](int p0, int np, float2* Z, float2* T, cudaStream_t s) {
        if constexpr (InterCfg<M>::OK) {
            using I = InterCfg<M>;
            constexpr int RJ = inter_ray_rows<M>(), RT = inter_row_tiles<M>() * (4 / I::LP);
            const dim3 gr((V + RJ - 1) / RJ, np / I::LP), gc(np / I::P, M / 2);
            bst_timing_mark(p, s, -1);
            if (prep)
                launch(chain, k_ray_inter<M, MAXR, NC, true>, gr, inter_ray_threads<M>(), I::S1, s, sino, slices, p0, N, V,
                       *prep, base_mode, g, two_alpha, Z, p->tw);
            else
                launch(chain, k_ray_inter<M, MAXR, NC, false>, gr, inter_ray_threads<M>(), I::S1, s, sino, slices, p0, N,
                       V, PrepArgs{}, base_mode, g, two_alpha, Z, p->tw);
            bst_timing_mark(p, s, 0);
            launch(chain, k_grid_inter<M, MAXR, NC>, pf ? gc : dim3(gc.y, gc.x), 2 * I::P * I::TPL, I::S2, s, Z, V, N,
                   p->geo_J, p->geo_f, T, p->tw, pf);
            bst_timing_mark(p, s, 1);
            launch(chain, k_row_inter<M, MAXR, NC>, dim3((N + RT - 1) / RT, np / I::LP),
                   4 * I::TPL * inter_row_tiles<M>(), I::S3, s, T, slices, p0, N, scale, vol, p->tw);
            bst_timing_mark(p, s, 2);
        }
    };
    // ... packed or paired
    auto run_pairs = [&](int p0, int np, float2* Z, float2* T, cudaStream_t s) {
        bst_timing_mark(p, s, -1);
        if (prep)
            launch(chain, k_ray_fft_prep<M, C::TPL, C::LPC1, MAXR, NC, C::ILV1>, dim3((V + C::LPC1 - 1) / C::LPC1, np),
                   C::TPL * C::LPC1, C::S1, s, sino, slices, p0, N, V, *prep, mode, Z, p->tw);
        else
            launch(chain, k_ray_fft<M, C::TPL, C::LPC1, MAXR, NC, C::ILV1>, dim3((V + C::LPC1 - 1) / C::LPC1, np),
                   C::TPL * C::LPC1, C::S1, s, sino, slices, p0, N, V, mode, g, two_alpha, Z, p->tw);
        bst_timing_mark(p, s, 0);
        if (kbg) {
            const bst_status_t ks = bst_launch_kb_col(p, Z, T, np, s);
            if (ks != BST_OK) return ks;
        } else if (paired && C::XCHG_OK && p->grid_xchg) {
            if constexpr (C::XCHG_OK) {
                launch(chain, k_grid_col_xchg<M, C::TPL, MAXR, NC>, pf ? dim3(np, M / 2) : dim3(M / 2, np), 2 * C::TPL,
                       C::S2X, s, Z, V, N, p->geo_J, p->geo_f, T, p->tw, pf);
            }
        } else if (paired) {
            const int ncg = (M / 2 + C::CPCP - 1) / C::CPCP;
            launch(chain, k_grid_col_paired<M, C::TPL, C::CPCP, MAXR, NC>, pf ? dim3(np, ncg) : dim3(ncg, np),
                   2 * C::TPL * C::CPCP, C::S2P, s, Z, V, N, p->geo_J, p->geo_f, T, p->tw, pf);
        } else {
            const int ncg = (M / 2 + C::CPC - 1) / C::CPC;
            launch(chain, k_grid_col<M, C::TPL, C::CPC, MAXR, NC>, pf ? dim3(np, ncg) : dim3(ncg, np), C::TPL * C::CPC,
                   C::S2, s, Z, V, N, p->geo_J, p->geo_f, T, p->tw, pf);
        }
        bst_timing_mark(p, s, 1);
        launch(chain, k_row_ifft<M, C::TPL, C::TPC, MAXR, NC>, dim3((row_tiles + C::TPC - 1) / C::TPC, np),
               4 * C::TPL * C::TPC, C::S3, s, T, slices, p0, N, scale, vol, p->tw, dk);
        bst_timing_mark(p, s, 2);
        return BST_OK;
    };
    for (int c = 0; c < nchunks; ++c) {
        const int p0 = c * chunk;
        const int np = std::min(chunk, pairs - p0);
        const int l = c % nl;
        cudaStream_t s = nl > 1 ? p->lane[l] : st;
        float2* Z = (float2*)ws + (size_t)l * lane_elems;
        float2* T = Z + (size_t)chunk * V * M;
        const int ni = inter ? np / InterCfg<M>::P * InterCfg<M>::P : 0;
        if (ni > 0) run_inter(p0, ni, Z, T, s);
        if (ni < np) {
            const bst_status_t rs = run_pairs(p0 + ni, np - ni, Z + (size_t)ni * V * M,
                                              T + (size_t)ni * ((N + 3) / 4) * 4 * M, s);
            if (rs != BST_OK) return rs;
        }
    }
    if (nl > 1) {
        for (int l = 0; l < nl; ++l) {
            if (cudaEventRecord(p->ev_join[l], p->lane[l]) != cudaSuccess) return BST_ERR_CUDA;
            if (cudaStreamWaitEvent(st, p->ev_join[l], 0) != cudaSuccess) return BST_ERR_CUDA;
        }
    }
    return cudaGetLastError() == cudaSuccess ? BST_OK : BST_ERR_CUDA;
}

}  // namespace bst

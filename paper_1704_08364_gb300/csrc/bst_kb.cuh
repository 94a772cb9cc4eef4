// bst_kb.cuh -- stage P5 as Kaiser-Bessel convolution gridding, fused with the
// column half of P6 (device part).
//
// Every polar sample Y_j[k] (k != 0, -M/2) carries the area of its polar cell:
// the ray stage has multiplied it by |k| W[|k|] (W[0] / 4 for the DC cell, the
// cell average of |k|) and the angular weight dtheta_j is applied here.  It sits
// at (c_s, r_s) = k (cos theta_j, sin theta_j) bins and is spread onto the W x W
// Cartesian points c' - c_s, r' - r_s in (-W/2, W/2] with the separable kernel
// phi(x) = (I0(beta sqrt(1 - (2x/W)^2)) - 1) / (I0(beta) - 1) (the KB kernel
// without its pedestal, zero at the support edge), on the M-periodic grid;
// phi is evaluated as a per-plan polynomial (KbArgs::poly).
// The division by phi's transform (deapodization) happens in the row stage.
//
// One block owns a strip of two consecutive Cartesian columns (storage order) of
// up to four slice pairs, kept in shared memory as padded FFT lines: the kernel
// weights of a sample are evaluated once for all of the pairs.  The plan lists,
// per strip, every sample whose footprint touches it, sorted by the first row of
// the footprint (the first rows' samples once more at the end, for the periodic
// wrap), and cuts the strip into bands of four rows: a band's samples are then
// one contiguous range of that list, cut into items of at most KB_ITEM entries.
// Four lanes take an item together, every fourth entry each, accumulate the
// band's 2 x 4 cell of every pair in registers (the weight of every sample at
// every cell point, zero outside the footprint), add the four partial cells by
// shuffles and store the sum (or add it atomically, if the band has several
// items: those near the origin, where the samples crowd).  A warp takes eight items
// at once, longest first, from a shared counter.  Then the inverse FFT along r' of each column runs in place
// and the N central rows go to T exactly as with the bilinear gather.  The V
// samples of the DC bin all sit at the origin; one warp sums them (with their
// angular weights) and spreads the sum once.
//
// Positions are exact to float rounding of a number below one: k cos(theta)
// is split into the nearest integer and a remainder with the double-float
// direction table and FMA, so the kernel weights do not lose the ~1e-4 bin
// that a plain float product loses at radius 2048.  Weights come from the
// exact distance to each cell point, so which samples the plan lists (in
// double precision) only has to be a superset of the float footprints up to
// the kernel's zero edge.
#pragma once
#include <cuda_runtime.h>

#include "bst_stages.cuh"

namespace bst {

constexpr int KB_POLY = 12;    // degree of the kernel polynomial (see KbArgs::poly)
constexpr int KB_WMAX = 8;
constexpr int KB_CS = 2;       // columns per strip
constexpr int KB_RB = 4;       // rows per band
constexpr int KB_ITEM = 128;   // entries per item at most
constexpr int KB_WARP = 8;     // items that a warp takes at once

struct KbArgs {
    // phi as a polynomial of degree kb_degree(W) <= KB_POLY in
    // t = 2 (2x/W)^2 - 1 (Chebyshev interpolation of phi at degree + 1 nodes,
    // built per plan in double precision; monomial coefficients, Horner in
    // float: absolute error below 3e-7 for every supported width and pad
    // factor); coefficients above the degree are zero
    float poly[KB_POLY + 1];
    float t_scale;         // 8 / W^2, so that t = x^2 t_scale - 1
    const int* istart;     // [nstrips + 1] offsets of the strips' items
    const int4* items;     // (band, first entry, end entry, 1 if the band has others), longest first in a strip
    const int* list;       // sample ids j M + kidx (natural-order bin index)
    const float* wq;       // [V] angular weights dtheta_j
    const float4* dir;     // [V + 2] (cos_hi, cos_lo, sin_hi, sin_lo) of theta_{j}, at j + 1
    int W;                 // kernel width in bins (even, <= KB_WMAX)
    int nstrips;
};

// most slice pairs a block: their strips fill at most 140 KB of shared memory
template <int M> __host__ __device__ constexpr int kb_pairs() { return M >= 3072 ? 2 : 4; }
// threads a block with P slice pairs: 16 warps an SM at 128 registers (the cells
// of four pairs take 64), two blocks of 256 threads where their strips fit; at
// least a warp
template <int M, int P> __host__ __device__ constexpr int kb_threads() {
    const int most = M > 1536 ? 512 : 256, lines = KB_CS * P * tpl_of<M>();
    const int n = lines < most ? lines : most;
    return n < 32 ? 32 : n;
}
template <int M, int P> __host__ __device__ constexpr size_t kb_smem_bytes() {
    const int lines = kb_threads<M, P>() / tpl_of<M>();   // of the FFT, some of them spare at the smallest lengths
    return (size_t)(lines > KB_CS * P ? lines : KB_CS * P) * smem_line_len(M) * sizeof(float2);
}

// phi(x): the plan's polynomial of degree DEG in t = 2 (2x/W)^2 - 1 on the
// support, zero for |x| >= W/2 (t >= 1).  Arithmetic only (the coefficients
// are kernel arguments), so the weights cost FMA issue instead of
// shared-memory lookups.  DEG = 10 serves W <= 6 (interpolation error below
// 1e-7), DEG = 12 all widths (the plan fits the degree it will use).
template <int DEG = KB_POLY>
__device__ __forceinline__ float kb_phi(const KbArgs& kb, float x) {
    const float t = fmaf(x * x, kb.t_scale, -1.f);
    float h = kb.poly[DEG];
#pragma unroll
    for (int i = DEG - 1; i >= 0; --i) h = fmaf(h, t, kb.poly[i]);
    return t < 1.f ? h : 0.f;
}

// phi at x, x + 1, ..., x + n - 1 (n even): two of them to a packed multiply-add
template <int DEG, int n>
__device__ __forceinline__ void kb_phis(const KbArgs& kb, float x, float (&w)[n]) {
#pragma unroll
    for (int i = 0; i < n; i += 2) {
        const float2 d = make_float2(x + (float)i, x + (float)(i + 1));
        const float2 t = __ffma2_rn(__fmul2_rn(d, d), make_float2(kb.t_scale, kb.t_scale), make_float2(-1.f, -1.f));
        float2 h = make_float2(kb.poly[DEG], kb.poly[DEG]);
#pragma unroll
        for (int k = DEG - 1; k >= 0; --k) h = __ffma2_rn(h, t, make_float2(kb.poly[k], kb.poly[k]));
        w[i] = t.x < 1.f ? h.x : 0.f;
        w[i + 1] = t.y < 1.f ? h.y : 0.f;
    }
}

// degree of the kernel polynomial for width W
__host__ __device__ constexpr int kb_degree(int W) { return W <= 6 ? 10 : KB_POLY; }

// k * (hi + lo) = n + d with n an integer (as float) and |d| <= ~0.5
__device__ __forceinline__ void kb_split(float k, float hi, float lo, float& n, float& d) {
    const float p = __fmul_rn(k, hi);
    const float e = fmaf(k, lo, fmaf(k, hi, -p));
    n = rintf(p);
    d = __fadd_rn(__fsub_rn(p, n), e);
}

// signed distance (in bins, periodic in M) from the sample at n + d to grid index g
template <int M>
__device__ __forceinline__ float kb_dist(int g, float n, float d) {
    int q = g - (int)n;
    q = q >= (M >> 1) ? q - M : (q < -(M >> 1) ? q + M : q);
    return (float)q - d;
}

// One entry of an item: the sample's direction, its value in P slice pairs and
// its angular weight (zero past the end of the item).
template <int P> struct KbEntry {
    float4 d;
    float2 z[P];
    float w;
};

// Four lanes (`ql` of a quad) accumulate the samples of entries [lo, hi) into the
// 2 x 4 cell (rows r0..r0+3, columns c0, c0 + 1) of P slice pairs (pair p's
// spectrum at Zp + min(p, np - 1) zs) and store or add it to the strip's lines
// (line 2 p + c).  The warp's eight quads run `iters` steps together; a lane's
// loads for its next entry (and the sample id two entries on) are issued before
// the current entry's arithmetic.
template <int M, int DEG, int P>
__device__ __forceinline__ void kb_band(float2* smem, const KbArgs& kb, const float2* __restrict__ Zp, size_t zs,
                                        int np, int c0, int r0, int lo, int hi, int iters, int ql, bool live,
                                        bool shared_band) {
    constexpr int LL = smem_line_len(M);
    float2 acc[P][KB_CS][KB_RB];
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
        for (int c = 0; c < KB_CS; ++c)
#pragma unroll
            for (int r = 0; r < KB_RB; ++r) acc[p][c][r] = make_float2(0.f, 0.f);
    const float2 zero = make_float2(0.f, 0.f);
    auto fetch = [&](int s, bool ok) {
        KbEntry<P> e;
        const int j = s / M;
        e.d = ok ? __ldg(kb.dir + j + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
        e.w = ok ? __ldg(kb.wq + j) : 0.f;
#pragma unroll
        for (int p = 0; p < P; ++p) e.z[p] = ok ? __ldg(Zp + min(p, np - 1) * zs + s) : zero;
        return e;
    };
    int e = lo + ql;
    int sn = e < hi ? __ldg(kb.list + e) : 0;           // sample id of the next entry
    int sn2 = e + 4 < hi ? __ldg(kb.list + e + 4) : 0;  // ... of the one after it
    KbEntry<P> n = fetch(sn, e < hi);
#pragma unroll 2
    for (int it = 0; it < iters; ++it) {
        const int s = sn;
        const KbEntry<P> v = n;
        e += 4;
        sn = sn2;
        sn2 = e + 4 < hi ? __ldg(kb.list + e + 4) : 0;
        n = fetch(sn, e < hi);
        const int kidx = s % M;
        const float k = (float)(kidx < (M >> 1) ? kidx : kidx - M);
        float nc, dc, nr, dr;
        kb_split(k, v.d.x, v.d.y, nc, dc);
        kb_split(k, v.d.z, v.d.w, nr, dr);
        // distances to the band's rows and the strip's columns: the first one
        // with the periodic wrap, the others one bin further each (a wrap
        // inside a run of four points only moves points that are at least
        // M/2 - 4 >= W/2 bins away, where phi is zero either way)
        float wr[KB_RB], wc[KB_CS];
        kb_phis<DEG>(kb, kb_dist<M>(r0, nr, dr), wr);
        kb_phis<DEG>(kb, kb_dist<M>(c0, nc, dc), wc);
#pragma unroll
        for (int c = 0; c < KB_CS; ++c) {
            const float w = v.w * wc[c];
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const float2 z = make_float2(w * v.z[p].x, w * v.z[p].y);
#pragma unroll
                for (int r = 0; r < KB_RB; ++r) acc[p][c][r] = __ffma2_rn(make_float2(wr[r], wr[r]), z, acc[p][c][r]);
            }
        }
    }
    // sum over the quad: lane (c, rh) ends with column c, rows 2 rh and 2 rh + 1
    const bool c1 = ql & 2, r1 = ql & 1;
    auto add = [](float2 keep, float2 send, int mask) {
        return make_float2(keep.x + __shfl_xor_sync(0xffffffffu, send.x, mask),
                           keep.y + __shfl_xor_sync(0xffffffffu, send.y, mask));
    };
#pragma unroll
    for (int p = 0; p < P; ++p) {
        float2 h[KB_RB];
#pragma unroll
        for (int r = 0; r < KB_RB; ++r) h[r] = add(c1 ? acc[p][1][r] : acc[p][0][r], c1 ? acc[p][0][r] : acc[p][1][r], 2);
        const float2 a = add(r1 ? h[2] : h[0], r1 ? h[0] : h[2], 1), b = add(r1 ? h[3] : h[1], r1 ? h[1] : h[3], 1);
        // the four rows lie in one group of 16
        float2* line = smem + (p * KB_CS + (c1 ? 1 : 0)) * LL + r0 + (r0 >> 4) + (r1 ? 2 : 0);
        if (live && !shared_band) {
            line[0] = a;
            line[1] = b;
        } else if (live) {
            atomicAdd(&line[0].x, a.x);
            atomicAdd(&line[0].y, a.y);
            atomicAdd(&line[1].x, b.x);
            atomicAdd(&line[1].y, b.y);
        }
    }
}

// the DC sample at the origin (value z) into the strip's columns
template <int M>
__device__ __forceinline__ void kb_spread_dc(float2* smem, const KbArgs& kb, int c0, float2 z) {
    constexpr int LL = smem_line_len(M);
    const int hw = kb.W >> 1;
    for (int c = 0; c < KB_CS; ++c) {
        const float x = kb_dist<M>(c0 + c, 0.f, 0.f);
        if (fabsf(x) >= (float)hw) continue;
        const float wc = kb_phi(kb, x);
        float2* line = smem + c * LL;
        for (int r = -hw + 1; r < hw; ++r) {
            const int rr = r < 0 ? r + M : r;
            const float w = wc * kb_phi(kb, (float)r);
            float2& v = line[rr + (rr >> 4)];
            v = make_float2(fmaf(w, z.x, v.x), fmaf(w, z.y, v.y));
        }
    }
}

// P5 (KB gridding) + column P6 for the strip of two columns starting at
// c0 = 2 strip of np (1 .. P) slice pairs, spectra zs and tiles ts apart
template <int M, int TPL, int MAXR, int P>
__device__ __forceinline__ void kb_col_unit(float2* smem, int strip, int np, int V, int N,
                                            const float2* __restrict__ Zp, size_t zs, const KbArgs& kb,
                                            float2* __restrict__ Tp, size_t ts, const float2* __restrict__ tw) {
    constexpr int NT = kb_threads<M, P>(), LL = smem_line_len(M);
    __shared__ int next;
    const int tid = threadIdx.x, lane = tid & 31;
    const int c0 = strip * KB_CS;
    const int i0 = __ldg(kb.istart + strip), i1 = __ldg(kb.istart + strip + 1);
    for (int i = tid; i < P * KB_CS * LL; i += NT) smem[i] = make_float2(0.f, 0.f);
    if (tid == 0) next = i0 + NT / 32 * KB_WARP;
    __syncthreads();

    // the items are ordered longest first; a warp takes the next eight when it
    // finishes (greedy longest-first), which evens out the warps' work before
    // the barrier of the column transform, and its quads have items of about the
    // same length
    for (int i = i0 + tid / 32 * KB_WARP; i < i1;) {
        const int at = i + lane / 4;
        const bool live = at < i1;
        const int4 it = live ? __ldg(kb.items + at) : make_int4(0, 0, 0, 0);
        const int iters = __shfl_sync(0xffffffffu, (it.z - it.y + 3) / 4, 0);   // the warp's longest item
        if (kb.W <= 6)
            kb_band<M, kb_degree(6), P>(smem, kb, Zp, zs, np, c0, KB_RB * it.x, it.y, it.z, iters, lane & 3, live,
                                        it.w != 0);
        else
            kb_band<M, kb_degree(8), P>(smem, kb, Zp, zs, np, c0, KB_RB * it.x, it.y, it.z, iters, lane & 3, live,
                                        it.w != 0);
        if (lane == 0) i = atomicAdd(&next, KB_WARP);
        i = __shfl_sync(0xffffffffu, i, 0);
    }
    __syncthreads();

    // the DC bin of every angle sits at the origin: one weighted sum per pair, spread once
    if (c0 < (kb.W >> 1) || c0 + KB_CS > M - (kb.W >> 1)) {
        if (tid < 32) {
            for (int p = 0; p < np; ++p) {
                const float2* z0 = Zp + p * zs;
                float sx = 0.f, sy = 0.f;
                for (int j = tid; j < V; j += 32) {
                    const float w = __ldg(kb.wq + j);
                    const float2 zz = __ldg(z0 + (size_t)j * M);
                    sx = fmaf(w, zz.x, sx);
                    sy = fmaf(w, zz.y, sy);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    sx += __shfl_xor_sync(0xffffffffu, sx, o);
                    sy += __shfl_xor_sync(0xffffffffu, sy, o);
                }
                if (tid == 0) kb_spread_dc<M>(smem + p * KB_CS * LL, kb, c0, make_float2(sx, sy));
            }
        }
        __syncthreads();
    }

    // inverse FFT along r' of each column in place, NT / TPL lines at a time; the
    // N central rows go to T
    constexpr int LPR = NT / TPL;
    static_assert(NT % TPL == 0, "whole lines");
    const int t = tid % TPL;
#pragma unroll 1
    for (int l0 = 0; l0 < P * KB_CS; l0 += LPR) {
        const int line = l0 + tid / TPL;
        const bool live = line < P * KB_CS;
        const int l = live ? line : 0, p = l / KB_CS, c = l % KB_CS;
        const SmemLine sm{smem + line * LL};   // a line past the last one is scratch
        const ColDst<> dst{Tp + p * ts, N, M, c0 + c, false, live && p < np};
        fft_line<M, TPL, true, MAXR>(t, sm, dst, sm, tw);
    }
}

}  // namespace bst

// bst_inter.cuh -- the forward path's three kernels with P slice pairs
// interleaved point by point (layout BST_LAYOUT_INTERLEAVED).
//
//   Z per group of P pairs: [V][M/2][2][P] complex64, slot k of a row holding
//     Z[+k] of the P pairs and then Z[-k] of the P pairs (bin 0 fills both; the
//     Nyquist bin, weight 0, is not stored): one bilinear tap of all P pairs and
//     of a point and its mirror is one contiguous piece of 16 P bytes (for P = 2
//     two halves of a 64-byte piece, inter_slot).
//   T per group: [N/G][M][G][P] complex64, G = 8 / P rows: a column writes
//     64-byte pieces, a row tile reads 32-byte sectors.  (32-byte pieces for P = 2
//     read faster and write slower: 64 x 2048 x 2048 4257 -> 4341 us.)
//
// Why: the gridding kernel is bound by the L1 data pipe (80 % of its
// wavefronts in the paired layout), most of it the tap gathers, which pay one
// wavefront for every 128-byte line that the 8 lanes of a quarter-warp touch.
// With one point a lane, 8 points fall on about 2.8 lines; with P pairs the
// quarter-warp covers 8 / P points of 16 P bytes each.  The column stores take
// 4 lines a warp instead of 8, and the geometry table is read once for P pairs.
// P = 256 / TPL (2 at M = 2048, 4 at 1024, 8 from 512 down) keeps a block at 512
// threads, 2 P column lines in 70 KB of shared memory and two blocks an SM; M >=
// 3072 takes P = 2 in one block of 1024 threads.
// Measured, us a pair, paired -> interleaved: M = 1024 (512 x 512) ray 2.53 -> 1.59,
// gridding 5.96 -> 4.26, row 1.94 -> 1.53; M = 4096 (2048 x 2048) ray 26.2 -> 23.4,
// gridding 89.4 -> 79.6, row 26.2 -> 26.5.  What bounds the gridding now is still the
// latency of its taps and their L1 wavefronts.
#pragma once
#include "bst_stages.cuh"

namespace bst {

template <int M> __host__ __device__ constexpr int inter_pairs() { return bsth::inter_pairs_of(M); }
// rows of a piece of T
template <int P> __host__ __device__ constexpr int inter_rows() { return 8 / P; }
// pairs whose lines share a warp in the ray and row kernels (32-byte pieces)
template <int P> __host__ __device__ constexpr int inter_lanes() { return P < 4 ? P : 4; }
// stride between lines whose lanes alternate over n lines: skewed by 32 / n banks
template <int M> __host__ __device__ constexpr int inter_stride(int n) { return smem_line_len(M, n) + 16 / n; }

// Place of slot k, sign s (0: +k, 1: -k) in a row, in complex values: [k][s][P],
// for P = 2 [k / 2][s][k % 2][P], so that the ray kernel writes whole sectors there
// too (consecutive bins of one sign).
template <int P> __host__ __device__ __forceinline__ int inter_slot(int k, int s) {
    return P == 2 ? (k >> 1) * 8 + s * 4 + (k & 1) * 2 : (k * 2 + s) * P;
}

// store of the weighted spectrum value of bin k into slot |k| of row j
template <int M, int P>
__device__ __forceinline__ void inter_store(float2* z, int j, int p, int k, float2 v) {
    constexpr int H = M / 2;
    float2* row = z + (size_t)j * M * P + p;
    if (k < H) {
        row[inter_slot<P>(k, 0)] = v;
        if (k == 0) row[inter_slot<P>(0, 1)] = v;
    } else if (k > H) {
        row[inter_slot<P>(M - k, 1)] = v;
    }
}
template <int M, int P> struct InterDst {
    float2* z;
    int j, p;
    const float* g;
    int mode;
    float two_alpha;
    bool live;
    static constexpr bool kSmem = false;
    __device__ __forceinline__ void store(int k, float2 v) const {
        if (live) inter_store<M, P>(z, j, p, k, cscale(v, bin_weight(k, M, mode, g, two_alpha)));
    }
};
template <int M, int P> struct InterDstPrep {
    float2* z;
    int j, p;
    const float2* cw;
    bool live;
    static constexpr bool kSmem = false;
    __device__ __forceinline__ void store(int k, float2 v) const {
        if (live) inter_store<M, P>(z, j, p, k, cmul(v, __ldg(cw + k)));
    }
};

// rows (angles) a block of the ray kernel
template <int M> __host__ __device__ constexpr int inter_ray_rows() {
    const int n = 256 / (tpl_of<M>() * inter_lanes<inter_pairs<M>()>());
    return n > 1 ? n : 1;
}
template <int M> __host__ __device__ constexpr int inter_ray_threads() {
    return inter_ray_rows<M>() * tpl_of<M>() * inter_lanes<inter_pairs<M>()>();
}

// P2 + P3 + P4 of LP pairs of a group (blockIdx.y: group and, for P = 8, half of
// it); lanes alternate over the pairs, so a warp stores whole 32-byte sectors
template <int M, int MAXR, int NC, bool PREP>
__global__ void __launch_bounds__(inter_ray_threads<M>(), 1024 / inter_ray_threads<M>())
    k_ray_inter(const float* __restrict__ sino, int slices, int pair0, int N, int V, PrepArgs pa, int mode,
                const float* __restrict__ g, float two_alpha, float2* __restrict__ Z, const float2* __restrict__ tw) {
    constexpr int TPL = tpl_of<M>(), P = inter_pairs<M>(), LP = inter_lanes<P>();
    extern __shared__ float2 smem[];
    chain_begin<M>();
    // the rays are read pair by pair, the spectrum is written with the pairs interleaved
    const int row = threadIdx.x / (LP * TPL);
    const LineMap m = ray_lines<M, TPL, LP, MAXR, true>(threadIdx.x % (LP * TPL));
    const int grp = blockIdx.y / (P / LP), pb = (blockIdx.y % (P / LP)) * LP;
    const int j = blockIdx.x * inter_ray_rows<M>() + row;
    const bool live = j < V;
    const int jj = live ? j : 0;
    const int sa = 2 * (pair0 + grp * P + pb + m.line0), sb = sa + 1;
    const bool hb = sb < slices;
    const float* ya = sino + ((size_t)sa * V + jj) * N;
    const float* yb = hb ? sino + ((size_t)sb * V + jj) * N : nullptr;
    float2* z = Z + (size_t)grp * V * M * P;
    const int p = pb + m.line1;
    const SmemLine sm0{smem + (row * LP + m.line0) * inter_stride<M>(LP)};
    const SmemLine sm1{smem + (row * LP + m.line1) * inter_stride<M>(LP)};
    if constexpr (PREP) {
        const PrepRays rays{ya,
                            yb,
                            pa.dark ? pa.dark + (size_t)sa * N : nullptr,
                            pa.dark && hb ? pa.dark + (size_t)sb * N : nullptr,
                            pa.flat ? pa.flat + (size_t)sa * N : nullptr,
                            pa.flat && hb ? pa.flat + (size_t)sb * N : nullptr,
                            pa.win};
        const InterDstPrep<M, P> dst{z, jj, p, pa.cw, live};
        float2 x[M / TPL];
        prep_gather<M, TPL, NC>(rays, m.t0, N, live, x);
        fft_line_regs<M, TPL, false, MAXR, InterDstPrep<M, P>, BlockSync, true>(m.t0, x, dst, sm0, m.t1, sm1, tw);
    } else {
        const RaySrc<NC> src{ya, yb, N, M, live};
        const InterDst<M, P> dst{z, jj, p, g, mode, two_alpha, live};
        fft_line_remap<M, TPL, false, MAXR, true, false>(m.t0, src, sm0, m.t1, dst, sm1, tw);
    }
}

template <int M, int P, int NC> struct InterColDst {
    float2* T;      // the group's T, at this pair
    int N, cidx;
    bool rev;
    static constexpr bool kSmem = false;
    // no output index p in [lo, hi) is kept (in either reading direction)
    static __host__ __device__ constexpr bool drop_group(int lo, int hi, int Mc) {
        return NC > 0 && lo >= NC / 2 + 1 && hi <= Mc - NC / 2;
    }
    __device__ __forceinline__ void store(int i, float2 v) const {
        constexpr int G = inter_rows<P>();
        const int n = NC > 0 ? NC : N;
        const int q = rev ? (i == 0 ? 0 : M - i) : i;
        const int r = signed_freq(q, M) + (n >> 1);
        if (r < 0 || r >= n) return;
        T[((size_t)(r / G) * M + cidx) * (G * P) + (r % G) * P] = v;
    }
};

// P0 + P5 + column P6 of the column pair (q, -q) for the P pairs of a group.
// The P lanes of a point hold its 16-byte pieces: lane e = h P/2 + u takes pairs
// 2u, 2u + 1 on the side of column q (h = 0) or -q (h = 1); the side, the half
// plane and the seam decide which sign's half of the slot it reads.  A lane owns
// the first FFT pass of pair 2u + w of its column, w = lane / 16: it gathers
// every second row for both pairs and swaps the other pair's value with lane
// ^ 16, so that it ends with its own sixteen (twelve) rows, as in grid_unit_xchg.
// PS points per gather step.
template <int M, int MAXR, int NC>
__global__ void __launch_bounds__(2 * inter_pairs<M>() * tpl_of<M>(), 1024 / (2 * inter_pairs<M>() * tpl_of<M>()))
    k_grid_inter(const float2* __restrict__ Z, int V, int N, const int* __restrict__ gJ,
                 const float2* __restrict__ gF, float2* __restrict__ T, const float2* __restrict__ tw,
                 int pair_fast) {
    constexpr int TPL = tpl_of<M>(), P = inter_pairs<M>(), H = M / 2, PS = 2;
    constexpr int RW = 16 / P;      // consecutive rows of a half-warp
    constexpr int PPL = M / TPL, PPT = PPL / 2;
    static_assert(TPL % RW == 0 && PPL % 4 == 0 && PPT % PS == 0, "steps of the upper and lower half rows");
    extern __shared__ float2 smem[];
    chain_begin<M>();
    const int grp = pair_fast ? blockIdx.x : blockIdx.y, q = pair_fast ? blockIdx.y : blockIdx.x;
    const int lane = threadIdx.x & 31, e = lane % P, w = lane >> 4;
    const int h = e / (P / 2), u = e % (P / 2);
    const int t = (threadIdx.x >> 5) * RW + (lane / P) % RW;
    const float4* Zg = reinterpret_cast<const float4*>(Z + (size_t)grp * V * M * P) + u;
    const int* gJq = gJ + (size_t)q * M + t + w * TPL;
    const float2* gFq = gF + (size_t)q * M + t + w * TPL;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    // xe[i] = input 2 i, xo[i] = input 2 i + 1 of the thread's first pass
    float2 xe[PPT], xo[PPT];
    int jn[PS];
    float2 fn[PS];
#pragma unroll
    for (int s = 0; s < PS; ++s) {
        jn[s] = __ldg(gJq + 2 * s * TPL);
        fn[s] = __ldg(gFq + 2 * s * TPL);
    }
#pragma unroll
    for (int i = 0; i < PPT; i += PS) {
        int jc[PS];
        float2 fc[PS];
#pragma unroll
        for (int s = 0; s < PS; ++s) {
            jc[s] = jn[s];
            fc[s] = fn[s];
        }
        if (i + PS < PPT) {
#pragma unroll
            for (int s = 0; s < PS; ++s) {
                jn[s] = __ldg(gJq + 2 * (i + PS + s) * TPL);
                fn[s] = __ldg(gFq + 2 * (i + PS + s) * TPL);
            }
        }
        float4 z[PS][4];
#pragma unroll
        for (int s = 0; s < PS; ++s) {
            const int Jt = jc[s] >> 16;
            const int k0 = jc[s] & 0xffff;
            // a table bracket >= -1 means the point is inside the band and not the origin
            const bool ok = Jt >= -1;
            // the row is below M/2 (kappa = +rho for the point) iff i + s < PPL / 4
            const bool up = (i + s) < PPL / 4;
            const int J = ok ? Jt : 0;
            const bool sA = J < 0, sB = J + 1 >= V;   // seam rows read row V - 1 or 0 at -k
            const int rowA = sA ? V - 1 : J;
            const int rowB = sB ? 0 : J + 1;
            const int hA = (up != sA ? 0 : 1) ^ h, hB = (up != sB ? 0 : 1) ^ h;
            const bool k1ok = ok && k0 + 1 < H;
            const float4* pa = Zg + rowA * H * P + inter_slot<P>(k0, hA) / 2;
            const float4* pb = Zg + rowB * H * P + inter_slot<P>(k0, hB) / 2;
            const int up1 = P == 2 ? ((k0 & 1) ? 3 : 1) : P;   // to the next bin
            z[s][0] = ok ? __ldg(pa) : zero4;
            z[s][1] = k1ok ? __ldg(pa + up1) : zero4;
            z[s][2] = ok ? __ldg(pb) : zero4;
            z[s][3] = k1ok ? __ldg(pb + up1) : zero4;
        }
#pragma unroll
        for (int s = 0; s < PS; ++s) {
            const float ft = fc[s].x, fk = fc[s].y;
            float2 v[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                auto half = [&](const float4& f) { return c ? make_float2(f.z, f.w) : make_float2(f.x, f.y); };
                const float2 a0 = half(z[s][0]), a1 = half(z[s][1]), b0 = half(z[s][2]), b1 = half(z[s][3]);
                const float2 kk = make_float2(fk, fk);
                const float2 A = __ffma2_rn(kk, csub(a1, a0), a0), B = __ffma2_rn(kk, csub(b1, b0), b0);
                v[c] = __ffma2_rn(make_float2(ft, ft), csub(B, A), A);
            }
            if (q == 0 && h) v[0] = v[1] = make_float2(0.f, 0.f);
            const float2 own = w ? v[1] : v[0], oth = w ? v[0] : v[1];
            const float2 rcv = make_float2(__shfl_xor_sync(0xffffffffu, oth.x, 16),
                                           __shfl_xor_sync(0xffffffffu, oth.y, 16));
            xe[i + s] = w ? rcv : own;
            xo[i + s] = w ? own : rcv;
        }
    }
    float2 x[PPL];
#pragma unroll
    for (int i = 0; i < PPT; ++i) {
        x[2 * i] = xe[i];
        x[2 * i + 1] = xo[i];
    }
    // the origin (row 0 of column 0, input 0 of thread t = 0, the gather gave 0
    // there) is single-valued: mean over angles of the DC bin, by the whole block
    // (thread: pair threadIdx.x % P, every 2 TPL-th angle)
    if (q == 0) {
        constexpr int NT = 2 * P * TPL, NW = NT / 32;
        const float2* z0 = Z + (size_t)grp * V * M * P + threadIdx.x % P;
        float2 s = make_float2(0.f, 0.f);
        for (int j = threadIdx.x / P; j < V; j += NT / P) s = cadd(s, __ldg(z0 + (size_t)j * M * P));
#pragma unroll
        for (int o = 16; o >= P; o >>= 1) {
            s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
            s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        }
        if (lane < P) smem[(threadIdx.x >> 5) * P + lane] = s;
        __syncthreads();
        if (h == 0 && t == 0) {
            s = make_float2(0.f, 0.f);
            for (int i = 0; i < NW; ++i) s = cadd(s, smem[i * P + 2 * u + w]);
            x[0] = make_float2(s.x / (float)V, s.y / (float)V);
        }
        __syncthreads();
    }
    const LineOf<P> sm{smem + (e + P * w) * inter_stride<M>(P)};
    const InterColDst<M, P, NC> dst{T + (size_t)grp * N * M * P + 2 * u + w, N,
                                    h == 0 ? q : (q == 0 ? H : M - q), h == 1 && q != 0};
    fft_line_regs<M, TPL, true, MAXR>(t, x, dst, sm, tw);
}

template <int M, int P> struct InterTileSrc {
    const float2* T;    // the group's T, at this row and pair
    static constexpr bool kSmem = false;
    __device__ __forceinline__ float2 load(int c) const { return __ldg(T + (size_t)c * (inter_rows<P>() * P)); }
};

// tiles of four lines a block of the row kernel
template <int M> __host__ __device__ constexpr int inter_row_tiles() {
    const int n = 128 / (4 * tpl_of<M>());
    return n > 1 ? n : 1;
}

// row P6 + P7 + P8: a tile is four lines, LP pairs of 4 / LP rows
// (blockIdx.y: group and, for P = 8, half of it)
template <int M, int MAXR, int NC>
__global__ void __launch_bounds__(4 * tpl_of<M>() * inter_row_tiles<M>(), 1024 / (4 * tpl_of<M>() * inter_row_tiles<M>()))
    k_row_inter(const float2* __restrict__ T, int slices, int pair0, int N, float scale, float* __restrict__ vol,
                const float2* __restrict__ tw) {
    constexpr int TPL = tpl_of<M>(), P = inter_pairs<M>(), LP = inter_lanes<P>(), G = inter_rows<P>();
    extern __shared__ float2 smem[];
    chain_begin<M>();
    const int tile = threadIdx.x / (4 * TPL);
    const LineMap m = tile_lines<M, TPL, 4, MAXR>(threadIdx.x % (4 * TPL));
    const int grp = blockIdx.y / (P / LP), pb = (blockIdx.y % (P / LP)) * LP;
    const int rb = (blockIdx.x * inter_row_tiles<M>() + tile) * (4 / LP);
    // line l: pair pb + l % LP of row rb + l / LP
    const int ra = rb + m.line0 / LP, pa = pb + m.line0 % LP;
    const int r = rb + m.line1 / LP, sa = 2 * (pair0 + grp * P + pb + m.line1 % LP), sb = sa + 1;
    const int rr = ra < N ? ra : 0;
    const InterTileSrc<M, P> src{T + (size_t)grp * N * M * P + (size_t)(rr / G) * M * G * P + (rr % G) * P + pa};
    const size_t at = (size_t)(r < N ? r : 0) * N;
    const VolDst<NC> dst{vol + (size_t)sa * N * N + at, sb < slices ? vol + (size_t)sb * N * N + at : nullptr,
                         N, M, scale, r < N, nullptr};
    float2* base = smem + tile * 4 * row_line_stride<M>();
    fft_line_remap<M, TPL, true, MAXR, false, true>(m.t0, src, LineOf<4>{base + m.line0 * row_line_stride<M>()}, m.t1, dst,
                                                   SmemLine{base + m.line1 * row_line_stride<M>()}, tw);
}

}  // namespace bst

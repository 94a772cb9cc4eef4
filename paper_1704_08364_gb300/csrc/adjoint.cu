// adjoint.cu -- the exact transpose of the discrete BST operator
// (radon_adjoint) and the gradient with respect to the filter taps
// (bst_fbp_filter_grad).
//
// Read backwards, the BST chain is a Fourier-slice projector (the FST dual of
// the BST, Sec. 2).  For a slice pair packed as f_a + i f_b:
//
//   k_adj_row_fft   transpose of the crop and the row inverse FFT: zero-extend
//                   each image row to M and FFT it (opposite exponent).
//   k_adj_col_fft   transpose of the column inverse FFT: zero-extend each
//                   column to M and FFT it, giving the full Cartesian spectrum,
//                   up to four slice pairs interleaved point by point.
//   k_adj_polar     transpose of the bilinear gridding in gather form: every
//                   polar sample (j, k) sums the weighted Cartesian values of
//                   the gridding cells that tap it (cell lists built once per
//                   plan, with the forward path's own coordinate function, so
//                   the weights are bitwise those of the forward gridding);
//                   plus the transpose of the DC mean; then the weight W and
//                   the inverse FFT along t, cropped to the N detector samples,
//                   scaled by dt dw^2, Re -> slice a, Im -> slice b.
//
// The filter gradient multiplies the rays' spectrum Y (no weight), recomputed
// block by block (k_fg_ray), by the polar pull-back lambda of the image
// gradient, and reduces Re(conj(lambda) Y) over angles, slices and +-k in a
// fixed order.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <vector>

#include "bst_stages.cuh"

namespace bst {

template <int M> __host__ __device__ constexpr int adj_tpl() { return (M % 3 == 0) ? M / 12 : M / 16; }
template <int M> __host__ __device__ constexpr int adj_row_stride() { return smem_line_len(M) + 4; }
// most slice pairs whose spectra are interleaved: four lines of 256 threads at
// M = 4096 would leave one block an SM
template <int M> __host__ __device__ constexpr int adj_pairs() { return M >= 3072 ? 2 : 4; }
// lines (columns times P pairs) of a block of the column kernel: 256 threads or
// more
template <int M, int P> __host__ __device__ constexpr int adj_col_lines() {
    const int n = 256 / (adj_tpl<M>() * P);
    return n > 1 ? n * P : P;
}
// lines (angle rows times P pairs) of a block of the polar kernel: its threads
// walk the rows one after the other, so four rows at most, two with few pairs (more
// only to fill a warp)
template <int M, int P> __host__ __device__ constexpr int adj_polar_lines() {
    const int warp = 32 / (adj_tpl<M>() * P), n = 256 / (adj_tpl<M>() * P), most = P < 4 ? 2 : 4;
    const int rows = n > most ? most : n;
    const int l = warp > rows ? warp : rows;
    return l > 1 ? l * P : P;
}
// threads of a block of the polar kernel: those of the lines' transforms, and up to
// M = 1024 with few pairs as many again as a row has bins, 512 at most: one pair
// alone fills the chip only so, and its walk is a chain of M (1 + 1 / rows) / threads
// steps (one slice of 64 x 64 30.7 -> 19.8 us; 33 x 400 x 512, whose last pair is alone,
// 204 -> 188).  From M = 1536 a pair has blocks enough (one slice of 900 x 1024 69.7 ->
// 74.0 us with them).
template <int M, int P> __host__ __device__ constexpr int adj_polar_threads() {
    const int fft = adj_tpl<M>() * adj_polar_lines<M, P>(), most = M < 512 ? M : 512;
    return M <= 1024 && P < 4 && most > fft ? most / fft * fft : fft;
}

// ---------------------------------------------------------------------------
// k_adj_row_fft

struct ImgRowSrc {
    const float* fa;
    const float* fb;
    int N, M;
    bool live;
    static constexpr bool kSmem = false;
    __device__ __forceinline__ float2 load(int p) const {
        const int c = signed_freq(p, M) + (N >> 1);
        if (!live || c < 0 || c >= N) return make_float2(0.f, 0.f);
        return make_float2(__ldg(fa + c), fb ? __ldg(fb + c) : 0.f);
    }
};

struct TileDst {
    float2* T;
    int M, rb, line;
    bool live;
    static constexpr bool kSmem = false;
    __device__ __forceinline__ void store(int k, float2 v) const {
        if (live) T[((size_t)rb * M + k) * 4 + line] = v;
    }
};

template <int M, int TPL, int TPC>
__global__ void __launch_bounds__(4 * TPL * TPC)
    k_adj_row_fft(const float* __restrict__ vol, int slices, int pair0, int N, float2* __restrict__ T,
                  const float2* __restrict__ tw) {
    extern __shared__ float2 smem[];
    const int pl = blockIdx.y;
    const int tile = threadIdx.x / (4 * TPL);
    // the image rows are read one by one, T is written with the four rows interleaved
    const LineMap m = ray_lines<M, TPL, 4, 16, true>(threadIdx.x % (4 * TPL));
    const int rb = blockIdx.x * TPC + tile;
    const int r = rb * 4 + m.line0;
    const bool live = r < N;
    const int rr = live ? r : 0;
    const int sa = 2 * (pair0 + pl), sb = sa + 1;
    const ImgRowSrc src{vol + ((size_t)sa * N + rr) * N, sb < slices ? vol + ((size_t)sb * N + rr) * N : nullptr, N, M,
                        live};
    const TileDst dst{T + (size_t)pl * ((N + 3) / 4) * 4 * M, M, rb, m.line1, rb * 4 < N};
    float2* base = smem + tile * 4 * adj_row_stride<M>();
    fft_line_remap<M, TPL, false, 16, false, false>(m.t0, src, SmemLine{base + m.line0 * adj_row_stride<M>()}, m.t1, dst,
                                  SmemLine{base + m.line1 * adj_row_stride<M>()}, tw);
}

// ---------------------------------------------------------------------------
// k_adj_col_fft

struct TileColSrc {
    const float2* T;
    int N, M, cidx;
    bool live;
    static constexpr bool kSmem = false;
    __device__ __forceinline__ float2 load(int p) const {
        const int r = signed_freq(p, M) + (N >> 1);
        if (!live || r < 0 || r >= N) return make_float2(0.f, 0.f);
        return __ldg(T + ((size_t)(r >> 2) * M + cidx) * 4 + (r & 3));
    }
};

// Points at radius M/2 and beyond are in no cell (polar_radius), so they are not
// stored: a fifth of X (33 x 400 x 512 adjoint 206.5 -> 205 us, 4 x 1024 x 1024
// 116 -> 113).
struct ColOut {
    float2* X;     // the column, of this pair among P
    int P, M;
    int most;      // stored while r'^2 <= most (negative: not at all)
    static constexpr bool kSmem = false;
    __device__ __forceinline__ void store(int k, float2 v) const {
        const int r = signed_freq(k, M);
        if (r * r <= most) X[(size_t)k * P] = v;
    }
};

// The spectra of P slice pairs interleaved, X[group][c][r][P], so that the
// polar kernel reads a Cartesian point of all P pairs as one 8 P byte piece.
// Lane order: pair, then position, so that the stores of a warp are contiguous;
// the pairs' lines are skewed by 32 / P banks.  Pairs beyond npairs are zero.
template <int M, int P> __host__ __device__ constexpr int adj_col_stride() {
    return smem_line_len(M, P) + (P > 1 ? 16 / P : 0);
}
template <int M, int TPL, int LINES, int P>
__global__ void __launch_bounds__(TPL * LINES)
    k_adj_col_fft(const float2* __restrict__ T, int N, int npairs, float2* __restrict__ X,
                  const float2* __restrict__ tw) {
    extern __shared__ float2 smem[];
    const int p = threadIdx.x % P, t = (threadIdx.x / P) % TPL, cl = threadIdx.x / (P * TPL);
    const int pl = blockIdx.y * P + p;
    const int c = blockIdx.x * (LINES / P) + cl;
    TileColSrc src{T + (size_t)pl * ((N + 3) / 4) * 4 * M, N, M, c, pl < npairs && c < M};
    const int cx = signed_freq(c, M);
    ColOut dst{X + ((size_t)blockIdx.y * M + c) * M * P + p, P, M, c < M ? M / 2 * (M / 2) - 1 - cx * cx : -1};
    LineOf<P> sm{smem + (cl * P + p) * adj_col_stride<M, P>()};
    fft_line<M, TPL, false>(t, src, dst, sm, tw);
}

// ---------------------------------------------------------------------------
// k_adj_polar

struct Cells {
    const int* __restrict__ start;   // [(V+1) M + 1]
    const int* __restrict__ pts;     // index c * M + r into the spectrum
    const float2* __restrict__ w;    // (fth, fk) of each point
};

// the values of P pairs at one Cartesian point
template <int P>
__device__ __forceinline__ void load_point(const float2* __restrict__ X, int pt, float2 (&x)[P]) {
    if constexpr (P == 1) {
        x[0] = __ldg(X + pt);
    } else {
        // (one 32-byte load for P = 4 measured slower: 358 against 280 us)
        const float4* q = reinterpret_cast<const float4*>(X + (size_t)pt * P);
#pragma unroll
        for (int i = 0; i < P / 2; ++i) {
            const float4 v = __ldg(q + i);
            x[2 * i] = make_float2(v.x, v.y);
            x[2 * i + 1] = make_float2(v.z, v.w);
        }
    }
}

template <int P>
__device__ __forceinline__ void axpy(float2 (&acc)[P], float w, const float2 (&x)[P]) {
#pragma unroll
    for (int p = 0; p < P; ++p) {
        acc[p].x = fmaf(w, x[p].x, acc[p].x);
        acc[p].y = fmaf(w, x[p].y, acc[p].y);
    }
}

// acc += the weighted Cartesian values of the cell (J, K0) for its tap `tap`
// (0: (J, K0), 1: (J, K0+1), 2: (J+1, K0), 3: (J+1, K0+1)).
template <int P>
__device__ __forceinline__ void add_cell(const Cells& cl, const float2* __restrict__ X, int M, int J, int K0, int tap,
                                         float2 (&acc)[P]) {
    if (K0 < -(M >> 1) || K0 > (M >> 1) - 1) return;
    const int cell = (J + 1) * M + (K0 + (M >> 1));
    const int b = __ldg(cl.start + cell), e = __ldg(cl.start + cell + 1);
    for (int i = b; i < e; ++i) {
        const float2 fw = __ldg(cl.w + i);
        float2 x[P];
        load_point<P>(X, __ldg(cl.pts + i), x);
        axpy<P>(acc, (tap & 2 ? fw.x : 1.f - fw.x) * (tap & 1 ? fw.y : 1.f - fw.y), x);
    }
}

// First-pass source of the inverse FFT along t: lambda from the shared line
// (plus the transpose of the mean at k = 0), kept in lam if asked for, times the
// weight W of `mode`.
struct PolarSrc {
    const float2* p;
    float2* lam;        // this pair's and angle's row, or null
    const float* g;
    float2 dc;          // spectrum value at (0, 0) / V
    int M, mode;
    float two_alpha;
    static constexpr bool kSmem = true;
    __device__ __forceinline__ float2 load(int k) const {
        float2 v = p[k + (k >> 4)];
        if (k == 0) v = cadd(v, dc);
        if (lam) lam[k] = v;
        const int ak = k <= (M >> 1) ? k : M - k;
        float w;
        if (ak == (M >> 1)) w = 0.f;
        else if (mode == BSTK_FILTER) w = g ? __ldg(g + ak) : 1.f;
        else w = ak == 0 ? 0.f : __fdiv_rn(two_alpha, (float)ak);
        return cscale(v, w);
    }
};

struct SinoCrop {
    float* ya;
    float* yb;
    int N, M;
    float scale;
    bool live;
    static constexpr bool kSmem = false;
    __device__ __forceinline__ void store(int m, float2 v) const {
        if (!live) return;
        const int i = signed_freq(m, M) + (N >> 1);
        if (i < 0 || i >= N) return;
        ya[i] = v.x * scale;
        if (yb) yb[i] = v.y * scale;
    }
};

// mode: BSTK_FILTER / BSTK_BACKPROJECT: weight, inverse FFT, crop -> sino;
//       BSTK_RAW: no sinogram.
// lam (may be null in the first two modes): lambda (no weight) to lam[pair][V][M]
//
// A block takes L = LINES / P angle rows j0 .. of P slice pairs.  Thread kappa
// walks the cells (J, K0 = kappa - M/2) of the brackets J = j0 - 1 .. j0 + L - 1
// and reads each list entry and its P-pair point once for the four polar
// samples it feeds: rows J and J + 1, bins K0 (its own) and K0 + 1 (handed to
// the next lane by a shuffle, across warps through `edge`).  Reading every cell
// once per sample and pair instead (four times, 8 bytes of each 32-byte sector)
// waited on the list-to-point chains (16 stall cycles per issue): 486 us for
// the 8 pairs of 16 x 1024 x 1024, 280 us with this form and 221 us with the next
// cell's list bounds read ahead.  What bounds it now is the latency of the chain
// from a list entry to its point (two thirds of the stall cycles), with the L1
// wavefronts of the point reads at 65 to 68 % of the peak.
template <int M, int TPL, int LINES, int P, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT)
    k_adj_polar(const float2* __restrict__ X, Cells cl, int V, int N, int slices, int pair0, int npairs, int mode,
                const float* __restrict__ g, float two_alpha, float scale, float* __restrict__ sino,
                float2* __restrict__ lam, const float2* __restrict__ tw) {
    constexpr int L = LINES / P, H = M / 2;
    constexpr int EDGES = (M - 1) / 32;   // warp boundaries within a row
    static_assert(NT % 32 == 0 && TPL * LINES % 32 == 0 && LINES % P == 0, "whole warps, whole groups of pairs");
    extern __shared__ float2 smem[];
    __shared__ float2 edge[EDGES > 0 ? EDGES : 1][LINES];
    const int tid = threadIdx.x, lane = tid & 31;
    const int j0 = blockIdx.x * L;
    const float2* Xp = X + (size_t)blockIdx.y * P * M * M;
    const float2 zero = make_float2(0.f, 0.f);
    // the list bounds of the next cell are read while this one is worked on
    auto bounds = [&](int k, int b, int& lo, int& hi) {
        const int J = j0 - 1 + b;
        lo = hi = 0;
        if (k < M && J < V) {
            const int cell = (J + 1) * M + k;
            lo = __ldg(cl.start + cell);
            hi = __ldg(cl.start + cell + 1);
        }
    };
    int sn, en;
    bounds(tid, 0, sn, en);
#pragma unroll 1
    for (int k0 = 0; k0 < M; k0 += NT) {
        const int kappa = k0 + tid;
        const bool act = kappa < M;
        const int K = kappa - H;
        float2 own[P], hi[P];   // of the row being completed, rows J + 1 of the brackets so far
#pragma unroll
        for (int p = 0; p < P; ++p) own[p] = hi[p] = zero;
#pragma unroll 1
        for (int b = 0; b <= L; ++b) {
            const int J = j0 - 1 + b;
            float2 own1[P], hi1[P];
#pragma unroll
            for (int p = 0; p < P; ++p) own1[p] = hi1[p] = zero;
            {
                const int e = en;
                int i = sn;
                bounds(b == L ? kappa + NT : kappa, b == L ? 0 : b + 1, sn, en);
                for (; i < e; ++i) {
                    const float2 fw = __ldg(cl.w + i);
                    float2 x[P];
                    load_point<P>(Xp, __ldg(cl.pts + i), x);
                    const float lo = 1.f - fw.x, l0 = 1.f - fw.y;
                    axpy<P>(own, lo * l0, x);
                    axpy<P>(hi, lo * fw.y, x);
                    axpy<P>(own1, fw.x * l0, x);
                    axpy<P>(hi1, fw.x * fw.y, x);
                }
            }
            if (b > 0) {
                const int j = J, l = b - 1;
                if (act && j == 0) {  // seam: the J + 1 = V taps of bracket V - 1 read row 0 at -k
                    add_cell<P>(cl, Xp, M, V - 1, -K, 2, own);
                    add_cell<P>(cl, Xp, M, V - 1, -K - 1, 3, own);
                }
                if (act && j == V - 1) {  // the J = -1 taps of bracket -1 read row V - 1 at -k
                    add_cell<P>(cl, Xp, M, -1, -K, 0, own);
                    add_cell<P>(cl, Xp, M, -1, -K - 1, 1, own);
                }
                const int k = K < 0 ? K + M : K;
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    const int line = l * P + p;
                    float2 up = make_float2(__shfl_up_sync(0xffffffffu, hi[p].x, 1),
                                            __shfl_up_sync(0xffffffffu, hi[p].y, 1));
                    if (lane == 0) up = zero;
                    if (act) {
                        // bin -M/2 is zero
                        SmemLine{smem + line * smem_line_len(M)}.store(k, K == -H ? zero : cadd(own[p], up));
                        if (lane == 31 && kappa + 1 < M) edge[kappa / 32][line] = hi[p];
                    }
                }
            }
#pragma unroll
            for (int p = 0; p < P; ++p) {
                own[p] = own1[p];
                hi[p] = hi1[p];
            }
        }
    }
    __syncthreads();
    for (int i = tid; i < EDGES * LINES; i += NT) {
        const int line = i % LINES, w = i / LINES;
        const int K = 32 * (w + 1) - H;
        const int k = K < 0 ? K + M : K;
        float2* q = smem + line * smem_line_len(M) + k + (k >> 4);
        *q = cadd(*q, edge[w][line]);
    }
    __syncthreads();
    if (tid >= TPL * LINES) return;   // the transforms' threads go on, with a barrier of their own
    const WorkerSync sync{1, TPL * LINES};
    const int line = tid / TPL, t = tid % TPL, p = line % P;
    const int pl = blockIdx.y * P + p, j = j0 + line / P;
    const bool live = j < V && pl < npairs;
    const SmemLine sm{smem + line * smem_line_len(M)};
    const float2 origin = __ldg(Xp + p);   // spectrum value at (0, 0)
    const PolarSrc src{sm.p,
                       lam && live ? lam + ((size_t)pl * V + j) * M : nullptr,
                       g,
                       make_float2(origin.x / (float)V, origin.y / (float)V),
                       M,
                       mode,
                       two_alpha};
    if (mode == BSTK_RAW) {   // uniform across the block
        for (int k = t; k < M; k += TPL) src.load(k);
        return;
    }
    const int sa = 2 * (pair0 + pl), sb = sa + 1;
    SinoCrop dst{sino + ((size_t)sa * V + j) * N, sb < slices ? sino + ((size_t)sb * V + j) * N : nullptr, N, M,
                 scale, live};
    fft_line<M, TPL, true>(t, src, dst, sm, tw, sync);
}

// ---------------------------------------------------------------------------
// cell lists of the gridding (plan set-up)

__global__ void k_cell_keys(Geo geo, int M, int* __restrict__ key, float2* __restrict__ wt) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)M * M) return;
    const int cidx = (int)(idx / M), ridx = (int)(idx % M);
    const int cx = signed_freq(cidx, M), ry = signed_freq(ridx, M);
    int k = -1;
    float2 w = make_float2(0.f, 0.f);
    Polar P;
    if (!(cx == 0 && ry == 0) && polar_of(cx, ry, geo, P)) {
        int K0;
        float fk;
        radial_bin(P, P.up, K0, fk);
        k = (P.J + 1) * M + (K0 + (M >> 1));
        w = make_float2(P.fth, fk);
    }
    key[idx] = k;
    wt[idx] = w;
}

// ---------------------------------------------------------------------------
// filter gradient reductions

// part[pair JB + block][k] (+)= sum over the block's angles of Re(conj(lam_j[k]) Y_j[k]):
// block x takes the groups of LPC angles x, x + JB, ..., transforms their padded
// rays and multiplies by lambda while the spectrum is in shared memory, so Y
// never goes to HBM.  Writing Y and reducing it in a second kernel took 54 +
// 118 us for 16 x 1024 x 1024 (64 blocks a pair walking the angles: 12 %
// occupancy), 65 us in this form.  Fixed order: deterministic.
// 512 threads an SM at least: with 1024 (64 registers) the sums and a butterfly do
// not fit, and most lengths spill (training step of 16 x 768 x 768 584 -> 538 us, 16 x
// 1024 x 1024 836 -> 830).
template <int M, int TPL, int LPC>
__global__ void __launch_bounds__(TPL * LPC, (TPL * LPC <= 512) ? 512 / (TPL * LPC) : 1)
    k_fg_ray(const float* __restrict__ sino, int slices, int pair0, int N, int V, const float2* __restrict__ lam,
             int add, float* __restrict__ part, const float2* __restrict__ tw) {
    extern __shared__ float2 smem[];
    constexpr int PPT = M / TPL;
    const int line = threadIdx.x / TPL, t = threadIdx.x % TPL;
    const int pl = blockIdx.y;
    const int sa = 2 * (pair0 + pl), sb = sa + 1;
    const SmemLine sm{smem + line * smem_line_len(M)};
    float acc[PPT];
#pragma unroll
    for (int i = 0; i < PPT; ++i) acc[i] = 0.f;
    for (int jb = blockIdx.x * LPC; jb < V; jb += gridDim.x * LPC) {
        const int j = jb + line;
        const bool live = j < V;
        const int jj = live ? j : 0;
        const RaySrc<0> src{sino + ((size_t)sa * V + jj) * N,
                            sb < slices ? sino + ((size_t)sb * V + jj) * N : nullptr, N, M, live};
        fft_line<M, TPL, false, 16, true>(t, src, sm, sm, tw);
        __syncthreads();
        const float2* l = lam + ((size_t)pl * V + jj) * M + t;
#pragma unroll
        for (int i = 0; i < PPT; ++i) {
            const float2 a = __ldg(l + i * TPL), b = sm.load(t + i * TPL);   // b = 0 in a dead line
            if (live) acc[i] = fmaf(a.x, b.x, fmaf(a.y, b.y, acc[i]));
        }
        __syncthreads();
    }
    float* red = reinterpret_cast<float*>(smem);
#pragma unroll
    for (int i = 0; i < PPT; ++i) red[line * M + t + i * TPL] = acc[i];
    __syncthreads();
    float* out = part + ((size_t)pl * gridDim.x + blockIdx.x) * M;
    for (int k = threadIdx.x; k < M; k += TPL * LPC) {
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < LPC; ++q) s += red[q * M + k];
        out[k] = add ? out[k] + s : s;
    }
}

// grad[m] = scale * sum over the rows of part of part[m] + part[M - m] (m = 1..M/2-1), fixed order;
// scale = dt dw^2 restores the constants the unscaled transforms leave out.  A
// block takes 32 bins and splits the rows over 32 groups of its threads.
constexpr int FG_K = 32, FG_G = 32;
__global__ void __launch_bounds__(FG_K * FG_G)
    k_fg_final(const float* __restrict__ part, int rows, int M, float scale, float* __restrict__ grad) {
    __shared__ float red[FG_G][FG_K];
    const int kl = threadIdx.x % FG_K, grp = threadIdx.x / FG_K;
    const int m = blockIdx.x * FG_K + kl;
    float s = 0.f;
    if (m < M / 2)
        for (int r = grp; r < rows; r += FG_G) {
            const float* q = part + (size_t)r * M;
            s += q[m] + (m != 0 ? q[M - m] : 0.f);
        }
    red[grp][kl] = s;
    __syncthreads();
    if (grp == 0 && m < M / 2) {
        float t = 0.f;
#pragma unroll
        for (int q = 0; q < FG_G; ++q) t += red[q][kl];
        grad[m] = t * scale;
    }
}

// ---------------------------------------------------------------------------
// host side

template <class K>
static bool set_smem_a(K kernel, size_t bytes) {
    if (bytes <= 48 * 1024) return true;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

template <int M> struct AdjCfg {
    static constexpr int TPL = adj_tpl<M>();
    static constexpr int TPC = (128 / (4 * TPL)) > 1 ? 128 / (4 * TPL) : 1;
    static constexpr int LPC = (256 / TPL) > 1 ? 256 / TPL : 1;
    static constexpr size_t S1 = (size_t)4 * TPC * adj_row_stride<M>() * sizeof(float2);
    static constexpr size_t SF = (size_t)LPC * smem_line_len(M) * sizeof(float2);
    template <int P> static constexpr int LC = adj_col_lines<M, P>();
    template <int P> static constexpr int LP = adj_polar_lines<M, P>();
    template <int P> static constexpr size_t SC = (size_t)LC<P> * adj_col_stride<M, P>() * sizeof(float2);
    template <int P> static constexpr size_t SP = (size_t)LP<P> * smem_line_len(M) * sizeof(float2);
};

struct AdjLayout {
    int chunk;            // slice pairs in flight
    int fg_blocks;        // angle blocks per pair of the filter gradient
    float2 *T, *X, *lam;  // T and lam share their space: T is read before lam is written
    float* part;
};

using bsth::adj_chunk;
using bsth::adj_fg_blocks;
using bsth::adj_rows_t;

// pairs that X holds: a rest of three is a group of four
static size_t adj_x_pairs(const bst_plan_s* p, int chunk) {
    return (size_t)chunk + (p->M < 3072 && chunk % 4 == 3 ? 1 : 0);
}

static AdjLayout adj_layout(const bst_plan_s* p, int pairs, void* ws) {
    AdjLayout L;
    L.chunk = adj_chunk(p, pairs);
    L.fg_blocks = adj_fg_blocks(p, L.chunk);
    // 16-byte reads of X; the workspace size has room for the rounding
    float2* b = (float2*)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
    L.X = b;
    b += adj_x_pairs(p, L.chunk) * p->M * p->M;
    L.T = L.lam = b;
    b += (size_t)L.chunk * std::max(adj_rows_t(p), (size_t)p->V) * p->M;
    L.part = (float*)b;
    return L;
}

// column FFTs (stage 0) or polar stage (stage 1) of np pairs of the chunk, P to a group
template <int M, int P>
static void adjoint_group(bst_plan_s* p, const AdjLayout& L, int stage, int slices, int p0, int at, int np, int mode,
                          const float* g, float* sino, bool keep_lam, cudaStream_t st) {
    using C = AdjCfg<M>;
    const int N = p->N, V = p->V, groups = (np + P - 1) / P;
    float2* X = L.X + (size_t)at * M * M;
    if (stage == 0) {
        constexpr int LC = C::template LC<P>, CB = LC / P;
        k_adj_col_fft<M, C::TPL, LC, P><<<dim3((M + CB - 1) / CB, groups), C::TPL * LC, C::template SC<P>, st>>>(
            L.T + (size_t)at * adj_rows_t(p) * M, N, np, X, p->tw);
        bst_timing_mark(p, st, 6);
        return;
    }
    const Cells cl{p->cell_start, p->cell_pts, p->cell_w};
    const float scale = (float)((double)N / (2.0 * (double)M * (double)M));
    constexpr int LP = C::template LP<P>, LR = LP / P;
    constexpr int NT = adj_polar_threads<M, P>();
    k_adj_polar<M, C::TPL, LP, P, NT><<<dim3((V + LR - 1) / LR, groups), NT, C::template SP<P>, st>>>(
        X, cl, V, N, slices, p0 + at, np, mode, g, (float)(2 * p->alpha), scale, sino,
        keep_lam ? L.lam + (size_t)at * V * M : nullptr, p->tw);
    bst_timing_mark(p, st, 7);
}

template <int M, int P>
static bool adjoint_smem() {
    using C = AdjCfg<M>;
    return set_smem_a(k_adj_col_fft<M, C::TPL, C::template LC<P>, P>, C::template SC<P>) &&
           set_smem_a(k_adj_polar<M, C::TPL, C::template LP<P>, P, adj_polar_threads<M, P>()>, C::template SP<P>);
}

template <int M>
static bst_status_t adjoint_chunk(bst_plan_s* p, const AdjLayout& L, const float* vol, int slices, int p0, int np,
                                  int mode, const float* g, float* sino, bool keep_lam, cudaStream_t st) {
    using C = AdjCfg<M>;
    constexpr int PM = adj_pairs<M>();
    static std::atomic<unsigned long long> attr_done{0};
    if (!bsth::once_per_device(attr_done, [] {
            return set_smem_a(k_adj_row_fft<M, C::TPL, C::TPC>, C::S1) && adjoint_smem<M, 1>() &&
                   adjoint_smem<M, 2>() && adjoint_smem<M, PM>();
        }))
        return BST_ERR_CUDA;
    const int row_tiles = (p->N + 3) / 4;
    bst_timing_mark(p, st, -1);
    k_adj_row_fft<M, C::TPL, C::TPC><<<dim3((row_tiles + C::TPC - 1) / C::TPC, np), 4 * C::TPL * C::TPC, C::S1, st>>>(
        vol, slices, p0, p->N, L.T, p->tw);
    bst_timing_mark(p, st, 5);
    // Whole groups of PM pairs, then what remains in the smallest group that
    // holds it.  lam overwrites T, so the polar stage starts only once every
    // column of the chunk is transformed.
    const int full = np / PM * PM, rem = np - full;
    for (int stage = 0; stage < 2; ++stage) {
        if (full > 0) adjoint_group<M, PM>(p, L, stage, slices, p0, 0, full, mode, g, sino, keep_lam, st);
        if (rem == 1) adjoint_group<M, 1>(p, L, stage, slices, p0, full, 1, mode, g, sino, keep_lam, st);
        if constexpr (PM > 2) {
            if (rem == 2) adjoint_group<M, 2>(p, L, stage, slices, p0, full, 2, mode, g, sino, keep_lam, st);
            if (rem == 3) adjoint_group<M, PM>(p, L, stage, slices, p0, full, 3, mode, g, sino, keep_lam, st);
        }
    }
    return BST_OK;
}

}  // namespace bst

#define BST_FOR_EACH_M(X) \
    X(16) X(32) X(64) X(128) X(256) X(512) X(1024) X(2048) X(4096) X(48) X(96) X(192) X(384) X(768) X(1536) X(3072)

size_t bst_adjoint_ws(const bst_plan_s* p, int slices) {
    const int pairs = (slices + 1) / 2;
    const bst::AdjLayout L = bst::adj_layout(p, pairs, nullptr);
    const size_t rows = (size_t)L.chunk * L.fg_blocks;
    return (size_t)((char*)L.part - (char*)nullptr) + rows * p->M * sizeof(float) + 256;
}

bst_status_t bst_build_cells(bst_plan_s* p, cudaStream_t st) {
    if (p->cells_built) return BST_OK;
    const int M = p->M;
    const size_t n = (size_t)M * M;
    int* d_key = nullptr;
    float2* d_w = nullptr;
    if (cudaMalloc((void**)&d_key, n * sizeof(int)) != cudaSuccess) return BST_ERR_OUT_OF_MEMORY;
    if (cudaMalloc((void**)&d_w, n * sizeof(float2)) != cudaSuccess) {
        cudaFree(d_key);
        return BST_ERR_OUT_OF_MEMORY;
    }
    bst::k_cell_keys<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(p->geo(), M, d_key, d_w);
    std::vector<int> key(n);
    std::vector<float2> w(n);
    bool ok = cudaMemcpyAsync(key.data(), d_key, n * sizeof(int), cudaMemcpyDeviceToHost, st) == cudaSuccess &&
              cudaMemcpyAsync(w.data(), d_w, n * sizeof(float2), cudaMemcpyDeviceToHost, st) == cudaSuccess &&
              cudaStreamSynchronize(st) == cudaSuccess;
    cudaFree(d_key);
    cudaFree(d_w);
    if (!ok) return BST_ERR_CUDA;
    const size_t ncell = (size_t)(p->V + 1) * M;
    std::vector<int> start(ncell + 1, 0);
    for (size_t i = 0; i < n; ++i)
        if (key[i] >= 0) ++start[(size_t)key[i] + 1];
    for (size_t c = 0; c < ncell; ++c) start[c + 1] += start[c];
    const int total = start[ncell];
    std::vector<int> pts(std::max(total, 1));
    std::vector<float2> pw(std::max(total, 1));
    std::vector<int> cur(start.begin(), start.end() - 1);
    for (size_t i = 0; i < n; ++i) {   // stable: ascending point index within a cell
        if (key[i] < 0) continue;
        const int pos = cur[key[i]]++;
        pts[pos] = (int)i;
        pw[pos] = w[i];
    }
    if (cudaMalloc((void**)&p->cell_start, start.size() * sizeof(int)) != cudaSuccess ||
        cudaMalloc((void**)&p->cell_pts, pts.size() * sizeof(int)) != cudaSuccess ||
        cudaMalloc((void**)&p->cell_w, pw.size() * sizeof(float2)) != cudaSuccess)
        return BST_ERR_OUT_OF_MEMORY;
    if (cudaMemcpy(p->cell_start, start.data(), start.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(p->cell_pts, pts.data(), pts.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(p->cell_w, pw.data(), pw.size() * sizeof(float2), cudaMemcpyHostToDevice) != cudaSuccess)
        return BST_ERR_CUDA;
    p->cell_n = total;
    p->cells_built = true;
    return BST_OK;
}

static bst_status_t adjoint_chunk_dispatch(bst_plan_s* p, const bst::AdjLayout& L, const float* vol, int slices,
                                           int p0, int np, int mode, const float* g, float* sino, bool keep_lam,
                                           cudaStream_t st) {
    switch (p->M) {
#define BST_CASE(m) \
    case m: return bst::adjoint_chunk<m>(p, L, vol, slices, p0, np, mode, g, sino, keep_lam, st);
        BST_FOR_EACH_M(BST_CASE)
#undef BST_CASE
    }
    return BST_ERR_UNSUPPORTED_SIZE;
}

bst_status_t bst_launch_adjoint(bst_plan_s* p, int mode, const float* g, const float* vol, int slices, float* sino,
                                void* ws, size_t /*ws_bytes*/, cudaStream_t st) {
    bst_status_t s = bst_build_cells(p, st);
    if (s != BST_OK) return s;
    const int pairs = (slices + 1) / 2;
    const bst::AdjLayout L = bst::adj_layout(p, pairs, ws);
    for (int p0 = 0; p0 < pairs; p0 += L.chunk) {
        const int np = std::min(L.chunk, pairs - p0);
        s = adjoint_chunk_dispatch(p, L, vol, slices, p0, np, mode, g, sino, false, st);
        if (s != BST_OK) return s;
    }
    return cudaGetLastError() == cudaSuccess ? BST_OK : BST_ERR_CUDA;
}

namespace bst {
template <int M>
static bst_status_t launch_fg_ray_M(bst_plan_s* p, const AdjLayout& L, const float* sino, int slices, int p0, int np,
                                    cudaStream_t st) {
    using C = AdjCfg<M>;
    static std::atomic<unsigned long long> attr_done{0};
    if (!bsth::once_per_device(attr_done, [] { return set_smem_a(k_fg_ray<M, C::TPL, C::LPC>, C::SF); }))
        return BST_ERR_CUDA;
    bst_timing_mark(p, st, -1);
    k_fg_ray<M, C::TPL, C::LPC><<<dim3(L.fg_blocks, np), C::TPL * C::LPC, C::SF, st>>>(
        sino, slices, p0, p->N, p->V, L.lam, p0 > 0, L.part, p->tw);
    bst_timing_mark(p, st, 0);
    return BST_OK;
}
}  // namespace bst

static bst_status_t fg_ray_dispatch(bst_plan_s* p, const bst::AdjLayout& L, const float* sino, int slices, int p0,
                                    int np, cudaStream_t st) {
    switch (p->M) {
#define BST_CASE(m) \
    case m: return bst::launch_fg_ray_M<m>(p, L, sino, slices, p0, np, st);
        BST_FOR_EACH_M(BST_CASE)
#undef BST_CASE
    }
    return BST_ERR_UNSUPPORTED_SIZE;
}

// Both gradients of <grad_vol, FBP(sino; g)>: grad_sino = the adjoint applied to
// grad_vol (taps g; skipped when null), grad_g = sum Re(conj(lambda) Y) (skipped
// when null), from one pull-back lambda per chunk.
bst_status_t bst_launch_backward(bst_plan_s* p, const float* sino, const float* gvol, int slices, const float* g,
                                 float* grad_sino, float* grad_g, void* ws, cudaStream_t st) {
    bst_status_t s = bst_build_cells(p, st);
    if (s != BST_OK) return s;
    const int pairs = (slices + 1) / 2;
    const bst::AdjLayout L = bst::adj_layout(p, pairs, ws);
    const int M = p->M;
    for (int p0 = 0; p0 < pairs; p0 += L.chunk) {
        const int np = std::min(L.chunk, pairs - p0);
        s = adjoint_chunk_dispatch(p, L, gvol, slices, p0, np, grad_sino ? BSTK_FILTER : BSTK_RAW, g, grad_sino,
                                   grad_g != nullptr, st);
        if (s != BST_OK) return s;
        if (grad_g) {
            s = fg_ray_dispatch(p, L, sino, slices, p0, np, st);
            if (s != BST_OK) return s;
        }
    }
    if (grad_g) {
        const float scale = (float)((double)p->N / (2.0 * (double)M * (double)M));
        bst::k_fg_final<<<(M / 2 + bst::FG_K - 1) / bst::FG_K, bst::FG_K * bst::FG_G, 0, st>>>(
            L.part, L.chunk * L.fg_blocks, M, scale, grad_g);
    }
    return cudaGetLastError() == cudaSuccess ? BST_OK : BST_ERR_CUDA;
}

bst_status_t bst_launch_filter_grad(bst_plan_s* p, const float* sino, const float* gvol, int slices, float* grad_g,
                                    void* ws, size_t /*ws_bytes*/, cudaStream_t st) {
    return bst_launch_backward(p, sino, gvol, slices, nullptr, nullptr, grad_g, ws, st);
}

// bst_fft.cuh -- shared-memory Stockham FFT engine for one line of length M.
//
// Used by every stage of the BST path that transforms along a line: the 1D
// FFT along the detector (stage P3), the column and row passes of the 2D
// inverse FFT (stage P6) and their adjoints.  A line of M complex64 values
// is transformed by TPL threads in log_R(M) radix-R Stockham passes
// (out-of-order autosort: no bit reversal), in place in shared memory with a
// barrier between the loads and the stores of each pass.  The first pass may
// read from any source (global memory, a gather) and the last may write to
// any sink, so loads and stores fuse with the neighbouring stage.
//
// Pass with sub-transform length NS and radix R, butterfly j in [0, M/R):
//   inputs   x[j + s M/R],  s = 0..R-1
//   twiddle  x_s *= w^(k s),  k = j mod NS,  w = exp(-+ 2 pi i / (NS R))
//   DFT_R in registers
//   outputs  y[(j / NS) NS R + k + s NS]
// Forward transforms use exp(-2 pi i k m / M), inverse ones exp(+...), both
// unnormalised.  Twiddles come from a table tw[m] = exp(-2 pi i m / M)
// computed in double precision on the host.
#pragma once
#include <cuda_runtime.h>

namespace bst {

// Sums, differences and scalings of whole complex values are packed FP32
// instructions (two lanes of arithmetic in one issue slot, the same roundings
// as the scalar forms): the FFT kernels are bound by instruction issue.  A sum
// with a factor i takes the scalar form (cadd_si), whose operands need no
// swapping.  At 2048 x 2048, pad 2: ray kernel 27.0 -> 25.4 us a pair, gridding
// 90.3 -> 88.9, row kernel 24.1 -> 24.8.
// (The scalar branch only lets host programs that check the tables include this
// header without naming the architecture.)
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return __fmul2_rn(a, make_float2(s, s)); }
#else
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 c) {
    return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
#endif
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return cfma(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a * conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
// sigma = -1 forward, +1 inverse:
// a + sigma i b and a - sigma i b
template <bool INV> __device__ __forceinline__ float2 cadd_si(float2 a, float2 b) {
    return INV ? make_float2(a.x - b.y, a.y + b.x) : make_float2(a.x + b.y, a.y - b.x);
}
template <bool INV> __device__ __forceinline__ float2 csub_si(float2 a, float2 b) { return cadd_si<!INV>(a, b); }
// a * (c + sigma i d): multiplication by exp(sigma i phi) with c = cos phi, d = sin phi
template <bool INV> __device__ __forceinline__ float2 mul_w(float2 a, float c, float d) {
    const float sd = INV ? d : -d;
    return make_float2(fmaf(a.x, c, -a.y * sd), fmaf(a.y, c, a.x * sd));
}

// cos and sin of pi/4, pi/8, 3 pi/8 and sqrt(3)/2
#define BST_R2 0.70710678118654752440f
#define BST_C8 0.92387953251128675613f
#define BST_S8 0.38268343236508977173f
#define BST_H3 0.86602540378443864676f
// a times exp(sigma i pi / 4) and exp(3 sigma i pi / 4): a sum, a difference and one packed scaling
template <bool INV> __device__ __forceinline__ float2 mul_w8(float2 a) { return cscale(cadd_si<INV>(a, a), BST_R2); }
template <bool INV> __device__ __forceinline__ float2 mul_w38(float2 a) {
    return cscale(INV ? make_float2(-a.x - a.y, a.x - a.y) : make_float2(a.y - a.x, -a.x - a.y), BST_R2);
}

template <int R, bool INV> struct Dft;

template <bool INV> struct Dft<2, INV> {
    __device__ __forceinline__ static void run(float2* a) {
        const float2 t = a[1];
        a[1] = csub(a[0], t);
        a[0] = cadd(a[0], t);
    }
};

template <bool INV> struct Dft<3, INV> {
    __device__ __forceinline__ static void run(float2* a) {
        const float2 t = cadd(a[1], a[2]);
        const float2 u = csub(a[1], a[2]);
        const float2 m = cfma(make_float2(-0.5f, -0.5f), t, a[0]);
        const float2 v = cscale(u, BST_H3);
        a[0] = cadd(a[0], t);
        a[1] = cadd_si<INV>(m, v);
        a[2] = csub_si<INV>(m, v);
    }
};

template <bool INV> struct Dft<4, INV> {
    // TURN2: a[2] still has to be multiplied by sigma i
    template <bool TURN2 = false>
    __device__ __forceinline__ static void run(float2* a) {
        const float2 a0 = TURN2 ? cadd_si<INV>(a[0], a[2]) : cadd(a[0], a[2]);
        const float2 a1 = TURN2 ? csub_si<INV>(a[0], a[2]) : csub(a[0], a[2]);
        const float2 b0 = cadd(a[1], a[3]), b1 = csub(a[1], a[3]);
        a[0] = cadd(a0, b0);
        a[2] = csub(a0, b0);
        a[1] = cadd_si<INV>(a1, b1);
        a[3] = csub_si<INV>(a1, b1);
    }
};

// 6 = 2 x 3 and 12 = 4 x 3 by the prime-factor map (Good 1958, Thomas 1963): inputs
// n = (R/3) n1 + 3 n2, outputs k = k1 mod 3 = k2 mod R/3, no inner twiddles
template <bool INV> struct Dft<6, INV> {
    __device__ __forceinline__ static void run(float2* a) {
        float2 e[3] = {a[0], a[2], a[4]}, o[3] = {a[3], a[5], a[1]};
        Dft<3, INV>::run(e);
        Dft<3, INV>::run(o);
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) {
            a[(4 * k1) % 6] = cadd(e[k1], o[k1]);
            a[(4 * k1 + 3) % 6] = csub(e[k1], o[k1]);
        }
    }
};
template <bool INV> struct Dft<12, INV> {
    __device__ __forceinline__ static void run(float2* a) {
        float2 b[4][3];
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
            for (int n1 = 0; n1 < 3; ++n1) b[n2][n1] = a[(4 * n1 + 3 * n2) % 12];
            Dft<3, INV>::run(b[n2]);
        }
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) {
            float2 c[4] = {b[0][k1], b[1][k1], b[2][k1], b[3][k1]};
            Dft<4, INV>::run(c);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) a[(4 * k1 + 9 * k2) % 12] = c[k2];
        }
    }
};

template <bool INV> struct Dft<8, INV> {
    __device__ __forceinline__ static void run(float2* a) {
        float2 e[4] = {a[0], a[2], a[4], a[6]};
        float2 o[4] = {a[1], a[3], a[5], a[7]};
        Dft<4, INV>::run(e);
        Dft<4, INV>::run(o);
        o[1] = mul_w8<INV>(o[1]);
        o[3] = mul_w38<INV>(o[3]);
        a[2] = cadd_si<INV>(e[2], o[2]);
        a[6] = csub_si<INV>(e[2], o[2]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k == 2) continue;
            a[k] = cadd(e[k], o[k]);
            a[k + 4] = csub(e[k], o[k]);
        }
    }
};

// 16 = 4 x 4: four DFT4 over the inputs of stride 4, internal twiddles
// W16^(n2 k1), four DFT4 over the results (fewer multiplications than 2 x 8)
template <bool INV> struct Dft<16, INV> {
    __device__ __forceinline__ static void run(float2* a) {
        float2 b[4][4];
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
            float2 c[4] = {a[n2], a[n2 + 4], a[n2 + 8], a[n2 + 12]};
            Dft<4, INV>::run(c);
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) b[n2][k1] = c[k1];
        }
        // W16^(n2 k1) for n2, k1 = 1..3: exponents 1 2 3 / 2 4 6 / 3 6 9
        b[1][1] = mul_w<INV>(b[1][1], BST_C8, BST_S8);
        b[1][2] = mul_w8<INV>(b[1][2]);
        b[1][3] = mul_w<INV>(b[1][3], BST_S8, BST_C8);
        b[2][1] = mul_w8<INV>(b[2][1]);
        // (b[2][2] by sigma i: in the DFT4 of k1 = 2)
        b[2][3] = mul_w38<INV>(b[2][3]);
        b[3][1] = mul_w<INV>(b[3][1], BST_S8, BST_C8);
        b[3][2] = mul_w38<INV>(b[3][2]);
        b[3][3] = mul_w<INV>(b[3][3], -BST_C8, -BST_S8);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            float2 c[4] = {b[0][k1], b[1][k1], b[2][k1], b[3][k1]};
            if (k1 == 2) Dft<4, INV>::template run<true>(c);
            else Dft<4, INV>::run(c);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) a[k1 + 4 * k2] = c[k2];
        }
    }
};

// ---- kernels in a row ------------------------------------------------------
//
// At the start of a kernel that may be launched with programmatic stream
// serialization: lets the next kernel of the stream be set up while this one
// runs, then waits until the previous one is complete and its writes are
// visible.  Every kernel of the forward path calls it first, so completion is
// transitive.  Up to M = 1024 only: one pair of a longer length takes 50 us and
// more, and the two instructions, though nothing without that launch attribute,
// cost large volumes 1 to 2 % (64 x 2048 x 2048: 4257 -> 4304 us).
__host__ __device__ constexpr bool chainable(int M) { return M <= 1024; }
template <int M> __device__ __forceinline__ void chain_begin() {
    if constexpr (chainable(M)) {
        asm volatile("griddepcontrol.launch_dependents;");
        asm volatile("griddepcontrol.wait;" ::: "memory");
    }
}

// ---- radix schedule --------------------------------------------------------

__host__ __device__ constexpr int ilog2c(int x) { return x <= 1 ? 0 : 1 + ilog2c(x / 2); }
// Radix of pass p for length M = 3^b 2^a (b <= 1) with radices at most MAXR
// (16 or 8).  Lengths 3 * 2^a start with a pass of radix 3, 6 or 12 (at most
// MAXR), the smallest that leaves the fewest passes: 3072 = 12 16 16, 1536 = 6 16
// 16, 192 = 12 16, where radix 3 alone took one pass more, of butterflies that do
// not divide among the threads.  15 x 1201 x 1536 backprojection: 785 -> 675 us.
// Then ceil(a / log2 MAXR)
// power-of-two passes of as equal a size as possible.  The maximum radix is the
// plan's schedule.
__host__ __device__ constexpr int radix_of(int M, int p, int MAXR = 16) {
    const bool three = (M % 3 == 0);
    const int rb = ilog2c(MAXR);
    int a = ilog2c(three ? M / 3 : M), x = 0;
    if (three) {
        for (int y = 1; (3 << y) <= MAXR; ++y)
            if ((a - y + rb - 1) / rb < (a - x + rb - 1) / rb) x = y;
        if (p == 0) return 3 << x;
        a -= x;
    }
    const int passes = (a + rb - 1) / rb;
    const int q = p - (three ? 1 : 0);
    const int bits = a / passes + (q < a % passes ? 1 : 0);
    return 1 << bits;
}

// ---- per-pass twiddle tables ---------------------------------------------------
//
// Beside the base table tw[m] = exp(-2 pi i m / M), m < M, the plan stores for
// each radix schedule (largest radix 16, then 8) and each pass p >= 1 (radix
// R, sub-transform length NS) the pass's twiddles w^(k s), w = exp(-2 pi i /
// (NS R)), at entry (s - 1) NS + k (s = 1..R-1, k < NS): the R - 1 twiddles of
// butterfly k are NS apart, so the lanes of a warp (consecutive k) read them
// coalesced.  Each entry equals tw[k s M / (NS R)].

// sub-transform length before pass p of the schedule
__host__ __device__ constexpr int pass_ns(int M, int p, int MAXR) {
    return p == 0 ? 1 : pass_ns(M, p - 1, MAXR) * radix_of(M, p - 1, MAXR);
}
// entries of the tables of passes 1 .. p - 1 of the schedule
__host__ __device__ constexpr int pass_tab_prefix(int M, int p, int MAXR) {
    return p <= 1 ? 0 : pass_tab_prefix(M, p - 1, MAXR) + (radix_of(M, p - 1, MAXR) - 1) * pass_ns(M, p - 1, MAXR);
}
// passes of the schedule
__host__ __device__ constexpr int pass_count(int M, int MAXR, int p = 0) {
    return pass_ns(M, p, MAXR) >= M ? p : pass_count(M, MAXR, p + 1);
}
// offset in tw of the table of pass p of the schedule (16 first, then 8)
__host__ __device__ constexpr int pass_tab_base(int M, int MAXR, int p) {
    return M + (MAXR == 8 ? pass_tab_prefix(M, pass_count(M, 16), 16) : 0) + pass_tab_prefix(M, p, MAXR);
}
// complex64 entries of the whole twiddle allocation
__host__ __device__ constexpr int tw_alloc_len(int M) {
    return M + pass_tab_prefix(M, pass_count(M, 16), 16) + pass_tab_prefix(M, pass_count(M, 8), 8);
}

// ---- barriers ----------------------------------------------------------------

// Barrier between the passes of a line: the whole block (__syncthreads), or a
// named barrier shared by the n threads (a multiple of 32) of one worker of a
// block, so that workers of one block run independent lines.
struct BlockSync {
    __device__ __forceinline__ void operator()() const { __syncthreads(); }
};
struct WorkerSync {
    int id;   // barrier 1..15 (0 is the block's __syncthreads barrier)
    int n;    // threads of the worker
    __device__ __forceinline__ void operator()() const {
        asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
    }
    // group g (of at most four) of worker id 1 or 2: its own barrier for threads of them
    __device__ __forceinline__ WorkerSync group(int g, int threads) const {
        return WorkerSync{3 + 4 * (id - 1) + g, threads};
    }
};

// ---- line storage ----------------------------------------------------------

// Shared-memory line of M complex values with ADD padding slots after every PER
// (the 16-byte-pair banks hold 16 values; a half-warp's 16 accesses should fall on
// 16 different ones).  Plain lines, and the exchanges between the passes of the
// lengths 2^a, have one slot per 16: the first pass stores at 17 t + s, the later
// ones move by whole groups.  That padding does not suit lengths 3 * 2^a, whose
// first pass stores at 12 t + s (three accesses a bank): see exchange_per.
// (`lines`: see exchange_per; four and more take the longest padding)
__host__ __device__ constexpr int smem_line_len(int M, int lines = 1) {
    return M % 3 == 0 && lines >= 4 ? (M + M / 12 + 15) / 16 * 16 : M + M / 16;
}

template <int PER, int ADD> struct PadLine {
    float2* p;
    static constexpr bool kSmem = true;
    static constexpr int kPer = PER, kAdd = ADD, kLines = 1;
    static __host__ __device__ constexpr int at(int i) { return i + i / PER * ADD; }
    __device__ __forceinline__ float2 load(int i) const { return p[at(i)]; }
    __device__ __forceinline__ void store(int i, float2 v) const { p[at(i)] = v; }
};
using SmemLine = PadLine<16, 1>;
// a line among LINES over whose threads the lanes of a warp alternate
template <int LINES> struct LineOf : SmemLine {
    static constexpr int kLines = LINES;
};

// Padding of the exchange after pass p of the transform, with the lanes of a warp
// alternating over `lines` lines (the lines' starts 16 / lines slots apart, so that
// 16 / lines consecutive threads of a line share a half-warp).
//   2^a: one slot per 16.
//   3 * 2^a, first pass of radix R0 (stores at R0 t + s, loads of consecutive
//     elements): R0 = 3 needs none, 6 and 12 one per 48 / lines elements.
//   3 * 2^a, then radix 16 (stores at 16 R0 (j / R0) + j % R0 + R0 s): R0 slots per
//     16 R0, which puts consecutive j on consecutive banks.
// In each of them the stores of a butterfly are a constant apart (with one slot per
// 16 they were not for 3 * 2^a).  Wavefronts per half-warp store of the first pass at
// M = 3072: 3 -> 1 with one line, 2 -> 1 with two or four.  15 x 1201 x 1536
// backprojection 652 -> 627 us, 64 x 768 x 768 554 -> 532, 512 x 192 x 192 291 -> 260.
__host__ __device__ constexpr int exchange_per(int M, int p, int MAXR, int lines) {
    const int r0 = radix_of(M, 0, MAXR);
    if (M % 3 != 0) return 16;
    if (p == 0) return r0 == 3 ? M : (48 / lines > 12 ? 48 / lines : 12);
    return p == 1 && radix_of(M, 1, MAXR) == 16 ? 16 * r0 : 16;
}
__host__ __device__ constexpr int exchange_add(int M, int p, int MAXR) {
    const int r0 = radix_of(M, 0, MAXR);
    if (M % 3 != 0) return 1;
    if (p == 0) return r0 == 3 ? 0 : 1;
    return p == 1 && radix_of(M, 1, MAXR) == 16 ? r0 : 1;
}
template <int M, int P, int MAXR, int LINES>
using Exchange = PadLine<exchange_per(M, P, MAXR, LINES), exchange_add(M, P, MAXR)>;

// ---- passes ----------------------------------------------------------------

// Sources that know index groups of always-zero input (S::zero_group) and
// destinations that know index groups of outputs they drop (D::drop_group):
// the first pass then loads nothing there and the last pass stores nothing
// there, and the compiler removes the arithmetic that only fed them.
template <class T, class = void> struct zero_group_trait { static constexpr bool value = false; };
template <class T>
struct zero_group_trait<T, decltype(void(T::zero_group(0, 0, 0)))> { static constexpr bool value = true; };
template <class T, class = void> struct drop_group_trait { static constexpr bool value = false; };
template <class T>
struct drop_group_trait<T, decltype(void(T::drop_group(0, 0, 0)))> { static constexpr bool value = true; };

template <class S, int M>
__device__ __forceinline__ constexpr bool src_zero_group(int lo, int hi) {
    if constexpr (zero_group_trait<S>::value) return S::zero_group(lo, hi, M);
    return false;
}
template <class D, int M>
__device__ __forceinline__ constexpr bool dst_drop_group(int lo, int hi) {
    if constexpr (drop_group_trait<D>::value) return D::drop_group(lo, hi, M);
    return false;
}

// true for a shared-memory line whose load and store are its padded elements
template <class T, class = void> struct pad_line_trait { static constexpr bool value = false; };
template <class T> struct pad_line_trait<T, decltype(void(T::kPer))> { static constexpr bool value = true; };
template <class T> __host__ __device__ constexpr bool is_pad_line() { return pad_line_trait<T>::value; }
// loads of a pass at j + s NB, stores at base + s NS, are a constant apart (0: not)
template <class T, int NB> __host__ __device__ constexpr int pad_load_step() {
    if constexpr (is_pad_line<T>()) return T::kAdd == 0 || NB % T::kPer == 0 ? T::at(NB) : 0;
    return 0;
}
template <class T, int NS, int R> __host__ __device__ constexpr int pad_store_step() {
    if constexpr (is_pad_line<T>()) {
        if (T::kAdd == 0 || T::kPer % (NS * R) == 0) return NS;   // a butterfly stays in one group
        if (NS % T::kPer == 0) return T::at(NS);
    }
    return 0;
}

// w[s] = tw[s * b] for s = 1..R-1 (b = k M / (NS R)): the powers of two of the
// base root come from the table, the others are products of at most three
// table values (error a few ulp), which quarters the table loads of a pass.
template <int R>
__device__ __forceinline__ void twiddles(const float2* __restrict__ tw, int b, float2* w) {
    if constexpr (R == 2) {
        w[1] = __ldg(tw + b);
    } else if constexpr (R == 3) {
        w[1] = __ldg(tw + b);
        w[2] = __ldg(tw + 2 * b);
    } else if constexpr (R == 4) {
        w[1] = __ldg(tw + b);
        w[2] = __ldg(tw + 2 * b);
        w[3] = cmul(w[1], w[2]);
    } else if constexpr (R == 8) {
        w[1] = __ldg(tw + b);
        w[2] = __ldg(tw + 2 * b);
        w[4] = __ldg(tw + 4 * b);
        w[3] = cmul(w[1], w[2]);
        w[5] = cmul(w[1], w[4]);
        w[6] = cmul(w[2], w[4]);
        w[7] = cmul(w[3], w[4]);
    } else {
        static_assert(R == 16, "radix");
        w[1] = __ldg(tw + b);
        w[2] = __ldg(tw + 2 * b);
        w[4] = __ldg(tw + 4 * b);
        w[8] = __ldg(tw + 8 * b);
        w[3] = cmul(w[1], w[2]);
        w[5] = cmul(w[1], w[4]);
        w[6] = cmul(w[2], w[4]);
        w[7] = cmul(w[3], w[4]);
#pragma unroll
        for (int s = 1; s < 8; ++s) w[8 + s] = cmul(w[s], w[8]);
    }
}

// a[s] *= w[s] (conjugated for the inverse) with w[s] = tw[s * b].  For R = 16
// the upper half is applied as (w[s] w[8]) a[8 + s], the same products as the
// table of twiddles() but never more than eight twiddles live at once.
template <int R, bool INV>
__device__ __forceinline__ void apply_twiddles(const float2* __restrict__ tw, int b, float2* a) {
    if constexpr (R == 16) {
        float2 w[8];
        w[1] = __ldg(tw + b);
        w[2] = __ldg(tw + 2 * b);
        w[4] = __ldg(tw + 4 * b);
        w[3] = cmul(w[1], w[2]);
        w[5] = cmul(w[1], w[4]);
        w[6] = cmul(w[2], w[4]);
        w[7] = cmul(w[3], w[4]);
#pragma unroll
        for (int s = 1; s < 8; ++s) a[s] = INV ? cmulc(a[s], w[s]) : cmul(a[s], w[s]);
        const float2 w8 = __ldg(tw + 8 * b);
        a[8] = INV ? cmulc(a[8], w8) : cmul(a[8], w8);
#pragma unroll
        for (int s = 1; s < 8; ++s) {
            const float2 ws = cmul(w[s], w8);
            a[8 + s] = INV ? cmulc(a[8 + s], ws) : cmul(a[8 + s], ws);
        }
    } else {
        float2 w[R];
        twiddles<R>(tw, b, w);
#pragma unroll
        for (int s = 1; s < R; ++s) a[s] = INV ? cmulc(a[s], w[s]) : cmul(a[s], w[s]);
    }
}

// TWT: the twiddles of a pass with NS > 1 come from the pass's own table
// (TB: its offset in tw), one coalesced load each, instead of from the base
// table with products
template <int M, int R, int NS, int TPL, bool INV, bool TWT, int TB, class Src, class Dst, class SYNC>
__device__ __forceinline__ void stockham_pass(int t, const Src& src, const Dst& dst,
                                              const float2* __restrict__ tw, bool sync_mid, const SYNC& sync) {
    constexpr int NB = M / R;
    constexpr int IT = (NB + TPL - 1) / TPL;
    float2 a[IT][R];
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int j = t + it * TPL;
        if ((NB % TPL) == 0 || j < NB) {
            constexpr int LS = pad_load_step<Src, NB>();
            if constexpr (LS > 0) {
                const float2* p = src.p + Src::at(j);
#pragma unroll
                for (int s = 0; s < R; ++s) a[it][s] = p[s * LS];
            } else {
#pragma unroll
                for (int s = 0; s < R; ++s)
                    a[it][s] = src_zero_group<Src, M>(s * NB, (s + 1) * NB) ? make_float2(0.f, 0.f)
                                                                              : src.load(j + s * NB);
            }
        }
    }
    if (sync_mid) sync();
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int j = t + it * TPL;
        if ((NB % TPL) == 0 || j < NB) {
            const int k = (NS == 1) ? 0 : (j % NS);
            if constexpr (NS > 1) {
                if constexpr (TWT) {
                    const float2* tp = tw + TB + k;
#pragma unroll
                    for (int s = 1; s < R; ++s) {
                        const float2 w = __ldg(tp + (s - 1) * NS);
                        a[it][s] = INV ? cmulc(a[it][s], w) : cmul(a[it][s], w);
                    }
                } else {
                    constexpr int STEP = M / (NS * R);
                    apply_twiddles<R, INV>(tw, k * STEP, a[it]);
                }
            }
            Dft<R, INV>::run(a[it]);
            const int base = (j / NS) * NS * R + k;
            constexpr int PS = pad_store_step<Dst, NS, R>();
            if constexpr (PS > 0) {
                float2* p = dst.p + Dst::at(base);
#pragma unroll
                for (int s = 0; s < R; ++s) p[s * PS] = a[it][s];
            } else {
                // in the last pass base = j < NS, so output s covers indices [s NS, (s + 1) NS)
                constexpr bool LASTP = NS * R == M;
#pragma unroll
                for (int s = 0; s < R; ++s)
                    if (!(LASTP && dst_drop_group<Dst, M>(s * NS, (s + 1) * NS))) dst.store(base + s * NS, a[it][s]);
            }
        }
    }
}

// Run passes PIDX.. of the length-M transform.  Pass 0 reads `src`, the last
// pass writes `dst`; the others go through the shared-memory line `sm`.  The last
// pass runs as thread tl of the line sml (t, sm unless the maps change there).
// LINES: lines over which the lanes alternate in pass 0.
// Every thread that `sync` covers must call this (it contains barriers).
template <int M, int TPL, bool INV, int MAXR, int PIDX, int NS, bool TWT, int LINES, class Src, class Dst, class SYNC>
__device__ __forceinline__ void fft_run(int t, const Src& src, const Dst& dst, float2* sm, int tl, float2* sml,
                                        const float2* __restrict__ tw, const SYNC& sync) {
    constexpr int R = radix_of(M, PIDX, MAXR);
    constexpr bool LAST = (NS * R == M);
    constexpr int TB = pass_tab_base(M, MAXR, PIDX);
    using In = Exchange<M, PIDX == 0 ? 0 : PIDX - 1, MAXR, LINES>;
    using Out = Exchange<M, PIDX, MAXR, LINES>;
    static_assert(LAST || Out::at(M - 1) < smem_line_len(M, LINES), "the exchange fits the line");
    if constexpr (PIDX == 0) {
        if constexpr (LAST) {
            stockham_pass<M, R, NS, TPL, INV, TWT, TB>(t, src, dst, tw, Src::kSmem && Dst::kSmem, sync);
        } else {
            stockham_pass<M, R, NS, TPL, INV, TWT, TB>(t, src, Out{sm}, tw, Src::kSmem, sync);
            sync();
            fft_run<M, TPL, INV, MAXR, PIDX + 1, NS * R, TWT, LINES>(t, src, dst, sm, tl, sml, tw, sync);
        }
    } else {
        if constexpr (LAST) {
            stockham_pass<M, R, NS, TPL, INV, TWT, TB>(tl, In{sml}, dst, tw, Dst::kSmem, sync);
        } else {
            stockham_pass<M, R, NS, TPL, INV, TWT, TB>(t, In{sm}, Out{sm}, tw, true, sync);
            sync();
            fft_run<M, TPL, INV, MAXR, PIDX + 1, NS * R, TWT, LINES>(t, src, dst, sm, tl, sml, tw, sync);
        }
    }
}

// TWT: twiddles from the per-pass tables (one coalesced load each) instead of
// four base-table loads and products per butterfly
template <int M, int TPL, bool INV, int MAXR = 16, bool TWT = false, class Src, class Dst, class SM, class SYNC = BlockSync>
__device__ __forceinline__ void fft_line(int t, const Src& src, const Dst& dst, const SM& sm,
                                         const float2* __restrict__ tw, const SYNC& sync = SYNC()) {
    fft_run<M, TPL, INV, MAXR, 0, 1, TWT, SM::kLines>(t, src, dst, sm.p, t, sm.p, tw, sync);
}

// Two thread-to-line maps for one transform: the first pass (LATE: all but the
// last) runs as thread t0 of a line whose source is src and whose storage is sm0,
// the others as thread t1 of a line with storage sm1 and sink dst.  A block may
// so read its lines one way (whole segments of a row, say) and write them another
// way (several lines interleaved), each coalesced.  With interleaved lines the
// base-table twiddles of a warp are those of fewer butterflies, so a transform
// without per-pass tables stays interleaved as long as it can.  `sync` covers the
// threads of all the lines.  A transform of a single pass cannot change maps
// (fft_remaps: then t0 = t1, sm0 = sm1).
template <int M, int MAXR = 16> __host__ __device__ constexpr bool fft_remaps() { return radix_of(M, 0, MAXR) < M; }
template <int M, int TPL, bool INV, int MAXR, bool TWT, bool LATE, class Src, class Dst, class SM0, class SM1,
          class SYNC = BlockSync>
__device__ __forceinline__ void fft_line_remap(int t0, const Src& src, const SM0& sm0, int t1, const Dst& dst,
                                               const SM1& sm1, const float2* __restrict__ tw,
                                               const SYNC& sync = SYNC()) {
    constexpr int R = radix_of(M, 0, MAXR);
    static_assert(!Src::kSmem, "a source outside the lines");
    if constexpr (LATE || !fft_remaps<M, MAXR>()) {
        fft_run<M, TPL, INV, MAXR, 0, 1, TWT, SM0::kLines>(t0, src, dst, sm0.p, t1, sm1.p, tw, sync);
    } else {
        stockham_pass<M, R, 1, TPL, INV, TWT, 0>(t0, src, Exchange<M, 0, MAXR, SM0::kLines>{sm0.p}, tw, false, sync);
        sync();
        fft_run<M, TPL, INV, MAXR, 1, R, TWT, SM0::kLines>(t1, src, dst, sm1.p, t1, sm1.p, tw, sync);
    }
}

// The transform of a line whose values thread t already holds in registers,
// x[i] = line[t + i TPL] for i < M / TPL (the order in which a gather fills the
// line).  These are exactly the first pass's inputs of butterflies
// j = t + it TPL: element j + s M/R is x[it + s IT].  So pass 0 runs on them
// directly and only its outputs go to the shared-memory line `sm`; the later
// passes are those of fft_line.  Call with every thread of the block; `sm`
// must be free for writing (the caller's barrier).
// sm1, t1: storage and thread of the later passes, as in fft_line_remap.
template <int M, int TPL, bool INV, int MAXR = 16, class Dst, class SYNC = BlockSync, bool TWT = false, class SM0, class SM1>
__device__ __forceinline__ void fft_line_regs(int t, float2 (&x)[M / TPL], const Dst& dst, const SM0& sm, int t1,
                                              const SM1& sm1, const float2* __restrict__ tw,
                                              const SYNC& sync = SYNC()) {
    constexpr int R = radix_of(M, 0, MAXR);
    constexpr int NB = M / R;
    static_assert(NB % TPL == 0, "one or more whole first-pass butterflies per thread");
    constexpr int IT = NB / TPL;
    if constexpr (R == M) {
        // a single pass: one thread holds the whole line
        Dft<R, INV>::run(x);
#pragma unroll
        for (int s = 0; s < R; ++s)
            if (!dst_drop_group<Dst, M>(s, s + 1)) dst.store(s, x[s]);
        return;
    }
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        float2 a[R];
#pragma unroll
        for (int s = 0; s < R; ++s) a[s] = x[it + s * IT];
        Dft<R, INV>::run(a);
        using Out = Exchange<M, 0, MAXR, SM0::kLines>;
        static_assert(pad_store_step<Out, 1, R>() == 1, "a butterfly's outputs side by side");
        float2* p = sm.p + Out::at((t + it * TPL) * R);
#pragma unroll
        for (int s = 0; s < R; ++s) p[s] = a[s];
    }
    if constexpr (R < M) {
        sync();
        fft_run<M, TPL, INV, MAXR, 1, R, TWT, SM0::kLines>(t1, sm1, dst, sm1.p, t1, sm1.p, tw, sync);
    }
}
template <int M, int TPL, bool INV, int MAXR = 16, class Dst, class SYNC = BlockSync, bool TWT = false, class SM>
__device__ __forceinline__ void fft_line_regs(int t, float2 (&x)[M / TPL], const Dst& dst, const SM& sm,
                                              const float2* __restrict__ tw, const SYNC& sync = SYNC()) {
    fft_line_regs<M, TPL, INV, MAXR, Dst, SYNC, TWT>(t, x, dst, sm, t, sm, tw, sync);
}

// signed frequency of natural-order index p
__device__ __forceinline__ int signed_freq(int p, int M) { return p < (M >> 1) ? p : p - M; }

}  // namespace bst

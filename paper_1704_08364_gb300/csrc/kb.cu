// kb.cu -- Kaiser-Bessel gridding for stage P5: plan tables (kernel polynomial,
// deapodization, per-strip sample lists), the gridding + column-FFT kernel
// and bst_plan_set_gridding.
//
// The paper leaves the interpolation kernel of P5 open.  With KB gridding the
// path computes, up to the gridding error, the polar quadrature of the inverse
// 2D Fourier integral x(u) = sum_{j,k} a_jk exp(2 pi i omega_jk . u) with
// a_jk = dtheta_j dsigma |sigma_k| W[|k|] Y_j[k] (Eq. 3 with the filter of
// P4), where bilinear interpolation in (kappa, theta) loses several digits.
// Kernel shape: beta = pi sqrt((W / alpha)^2 (alpha - 1/2)^2 - 0.8) for the
// grid oversampling alpha = M / N (Beatty, Nishimura and Pauly, 2005).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <new>
#include <vector>

#include "bst_kb.cuh"
#include "bst_parallel.h"

namespace bst {

// P slice pairs per block (blockIdx.y: group of P of the np pairs).
// What bounds it: the latency of the samples' loads at 16 warps an SM (long scoreboard
// leads the stalls) and the L1 wavefronts of these scattered 8-byte reads (66 % of
// the peak with four pairs a block, 59 % with two), before instruction issue (48 and
// 57 %).  With one pair a block, strips of four columns
// and an item a thread, every pair evaluated its own kernel values: 187 us a pair
// at 1024 x 1024 (W = 6), 66 us with four pairs a block.
template <int M, int MAXR, int P>
__global__ void __launch_bounds__(kb_threads<M, P>(), kb_threads<M, P>() > 256 ? 1 : 2)
    k_kb_col(const float2* __restrict__ Z, int np, int V, int N, KbArgs kb, float2* __restrict__ T,
             const float2* __restrict__ tw) {
    extern __shared__ float2 smem[];
    const int pl = blockIdx.y * P;
    // strips nearest the column c' = 0 carry the most samples: start there
    const int b = blockIdx.x;
    const int strip = (b & 1) ? kb.nstrips - 1 - (b >> 1) : (b >> 1);
    const size_t zs = (size_t)V * M, ts = (size_t)((N + 3) / 4) * 4 * M;
    kb_col_unit<M, tpl_of<M>(), MAXR, P>(smem, strip, min(P, np - pl), V, N, Z + pl * zs, zs, kb, T + pl * ts, ts, tw);
}

template <int M, int MAXR, int P>
static bst_status_t launch_kb_col_P(const bst_plan_s* p, const KbArgs& a, const float2* Z, float2* T, int np,
                                    cudaStream_t st) {
    constexpr size_t smem = kb_smem_bytes<M, P>();
    static std::atomic<unsigned long long> attr_done{0};
    if (!bsth::once_per_device(attr_done, [] {
            return cudaFuncSetAttribute(k_kb_col<M, MAXR, P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem) == cudaSuccess;
        }))
        return BST_ERR_CUDA;
    k_kb_col<M, MAXR, P><<<dim3(p->kb_nstrips, (np + P - 1) / P), kb_threads<M, P>(), smem, st>>>(Z, np, p->V, p->N, a,
                                                                                                T, p->tw);
    return BST_OK;
}

// Whole groups of kb_pairs pairs, then what remains in the smallest group that
// holds it.
template <int M, int MAXR>
bst_status_t launch_kb_col_M(bst_plan_s* p, const float2* Z, float2* T, int np, cudaStream_t st) {
    KbArgs a;
    static_assert(sizeof(a.poly) == sizeof(p->kb_poly), "polynomial size");
    for (int i = 0; i <= KB_POLY; ++i) a.poly[i] = p->kb_poly[i];
    a.t_scale = 8.f / (float)(p->kb_w * p->kb_w);
    a.istart = p->kb_start;
    a.items = p->kb_items;
    a.list = p->kb_list;
    a.dir = p->dir;
    a.wq = p->wq;
    a.W = p->kb_w;
    a.nstrips = p->kb_nstrips;
    constexpr int PM = kb_pairs<M>();
    const size_t zs = (size_t)p->V * M, ts = (size_t)((p->N + 3) / 4) * 4 * M;
    const int full = np % PM == 3 ? np : np / PM * PM, rem = np - full;
    bst_status_t s = BST_OK;
    if (full > 0) s = launch_kb_col_P<M, MAXR, PM>(p, a, Z, T, full, st);
    if (s == BST_OK && rem == 1) s = launch_kb_col_P<M, MAXR, 1>(p, a, Z + full * zs, T + full * ts, 1, st);
    if constexpr (PM > 2) {
        if (s == BST_OK && rem == 2) s = launch_kb_col_P<M, MAXR, 2>(p, a, Z + full * zs, T + full * ts, 2, st);
    }
    return s;
}

}  // namespace bst

#define BST_FOR_EACH_M(X) \
    X(16) X(32) X(64) X(128) X(256) X(512) X(1024) X(2048) X(4096) X(48) X(96) X(192) X(384) X(768) X(1536) X(3072)

bst_status_t bst_launch_kb_col(bst_plan_s* p, const float2* Z, float2* T, int np, cudaStream_t st) {
    switch (p->M) {
#define BST_CASE(m)                                                                            \
    case m:                                                                                    \
        return p->maxr == 8 ? bst::launch_kb_col_M<m, 8>(p, Z, T, np, st)                      \
                            : bst::launch_kb_col_M<m, 16>(p, Z, T, np, st);
        BST_FOR_EACH_M(BST_CASE)
#undef BST_CASE
    }
    return BST_ERR_UNSUPPORTED_SIZE;
}

double bst_bessel_i0(double x) {
    double term = 1.0, sum = 1.0;
    const double q = 0.25 * x * x;
    for (int k = 1; k < 500 && term > 1e-18 * sum; ++k) {
        term *= q / ((double)k * (double)k);
        sum += term;
    }
    return sum;
}

void bst_free_kb(bst_plan_s* p) {
    cudaFree(p->kb_dk);
    cudaFree(p->kb_start);
    cudaFree(p->kb_list);
    cudaFree(p->kb_items);
    p->kb_dk = nullptr;
    for (float& c : p->kb_poly) c = 0.f;
    p->kb_start = p->kb_list = nullptr;
    p->kb_items = nullptr;
    p->kb_w = 0;
    p->kb_n = 0;
    p->kb_nstrips = 0;
}

template <class T>
static bool upload_vec(T** d, const std::vector<T>& h) {
    if (cudaMalloc((void**)d, std::max<size_t>(h.size(), 1) * sizeof(T)) != cudaSuccess) return false;
    return h.empty() || cudaMemcpy(*d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice) == cudaSuccess;
}

// Tables of KB gridding of width W for the plan, host-built in double:
//   the kernel polynomial and the deapodization;
//   per strip of two columns, every sample (j, k), k != 0, -M/2, whose
//   footprint (the W columns c' - c_s in (-W/2, W/2]) meets the strip, sorted
//   by the first row of its footprint (r' - r_s > -W/2, taken mod M), then by
//   sample; the samples of the first KB_WMAX rows once more at the end;
//   per band of four rows of the strip, the range of that list whose footprint
//   meets the band, cut into items of at most KB_ITEM entries; a strip's items
//   ordered longest first.
// The strips are divided over host threads.
static bst_status_t build_kb(bst_plan_s* p, int W) {
    using bst::KB_CS;
    using bst::KB_ITEM;
    using bst::KB_RB;
    const int M = p->M, V = p->V, N = p->N;
    const int ns = M / KB_CS, nb = M / KB_RB;
    const double alpha = (double)M / (double)N;
    const double beta = M_PI * std::sqrt((W / alpha) * (W / alpha) * (alpha - 0.5) * (alpha - 0.5) - 0.8);
    const double i0b = bst_bessel_i0(beta);

    // phi(x) = (I0(beta sqrt(1 - (2x/W)^2)) - 1) / (I0(beta) - 1): the KB kernel
    // without its pedestal, zero at |x| = W/2, so that a footprint edge falling
    // exactly on a grid point adds nothing and the gridded spectrum of a real
    // slice stays Hermitian (the pair packing relies on it)
    // evaluated on the GPU as a polynomial of degree KB_POLY in t = 2u - 1,
    // u = (2x/W)^2 in [0, 1] (phi is an entire function of u): interpolation
    // at the Chebyshev nodes of t, then the Chebyshev series rewritten in
    // powers of t (all in double; the monomial coefficients stay below 1 in
    // magnitude, so Horner's rule in float loses only a few ulp)
    constexpr int DMAX = bst::KB_POLY;
    const int D = bst::kb_degree(W);
    double cheb[DMAX + 1] = {0};
    for (int i = 0; i <= D; ++i) {
        const double th = M_PI * (i + 0.5) / (D + 1);
        const double t = std::cos(th);
        const double u = 0.5 * (t + 1.0);
        const double f = (bst_bessel_i0(beta * std::sqrt(std::max(1.0 - u, 0.0))) - 1.0) / (i0b - 1.0);
        for (int k = 0; k <= D; ++k) cheb[k] += f * std::cos(k * th) * (2.0 / (D + 1));
    }
    cheb[0] *= 0.5;
    double mono[DMAX + 1] = {0}, tk[DMAX + 1] = {0}, tkm1[DMAX + 1] = {0};
    tkm1[0] = 1.0;                       // T_0
    tk[1] = 1.0;                         // T_1
    mono[0] += cheb[0];
    mono[1] += cheb[1];
    for (int k = 2; k <= D; ++k) {       // T_k = 2 t T_{k-1} - T_{k-2}
        double nx[DMAX + 1] = {0};
        for (int m = 0; m <= D; ++m) {
            if (m > 0) nx[m] += 2.0 * tk[m - 1];
            nx[m] -= tkm1[m];
        }
        for (int m = 0; m <= D; ++m) {
            tkm1[m] = tk[m];
            tk[m] = nx[m];
            mono[m] += cheb[k] * nx[m];
        }
    }

    // 1 / C(nu), C(nu) = W (sinh(z) / z - sinc(W nu)) / (I0(beta) - 1),
    // z = sqrt(beta^2 - (pi W nu)^2), sinc(x) = sin(pi x) / (pi x)
    std::vector<float> dk(N);
    for (int i = 0; i < N; ++i) {
        const double nu = (double)(i - N / 2) / (double)M;
        const double z2 = beta * beta - (M_PI * W * nu) * (M_PI * W * nu);
        const double z = std::sqrt(std::fabs(z2));
        const double r = z < 1e-8 ? 1.0 : (z2 >= 0 ? std::sinh(z) / z : std::sin(z) / z);
        const double a = M_PI * W * nu;
        const double sn = a == 0.0 ? 1.0 : std::sin(a) / a;
        dk[i] = (float)((i0b - 1.0) / (W * (r - sn)));
    }

    // footprint starts (first column and first row, mod M) of every sample
    std::vector<uint16_t> fc((size_t)V * M), fr((size_t)V * M);
    auto first = [&](double x) {
        const int f = (int)std::floor(x - 0.5 * W) + 1;
        return (uint16_t)(f < 0 ? f + M : (f >= M ? f - M : f));
    };
    bsth::parallel(V, [&](int j0, int j1) {
        for (int j = j0; j < j1; ++j) {
            const double c = std::cos(p->theta[j]), s = std::sin(p->theta[j]);
            for (int i = 0; i < M; ++i) {
                const double k = (double)(i < M / 2 ? i : i - M);
                fc[(size_t)j * M + i] = first(k * c);
                fr[(size_t)j * M + i] = first(k * s);
            }
        }
    });
    // fn(strip, first row, sample) for the samples of strips [s0, s1), ascending by sample
    auto each = [&](int s0, int s1, auto&& fn) {
        for (int j = 0; j < V; ++j)
            for (int i = 1; i < M; ++i) {
                if (i == M / 2) continue;
                const size_t at = (size_t)j * M + i;
                // the strips of columns fc .. fc + W - 1 (mod M), each once
                int s = fc[at] / KB_CS;
                const int n = (fc[at] % KB_CS + W - 1) / KB_CS + 1;
                for (int d = 0; d < n && d < ns; ++d, s = s + 1 == ns ? 0 : s + 1)
                    if (s >= s0 && s < s1) fn(s, (int)fr[at], (int)at);
            }
    };
    // entries per (strip, first row), then the lists
    const int wrap = std::min(bst::KB_WMAX, M);
    std::vector<int> row((size_t)ns * (M + 1), 0);   // row[s][r]: entries of the strip with first row < r
    std::vector<size_t> start(ns + 1, 0);            // the strip's place in the list
    bsth::parallel(ns, [&](int s0, int s1) {
        each(s0, s1, [&](int s, int r, int) { ++row[(size_t)s * (M + 1) + r + 1]; });
        for (int s = s0; s < s1; ++s)
            for (int r = 0; r < M; ++r) row[(size_t)s * (M + 1) + r + 1] += row[(size_t)s * (M + 1) + r];
    });
    for (int s = 0; s < ns; ++s) {
        const int* q = &row[(size_t)s * (M + 1)];
        start[s + 1] = start[s] + q[M] + q[wrap];
    }
    const size_t n = start[ns];
    if (n >= (size_t)INT32_MAX) return BST_ERR_UNSUPPORTED_SIZE;
    // first entry of strip s with first row >= r, rows r >= M being those of the copy
    auto pos = [&](int s, int r) {
        const int* q = &row[(size_t)s * (M + 1)];
        return (int)start[s] + (r < M ? q[r] : q[M] + q[r - M]);
    };
    // the entries [lo, hi) of band b of strip s: first rows [KB_RB b - W + 1, KB_RB b + KB_RB) mod M
    auto band = [&](int s, int b) {
        int lo = KB_RB * b - W + 1, hi = KB_RB * b + KB_RB;
        if (lo < 0) {
            lo += M;
            hi += M;
        }
        return make_int2(pos(s, lo), pos(s, hi));
    };
    std::vector<int> istart(ns + 1, 0);
    for (int s = 0; s < ns; ++s) {
        istart[s + 1] = istart[s];
        for (int b = 0; b < nb; ++b) {
            const int2 e = band(s, b);
            istart[s + 1] += (e.y - e.x + KB_ITEM - 1) / KB_ITEM;
        }
    }
    std::vector<int> list(n), fill((size_t)ns * M);
    std::vector<int4> items(istart[ns]);
    bsth::parallel(ns, [&](int s0, int s1) {
        for (int s = s0; s < s1; ++s)
            for (int r = 0; r < M; ++r) fill[(size_t)s * M + r] = pos(s, r);
        each(s0, s1, [&](int s, int r, int at) { list[fill[(size_t)s * M + r]++] = at; });
        for (int s = s0; s < s1; ++s) {
            const int* q = &row[(size_t)s * (M + 1)];
            std::copy_n(list.begin() + start[s], q[wrap], list.begin() + start[s] + q[M]);
            int4* it = items.data() + istart[s];
            for (int b = 0; b < nb; ++b) {
                const int2 e = band(s, b);
                for (int i = e.x; i < e.y; i += KB_ITEM)
                    *it++ = make_int4(b, i, std::min(e.y, i + KB_ITEM), e.y - e.x > KB_ITEM);
            }
            std::stable_sort(items.begin() + istart[s], items.begin() + istart[s + 1],
                             [](const int4& a, const int4& b) { return a.z - a.y > b.z - b.y; });
        }
    });

    bst_free_kb(p);
    const bool ok = upload_vec(&p->kb_dk, dk) && upload_vec(&p->kb_start, istart) && upload_vec(&p->kb_list, list) && upload_vec(&p->kb_items, items);
    if (!ok) {
        cudaGetLastError();
        bst_free_kb(p);
        return BST_ERR_OUT_OF_MEMORY;
    }
    for (int i = 0; i <= DMAX; ++i) p->kb_poly[i] = i <= D ? (float)mono[i] : 0.f;
    p->kb_w = W;
    p->kb_n = n;
    p->kb_nstrips = ns;
    return BST_OK;
}

extern "C" {

bst_status_t bst_plan_set_gridding(bst_plan_t p, int kind, int width) {
    if (!p) return BST_ERR_INVALID_ARGUMENT;
    if (!bsth::on_plan_device(p)) return BST_ERR_INVALID_ARGUMENT;
    if (kind == BST_GRID_BILINEAR) {
        cudaDeviceSynchronize();
        bst_free_kb(p);
        p->grid_kind = BST_GRID_BILINEAR;
        return BST_OK;
    }
    if (kind != BST_GRID_KAISER_BESSEL || width < 2 || width > bst::KB_WMAX || width % 2 != 0)
        return BST_ERR_INVALID_ARGUMENT;
    if (p->grid_kind == BST_GRID_KAISER_BESSEL && p->kb_w == width) return BST_OK;
    cudaDeviceSynchronize();
    bst_status_t s;
    try {
        s = build_kb(p, width);
    } catch (const std::bad_alloc&) {
        s = BST_ERR_OUT_OF_MEMORY;
    }
    if (s != BST_OK) {
        p->grid_kind = BST_GRID_BILINEAR;
        return s;
    }
    p->grid_kind = BST_GRID_KAISER_BESSEL;
    return BST_OK;
}

bst_status_t bst_plan_get_gridding(bst_plan_t p, int* kind, int* width) {
    if (!p || !kind || !width) return BST_ERR_INVALID_ARGUMENT;
    *kind = p->grid_kind;
    *width = p->grid_kind == BST_GRID_KAISER_BESSEL ? p->kb_w : 2;
    return BST_OK;
}

}  // extern "C"

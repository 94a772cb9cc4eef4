// Test-only translation unit (compiled by tests/test_kernel_resources_default.py,
// never linked): the kernels that plans use as they are created, at the lengths of
// the 2048^3 and 512^3 workloads and, for Kaiser-Bessel gridding, both group sizes.
#include "bst_inter.cuh"
#include "bst_kb.cuh"

#define INTER(M, N)                                                                                                    \
    template __global__ void bst::k_ray_inter<M, 16, N, false>(const float*, int, int, int, int, bst::PrepArgs, int,  \
                                                                const float*, float, float2*, const float2*);         \
    template __global__ void bst::k_ray_inter<M, 16, N, true>(const float*, int, int, int, int, bst::PrepArgs, int,   \
                                                               const float*, float, float2*, const float2*);          \
    template __global__ void bst::k_grid_inter<M, 16, N>(const float2*, int, int, const int*, const float2*, float2*, \
                                                          const float2*, int);                                        \
    template __global__ void bst::k_row_inter<M, 16, N>(const float2*, int, int, int, float, float*, const float2*);
INTER(4096, 2048)
INTER(3072, 1536)
INTER(1024, 512)

// kb_col_unit with the launch bounds of its kernel
template <int M, int P>
__global__ void __launch_bounds__(bst::kb_threads<M, P>(), bst::kb_threads<M, P>() > 256 ? 1 : 2)
    kb_unit(const float2* __restrict__ Z, int np, int V, int N, bst::KbArgs kb, float2* __restrict__ T,
            const float2* __restrict__ tw) {
    extern __shared__ float2 smem[];
    bst::kb_col_unit<M, bst::tpl_of<M>(), 16, P>(smem, blockIdx.x, np, V, N, Z, (size_t)V * M, kb, T, (size_t)N * M, tw);
}
template __global__ void kb_unit<4096, 2>(const float2*, int, int, int, bst::KbArgs, float2*, const float2*);
template __global__ void kb_unit<2048, 4>(const float2*, int, int, int, bst::KbArgs, float2*, const float2*);

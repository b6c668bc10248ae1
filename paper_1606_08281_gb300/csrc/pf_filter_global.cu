// The filter kernel with populations in global memory.
#include "pf_filter.cuh"

namespace pf {
namespace {

using namespace dev;

// Populations too large for shared memory: a grid of resident blocks walks
// the filters (grid stride), each block keeping its population in its own slab
// of global memory (N (16 + 8U) bytes), which stays in L1/L2 while it runs.
template <int RM, int UM>
__global__ void __launch_bounds__(kMaxThreads, kMinBlocks<RM, kMaxThreads>)
filter_kernel_global(const __grid_constant__ FilterArgs args, unsigned char *slabs, size_t slab_bytes) {
    load_head(args);
    unsigned char *arrays = slabs + static_cast<size_t>(blockIdx.x) * slab_bytes;
    const int64_t F = args.M * args.T;
    for (int64_t slot = blockIdx.x; slot < F; slot += gridDim.x) {
        __syncthreads();
        run_filter<RM, UM>(filter_job(args, slot), block_head(), ParamKeys{args.round_keys}, args.fast != 0, arrays);
    }
}

template <int RM, int UM>
int launch_tier_global(const FilterArgs &a, int B, unsigned char *slabs, size_t slab_bytes,
                       int grid, cudaStream_t s) {
    const cudaError_t e = static_cast<cudaError_t>(
        raise_smem_limit(reinterpret_cast<const void *>(filter_kernel_global<RM, UM>)));
    if (e != cudaSuccess) return e;
    filter_kernel_global<RM, UM><<<grid, B, kHeadBytes + a.fast, s>>>(a, slabs, slab_bytes);
    return cudaGetLastError();
}

}  // namespace

int launch_filter_global(const FilterArgs &a, int B, unsigned char *slabs, size_t slab_bytes, int grid,
                         cudaStream_t s) {
    const bool small_u = a.net.U <= 4, tiny_u = a.net.U <= 2;
    switch (reaction_tier(a.net.R)) {
        case 4: return tiny_u ? launch_tier_global<4, 2>(a, B, slabs, slab_bytes, grid, s) : small_u ? launch_tier_global<4, 4>(a, B, slabs, slab_bytes, grid, s) : launch_tier_global<4, 0>(a, B, slabs, slab_bytes, grid, s);
        case 8: return small_u ? launch_tier_global<8, 4>(a, B, slabs, slab_bytes, grid, s) : launch_tier_global<8, 0>(a, B, slabs, slab_bytes, grid, s);
        case 16: return launch_tier_global<16, 0>(a, B, slabs, slab_bytes, grid, s);
        default: return launch_tier_global<32, 0>(a, B, slabs, slab_bytes, grid, s);
    }
}

}  // namespace pf

// The filter kernel over thread-block clusters (pf_filter.cuh, run_filter_cluster).
#include "pf_filter.cuh"

namespace pf {
namespace {

using namespace dev;

// A filter split over the C blocks of a thread-block cluster (cluster size
// set at launch): cluster c runs filter slot c, its blocks on C SMs.
template <int RM, int UM, int MT>
__global__ void __launch_bounds__(MT, kMinBlocks<RM, MT>) filter_kernel_cluster(const __grid_constant__ FilterArgs args) {
    load_head(args);
    __syncthreads();
    const FilterJob job = filter_job(args, blockIdx.x / cooperative_groups::this_cluster().num_blocks());
    run_filter_cluster<RM, UM>(job, block_head(), ParamKeys{args.round_keys}, args.fast != 0,
                               g_smem + kHeadBytes + args.fast);
}

// The instance for B threads: small networks have one for blocks of up to 128.
template <int RM, int UM>
auto cluster_instance(int B) {
    if constexpr (RM <= 8) return B <= 128 ? filter_kernel_cluster<RM, UM, 128> : filter_kernel_cluster<RM, UM, kMaxThreads>;
    else return filter_kernel_cluster<RM, UM, kMaxThreads>;
}

template <int RM, int UM>
int launch_tier_cluster(const FilterArgs &a, int B, size_t smem, int C, cudaStream_t s) {
    const auto kernel = cluster_instance<RM, UM>(B);
    cudaError_t e = static_cast<cudaError_t>(raise_smem_limit(reinterpret_cast<const void *>(kernel)));
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(a.M * a.T * C));
    cfg.blockDim = dim3(static_cast<unsigned>(B));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(C);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel, a);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace

int launch_filter_cluster(const FilterArgs &a, int B, size_t smem, cudaStream_t s) {
    const bool small_u = a.net.U <= 4, tiny_u = a.net.U <= 2;
    switch (reaction_tier(a.net.R)) {
        case 4: return tiny_u ? launch_tier_cluster<4, 2>(a, B, smem, a.cluster, s) : small_u ? launch_tier_cluster<4, 4>(a, B, smem, a.cluster, s) : launch_tier_cluster<4, 0>(a, B, smem, a.cluster, s);
        case 8: return small_u ? launch_tier_cluster<8, 4>(a, B, smem, a.cluster, s) : launch_tier_cluster<8, 0>(a, B, smem, a.cluster, s);
        case 16: return launch_tier_cluster<16, 0>(a, B, smem, a.cluster, s);
        default: return launch_tier_cluster<32, 0>(a, B, smem, a.cluster, s);
    }
}

}  // namespace pf

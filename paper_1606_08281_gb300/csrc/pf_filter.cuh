// What the filter kernels' translation units share (one unit per launch form, so
// that they compile in parallel).
#pragma once
#include "pf_device.cuh"

namespace pf {
namespace dev {

// Resident blocks the register allocation aims at.  Blocks of up to 128 threads
// (populations below 512, where the chain of one particle's events sets the
// time): 4, with 128 registers and no spills.  Blocks of 256 (where issue does):
// small networks 3 with 80 registers (gene expression 1000 x 1000: 164 ms; 2
// blocks 189), the others 2 (cascade 153 ms; 3 blocks 160; 128 threads 217).
template <int RM, int MT>
constexpr int kMinBlocks = MT == 128 ? 4 : RM <= 8 ? 3 : 2;

// Filter `slot` of the launch: its job, from the launch's arguments.
__device__ __forceinline__ FilterJob filter_job(const FilterArgs &args, int64_t slot) {
    const int T = args.T;
    int64_t mrow = slot / T;
    const int traj = static_cast<int>(slot - mrow * T);
    if (args.row_order) mrow = args.row_order[mrow];
    const int64_t f = mrow * T + traj;
    FilterJob job;
    job.theta = args.thetas + mrow * args.net.d;
    job.obs_times = args.obs_times;
    job.y = args.y + static_cast<int64_t>(traj) * args.K * args.net.P;
    job.K = args.K;
    job.N = args.N;
    job.mrow = args.theta_ids ? args.theta_ids[mrow] : static_cast<uint32_t>(mrow);
    job.traj = traj;
    job.seed = args.seed;
    job.budget = args.budget;
    job.ll_out = args.ll_f + f;
    job.st_out = args.st_f + f;
    job.ev_out = reinterpret_cast<unsigned long long *>(args.ev_f) + f;
    job.dg_out = args.dg_f ? reinterpret_cast<unsigned long long *>(args.dg_f) + f : nullptr;
    job.fs_out = args.final_states ? args.final_states + f * static_cast<int64_t>(args.N) * args.net.U
                                   : nullptr;
    job.ph_out = args.phase_f ? reinterpret_cast<unsigned long long *>(args.phase_f) + 3 * f : nullptr;
    job.acc = args.acc ? args.acc + mrow : nullptr;
    job.reject_below = args.reject_below;
    job.slack = args.slack;
    return job;
}

// A block's head: network tables and ziggurat (the caller synchronises).
__device__ __forceinline__ void load_head(const FilterArgs &args) {
    SharedHead &sh = block_head();
    const uint32_t *src = reinterpret_cast<const uint32_t *>(&args.net);
    uint32_t *dst = reinterpret_cast<uint32_t *>(&sh.net);
    for (int i = threadIdx.x; i < static_cast<int>(sizeof(NetTables) / 4); i += blockDim.x) dst[i] = src[i];
    if (args.fast) load_fast_zig(args.zig);
    if (threadIdx.x == 0) sh.zig_g = args.zig;
}

}  // namespace dev
}  // namespace pf

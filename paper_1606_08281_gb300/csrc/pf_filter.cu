// Particle-filter kernels for sm_103a.
//
// One thread block runs one filter, i.e. one (theta row, observed trajectory)
// pair, through all K observation times (Supp. I, algorithm "Likelihood
// Approximation using particle filter"); on request the filter is split over
// the blocks of a thread-block cluster instead (filter_kernel_cluster):
//   resample by the previous weights -> simulate every particle to t_k with
//   the direct-method SSA -> Gaussian weight -> log-sum-exp increment.
// (run_filter in pf_device.cuh).
//
// Arithmetic that decides integer outcomes (propensities, their prefix sums,
// event times, the Gaussian exponent) uses explicit round-to-nearest
// intrinsics so that the compiler cannot fuse a multiply and an add; the
// results then match a plain sequential FP64 restatement bit for bit, except
// where CUDA's log/exp differ from another libm in the last place.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <utility>
#include <vector>

#include "pf_filter.cuh"

namespace pf {
namespace {

using namespace dev;

template <int RM, int UM, int MT>
__global__ void __launch_bounds__(MT, kMinBlocks<RM, MT>) filter_kernel(const __grid_constant__ FilterArgs args) {
    load_head(args);
    __syncthreads();
    run_filter<RM, UM>(filter_job(args, blockIdx.x), block_head(), ParamKeys{args.round_keys}, args.fast != 0,
                       g_smem + kHeadBytes + args.fast);
}

// loglik[m] = sum over trajectories (in order) of the filter estimates (Supp. I).
__global__ void reduce_kernel(const double *ll_f, const uint8_t *st_f, int64_t M, int T,
                              double *loglik, uint8_t *status) {
    const int64_t m = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (m >= M) return;
    double sum = 0.0;
    int st = PF_ST_OK;
    for (int t = 0; t < T; ++t) {
        const int s = st_f[m * T + t];
        if (st == PF_ST_OK && s != PF_ST_OK) st = s;
        sum = __dadd_rn(sum, ll_f[m * T + t]);
    }
    double out = sum;
    if (st == PF_ST_INVALID_THETA) out = __longlong_as_double(0x7FF8000000000000ll);
    else if (st != PF_ST_OK) out = -INFINITY;
    loglik[m] = out;
    if (status) status[m] = static_cast<uint8_t>(st);
}

// One unconditioned direct-method path per theta row over [0, t_K], counting
// events (at most `cap`): a cost estimate for scheduling only.  Its random
// stream (particle lane 0xFFFFFFFE, interval word 0xFFFFFFFF) is disjoint from
// the filters' streams.
template <int RM>
__global__ void __launch_bounds__(128) pilot_kernel(const FilterArgs args, uint32_t *cost,
                                                    uint32_t cap) {
    __shared__ NetTables net;
    __shared__ LogTab logt;
    {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(&args.net);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&net);
        for (int i = threadIdx.x; i < static_cast<int>(sizeof(NetTables) / 4); i += blockDim.x)
            dst[i] = src[i];
    }
    load_log_table(logt);
    __syncthreads();
    const int64_t m = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (m >= args.M) return;
    const int R = net.R, U = net.U, d = net.d;
    const double *theta = args.thetas + m * d;
    bool ok = true;
    for (int c = 0; c < d; ++c) ok = ok && isfinite(theta[c]) && theta[c] >= 0.0;
    if (!ok) {
        cost[m] = 0;
        return;
    }
    double rate[RM];
#pragma unroll
    for (int r = 0; r < RM; ++r) rate[r] = r < R ? reaction_rate(net, theta, r) : 0.0;
    int x[PF_MAX_SPECIES];
    for (int u = 0; u < PF_MAX_SPECIES; ++u) x[u] = u < U ? net.x0[u] : 0;
    const uint32_t key0 = static_cast<uint32_t>(args.seed);
    const uint32_t key1 = static_cast<uint32_t>(args.seed >> 32);
    const long long t_end_bits = __double_as_longlong(args.obs_times[args.K - 1]);
    double t = 0.0;
    uint32_t events = 0;
    while (events < cap) {
        double a[RM], S[RM], run = 0.0;
#pragma unroll
        for (int r = 0; r < RM; ++r) {
            long long h = 1;
            if (r < R) {
                if (net.sp_a[r] >= 0) h = binom_small(x[net.sp_a[r]], net.ord_a[r]);
                if (net.sp_b[r] >= 0) h *= binom_small(x[net.sp_b[r]], net.ord_b[r]);
            }
            a[r] = r < R ? __dmul_rn(rate[r], count_to_double(h)) : 0.0;
            run = r == 0 ? a[0] : __dadd_rn(run, a[r]);
            S[r] = run;
        }
        if (__double_as_longlong(run) == 0) break;
        const Philox4 w = philox4x32_10(events, 0xFFFFFFFEu, 0xFFFFFFFFu, static_cast<uint32_t>(m),
                                        key0, key1);
        const uint64_t r0 = (static_cast<uint64_t>(w.w1) << 32) | w.w0;
        const uint64_t v2 = ((static_cast<uint64_t>(w.w3) << 32) | w.w2) >> 11;
        t = __dadd_rn(t, __ddiv_rn(neg_log_u53((r0 >> 11) + 1ull, logt), run));
        if (__double_as_longlong(t) > t_end_bits) break;
        const long long tb = __double_as_longlong(__dmul_rn(scaled_u53_or_zero(v2), run));
        int chosen = 0;
#pragma unroll
        for (int r = 0; r < RM; ++r) chosen += (r < R && __double_as_longlong(S[r]) <= tb) ? 1 : 0;
        if (chosen >= R) {
            chosen = 0;
#pragma unroll
            for (int r = 0; r < RM; ++r)
                if (r < R && __double_as_longlong(a[r]) != 0) chosen = r;
        }
        for (int i = 0; i < net.n_change[chosen]; ++i) x[net.ch_sp[chosen][i]] += net.ch_delta[chosen][i];
        ++events;
    }
    cost[m] = events;
}

// Expected events of every theta row by the mean-field equations from x0 (FP32,
// kMeanSteps steps to t_K; losses are taken implicitly, so that a stiff row
// stays bounded): a cost estimate for scheduling only.  One thread per row,
// about 20 us for four reactions.
constexpr int kMeanSteps = 64;
__global__ void __launch_bounds__(128) mean_field_kernel(const FilterArgs args, uint32_t *cost) {
    __shared__ NetTables net;
    {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(&args.net);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&net);
        for (int i = threadIdx.x; i < static_cast<int>(sizeof(NetTables) / 4); i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    const int64_t m = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (m >= args.M) return;
    const int R = net.R, U = net.U;
    float rate[PF_MAX_REACTIONS], x[PF_MAX_SPECIES], gain[PF_MAX_SPECIES], loss[PF_MAX_SPECIES];
    for (int r = 0; r < R; ++r) rate[r] = static_cast<float>(reaction_rate(net, args.thetas + m * net.d, r));
    for (int u = 0; u < U; ++u) x[u] = 0.5f * (static_cast<float>(net.x0[u]) + static_cast<float>(net.x0_hi[u]));
    const float dt = static_cast<float>(args.obs_times[args.K - 1]) / kMeanSteps;
    float events = 0.0f;
    for (int s = 0; s < kMeanSteps; ++s) {
        for (int u = 0; u < U; ++u) gain[u] = loss[u] = 0.0f;
        for (int r = 0; r < R; ++r) {
            const int sa = net.sp_a[r], sb = net.sp_b[r];
            float a = rate[r];
            if (sa >= 0) a *= net.ord_a[r] == 2 ? 0.5f * x[sa] * x[sa] : x[sa];
            if (sb >= 0) a *= x[sb];
            events += a * dt;
            for (int i = 0; i < net.n_change[r]; ++i) {
                const int u = net.ch_sp[r][i];
                const float c = a * static_cast<float>(net.ch_delta[r][i]);
                if (c > 0.0f) gain[u] += c;
                else loss[u] -= c;
            }
        }
        for (int u = 0; u < U; ++u) x[u] = (x[u] + dt * gain[u]) / (1.0f + dt * loss[u] / fmaxf(x[u], 1e-3f));
    }
    // invalid rows and overflows order anywhere
    cost[m] = events >= 0.0f && events < 4e9f ? static_cast<uint32_t>(events) : 0xFFFFFFFFu;
}

// Counting sort of theta rows by estimated cost, heaviest first (4 buckets per
// octave).  One block.
__global__ void __launch_bounds__(1024) order_kernel(const uint32_t *cost, int64_t M,
                                                      uint32_t *order) {
    constexpr int kOrder = 128;
    __shared__ int hist[kOrder];
    auto bucket = [](uint32_t c) {
        const int lg = c == 0 ? 0 : static_cast<int>(4.0f * __log2f(static_cast<float>(c)));
        return kOrder - 1 - min(kOrder - 1, max(0, lg));
    };
    if (threadIdx.x < kOrder) hist[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t m = threadIdx.x; m < M; m += blockDim.x) atomicAdd(&hist[bucket(cost[m])], 1);
    __syncthreads();
    if (threadIdx.x < 32) {                   // exclusive sums, four buckets a lane
        int c[4], own = 0;
        for (int i = 0; i < 4; ++i) {
            c[i] = hist[4 * threadIdx.x + i];
            own += c[i];
        }
        int run = own;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kFull, run, o);
            if (static_cast<int>(threadIdx.x) >= o) run += v;
        }
        run -= own;
        for (int i = 0; i < 4; ++i) {
            hist[4 * threadIdx.x + i] = run;
            run += c[i];
        }
    }
    __syncthreads();
    for (int64_t m = threadIdx.x; m < M; m += blockDim.x)
        order[atomicAdd(&hist[bucket(cost[m])], 1)] = static_cast<uint32_t>(m);
}

__global__ void fill_kernel(double *p, int64_t n, double v) {
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        p[i] = v;
}

__global__ void philox_kernel(const uint32_t *ctr, const uint32_t *key, uint32_t *out, int64_t n) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Philox4 w = philox4x32_10(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3],
                                    key[2 * i], key[2 * i + 1]);
    out[4 * i] = w.w0;
    out[4 * i + 1] = w.w1;
    out[4 * i + 2] = w.w2;
    out[4 * i + 3] = w.w3;
}

// The instance for B threads: small networks have one for blocks of up to 128.
template <int RM, int UM>
auto filter_instance(int B) {
    if constexpr (RM <= 8) return B <= 128 ? filter_kernel<RM, UM, 128> : filter_kernel<RM, UM, kMaxThreads>;
    else return filter_kernel<RM, UM, kMaxThreads>;
}
template <int RM, int UM>
int launch_tier(const FilterArgs &a, int B, size_t smem, cudaStream_t s) {
    const auto kernel = filter_instance<RM, UM>(B);
    cudaError_t e = static_cast<cudaError_t>(raise_smem_limit(reinterpret_cast<const void *>(kernel)));
    if (e != cudaSuccess) return e;
    const int64_t F = a.M * a.T;
    kernel<<<static_cast<unsigned>(F), B, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

static int launch_filter_plain(const FilterArgs &a, int B, size_t smem, cudaStream_t s) {
    const bool small_u = a.net.U <= 4, tiny_u = a.net.U <= 2;
    switch (reaction_tier(a.net.R)) {
        case 4: return tiny_u ? launch_tier<4, 2>(a, B, smem, s) : small_u ? launch_tier<4, 4>(a, B, smem, s) : launch_tier<4, 0>(a, B, smem, s);
        case 8: return small_u ? launch_tier<8, 4>(a, B, smem, s) : launch_tier<8, 0>(a, B, smem, s);
        case 16: return launch_tier<16, 0>(a, B, smem, s);
        default: return launch_tier<32, 0>(a, B, smem, s);
    }
}

// The dynamic shared-memory limit of a kernel is a process-wide attribute.
// It is raised once per kernel and device to the largest size a launch of it
// can use (the device's opt-in maximum less the kernel's static shared
// memory) and never lowered, so concurrent callers with different
// populations cannot change it under each other's launches.
int raise_smem_limit(const void *kernel) {
    static std::mutex mu;
    static std::vector<std::pair<const void *, int>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    for (const auto &kd : done)
        if (kd.first == kernel && kd.second == dev) return cudaSuccess;
    int optin = 0;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             optin - static_cast<int>(fa.sharedSizeBytes));
    if (e != cudaSuccess) return e;
    done.emplace_back(kernel, dev);
    return cudaSuccess;
}

size_t cluster_smem_bytes(int N, int C, int U, bool digest) {
    return cluster_share_bytes(N, C, U, digest);
}

size_t filter_smem_bytes(int N, int U, bool digest) {
    return static_cast<size_t>(N) * (8 + 4 * static_cast<size_t>(U) + 4 + (digest ? 4 : 0)) + 16;
}

int reaction_tier(int R) {
    if (R <= 4) return 4;
    if (R <= 8) return 8;
    if (R <= 16) return 16;
    return 32;
}

int global_grid(int sms) { return sms * 2; }

size_t filter_static_smem() { return 30104; }

// Bytes of the fast path's tables and columns ahead of `population` bytes of
// dynamic shared memory, or 0 when both do not fit a block together.
int fast_smem(int U, int B, size_t population) {
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return 0;
    const size_t f = fast_smem_bytes(U, B);
    return kHeadBytes + f + population + 512 <= static_cast<size_t>(optin) ? static_cast<int>(f) : 0;
}

int launch_filter(const FilterArgs &args, int B, double *loglik, uint8_t *status, void *stream,
                  unsigned char *slabs, size_t slab_bytes, int grid) {
    if (args.M == 0) return cudaSuccess;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    FilterArgs a = args;
    size_t smem = filter_smem_bytes(a.N, a.net.U, a.dg_f != nullptr);
    if (a.cluster > 1) smem = cluster_smem_bytes(a.N, a.cluster, a.net.U, a.dg_f != nullptr);
    a.fast = fast_smem(a.net.U, B, slabs ? 0 : smem);
    for (uint32_t i = 0; i < 10; ++i) {
        a.round_keys[i] = static_cast<uint32_t>(a.seed) + i * 0x9E3779B9u;
        a.round_keys[10 + i] = static_cast<uint32_t>(a.seed >> 32) + i * 0xBB67AE85u;
    }
    smem += kHeadBytes + a.fast;
    const int e = slabs ? launch_filter_global(a, B, slabs, slab_bytes, grid, s)
                  : a.cluster > 1 ? launch_filter_cluster(a, B, smem, s)
                                  : launch_filter_plain(a, B, smem, s);
    if (e != cudaSuccess) return e;
    const int rb = 128;
    reduce_kernel<<<static_cast<unsigned>((a.M + rb - 1) / rb), rb, 0, s>>>(a.ll_f, a.st_f, a.M,
                                                                           a.T, loglik, status);
    return cudaGetLastError();
}

int launch_schedule(const FilterArgs &a, uint32_t *cost, uint32_t *order, uint32_t cap,
                    void *stream) {
    if (a.M == 0) return cudaSuccess;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const unsigned g = static_cast<unsigned>((a.M + 127) / 128);
    if (cap == 0) mean_field_kernel<<<g, 128, 0, s>>>(a, cost);
    else switch (reaction_tier(a.net.R)) {
        case 4: pilot_kernel<4><<<g, 128, 0, s>>>(a, cost, cap); break;
        case 8: pilot_kernel<8><<<g, 128, 0, s>>>(a, cost, cap); break;
        case 16: pilot_kernel<16><<<g, 128, 0, s>>>(a, cost, cap); break;
        default: pilot_kernel<32><<<g, 128, 0, s>>>(a, cost, cap); break;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    order_kernel<<<1, 1024, 0, s>>>(cost, a.M, order);
    return cudaGetLastError();
}

static __device__ ZigTab g_zig_table;

// The ziggurat table, written from its recurrence with the host C library's
// exp and log (x_1 = r, x_{i+1} = -log(v / x_i + exp(-x_i)), x_2048 = 0,
// x_0 = v / exp(-r), f_i = exp(-x_i)), and each wedge's bounding lines.
static void build_zig_table(ZigTab &t) {
    t.x[0] = kZigV / std::exp(-kZigR);
    t.x[1] = kZigR;
    for (int i = 1; i < kZigLayers - 1; ++i) t.x[i + 1] = -std::log(kZigV / t.x[i] + std::exp(-t.x[i]));
    t.x[kZigLayers] = 0.0;
    for (int i = 0; i < kZigLayers; ++i) {
        const double f = std::exp(-t.x[i]), f1 = std::exp(-t.x[i + 1]);
        const double m = std::ldexp(f1, -48);
        ZigLayer &L = t.layer[i];
        L.f = f;
        L.df = f1 - f;
        L.lo = f - m;
        L.hi = f + m;
        L.slope = i == 0 ? 0.0 : L.df / (t.x[i] - t.x[i + 1]);
    }
    for (int i = 0; i < kExpTable; ++i)
        t.exp_t[i] = static_cast<uint64_t>(std::ldexp(std::exp(-i * 0.693147180559945309417232121458176568L / kExpTable), 63) + 0.5L);
    for (int i = 0; i < kZigLayers; ++i) {
        const float hi = static_cast<float>(t.x[i]);
        t.fast_hi[i] = std::ldexp(hi, -24);
        const float lo = std::ldexp(static_cast<float>(t.x[i] - static_cast<double>(hi)), -24);
        uint32_t lo_bits;
        memcpy(&lo_bits, &lo, 4);
        lo_bits = (lo_bits + 0x8000u) & 0xFFFF0000u;      // to 16 bits (2^-8 of it)
        t.wedge[i] = static_cast<float>(1.0 / std::expm1(t.x[i] - t.x[i + 1]));
        // the product is monotone in u, so the test of the largest u with these
        // upper 16 bits decides for all of them
        int n = static_cast<int>(t.x[i + 1] / t.x[i] * 65536.0) + 1;
        auto passes = [&](int top) {
            const uint64_t uv = (static_cast<uint64_t>(top) << 37) - 1;
            return std::ldexp(static_cast<double>(uv), -53) * t.x[i] < t.x[i + 1];
        };
        while (n > 0 && !passes(n)) --n;
        t.fast_lo[i] = lo_bits | static_cast<uint32_t>(std::max(0, std::min(n, 65536) - 16));
    }
}

const ZigTab *zig_table_device(int *err) {
    static std::mutex mu;
    static const ZigTab *addr[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess && (dev < 0 || dev >= 64)) e = cudaErrorInvalidDevice;
    if (e != cudaSuccess) {
        *err = e;
        return nullptr;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        ZigTab host;
        build_zig_table(host);
        void *p = nullptr;
        e = cudaMemcpyToSymbol(g_zig_table, &host, sizeof(ZigTab));
        if (e == cudaSuccess) e = cudaGetSymbolAddress(&p, g_zig_table);
        if (e != cudaSuccess) {
            *err = e;
            return nullptr;
        }
        addr[dev] = static_cast<const ZigTab *>(p);
    }
    *err = cudaSuccess;
    return addr[dev];
}

int launch_fill(double *p, int64_t n, double value, void *stream) {
    if (n == 0) return cudaSuccess;
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, 4096);
    fill_kernel<<<static_cast<unsigned>(blocks), 256, 0, static_cast<cudaStream_t>(stream)>>>(p, n, value);
    return cudaGetLastError();
}

double increment_slack(const NetTables &t) {
    double lognorm = 0.0;
    for (int p = 0; p < t.P; ++p) lognorm += std::log(t.sigma[p]);
    lognorm += 0.5 * t.P * std::log(2.0 * M_PI);
    // a positive bound is enlarged by a relative 1e-9 so that it stays an upper
    // bound whatever the last-place differences of the device's logarithm
    return lognorm >= 0.0 ? 0.0 : -lognorm * (1.0 + 1e-9);
}

int launch_philox(const uint32_t *ctr, const uint32_t *key, uint32_t *out, int64_t n,
                  void *stream) {
    if (n == 0) return cudaSuccess;
    philox_kernel<<<static_cast<unsigned>((n + 127) / 128), 128, 0,
                    static_cast<cudaStream_t>(stream)>>>(ctr, key, out, n);
    return cudaGetLastError();
}

}  // namespace pf

// The direct-method SSA without FP64 arithmetic, with the same outcome.
//
// What the filter keeps of a simulated interval is integers: each particle's
// counts at t_end and how many draws it took.  They follow from three
// decisions per draw -- which ziggurat branch the waiting time takes, which
// reaction fires, whether the event falls before t_end -- defined by FP64
// arithmetic (ssa_interval in pf_device.cuh).  GB300 executes FP64 at 2 lanes
// per clock and SM, 1/64 of its integer and FP32 rate, so this path takes
// every decision from integer and FP32 arithmetic whose error is bounded, and
// hands the decisions that the bound leaves open to the FP64 definition:
//
//   * propensities are 64-bit integers in units of 2^-k: a_r = A_r h_r(x) with
//     A_r = RN(rate_r 2^k), so the prefix sums are exact and cost two integer
//     multiply-adds per reaction.  k is chosen per filter and interval so that
//     the sum stays below 2^62 while every count stays below a cap (four times
//     the largest count in the population, plus room); a particle that leaves
//     the caps is handed over (below).  A_r >= 2^30 is within 2^-31 of the
//     rate; smaller ones contribute at most h_r / 2 units, bounded by e_abs.
//   * the waiting time's variate is u x_i (ziggurat layer i) in two-float
//     arithmetic from 48 bits of u >= 2^-12 and x_i to 2^-32; draws whose layer
//     test w1 < T_i (an integer threshold, a lower bound of the FP64 test) does
//     not accept, 0.4 % of them, take the wedge tests in FP32, and the FP64
//     ziggurat where those are too close (0.03 %).
//   * tau = E / a0 from the approximate reciprocal of a0's 24 leading bits,
//     corrected to all of its 32 leading bits; relative error below
//     2^-31 (rates) + 2^-31 (a0 truncated) + 2^-36 (u) + 2^-42 (reciprocal,
//     products) + 2^-32 (x_i) < 2^-29.8.  Times are 64-bit integers with the interval scaled
//     to [2^49, 2^50) units, so sums add one unit of rounding per event.
//   * an event at t is in time when t < D - b and late when t > D + b, with
//     D the interval's length and b = 2^-28 D + (c units per draw) + the
//     e_abs contribution accumulated along the path; c covers this path's
//     rounding and the FP64 definition's own (2^-53 t_end per event).
//     Otherwise the particle is replayed from its state at the interval's
//     start by ssa_interval (about 1 in 10^8 events).
//   * the reaction is the number of prefix sums at or below u2 a0, compared on
//     31 leading bits; closer than a margin above all errors (16 units, or 2^14
//     when e_abs > 0), this one choice is recomputed in FP64 (exact_step).
//
// So states, draw counts and event counts equal the FP64 definition's, bit for
// bit.  What bounds the path is instruction issue (64 % of the cycles with 24
// warps per SM) and, for few filters, the latency of one event's chain, about
// 1500 cycles: gene expression (1024 rows x 10 x 1000 particles x 50 times)
// 373-417 ms by the FP64 path, 161 ms; the cascade (64 x 16 x 512 x 60, 20
// reactions) 561-597 ms and 125 ms.
//
// Each lane simulates its particle in a private column of shared memory
// (conflict-free, whatever the particle's index, and the same for populations
// in global memory); the population keeps the particle's starting state until
// it has finished, which is what a replay starts from.
#pragma once
#include "fastmath.cuh"
#include "philox.cuh"
#include "ziggurat.cuh"

namespace pf {
namespace dev {

// Largest block of the filter kernels.
constexpr int kMaxThreads = 256;
// A warp parks at most kParkLanes - 1 particles a round.
static_assert(kMaxThreads / 32 * (kParkLanes - 1) <= kMaxRemnants, "the parked particles' lists are too short");
constexpr int kCheckTrips = 32;    // trips between two looks at the counts' caps

// One reaction: A_r and the byte offsets of its reactants' rows in a column.
// Row U of every column holds 1, so h = x_a for orders 0 and 1; otherwise
// h = x_a (x_b - same) >> same (same = 1 for X + X).
struct FastReac {
    uint32_t lo, hi, a, b;     // b: offset << 1 | same
};

struct __align__(16) FastShared {
    float2 zx[kZigLayers];               // x_i 2^-24; trailing part in 16 bits | layer test in 16 bits
    FastReac reac[PF_MAX_REACTIONS];
    uint4 change[PF_MAX_REACTIONS];      // up to four words: row offset << 16 | delta
    int mx[PF_MAX_SPECIES];              // the population's largest counts
    int lim[PF_MAX_SPECIES];             // a count above leaves the caps within kCheckTrips events
    unsigned long long D;                // interval length in time units
    unsigned long long b0;               // b without its per-draw and e_abs parts
    double unit;                         // time units per unit of time (a power of two)
    uint32_t quick_lo, quick_hi;         // times' bits from 2^30 on that decide most events
    uint32_t c;                          // units per draw in b
    uint32_t hi_min;                     // a0's upper word below this: exact_step
    uint32_t margin;                     // reaction choice
    uint32_t scale;                      // exponent bits of the time scale
    float ecoef;                         // e_abs in the units the path's bound needs
    float rate_up[PF_MAX_REACTIONS];     // rates rounded up (0: a rate outside 2^-80 .. 2^80 and not 0)
    uint32_t mask2;                      // reactions of order 2
    int gain;                            // largest count a reaction adds
    int possible;                        // the network's part of the conditions
    int on;                              // this interval runs here
    int n_exact;                         // particles to replay
    uint16_t rem_slot[2][kMaxRemnants];  // parked particles' columns
    float rem_err[2][kMaxRemnants];      // and accumulated bounds
};

// Dynamic shared memory of a filter block: the block's head; then, where this
// path runs, its tables and U + 1 rows of one column per thread; then the
// population (unless it is in global memory).  The parts are reached through
// these functions so that code called out of line still addresses them as
// shared memory.
constexpr size_t kHeadBytes = (sizeof(SharedHead) + 15) & ~static_cast<size_t>(15);
__host__ __device__ __forceinline__ size_t fast_smem_bytes(int U, int threads) {
    return (sizeof(FastShared) + sizeof(int) * static_cast<size_t>(U + 1) * threads + 15) & ~static_cast<size_t>(15);
}
extern __shared__ __align__(16) unsigned char g_smem[];
__device__ __forceinline__ SharedHead &block_head() { return *reinterpret_cast<SharedHead *>(g_smem); }
__device__ __forceinline__ FastShared &block_fast() { return *reinterpret_cast<FastShared *>(g_smem + kHeadBytes); }
__device__ __forceinline__ int *block_columns() {
    return reinterpret_cast<int *>(g_smem + kHeadBytes + sizeof(FastShared));
}

__device__ __forceinline__ void load_fast_zig(const ZigTab *src) {
    FastShared &fs = block_fast();
    for (int i = threadIdx.x; i < kZigLayers; i += blockDim.x) {
        fs.zx[i] = make_float2(src->fast_hi[i], __uint_as_float(src->fast_lo[i]));
    }
}

// Per-filter part of the set-up (the network's tables are loaded); the caller
// synchronises afterwards.
__device__ __forceinline__ void fast_network() {
    FastShared &fs = block_fast();
    int *const cols = block_columns();
    const NetTables &n = block_head().net;
    const int tid = threadIdx.x, B = blockDim.x;
    const uint32_t row = 4u * B;
    cols[n.U * B + tid] = 1;
    if (tid < 32) {
        const int r = tid;
        int gain = 0;
        bool ok = true, second = false;
        uint32_t a = n.U * row, b = n.U * row << 1;
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        if (r < n.R) {
            const int sa = n.sp_a[r], sb = n.sp_b[r];
            if (sa >= 0) a = sa * row;
            if (sa >= 0 && n.ord_a[r] == 2) {
                b = (a << 1) | 1u;
                second = true;
            } else if (sb >= 0) {
                b = sb * row << 1;
                second = true;
            }
            ok = n.n_change[r] <= 4;
            for (int i = 0; i < n.n_change[r] && i < 4; ++i) {
                const int dl = n.ch_delta[r][i];
                w[i] = (static_cast<uint32_t>(n.ch_sp[r][i]) * row << 16) | (static_cast<uint32_t>(dl) & 0xFFFFu);
                gain = max(gain, dl);
            }
        }
        fs.reac[r] = FastReac{0u, 0u, a, b};
        fs.change[r] = make_uint4(w[0], w[1], w[2], w[3]);
        gain = __reduce_max_sync(0xFFFFFFFFu, gain);
        const uint32_t m2 = __ballot_sync(0xFFFFFFFFu, second);
        const bool all_ok = __all_sync(0xFFFFFFFFu, ok);
        if (r == 0) {
            fs.gain = gain;
            fs.mask2 = m2;
            fs.possible = all_ok;
        }
        if (r < PF_MAX_SPECIES) fs.mx[r] = 0;
    }
}

// Exponent of a positive normal double.
__device__ __forceinline__ int exponent_of(double v) {
    return static_cast<int>(__double_as_longlong(v) >> 52) - 1023;
}

// Per-filter part that needs the rates (set by the threads r < R); the caller
// synchronises afterwards.
__device__ __forceinline__ void fast_rate(int r, double rate) {
    const int ex = exponent_of(rate);
    const bool zero = __double_as_longlong(rate) == 0;
    if (!zero && !(ex > -80 && ex < 80)) atomicAnd(&block_fast().possible, 0);
    block_fast().rate_up[r] = zero ? 0.0f : __double2float_ru(rate);
}

// Per-interval set-up by the whole block: caps, k, A_r, time scale and bounds.
// Returns whether the interval can run here (the same in every thread); the
// caller has synchronised after the last write to xs.
static __device__ __noinline__ bool fast_interval(const int *xs, int Np, int N, double t_prev, double t_end,
                                           uint64_t budget) {
    FastShared &fs = block_fast();
    if (!fs.possible) return false;
    const NetTables &n = block_head().net;
    const double *rate = block_head().rate;
    const int tid = threadIdx.x, B = blockDim.x, U = n.U;
    for (int u = 0; u < U; ++u) {
        int m = 0;
        for (int j = tid; j < N; j += B) m = max(m, xs[u * Np + j]);
        m = __reduce_max_sync(0xFFFFFFFFu, m);
        if ((tid & 31) == 0) atomicMax(&fs.mx[u], m);
    }
    __syncthreads();
    if (tid < 32) {
        const int r = tid;
        const uint32_t room = static_cast<uint32_t>(kCheckTrips * fs.gain);
        auto cap_of = [&](uint32_t row_off) -> uint64_t {
            const int u = static_cast<int>(row_off / (4u * B));
            if (u >= U) return 1ull;
            return 4ull * static_cast<uint32_t>(fs.mx[u]) + 1024ull + room;
        };
        bool ok = true;
        float up = 0.0f;
        uint64_t h = 1;
        if (r < n.R) {
            up = fs.rate_up[r];
            const FastReac &q = fs.reac[r];
            const uint64_t ca = cap_of(q.a), cb = cap_of(q.b >> 1);
            h = ca * cb;                     // the product formed before the shift must fit 32 bits
            ok = ca < (1ull << 28) && cb < (1ull << 28) && h < (1ull << 32);
            if (q.b & 1u) h >>= 1;
        }
        const float hf = __uint2float_ru(static_cast<uint32_t>(h));
        // sum of rate times the largest h, rounded up
        float sum = __fmul_ru(up, hf);
        for (int o = 16; o > 0; o >>= 1) sum = __fadd_ru(sum, __shfl_xor_sync(0xFFFFFFFFu, sum, o));
        ok = ok && sum > 0.0f && sum < 1e36f;
        const int k = 61 - ((__float_as_int(sum) >> 23) - 127);     // sum 2^k < 2^62
        uint64_t A = 0;
        if (ok && up > 0.0f) {
            const long long rb = __double_as_longlong(rate[r]);
            const uint64_t m53 = (static_cast<uint64_t>(rb) & ((1ull << 52) - 1ull)) | (1ull << 52);
            const int sh = static_cast<int>(rb >> 52) - 1075 + k;
            if (sh >= 0) A = m53 << min(sh, 63);
            else if (sh > -63) A = (m53 + (1ull << (-sh - 1))) >> -sh;
        }
        if (r < n.R) {
            fs.reac[r].lo = static_cast<uint32_t>(A);
            fs.reac[r].hi = static_cast<uint32_t>(A >> 32);
        }
        // absolute error of the sums from the coarsely represented rates
        const bool coarse = up > 0.0f && A < (1ull << 30);
        float e_abs = coarse ? 0.5f * hf : 0.0f;
        for (int o = 16; o > 0; o >>= 1) e_abs = __fadd_ru(e_abs, __shfl_xor_sync(0xFFFFFFFFu, e_abs, o));
        ok = ok && e_abs < 1073741824.0f;
        // time scale: D = (t_end - t_prev) 2^q in [2^49, 2^50)
        const double d = __dsub_rn(t_end, t_prev);
        const int ed = exponent_of(d), q = 49 - ed;
        const uint64_t D = ((static_cast<uint64_t>(__double_as_longlong(d)) & ((1ull << 52) - 1ull)) | (1ull << 52)) >> 3;
        const int far = exponent_of(t_end) + 1 - ed;              // t_end < 2^far D
        ok = ok && ed > -500 && ed < 500 && far <= 14;
        const int kq = k + q;
        ok = ok && kq >= 40 && kq <= 120;
        const uint32_t c = 4u + (ok ? 1u << max(far - 2, 0) : 0u);
        const uint64_t per_draws = c * (budget < (1ull << 40) ? budget : (1ull << 40));
        const uint64_t b_quick = (D >> 16) + per_draws;
        ok = ok && b_quick < (D >> 2);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (r < U) {
            const uint64_t most = 4ull * static_cast<uint32_t>(fs.mx[r]) + 1024ull;
            fs.lim[r] = static_cast<int>(most < (1ull << 28) ? most : (1ull << 28));
            fs.mx[r] = 0;                     // for the next interval
        }
        if (r == 0) {
            fs.D = D;
            fs.unit = __longlong_as_double(static_cast<long long>(1023 + (ok ? q : 0)) << 52);
            fs.b0 = D >> 28;
            fs.quick_lo = static_cast<uint32_t>((D - b_quick) >> 30);
            fs.quick_hi = static_cast<uint32_t>((D + b_quick) >> 30);
            fs.c = c;
            // e_abs / a0 stays below 2^-18: well inside the quick bound's 2^-16 D
            // and, in 31-bit units, below half the margin of 2^14
            fs.hi_min = 1u + static_cast<uint32_t>(e_abs * (1.0f / 16384.0f));
            fs.margin = e_abs > 0.0f ? 16384u : 16u;
            fs.scale = static_cast<uint32_t>(127 + kq - 32) << 23;
            fs.ecoef = ok ? __fmul_ru(__fmul_ru(e_abs, 1.01f), __int_as_float((127 - kq) << 23)) : 0.0f;
            fs.on = ok;
            fs.n_exact = 0;
        }
    }
    __syncthreads();
    return fs.on != 0;
}

// One draw by the FP64 definition from the counts in the column `col` (rows
// `row` bytes apart): the reaction (or -1 when a_0 = 0) and tau = E / a_0.
static __device__ __noinline__ int exact_step(const NetTables &n, const double *rate, const int *col,
                                              int stride, double E, uint64_t v2, double &tau) {
    auto prop = [&](int r) {
        long long h = 1;
        const int sa = n.sp_a[r], sb = n.sp_b[r];
        if (sa >= 0) {
            const long long x = col[sa * stride];
            h = n.ord_a[r] == 2 ? (x >= 2 ? x * (x - 1) / 2 : 0) : x;
        }
        if (sb >= 0) h *= col[sb * stride];
        return __dmul_rn(rate[r], count_to_double(h));
    };
    const int R = n.R;
    double a0 = prop(0);
    for (int r = 1; r < R; ++r) a0 = __dadd_rn(a0, prop(r));
    if (__double_as_longlong(a0) == 0) return -1;
    tau = div_pos(E, a0);
    const long long tb = __double_as_longlong(__dmul_rn(scaled_u53_or_zero(v2), a0));
    int chosen = 0, last = 0;
    double run = 0.0;
    for (int r = 0; r < R; ++r) {
        const double a = prop(r);
        run = r == 0 ? a : __dadd_rn(run, a);
        if (__double_as_longlong(run) <= tb) ++chosen;
        if (__double_as_longlong(a) != 0) last = r;
    }
    return chosen >= R ? last : chosen;
}

// One attempt of the ziggurat: u x_i as a sum of two floats, u from the 48 upper
// bits of the word (w1, w0), and whether the layer's test accepts it.
__device__ __forceinline__ bool zig_first(const FastShared &fs, int layer, uint32_t w1, uint32_t w0, float &Eh,
                                          float &El) {
    const float2 zx = fs.zx[layer];
    const uint32_t z = __float_as_uint(zx.y);
    const float uh = static_cast<float>(w1 >> 8);
    const float ul = static_cast<float>(__byte_perm(w0, w1, 0x4432) & 0xFFFFFFu) * 5.9604644775390625e-8f;
    const float p = __fmul_rn(uh, zx.x);
    float q = __fmaf_rn(uh, zx.x, -p);
    q = __fmaf_rn(ul, zx.x, q);
    q = __fmaf_rn(uh, __uint_as_float(z & 0xFFFF0000u), q);
    Eh = __fadd_rn(p, q);
    El = __fsub_rn(q, __fsub_rn(Eh, p));
    return (w1 >> 16) - 16u < (z & 0xFFFFu);
}

// A draw whose first word (layer, w1, w0) passes no layer test: the wedge tests
// U < (e^d - 1) / (e^D - 1), d = x_i - x, D = x_i - x_{i+1} (the ziggurat's
// f_i + U (f_{i+1} - f_i) < e^-x divided by f_i), and further attempts, as
// zig_exp does them.  Both sides are within 2^-19 of their FP64 values; false
// when they are closer than 2^-15, or for the tail and for small u: zig_exp
// then decides (1 draw in 3000).
static __device__ __noinline__ bool zig_wedges(const FastShared &fs, const ZigTab *zig, int layer, uint32_t w1,
                                               uint32_t w0, uint32_t draws, uint32_t particle, uint32_t lane,
                                               uint32_t mrow, uint32_t key0, uint32_t key1, float &Eh, float &El) {
    for (uint32_t s = 1; s < 32; ++s) {
        if (layer == 0 || (w1 >> 16) < 16u) return false;
        const Philox4 x = philox4x32_10(draws, particle | (s << 16), lane, mrow, key0, key1);
        const float xi = fs.zx[layer].x * 16777216.0f;
        const float d = static_cast<float>(~w1) * 2.3283064365386963e-10f * xi;
        const float g = expm1f(d) * __ldg(&zig->wedge[layer]);
        const float U = static_cast<float>(x.w1) * 2.3283064365386963e-10f;
        if (fabsf(U - g) < 3.0517578125e-5f) return false;
        if (U < g) return true;
        w1 = x.w3;
        w0 = x.w2;
        layer = static_cast<int>(w0 & 0x7FFu);
        if ((w1 >> 16) < 16u) return false;
        if (zig_first(fs, layer, w1, w0, Eh, El)) return true;
    }
    return false;
}

// Shared-memory accesses by 32-bit address (columns are private to a lane).
__device__ __forceinline__ uint32_t shared_addr(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint32_t col_load(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void col_store(uint32_t addr, uint32_t v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// Philox round keys: from the seed, or precomputed in the kernel's parameters
// (constant-bank operands: no additions and no registers).
struct SeedKeys {
    uint32_t key0, key1;
    __device__ __forceinline__ uint32_t k0(uint32_t round) const { return key0 + round * 0x9E3779B9u; }
    __device__ __forceinline__ uint32_t k1(uint32_t round) const { return key1 + round * 0xBB67AE85u; }
};
struct ParamKeys {
    const uint32_t *rk;        // k0 of rounds 0..9, then k1
    __device__ __forceinline__ uint32_t k0(uint32_t round) const { return rk[round]; }
    __device__ __forceinline__ uint32_t k1(uint32_t round) const { return rk[10 + round]; }
};

static __device__ __noinline__ double zig_call(uint32_t w1, uint32_t w0, uint32_t draws, uint32_t particle, uint32_t lane,
                                               uint32_t mrow, uint32_t key0, uint32_t key1, const ZigTab *zig) {
    return zig_exp((static_cast<uint64_t>(w1) << 32) | w0, draws, particle, lane, mrow, key0, key1, zig->x, zig);
}

// Simulate the interval's particles (see the head of this file).  Particles
// that must be replayed are appended to `redo`, their state untouched.
// Returns the reactions that this thread's finished particles fired.
// Preconditions: fast_interval returned true, sh.pool_next = blockDim.x,
// sh.rem_n = {0, 0}.
//
// Up to eight reactions keep their prefix sums in registers and compare all of
// them with the target.  More keep only every fourth sum: the choice picks a
// group of four by those and computes the group's sums again, which costs the
// same instructions (20 reactions: 9 compares instead of 20, three sums again)
// and 16 registers instead of 64, so that 24 warps fit on an SM instead of 16.
template <int RM, int UM, class Keys>
__device__ __forceinline__ unsigned long long ssa_fast(int *xs, int Np, int N, const Keys &keys, uint32_t lane,
                                                       uint32_t mrow, uint32_t budget32, uint32_t j0, int *redo) {
    constexpr uint32_t kMulA = 0xD2511F53u, kMulB = 0xCD9E8D57u;
    constexpr bool kHoist = RM <= 4;             // reactions in registers
    constexpr bool kGroups4 = RM > 8;            // prefix sums by groups of four
    SharedHead &sh = block_head();
    FastShared &fs = block_fast();
    int *const cols = block_columns();
    const int R4 = (sh.net.R + 3) & ~3, U = sh.net.U;
    const uint32_t row = 4u * blockDim.x;
    const uint32_t cols_addr = shared_addr(cols);
    const uint32_t mask2 = fs.mask2, hi_min = fs.hi_min, margin = fs.margin;
    const uint32_t quick_lo = fs.quick_lo, quick_hi = fs.quick_hi, scale = fs.scale;
    const float ecoef = fs.ecoef;
    unsigned long long fired = 0;
    uint32_t col = cols_addr + 4u * threadIdx.x;
    // Philox rounds 1 and 2 depend on the draw counter only in part
    const uint64_t pB = static_cast<uint64_t>(kMulB) * lane;
    uint32_t pA_hi = 0, pA_lo = 0;
    int j = 0;
    auto set_particle = [&]() {
        const uint32_t n0 = static_cast<uint32_t>(pB >> 32) ^ (j0 + static_cast<uint32_t>(j)) ^ keys.k0(0);
        const uint64_t p = static_cast<uint64_t>(kMulA) * n0;
        pA_hi = static_cast<uint32_t>(p >> 32) ^ keys.k1(1);
        pA_lo = static_cast<uint32_t>(p);
    };
    bool active = false;
    uint32_t t_hi = 0, t_lo = 0;                 // time: t_hi 2^30 + t_lo units, t_lo < 2^30
    uint32_t draws = 0;
    float err = 0.0f;
    auto load_state = [&]() {
        if constexpr (UM > 0) {
#pragma unroll
            for (int u = 0; u < UM; ++u)
                if (u < U) col_store(col + u * row, static_cast<uint32_t>(xs[u * Np + j]));
        } else {
            for (int u = 0; u < U; ++u) col_store(col + u * row, static_cast<uint32_t>(xs[u * Np + j]));
        }
    };
    auto store_state = [&]() {
        if constexpr (UM > 0) {
#pragma unroll
            for (int u = 0; u < UM; ++u)
                if (u < U) xs[u * Np + j] = static_cast<int>(col_load(col + u * row));
        } else {
            for (int u = 0; u < U; ++u) xs[u * Np + j] = static_cast<int>(col_load(col + u * row));
        }
    };
    auto start = [&](int slot) {
        active = slot < N;
        if (active) {
            j = slot;
            load_state();
            set_particle();
            t_hi = 0;
            t_lo = 0;
            draws = 0;
            err = 0.0f;
        }
    };
    FastReac reg[kHoist ? RM : 1];
    if constexpr (kHoist) {
#pragma unroll
        for (int r = 0; r < RM; ++r) reg[r] = fs.reac[r];
    }
    // h_r(x) of the reaction at the lane's column
    auto count = [&](const FastReac &q, bool second) -> uint32_t {
        uint32_t h = col_load(col + q.a);
        if (second) {
            const uint32_t same = q.b & 1u;
            h = (h * (col_load(col + (q.b >> 1)) - same)) >> same;
        }
        return h;
    };
    auto add = [](unsigned long long run, const FastReac &q, uint32_t h) {
        run += static_cast<unsigned long long>(q.lo) * h;
        return run + (static_cast<unsigned long long>(q.hi * h) << 32);
    };
    int src = 0, remaining = N;
    bool first = true;
    for (;;) {
        if (first) {
            start(static_cast<int>(threadIdx.x));
        } else {
            active = static_cast<int>(threadIdx.x) < remaining;
            if (active) {
                const int i = threadIdx.x;
                j = sh.rem_j[src][i];
                const unsigned long long t = static_cast<unsigned long long>(__double_as_longlong(sh.rem_t[src][i]));
                t_hi = static_cast<uint32_t>(t >> 32);
                t_lo = static_cast<uint32_t>(t);
                draws = sh.rem_draws[src][i];
                err = fs.rem_err[src][i];
                col = cols_addr + 4u * fs.rem_slot[src][i];
                set_particle();
            }
        }
        const int dst = src ^ 1;
        const bool may_park = remaining > 32;
        for (uint32_t trip = 0;; ++trip) {
            const unsigned busy = __ballot_sync(kFull, active);
            if (busy == 0) break;
            if (may_park && __popc(busy) < kParkLanes) {
                const int pool_now = __shfl_sync(kFull, *reinterpret_cast<volatile int *>(&sh.pool_next), 0);
                if (pool_now >= N) {
                    if (active) {
                        const int slot = atomicAdd(&sh.rem_n[dst], 1);
                        sh.rem_j[dst][slot] = j;
                        sh.rem_t[dst][slot] = __longlong_as_double(
                            static_cast<long long>((static_cast<unsigned long long>(t_hi) << 32) | t_lo));
                        sh.rem_draws[dst][slot] = draws;
                        fs.rem_err[dst][slot] = err;
                        fs.rem_slot[dst][slot] = static_cast<uint16_t>((col - cols_addr) >> 2);
                    }
                    break;
                }
            }
            if (!active) continue;
            int fin = 0;               // 1: at t_end, 2: to be replayed
            if (trip % kCheckTrips == 0) {
                for (int u = 0; u < U; ++u)
                    if (static_cast<int>(col_load(col + u * row)) > fs.lim[u]) fin = 2;
            }
            if (fin == 0) {
                // the draw's random words: Philox4x32-10 of (draws, particle, lane, row)
                uint32_t w0, w1, w2, w3;
                {
                    const uint64_t p1 = static_cast<uint64_t>(kMulA) * draws;
                    const uint32_t n2 = static_cast<uint32_t>(p1 >> 32) ^ mrow ^ keys.k1(0);
                    const uint64_t q1 = static_cast<uint64_t>(kMulB) * n2;
                    w0 = static_cast<uint32_t>(q1 >> 32) ^ static_cast<uint32_t>(pB) ^ keys.k0(1);
                    w1 = static_cast<uint32_t>(q1);
                    w2 = pA_hi ^ static_cast<uint32_t>(p1);
                    w3 = pA_lo;
#pragma unroll
                    for (uint32_t round = 2; round < 10; ++round) {
                        const uint64_t a = static_cast<uint64_t>(kMulA) * w0;
                        const uint64_t b = static_cast<uint64_t>(kMulB) * w2;
                        w0 = static_cast<uint32_t>(b >> 32) ^ w1 ^ keys.k0(round);
                        w1 = static_cast<uint32_t>(b);
                        w2 = static_cast<uint32_t>(a >> 32) ^ w3 ^ keys.k1(round);
                        w3 = static_cast<uint32_t>(a);
                    }
                }
                // prefix sums of the propensities (each, or every fourth)
                constexpr int kSums = kGroups4 ? RM / 4 : RM;
                unsigned long long S[kSums], run = 0;
#pragma unroll
                for (int r0 = 0; r0 < RM; r0 += 4) {
                    if (r0 < R4) {
                        const bool second = ((mask2 >> r0) & 15u) != 0;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            FastReac q;
                            if constexpr (kHoist) q = reg[r0 + i];
                            else q = fs.reac[r0 + i];
                            run = add(run, q, count(q, second));
                            if constexpr (!kGroups4) S[r0 + i] = run;
                        }
                    } else if constexpr (!kGroups4) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) S[r0 + i] = run;
                    }
                    if constexpr (kGroups4) S[r0 / 4] = run;
                }
                const uint32_t a_hi = static_cast<uint32_t>(run >> 32);
                int chosen;
                uint32_t n_hi = t_hi, n_lo = t_lo;       // time of the event
                if (a_hi >= hi_min) {
                    if (draws >= budget32) {
                        sh.status = PF_ST_BUDGET;
                        fin = 1;
                    }
                    // E as a sum of two floats
                    const int layer = static_cast<int>(w0 & 0x7FFu);
                    float Eh, El;
                    if (!zig_first(fs, layer, w1, w0, Eh, El) &&
                        !zig_wedges(fs, sh.zig_g, layer, w1, w0, draws, j0 + static_cast<uint32_t>(j), lane, mrow,
                                    keys.k0(0), keys.k1(0), Eh, El)) {
                        const double E = zig_call(w1, w0, draws, j0 + static_cast<uint32_t>(j), lane, mrow, keys.k0(0),
                                                  keys.k1(0), sh.zig_g);
                        Eh = __double2float_rn(E);
                        El = __double2float_rn(__dsub_rn(E, static_cast<double>(Eh)));
                    }
                    // tau = E / a0 in time units: a0's 32 leading bits as f + g
                    const int s = 158 - (__float_as_int(__uint2float_rz(a_hi)) >> 23);
                    const uint32_t mh = __funnelshift_l(static_cast<uint32_t>(run), a_hi, s);
                    const float f = static_cast<float>(mh & 0xFFFFFF00u), g = static_cast<float>(mh & 0xFFu);
                    float rc;
                    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rc) : "f"(f));
                    const float e = __fmaf_rn(-g, rc, __fmaf_rn(-f, rc, 1.0f));
                    const float rs = __fmul_rn(rc, __int_as_float(static_cast<int>(scale + (static_cast<uint32_t>(s) << 23))));
                    const float ph = __fmul_rn(Eh, rs);
                    float pl = __fmaf_rn(Eh, rs, -ph);
                    pl = __fmaf_rn(El, rs, pl);
                    pl = __fmaf_rn(ph, e, pl);
                    err = __fmaf_ru(ph, __fmul_ru(rs, ecoef), err);
                    // tau to an integer in two parts (64-bit conversions run on
                    // the FP64 pipe): a multiple of 2^30 by adding 1.5 2^23, and
                    // the rest; from 2^52 on the event is late whatever its size.
                    // |rest| <= 2^29 and |pl| < 2^-21.5 ph: for ph up to 1.3 2^50,
                    // beyond which the event is late whatever lo's carry, lo fits
                    const float pc = fminf(ph, 4503599627370496.0f);
                    const float top = __fmaf_rn(pc, 9.31322574615478515625e-10f, 12582912.0f);
                    const float rest = __fmaf_rn(-1073741824.0f, __fsub_rn(top, 12582912.0f), pc);
                    const uint32_t lo = t_lo + static_cast<uint32_t>(__float2int_rn(__fadd_rn(rest, pl)));
                    n_hi = t_hi + (__float_as_uint(top) - 0x4B400000u) + static_cast<uint32_t>(static_cast<int>(lo) >> 30);
                    n_lo = lo & 0x3FFFFFFFu;
                    // the reaction: the prefix sums at or below u2 a0, on 31
                    // leading bits; a target next to a0 itself counts as near
                    const uint32_t tgt = __umulhi(w3, mh) >> 1;
                    uint32_t near = ~w3;
                    auto below = [&](unsigned long long v) -> int {      // 0 when the sum is at or below the target, else -1
                        const uint32_t d = tgt - __funnelshift_l(static_cast<uint32_t>(v), static_cast<uint32_t>(v >> 32), s - 1);
                        near = min(near, d + margin);
                        return static_cast<int>(d) >> 31;
                    };
                    if constexpr (kGroups4) {
                        int above = 0;
                        unsigned long long base = 0;
#pragma unroll
                        for (int q = 0; q < RM / 4 - 1; ++q) {
                            if (4 * q < R4) {
                                const int b = below(S[q]);
                                above += b + 1;
                                base = b ? base : S[q];
                            }
                        }
                        chosen = min(4 * above, R4 - 4);
                        int inner = 3;
#pragma unroll
                        for (int i = 0; i < 3; ++i) {
                            const FastReac q = fs.reac[chosen + i];
                            base = add(base, q, count(q, mask2 != 0));
                            inner += below(base);
                        }
                        chosen += inner;
                    } else {
                        chosen = RM - 1;
#pragma unroll
                        for (int r = 0; r < RM - 1; ++r) chosen += below(S[r]);
                    }
                    if (near < 2u * margin) {
                        double tau;
                        chosen = exact_step(sh.net, sh.rate, cols + ((col - cols_addr) >> 2), blockDim.x, 1.0,
                                            ((static_cast<uint64_t>(w3) << 32) | w2) >> 11, tau);
                    }
                } else {
                    // a0 is zero or too small for its relative error
                    const double E = zig_call(w1, w0, draws, j0 + static_cast<uint32_t>(j), lane, mrow, keys.k0(0),
                                              keys.k1(0), sh.zig_g);
                    double tau = 0.0;
                    chosen = exact_step(sh.net, sh.rate, cols + ((col - cols_addr) >> 2), blockDim.x, E,
                                        ((static_cast<uint64_t>(w3) << 32) | w2) >> 11, tau);
                    if (chosen < 0) {
                        fin = 1;                           // absorbing: nothing can fire
                    } else if (draws >= budget32) {
                        sh.status = PF_ST_BUDGET;
                        fin = 1;
                    } else {
                        const double d = fmin(__dmul_rn(tau, fs.unit), 4503599627370496.0);
                        const unsigned long long t = static_cast<unsigned long long>(__double2ll_rn(d)) + t_lo;
                        n_hi = t_hi + static_cast<uint32_t>(t >> 30);
                        n_lo = static_cast<uint32_t>(t) & 0x3FFFFFFFu;
                    }
                }
                if (fin) {
                    fired += draws;
                } else {
                    ++draws;
                    if (n_hi >= quick_lo) {
                        if (n_hi > quick_hi) {
                            fin = 1;
                        } else {
                            const unsigned long long t = (static_cast<unsigned long long>(n_hi) << 30) | n_lo;
                            const unsigned long long b = fs.b0 + static_cast<unsigned long long>(fs.c) * draws +
                                                         static_cast<unsigned long long>(__float2ll_ru(err)) + 2ull;
                            if (t > fs.D + b) fin = 1;
                            else if (t + b >= fs.D) fin = 2;
                        }
                    }
                    if (fin == 0) {
                        t_hi = n_hi;
                        t_lo = n_lo;
                        const uint4 ch = fs.change[chosen];
                        auto apply = [&](uint32_t w) {
                            const uint32_t p = col + (w >> 16);
                            col_store(p, col_load(p) + static_cast<uint32_t>(static_cast<int>(static_cast<int16_t>(w & 0xFFFFu))));
                        };
                        if (ch.x) apply(ch.x);
                        if (ch.y) {
                            apply(ch.y);
                            if (ch.z) apply(ch.z);
                            if (ch.w) apply(ch.w);
                        }
                    } else if (fin == 1) {
                        fired += draws - 1;
                    }
                }
            }
            if (fin) {
                if (fin == 1) store_state();
                else redo[atomicAdd(&fs.n_exact, 1)] = j;
                active = false;
                if (first) start(atomicAdd(&sh.pool_next, 1));
            }
        }
        __syncthreads();
        remaining = sh.rem_n[dst];
        if (remaining == 0) break;
        if (threadIdx.x == 0) sh.rem_n[src] = 0;
        __syncthreads();
        src = dst;
        first = false;
    }
    return fired;
}

}  // namespace dev
}  // namespace pf

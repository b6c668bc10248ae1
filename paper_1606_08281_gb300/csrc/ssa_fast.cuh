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
//     arithmetic from 48 bits of u >= 2^-12 and x_i to 2^-48; draws whose layer
//     test w1 < T_i (an integer threshold, a lower bound of the FP64 test) does
//     not accept, 0.4 % of them, take the FP64 ziggurat.
//   * tau = E / a0 from the approximate reciprocal of a0's 24 leading bits,
//     corrected to all of its 32 leading bits; relative error below
//     2^-31 (rates) + 2^-31 (a0 truncated) + 2^-36 (u) + 2^-42 (reciprocal,
//     products) < 2^-29.9.  Times are 64-bit integers with the interval scaled
//     to [2^50, 2^51) units, so sums add one unit of rounding per event.
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
// bit.  What bounds the path is instruction issue: gene expression (R = 4)
// spends about 190 warp instructions per event instead of 580 with 16 FP64
// ones of 16 cycles each.
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
constexpr int kMaxThreads = 128;
constexpr int kCheckTrips = 32;    // trips between two looks at the counts' caps

// One reaction: A_r and the byte offsets of its reactants' rows in a column.
// Row U of every column holds 1, so h = x_a for orders 0 and 1; otherwise
// h = x_a (x_b - same) >> same (same = 1 for X + X).
struct FastReac {
    uint32_t lo, hi, a, b;     // b: offset << 1 | same
};

struct __align__(16) FastShared {
    float2 zx[kZigLayers];               // x_i 2^-24, leading and trailing part
    uint16_t zt[kZigLayers];             // accept when (w1 >> 16) - 16 < zt (unsigned)
    FastReac reac[PF_MAX_REACTIONS];
    uint4 change[PF_MAX_REACTIONS];      // up to four words: row offset << 16 | delta
    int mx[PF_MAX_SPECIES];              // the population's largest counts
    int lim[PF_MAX_SPECIES];             // a count above leaves the caps within kCheckTrips events
    unsigned long long D;                // interval length in time units
    unsigned long long b0;               // b without its per-draw and e_abs parts
    double unit;                         // time units per unit of time (a power of two)
    uint32_t quick_lo, quick_hi;         // upper words that decide most events
    uint32_t c;                          // units per draw in b
    uint32_t hi_min;                     // a0's upper word below this: exact_step
    uint32_t margin;                     // reaction choice
    uint32_t scale;                      // exponent bits of the time scale
    float ecoef;                         // e_abs in the units the path's bound needs
    uint32_t mask2;                      // reactions of order 2
    int gain;                            // largest count a reaction adds
    int possible;                        // the network's part of the conditions
    int on;                              // this interval runs here
    int n_exact;                         // particles to replay
    uint16_t rem_slot[2][kMaxThreads];   // parked particles' columns
    float rem_err[2][kMaxThreads];       // and accumulated bounds
};

// Shared memory of the path: tables, and U + 1 rows of one column per thread.
__host__ __device__ __forceinline__ size_t fast_smem_bytes(int U, int threads) {
    return sizeof(FastShared) + sizeof(int) * static_cast<size_t>(U + 1) * threads;
}

__device__ __forceinline__ void load_fast_zig(FastShared &fs, const ZigTab *src) {
    for (int i = threadIdx.x; i < kZigLayers; i += blockDim.x) {
        fs.zx[i] = make_float2(src->fast_hi[i], src->fast_lo[i]);
        fs.zt[i] = src->fast_t[i];
    }
}

// Per-filter part of the set-up (the network's tables are loaded); the caller
// synchronises afterwards.
__device__ __forceinline__ void fast_network(FastShared &fs, int *cols, const NetTables &n) {
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

// Per-interval set-up by the whole block: caps, k, A_r, time scale and bounds.
// Returns whether the interval can run here (the same in every thread); the
// caller has synchronised after the last write to xs.
__device__ __forceinline__ bool fast_interval(FastShared &fs, const NetTables &n, const double *rate,
                                              const int *xs, int Np, int N, double t_prev,
                                              double t_end, uint64_t budget) {
    if (!fs.possible) return false;
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
        double rt = 0.0;
        uint64_t h = 1;
        if (r < n.R) {
            rt = rate[r];
            const FastReac &q = fs.reac[r];
            const uint64_t ca = cap_of(q.a), cb = cap_of(q.b >> 1);
            ok = ca < (1ull << 28) && cb < (1ull << 28);
            h = ca * cb;                     // the product formed before the shift must fit 32 bits
            ok = ok && h < (1ull << 32);
            if (q.b & 1u) h >>= 1;
            const int ex = exponent_of(rt);
            ok = ok && (__double_as_longlong(rt) == 0 || (ex > -80 && ex < 80));
        }
        // sum of rate times the largest h, rounded up
        float sum = r < n.R ? __fmul_ru(__double2float_ru(rt), __ull2float_ru(h)) : 0.0f;
        for (int o = 16; o > 0; o >>= 1) sum = __fadd_ru(sum, __shfl_xor_sync(0xFFFFFFFFu, sum, o));
        ok = ok && sum > 0.0f && sum < 1e36f;
        const int k = 61 - ((__float_as_int(sum) >> 23) - 127);     // sum 2^k < 2^62
        uint64_t A = 0;
        if (ok && __double_as_longlong(rt) != 0) {
            const uint64_t m53 = (static_cast<uint64_t>(__double_as_longlong(rt)) & ((1ull << 52) - 1ull)) | (1ull << 52);
            const int sh = exponent_of(rt) - 52 + k;
            if (sh >= 0) A = m53 << min(sh, 63);
            else if (sh > -63) A = (m53 + (1ull << (-sh - 1))) >> -sh;
        }
        if (r < n.R) {
            fs.reac[r].lo = static_cast<uint32_t>(A);
            fs.reac[r].hi = static_cast<uint32_t>(A >> 32);
        }
        // absolute error of the sums from the coarsely represented rates
        const bool coarse = __double_as_longlong(rt) != 0 && A < (1ull << 30);
        float e_abs = coarse ? __fmul_ru(0.5f, __ull2float_ru(h)) : 0.0f;
        for (int o = 16; o > 0; o >>= 1) e_abs = __fadd_ru(e_abs, __shfl_xor_sync(0xFFFFFFFFu, e_abs, o));
        ok = ok && e_abs < 1073741824.0f;
        // time scale: D = (t_end - t_prev) 2^q in [2^50, 2^51)
        const double d = __dsub_rn(t_end, t_prev);
        const int ed = exponent_of(d), q = 50 - ed;
        const uint64_t D = ((static_cast<uint64_t>(__double_as_longlong(d)) & ((1ull << 52) - 1ull)) | (1ull << 52)) >> 2;
        const float ratio = __fdiv_ru(__double2float_ru(t_end), __double2float_rd(d));
        ok = ok && ed > -500 && ed < 500 && ratio < 16384.0f;
        const int kq = k + q;
        ok = ok && kq >= 40 && kq <= 120;
        const uint32_t c = ok ? 4u + static_cast<uint32_t>(ratio) : 4u;
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
            fs.quick_lo = static_cast<uint32_t>((D - b_quick) >> 32);
            fs.quick_hi = static_cast<uint32_t>((D + b_quick) >> 32);
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

// Simulate the interval's particles (see the head of this file).  Particles
// that must be replayed are appended to `redo`, their state untouched.
// Preconditions: fast_interval returned true, sh.pool_next = blockDim.x,
// sh.rem_n = {0, 0}.
template <int RM>
__device__ __forceinline__ void ssa_fast(SharedHead &sh, FastShared &fs, int *cols, int *xs, int Np, int N,
                                         uint32_t key0, uint32_t key1, uint32_t lane, uint32_t mrow,
                                         uint64_t budget, unsigned long long &fired, uint32_t j0, int *redo) {
    constexpr uint32_t kMulA = 0xD2511F53u, kMulB = 0xCD9E8D57u;
    constexpr uint32_t kWeylA = 0x9E3779B9u, kWeylB = 0xBB67AE85u;
    const int R4 = (sh.net.R + 3) & ~3, U = sh.net.U, B = blockDim.x;
    const uint32_t mask2 = fs.mask2, hi_min = fs.hi_min, margin = fs.margin;
    const uint32_t quick_lo = fs.quick_lo, quick_hi = fs.quick_hi, scale = fs.scale;
    const float ecoef = fs.ecoef;
    const uint32_t budget32 = static_cast<uint32_t>(budget);
    char *col = reinterpret_cast<char *>(cols + threadIdx.x);
    // Philox rounds 1 and 2 depend on the draw counter only in part
    const uint64_t pB = static_cast<uint64_t>(kMulB) * lane;
    uint32_t pn0 = 0, pA_hi = 0, pA_lo = 0;
    int j = 0;
    auto set_particle = [&]() {
        pn0 = static_cast<uint32_t>(pB >> 32) ^ (j0 + static_cast<uint32_t>(j)) ^ key0;
        const uint64_t p = static_cast<uint64_t>(kMulA) * pn0;
        pA_hi = static_cast<uint32_t>(p >> 32) ^ (key1 + kWeylB);
        pA_lo = static_cast<uint32_t>(p);
    };
    bool active = false;
    unsigned long long t = 0;
    uint32_t draws = 0;
    float err = 0.0f;
    auto start = [&](int slot) {
        active = slot < N;
        if (active) {
            j = slot;
            for (int u = 0; u < U; ++u) *reinterpret_cast<int *>(col + u * 4 * B) = xs[u * Np + j];
            set_particle();
            t = 0;
            draws = 0;
            err = 0.0f;
        }
    };
    // small networks keep the reactions in registers
    constexpr bool kHoist = RM <= 4;
    FastReac reg[kHoist ? RM : 1];
    if constexpr (kHoist) {
#pragma unroll
        for (int r = 0; r < RM; ++r) reg[r] = fs.reac[r];
    }
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
                t = static_cast<unsigned long long>(__double_as_longlong(sh.rem_t[src][i]));
                draws = sh.rem_draws[src][i];
                err = fs.rem_err[src][i];
                col = reinterpret_cast<char *>(cols + fs.rem_slot[src][i]);
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
                        sh.rem_t[dst][slot] = __longlong_as_double(static_cast<long long>(t));
                        sh.rem_draws[dst][slot] = draws;
                        fs.rem_err[dst][slot] = err;
                        fs.rem_slot[dst][slot] = static_cast<uint16_t>(reinterpret_cast<int *>(col) - cols);
                    }
                    break;
                }
            }
            if (!active) continue;
            int fin = 0;               // 1: at t_end, 2: to be replayed
            if (trip % kCheckTrips == 0) {
                for (int u = 0; u < U; ++u)
                    if (*reinterpret_cast<int *>(col + u * 4 * B) > fs.lim[u]) fin = 2;
            }
            if (fin == 0) {
                // the draw's random words: Philox4x32-10 of (draws, particle, lane, row)
                uint32_t w0, w1, w2, w3;
                {
                    const uint64_t p1 = static_cast<uint64_t>(kMulA) * draws;
                    const uint32_t n2 = static_cast<uint32_t>(p1 >> 32) ^ mrow ^ key1;
                    const uint64_t q1 = static_cast<uint64_t>(kMulB) * n2;
                    uint32_t c0 = static_cast<uint32_t>(q1 >> 32) ^ static_cast<uint32_t>(pB) ^ (key0 + kWeylA);
                    uint32_t c1 = static_cast<uint32_t>(q1);
                    uint32_t c2 = pA_hi ^ static_cast<uint32_t>(p1);
                    uint32_t c3 = pA_lo;
#pragma unroll
                    for (uint32_t round = 2; round < 10; ++round) {
                        const uint64_t a = static_cast<uint64_t>(kMulA) * c0;
                        const uint64_t b = static_cast<uint64_t>(kMulB) * c2;
                        c0 = static_cast<uint32_t>(b >> 32) ^ c1 ^ (key0 + round * kWeylA);
                        c1 = static_cast<uint32_t>(b);
                        c2 = static_cast<uint32_t>(a >> 32) ^ c3 ^ (key1 + round * kWeylB);
                        c3 = static_cast<uint32_t>(a);
                    }
                    w0 = c0;
                    w1 = c1;
                    w2 = c2;
                    w3 = c3;
                }
                // prefix sums of the propensities
                unsigned long long S[RM], run = 0;
#pragma unroll
                for (int r0 = 0; r0 < RM; r0 += 4) {
                    if (r0 < R4) {
                        const bool second = ((mask2 >> r0) & 15u) != 0;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int r = r0 + i;
                            FastReac q;
                            if constexpr (kHoist) q = reg[r];
                            else q = fs.reac[r];
                            uint32_t h = *reinterpret_cast<uint32_t *>(col + q.a);
                            if (second) {
                                const uint32_t same = q.b & 1u;
                                h = (h * (*reinterpret_cast<uint32_t *>(col + (q.b >> 1)) - same)) >> same;
                            }
                            run += static_cast<unsigned long long>(q.lo) * h;
                            run += static_cast<unsigned long long>(q.hi * h) << 32;
                            S[r] = run;
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i) S[r0 + i] = run;
                    }
                }
                const uint64_t v2 = ((static_cast<uint64_t>(w3) << 32) | w2) >> 11;
                const uint32_t a_hi = static_cast<uint32_t>(run >> 32);
                int chosen;
                unsigned long long t_next = t;
                if (a_hi >= hi_min) {
                    if (draws >= budget32) {
                        sh.status = PF_ST_BUDGET;
                        fin = 1;
                    }
                    // E as a sum of two floats
                    const int layer = static_cast<int>(w0 & 0x7FFu);
                    const float2 zx = fs.zx[layer];
                    float Eh, El;
                    {
                        const float uh = static_cast<float>(w1 >> 8);
                        const float ul = static_cast<float>(((w1 & 0xFFu) << 16) | (w0 >> 16)) * 5.9604644775390625e-8f;
                        const float p = __fmul_rn(uh, zx.x);
                        float q = __fmaf_rn(uh, zx.x, -p);
                        q = __fmaf_rn(ul, zx.x, q);
                        q = __fmaf_rn(uh, zx.y, q);
                        Eh = __fadd_rn(p, q);
                        El = __fsub_rn(q, __fsub_rn(Eh, p));
                    }
                    if ((w1 >> 16) - 16u >= static_cast<uint32_t>(fs.zt[layer])) {
                        const uint64_t r0 = (static_cast<uint64_t>(w1) << 32) | w0;
                        const double E = zig_exp(r0, draws, j0 + static_cast<uint32_t>(j), lane, mrow, key0, key1,
                                                 sh.zig_g->x, sh.zig_g);
                        Eh = __double2float_rn(E);
                        El = __double2float_rn(__dsub_rn(E, static_cast<double>(Eh)));
                    }
                    // tau = E / a0 in time units
                    const int s = __clz(static_cast<int>(a_hi));
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
                    t_next = t + static_cast<unsigned long long>(__float2ll_rn(ph)) +
                             static_cast<unsigned long long>(static_cast<long long>(__float2int_rn(pl)));
                    // the reaction
                    const uint32_t tgt = __umulhi(w3, mh) >> 1;
                    int neg = 0;
                    uint32_t near = 0xFFFFFFFFu;
#pragma unroll
                    for (int r0 = 0; r0 < RM; r0 += 4) {
                        if (r0 < R4) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const uint32_t Sn = __funnelshift_l(static_cast<uint32_t>(S[r0 + i]),
                                                                    static_cast<uint32_t>(S[r0 + i] >> 32), s - 1);
                                const uint32_t dd = tgt - Sn;
                                neg += static_cast<int>(dd) >> 31;
                                near = min(near, dd + margin);
                            }
                        }
                    }
                    chosen = R4 + neg;
                    if (near < 2u * margin) {
                        double tau;
                        chosen = exact_step(sh.net, sh.rate, reinterpret_cast<int *>(col), B, 1.0, v2, tau);
                    }
                } else {
                    // a0 is zero or too small for its relative error
                    const uint64_t r0 = (static_cast<uint64_t>(w1) << 32) | w0;
                    const double E = zig_exp(r0, draws, j0 + static_cast<uint32_t>(j), lane, mrow, key0, key1,
                                             sh.zig_g->x, sh.zig_g);
                    double tau = 0.0;
                    chosen = exact_step(sh.net, sh.rate, reinterpret_cast<int *>(col), B, E, v2, tau);
                    if (chosen < 0) {
                        fin = 1;                           // absorbing: nothing can fire
                    } else if (draws >= budget32) {
                        sh.status = PF_ST_BUDGET;
                        fin = 1;
                    } else {
                        const double d = __dmul_rn(tau, fs.unit);
                        t_next = t + static_cast<unsigned long long>(__double2ll_rn(fmin(d, 1.4411518807585587e17)));
                    }
                }
                if (fin) {
                    fired += draws;
                } else {
                    ++draws;
                    const uint32_t th = static_cast<uint32_t>(t_next >> 32);
                    if (th >= quick_lo) {
                        if (th > quick_hi) {
                            fin = 1;
                        } else {
                            const unsigned long long b = fs.b0 + static_cast<unsigned long long>(fs.c) * draws +
                                                         static_cast<unsigned long long>(__float2ll_ru(err)) + 2ull;
                            if (t_next > fs.D + b) fin = 1;
                            else if (t_next + b >= fs.D) fin = 2;
                        }
                    }
                    if (fin == 0) {
                        t = t_next;
                        const uint4 ch = fs.change[chosen];
                        auto apply = [&](uint32_t w) {
                            int *p = reinterpret_cast<int *>(col + (w >> 16));
                            *p += static_cast<int>(static_cast<int16_t>(w & 0xFFFFu));
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
                if (fin == 1) {
                    for (int u = 0; u < U; ++u) xs[u * Np + j] = *reinterpret_cast<int *>(col + u * 4 * B);
                } else {
                    redo[atomicAdd(&fs.n_exact, 1)] = j;
                }
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
}

}  // namespace dev
}  // namespace pf

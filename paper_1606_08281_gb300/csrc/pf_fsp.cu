// Exact (truncated) trajectory likelihood by the finite state projection.
//
// The paper checks its sampler against the "(almost) exact" likelihood that
// the finite state projection (FSP) of the chemical master equation gives
// (Supp. "Verification of approximated posterior", the RNA model).  On the
// box B = {x : 0 <= x_u <= n_u} the generator moves probability out of every
// state x at rate a_0(x) and into x + nu_r at rate a_r(x) when that state is in
// B; probability whose next state leaves B is dropped (the FSP lower bound).
// With the particle filter's observation model, the likelihood factorises over
// observation times like the filter's estimate (Supp. I), and the forward
// algorithm computes each factor exactly:
//     alpha <- alpha exp(Q dt_k);  alpha <- alpha * p(y_k | x);
//     c_k = sum alpha;  log p(y) += log c_k;  alpha <- alpha / c_k.
//
// GB300 layout: one block per (theta row, observed trajectory).  The whole
// probability vector lives in shared memory (three S-vectors: the current
// Krylov term, the next one, and the running sum) and never touches HBM.
// exp(Q dt) acts by uniformization (Jensen's method): with lambda >= max_x
// a_0(x) and P = I + Q / lambda (substochastic),
//     alpha exp(Q h) = sum_j Pois(j; lambda h) alpha P^j,
// truncated where the Poisson tail is below 1e-17; intervals with
// lambda dt > kMaxLambdaH are split into equal sub-steps.  One product
// alpha P is a pull-form stencil (each state gathers from its predecessors
// x - nu_r), race-free and in a fixed order, with the coefficients -- per state
// the diagonal 1 - a_0(x)/lambda and the inflow weights a_r(x - nu_r)/lambda --
// in shared memory.  Three kernels differ in the states they run on: the
// reachable ones (fsp_compact_kernel), a window of a one-species box
// (fsp_window_kernel), and the whole box where neither fits (fsp_kernel).  The
// FP64 pipe bounds all of them (one warp instruction per 19 cycles and SM).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <utility>
#include <vector>

#include "pf1606.h"
#include "pf_device.cuh"
#include "pf_internal.h"

namespace pf {
namespace {

constexpr int kFspMaxTerms = 2048;       // Poisson terms per sub-step (weights in shared memory)
constexpr double kMaxLambdaH = 1500.0;   // lambda h + 8.5 sqrt(lambda h) + 20 < kFspMaxTerms
constexpr int kFspMaxThreads = 512;

struct FspArgs {
    NetTables net;
    const double *thetas;     // [M][d]
    const double *obs_times;  // [K]
    const double *y;          // [T][K][P]
    int64_t M;
    int32_t K, T, S;
    int32_t box[PF_MAX_SPECIES];
    int32_t stride[PF_MAX_SPECIES];
    int32_t off[PF_MAX_REACTIONS];    // index(x) - index(x - nu_r)
    int8_t nu_a[PF_MAX_REACTIONS];    // nu_r at the first reactant species (sp_a)
    int8_t nu_b[PF_MAX_REACTIONS];    // nu_r at the second reactant species (sp_b)
    int32_t coef_smem;                // stencil coefficients precomputed in shared memory
    // the states reachable from the initial ones, most inflows first, and each
    // one's inflows in reaction order (fsp_compact_kernel)
    int32_t Sc, E;                    // states, largest number of inflows
    const uint16_t *st_idx;           // [Sc] index in the box
    const uint16_t *in_src;           // [E][Sc] predecessor, in compact numbering
    const uint8_t *in_reac;           // [E][Sc] its reaction
    const uint8_t *in_n;              // [Sc] number of inflows
    int32_t reach;                    // one species: largest change of a reaction
    double *ll_f;                     // [M*T]
    double *leak_f;                   // [M*T] or null
    uint8_t *st_f;                    // [M*T]
};

struct FspShared {
    double rate_s[PF_MAX_REACTIONS];  // rate_r / lambda
    double red[kFspMaxThreads / 32];
    double bcast;
    int valid;
};

__device__ __forceinline__ long long h_of(int x, int p) { return dev::binom_small(x, p); }

// Block-wide max / sum of one double per thread (every thread gets the result).
__device__ double fsp_block_max(double v, FspShared &sh) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh.red[w] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = sh.red[0];
        for (int i = 1; i < nw; ++i) m = fmax(m, sh.red[i]);
        sh.bcast = m;
    }
    __syncthreads();
    return sh.bcast;
}

__device__ double fsp_block_sum(double v, FspShared &sh) {
    for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh.red[w] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < nw; ++i) s = __dadd_rn(s, sh.red[i]);
        sh.bcast = s;
    }
    __syncthreads();
    return sh.bcast;
}

// Multi-index of state i (last species fastest).
__device__ __forceinline__ void decode(const FspArgs &a, int i, int *x) {
    if (a.net.U == 1) {
        x[0] = i;
        return;
    }
    int rem = i;
    for (int u = 0; u < a.net.U; ++u) {
        x[u] = rem / a.stride[u];
        rem -= x[u] * a.stride[u];
    }
}

__device__ __forceinline__ long long combos_at(const NetTables &n, int r, const int *x, int da,
                                               int db) {
    long long h = 1;
    if (n.sp_a[r] >= 0) h = h_of(x[n.sp_a[r]] - da, n.ord_a[r]);
    if (n.sp_b[r] >= 0) h *= h_of(x[n.sp_b[r]] - db, n.ord_b[r]);
    return h;
}

// Poisson probability of j by the saddle-point form (C. Loader, "Fast and
// accurate computation of binomial probabilities", 2000):
// exp(-D(j, lh) - delta(j)) / sqrt(2 pi j), D = j log(j / lh) + lh - j as a series
// in v = (j - lh) / (j + lh) near the mode, delta the error of Stirling's formula.
// exp(-lh + j log lh - lgamma(j + 1)) loses the digits of its largest term
// (error 1e-12 at lh = 1500) and lgamma alone is some 200 FP64 instructions.
__device__ __forceinline__ double poisson_weight(int j, double lh, double llh) {
    const double x = j;
    if (j < 16) return exp(-lh + x * llh - lgamma(x + 1.0));
    const double r = 1.0 / x, r2 = r * r;
    const double delta =
        r * (1.0 / 12.0 - r2 * (1.0 / 360.0 - r2 * (1.0 / 1260.0 - r2 * (1.0 / 1680.0 - r2 * (1.0 / 1188.0)))));
    const double d = x - lh;
    double D;
    if (fabs(d) < 0.1 * (x + lh)) {
        const double v = d / (x + lh), v2 = v * v;
        double ej = 2.0 * x * v;
        D = d * v;
        for (int k = 3; k < 40; k += 2) {
            ej *= v2;
            const double next = D + ej / k;
            if (next == D) break;
            D = next;
        }
    } else {
        D = x * log(x / lh) - d;
    }
    return exp(-D - delta) * rsqrt(6.283185307179586476925 * x);
}

// Poisson weights of one sub-step of length h, lh = lambda h, into wts[0..jmax];
// returns jmax (the tail beyond it is below 1e-17).  The caller synchronises.
__device__ __forceinline__ int poisson_weights(double lh, double *wts) {
    const int jmax = min(kFspMaxTerms - 1, static_cast<int>(ceil(lh + 8.5 * sqrt(lh) + 20.0)));
    const double llh = log(lh);
    for (int j = threadIdx.x; j <= jmax; j += blockDim.x) wts[j] = poisson_weight(j, lh, llh);
    return jmax;
}

// Whether the theta row is valid (every thread learns it); reports it if not.
__device__ __forceinline__ bool fsp_valid(const FspArgs &a, FspShared &sh, const double *theta, int64_t f) {
    if (threadIdx.x == 0) {
        int ok = 1;
        for (int c = 0; c < a.net.d; ++c) ok &= (isfinite(theta[c]) && theta[c] >= 0.0) ? 1 : 0;
        sh.valid = ok;
        if (!ok) {
            a.ll_f[f] = __longlong_as_double(0x7FF8000000000000ll);
            a.st_f[f] = PF_ST_INVALID_THETA;
            if (a.leak_f) a.leak_f[f] = 0.0;
        }
    }
    __syncthreads();
    return sh.valid != 0;
}

// Constant part of the log emission.
__device__ __forceinline__ double fsp_lconst(const FspArgs &a) {
    double lconst = -0.5 * static_cast<double>(a.net.P) * log(2.0 * M_PI);
    if (!a.net.obs_state_var)
        for (int p = 0; p < a.net.P; ++p) lconst -= log(a.net.sigma[p]);
    return lconst;
}

// log p(y_k | x)
__device__ __forceinline__ double fsp_emission(const FspArgs &a, const int *x, const double *yk, double lconst) {
    double le = lconst;
    for (int p = 0; p < a.net.P; ++p) {
        double mu = a.net.obs_offset[p];
        for (int u = 0; u < a.net.U; ++u) mu = fma(a.net.C[p][u], static_cast<double>(x[u]), mu);
        const double dv = yk[p] - mu;
        if (a.net.obs_state_var) {
            double v = a.net.sigma[p] * a.net.sigma[p];
            for (int u = 0; u < a.net.U; ++u) v = fma(a.net.obs_var[p][u], static_cast<double>(x[u]), v);
            le -= 0.5 * (dv * dv / v + log(v));
        } else {
            const double z = dv / a.net.sigma[p];
            le -= 0.5 * z * z;
        }
    }
    return le;
}

// a_0(x) = sum_r rate_r h_r(x)
__device__ __forceinline__ double total_propensity(const FspArgs &a, const double *rate, const int *x) {
    double a0 = 0.0;
    for (int r = 0; r < a.net.R; ++r)
        a0 = __dadd_rn(a0, __dmul_rn(rate[r], static_cast<double>(combos_at(a.net, r, x, 0, 0))));
    return a0;
}

// Probability of state x at time 0: x0, or uniform over the box x0..x0_hi.
__device__ __forceinline__ double initial_probability(const FspArgs &a, const int *x) {
    double cnt = 1.0;
    bool in = true;
    for (int u = 0; u < a.net.U; ++u) {
        cnt *= static_cast<double>(a.net.x0_hi[u] - a.net.x0[u] + 1);
        in = in && x[u] >= a.net.x0[u] && x[u] <= a.net.x0_hi[u];
    }
    return in ? 1.0 / cnt : 0.0;
}

// The interval's end: dropped mass, emission, normalisation of cur[0..S)
// (le: scratch); state(i, x) gives state i's counts.  False when the
// observation has no probability.
template <class State>
__device__ __forceinline__ bool fsp_observe(const FspArgs &a, FspShared &sh, int S, double *cur, double *le,
                                            const double *yk, double lconst, State state, double &ll, double &leak) {
    const int tid = threadIdx.x, B = blockDim.x;
    int x[PF_MAX_SPECIES];
    double msum = 0.0;
    for (int i = tid; i < S; i += B) msum += fmax(cur[i], 0.0);
    const double mass = fsp_block_sum(msum, sh);
    leak += 1.0 - mass;
    double lmax = -INFINITY;
    for (int i = tid; i < S; i += B) {
        state(i, x);
        le[i] = fsp_emission(a, x, yk, lconst);
        const double pi = fmax(cur[i], 0.0);
        cur[i] = pi;
        if (pi > 0.0) lmax = fmax(lmax, le[i]);
    }
    const double emax = fsp_block_max(lmax, sh);
    double csum = 0.0;
    for (int i = tid; i < S; i += B) {
        const double v = cur[i] > 0.0 ? cur[i] * exp(le[i] - emax) : 0.0;
        cur[i] = v;
        csum += v;
    }
    const double c = fsp_block_sum(csum, sh);
    if (!(c > 0.0) || !isfinite(emax)) return false;
    ll += emax + log(c);
    const double inv = 1.0 / c;
    for (int i = tid; i < S; i += B) cur[i] *= inv;
    __syncthreads();
    return true;
}

__device__ __forceinline__ void fsp_report(const FspArgs &a, int64_t f, int status, double ll, double leak) {
    if (threadIdx.x == 0) {
        a.ll_f[f] = status == PF_ST_OK ? ll : -INFINITY;
        a.st_f[f] = static_cast<uint8_t>(status);
        if (a.leak_f) a.leak_f[f] = leak;
    }
}

// Networks whose stencil over the reachable states fits in shared memory.  The
// FP64 pipe bounds it: a product costs (inflows + 2) FMAs per state.  States
// that no sequence of reactions reaches hold probability 0 for ever, and an
// inflow whose predecessor is outside the box, unreachable or has no
// reactants is 0: neither is stored (telegraph: 122 of the box's 244 states,
// 4.5 FMAs per state instead of 6).  States are numbered by their number of
// inflows, so that a warp's lanes loop alike.
__global__ void __launch_bounds__(kFspMaxThreads) fsp_compact_kernel(const FspArgs a) {
    extern __shared__ __align__(16) double fsm[];
    __shared__ FspShared sh;
    const int S = a.Sc, E = a.E, tid = threadIdx.x, B = blockDim.x;
    const int64_t f = blockIdx.x;
    const int64_t m = f / a.T;
    const int traj = static_cast<int>(f - m * a.T);
    const double *theta = a.thetas + m * a.net.d;
    double *cur = fsm, *nxt = fsm + S, *acc = fsm + 2 * S, *wts = fsm + 3 * S;
    double *diag = wts + kFspMaxTerms, *cin = diag + S;                    // [S], [E][S]
    uint16_t *src = reinterpret_cast<uint16_t *>(cin + static_cast<size_t>(E) * S);   // [E][S]
    if (!fsp_valid(a, sh, theta, f)) return;
    double rate[PF_MAX_REACTIONS];
    for (int r = 0; r < a.net.R; ++r) rate[r] = dev::reaction_rate(a.net, theta, r);
    auto state = [&](int i, int *x) { decode(a, a.st_idx[i], x); };
    int x[PF_MAX_SPECIES];
    double amax = 0.0;
    for (int i = tid; i < S; i += B) {
        state(i, x);
        amax = fmax(amax, total_propensity(a, rate, x));
    }
    const double lambda = fsp_block_max(amax, sh);
    if (tid < a.net.R) sh.rate_s[tid] = lambda > 0.0 ? __ddiv_rn(rate[tid], lambda) : 0.0;
    __syncthreads();
    for (int i = tid; i < S; i += B) {
        state(i, x);
        double a0 = 0.0;
        for (int r = 0; r < a.net.R; ++r)
            a0 = fma(sh.rate_s[r], static_cast<double>(combos_at(a.net, r, x, 0, 0)), a0);
        diag[i] = 1.0 - a0;
        cur[i] = initial_probability(a, x);
        for (int e = 0; e < a.in_n[i]; ++e) {
            const int r = a.in_reac[e * S + i];
            src[e * S + i] = a.in_src[e * S + i];
            cin[e * S + i] = sh.rate_s[r] * static_cast<double>(combos_at(a.net, r, x, a.nu_a[r], a.nu_b[r]));
        }
    }
    __syncthreads();
    const double lconst = fsp_lconst(a);
    const int n0 = tid < S ? a.in_n[tid] : 0;      // the thread's first state, kept in registers below
    double ll = 0.0, leak = 0.0, t_prev = 0.0, lh_of = -1.0;
    int status = PF_ST_OK, jmax = 0;
    for (int k = 0; k < a.K; ++k) {
        const double dt = a.obs_times[k] - t_prev;
        if (dt > 0.0 && lambda > 0.0) {
            const int nsub = static_cast<int>(ceil(lambda * dt / kMaxLambdaH));
            const double lh = lambda * (dt / nsub);
            if (lh != lh_of) {                     // equal intervals share their weights
                jmax = poisson_weights(lh, wts);
                lh_of = lh;
            }
            __syncthreads();
            for (int sub = 0; sub < nsub; ++sub) {
                const double w0 = wts[0];
                for (int i = tid; i < S; i += B) acc[i] = w0 * cur[i];
                for (int j = 1; j <= jmax; ++j) {
                    __syncthreads();  // cur complete
                    const double wj = wts[j];
                    int n = n0;
                    for (int i = tid; i < S; i += B) {
                        if (i != tid) n = a.in_n[i];
                        double out = diag[i] * cur[i];
                        for (int e = 0; e < n; ++e) out = fma(cin[e * S + i], cur[src[e * S + i]], out);
                        nxt[i] = out;
                        acc[i] = fma(wj, out, acc[i]);
                    }
                    double *tmp = cur;
                    cur = nxt;
                    nxt = tmp;
                }
                __syncthreads();
                double *tmp = cur;  // the sum becomes the distribution
                cur = acc;
                acc = tmp;
            }
        }
        if (!fsp_observe(a, sh, S, cur, nxt, a.y + (static_cast<int64_t>(traj) * a.K + k) * a.net.P, lconst, state, ll,
                         leak)) {
            status = PF_ST_NONFINITE;
            break;
        }
        t_prev = a.obs_times[k];
    }
    fsp_report(a, f, status, ll, leak);
}

// One species: the same on a window lo..hi of the box that follows the
// probability.  After an observation the weights exp(-(y - x)^2 / 2 sigma^2)
// leave only some tens of states above 1e-300, and an interval's events spread
// them by a few hundred at that level, while the uniformization rate and so the
// number of products grow with the box's upper end.  An interval runs on the
// support widened by some states on either side; if any product leaves more
// than 1e-290 within a reaction's reach of a window edge that is not an edge of
// the box, the interval is repeated from its start with half as much again.
// What is left out is then below 1e-290 times the number of products -- the
// likelihoods that come from far tails (1e-60 and below for poor thetas) keep
// their accuracy.  Birth-death (200 thetas, 1201 states): the heaviest rows
// take 480 states and 550 products per unit of time instead of 1201 and 1250.
constexpr double kWindowEdge = 1e-290;
__global__ void __launch_bounds__(kFspMaxThreads) fsp_window_kernel(const FspArgs a) {
    extern __shared__ __align__(16) double fsm[];
    __shared__ FspShared sh;
    __shared__ int sup_lo, sup_hi, touched[2], seen;
    const int S = a.S, R = a.net.R, tid = threadIdx.x, B = blockDim.x;
    const int64_t f = blockIdx.x;
    const int64_t m = f / a.T;
    const int traj = static_cast<int>(f - m * a.T);
    const double *theta = a.thetas + m * a.net.d;
    // [S] each: the distribution at the interval's start (by state of the box),
    // two product vectors and the sum (by state of the window), the stencil
    double *dist = fsm, *va = fsm + S, *vb = fsm + 2 * S, *vs = fsm + 3 * S, *wts = fsm + 4 * S;
    double *diag = wts + kFspMaxTerms, *cin = diag + S;                    // [S], [R][S]
    if (!fsp_valid(a, sh, theta, f)) return;
    double rate[PF_MAX_REACTIONS];
    for (int r = 0; r < R; ++r) rate[r] = dev::reaction_rate(a.net, theta, r);
    for (int i = tid; i < S; i += B) dist[i] = initial_probability(a, &i);
    __syncthreads();
    const double lconst = fsp_lconst(a);
    const long long edge = __double_as_longlong(kWindowEdge);
    int grow_lo = 64, grow_hi = 64, jmax = 0;
    double ll = 0.0, leak = 0.0, t_prev = 0.0, lambda = 0.0, lh_of = -1.0;
    int status = PF_ST_OK;
    int lo = 0, n = S;                             // the window lo .. lo + n - 1
    double *fin = dist;                            // the distribution at t_k, on the window
    for (int k = 0; k < a.K; ++k) {
        const double dt = a.obs_times[k] - t_prev;
        lo = 0;
        n = S;
        fin = dist;
        if (dt > 0.0) {
            if (tid == 0) {
                sup_lo = S;
                sup_hi = -1;
            }
            __syncthreads();
            int mn = S, mx = -1;
            for (int i = tid; i < S; i += B)
                if (__double_as_longlong(dist[i]) > edge) {
                    mn = min(mn, i);
                    mx = i;
                }
            mn = __reduce_min_sync(0xFFFFFFFFu, mn);
            mx = __reduce_max_sync(0xFFFFFFFFu, mx);
            if ((tid & 31) == 0) {
                atomicMin(&sup_lo, mn);
                atomicMax(&sup_hi, mx);
            }
            __syncthreads();
            for (;;) {
                lo = max(0, sup_lo - grow_lo);
                n = min(S - 1, sup_hi + grow_hi) - lo + 1;
                // stencil on the window
                double amax = 0.0;
                for (int i = tid; i < n; i += B) {
                    const int x = lo + i;
                    amax = fmax(amax, total_propensity(a, rate, &x));
                }
                const double top = fsp_block_max(amax, sh);
                if (!(top > 0.0)) {                // nothing can happen on the support
                    lo = 0;
                    n = S;
                    break;
                }
                // a slightly larger rate serves as well: the last one is kept, and
                // with it the Poisson weights of an equal interval
                if (!(top <= lambda && lambda <= 1.2 * top)) lambda = top;
                if (tid < R) sh.rate_s[tid] = __ddiv_rn(rate[tid], lambda);
                if (tid == 0) touched[0] = touched[1] = seen = 0;
                __syncthreads();
                for (int i = tid; i < n; i += B) {
                    const int x = lo + i;
                    double a0 = 0.0;
                    for (int r = 0; r < R; ++r) {
                        a0 = fma(sh.rate_s[r], static_cast<double>(combos_at(a.net, r, &x, 0, 0)), a0);
                        const int z = x - a.off[r];
                        const bool in = sh.rate_s[r] > 0.0 && z >= lo && z < lo + n;
                        cin[r * S + i] =
                            in ? sh.rate_s[r] * static_cast<double>(combos_at(a.net, r, &x, a.nu_a[r], a.nu_b[r])) : 0.0;
                    }
                    diag[i] = 1.0 - a0;
                    va[i] = x >= sup_lo && x <= sup_hi ? dist[x] : 0.0;
                    vb[i] = 0.0;
                }
                const int nsub = static_cast<int>(ceil(lambda * dt / kMaxLambdaH));
                const double lh = lambda * (dt / nsub);
                if (lh != lh_of) {
                    jmax = poisson_weights(lh, wts);
                    lh_of = lh;
                }
                __syncthreads();
                // states whose probability tells that the window is too small
                const int first = lo > 0 ? a.reach : 0, last = lo + n < S ? n - a.reach : n;
                double *cur = va, *nxt = vb, *acc = vs;
                bool big = false;
                // a product widens the states that are not 0 by the reach: the others
                // are left out (both vectors hold 0 there)
                int from = sup_lo - lo, to = sup_hi - lo + 1;
                for (int sub = 0; sub < nsub && !big; ++sub) {
                    const double w0 = wts[0];
                    for (int i = tid; i < n; i += B) acc[i] = w0 * cur[i];
                    for (int j = 1; j <= jmax; ++j) {
                        __syncthreads();  // cur complete
                        if ((j & 31) == 1 && seen != 0) {    // written by thread 0 at (j & 31) == 0 only
                            big = true;
                            break;
                        }
                        const double wj = wts[j];
                        from = max(0, from - a.reach);
                        to = min(n, to + a.reach);
                        for (int i = from + tid; i < to; i += B) {
                            double out = diag[i] * cur[i];
                            for (int r = 0; r < R; ++r) {
                                const double c = cin[r * S + i];
                                // c >= +0: its bits are nonzero iff c != 0 (an integer test)
                                const int s = __double_as_longlong(c) != 0 ? i - a.off[r] : i;
                                out = fma(c, cur[s], out);
                            }
                            nxt[i] = out;
                            acc[i] = fma(wj, out, acc[i]);
                            if (i < first && __double_as_longlong(out) > edge) touched[0] = 1;
                            if (i >= last && __double_as_longlong(out) > edge) touched[1] = 1;
                        }
                        if ((j & 31) == 0 && tid == 0) seen = touched[0] | touched[1];
                        double *tmp = cur;
                        cur = nxt;
                        nxt = tmp;
                    }
                    __syncthreads();
                    big = big || (touched[0] | touched[1]) != 0;
                    double *tmp = cur;  // the sum becomes the distribution
                    cur = acc;
                    acc = tmp;
                }
                fin = cur;
                if (!big) break;
                if (touched[0]) grow_lo += grow_lo / 2;
                if (touched[1]) grow_hi += grow_hi / 2;
                __syncthreads();
            }
        }
        double *le = fin == va ? vb : va;
        auto state = [&](int i, int *x) { x[0] = lo + i; };
        if (!fsp_observe(a, sh, n, fin, le, a.y + (static_cast<int64_t>(traj) * a.K + k) * a.net.P, lconst, state, ll,
                         leak)) {
            status = PF_ST_NONFINITE;
            break;
        }
        if (fin != dist) {                         // back to the states of the box
            for (int i = tid; i < S; i += B) dist[i] = i >= lo && i < lo + n ? fin[i - lo] : 0.0;
            __syncthreads();
        }
        t_prev = a.obs_times[k];
    }
    fsp_report(a, f, status, ll, leak);
}

// Boxes whose stencil does not fit beside the vectors in the forms above.
__global__ void __launch_bounds__(kFspMaxThreads) fsp_kernel(const FspArgs a) {
    extern __shared__ __align__(16) double fsm[];
    __shared__ FspShared sh;
    const int S = a.S, R = a.net.R;
    const int tid = threadIdx.x, B = blockDim.x;
    const int64_t f = blockIdx.x;
    const int64_t m = f / a.T;
    const int traj = static_cast<int>(f - m * a.T);
    const double *theta = a.thetas + m * a.net.d;
    double *cur = fsm, *nxt = fsm + S, *acc = fsm + 2 * S, *wts = fsm + 3 * S;
    double *diag = wts + kFspMaxTerms, *cin = diag + S;   // [S], [R][S] when coef_smem
    if (!fsp_valid(a, sh, theta, f)) return;
    // rates, and the uniformization rate lambda = max over the box of a_0(x)
    double rate[PF_MAX_REACTIONS];
    for (int r = 0; r < R; ++r) rate[r] = dev::reaction_rate(a.net, theta, r);
    double amax = 0.0;
    int x[PF_MAX_SPECIES];
    for (int i = tid; i < S; i += B) {
        decode(a, i, x);
        amax = fmax(amax, total_propensity(a, rate, x));
    }
    const double lambda = fsp_block_max(amax, sh);
    if (tid < R) sh.rate_s[tid] = lambda > 0.0 ? __ddiv_rn(rate[tid], lambda) : 0.0;
    __syncthreads();
    // the diagonal 1 - a_0(x) / lambda, and reaction r's inflow weight (0: none)
    auto outflow = [&](const int *x) {
        double a0 = 0.0;
        for (int r = 0; r < R; ++r)
            a0 = fma(sh.rate_s[r], static_cast<double>(combos_at(a.net, r, x, 0, 0)), a0);
        return a0;
    };
    auto inflow_weight = [&](int r, const int *x) {
        const double rs = sh.rate_s[r];
        bool in = rs > 0.0;
        for (int c = 0; c < a.net.n_change[r] && in; ++c) {
            const int sp = a.net.ch_sp[r][c];
            const int z = x[sp] - a.net.ch_delta[r][c];
            in = z >= 0 && z <= a.box[sp];
        }
        return in ? rs * static_cast<double>(combos_at(a.net, r, x, a.nu_a[r], a.nu_b[r])) : 0.0;
    };
    for (int i = tid; i < S; i += B) {
        decode(a, i, x);
        cur[i] = initial_probability(a, x);
        if (a.coef_smem) {
            for (int r = 0; r < R; ++r) cin[r * S + i] = inflow_weight(r, x);
            diag[i] = 1.0 - outflow(x);
        }
    }
    __syncthreads();
    const double lconst = fsp_lconst(a);
    double ll = 0.0, leak = 0.0, t_prev = 0.0;
    int status = PF_ST_OK;
    for (int k = 0; k < a.K; ++k) {
        const double dt = a.obs_times[k] - t_prev;
        if (dt > 0.0 && lambda > 0.0) {
            const int nsub = static_cast<int>(ceil(lambda * dt / kMaxLambdaH));
            const int jmax = poisson_weights(lambda * (dt / nsub), wts);
            __syncthreads();
            for (int sub = 0; sub < nsub; ++sub) {
                const double w0 = wts[0];
                for (int i = tid; i < S; i += B) acc[i] = w0 * cur[i];
                for (int j = 1; j <= jmax; ++j) {
                    __syncthreads();  // cur complete
                    const double wj = wts[j];
                    if (a.coef_smem) {
                        for (int i = tid; i < S; i += B) {
                            double out = diag[i] * cur[i];
                            for (int r = 0; r < R; ++r) {
                                const double c = cin[r * S + i];
                                // c >= +0: its bits are nonzero iff c != 0 (an integer test)
                                const int src = __double_as_longlong(c) != 0 ? i - a.off[r] : i;
                                out = fma(c, cur[src], out);
                            }
                            nxt[i] = out;
                            acc[i] = fma(wj, out, acc[i]);
                        }
                    } else for (int i = tid; i < S; i += B) {
                        decode(a, i, x);
                        double inflow = 0.0;
                        for (int r = 0; r < R; ++r) {
                            const double c = inflow_weight(r, x);
                            if (__double_as_longlong(c) != 0) inflow = fma(c, cur[i - a.off[r]], inflow);
                        }
                        const double out = fma(cur[i], 1.0 - outflow(x), inflow);
                        nxt[i] = out;
                        acc[i] = fma(wj, out, acc[i]);
                    }
                    double *tmp = cur;
                    cur = nxt;
                    nxt = tmp;
                }
                __syncthreads();
                double *tmp = cur;  // the sum becomes the distribution
                cur = acc;
                acc = tmp;
            }
        }
        if (!fsp_observe(a, sh, S, cur, nxt, a.y + (static_cast<int64_t>(traj) * a.K + k) * a.net.P, lconst,
                         [&](int i, int *z) { decode(a, i, z); }, ll, leak)) {
            status = PF_ST_NONFINITE;
            break;
        }
        t_prev = a.obs_times[k];
    }
    fsp_report(a, f, status, ll, leak);
}

__global__ void fsp_reduce_kernel(const double *ll_f, const uint8_t *st_f, int64_t M, int T,
                                  double *loglik, uint8_t *status) {
    const int64_t m = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (m >= M) return;
    double sum = 0.0;
    int st = PF_ST_OK;
    for (int t = 0; t < T; ++t) {
        const int s = st_f[m * T + t];
        if (st == PF_ST_OK && s != PF_ST_OK) st = s;
        sum += ll_f[m * T + t];
    }
    double out = sum;
    if (st == PF_ST_INVALID_THETA) out = __longlong_as_double(0x7FF8000000000000ll);
    else if (st != PF_ST_OK) out = -INFINITY;
    loglik[m] = out;
    if (status) status[m] = static_cast<uint8_t>(st);
}

// The reachable states of the box and their inflows (fsp_compact_kernel's
// tables), from the initial states by reactions with enough reactants whose
// result stays in the box, whatever their rates.
struct Compact {
    std::vector<uint16_t> idx, src;
    std::vector<uint8_t> reac, n;
    int E = 0;
};
Compact reachable_states(const FspArgs &a) {
    const NetTables &t = a.net;
    const int S = a.S, U = t.U, R = t.R;
    auto counts = [&](int i, int *x) {
        for (int u = 0; u < U; ++u) {
            x[u] = i / a.stride[u];
            i -= x[u] * a.stride[u];
        }
    };
    // the state that reaction r takes x to, or -1
    auto next = [&](int i, const int *x, int r) {
        const int sa = t.sp_a[r], sb = t.sp_b[r];
        if ((sa >= 0 && x[sa] < t.ord_a[r]) || (sb >= 0 && x[sb] < t.ord_b[r])) return -1;
        for (int c = 0; c < t.n_change[r]; ++c) {
            const int z = x[t.ch_sp[r][c]] + t.ch_delta[r][c];
            if (z < 0 || z > a.box[t.ch_sp[r][c]]) return -1;
        }
        return i + a.off[r];
    };
    std::vector<int32_t> number(S, -1);        // reached: >= 0, later the compact number
    std::vector<int32_t> todo;
    int x[PF_MAX_SPECIES];
    for (int i = 0; i < S; ++i) {
        counts(i, x);
        bool in = true;
        for (int u = 0; u < U; ++u) in = in && x[u] >= t.x0[u] && x[u] <= t.x0_hi[u];
        if (in) {
            number[i] = 0;
            todo.push_back(i);
        }
    }
    std::vector<std::vector<std::pair<uint8_t, int32_t>>> in(S);   // (reaction, predecessor)
    for (size_t q = 0; q < todo.size(); ++q) {
        const int i = todo[q];
        counts(i, x);
        for (int r = 0; r < R; ++r) {
            const int z = next(i, x, r);
            if (z < 0) continue;
            in[z].emplace_back(static_cast<uint8_t>(r), i);
            if (number[z] < 0) {
                number[z] = 0;
                todo.push_back(z);
            }
        }
    }
    std::sort(todo.begin(), todo.end());
    std::stable_sort(todo.begin(), todo.end(), [&](int p, int q) { return in[p].size() > in[q].size(); });
    Compact c;
    const size_t Sc = todo.size();
    for (size_t i = 0; i < Sc; ++i) {
        number[todo[i]] = static_cast<int32_t>(i);
        c.E = std::max(c.E, static_cast<int>(in[todo[i]].size()));
    }
    c.idx.resize(Sc);
    c.n.resize(Sc);
    c.src.assign(Sc * c.E, 0);
    c.reac.assign(Sc * c.E, 0);
    for (size_t i = 0; i < Sc; ++i) {
        auto &v = in[todo[i]];
        std::stable_sort(v.begin(), v.end(), [](const auto &p, const auto &q) { return p.first < q.first; });
        c.idx[i] = static_cast<uint16_t>(todo[i]);
        c.n[i] = static_cast<uint8_t>(v.size());
        for (size_t e = 0; e < v.size(); ++e) {
            c.src[e * Sc + i] = static_cast<uint16_t>(number[v[e].second]);
            c.reac[e * Sc + i] = v[e].first;
        }
    }
    return c;
}

struct Buf {
    void *p = nullptr;
    cudaStream_t s = nullptr;
    ~Buf() { if (p) cudaFreeAsync(p, s); }
    cudaError_t alloc(size_t bytes, cudaStream_t st) {
        s = st;
        return bytes ? static_cast<cudaError_t>(alloc_scratch(&p, bytes, st)) : cudaSuccess;
    }
};

}  // namespace
}  // namespace pf

#define FSP_CUDA(call, what)                                          \
    do {                                                              \
        cudaError_t e_ = (call);                                      \
        if (e_ != cudaSuccess) return pf::cuda_fail(e_, what);        \
    } while (0)

extern "C" int pf_fsp_loglik(const pf_network *net, const double *thetas, int64_t M, int32_t d,
                             const int32_t *x0, const int32_t *box_max, const double *obs_times,
                             int32_t K, const double *y, int32_t T, int32_t P, const double *C,
                             const double *sigma, double *loglik, uint8_t *status,
                             const pf_fsp_options *opt) {
    using pf::fail;
    pf::clear_error();
    pf_fsp_options o{};
    if (opt) o = *opt;
    if (M < 0) return fail(PF_EINVAL, "M < 0");
    if (K < 1 || K >= (1 << 20)) return fail(PF_EINVAL, "K %d outside 1..2^20-1", K);
    if (T < 1 || T >= 4096) return fail(PF_EINVAL, "T %d outside 1..4095", T);
    if (!obs_times || !box_max) return fail(PF_EINVAL, "obs_times and box_max are required");
    if (M > 0 && (!thetas || !y || !loglik)) return fail(PF_EINVAL, "NULL array argument");
    if (M * (int64_t)T > 0x7FFFFFFFll) return fail(PF_EINVAL, "M * T must be < 2^31");
    pf::FspArgs a{};
    int rc = pf::build_tables(net, d, x0, P, C, sigma, o.model, a.net);
    if (rc) return rc;
    rc = pf::check_obs_times(obs_times, K);
    if (rc) return rc;
    const int U = a.net.U;
    int64_t S = 1;
    for (int u = 0; u < U; ++u) {
        if (box_max[u] < 0) return fail(PF_EINVAL, "box_max[%d] = %d < 0", u, box_max[u]);
        if (a.net.x0_hi[u] > box_max[u])
            return fail(PF_EINVAL, "initial count of species %d (up to %d) outside the box 0..%d", u,
                        a.net.x0_hi[u], box_max[u]);
        a.box[u] = box_max[u];
        S *= (int64_t)box_max[u] + 1;
        if (S > PF_FSP_MAX_STATES)
            return fail(PF_EINVAL, "the box has more than %d states", PF_FSP_MAX_STATES);
    }
    a.S = (int32_t)S;
    a.stride[U - 1] = 1;
    for (int u = U - 2; u >= 0; --u) a.stride[u] = a.stride[u + 1] * (a.box[u + 1] + 1);
    for (int r = 0; r < a.net.R; ++r) {
        int off = 0, nua = 0, nub = 0;
        for (int c = 0; c < a.net.n_change[r]; ++c) {
            const int sp = a.net.ch_sp[r][c], dl = a.net.ch_delta[r][c];
            off += dl * a.stride[sp];
            if (sp == a.net.sp_a[r]) nua = dl;
            if (sp == a.net.sp_b[r]) nub = dl;
        }
        a.off[r] = off;
        a.nu_a[r] = (int8_t)nua;
        a.nu_b[r] = (int8_t)nub;
    }
    if (M == 0) return PF_OK;

    cudaStream_t s = static_cast<cudaStream_t>(o.stream);
    const int64_t F = M * T;
    a.M = M; a.K = K; a.T = T;
    pf::Buf b_theta, b_times, b_y, b_ll, b_st, b_llf, b_leak, b_stf;
    const size_t n_th = sizeof(double) * (size_t)M * d, n_y = sizeof(double) * (size_t)T * K * P;
    double *d_ll = loglik;
    uint8_t *d_st = status;
    // Which kernel: one species on a box of 256 states or more runs on a window
    // of it (birth-death's 1201 states: 63-72 -> 15 ms for 200 rows), everything
    // else on the reachable states (telegraph: 17.9 -> 7.1 ms for 4096 rows);
    // what does not fit a block's shared memory in that form runs on the box.
    int dev = 0, smem_max = 0;
    FSP_CUDA(cudaGetDevice(&dev), "cudaGetDevice");
    FSP_CUDA(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev), "cudaDeviceGetAttribute");
    const size_t D = sizeof(double), room = (size_t)smem_max - 1024;
    void (*kernel)(const pf::FspArgs) = pf::fsp_kernel;
    size_t smem = D * (3 * (size_t)S + pf::kFspMaxTerms), n_run = (size_t)S;
    pf::Compact compact;
    const size_t window = D * ((5 + (size_t)a.net.R) * S + pf::kFspMaxTerms);
    if (U == 1 && S >= 256 && window <= room) {
        kernel = pf::fsp_window_kernel;
        smem = window;
        for (int r = 0; r < a.net.R; ++r) a.reach = std::max(a.reach, std::abs(a.off[r]));
    } else {
        compact = pf::reachable_states(a);
        const size_t Sc = compact.idx.size(), E = (size_t)compact.E;
        const size_t bytes = D * ((4 + E) * Sc + pf::kFspMaxTerms) + sizeof(uint16_t) * E * Sc;
        if (bytes <= room) {
            kernel = pf::fsp_compact_kernel;
            smem = bytes;
            n_run = Sc;
            a.Sc = (int32_t)Sc;
            a.E = compact.E;
        } else if (smem + D * (size_t)(a.net.R + 1) * S <= room) {
            smem += D * (size_t)(a.net.R + 1) * S;
            a.coef_smem = 1;
        }
    }
    // observation times and the compact tables: one host-to-device copy
    const size_t Sc = (size_t)a.Sc, n_src = Sc * (size_t)a.E;
    std::vector<unsigned char> tab(D * K + sizeof(uint16_t) * (Sc + n_src) + n_src + Sc);
    unsigned char *tp = tab.data();
    auto put = [&](const void *v, size_t n) {
        const size_t at = (size_t)(tp - tab.data());
        if (n) memcpy(tp, v, n);
        tp += n;
        return at;
    };
    const size_t at_t = put(obs_times, D * K);
    size_t at_idx = 0, at_src = 0, at_reac = 0, at_n = 0;
    if (Sc) {
        at_idx = put(compact.idx.data(), sizeof(uint16_t) * Sc);
        at_src = put(compact.src.data(), sizeof(uint16_t) * n_src);
        at_reac = put(compact.reac.data(), n_src);
        at_n = put(compact.n.data(), Sc);
    }
    FSP_CUDA(b_times.alloc(tab.size(), s), "alloc tables");
    FSP_CUDA(cudaMemcpyAsync(b_times.p, tab.data(), tab.size(), cudaMemcpyHostToDevice, s), "copy tables");
    const unsigned char *dt = (const unsigned char *)b_times.p;
    a.obs_times = (const double *)(dt + at_t);
    a.st_idx = (const uint16_t *)(dt + at_idx);
    a.in_src = (const uint16_t *)(dt + at_src);
    a.in_reac = dt + at_reac;
    a.in_n = dt + at_n;
    if (o.device_ptrs) {
        a.thetas = thetas;
        a.y = y;
    } else {
        FSP_CUDA(b_theta.alloc(n_th, s), "alloc thetas");
        FSP_CUDA(b_y.alloc(n_y, s), "alloc y");
        FSP_CUDA(b_ll.alloc(sizeof(double) * M, s), "alloc loglik");
        FSP_CUDA(b_st.alloc(M, s), "alloc status");
        FSP_CUDA(cudaMemcpyAsync(b_theta.p, thetas, n_th, cudaMemcpyHostToDevice, s), "copy thetas");
        FSP_CUDA(cudaMemcpyAsync(b_y.p, y, n_y, cudaMemcpyHostToDevice, s), "copy y");
        a.thetas = (const double *)b_theta.p;
        a.y = (const double *)b_y.p;
        d_ll = (double *)b_ll.p;
        d_st = (uint8_t *)b_st.p;
    }
    if (o.ll_traj && o.device_ptrs) {
        a.ll_f = o.ll_traj;
    } else {
        FSP_CUDA(b_llf.alloc(sizeof(double) * F, s), "alloc ll_traj");
        a.ll_f = (double *)b_llf.p;
    }
    if (o.leak && o.device_ptrs) {
        a.leak_f = o.leak;
    } else if (o.leak) {
        FSP_CUDA(b_leak.alloc(sizeof(double) * F, s), "alloc leak");
        a.leak_f = (double *)b_leak.p;
    }
    FSP_CUDA(b_stf.alloc(F, s), "alloc status_traj");
    a.st_f = (uint8_t *)b_stf.p;

    // a window is mostly some 500 states (birth-death: 384 threads 17.1 ms, 512 18.8, 256 20.4)
    const int most = kernel == pf::fsp_window_kernel ? 384 : pf::kFspMaxThreads;
    const int threads = std::min(most, std::max(64, (int)((n_run + 31) / 32) * 32));
    FSP_CUDA(static_cast<cudaError_t>(pf::raise_smem_limit(reinterpret_cast<const void *>(kernel))), "fsp smem attribute");
    kernel<<<(unsigned)F, threads, smem, s>>>(a);
    FSP_CUDA(cudaGetLastError(), "fsp launch");
    pf::fsp_reduce_kernel<<<(unsigned)((M + 255) / 256), 256, 0, s>>>(a.ll_f, a.st_f, M, T, d_ll, d_st);
    FSP_CUDA(cudaGetLastError(), "fsp reduce launch");
    if (!o.device_ptrs) {
        FSP_CUDA(cudaMemcpyAsync(loglik, d_ll, sizeof(double) * M, cudaMemcpyDeviceToHost, s), "copy loglik");
        if (status) FSP_CUDA(cudaMemcpyAsync(status, d_st, M, cudaMemcpyDeviceToHost, s), "copy status");
        if (o.ll_traj) FSP_CUDA(cudaMemcpyAsync(o.ll_traj, a.ll_f, sizeof(double) * F, cudaMemcpyDeviceToHost, s), "copy ll_traj");
        if (o.leak) FSP_CUDA(cudaMemcpyAsync(o.leak, a.leak_f, sizeof(double) * F, cudaMemcpyDeviceToHost, s), "copy leak");
        FSP_CUDA(cudaStreamSynchronize(s), "synchronize");
    }
    return PF_OK;
}

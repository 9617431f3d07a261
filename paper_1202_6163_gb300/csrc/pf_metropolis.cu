// Metropolis resampler (Figure 1d, Section 2).
//
// Thread i runs chain i: k = i, then B steps, each proposing j uniformly over
// all P indices and moving to it when lw_j >= lw_k or when u < exp(lw_j - lw_k).
// No sum of weights is formed, so there is no collective step and one launch
// suffices.  Each Philox-4x32-10 call supplies the (proposal, uniform) pairs of
// two consecutive steps.
//
// When the P weights fit shared memory, each CTA stages them once as
// w_i = exp(lw_i - m) (m the largest log-weight, the subtraction error-free)
// and a step accepts when u w_k < w_j: one product instead of an exponential
// per step.  Each w carries at most 2.5 ulp of error (expf's 2 ulp and one
// rounding), so the decision can differ from the exact rule only where u lies
// within 7e-7 r of r = exp(lw_j - lw_k).  A state whose weight is below 2^-100
// (zero, or too small for the product to stay a normal float) decides in log
// space from the global log-weights instead.  Larger P reads the log-weights
// through L2 (ld.global.nc), where the 4 MiB of P = 2^20 stays resident.
#include "pf_device.cuh"

namespace pf {

constexpr int kMetroThreads = 256;
constexpr int kMetroSmemFloats = 48 * 1024;  // 192 KiB staging limit
constexpr float kWeightFloor = 0x1p-100f;    // staged weights below it decide in log space

// Accept a move from k to j (log-weights lk, lj) with uniform u.
__device__ __forceinline__ bool metropolis_accept(float lj, float lk, float u) {
    if (lj >= lk) return true;  // also covers lk = -inf
    float s, e;
    two_sum(lj, -lk, s, e);
    const float x = expf(s);
    const float r = x > 0.f ? __fmaf_rn(x, e, x) : 0.f;
    return u < r;
}

// The chain's Philox stream with everything taken out of the steps that does not
// depend on the step.  Of the counter (i, step / 2, filter, tag) only one word varies, so
// the first three rounds come down to two products: round 0 multiplies i and filter,
// round 1 multiplies the step's word (xored with a constant) and a constant, round 2 a
// constant and what round 1 made of the step.  The later rounds' keys are kept in
// registers (opaque to the compiler, which otherwise forms them anew in every call: two
// additions a round).  34 instructions a call instead of about 60; a call serves two steps.
constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;

template <int ROUNDS>
struct ChainStream {
    uint32_t f0, e2, h0, j2, g3;
    uint32_t k0[ROUNDS - 3], k1[ROUNDS - 3];

    __device__ __forceinline__ void set_key(uint32_t key0, uint32_t key1) {
#pragma unroll
        for (int r = 3; r < ROUNDS; ++r) {
            k0[r - 3] = key0 + (uint32_t)r * 0x9E3779B9u;
            k1[r - 3] = key1 + (uint32_t)r * 0xBB67AE85u;
            asm volatile("" : "+r"(k0[r - 3]), "+r"(k1[r - 3]));
        }
    }
    __device__ __forceinline__ void set_chain(uint32_t i, uint32_t filter, uint32_t key0, uint32_t key1) {
        const uint64_t b0 = (uint64_t)kPhiloxM1 * filter, a0 = (uint64_t)kPhiloxM0 * i;
        f0 = (uint32_t)(b0 >> 32) ^ key0;
        const uint32_t c2 = (uint32_t)(a0 >> 32) ^ (uint32_t)TAG_METRO ^ key1;
        const uint64_t b1 = (uint64_t)kPhiloxM1 * c2;
        const uint32_t d0 = (uint32_t)(b1 >> 32) ^ (uint32_t)b0 ^ (key0 + 0x9E3779B9u);
        e2 = (uint32_t)a0 ^ (key1 + 0xBB67AE85u);
        h0 = (uint32_t)b1 ^ (key0 + 2u * 0x9E3779B9u);
        const uint64_t a2 = (uint64_t)kPhiloxM0 * d0;
        j2 = (uint32_t)(a2 >> 32) ^ (key1 + 2u * 0xBB67AE85u);
        g3 = (uint32_t)a2;
    }
    __device__ __forceinline__ u32x4 words(uint32_t half_step) const {
        const uint64_t a1 = (uint64_t)kPhiloxM0 * (f0 ^ half_step);
        const uint64_t b2 = (uint64_t)kPhiloxM1 * ((uint32_t)(a1 >> 32) ^ e2);
        uint32_t c0 = (uint32_t)(b2 >> 32) ^ h0, c1 = (uint32_t)b2, c2 = (uint32_t)a1 ^ j2, c3 = g3;
#pragma unroll
        for (int r = 0; r < ROUNDS - 3; ++r) {
            const uint64_t a = (uint64_t)kPhiloxM0 * c0, b = (uint64_t)kPhiloxM1 * c2;
            c0 = (uint32_t)(b >> 32) ^ c1 ^ k0[r];
            c1 = (uint32_t)b;
            c2 = (uint32_t)(a >> 32) ^ c3 ^ k1[r];
            c3 = (uint32_t)a;
        }
        return {c0, c1, c2, c3};
    }
};

// Proposals and uniforms of steps b0 .. b0 + kAhead - 1 (b0 even).
constexpr int kAhead = 4;

template <int ROUNDS>
__device__ __forceinline__ void draw_steps(const ChainStream<ROUNDS>& rng, int b0, uint32_t Pu, uint32_t (&jj)[kAhead],
                                           float (&uu)[kAhead]) {
#pragma unroll
    for (int q = 0; q < kAhead / 2; ++q) {
        const u32x4 r = rng.words((uint32_t)((b0 >> 1) + q));
        jj[2 * q] = draw_index(r.x, Pu);
        uu[2 * q] = u23f(r.y);
        jj[2 * q + 1] = draw_index(r.z, Pu);
        uu[2 * q + 1] = u23f(r.w);
    }
}

// A log-weight read at random.  Where the read-only path is closed (ld_input) the load stays
// where it is written: moved about by the compiler, the chain's loads took seven registers
// more, and with them a quarter of the resident warps.
template <bool RO>
__device__ __forceinline__ float read_logw(const float* p) {
    if constexpr (RO) return ld_input<true>(p);
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// B steps of a chain from state (k, lk).  The proposals do not depend on the
// chain's state, so each group of kAhead steps draws its proposals first and
// issues all their log-weight loads before resolving the steps in order.
template <int ROUNDS, bool RO>
__device__ __forceinline__ void run_chain(const float* lw, uint32_t Pu, const ChainStream<ROUNDS>& rng,
                                          int steps, uint32_t& k, float& lk) {
    for (int b0 = 0; b0 < steps; b0 += kAhead) {
        uint32_t jj[kAhead];
        float uu[kAhead], ll[kAhead];
        draw_steps(rng, b0, Pu, jj, uu);
#pragma unroll
        for (int s = 0; s < kAhead; ++s) ll[s] = read_logw<RO>(lw + jj[s]);
#pragma unroll
        for (int s = 0; s < kAhead; ++s) {
            if (b0 + s < steps && metropolis_accept(ll[s], lk, uu[s])) {
                k = jj[s];
                lk = ll[s];
            }
        }
    }
}

// A filter's staged weights: those below `held` in shared memory, the rest (SPLIT) in
// global memory.
struct StagedWeights {
    float* w;
    float* rest;    // weight of particle held + i at rest[i]
    uint32_t held;
    template <bool SPLIT>
    __device__ __forceinline__ float at(uint32_t j) const {
        if (!SPLIT || j < held) return w[j];
        return rest[j - held];
    }
};

// B steps of a chain from state k over staged weights.  CLEAN: every staged weight is
// at least kWeightFloor, so no step looks at the log-weights.  SPLIT: a filter
// beyond shared memory, whose steps decide by the rule on log-weights: the product
// decides where it is further from a tie than the weights' errors reach (7e-7
// relative, five times over), and the log-weights where it is not.
constexpr float kTieBand = 4e-6f;

template <int ROUNDS, bool CLEAN, bool SPLIT, bool RO>
__device__ __forceinline__ void run_chain_w(const float* lw, const StagedWeights& sw, uint32_t Pu,
                                            const ChainStream<ROUNDS>& rng, int steps, uint32_t& k) {
    float wk = sw.at<SPLIT>(k);
    auto step = [&](uint32_t j, float u, float wj) {
        const float t = __fmul_rn(u, wk);
        bool acc = t < wj;
        if ((!CLEAN && !(wk >= kWeightFloor)) || (SPLIT && fabsf(__fsub_rn(t, wj)) <= kTieBand * wj))
            acc = metropolis_accept(ld_input<RO>(lw + j), ld_input<RO>(lw + k), u);
        if (acc) {
            k = j;
            wk = wj;
        }
    };
    uint32_t jj[kAhead];
    float uu[kAhead], ww[kAhead];
    int b0 = 0;
    for (; b0 + kAhead <= steps; b0 += kAhead) {
        draw_steps(rng, b0, Pu, jj, uu);
#pragma unroll
        for (int s = 0; s < kAhead; ++s) ww[s] = sw.at<SPLIT>(jj[s]);
#pragma unroll
        for (int s = 0; s < kAhead; ++s) step(jj[s], uu[s], ww[s]);
    }
    if (b0 < steps) {
        draw_steps(rng, b0, Pu, jj, uu);
#pragma unroll
        for (int s = 0; s < kAhead; ++s)
            if (b0 + s < steps) step(jj[s], uu[s], sw.at<SPLIT>(jj[s]));
    }
}

// Chain i of a filter with staged weights, written to anc[i].
template <int ROUNDS, bool SPLIT, bool RO>
__device__ __forceinline__ void run_staged(const float* lw, const StagedWeights& sw, bool clean, uint32_t Pu, uint32_t i,
                                           int steps, uint32_t filter, uint32_t key0, uint32_t key1,
                                           ChainStream<ROUNDS>& rng, int32_t* anc) {
    uint32_t k = i;
    rng.set_chain(i, filter, key0, key1);
    if (clean) run_chain_w<ROUNDS, true, SPLIT, RO>(lw, sw, Pu, rng, steps, k);
    else run_chain_w<ROUNDS, false, SPLIT, RO>(lw, sw, Pu, rng, steps, k);
    anc[i] = (int32_t)k;
}

template <int ROUNDS, bool RO>
__device__ __forceinline__ void run_unstaged(const float* lw, uint32_t Pu, uint32_t i, int steps,
                                             uint32_t filter, uint32_t key0, uint32_t key1, ChainStream<ROUNDS>& rng,
                                             int32_t* anc, uint32_t* ctl) {
    uint32_t k = i;
    float lk = read_logw<RO>(lw + i);
    if (!(lk <= 3.402823466e38f)) set_status(ctl + CTL_STATUS, ST_DOMAIN);  // NaN or +inf
    rng.set_chain(i, filter, key0, key1);
    run_chain<ROUNDS, RO>(lw, Pu, rng, steps, k, lk);
    anc[i] = (int32_t)k;
}

// Block-wide: copy lw[0..n) as weights exp(lw - m), m = max lw (0 when every weight is
// zero), to shared memory and, from sw.held on, to sw.rest; records PF_ERR_DOMAIN
// for a NaN or +inf log-weight.  Returns whether every weight is at least kWeightFloor.
// Bound by the latency of its reads, as every CTA reads the whole filter: with four in flight
// and the weights formed four at a time, 20011 particles, B = 8, 6.3 us a call (7.2 one by one).
template <int THREADS, bool RO>
__device__ bool stage_weights(const float* lw, int64_t n, const StagedWeights& sw, float* red,
                              uint32_t* ctl) {
    const int tid = threadIdx.x;
    const int64_t ns = n < (int64_t)sw.held ? n : (int64_t)sw.held;  // those held in shared memory
    float m = -INFINITY;
    int bad = 0;
    auto see = [&](float x) {
        m = fmaxf(m, x);
        bad |= !(x <= 3.402823466e38f);
    };
    const int64_t n4 = (((uintptr_t)lw) & 15u) == 0 ? ns >> 2 : 0;
    constexpr int kBatch = RO ? 1 : 4;  // reads in flight per thread (RO: as many as the compiler sees fit)
    for (int64_t q0 = tid; q0 < n4; q0 += kBatch * THREADS) {
        float4 v[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
            if (q0 + u * THREADS < n4) v[u] = ld_input<RO>(reinterpret_cast<const float4*>(lw) + q0 + u * THREADS);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            if (q0 + u * THREADS < n4) {
                reinterpret_cast<float4*>(sw.w)[q0 + u * THREADS] = v[u];
                see(v[u].x);
                see(v[u].y);
                see(v[u].z);
                see(v[u].w);
            }
        }
    }
    for (int64_t q0 = 4 * n4 + tid; q0 < ns; q0 += kBatch * THREADS) {
        float x[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
            if (q0 + u * THREADS < ns) x[u] = ld_input<RO>(lw + q0 + u * THREADS);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            if (q0 + u * THREADS < ns) {
                sw.w[q0 + u * THREADS] = x[u];
                see(x[u]);
            }
        }
    }
    for (int64_t q = ns + tid; q < n; q += THREADS) see(ld_input<RO>(lw + q));
    m = warp_max(m);
    if ((tid & 31) == 0) red[tid >> 5] = m;
    bad = __syncthreads_or(bad);
    if (bad && tid == 0) set_status(ctl + CTL_STATUS, ST_DOMAIN);
    float mt = red[0];
#pragma unroll
    for (int q = 1; q < THREADS / 32; ++q) mt = fmaxf(mt, red[q]);
    const fpair R = {mt > -INFINITY ? mt : 0.f, 0.f};
    float least = INFINITY;
    for (int q = tid; q < (int)(ns >> 2); q += THREADS) {
        float4 x = reinterpret_cast<const float4*>(sw.w)[q];
        x = make_float4(weight_rel(x.x, R), weight_rel(x.y, R), weight_rel(x.z, R), weight_rel(x.w, R));
        reinterpret_cast<float4*>(sw.w)[q] = x;
        least = fminf(least, fminf(fminf(x.x, x.y), fminf(x.z, x.w)));
    }
    for (int q = (int)(ns & ~(int64_t)3) + tid; q < (int)ns; q += THREADS)
        least = fminf(least, sw.w[q] = weight_rel(sw.w[q], R));
    for (int64_t q = ns + tid; q < n; q += THREADS)
        least = fminf(least, sw.rest[q - ns] = weight_rel(ld_input<RO>(lw + q), R));
    return __syncthreads_and(least >= kWeightFloor) != 0;
}

// Block-wide: the largest normalised weight w_max = max_i w_i / sum_i w_i of
// lw[0..n) (Section 2, Eq. 5's w_max), from the staged weights w (STAGED: w_i =
// exp(lw_i - m), the largest is 1) or from the log-weights in global memory (one
// pass of running (max, sum) pairs, rescaled as the maximum grows).  Returns
// 0 when every weight is zero.  red: THREADS/32 floats of shared memory.
template <int THREADS, bool STAGED>
__device__ float largest_weight(const float* lw, const float* w, int64_t n, float* red) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float m = -INFINITY, sum = 0.f, c = 0.f;
    for (int64_t q = tid; q < n; q += THREADS) {
        if (STAGED) {
            const float y = __fsub_rn(w[q], c);  // compensated sum of the staged weights (max 1)
            const float t = __fadd_rn(sum, y);
            c = __fsub_rn(__fsub_rn(t, sum), y);
            sum = t;
        } else {
            const float x = ld_input<kReadOnly>(lw + q);
            if (x > m) {
                sum = (m > -INFINITY ? sum * expf(m - x) : 0.f) + 1.f;
                m = x;
            } else if (x > -INFINITY) {
                sum += expf(x - m);
            }
        }
    }
    if (STAGED) {
        sum = __fsub_rn(sum, c);
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) red[warp] = sum;
        __syncthreads();
        float tot = 0.f;
        for (int q = 0; q < THREADS / 32; ++q) tot += red[q];
        __syncthreads();  // red is reused
        return tot > 0.f ? 1.f / tot : 0.f;
    }
    // combine (max, sum) pairs: first the maximum, then every sum rescaled to it
    const float mw = warp_max(m);
    if (lane == 0) red[warp] = mw;
    __syncthreads();
    float M = red[0];
    for (int q = 1; q < THREADS / 32; ++q) M = fmaxf(M, red[q]);
    __syncthreads();
    float s2 = m > -INFINITY ? sum * expf(m - M) : 0.f;
    for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    if (lane == 0) red[warp] = s2;
    __syncthreads();
    float tot = 0.f;
    for (int q = 0; q < THREADS / 32; ++q) tot += red[q];
    __syncthreads();
    return (M > -INFINITY && tot > 0.f) ? 1.f / tot : 0.f;
}

// Eq. 5 (Section 2) on the device, in double precision, as pf_metropolis_B
// computes it on the host: the smallest B with lambda^B <= eps (alpha + beta) /
// max(alpha, beta), beta = 1/P, alpha = (1 - w_max)/(P w_max), lambda = 1 -
// alpha - beta; capped at cap (also for w_max = 0).
__device__ uint32_t bound_B(int64_t P, double w_max, double eps, uint32_t cap) {
    if (!(w_max > 0.0)) return cap;
    if (w_max > 1.0) w_max = 1.0;
    const double beta = 1.0 / (double)P;
    const double alpha = (1.0 - w_max) / ((double)P * w_max);
    const double lambda = 1.0 - alpha - beta;
    const double target = eps * (alpha + beta) / (alpha > beta ? alpha : beta);
    if (target >= 1.0) return 0;
    if (lambda <= 0.0) return 1;
    double b = ceil(log(target) / log(lambda));
    if (b >= 1.0 && pow(lambda, b - 1.0) <= target) b -= 1.0;
    if (!(b >= 0.0)) return cap;
    return b < (double)cap ? (uint32_t)b : cap;
}

template <bool STAGED, int ROUNDS>
__global__ void __launch_bounds__(kMetroThreads) k_metropolis(const float* lw, int64_t P, int B,
                                                              const uint32_t* B_dev, uint32_t key0, uint32_t key1,
                                                              uint32_t filter, int32_t* anc, uint32_t* ctl) {
    extern __shared__ float wsm[];
    __shared__ float red[kMetroThreads / 32];
    grid_begin();
    bool clean = false;
    const StagedWeights sw = {wsm, nullptr, 0xffffffffu};
    if (STAGED) clean = stage_weights<kMetroThreads, false>(lw, P, sw, red, ctl);  // every CTA: the whole vector
    const int steps = B_dev ? (int)*B_dev : B;
    const uint32_t Pu = (uint32_t)P;
    ChainStream<ROUNDS> rng;
    rng.set_key(key0, key1);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        if (STAGED)
            run_staged<ROUNDS, false, false>(lw, sw, clean, Pu, (uint32_t)i, steps, filter, key0, key1, rng, anc);
        else run_unstaged<ROUNDS, false>(lw, Pu, (uint32_t)i, steps, filter, key0, key1, rng, anc, ctl);
    }
}

// Once per device: allow the staged variant its full shared-memory copy.
cudaError_t prepare_metropolis() {
    cudaError_t e = cudaFuncSetAttribute(k_metropolis<true, 10>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kMetroSmemFloats * (int)sizeof(float));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_metropolis<true, 7>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kMetroSmemFloats * (int)sizeof(float));
    return e;
}

template <int ROUNDS>
static cudaError_t launch_metropolis_r(const float* lw, int64_t P, int B, const uint32_t* B_dev, uint32_t key0,
                                       uint32_t key1, uint32_t filter, int32_t* anc, uint32_t* ctl, int num_sms,
                                       cudaStream_t s) {
    const bool staged = P <= kMetroSmemFloats;
    const int64_t blocks_needed = (P + kMetroThreads - 1) / kMetroThreads;
    if (staged) {
        // every CTA stages the full vector, so keep the grid to what runs at once
        const size_t smem = (size_t)P * sizeof(float);
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_metropolis<true, ROUNDS>, kMetroThreads, smem);
        if (per_sm < 1) per_sm = 1;
        const int64_t grid = blocks_needed < (int64_t)num_sms * per_sm ? blocks_needed : (int64_t)num_sms * per_sm;
        return launch_overlapped(k_metropolis<true, ROUNDS>, (unsigned)grid, kMetroThreads, smem, s, lw, P, B, B_dev, key0,
                                 key1, filter, anc, ctl);
    } else {
        const int64_t cap = (int64_t)num_sms * 64;
        const int64_t grid = blocks_needed < cap ? blocks_needed : cap;
        return launch_overlapped(k_metropolis<false, ROUNDS>, (unsigned)grid, kMetroThreads, 0, s, lw, P, B, B_dev, key0,
                                 key1, filter, anc, ctl);
    }
}

cudaError_t launch_metropolis(const float* lw, int64_t P, int B, const uint32_t* B_dev, uint32_t key0, uint32_t key1,
                              uint32_t filter, int32_t* anc, uint32_t* ctl, int num_sms, cudaStream_t s, int rounds) {
    if (rounds == 7) return launch_metropolis_r<7>(lw, P, B, B_dev, key0, key1, filter, anc, ctl, num_sms, s);
    return launch_metropolis_r<10>(lw, P, B, B_dev, key0, key1, filter, anc, ctl, num_sms, s);
}

// ---------------------------------------------------------------------------
// Batched: each CTA takes whole filters from a ticket counter, copies the
// filter's log-weights to shared memory when they fit, and runs its chains
// (filter-local indices, Philox filter id f, key seeds[f]).  One 1024-thread
// CTA per SM stages up to 56 Ki log-weights (224 KiB): a staged chain step is
// bound by its Philox and acceptance arithmetic, an unstaged one by random
// L2 reads, which sustain fewer steps per second.
// ---------------------------------------------------------------------------
constexpr int kMetroBThreads = 1024;
constexpr int kMetroBStage = 56 * 1024;  // floats staged per CTA (224 KiB)
constexpr uint32_t kBatchedBCap = 1u << 24;  // largest step count chosen for B < 0
// A filter of up to twice the staging holds the rest of its weights in the CTA's
// scratch: its steps then cost L2 only for the proposals that fall there.  Without, the
// CTA's 32 random L2 reads a warp step bound it: 65 cycles a warp step at 65536
// particles against 13 staged and 18 split; beyond, half or more of the reads go
// to L2 either way.
constexpr int64_t kMetroBSplit = 2 * (int64_t)kMetroBStage;
static_assert(kMetroBSplit - kMetroBStage <= kMetroScratchFloats, "the CTA's scratch holds the rest");

// How a filter's weights are reached.
enum WeightsAt { kAllStaged, kSplit, kUnstaged };
__device__ __forceinline__ WeightsAt weights_at(int64_t Pf) {
    return Pf <= kMetroBStage ? kAllStaged : (Pf <= kMetroBSplit ? kSplit : kUnstaged);
}

// Chain blocks of a filter shared by several CTAs: a filter whose chains
// number more than one block and whose work P_f B_f reaches kHeavyWork steps
// is put on a list after its owner (the CTA that took its ticket) has
// published its step count; CTAs that find the ticket queue empty join the
// listed filters.  Blocks of kMetroBThreads chains are claimed through a 64-bit
// word per filter, (launch epoch, claims): a word from an earlier launch is
// replaced by the first claimer, so no pass clears the words between launches.
// Every chain depends only on (f, i, B_f), so which CTA runs it does not
// change the result.
constexpr long long kHeavyWork = 1LL << 22;

// Claims the next block of the filter's word (thread 0 only).
__device__ __forceinline__ uint32_t claim_block(unsigned long long* w, uint32_t epoch) {
    for (;;) {
        const unsigned long long old = (unsigned long long)ld_relaxed_u64(reinterpret_cast<const uint64_t*>(w));
        if ((uint32_t)(old >> 32) != epoch) {
            if (atomicCAS(w, old, ((unsigned long long)epoch << 32) | 1ull) == old) return 0u;
            continue;
        }
        return (uint32_t)atomicAdd(w, 1ull);
    }
}

// Chain i of a batched filter.
template <int ROUNDS>
__device__ __forceinline__ void run_batched_chain(const BatchParams& bp, const float* lw, const StagedWeights& sw,
                                                  WeightsAt where, bool clean, uint32_t Pu, int64_t off0, uint32_t i,
                                                  int steps, int f, uint32_t key0, uint32_t key1,
                                                  ChainStream<ROUNDS>& rng) {
    int32_t* anc = bp.anc + off0;
    const uint32_t filter = (uint32_t)f;
    if (where == kAllStaged)
        run_staged<ROUNDS, false, kReadOnly>(lw, sw, clean, Pu, i, steps, filter, key0, key1, rng, anc);
    else if (where == kSplit)
        run_staged<ROUNDS, true, kReadOnly>(lw, sw, clean, Pu, i, steps, filter, key0, key1, rng, anc);
    else
        run_unstaged<ROUNDS, kReadOnly>(lw, Pu, i, steps, filter, key0, key1, rng, anc, bp.ctl);
}

// The chains of blocks claimed from filter f (block-wide; the weights are staged).
template <int ROUNDS>
__device__ __forceinline__ void run_claimed_blocks(const BatchParams& bp, const float* lw, const StagedWeights& sw,
                                                   WeightsAt where, bool clean, int64_t Pf, int64_t off0, int steps,
                                                   int f, uint32_t epoch, uint32_t key0, uint32_t key1,
                                                   ChainStream<ROUNDS>& rng, int* blk_sm) {
    const int tid = threadIdx.x;
    const uint32_t Pu = (uint32_t)Pf;
    const int64_t nblk = (Pf + kMetroBThreads - 1) / kMetroBThreads;
    for (;;) {
        if (tid == 0) *blk_sm = (int)claim_block(bp.metro + 2 * (int64_t)f, epoch);
        __syncthreads();
        const int64_t blk = *blk_sm;
        __syncthreads();
        if (blk >= nblk) break;
        const int64_t i = blk * kMetroBThreads + tid;
        if (i < Pf)
            run_batched_chain<ROUNDS>(bp, lw, sw, where, clean, Pu, off0, (uint32_t)i, steps, f, key0, key1, rng);
    }
}

template <int ROUNDS>
__global__ void __launch_bounds__(kMetroBThreads) k_batched_metropolis(BatchParams bp) {
    extern __shared__ float wsm[];
    __shared__ int f_sm, f_B, blk_sm;
    __shared__ float red[kMetroBThreads / 32];
    const int tid = threadIdx.x;
    const int n_items = (int)ld_relaxed_u32(bp.ctl + CTL_ITEMS);
    const uint32_t epoch = ld_relaxed_u32(bp.ctl + CTL_METRO_EPOCH);
    ChainStream<ROUNDS> rng;
    const StagedWeights sw = {wsm, bp.scratch + (int64_t)blockIdx.x * bp.scratch_per_cta, (uint32_t)kMetroBStage};
    for (;;) {
        if (tid == 0) f_sm = (int)atomicAdd(bp.ctl + CTL_QUEUE, 1u);
        __syncthreads();
        const int ticket = f_sm;
        __syncthreads();
        if (ticket >= n_items) break;
        const int f = bp.items[ticket] >> 5;
        const int64_t off0 = bp.offsets[f], off1 = bp.offsets[f + 1];
        const int64_t Pf = off1 - off0;
        if (Pf <= 0 || Pf > 0x7fffffffLL) {
            if (Pf != 0 && tid == 0) set_status(bp.ctl + CTL_STATUS, ST_INVALID);
            continue;
        }
        const float* lw = bp.lw + off0;
        const WeightsAt where = weights_at(Pf);
        const bool staged = where == kAllStaged;
        if (bp.trace) {
            trace_stamp(bp.trace, bp.trace_cap, ticket, 0);
            trace_put(bp.trace, bp.trace_cap, ticket, 5, blockIdx.x);
            trace_put(bp.trace, bp.trace_cap, ticket, 6, (uint64_t)f);
            trace_put(bp.trace, bp.trace_cap, ticket, 7, (uint64_t)(bp.items[ticket] & 31));
        }
        bool clean = false;
        if (where != kUnstaged) clean = stage_weights<kMetroBThreads, kReadOnly>(lw, Pf, sw, red, bp.ctl);
        for (int w = 1; w <= 2; ++w) trace_stamp(bp.trace, bp.trace_cap, ticket, w);
        // B < 0: this filter's own step count from Eq. 5 and its largest normalised weight
        int steps = bp.B;
        if (bp.B < 0) {
            const float wmax = staged ? largest_weight<kMetroBThreads, true>(lw, wsm, Pf, red)
                                      : largest_weight<kMetroBThreads, false>(lw, wsm, Pf, red);
            if (tid == 0) {
                f_B = (int)bound_B(Pf, (double)wmax, bp.eps, kBatchedBCap);
                if (bp.B_out) bp.B_out[f] = f_B;
            }
            __syncthreads();
            steps = f_B;
        }
        trace_stamp(bp.trace, bp.trace_cap, ticket, 3);
        const uint64_t seed = bp.seeds[f];
        const uint32_t key0 = (uint32_t)(seed & 0xffffffffu), key1 = (uint32_t)(seed >> 32);
        const uint32_t Pu = (uint32_t)Pf;
        rng.set_key(key0, key1);
        const bool heavy = bp.metro != nullptr && Pf > kMetroBThreads && Pf * (long long)max(steps, 1) >= kHeavyWork;
        if (heavy) {
            // publish the step count, then list the filter for CTAs with nothing left to take
            if (tid == 0) {
                st_release_u64(reinterpret_cast<uint64_t*>(bp.metro + 2 * (int64_t)f + 1),
                               ((uint64_t)epoch << 32) | (uint32_t)steps);
                const uint32_t h = atomicAdd(bp.ctl + CTL_HEAVY, 1u);
                if (h < (uint32_t)kMaxHeavy) {  // the list lives after the items (scratch the plan cleared)
                    int32_t* list = const_cast<int32_t*>(bp.items) + bp.F;
                    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(list + h), "r"(f + 1) : "memory");
                }
            }
            run_claimed_blocks<ROUNDS>(bp, lw, sw, where, clean, Pf, off0, steps, f, epoch, key0, key1, rng, &blk_sm);
        } else {
            for (int64_t i = tid; i < Pf; i += kMetroBThreads)
                run_batched_chain<ROUNDS>(bp, lw, sw, where, clean, Pu, off0, (uint32_t)i, steps, f, key0, key1, rng);
        }
        __syncthreads();  // the staging buffer is reused by the next filter
        trace_stamp(bp.trace, bp.trace_cap, ticket, 4);
    }
    // the queue is empty: join the listed filters that still have unclaimed blocks
    if (bp.metro != nullptr) {
        const uint64_t t_start = global_ns();
        for (int h = 0;; ++h) {
            if (tid == 0) {
                const int H = (int)min(ld_acquire_u32(bp.ctl + CTL_HEAVY), (uint32_t)kMaxHeavy);
                int f = -1;
                if (h < H) {
                    // the owner lists the filter right after counting it: wait (bounded) for the entry
                    for (uint32_t it = 0;; ++it) {
                        const uint32_t e = ld_acquire_u32(reinterpret_cast<const uint32_t*>(bp.items + bp.F + h));
                        if (e != 0u) {
                            f = (int)e - 1;
                            break;
                        }
                        if ((it & 63u) == 63u && global_ns() - t_start > bp.wait_ns) break;
                    }
                }
                f_sm = h < H ? f : -2;
                if (f >= 0) {
                    const uint64_t pw = ld_acquire_u64(reinterpret_cast<const uint64_t*>(bp.metro + 2 * (int64_t)f + 1));
                    const uint64_t cw = ld_relaxed_u64(reinterpret_cast<const uint64_t*>(bp.metro + 2 * (int64_t)f));
                    const int64_t nblk = (bp.offsets[f + 1] - bp.offsets[f] + kMetroBThreads - 1) / kMetroBThreads;
                    const bool done = (uint32_t)(cw >> 32) == epoch && (int64_t)(uint32_t)cw >= nblk;
                    if ((uint32_t)(pw >> 32) != epoch || done) f_sm = -1;  // nothing to join here
                    else f_B = (int)(uint32_t)pw;
                }
            }
            __syncthreads();
            const int f = f_sm;
            const int steps = f_B;
            __syncthreads();
            if (f == -2) break;  // past the end of the list
            if (f < 0) continue;
            const int64_t off0 = bp.offsets[f];
            const int64_t Pf = bp.offsets[f + 1] - off0;
            const float* lw = bp.lw + off0;
            const WeightsAt where = weights_at(Pf);
            bool clean = false;
            if (where != kUnstaged) clean = stage_weights<kMetroBThreads, kReadOnly>(lw, Pf, sw, red, bp.ctl);
            const uint64_t seed = bp.seeds[f];
            const uint32_t key0 = (uint32_t)(seed & 0xffffffffu), key1 = (uint32_t)(seed >> 32);
            rng.set_key(key0, key1);
            run_claimed_blocks<ROUNDS>(bp, lw, sw, where, clean, Pf, off0, steps, f, epoch, key0, key1, rng, &blk_sm);
            __syncthreads();  // the staging buffer is reused by the next listed filter
        }
    }
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(bp.ctl + CTL_QUEUE_DONE, 1u) == gridDim.x - 1) {
            atomicExch(bp.ctl + CTL_QUEUE, 0u);
            atomicExch(bp.ctl + CTL_QUEUE_DONE, 0u);
        }
    }
}

int batched_metropolis_blocks_per_sm() {
    const size_t smem = kMetroBStage * sizeof(float);
    int nb10 = 0, nb7 = 0;
    if (cudaFuncSetAttribute(k_batched_metropolis<10>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
            cudaSuccess ||
        cudaFuncSetAttribute(k_batched_metropolis<7>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
            cudaSuccess)
        return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb10, k_batched_metropolis<10>, kMetroBThreads, smem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb7, k_batched_metropolis<7>, kMetroBThreads, smem) !=
            cudaSuccess)
        return 0;
    return nb10 < nb7 ? nb10 : nb7;
}

cudaError_t launch_batched_metropolis(const BatchParams& bp, int grid, cudaStream_t s) {
    if (bp.rounds == 7)
        k_batched_metropolis<7><<<grid, kMetroBThreads, kMetroBStage * sizeof(float), s>>>(bp);
    else
        k_batched_metropolis<10><<<grid, kMetroBThreads, kMetroBStage * sizeof(float), s>>>(bp);
    return cudaGetLastError();
}

}  // namespace pf

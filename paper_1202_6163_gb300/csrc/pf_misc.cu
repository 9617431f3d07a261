// Ancestor gather (Section 1, step 4) and the weight reduction behind the
// effective sample size (Section 3) and the device-side choice of the
// Metropolis step count (Section 2, Eqs. 1-5).
#include <climits>

#include "pf_fixed.cuh"
#include "pf_rows.cuh"

namespace pf {

// ---------------------------------------------------------------------------
// Gather: dst row j <- src row anc[j].  One thread moves U chunks of VT, adjacent
// blocks of a CTA's threads, issuing all loads before the stores so that several
// random row reads are in flight; the next piece's ancestors are asked for while a piece
// is on its way.  Bound by DRAM writes and the latency of the row reads.  Rows of a
// multiple of 32 bytes move in 256-bit accesses, two a thread: systematic ancestors of
// N(0,1) log-weights, 2^24 rows of 32 bytes 161 us, 2^22 rows of 64 bytes 76 us, of 128
// bytes 128 us, against 170, 81 and 146 for four 128-bit chunks a thread spaced a grid apart.
// The fewer CTAs stride over the chunks the better, down to what covers the latency (the
// waves in launch_gather): with eight of them per SM for every type 2^24 rows of 4 and 12
// bytes took 44 and 145 us, now 34 and 87; 3000017 random rows of 16 bytes 21.0, now 18.8, of
// 68 bytes 155, now 95.
// ---------------------------------------------------------------------------
constexpr int kGatherThreads = 256;

// CTAs per SM that the registers must leave room for (0: as they fall): 256-bit chunks come out two
// registers above six CTAs otherwise.
template <typename VT, typename Place>
constexpr int gather_ctas() {
    return sizeof(VT) == 32 && sizeof(Place) == 4 ? 6 : 0;
}

template <typename VT, int U, bool POW2, typename Place = uint32_t>  // Place: as RowSplit
__global__ void __launch_bounds__(kGatherThreads, gather_ctas<VT, Place>())
    k_gather(const VT* src, int64_t P_src, RowSplit split, const int32_t* anc, int64_t total, VT* dst, uint32_t* ctl) {
    grid_begin();
    const int64_t stride = (int64_t)gridDim.x * (kGatherThreads * U);
    int64_t base = (int64_t)blockIdx.x * (kGatherThreads * U) + threadIdx.x;
    int32_t a[U];  // this piece's ancestors, and (POW2: formed anew) the chunks' places in their rows
    Place c[U] = {};
    auto ancestors = [&](int64_t b, int32_t (&e)[U], Place (&at)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = b + u * kGatherThreads;
            e[u] = 0;
            at[u] = 0;
            if (i < total) e[u] = anc[split.row<POW2>(i, at[u])];
        }
    };
    auto place = [&](int u) -> Place {
        return POW2 ? (Place)((base + u * kGatherThreads) & (split.vecs - 1)) : c[u];
    };
    ancestors(base, a, c);
    for (; base < total; base += stride) {
        VT v[U];
        bool ok[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            // an ancestor in range by one unsigned comparison (negative ones wrap beyond every P_src): 20011
            // rows of 16 bytes 1.87 us with two signed ones, so 1.68; beside the 256-bit loads it spills
            // (2^20 rows of 32 bytes 6.8 us, so 8.3)
            if constexpr (sizeof(VT) == 32)
                ok[u] = base + u * kGatherThreads < total && a[u] >= 0 && a[u] < P_src;
            else
                ok[u] = base + u * kGatherThreads < total && (uint64_t)(int64_t)a[u] < (uint64_t)P_src;
            if (ok[u]) v[u] = load_chunk(src + (int64_t)a[u] * split.vecs + place(u));
        }
        int32_t an[U];
        Place cn[U];
        ancestors(base + stride, an, cn);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (ok[u]) store_chunk_cs(dst + base + u * kGatherThreads, v[u]);
            else if (base + u * kGatherThreads < total && place(u) == 0) set_status(ctl + CTL_STATUS, ST_INVALID);
            a[u] = an[u];
            c[u] = cn[u];
        }
    }
}

template <typename VT, int U>
static cudaError_t gather_vt(const void* src, int64_t P_src, int64_t row_bytes, const int32_t* anc, int64_t P_dst,
                             void* dst, uint32_t* ctl, int num_sms, cudaStream_t s, int wave, int from = 8,
                             int full = 40) {
    const int64_t vecs = row_bytes / (int64_t)sizeof(VT);
    const int64_t total = P_dst * vecs;
    const RowSplit split = row_split(vecs, total);
    const unsigned blocks = chunk_grid(total, kGatherThreads * U, num_sms, wave, full, from);
    return launch_overlapped(split.wide()   ? k_gather<VT, U, false, uint64_t>
                             : split.pow2 ? k_gather<VT, U, true>
                                          : k_gather<VT, U, false>,
                             blocks, kGatherThreads, 0, s, (const VT*)src, P_src, split, anc, total, (VT*)dst, ctl);
}

cudaError_t launch_gather(const void* src, int64_t P_src, int64_t row_bytes, const int32_t* anc, int64_t P_dst,
                          void* dst, uint32_t* ctl, int num_sms, cudaStream_t s) {
    const uintptr_t a = (uintptr_t)src | (uintptr_t)dst | (uintptr_t)row_bytes;
    // CTAs per SM of a wave.  us with more of them: 2^22 random rows of 16 bytes, eight 31.5 and five
    // 27.8 (rows of 48 bytes, whose kernel leaves room for four at a time, need the eight: 2^20 of
    // them 13.3 and 16.0); 2^20 sorted rows of 64 bytes, eight 18.8 and six 18.1; 2^22 random rows
    // of 8 bytes 21.8 and 20.3; 2^24 sorted rows of 4 bytes 42 and 34.
    constexpr int kNever = 1 << 22;  // one resident wave however many pieces there are
    if ((a & 31) == 0) return gather_vt<u32x8, 2>(src, P_src, row_bytes, anc, P_dst, dst, ctl, num_sms, s, 6);
    if ((a & 15) == 0) {
        const int wave = (row_bytes & (row_bytes - 1)) == 0 ? 5 : 8;
        return gather_vt<uint4, 4>(src, P_src, row_bytes, anc, P_dst, dst, ctl, num_sms, s, wave);
    }
    if ((a & 7) == 0) return gather_vt<uint2, 4>(src, P_src, row_bytes, anc, P_dst, dst, ctl, num_sms, s, 6);
    return gather_vt<uint32_t, 4>(src, P_src, row_bytes, anc, P_dst, dst, ctl, num_sms, s, 6, 6, kNever);
}

// ---------------------------------------------------------------------------
// Weight reduction: per tile (k_t, sum w, sum w^2, max lw) with weights taken
// relative to 2^k_t; the last CTA to finish combines the tiles in index order
// in FP64 and writes ESS = (sum w)^2 / sum w^2, log sum exp(lw), and, when
// asked, the Metropolis step bound of Eq. 5 for the actual w_max.
// ---------------------------------------------------------------------------
constexpr int kRedThreads = 256;
constexpr int kRedPerThread = 16;
constexpr int kRedTile = kRedThreads * kRedPerThread;

struct RedRecord {  // 32 bytes, read back as two 16-byte halves
    int32_t k;
    float m;
    float s_hi, s_lo, q_hi, q_lo;
    uint32_t bad, pad;
};
static_assert(sizeof(RedRecord) == 32, "record layout");

__device__ __forceinline__ void kahan_add(float& s, float& c, float w) {
    const float y = __fsub_rn(w, c);
    const float t = __fadd_rn(s, y);
    c = __fsub_rn(__fsub_rn(t, s), y);
    s = t;
}

__device__ __forceinline__ i128 shfl_xor_i128(i128 v, int o) {
    const unsigned long long lo = (unsigned long long)v, hi = (unsigned long long)(v >> 64);
    const unsigned long long l2 = __shfl_xor_sync(0xffffffffu, lo, o);
    const unsigned long long h2 = __shfl_xor_sync(0xffffffffu, hi, o);
    return (i128)(((unsigned __int128)h2 << 64) | l2);
}

__global__ void __launch_bounds__(kRedThreads) k_reduce(const float* lw, int64_t P, RedRecord* rec,
                                                        uint32_t* ctl, float* ess_out, double* log_sum_out,
                                                        uint32_t* B_out, double eps, uint32_t B_cap) {
    __shared__ float rm[kRedThreads / 32];
    __shared__ fpair rs[kRedThreads / 32], rq[kRedThreads / 32];
    __shared__ int rk[kRedThreads / 32];
    __shared__ i128 rS[kRedThreads / 32], rQ[kRedThreads / 32];
    __shared__ int last;
    grid_begin();
    const float eps_f = (float)eps;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t t0 = (int64_t)blockIdx.x * kRedTile;
    const int n = (int)min((int64_t)kRedTile, P - t0);
    const float* base = lw + t0;

    float x[kRedPerThread];
#pragma unroll
    for (int q = 0; q < kRedPerThread / 4; ++q) {
        // coalesced: thread tid reads vector q*kRedThreads + tid
        const int e = 4 * (q * kRedThreads + tid);
        if (e + 3 < n) {
            const float4 v = *reinterpret_cast<const float4*>(base + e);
            x[4 * q] = v.x;
            x[4 * q + 1] = v.y;
            x[4 * q + 2] = v.z;
            x[4 * q + 3] = v.w;
        } else {
#pragma unroll
            for (int r = 0; r < 4; ++r) x[4 * q + r] = (e + r < n) ? base[e + r] : -INFINITY;
        }
    }
    float m = -INFINITY;
    int bad = 0;
#pragma unroll
    for (int i = 0; i < kRedPerThread; ++i) {
        bad |= !(x[i] <= 3.402823466e38f);
        m = fmaxf(m, x[i]);
    }
    m = warp_max(m);
    if (lane == 0) rm[warp] = m;
    bad = __syncthreads_or(bad);
    float mt = rm[0];
#pragma unroll
    for (int w = 1; w < kRedThreads / 32; ++w) mt = fmaxf(mt, rm[w]);
    const int k = tile_exponent(mt);
    const fpair R = tile_reference(k);
    float s = 0.f, sc = 0.f, q = 0.f, qc = 0.f;
#pragma unroll
    for (int i = 0; i < kRedPerThread; ++i) {
        const float w = weight_rel(x[i], R);
        kahan_add(s, sc, w);
        kahan_add(q, qc, w * w);
    }
    fpair ps = {s, -sc}, pq = {q, -qc};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ps = pair_add(ps, {__shfl_xor_sync(0xffffffffu, ps.hi, o), __shfl_xor_sync(0xffffffffu, ps.lo, o)});
        pq = pair_add(pq, {__shfl_xor_sync(0xffffffffu, pq.hi, o), __shfl_xor_sync(0xffffffffu, pq.lo, o)});
    }
    if (lane == 0) {
        rs[warp] = ps;
        rq[warp] = pq;
    }
    __syncthreads();
    if (tid == 0) {
        fpair S = rs[0], Q = rq[0];
        for (int w = 1; w < kRedThreads / 32; ++w) {
            S = pair_add(S, rs[w]);
            Q = pair_add(Q, rq[w]);
        }
        RedRecord r;
        r.k = k;
        r.m = mt;
        r.s_hi = S.hi;
        r.s_lo = S.lo;
        r.q_hi = Q.hi;
        r.q_lo = Q.lo;
        r.bad = bad;
        r.pad = 0;
        rec[blockIdx.x] = r;
        __threadfence();
        const uint32_t prev = atomicAdd(ctl + CTL_ESS_COUNT, 1u);
        last = (prev == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // last CTA: combine all tiles (exact fixed-point sums, all threads)
    const int T = gridDim.x;
    int kmax = INT_MIN, anybad = 0;
    float mmax = -INFINITY;
    // each record as two 16-byte loads; the first one a thread reads stays in
    // registers for the second pass (the only one when T <= kRedThreads)
    const uint32_t* rw = reinterpret_cast<const uint32_t*>(rec);
    uint4 r0 = make_uint4(0, 0, 0, 0), r1 = make_uint4(0, 0, 0, 0);
    for (int t = tid; t < T; t += kRedThreads) {
        const uint4 a = ld_cg_v4_u32(rw + 8 * t), b = ld_cg_v4_u32(rw + 8 * t + 4);
        if (t == tid) {
            r0 = a;
            r1 = b;
        }
        anybad |= (int)b.z;
        if (__uint_as_float(a.z) > 0.f) kmax = max(kmax, (int)a.x);
        mmax = fmaxf(mmax, __uint_as_float(a.y));
    }
    kmax = warp_max_i(kmax);
    mmax = warp_max(mmax);
    if (lane == 0) {
        rk[warp] = kmax;
        rm[warp] = mmax;
    }
    anybad = __syncthreads_or(anybad);
    int K = rk[0];
    float M = rm[0];
#pragma unroll
    for (int w = 1; w < kRedThreads / 32; ++w) {
        K = max(K, rk[w]);
        M = fmaxf(M, rm[w]);
    }
    if (anybad || K == INT_MIN) {
        if (tid == 0) {
            set_status(ctl + CTL_STATUS, ST_DOMAIN);
            if (ess_out) *ess_out = NAN;
            if (log_sum_out) *log_sum_out = NAN;
            if (B_out) *B_out = 0;
            ctl[CTL_ESS_COUNT] = 0;
        }
        return;
    }
    i128 S = 0, Q = 0;
    for (int t = tid; t < T; t += kRedThreads) {
        uint4 a = r0, b = r1;
        if (t != tid) {
            a = ld_cg_v4_u32(rw + 8 * t);
            b = ld_cg_v4_u32(rw + 8 * t + 4);
        }
        const int sh = (int)a.x - K;
        S += fixed_of(__uint_as_float(a.z), sh) + fixed_of(__uint_as_float(a.w), sh);
        Q += fixed_of(__uint_as_float(b.x), 2 * sh) + fixed_of(__uint_as_float(b.y), 2 * sh);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        S += shfl_xor_i128(S, o);
        Q += shfl_xor_i128(Q, o);
    }
    if (lane == 0) {
        rS[warp] = S;
        rQ[warp] = Q;
    }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < kRedThreads / 32; ++w) {
            S += rS[w];
            Q += rQ[w];
        }
        const fpair Sp = fixed_to_pair(S), Qp = fixed_to_pair(Q);
        // ESS = S^2 / Q in float (first order in the low parts)
        const float ratio = Sp.hi * (Sp.hi / Qp.hi);
        const float corr = 2.f * (Sp.lo / Sp.hi) - Qp.lo / Qp.hi;
        if (ess_out) *ess_out = __fmaf_rn(ratio, corr, ratio);
        // log sum exp(lw) = K ln 2 + log S
        const float logS = logf(Sp.hi) + Sp.lo / Sp.hi;
        const double log_sum = (double)K * kLn2 + (double)logS;
        if (log_sum_out) *log_sum_out = log_sum;
        if (B_out) {
            // Eq. 5 with the actual largest normalised weight
            const float ls = (float)((double)K * kLn2 - (double)M) + logS;  // log W - m
            const float w_max = fminf(1.f, expf(-ls));
            float b;
            if (!(w_max > 0.f)) {
                b = (float)B_cap;
            } else {
                const float beta = 1.f / (float)P;
                const float alpha = (1.f - w_max) / ((float)P * w_max);
                const float target = eps_f * (alpha + beta) / fmaxf(alpha, beta);
                if (target >= 1.f) b = 0.f;
                else b = ceilf(logf(target) / log1pf(-(alpha + beta)));
            }
            if (!(b >= 0.f)) b = (float)B_cap;
            *B_out = (uint32_t)fminf(b, (float)B_cap);
        }
        ctl[CTL_ESS_COUNT] = 0;  // ready for the next reduction on this stream
    }
}

// ---------------------------------------------------------------------------
// Diagnostic: the rate of random 4-byte reads from a buffer held in L2, the
// ceiling of the Metropolis resampler at P of a few million (its chains read
// one random log-weight per step).  Each thread makes `reads` independent
// reads at hashed indices, eight in flight.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t probe_hash(uint32_t x) {
    x ^= x >> 16;
    x *= 0x7feb352du;
    x ^= x >> 15;
    x *= 0x846ca68bu;
    x ^= x >> 16;
    return x;
}

__global__ void __launch_bounds__(256) k_probe_l2(const float* __restrict__ buf, uint32_t n, int reads, float* sink) {
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    float acc = 0.f;
    for (int l = 0; l < reads; l += 8) {
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = __ldg(buf + __umulhi(probe_hash(t * 977u + (uint32_t)(l + q) * 131071u), n));
#pragma unroll
        for (int q = 0; q < 8; ++q) acc += v[q];
    }
    if (acc == -1.2345e38f) sink[0] = acc;  // keeps the loads; never true for finite data
}

cudaError_t probe_l2_random_reads(const float* buf, int64_t n, int reads, int num_sms, double* rate) {
    if (n < 1 || n > 0xffffffffLL || reads < 8) return cudaErrorInvalidValue;
    const int blocks = num_sms * 16;
    cudaEvent_t a, b;
    cudaError_t e = cudaEventCreate(&a);
    if (e != cudaSuccess) return e;
    e = cudaEventCreate(&b);
    if (e != cudaSuccess) return e;
    float* sink = const_cast<float*>(buf);
    k_probe_l2<<<blocks, 256>>>(buf, (uint32_t)n, reads, sink);  // warm L2
    cudaEventRecord(a);
    for (int r = 0; r < 5; ++r) k_probe_l2<<<blocks, 256>>>(buf, (uint32_t)n, reads, sink);
    cudaEventRecord(b);
    e = cudaEventSynchronize(b);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (e != cudaSuccess) return e;
    *rate = 5.0 * blocks * 256.0 * (reads & ~7) / (ms * 1e-3);
    return cudaGetLastError();
}

// Diagnostic: the tile weights the scans use, out[i] = exp(lw[i] - k ln 2).
__global__ void k_tile_weights(const float* __restrict__ lw, int64_t n, int k, float* __restrict__ out) {
    const fpair R = tile_reference(k);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = weight_rel(lw[i], R);
}

cudaError_t launch_tile_weights(const float* lw, int64_t n, int k, float* out, cudaStream_t s) {
    const int64_t blocks = (n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096;
    k_tile_weights<<<(unsigned)(blocks > 0 ? blocks : 1), 256, 0, s>>>(lw, n, k, out);
    return cudaGetLastError();
}

int reduce_tiles(int64_t P) { return (int)((P + kRedTile - 1) / kRedTile); }
size_t reduce_record_bytes() { return sizeof(RedRecord); }

cudaError_t launch_reduce(const float* lw, int64_t P, void* rec, uint32_t* ctl, float* ess_out, double* log_sum_out,
                          uint32_t* B_out, double eps, uint32_t B_cap, cudaStream_t s) {
    return launch_overlapped(k_reduce, reduce_tiles(P), kRedThreads, 0, s, lw, P, (RedRecord*)rec, ctl, ess_out,
                             log_sum_out, B_out, eps, B_cap);
}

}  // namespace pf

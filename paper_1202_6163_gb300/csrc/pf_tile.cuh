// Tile scan: the per-tile half of the collective prefix sum of weights
// (Section 2: multinomial, stratified and systematic resamplers need the
// cumulative weights c_i).
//
// One CTA of kThreads threads owns a tile of n <= kTileMax consecutive
// log-weights.  Thread k holds K consecutive elements (K in {4, 8, 16}) in
// registers, loaded with 128-bit accesses.  The tile:
//   1. finds its largest log-weight m_t and exponent k_t ~ m_t log2 e;
//   2. forms w_i = exp(lw_i - k_t ln 2) with an error-free subtraction;
//   3. runs a Kahan-compensated serial scan per thread and an exact block scan
//      of the per-thread totals in 64-bit fixed point;
//   4. leaves in registers the tile-local inclusive cumulative weights v_i
//      (float, monotone across threads) and a bit mask of the elements with
//      positive weight.
//
// Bound by instruction issue (the exponential's and the compensated sum's serial
// arithmetic), so the weights are formed two at a time in packed single precision,
// threads without a zero weight skip the zero handling, and the 64-bit fixed-point
// conversions are built from 32-bit ones (the 64-bit ones run on the FP64 pipe, 16
// cycles a warp).  P = 2^25 + 4096, the scan launch of pf_large.cu: 96 -> 77 us, 55.8 ->
// 43.9 M warp instructions, with the same bits; the floor of its 8 bytes per particle is 40 us.
#pragma once

#include "pf_device.cuh"

namespace pf {

constexpr int kWarps = kThreads / 32;

struct TileShared {
    long long wtot[kWarps];  // per-warp sums of the thread totals (fixed point)
    float redf[kWarps];
    int wlast[kWarps];  // per-warp last positive element
};

struct TileSummary {
    int k;        // tile exponent
    fpair S;      // tile sum relative to 2^k (compensated pair); thread 0 only
    int i_last;   // tile-local index of the last positive weight, -1 if none
    int bad;      // a NaN or +inf log-weight was seen
    long long total;  // tile sum in fixed point (2^-48 relative to 2^k)
};

// This thread's share of the tile.
struct TileThread {
    float v[kMaxPerThread];  // tile-local inclusive cumulative weight of element e0 + i
    float base;              // that of element e0 - 1 (0 for e0 = 0)
    uint32_t pos;            // bit i: element e0 + i has positive weight
    int K;                   // elements per thread
    int e0;                  // first tile-local element of this thread
};

__device__ __forceinline__ int per_thread_count(int n) {
    const int q = (n + kThreads - 1) / kThreads;
    return q <= 4 ? 4 : (q <= 8 ? 8 : 16);
}

__device__ __forceinline__ bool zero_flag(float v) { return __float_as_uint(v) >> 31; }

// A tile staged in shared memory (16 elements per thread): 16-byte chunk (t, q), the
// q-th of thread t's four, lies at place (q + t / 2) mod 4 of the thread's 64 bytes, so
// that eight neighbouring threads' reads of their q-th chunks meet no bank conflict
// (in plain order they meet four-way ones).
__device__ __forceinline__ int stage_place(int t, int q) { return 16 * t + 4 * ((q + (t >> 1)) & 3); }

// Block-wide: this CTA's asynchronous copies of the whole 16-byte chunks of src[0..n) (src 16-byte
// aligned) into buf, as one group per thread; the caller waits for the group and meets a barrier.
__device__ __forceinline__ void stage_tile(const float* src, int n, float* buf) {
    const int c0 = threadIdx.x;  // chunk q kThreads + c0: coalesced
    float* to = buf + stage_place(c0 >> 2, c0 & 3);
    const float* from = src + 4 * c0;
#pragma unroll
    for (int q = 0; q < kMaxPerThread / 4; ++q)
        if (n == kTileMax || 4 * (q * kThreads + c0) + 3 < n)
            async_copy16(to + q * kThreads * 4, from + q * kThreads * 4);
    async_commit();
}
static_assert((kThreads / 4) % 8 == 0, "chunks a CTA apart have the same place");

// Loads this thread's KK elements (tile-local e0 .. e0+KK) of base[lo..n);
// base is 16-byte aligned in global memory, or (SMEM) a tile staged by stage_tile.
// Slots outside [lo, n) read as -inf (zero weight).
template <int KK, bool SMEM = false, bool RO = false>
__device__ __forceinline__ void tile_load_k(const float* base, int lo, int n, int e0,
                                            float (&x)[kMaxPerThread]) {
    static_assert(!SMEM || KK == kMaxPerThread, "tiles are staged in full");
    if (e0 >= lo && e0 + KK <= n) {  // nearly every thread
#pragma unroll
        for (int q = 0; q < KK / 4; ++q) {
            const float4 v = SMEM ? *reinterpret_cast<const float4*>(base + stage_place(threadIdx.x, q))
                                  : ld_input<RO>(reinterpret_cast<const float4*>(base + e0 + 4 * q));
            x[4 * q + 0] = v.x;
            x[4 * q + 1] = v.y;
            x[4 * q + 2] = v.z;
            x[4 * q + 3] = v.w;
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < KK; ++i) {
        const float* src = SMEM ? base + stage_place(threadIdx.x, i >> 2) + (i & 3) : base + e0 + i;
        x[i] = (e0 + i >= lo && e0 + i < n) ? (SMEM ? *src : ld_input<RO>(src)) : -INFINITY;
    }
}

// A tile's sum as a pair, from its fixed-point total.
__device__ __forceinline__ fpair tile_sum_pair(long long total) {
    const float hi = (float)total;
    return {hi * 0x1p-48f, (float)(total - (long long)hi) * 0x1p-48f};
}

// Block-wide; every thread of the CTA must call it.  Scans base[0..n) with the
// first `lo` slots taken as zero weights; fills th (this thread's elements) and
// returns the tile summary (identical in every thread, but S in thread 0 alone).
// KK elements per thread (n <= KK * kThreads); tile_scan picks KK from n.  RO: as ld_input.
template <int KK, bool SMEM = false, bool RO = false>  // SMEM: base is a copy of the tile in shared memory
__device__ __forceinline__ TileSummary tile_scan_k(const float* base, int lo, int n, TileShared& sm,
                                                   TileThread& th) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int e0 = tid * KK;
    th.K = KK;
    th.e0 = e0;

    float* x = th.v;
    tile_load_k<KK, SMEM, RO>(base, lo, n, e0, th.v);

    // 1. tile maximum and domain check: the maxima propagate NaN (which the
    // integer reduction places above +inf), so the tile's maximum alone tells
    // whether the tile holds a NaN or +inf
    float m = fmax_nan(x[0], x[1]);
#pragma unroll
    for (int i = 2; i < KK; i += 2) m = fmax3_nan(m, x[i], x[i + 1]);
    m = warp_max_redux(m);
    if (lane == 0) sm.redf[warp] = m;
    __syncthreads();
    const float mt = warp_max_redux(lane < kWarps ? sm.redf[lane] : -INFINITY);
    const int bad = !(mt <= 3.402823466e38f);
    const int k = tile_exponent(mt);
    const fpair R = tile_reference(k);

    // 2. weights, two at a time; a thread all of whose weights are positive (the
    // minimum propagates the NaN of a zero weight) skips the zero handling
    const float2 nhi = make_float2(-R.hi, -R.hi), nlo = make_float2(-R.lo, -R.lo);
    float mn;
#pragma unroll
    for (int i = 0; i < KK; i += 2) {
        const float2 w = weight_rel2(make_float2(x[i], x[i + 1]), nhi, nlo);
        x[i] = w.x;
        x[i + 1] = w.y;
        mn = i ? fmin3_nan(mn, w.x, w.y) : fmin3_nan(w.x, w.x, w.y);
    }
    int p = KK - 1;
    uint32_t posbits = (1u << KK) - 1u;
    if (!(mn > 0.f)) {
        p = -1;
        posbits = 0;
#pragma unroll
        for (int i = 0; i < KK; ++i) {
            if (x[i] > 0.f) {
                p = i;
                posbits |= 1u << i;
            } else {
                x[i] = 0.f;
            }
        }
    }
    th.pos = posbits;

    // 3. the compensated per-thread scan (x[] becomes the running sum)
    float s = 0.f, c = 0.f;
#pragma unroll
    for (int i = 0; i < KK; ++i) {
        const float y = __fsub_rn(x[i], c);
        const float t = __fadd_rn(s, y);
        c = __fsub_rn(__fsub_rn(t, s), y);
        s = t;
        x[i] = s;
    }

    // block exclusive scan of the per-thread totals in exact 64-bit fixed point
    // (resolution 2^-48 relative to 2^k; a tile sum is below 2^14): exact
    // sums are monotone, and every thread knows its own next base
    const long long tot = fixed48_of(s, c);
    long long inc = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long h = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += h;
    }
    if (lane == 31) sm.wtot[warp] = inc;
    const int il = __reduce_max_sync(0xffffffffu, p >= 0 ? e0 + p : -1);
    if (lane == 0) sm.wlast[warp] = il;
    __syncthreads();
    // every warp scans the kWarps warp totals (lane w holds warp w's)
    long long ws = lane < kWarps ? sm.wtot[lane] : 0;
    const int i_last = __reduce_max_sync(0xffffffffu, lane < kWarps ? sm.wlast[lane] : -1);
#pragma unroll
    for (int o = 1; o < kWarps; o <<= 1) {
        const long long h = __shfl_up_sync(0xffffffffu, ws, o);
        if (lane >= o) ws += h;
    }
    const long long total = __shfl_sync(0xffffffffu, ws, kWarps - 1);
    const long long wbase = warp > 0 ? __shfl_sync(0xffffffffu, ws, warp - 1) : 0;
    const long long excl = wbase + inc - tot;
    const float Vk = fixed48_to_float(excl), Vn = fixed48_to_float(excl + tot);
    th.base = Vk;

    // 4. tile-local cumulative weights; elements from the last positive one on
    // take the next base so that no gap is left between threads
    if (p == KK - 1) {
        const float2 Vk2 = make_float2(Vk, Vk);
#pragma unroll
        for (int i = 0; i < KK; i += 2) {
            const float2 v = __fadd2_rn(Vk2, make_float2(x[i], x[i + 1]));
            x[i] = fminf(v.x, Vn);
            x[i + 1] = i + 1 < KK - 1 ? fminf(v.y, Vn) : Vn;
        }
    } else {
#pragma unroll
        for (int i = 0; i < KK; ++i) x[i] = (i >= p) ? Vn : fminf(__fadd_rn(Vk, x[i]), Vn);
    }

    TileSummary ts;
    ts.k = k;
    ts.S = {0.f, 0.f};
    if (tid == 0) ts.S = tile_sum_pair(total);  // thread 0 records it
    ts.total = total;
    ts.i_last = i_last;
    ts.bad = bad;
    return ts;
}

// Block-wide; KK from the tile length (4, 8 or 16 elements per thread).
template <bool RO = false>
__device__ __forceinline__ TileSummary tile_scan(const float* base, int lo, int n, TileShared& sm,
                                                 TileThread& th) {
    const int K = per_thread_count(n);
    if (K == 4) return tile_scan_k<4, false, RO>(base, lo, n, sm, th);
    if (K == 8) return tile_scan_k<8, false, RO>(base, lo, n, sm, th);
    return tile_scan_k<16, false, RO>(base, lo, n, sm, th);
}

}  // namespace pf

// Assignment of offsets to a tile's elements, shared by the single-launch and
// the batched kernels (Section 2: systematic and stratified resampling give
// offspring counts; multinomial resampling a binary search per draw).
#pragma once

#include "pf_fixed.cuh"
#include "pf_index.h"
#include "pf_tile.cuh"

namespace pf {

enum { KIND_MULTI = 0, KIND_STRAT = 1, KIND_SYS = 2 };
// Staging entries of the run-length decode (per buffer): a chunk of the CTA-wide
// decode holds up to CAP - 4 offsets, a warp's its share.  kIoCap serves tiles of up to
// 8192 elements, kIoCapSmall of up to 4096.
constexpr int kIoCap = 10240;
constexpr int kIoCapSmall = 8192;
static_assert(kIoCap % (4 * 512) == 0 && kIoCapSmall % (4 * 512) == 0, "decode chunks use 4-entry groups per thread");

struct TableEntry {  // multinomial: one tile's lower boundary and scale
    float bhi, blo;  // B_t as a float pair (units of 2^K)
    float sc;        // 2^(K - k_t): global units -> tile-local units
    int il;          // last positive element of the tile, -1 if none
};

// Shared-memory fields of one filter's assignment.
constexpr int kMaxRuns = 128;  // long runs of a tile stored ahead of its decode

struct AssignShared {
    i128 Wt;       // total mass W (fixed point, units of 2^K)
    int K;         // largest tile exponent
    int noff;      // offsets of the tile being assigned
    long long jlo; // first offset of that tile
    float tau0, inv_rho, W_hi, W_lo;
    int red_n[kWarps];
    int n_runs;  // long runs of the tile, stored ahead of its decode
    int run_lo[kMaxRuns], run_hi[kMaxRuns];
    int32_t run_of[kMaxRuns];
};

// ---------------------------------------------------------------------------
// Offspring-count assignment (systematic, stratified).
// ---------------------------------------------------------------------------
// Per-tile scalars (lanes 0 and 1 of warp 0), in float pairs: the tile's
// offset range and the map from tile-local cumulative weight v to the offset
// coordinate y = v * inv_rho + x0 (offsets counted from jlo).
// One end of a tile's offset range: the offsets below boundary B (B_t for
// the lower end, B_{t+1} for the upper), the same function of B for both, so
// adjacent tiles share their common end exactly.  A boundary at 0 gives 0 and
// one at the total mass W gives P.  Lower end (SYS, STRAT): x0 of the map.
// (a.hi - j) + a.lo for an integer j near a.hi: the subtraction is exact even
// where j has no float representation (odd j above 2^24, with P up to 2^31),
// as a small integer plus the exact fraction of a.hi.
__device__ __forceinline__ float pair_minus_int(fpair a, long long j) {
    const float fh = floorf(a.hi);
    return __fadd_rn(__fadd_rn((float)((long long)fh - j), __fsub_rn(a.hi, fh)), a.lo);
}

// The uniform of the systematic scheme; the multinomial guide places its offsets at (j / P) W: none.
__device__ __forceinline__ float offset_uniform(const SortedParams& p) {
    return p.guide ? 0.f : u23f(philox(0u, 0u, p.filter, TAG_SYS, p.key0, p.key1).x);
}

template <int KIND>
__device__ __forceinline__ long long offsets_below(const SortedParams& p, const AssignShared& sm, fpair PW, i128 B_i,
                                                   float u, float& x0) {
    const fpair y = pair_mul(fixed_to_pair(B_i), PW);  // B P / W
    long long j;
    if (KIND == KIND_SYS) {
        const fpair d = pair_sub_f(y, u);
        j = B_i <= 0 ? 0 : (B_i >= sm.Wt ? p.P : max(0LL, min((long long)p.P, pair_ceil(d))));
        x0 = pair_minus_int(d, j);  // N(v) = ceil(v * inv_rho + x0)
    } else {
        j = 0;
        if (B_i >= sm.Wt) {
            j = p.P;
        } else if (B_i > 0) {
            const long long f = pair_floor(y);
            if (f >= p.P) {
                j = p.P;
            } else {
                const float frac = pair_minus_int(y, f);
                const u32x4 r = philox((uint32_t)(f >> 2), 0u, p.filter, TAG_STRAT, p.key0, p.key1);
                j = max(0LL, f + (u23f(word_of(r, (int)(f & 3))) < frac ? 1 : 0));
            }
        }
        x0 = pair_minus_int(y, j);  // y(v) = v * inv_rho + x0
    }
    return j;
}

// A tile's offset range [jlo, jlo + noff) and the map from its tile-local
// cumulative weight v to offsets: N(v) = ceil(v * ir + x0) (systematic) or the
// stratum test on y(v) = v * ir + x0 (stratified), offsets counted from jlo.
struct TileMap {
    long long jlo;
    int noff;
    float x0, ir;
};

// The map of a tile with boundaries [Bl_i, Bh_i), formed by two lanes of one
// warp together: the even lane forms the lower end, the odd lane the upper;
// `mask` names the participating lanes (both lanes of every pair).  Both lanes
// return the map.
// u: offset_uniform (systematic).
template <int KIND>
__device__ __forceinline__ TileMap tile_map_pair(const SortedParams& p, const AssignShared& sm, i128 Bl_i, i128 Bh_i,
                                                 int k_tile, unsigned mask, float u) {
    const int lane = threadIdx.x & 31;
    const bool upper = lane & 1;
    const fpair W = {sm.W_hi, sm.W_lo};
    const fpair Pp = fast_two_sum((float)p.P, (float)(p.P - (int64_t)(float)p.P));  // P exactly
    const fpair PW = pair_div(Pp, W);
    float x0;
    const long long j = offsets_below<KIND>(p, sm, PW, upper ? Bh_i : Bl_i, u, x0);
    const long long jl = __shfl_sync(mask, j, lane & ~1);
    const long long jh = __shfl_sync(mask, j, lane | 1);
    const float x0l = __shfl_sync(mask, x0, lane & ~1);
    return {jl, (int)max(0LL, jh - jl), x0l, PW.hi * pow2f(k_tile - sm.K)};
}

template <int KIND>
__device__ __forceinline__ TileMap tile_map_pair(const SortedParams& p, const AssignShared& sm, i128 Bl_i, i128 Bh_i,
                                                 int k_tile, unsigned mask) {
    return tile_map_pair<KIND>(p, sm, Bl_i, Bh_i, k_tile, mask, KIND == KIND_SYS ? offset_uniform(p) : 0.f);
}

// The same for one tile into sm (lanes 0 and 1 of warp 0 together).
template <int KIND>
__device__ void tile_offsets(const SortedParams& p, AssignShared& sm, i128 Bl_i, i128 Bh_i, int k_tile) {
    const TileMap m = tile_map_pair<KIND>(p, sm, Bl_i, Bh_i, k_tile, 0x3u);
    if (threadIdx.x == 0) {
        sm.jlo = m.jlo;
        sm.noff = m.noff;
        sm.tau0 = m.x0;
        sm.inv_rho = m.ir;
    }
}

// Run-length decode staging: two buffers of kIoCap entries, used by
// successive chunks in turn.  A chunk's entries are tagged with the chunk's
// epoch, (epoch << kLocalBits) | element, so entries left by earlier chunks
// are smaller than all of its own and no clearing pass is needed; alternating
// the buffers lets a chunk start before every thread has stored the previous
// one.  stage_init fills both buffers with -1 (below every tag) and must run
// once per launch before the first chunk.
constexpr int kLocalBits = 13;  // tile-local element index
static_assert(kTileMax <= (1 << kLocalBits), "element index must fit the tag's low bits");
constexpr uint32_t kEpochMax = (1u << (31 - kLocalBits)) - 1;  // tags stay positive as int32

template <int CAP>
__device__ __forceinline__ void stage_init(int32_t* stage) {  // stage: 16-byte aligned
    for (int i = threadIdx.x; i < 2 * CAP / 4; i += kThreads)
        reinterpret_cast<int4*>(stage)[i] = make_int4(-1, -1, -1, -1);
}

// The run that covers offset c0 and where the next one begins, over this thread's elements
// (counts N in v, starting from start0): cur the last element whose run covers c0 (-1:
// none), next the first start beyond c0 (INT_MAX: none).
template <int KK>
__device__ __forceinline__ void run_at(const TileThread& th, int start0, int c0, int& cur, int& next) {
    cur = -1;
    next = INT_MAX;
    int a = start0;
#pragma unroll
    for (int i = 0; i < KK; ++i) {
        if ((th.pos >> i) & 1u) {
            const int b = __float_as_int(th.v[i]);
            if (b > a) {
                if (a > c0) next = min(next, a);
                else if (b > c0) cur = i;
            }
            a = b;
        }
    }
}

// The longest run of this thread's elements (as run_at).
template <int KK>
__device__ __forceinline__ int longest_run(const TileThread& th, int start0) {
    int a = start0, longest = 0;
#pragma unroll
    for (int i = 0; i < KK; ++i) {
        if ((th.pos >> i) & 1u) {
            const int b = __float_as_int(th.v[i]);
            longest = max(longest, b - a);
            a = b;
        }
    }
    return longest;
}

// dst[0, n) = v by `threads` threads, this one the t-th; 16-byte stores between the ends.
__device__ __forceinline__ void fill_run(int32_t* dst, int n, int32_t v, int t, int threads) {
    const int head = min((int)((4u - (uint32_t)((uintptr_t)dst >> 2)) & 3u), n), body = (n - head) & ~3;
    if (t < head) dst[t] = v;
    for (FillPieces f(head, body, t, threads); f.x < f.end; f.x += f.step)
        *reinterpret_cast<int4*>(dst + f.x) = make_int4(v, v, v, v);
    if (t < n - head - body) dst[head + body + t] = v;
}

// One chunk [c0, c1) of the tile's offsets: each positive element marks the
// first slot of its run [N_{i-1}, N_i) with its tagged tile-local index (runs
// of later elements start later, so tags increase along the chunk), the
// element whose run covers the chunk's first slot marks that slot, and an
// inclusive max-scan over the chunk fills every run.  Chunk slot s sits at
// out[s + shift] so that out[x] maps to the 16-byte aligned global position
// gb + x; each thread scans and stores S consecutive entries
// (S * kThreads >= c1 - c0 + shift).  Ancestor = tile_base + element.
template <int S, int KK>
__device__ __forceinline__ void decode_chunk(const SortedParams& p, AssignShared& sm, int32_t* out,
                                             const TileThread& th, long long jlo, int c0, int c1, int shift,
                                             int start0, int32_t tile_base, int32_t tag) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int x0i = tid * S;
    const int32_t mark0 = tag | th.e0;
    int a = start0;
#pragma unroll
    for (int i = 0; i < KK; ++i) {
        if ((th.pos >> i) & 1u) {
            const int b = __float_as_int(th.v[i]);
            if (b > a) {
                if (a >= c0 && a < c1) out[a - c0 + shift] = mark0 + i;
                else if (a < c0 && b > c0) out[shift] = mark0 + i;
            }
            a = b;
        }
    }
    __syncthreads();
    // pass A: this thread's maximum, then the exclusive maximum over the block
    int run = -1;
#pragma unroll
    for (int q = 0; q < S / 4; ++q) {
        const int4 v = *reinterpret_cast<const int4*>(&out[x0i + 4 * q]);
        run = max(run, max(max(v.x, v.y), max(v.z, v.w)));
    }
    int mm = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int h = __shfl_up_sync(0xffffffffu, mm, o);
        if (lane >= o) mm = max(mm, h);
    }
    int carry = __shfl_up_sync(0xffffffffu, mm, 1);
    if (lane == 0) carry = -1;
    if (lane == 31) sm.red_n[warp] = mm;
    __syncthreads();
    carry = max(carry, __reduce_max_sync(0xffffffffu, lane < warp ? sm.red_n[lane] : -1));
    // pass B: the entries again (the buffer is not written again before the
    // chunk after next), as running maxima from the carry, stored.  Entries x in
    // [x0i, x0i + S) hold chunk slots x - shift; every slot of the chunk carries
    // this chunk's tag (its first slot is marked).
    const int lo = max(x0i, shift), hi = min(x0i + S, shift + (c1 - c0));
    if (hi > lo) {
        int32_t* g = p.anc + (jlo + c0 - shift) + x0i;  // 16-byte aligned
        const bool whole = lo == x0i && hi == x0i + S;
        int rr = carry;
        // every filled slot holds tag | element with this chunk's tag, so one
        // add turns it into the ancestor tile_base + element
        const int32_t delta = tile_base - tag;
#pragma unroll
        for (int q = 0; q < S / 4; ++q) {
            const int4 v = *reinterpret_cast<const int4*>(&out[x0i + 4 * q]);
            int4 a4;
            a4.x = delta + (rr = max(rr, v.x));
            a4.y = delta + (rr = max(rr, v.y));
            a4.z = delta + (rr = max(rr, v.z));
            a4.w = delta + (rr = max(rr, v.w));
            if (whole) {
                *reinterpret_cast<int4*>(g + 4 * q) = a4;
            } else {
                const int v4[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
                for (int z = 0; z < 4; ++z)
                    if (x0i + 4 * q + z >= lo && x0i + 4 * q + z < hi) g[4 * q + z] = v4[z];
            }
        }
    }
    // no trailing barrier: the next chunk marks the other buffer, and it reuses
    // sm.red_n only after its own mark barrier, which every thread reaches after
    // finishing this chunk's reads of sm.red_n
}

// The assignment of a tile of many offsets (more than any chunk holds) by the whole CTA.
// stage: the two staging buffers (2 * CAP entries, stage_init<CAP>'ed); epoch: the chunk
// counter, identical in every thread.
template <int KIND, int KK, int CAP, bool LONG>  // LONG: look for long runs
__device__ void assign_offspring(const SortedParams& p, AssignShared& sm, const TileMap map, int32_t* stage,
                                 uint32_t& epoch, TileThread& th, const TileSummary& ts, int64_t index0) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int noff = map.noff;
    const long long jlo = map.jlo;
    const float x0 = map.x0, ir = map.ir;
    // N_i: offsets of the tile below the element's cumulative weight (kept in v[] as int bits).
    // Systematic: N = min(ceil(y), noff), the conversion rounding up and saturating at 0.
    // Stratified: with k = floor(y), N = k + [u_k < y - k], capped at noff (y - k is exact); each
    // thread draws the Philox blocks its elements need.  The tile's last positive element takes noff.
    int last_n = -1;
    uint32_t cq = 0xffffffffu;
    u32x4 cw = {0, 0, 0, 0};
#pragma unroll
    for (int i = 0; i < KK; ++i) {
        if ((th.pos >> i) & 1u) {
            const float y = __fmaf_rn(th.v[i], ir, x0);
            int n;
            if (th.e0 + i == ts.i_last) {
                n = noff;
            } else if (KIND == KIND_SYS) {
                n = (int)min(__float2uint_ru(y), (uint32_t)noff);
            } else if (y <= 0.f) {
                n = 0;
            } else {
                const float fl = floorf(y);
                if (fl >= (float)noff) {
                    n = noff;
                } else {
                    const long long j = jlo + (long long)fl;
                    const uint32_t q = (uint32_t)(j >> 2);
                    if (q != cq) {
                        cq = q;
                        cw = philox(q, 0u, p.filter, TAG_STRAT, p.key0, p.key1);
                    }
                    n = min(noff, (int)fl + (u23f(word_of(cw, (int)(j & 3))) < y - fl ? 1 : 0));
                }
            }
            th.v[i] = __int_as_float(n);
            last_n = n;
        }
    }
    // exclusive running maximum of the threads' last counts: where this thread's first run starts
    int m = last_n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int h = __shfl_up_sync(0xffffffffu, m, o);
        if (lane >= o) m = max(m, h);
    }
    int prev = __shfl_up_sync(0xffffffffu, m, 1);
    if (lane == 0) prev = -1;
    if (lane == 31) sm.red_n[warp] = m;
    __syncthreads();
    prev = max(prev, __reduce_max_sync(0xffffffffu, lane < warp ? sm.red_n[lane] : -1));
    const int start0 = max(prev, 0);
    const int32_t tile_base = (int32_t)index0;  // particle index of the tile's element 0

    // Runs of a chunk or more are stored as they are, all of them one after another (those
    // found beyond kMaxRuns stay with the decode), and the chunks below pass over them.  A
    // run's stored part ends where a later one may begin: at the least of the counts from its
    // own element on (a compensated sum may step back by an ulp).  300 equally heavy neighbours
    // among 2^24 particles, systematic: 536 us chunk by chunk, 633 with a search for the next
    // run between every two, 443 this way (one SM's stores: 55 GB/s).
    constexpr int kLongRun = CAP;
    int n_runs = 0;
    if (LONG && noff >= 2 * kLongRun) {  // block-uniform
        if (tid == 0) sm.n_runs = 0;
        __syncthreads();
        int a = start0, lo = 0, hi = 0, of = -1;
        auto put = [&] {
            if (of >= 0 && hi - lo >= kLongRun) {
                const int r = atomicAdd(&sm.n_runs, 1);
                if (r < kMaxRuns) {
                    sm.run_lo[r] = lo;
                    sm.run_hi[r] = hi;
                    sm.run_of[r] = tile_base + th.e0 + of;
                }
            }
        };
#pragma unroll
        for (int i = 0; i < KK; ++i) {
            if ((th.pos >> i) & 1u) {
                const int b = __float_as_int(th.v[i]);
                if (b - a >= kLongRun) {
                    put();
                    lo = a;
                    hi = b;
                    of = i;
                } else if (of >= 0) {
                    hi = min(hi, b);
                }
                a = b;
            }
        }
        put();
        __syncthreads();
        n_runs = min(sm.n_runs, kMaxRuns);
        for (int r = 0; r < n_runs; ++r)
            fill_run(p.anc + jlo + sm.run_lo[r], sm.run_hi[r] - sm.run_lo[r], sm.run_of[r], tid, kThreads);
    }

    // Run-length decode, one staging chunk at a time (decode_chunk); chunks
    // of at most 2044 / 4092 / 8188 offsets use 4 / 8 / 16 staging entries per
    // thread, larger ones 20.
    constexpr int kChunk = CAP - 4;  // offsets per chunk (room for the shift)
    for (int c0 = 0; c0 < noff;) {
        int c1 = chunk_end(c0, noff, kChunk);
        if (n_runs > 0) {  // block-uniform
            int beyond = 0, next = INT_MAX;
            for (int r = lane; r < n_runs; r += 32) {
                const int lo = sm.run_lo[r], hi = sm.run_hi[r];
                if (lo > c0) next = min(next, lo);
                else if (c0 < hi) beyond = hi;
            }
            beyond = __reduce_max_sync(0xffffffffu, beyond);
            if (beyond > 0) {
                c0 = beyond;
                continue;
            }
            c1 = min(c1, __reduce_min_sync(0xffffffffu, next));
        }
        if (++epoch > kEpochMax) {  // tags exhausted (uniform): clear both buffers and restart
            __syncthreads();
            stage_init<CAP>(stage);
            __syncthreads();
            epoch = 1;
        }
        int32_t* out = stage + (epoch & 1u) * CAP;
        const int32_t tag = (int32_t)(epoch << kLocalBits);
        const int shift = (int)(((uintptr_t)(p.anc + jlo + c0) >> 2) & 3u);  // to a 16-byte boundary
        const int need = c1 - c0 + shift;
        if (CAP <= 4 * kThreads || need <= 4 * kThreads)  // the multinomial guide's staging: always
            decode_chunk<4, KK>(p, sm, out, th, jlo, c0, c1, shift, start0, tile_base, tag);
        else if (need <= 8 * kThreads)
            decode_chunk<8, KK>(p, sm, out, th, jlo, c0, c1, shift, start0, tile_base, tag);
        else if (CAP == 16 * kThreads || need <= 16 * kThreads)
            decode_chunk<16, KK>(p, sm, out, th, jlo, c0, c1, shift, start0, tile_base, tag);
        else
            decode_chunk<(CAP > 16 * kThreads ? CAP : 16 * kThreads + 4) / kThreads, KK>(
                p, sm, out, th, jlo, c0, c1, shift, start0, tile_base, tag);
        c0 = c1;
    }
}

// ---------------------------------------------------------------------------
// The same assignment warp by warp, for tiles of at most kWarpOffsets offsets
// (nearly all: a tile's count varies around its length).  No barrier of the CTA:
// a warp's elements own one contiguous range of the tile's offsets, and where
// that range begins follows from the thread's base (the cumulative weight of the
// element before its first), because the element before it has exactly that
// cumulative weight and so the same count N.  Each warp marks its runs in its
// own 32 S staging entries (all -1 between chunks), a warp max-scan fills them,
// and the entries are set back to -1 as they are read for the last time.
//
// Bound by instruction issue and latency at two CTAs an SM.  The CTA-wide decode waited at
// three barriers a tile with 40% of the issue slots used: the assignment launch at P = 2^25 +
// 4096 took 94 us systematic and 156 stratified, this way 53 and 79 (pf_large.cu); stratified
// at 10^8 particles 691 and 391 us in all.
//
// N by a rounded addition: y + 1.5 2^23 rounded up (down) has ceil(y)
// (floor(y)) in its low bits, exact for |y| < 2^22; it replaces the conversion,
// which issues at a quarter of the rate.  y is monotone along the thread, so only
// a thread whose first or last count falls outside the tile's range clamps.
//
// Skewed weights: a warp whose offsets are several chunks looks for a run that goes on
// for two chunks or more and stores it as it is, and a warp with more strata than its
// buffers hold draws them one buffer at a time, passing over those inside a run.  With
// every chunk decoded and each thread drawing its own strata, systematic, exp(4 N(0,1))
// weights: 2^20 particles 66 us, so 27; 2^24 394 and 150; stratified 2^20 41 and 26.
// ---------------------------------------------------------------------------
// A tile with more offsets than this goes to the CTA-wide decode.  One warp may own nearly
// all of a tile's offsets (one heavy particle, or many): long runs it stores as they are,
// and where it must decode chunk by chunk, 640 offsets at a time, the CTA's 10236 at a
// time behind three barriers and two clears of the staging are quicker only for a great
// many.  2^24 particles, systematic, weights exp(3 N(0,1)): 98 us with the line at 16384, 80 at
// 65536, 79 at 262144; exp(4 N) at 6e4 particles, stratified: 14.7, 12.4, 11.7; 300 equally
// heavy particles side by side among 2^20: 56, 50, 89.
// Without the look for long runs (LONG false) the line is at 16384.
constexpr int kWarpOffsets = 8 * kTileMax, kWarpOffsetsShort = 2 * kTileMax;
// A run of so many offsets of one particle, two of the warp's chunks, is stored as it is.
constexpr int kRunFill = 1280;
constexpr float kRoundMagic = 12582912.f;      // 1.5 2^23
constexpr int kRoundMagicBits = 0x4b400000;

// Staging entries per lane: 32 S covers a warp's usual range (its 32 KK elements'
// worth of offsets and four standard deviations of N(0,1) weights) in one chunk, and an
// odd multiple of four words between lanes keeps the 16-byte reads free of bank conflicts.
__host__ __device__ constexpr int warp_stage_per_lane(int KK) { return KK == 16 ? 20 : (KK == 8 ? 12 : 8); }

// marks: this warp's STRIDE entries (32 S used), 16-byte aligned, all -1 on entry and on return;
// stratified: STRIDE floats for the strata's uniforms follow.
template <int KIND, int KK, int S, int STRIDE, bool LONG, bool SPILL>
__device__ __forceinline__ void assign_warp(const SortedParams& p, const TileMap map, int32_t* marks, TileThread& th,
                                            int i_last, int64_t index0) {
    const int lane = threadIdx.x & 31;
    const int noff = map.noff;
    if (noff <= 0) return;
    const float x0 = map.x0, ir = map.ir;
    constexpr uint32_t kFull = (1u << KK) - 1u;
    const uint32_t pos = th.pos;
    if (!__any_sync(0xffffffffu, pos != 0u)) return;  // no positive weight in the warp
    const int il = i_last - th.e0;  // this thread's index of the tile's last positive element, if any
    const float yb = __fmaf_rn(th.base, ir, x0), yl = __fmaf_rn(th.v[KK - 1], ir, x0);
    int start0;  // offsets below the element before this thread's first
    if (KIND == KIND_SYS) {
        const int nb = __float_as_int(__fadd_ru(yb, kRoundMagic)) - kRoundMagicBits;
        const int nl = __float_as_int(__fadd_ru(yl, kRoundMagic)) - kRoundMagicBits;
        start0 = min(max(nb, 0), noff);
        const bool clamp = nb < 0 || nl > noff;
#pragma unroll
        for (int i = 0; i < KK; ++i)
            th.v[i] =
                __int_as_float(__float_as_int(__fadd_ru(__fmaf_rn(th.v[i], ir, x0), kRoundMagic)) - kRoundMagicBits);
        if (clamp) {
#pragma unroll
            for (int i = 0; i < KK; ++i)
                th.v[i] = __int_as_float(min(max(__float_as_int(th.v[i]), 0), noff));
        }
    } else {
        const int kmax = noff - 1;
        // stratum of a coordinate and the coordinate's place in it
        auto stratum = [&](float y, float& frac) -> int {
            const float t = __fadd_rd(y, kRoundMagic);
            int k = __float_as_int(t) - kRoundMagicBits;
            frac = __fsub_rn(y, __fsub_rn(t, kRoundMagic));
            return k;
        };
        float fb, fl;
        const int kb0 = stratum(yb, fb), kl0 = stratum(yl, fl);
        const bool clamp = strata_clamped(kb0, kl0, kmax, pos);
        const int kb = min(max(kb0, 0), kmax), kl = min(max(kl0, 0), kmax);
        if (clamp) fb = __fsub_rn(yb, (float)kb);
        // the uniforms of the warp's strata, four per Philox block, drawn once into ubuf
        const int k_first = __shfl_sync(0xffffffffu, kb, 0);
        // one more than the last count's: a compensated sum may step back by an ulp at the end
        const int k_last = min(__reduce_max_sync(0xffffffffu, max(kb, kl)) + 1, kmax);
        const long long g0 = strata_block(map.jlo, k_first);
        const int blocks = (int)(strata_block(map.jlo, k_last) - g0) + 1;
        const int at = strata_at(map.jlo, g0);  // ubuf index of stratum 0 (may be negative)
        if (blocks <= STRIDE / (SPILL ? 2 : 4)) {
            // SPILL: where the buffer does not hold them all, the marks' entries in front of it take their
            // share (2^21 particles, weights u^100, u uniform: a buffer at a time 22.3 us, so 18.8)
            const bool spill = SPILL && blocks > STRIDE / 4;
            const int from = spill ? 0 : STRIDE;
            float* ubuf = reinterpret_cast<float*>(marks);
            __syncwarp();  // the last tile's reads of the buffer
            for (int b = lane; b < blocks; b += 32) {
                const u32x4 r = philox((uint32_t)(g0 + b), 0u, p.filter, TAG_STRAT, p.key0, p.key1);
                *reinterpret_cast<float4*>(ubuf + from + 4 * b) =
                    make_float4(u23f(r.x), u23f(r.y), u23f(r.z), u23f(r.w));
            }
            __syncwarp();
            start0 = min(noff, kb + (ubuf[from + strata_index(at, kb)] < fb ? 1 : 0));
            if (!clamp) {
#pragma unroll
                for (int i = 0; i < KK; ++i) {
                    float frac;
                    const int k = stratum(__fmaf_rn(th.v[i], ir, x0), frac);
                    th.v[i] = __int_as_float(k + (ubuf[from + at + k] < frac ? 1 : 0));
                }
            } else {
#pragma unroll
                for (int i = 0; i < KK; ++i) {
                    const float y = __fmaf_rn(th.v[i], ir, x0);
                    float frac;
                    const int k = min(max(stratum(y, frac), 0), kmax);
                    th.v[i] = __int_as_float(
                        min(noff, k + (ubuf[from + strata_index(at, k)] < __fsub_rn(y, (float)k) ? 1 : 0)));
                }
            }
            if (spill) {
                __syncwarp();
                for (int b = lane; b < STRIDE / 4; b += 32)
                    reinterpret_cast<int4*>(marks)[b] = make_int4(-1, -1, -1, -1);
                __syncwarp();
            }
        } else {
            float* ubuf = reinterpret_cast<float*>(marks + STRIDE);
            // strata beyond the buffer: one buffer of them at a time, those without a
            // coordinate (inside a dominant particle's run) passed over.  The whole buffer each
            // time: draws cut off at the last stratum measured slower (no longer unrolled)
            uint32_t open = kFull;  // elements whose stratum is still to come
            bool open0 = true;
            for (int w = k_first; w < INT_MAX;) {
                const long long g = strata_block(map.jlo, w);
                const int w_at = strata_at(map.jlo, g), w_end = 32 * S - w_at;  // strata [w, w_end) are in ubuf
                __syncwarp();
                for (int b = lane; b < 8 * S; b += 32) {
                    const u32x4 r = philox((uint32_t)(g + b), 0u, p.filter, TAG_STRAT, p.key0, p.key1);
                    *reinterpret_cast<float4*>(ubuf + 4 * b) = make_float4(u23f(r.x), u23f(r.y), u23f(r.z), u23f(r.w));
                }
                __syncwarp();
                int next = INT_MAX;
                if (open0) {
                    if (kb < w_end) {
                        start0 = min(noff, kb + (ubuf[strata_index(w_at, kb)] < fb ? 1 : 0));
                        open0 = false;
                    } else {
                        next = kb;
                    }
                }
#pragma unroll
                for (int i = 0; i < KK; ++i) {
                    if ((open >> i) & 1u) {
                        const float y = __fmaf_rn(th.v[i], ir, x0);
                        float frac;
                        const int k = min(max(stratum(y, frac), 0), kmax);
                        if (k < w_end) {
                            th.v[i] = __int_as_float(
                                min(noff, k + (ubuf[strata_index(w_at, k)] < __fsub_rn(y, (float)k) ? 1 : 0)));
                            open &= ~(1u << i);
                        } else {
                            next = min(next, k);
                        }
                    }
                }
                w = __reduce_min_sync(0xffffffffu, next);
            }
        }
    }
    int last_n;  // count at this thread's last positive element
    if ((uint32_t)il < (uint32_t)KK || pos != kFull) {
        last_n = start0;
#pragma unroll
        for (int i = 0; i < KK; ++i) {
            if (i == il) th.v[i] = __int_as_float(noff);  // the tile's last positive element takes the rest
            if ((pos >> i) & 1u) last_n = __float_as_int(th.v[i]);
        }
    } else {
        last_n = __float_as_int(th.v[KK - 1]);
    }
    const int A = __shfl_sync(0xffffffffu, start0, 0);
    const int B = __reduce_max_sync(0xffffffffu, pos ? last_n : 0);
    const int32_t e_base = (int32_t)index0 + th.e0;  // ancestor of this thread's element 0
    const int xl = lane * S;
    const bool long_runs = LONG && B - A > 32 * S && __any_sync(0xffffffffu, longest_run<KK>(th, start0) >= kRunFill);
    for (int c0 = A; c0 < B;) {
        const int shift = (int)(((uintptr_t)(p.anc + map.jlo + c0) >> 2) & 3u);  // to a 16-byte boundary
        const int c1 = min(B, c0 + 32 * S - shift);
        if (long_runs && B - c0 >= kRunFill) {
            // a run that goes on for kRunFill offsets or more is stored as it is
            int cur, next;
            run_at<KK>(th, start0, c0, cur, next);
            cur = __reduce_max_sync(0xffffffffu, cur < 0 ? -1 : e_base + cur);
            next = min(__reduce_min_sync(0xffffffffu, next), B);
            if (cur >= 0 && next - c0 >= kRunFill) {
                fill_run(p.anc + map.jlo + c0, next - c0, cur, lane, 32);
                c0 = next;
                continue;
            }
        }
        // marks: each run's first slot in the chunk
        int a = start0;
        int32_t* mk = marks + (shift - c0);
        if (c0 == A && c1 == B && pos == kFull) {  // the usual case: one chunk, every weight positive
#pragma unroll
            for (int i = 0; i < KK; ++i) {
                const int b = __float_as_int(th.v[i]);
                if (b > a) mk[a] = e_base + i;
                a = b;
            }
        } else {
#pragma unroll
            for (int i = 0; i < KK; ++i) {
                if ((pos >> i) & 1u) {
                    const int b = __float_as_int(th.v[i]);
                    const int m = max(a, c0);
                    if (b > m && m < c1) mk[m] = e_base + i;
                    a = b;
                }
            }
        }
        __syncwarp();
        int run = -1;
#pragma unroll
        for (int q = 0; q < S / 4; ++q) {
            const int4 v = *reinterpret_cast<const int4*>(&marks[xl + 4 * q]);
            run = max(run, max(max(v.x, v.y), max(v.z, v.w)));
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int h = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run = max(run, h);
        }
        int rr = __shfl_up_sync(0xffffffffu, run, 1);
        if (lane == 0) rr = -1;
        const int end = shift + (c1 - c0);  // the chunk's entries: [shift, end)
        int32_t* g = p.anc + (map.jlo + c0 - shift) + xl;  // 16-byte aligned
#pragma unroll
        for (int q = 0; q < S / 4; ++q) {
            const int x = xl + 4 * q;
            int4 v = *reinterpret_cast<const int4*>(&marks[x]);
            *reinterpret_cast<int4*>(&marks[x]) = make_int4(-1, -1, -1, -1);
            v.x = rr = max(rr, v.x);
            v.y = rr = max(rr, v.y);
            v.z = rr = max(rr, v.z);
            v.w = rr = max(rr, v.w);
            if (x >= shift && x + 4 <= end) {
                *reinterpret_cast<int4*>(g + 4 * q) = v;
            } else if (x + 4 > shift && x < end) {
                if (x >= shift) g[4 * q] = v.x;
                if (x + 1 >= shift && x + 1 < end) g[4 * q + 1] = v.y;
                if (x + 2 >= shift && x + 2 < end) g[4 * q + 2] = v.z;
                if (x + 3 < end) g[4 * q + 3] = v.w;
            }
        }
        __syncwarp();  // the entries are clear before the next marks
        c0 = c1;
    }
}

// A warp's entries in the staging, and where they begin: the same place whatever KK and S, as
// the CTA's warps may be in different tiles, of different KK.
template <int KIND, int CAP>
__host__ __device__ constexpr int warp_stage_stride() {
    return (KIND == KIND_STRAT || CAP >= kIoCapSmall ? CAP : 2 * CAP) / kWarps;
}
template <int KIND, int CAP>
__device__ __forceinline__ int32_t* warp_stage(int32_t* stage) {  // stratified: the uniforms' buffer behind each warp's
    return stage + (int)(threadIdx.x >> 5) * (KIND == KIND_STRAT ? 2 : 1) * warp_stage_stride<KIND, CAP>();
}

// Sets this warp's entries to -1 (once, before its first tile).
template <int KIND, int CAP>
__device__ __forceinline__ void warp_stage_init(int32_t* stage) {
    constexpr int kStride = warp_stage_stride<KIND, CAP>();
    int4* mine = reinterpret_cast<int4*>(warp_stage<KIND, CAP>(stage));
#pragma unroll
    for (int i = threadIdx.x & 31; i < kStride / 4; i += 32) mine[i] = make_int4(-1, -1, -1, -1);
    __syncwarp();
}

// W of a one-tile filter as a pair, as fixed_to_pair gives it for the tile sum's 128-bit
// value: the top 24 bits and the next 24 of the pair's exact sum.
__device__ __forceinline__ fpair total_pair(long long total) {
    const float hi = (float)total;
    const long long sum = (long long)hi + (long long)(float)(total - (long long)hi);
    const int n = 64 - __clzll(sum), s = max(n - 24, 0);
    const uint32_t top = (uint32_t)(sum >> s);
    const long long rem = sum - ((long long)top << s);
    const int s2 = max(s - 24, 0);
    return {(float)top * pow2f(s - 48), (float)(uint32_t)(rem >> s2) * pow2f(s2 - 48)};
}

// The map of a tile that owns every offset (tile_map_pair with the boundaries 0 and W).
template <int KIND>
__device__ __forceinline__ TileMap only_tile_map(const SortedParams& p, fpair W) {
    const fpair Pp = fast_two_sum((float)p.P, (float)(p.P - (int64_t)(float)p.P));
    const float u = KIND == KIND_SYS ? u23f(philox(0u, 0u, p.filter, TAG_SYS, p.key0, p.key1).x) : 0.f;
    return {0, (int)p.P, -u, pair_div(Pp, W).hi};
}

// One tile's assignment: warp by warp, or, for a tile that owns so many offsets
// that one warp's share could be most of them, chunk by chunk over the CTA (which sets
// the staging before, and back to -1 after).  Block-uniform choice.  The warp's
// entries are -1 on entry (warp_stage_init) and on return.
template <int KIND, int KK, int CAP, int S = warp_stage_per_lane(KK), bool LONG = true,  // LONG: as assign_offspring
          bool SPILL = true>                                                             // SPILL: as assign_warp
__device__ __forceinline__ void assign_tile(const SortedParams& p, AssignShared& sm, const TileMap map, int32_t* stage,
                                            TileThread& th, const TileSummary& ts, int64_t index0) {
    constexpr int kStride = warp_stage_stride<KIND, CAP>();
    static_assert(32 * S <= kStride && kStride % 4 == 0, "a warp's entries fit its share of the staging");
    if (map.noff <= (LONG ? kWarpOffsets : kWarpOffsetsShort)) {
        assign_warp<KIND, KK, S, kStride, LONG, SPILL>(p, map, warp_stage<KIND, CAP>(stage), th, ts.i_last, index0);
        return;
    }
    __syncthreads();
    stage_init<CAP>(stage);
    __syncthreads();
    uint32_t epoch = 0;
    assign_offspring<KIND, KK, CAP, LONG>(p, sm, map, stage, epoch, th, ts, index0);
    __syncthreads();
    stage_init<CAP>(stage);
    __syncthreads();
}

// Four multinomial draws (the words of one Philox block) of one filter
// (Figure 1a).  Draw s targets u_s W (float pair); a binary search over the
// tile table (shared memory) finds the last tile whose carry is <= the
// target, then a lower-bound search in that tile's cumulative weights finds
// the first element whose weight exceeds the tile-local target.  The four
// in-tile searches advance in lockstep, so their loads overlap.
//   table[T]  tile entries;  v(t, b, i)  reads element i of tile t, whose first is b, of the
//   cumulative weights (sign bit: zero weight);  tile  tile length;  PA = P + lead.
//   Writes filter-local ancestors to a[].
// v takes the tile both ways, as forming the address from b keeps four 64-bit values in
// registers and from t costs a multiplication a step: 2^25 particles, one log-weight in a hundred
// raised by 10 (their draws end here) 1323 and 1273 us, 20011 without allocation 22.9 and 23.8.
template <class V>
__device__ __forceinline__ void multinomial_draws4(const u32x4& r, const TableEntry* table, int T, V v, int tile,
                                                   int64_t PA, int lead, float Wh, float Wl, int32_t (&a)[4]) {
    float xh[4], xl[4];
    int lo[4], n[4], il[4], at[4];
    int64_t b0[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        float uh, ul;
        u32_pair(word_of(r, s), uh, ul);
        const float th = __fmul_rn(uh, Wh);
        const float tl = __fmaf_rn(uh, Wl, __fmaf_rn(ul, Wh, __fmaf_rn(uh, Wh, -th)));
        int tlo = 0, thi = T - 1;
        while (tlo < thi) {
            const int mid = (tlo + thi + 1) >> 1;
            const float d = __fadd_rn(__fsub_rn(table[mid].bhi, th), __fsub_rn(table[mid].blo, tl));
            if (d <= 0.f) tlo = mid;
            else thi = mid - 1;
        }
        while (tlo > 0 && table[tlo].il < 0) --tlo;  // never settle on a tile without weight
        const TableEntry e = table[tlo];
        float h = __fmul_rn(__fsub_rn(th, e.bhi), e.sc);
        float l = __fmul_rn(__fsub_rn(tl, e.blo), e.sc);
        if (h + l < 0.f) {
            h = 0.f;
            l = 0.f;
        }
        xh[s] = h;
        xl[s] = l;
        at[s] = tlo;
        b0[s] = (int64_t)tlo * tile;
        n[s] = (int)min((int64_t)tile, PA - b0[s]);
        lo[s] = 0;
        il[s] = e.il;
    }
    const int nt[4] = {n[0], n[1], n[2], n[3]};
    // lower bound: first i with |v_i| - xh > xl (|v| - xh is exact near the decision)
    for (int it = 0; it < 15 && (n[0] | n[1] | n[2] | n[3]) > 0; ++it) {
        float val[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            val[s] = n[s] > 0 ? v(at[s], b0[s], lo[s] + (n[s] >> 1)) : 0.f;
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            if (n[s] > 0) {
                const int half = n[s] >> 1;
                if (__fsub_rn(fabsf(val[s]), xh[s]) > xl[s]) {
                    n[s] = half;
                } else {
                    lo[s] += half + 1;
                    n[s] -= half + 1;
                }
            }
        }
    }
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        auto ld = [&](int i) -> float { return v(at[s], b0[s], i); };
        int idx = il[s];
        if (lo[s] < nt[s]) {
            idx = lo[s];
            if (zero_flag(ld(idx))) {  // rounding landed on a zero weight: the next positive one
                int f = il[s];
                for (int z = idx + 1; z < nt[s]; ++z)
                    if (!zero_flag(ld(z))) {
                        f = z;
                        break;
                    }
                idx = f;
            }
        }
        a[s] = (int32_t)(b0[s] + idx - lead);
    }
}

// Quad-cooperative window count.  Every lane of the warp calls it at the same
// point (the shuffles span the full warp).  Each lane brings a window of n <= 16
// monotone entries at base + off (base the same in every lane, base + off
// 16-byte aligned; n = 0: none) and its target (xh, xl); the four lanes of each
// aligned quad read each other's windows, one 16-byte piece per lane, so one
// load instruction touches the lines of 8 windows instead of 32 scattered
// pieces.  Returns the count of this lane's window entries at or below its
// target and (FLAGS) the window's zero-weight flags in zmask (sign bits, bit i
// for entry i).
template <bool FLAGS>
__device__ __forceinline__ int quad_window_below(const float* base, int off, int n, float xh, float xl,
                                                 uint32_t& zmask) {
    const int lane = threadIdx.x & 31, q = lane & 3;
    // all four pieces are requested before any is used, so their latencies overlap
    float t[4][4], hr[4], lr[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int src = (lane & ~3) | r;
        const float* wr = base + __shfl_sync(0xffffffffu, off, src);
        const int nr = __shfl_sync(0xffffffffu, n, src);
        hr[r] = __shfl_sync(0xffffffffu, xh, src);
        lr[r] = __shfl_sync(0xffffffffu, xl, src);
        if (4 * q + 3 < nr) {
            const float4 t4 = __ldcg(reinterpret_cast<const float4*>(wr + 4 * q));
            t[r][0] = t4.x;
            t[r][1] = t4.y;
            t[r][2] = t4.z;
            t[r][3] = t4.w;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) t[r][i] = 4 * q + i < nr ? __ldcg(wr + 4 * q + i) : INFINITY;
        }
    }
    // this lane's share of each window: count in bits 0-4, flags from bit 5 (the
    // lanes' flag bits are disjoint, so adding shares also merges the flags)
    int part[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        int cnt = 0;
        uint32_t z = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            cnt += __fsub_rn(fabsf(t[r][i]), hr[r]) > lr[r] ? 0 : 1;  // +inf padding counts as above
            if (FLAGS) z |= (__float_as_uint(t[r][i]) >> 31) << (4 * q + i);
        }
        part[r] = cnt + (int)(z << 5);
    }
    // transposed sum over the quad: lane q ends with window q's total
    const bool odd = q & 1, high = q & 2;
    int s0 = odd ? part[1] : part[0], s1 = odd ? part[3] : part[2];  // windows q&1 and 2 + (q&1)
    s0 += __shfl_xor_sync(0xffffffffu, odd ? part[0] : part[1], 1);
    s1 += __shfl_xor_sync(0xffffffffu, odd ? part[2] : part[3], 1);
    int mine = high ? s1 : s0;
    mine += __shfl_xor_sync(0xffffffffu, high ? s0 : s1, 2);
    zmask = FLAGS ? ((uint32_t)mine >> 5) : 0u;
    return mine & 31;
}

// One multinomial draw of a filter whose tiles' cumulative weights v are in
// global memory (L2) and whose every 16th |v| (and each tile's last one) is
// in shared memory: tile search in the table, then a search in the tile's
// coarse samples for the first window of 16 elements whose last sample exceeds
// the tile-local target, then that window read whole (64 bytes, 16-byte
// aligned, quad-cooperatively: every lane of the warp must call it) and the
// first element above the target counted in registers.  Same predicate on the
// same monotone sequence as the plain search, so the same result; one 64-byte
// read from L2 per draw instead of a dozen.
constexpr int kWinShift = 4;
constexpr int kWin = 1 << kWinShift;
__device__ __forceinline__ int32_t multinomial_draw_windowed(uint32_t x, const TableEntry* table, int T,
                                                             const float* v, const float* coarse, int cpt, int tile,
                                                             int64_t PA, int lead, float Wh, float Wl) {
    float uh, ul;
    u32_pair(x, uh, ul);
    const float th = __fmul_rn(uh, Wh);
    const float tl = __fmaf_rn(uh, Wl, __fmaf_rn(ul, Wh, __fmaf_rn(uh, Wh, -th)));
    int lo = 0, hi = T - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        const float d = __fadd_rn(__fsub_rn(table[mid].bhi, th), __fsub_rn(table[mid].blo, tl));
        if (d <= 0.f) lo = mid;
        else hi = mid - 1;
    }
    while (lo > 0 && table[lo].il < 0) --lo;
    const TableEntry e = table[lo];
    float xh = __fmul_rn(__fsub_rn(th, e.bhi), e.sc);
    float xl = __fmul_rn(__fsub_rn(tl, e.blo), e.sc);
    if (xh + xl < 0.f) {
        xh = 0.f;
        xl = 0.f;
    }
    const int64_t b0 = (int64_t)lo * tile;
    const int nt = (int)min((int64_t)tile, PA - b0);
    // coarse: first window whose last sample is above the target
    const float* c = coarse + lo * cpt;
    int cl = 0, cn = (nt + kWin - 1) >> kWinShift;
    while (cn > 0) {
        const int half = cn >> 1;
        if (__fsub_rn(c[cl + half], xh) > xl) {
            cn = half;
        } else {
            cl += half + 1;
            cn -= half + 1;
        }
    }
    // the window is read quad-cooperatively: every lane of the warp comes here
    // (wn = 0 where the target lies past the tile's samples)
    const int w0 = cl << kWinShift;
    const int wn = w0 < nt ? min(kWin, nt - w0) : 0;
    uint32_t zmask;
    const int below = quad_window_below<true>(v, (int)(b0 + w0), wn, xh, xl, zmask);  // elements at or below the target
    int idx = e.il;
    if (below < wn) {
        idx = w0 + below;
        if ((zmask >> below) & 1u) {  // rounding landed on a zero weight: the next positive one
            int f = e.il;
            for (int z = idx + 1; z < nt; ++z)
                if (!zero_flag(__ldcg(v + b0 + z))) {
                    f = z;
                    break;
                }
            idx = f;
        }
    }
    return (int32_t)(b0 + idx - lead);
}

// Every 16th |v| of a tile (and its last one), from this thread's elements,
// into the tile's coarse samples (shared memory).
__device__ __forceinline__ void write_tile_coarse(const TileThread& th, int n, float* c) {
#pragma unroll
    for (int i = 0; i < kMaxPerThread; ++i) {
        const int e = th.e0 + i;
        if (i < th.K && e < n && (((e + 1) & (kWin - 1)) == 0 || e == n - 1)) c[e >> kWinShift] = fabsf(th.v[i]);
    }
}

// Tile lookup of the single-launch multinomial draws: lut[k], k = 0..kLut, is
// the last tile t whose boundary B_t is at or below the target (k / kLut) W
// under the draws' own comparison.  A draw whose uniform lies in
// (k / kLut, (k+1) / kLut) then lies in tiles lut[k]..lut[k+1], which narrows
// the search over the table to a tile or two.
constexpr int kLutBits = 12;
constexpr int kLut = 1 << kLutBits;

// The draws' comparison: is tile e's boundary at or below the target (th, tl)?
__device__ __forceinline__ bool boundary_at_or_below(const TableEntry& e, float th, float tl) {
    return __fadd_rn(__fsub_rn(e.bhi, th), __fsub_rn(e.blo, tl)) <= 0.f;
}

// Target u W of a uniform given as an exact pair (uh, ul), W = (Wh, Wl).
__device__ __forceinline__ void draw_target(float uh, float ul, float Wh, float Wl, float& th, float& tl) {
    th = __fmul_rn(uh, Wh);
    tl = __fmaf_rn(uh, Wl, __fmaf_rn(ul, Wh, __fmaf_rn(uh, Wh, -th)));
}

// Block-wide (kThreads): fills lut[0..kLut] from table[0..T); red: kWarps ints.
__device__ inline void build_tile_lut(const TableEntry* table, int T, float Wh, float Wl, int* lut, int* red) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int k = tid; k <= kLut; k += kThreads) lut[k] = 0;
    __syncthreads();
    // each tile t >= 1 marks the first lookup point whose target reaches B_t
    for (int t = 1 + tid; t < T; t += kThreads) {
        const TableEntry e = table[t];
        auto reaches = [&](int k) {
            float th, tl;
            draw_target((float)k * (1.f / kLut), 0.f, Wh, Wl, th, tl);
            return boundary_at_or_below(e, th, tl);
        };
        int k = (int)fminf(fmaxf(ceilf(e.bhi / Wh * (float)kLut), 0.f), (float)kLut);
        while (k > 0 && reaches(k - 1)) --k;
        while (k <= kLut && !reaches(k)) ++k;
        if (k <= kLut) atomicMax(&lut[k], t);
    }
    __syncthreads();
    // running maximum over lut[0..kLut): kLut / kThreads consecutive entries per thread
    constexpr int per = kLut / kThreads;
    int m = 0;
#pragma unroll
    for (int i = 0; i < per; ++i) m = max(m, lut[tid * per + i]);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int h = __shfl_up_sync(0xffffffffu, m, o);
        if (lane >= o) m = max(m, h);
    }
    if (lane == 31) red[warp] = m;
    int prev = __shfl_up_sync(0xffffffffu, m, 1);
    if (lane == 0) prev = 0;
    __syncthreads();
    for (int w = 0; w < warp; ++w) prev = max(prev, red[w]);
    int run = prev;
#pragma unroll
    for (int i = 0; i < per; ++i) {
        run = max(run, lut[tid * per + i]);
        lut[tid * per + i] = run;
    }
    if (tid == kThreads - 1) lut[kLut] = max(lut[kLut], run);
    __syncthreads();
}

// Single-launch multinomial draw over three levels of the tiles' cumulative
// weights: every 2^c1shift-th |v| of each tile (c1, shared memory, c1shift >=
// 8), every 16th (c2, global, cpt2 per tile, each tile's block 64-byte
// aligned) and v itself (global).  Level 1 narrows to 2^(c1shift-4) samples of
// c2; when that is more than 16, a binary search over their 16-entry blocks
// (one 4-byte read a level) picks the block; each remaining level reads one
// 16-entry window whole.  The predicate and the monotone sequence are those of
// the plain search, so the result is the same, with two dependent 64-byte
// reads per draw (plus c1shift - 8 small ones) instead of a dozen 4-byte ones.
__device__ __forceinline__ int last_tile_at_or_below(const TableEntry* table, int lo, int hi, float th, float tl) {
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (boundary_at_or_below(table[mid], th, tl)) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int32_t multinomial_draw_3level(uint32_t x, const TableEntry* table, const int* lut, int T,
                                                           const float* v, const float* c2, int cpt2, const float* c1,
                                                           int cpt1, int c1shift, int tile, int64_t PA, int lead,
                                                           float Wh, float Wl) {
    float uh, ul, th, tl;
    u32_pair(x, uh, ul);
    draw_target(uh, ul, Wh, Wl, th, tl);
    // the last tile whose boundary is at or below the target: searched between
    // the lookup points around u, then confirmed (the predicate is monotone in
    // t, so a confirmed tile is the plain binary search's result over all T)
    const int kq = (int)(x >> (32 - kLutBits));
    int lo = last_tile_at_or_below(table, lut[kq], min(lut[kq + 1], T - 1), th, tl);
    if (!boundary_at_or_below(table[lo], th, tl) || (lo + 1 < T && boundary_at_or_below(table[lo + 1], th, tl)))
        lo = last_tile_at_or_below(table, 0, T - 1, th, tl);
    while (lo > 0 && table[lo].il < 0) --lo;
    const TableEntry e = table[lo];
    float xh = __fmul_rn(__fsub_rn(th, e.bhi), e.sc);
    float xl = __fmul_rn(__fsub_rn(tl, e.blo), e.sc);
    if (xh + xl < 0.f) {
        xh = 0.f;
        xl = 0.f;
    }
    const int64_t b0 = (int64_t)lo * tile;
    const int nt = (int)min((int64_t)tile, PA - b0);
    const int n2 = (nt + 15) >> 4, n1 = (nt + (1 << c1shift) - 1) >> c1shift;
    // level 1: first window whose last sample is above the target
    const float* c = c1 + lo * cpt1;
    int cl = 0, cn = n1;
    while (cn > 0) {
        const int half = cn >> 1;
        if (__fsub_rn(c[cl + half], xh) > xl) {
            cn = half;
        } else {
            cl += half + 1;
            cn -= half + 1;
        }
    }
    // levels 2 and 3 read their 16-entry windows quad-cooperatively, so every
    // lane of the warp takes this path (n = 0 where no window is read)
    const bool has = cl < n1;
    const float* c2t = c2 + (int64_t)lo * cpt2;
    int m2 = cl << (c1shift - 4);  // first c2 sample of the window
    if (has && c1shift > 8) {
        // several 16-sample blocks: the first whose last sample is above the target
        int bl = 0, bn = min(1 << (c1shift - 8), (n2 - m2 + 15) >> 4);
        while (bn > 0) {
            const int half = bn >> 1;
            const int last = min(m2 + ((bl + half + 1) << 4), n2) - 1;
            if (__fsub_rn(__ldcg(c2t + last), xh) > xl) {
                bn = half;
            } else {
                bl += half + 1;
                bn -= half + 1;
            }
        }
        m2 += bl << 4;
    }
    // level 2: the block of 16 samples, then level 3: the 16 elements
    uint32_t zmask;
    m2 += quad_window_below<false>(c2, lo * cpt2 + m2, has ? min(16, n2 - m2) : 0, xh, xl, zmask);
    const int w0 = m2 << 4;
    const int wn = has ? min(16, nt - w0) : 0;
    const int below = quad_window_below<true>(v, (int)(b0 + w0), wn, xh, xl, zmask);
    int idx = e.il;
    if (has) {
        idx = w0 + below;
        if (below >= wn) idx = e.il;  // not reached: the window's last sample is above the target
        else if ((zmask >> below) & 1u) {  // rounding landed on a zero weight: the next positive one
            int f = e.il;
            for (int z = idx + 1; z < nt; ++z)
                if (!zero_flag(__ldcg(v + b0 + z))) {
                    f = z;
                    break;
                }
            idx = f;
        }
    }
    return (int32_t)(b0 + idx - lead);
}

// Single-launch multinomial draw through the guide table g[0..M): g[b] is the
// first particle whose cumulative weight exceeds the bucket edge (b / M) W (the
// systematic assignment's arithmetic with M offsets and no uniform shift).  A
// draw whose uniform lies in bucket b = floor(u M) has its answer at or after
// g[b], up to the rounding that separates the two arithmetics, so the draw
// takes the tile holding particle g[b] - 1, confirms it with its own boundary
// test (the tile's boundary at or below the target, the next one above it),
// reads the 16-element window of v that starts at or just below g[b] - 1 and
// counts the elements at or below its target.  That is the plain search's
// result exactly when the window's first element is at or below the target (or
// is the tile's first), and some element of the window is above it (or the
// window ends the tile): the same predicate on the same monotone sequence.
// Otherwise (a bucket holding more than ~12 particles, or an empty tile) ok is
// false and the caller takes the three-level draw.  Every lane of the warp must
// call it (quad-cooperative window read).
__device__ __forceinline__ int32_t multinomial_draw_guided(uint32_t x, const TableEntry* table, int T,
                                                           const float* v, const int32_t* g, int64_t M, int tile,
                                                           int64_t PA, int lead, float Wh, float Wl, bool& ok) {
    float uh, ul, th, tl;
    u32_pair(x, uh, ul);
    draw_target(uh, ul, Wh, Wl, th, tl);
    // bucket of u = (2x + 1) 2^-33: floor(u M), exact in 64-bit integers
    const int64_t b = (int64_t)(((2ull * x + 1ull) * (unsigned long long)M) >> 33);
    int64_t h = (int64_t)__ldcg(g + b) - 1 + lead;  // aligned-window position of particle g[b] - 1
    h = h < lead ? (int64_t)lead : (h > PA - 1 ? PA - 1 : h);
    static_assert((1 << kLocalBits) == kTileMax, "full tiles are 2^kLocalBits elements");
    const int lo = tile == kTileMax ? (int)((uint64_t)h >> kLocalBits) : (int)(h / tile);
    const bool good = boundary_at_or_below(table[lo], th, tl) &&
                      (lo + 1 >= T || !boundary_at_or_below(table[lo + 1], th, tl)) && table[lo].il >= 0;
    const TableEntry e = table[lo];
    float xh = __fmul_rn(__fsub_rn(th, e.bhi), e.sc);
    float xl = __fmul_rn(__fsub_rn(tl, e.blo), e.sc);
    if (xh + xl < 0.f) {
        xh = 0.f;
        xl = 0.f;
    }
    const int64_t b0 = (int64_t)lo * tile;
    const int nt = (int)min((int64_t)tile, PA - b0);
    const int w0 = (int)(h - b0) & ~3;
    const int wn = good ? min(16, nt - w0) : 0;
    uint32_t zmask;
    const int below = quad_window_below<true>(v, (int)(b0 + w0), wn, xh, xl, zmask);
    ok = good && (w0 == 0 || below >= 1) && (below < wn || w0 + wn >= nt);
    int idx = e.il;
    if (ok && below < wn) {
        idx = w0 + below;
        if ((zmask >> below) & 1u) {  // rounding landed on a zero weight: the next positive one
            int f = e.il;
            for (int z = idx + 1; z < nt; ++z)
                if (!zero_flag(__ldcg(v + b0 + z))) {
                    f = z;
                    break;
                }
            idx = f;
        }
    }
    return (int32_t)(b0 + idx - lead);
}

// This thread's samples of its tile: every 16th |v| (and the tile's last)
// into c2, every 2^c1shift-th (and the last) into c1.
template <int KK>
__device__ __forceinline__ void write_tile_samples(const TileThread& th, int n, float* c2, float* c1, int c1shift) {
    const int m1 = (1 << c1shift) - 1;
#pragma unroll
    for (int i = 0; i < KK; ++i) {
        const int e = th.e0 + i;
        if (e < n) {
            const bool lastel = e == n - 1;
            if (((e + 1) & 15) == 0 || lastel) c2[e >> 4] = fabsf(th.v[i]);
            if (((e + 1) & m1) == 0 || lastel) c1[e >> c1shift] = fabsf(th.v[i]);
        }
    }
}

// Eight floats in one 256-bit access (32-byte aligned): a thread's share of a tile
// is 64 bytes, so each access moves whole 32-byte sectors where two 128-bit ones
// move each sector twice.
__device__ __forceinline__ void ld_cg_v8(const float* p, float* o) {
    asm volatile("ld.global.cg.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3]), "=f"(o[4]), "=f"(o[5]), "=f"(o[6]), "=f"(o[7])
                 : "l"(p)
                 : "memory");
}

__device__ __forceinline__ void st_v8(float* p, const float* o) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(o[0]), "f"(o[1]), "f"(o[2]),
                 "f"(o[3]), "f"(o[4]), "f"(o[5]), "f"(o[6]), "f"(o[7])
                 : "memory");
}

// Reloads a tile stored by write_tile_v into th (elements of tile-local
// indices [0, n), KK a thread as scanned): v from the magnitudes, the positive-weight mask from
// the sign bits.  Slots at or beyond n are not read: they and, in threads wholly past n, the
// base hold the last element's v, as after a scan.  Every lane of the warp must call it
// (the bases come from the lane below).
template <int KK>
__device__ __forceinline__ void read_tile_v(const float* vg0, int n, TileThread& th) {
    th.K = KK;
    th.e0 = threadIdx.x * KK;
    const float* vg = vg0 + th.e0;
    if (KK >= 8 && th.e0 + KK <= n && (((uintptr_t)vg) & 31u) == 0) {
#pragma unroll
        for (int q = 0; q < KK / 8; ++q) ld_cg_v8(vg + 8 * q, th.v + 8 * q);
    } else {
#pragma unroll
        for (int q = 0; q < KK / 4; ++q) {
            if (th.e0 + 4 * q + 3 < n) {
                const float4 t = __ldcg(reinterpret_cast<const float4*>(vg + 4 * q));
                th.v[4 * q] = t.x;
                th.v[4 * q + 1] = t.y;
                th.v[4 * q + 2] = t.z;
                th.v[4 * q + 3] = t.w;
            } else {
#pragma unroll
                for (int r = 0; r < 4; ++r) th.v[4 * q + r] = th.e0 + 4 * q + r < n ? __ldcg(vg + 4 * q + r) : -0.0f;
            }
        }
    }
    // the sign bits: none set in the usual thread
    uint32_t any = 0, pos = (1u << KK) - 1u;
#pragma unroll
    for (int i = 0; i < KK; ++i) any |= __float_as_uint(th.v[i]);
    if (any >> 31) {
        pos = 0;
        float run = th.e0 >= n ? fabsf(__ldcg(vg0 + n - 1)) : 0.f;
#pragma unroll
        for (int i = 0; i < KK; ++i) {
            if (!zero_flag(th.v[i])) pos |= 1u << i;
            if (th.e0 + i < n) run = fabsf(th.v[i]);
            th.v[i] = run;  // past the tile's end: the last element's
        }
    }
    th.pos = pos;
    // the element before this thread's first: the lane below's last, or a load by lane 0
    th.base = __shfl_up_sync(0xffffffffu, th.v[KK - 1], 1);
    if ((threadIdx.x & 31) == 0) th.base = th.e0 == 0 ? 0.f : (th.e0 <= n ? fabsf(__ldcg(vg - 1)) : th.v[0]);
}

// The tile's cumulative weights to global memory (sign bit: zero weight), for the searches.
template <int KK = 0>
__device__ __forceinline__ void write_tile_v(const SortedParams& p, const TileThread& th, int64_t t0, int n) {
    float* vg = p.v_out + t0 + th.e0;
    const int K = KK ? KK : th.K;
    if (KK && th.pos == (1u << KK) - 1u && th.e0 + K <= n) {  // the usual thread: whole, every weight positive
        if (KK >= 8 && (((uintptr_t)vg) & 31u) == 0) {
#pragma unroll
            for (int q = 0; q < KK / 8; ++q) st_v8(vg + 8 * q, th.v + 8 * q);
        } else {
#pragma unroll
            for (int q = 0; q < KK / 4; ++q)
                *reinterpret_cast<float4*>(vg + 4 * q) =
                    make_float4(th.v[4 * q], th.v[4 * q + 1], th.v[4 * q + 2], th.v[4 * q + 3]);
        }
        return;
    }
#pragma unroll
    for (int q = 0; q < (KK ? KK : kMaxPerThread) / 4; ++q) {
        if (KK || 4 * q < th.K) {
            float o[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int i = 4 * q + r;
                o[r] = ((th.pos >> i) & 1u) ? th.v[i] : -th.v[i];
            }
            if (th.e0 + 4 * q + 3 < n) {
                *reinterpret_cast<float4*>(vg + 4 * q) = make_float4(o[0], o[1], o[2], o[3]);
            } else {
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    if (th.e0 + 4 * q + r < n) vg[4 * q + r] = o[r];
            }
        }
    }
}

}  // namespace pf

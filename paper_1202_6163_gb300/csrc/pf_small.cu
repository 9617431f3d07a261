// Cumulative resamplers of small single filters (Figure 1a-c): up to 16 tiles, one
// per CTA of one thread-block cluster.  The cluster's CTAs are scheduled together, so
// the call is an ordinary launch (a cooperative one costs 2.5 us more between calls on
// a stream), the tiles' records are exchanged through distributed shared memory and the
// hardware's cluster barrier instead of global memory and an arrival counter, and
// the multinomial's draws search the cumulative weights in shared memory.  A filter of one
// tile needs no exchange at all: every thread forms the filter's offset map from the
// tile's total.
//
// Bound by latency: the load, the scan's shuffles and barriers, the boundaries' 128-bit
// arithmetic and two divisions follow one another.  Calls back to back in a graph,
// cooperative launch and here: systematic P = 1000 8.2 and 4.1 us, 20011 8.5 and 6.0, stratified
// 8.9 and 4.3, 9.4 and 6.6, multinomial 13.6 and 5.4, 16.9 and 13.2 (32768: 17.0 and 16.6).
// Sixteen CTAs are the largest cluster the hardware takes.
//
// The tiles and all arithmetic are those of the single-launch kernels (pf_persistent.cu).
#include <cfloat>
#include <climits>

#include <cooperative_groups.h>

#include "pf_assign.cuh"

namespace pf {

namespace cg = cooperative_groups;

namespace {

constexpr int kMaxCluster = 16;  // CTAs of a cluster (beyond 8: opt-in)

struct SmallShared {
    TileShared tile;
    AssignShared as;
    uint4 rec;  // this CTA's tile: exponent, sum (NaN: a bad weight), last positive element
    TileMap map;
    TableEntry table[kMaxCluster];
    int ok;
};

__host__ __device__ constexpr int small_stage_cap(int KK) { return KK == 16 ? kIoCap : kIoCapSmall; }
__host__ __device__ constexpr size_t small_header() { return (sizeof(SmallShared) + 15) & ~(size_t)15; }
// Behind it: the decode's staging (systematic, stratified), or the filter's cumulative
// weights (multinomial): every CTA holds all tiles', so that a draw's search stays in
// its own shared memory (eleven dependent reads of a neighbour's took 25 us at P = 20011).
__host__ __device__ constexpr size_t small_smem(int kind, int KK) {
    return small_header() + (kind == KIND_MULTI ? 0 : 2 * (size_t)small_stage_cap(KK) * sizeof(int32_t));
}
constexpr int kSmallWeights = 48 * 1024;  // cumulative weights a multinomial call may hold (192 KiB)
__host__ __device__ constexpr int weight_slot(int tile) { return (tile + 31) & ~31; }  // floats per tile
// Element i's place in its tile's slot: the 16-byte pieces of every 128 bytes are
// rotated among themselves, as the pivots of a search over a power of two elements
// otherwise all fall in one bank (P = 2048: 8.2 us, 2000: 5.9).
__device__ __forceinline__ int weight_place(int i) { return i ^ ((i >> 3) & 0x1c); }

// Two multinomial draws, their searches in lockstep and without branches: the last tile
// whose boundary is at or below the target, then the number of the tile's elements at or
// below it.
template <bool ONE>
__device__ __forceinline__ void small_draws2(const uint32_t (&x)[2], const TableEntry* table, const float* vall, int slot,
                                             const SortedParams& p, int PA, fpair W, int32_t (&a)[2]) {
    float th[2], tl[2], xh[2], xl[2];
    int tile[2] = {0, 0}, n[2], pos[2] = {0, 0}, il[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        float uh, ul;
        u32_pair(x[s], uh, ul);
        draw_target(uh, ul, W.hi, W.lo, th[s], tl[s]);
    }
    if (!ONE) {
#pragma unroll
        for (int st = kMaxCluster / 2; st > 0; st >>= 1) {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int u = tile[s] + st;
                if (u < p.n_tiles && boundary_at_or_below(table[u], th[s], tl[s])) tile[s] = u;
            }
        }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        while (tile[s] > 0 && table[tile[s]].il < 0) --tile[s];  // never settle on a tile without weight
        const TableEntry e = table[tile[s]];
        xh[s] = __fmul_rn(__fsub_rn(th[s], e.bhi), e.sc);
        xl[s] = __fmul_rn(__fsub_rn(tl[s], e.blo), e.sc);
        if (xh[s] + xl[s] < 0.f) {
            xh[s] = 0.f;
            xl[s] = 0.f;
        }
        n[s] = min(p.tile, PA - tile[s] * p.tile);
        il[s] = e.il;
    }
    const int top = 1 << (31 - __clz(min(p.tile, PA)));
    const float* v[2] = {vall + tile[0] * slot, vall + tile[1] * slot};
    for (int st = top; st > 0; st >>= 1) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int i = pos[s] + st;
            const float val = fabsf(v[s][weight_place(min(i, n[s]) - 1)]);
            if (i <= n[s] && !(__fsub_rn(val, xh[s]) > xl[s])) pos[s] = i;
        }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        // rounding landed on a zero weight: the next positive one
        while (pos[s] < n[s] && zero_flag(v[s][weight_place(pos[s])])) ++pos[s];
        a[s] = tile[s] * p.tile + (pos[s] < n[s] ? pos[s] : il[s]) - p.lead;
    }
}

template <int KIND, int KK, bool ONE>
__global__ void __launch_bounds__(kThreads) k_small(SortedParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallShared& sm = *reinterpret_cast<SmallShared*>(smem_raw);
    unsigned char* region = smem_raw + small_header();
    int32_t* stage = reinterpret_cast<int32_t*>(region);
    float* vall = reinterpret_cast<float*>(region);  // multinomial: tile u's cumulative weights at u slot
    const int slot = weight_slot(p.tile);
    constexpr int CAP = small_stage_cap(KK);
    const int tid = threadIdx.x, lane = tid & 31, t = blockIdx.x, T = p.n_tiles;
    grid_begin();
    uint64_t* const trace = t < T ? p.trace : nullptr;  // CTAs beyond the tiles write no record
    if (trace) {
        trace_stamp(trace, p.trace_cap, t, 0);
        trace_put(trace, p.trace_cap, t, 5, t);
        trace_put(trace, p.trace_cap, t, 6, 0);
        trace_put(trace, p.trace_cap, t, 7, 1);
    }
    const int64_t PA = p.P + p.lead, t0 = (int64_t)t * p.tile;
    const int n = (int)max((int64_t)0, min((int64_t)p.tile, PA - t0));  // CTAs beyond the tiles have none
    TileThread th;
    const TileSummary ts = tile_scan_k<KK>(p.lw + t0, t == 0 ? p.lead : 0, n, sm.tile, th);
    if (KIND == KIND_MULTI) {
#pragma unroll
        for (int q = 0; q < KK / 4; ++q) {
            float o[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int i = 4 * q + r;
                o[r] = ((th.pos >> i) & 1u) ? th.v[i] : -th.v[i];
            }
            if (th.e0 + 4 * q < n)  // a whole piece of four: the slots between n and it belong to this tile
                *reinterpret_cast<float4*>(vall + t * slot + weight_place(th.e0 + 4 * q)) =
                    make_float4(o[0], o[1], o[2], o[3]);
        }
    } else {
        warp_stage_init<KIND, CAP>(stage);
    }
    trace_stamp(trace, p.trace_cap, t, 1);

    TileMap map = {0, 0, 0.f, 0.f};
    fpair W = {0.f, 0.f};
    bool ok;
    if (ONE) {
        ok = !ts.bad && ts.total > 0;
        W = total_pair(ts.total);
        if (KIND != KIND_MULTI) {
            map = only_tile_map<KIND>(p, W);
        } else {
            if (tid == 0) sm.table[0] = {0.f, 0.f, 1.f, ts.i_last};
            __syncthreads();
        }
        trace_stamp(trace, p.trace_cap, t, 2);
    } else {
        if (tid == 0)
            sm.rec = make_uint4((uint32_t)ts.k, __float_as_uint(ts.bad ? NAN : ts.S.hi), __float_as_uint(ts.S.lo),
                                (uint32_t)ts.i_last);
        cg::cluster_group cluster = cg::this_cluster();
        cluster.sync();
        trace_stamp(trace, p.trace_cap, t, 2);
        const int warp = tid >> 5;
        if (KIND == KIND_MULTI && t < T && warp > 0 && warp < T) {
            // another tile's cumulative weights per warp, eight pieces in flight, while warp 0 forms the table
            const int u = t + warp < T ? t + warp : t + warp - T;
            float4* mine = reinterpret_cast<float4*>(vall + u * slot);
            const float4* theirs = cluster.map_shared_rank(mine, u);
            const int n4 = weight_slot((int)min((int64_t)p.tile, PA - (int64_t)u * p.tile)) >> 2;
            for (int i0 = lane; i0 < n4; i0 += 8 * 32) {
                float4 v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (i0 + 32 * k < n4) v[k] = theirs[i0 + 32 * k];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (i0 + 32 * k < n4) mine[i0 + 32 * k] = v[k];
            }
        }
        if (tid < 32) {
            uint4 r = make_uint4(0u, 0u, 0u, 0xffffffffu);
            if (lane < T) r = *cluster.map_shared_rank(&sm.rec, lane);
            const float sh = __uint_as_float(r.y);
            const bool bad = __any_sync(0xffffffffu, !(sh <= FLT_MAX));
            const int K = __reduce_max_sync(0xffffffffu, sh > 0.f ? (int)r.x : INT_MIN);
            const bool good = !bad && K != INT_MIN;
            if (good) {
                i128 m = 0;
                if (KIND == KIND_MULTI) {  // as the single-launch kernel forms its table
                    const int s = (int)r.x - K;
                    if (lane < T) m = fixed_of(sh, s) + fixed_of(__uint_as_float(r.z), s);
                } else if (sh > 0.f) {  // as it sums its CTAs' records
                    const int s = K - (int)r.x;
                    m = s >= 127 ? (i128)0 : (fixed_of(sh, 0) + fixed_of(__uint_as_float(r.z), 0)) >> s;
                }
                const i128 inc = warp_scan_i128(m, lane);
                const i128 Wt = shfl_i128(inc, 31);
                const fpair Wp = fixed_to_pair(Wt);
                if (KIND == KIND_MULTI) {
                    if (lane < T) {
                        const fpair b = fixed_to_pair(inc - m);
                        sm.table[lane] = {b.hi, b.lo, pow2f(K - (int)r.x), (int)r.w};
                    }
                } else {
                    AssignShared as;
                    as.Wt = Wt;
                    as.K = K;
                    as.W_hi = Wp.hi;
                    as.W_lo = Wp.lo;
                    const int mine = min(t, T - 1);
                    const i128 hi = shfl_i128(inc, mine), lo = hi - shfl_i128(m, mine);
                    const TileMap mp = tile_map_pair<KIND>(p, as, lo, hi, ts.k, 0xffffffffu);
                    if (lane == 0) sm.map = mp;
                }
                if (lane == 0) {
                    sm.as.W_hi = Wp.hi;
                    sm.as.W_lo = Wp.lo;
                }
            }
            if (lane == 0) sm.ok = good;
        }
        __syncthreads();
        ok = sm.ok != 0;
        if (KIND != KIND_MULTI) map = sm.map;
        else W = {sm.as.W_hi, sm.as.W_lo};
    }
    trace_stamp(trace, p.trace_cap, t, 3);
    if (!ok && tid == 0 && t == 0) set_status(p.ctl + CTL_STATUS, ST_DOMAIN);  // NaN/+inf or all weights zero
    if (ok) {
        if (KIND == KIND_MULTI) {
            // two draws per thread (half a Philox block), so that twice as many warps share the searches
            const int n2 = (int)((p.P + 1) >> 1), h_end = (int)((int64_t)n2 * (t + 1) / T);
            for (int h = (int)((int64_t)n2 * t / T) + tid; h < h_end && t < T; h += kThreads) {
                const u32x4 r = philox((uint32_t)h >> 1, 0u, p.filter, TAG_MULTI, p.key0, p.key1);
                const uint32_t x[2] = {h & 1 ? r.z : r.x, h & 1 ? r.w : r.y};
                int32_t a[2];
                small_draws2<ONE>(x, sm.table, vall, slot, p, (int)PA, W, a);
                p.anc[2 * h] = a[0];
                if (2 * h + 1 < p.P) p.anc[2 * h + 1] = a[1];
            }
        } else if (t < T) {
            assign_tile<KIND, KK, CAP>(p, sm.as, map, stage, th, ts, t0 - p.lead);
        }
    }
    if (trace) {
        __syncthreads();
        trace_stamp(trace, p.trace_cap, t, 4);
    }
    // no CTA leaves while another may still read its record or its cumulative weights
    if (!ONE) cg::this_cluster().sync();
}

template <int KIND, int KK>
cudaError_t launch_kk(const SortedParams& p, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = small_smem(KIND, KK);
    if (KIND == KIND_MULTI) cfg.dynamicSmemBytes += (size_t)p.n_tiles * weight_slot(p.tile) * sizeof(float);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (p.n_tiles == 1) {
        cfg.gridDim = dim3(1);
        return cudaLaunchKernelEx(&cfg, k_small<KIND, KK, true>, p);
    }
    int c = 2;
    while (c < p.n_tiles) c *= 2;
    cfg.gridDim = dim3(c);
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = c;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k_small<KIND, KK, false>, p);
}

template <int KIND>
cudaError_t launch_kind(const SortedParams& p, cudaStream_t s) {
    const int q = (p.tile + kThreads - 1) / kThreads;  // elements per thread of a full tile
    if (q <= 4) return launch_kk<KIND, 4>(p, s);
    if (q <= 8) return launch_kk<KIND, 8>(p, s);
    return launch_kk<KIND, 16>(p, s);
}

// Raises the kernels' limits; returns the largest cluster every one of them can be launched with.
template <int KIND, int KK>
int prepare_kk(cudaError_t& e) {
    const int smem = (int)(small_smem(KIND, KK) + (KIND == KIND_MULTI ? kSmallWeights * sizeof(float) : 0));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_small<KIND, KK, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_small<KIND, KK, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_small<KIND, KK, false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return 0;
    for (int c = kMaxCluster; c >= 2; c /= 2) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = (size_t)smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = c;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, k_small<KIND, KK, false>, &cfg) == cudaSuccess && clusters >= 1)
            return c;
        cudaGetLastError();  // a cluster this device cannot hold: try a smaller one
    }
    return 1;
}

template <int KIND>
int prepare_kind(cudaError_t& e) {
    const int a = prepare_kk<KIND, 4>(e), b = prepare_kk<KIND, 8>(e), c = prepare_kk<KIND, 16>(e);
    return a < b ? (a < c ? a : c) : (b < c ? b : c);
}

}  // namespace

// Once per device: the largest number of tiles a small call of each kind may have.
cudaError_t prepare_small(int (&tiles)[3]) {
    cudaError_t e = cudaSuccess;
    tiles[KIND_MULTI] = prepare_kind<KIND_MULTI>(e);
    tiles[KIND_STRAT] = prepare_kind<KIND_STRAT>(e);
    tiles[KIND_SYS] = prepare_kind<KIND_SYS>(e);
    return e;
}

// Whether a call of p.n_tiles tiles of p.tile elements is served here.
bool small_fits(int kind, const SortedParams& p, int tiles) {
    return p.n_tiles <= tiles && (kind != KIND_MULTI || p.n_tiles * weight_slot(p.tile) <= kSmallWeights);
}

cudaError_t launch_small(int kind, const SortedParams& p, cudaStream_t s) {
    if (p.n_tiles < 1 || p.n_tiles > kMaxCluster || p.tile < 4 || p.tile > kTileMax) return cudaErrorInvalidValue;
    switch (kind) {
    case KIND_MULTI: return launch_kind<KIND_MULTI>(p, s);
    case KIND_STRAT: return launch_kind<KIND_STRAT>(p, s);
    case KIND_SYS: return launch_kind<KIND_SYS>(p, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace pf

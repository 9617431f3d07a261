// Single filters beyond the tiles of one cooperative launch: the cumulative
// schemes (Section 2, Figure 1a-c) for P + lead > PF_MAX_CUMULATIVE, up to
// 2^31 - 1 particles.  Three ordinary launches in stream order, with no wait of
// one CTA on another:
//   1. k_large_scan: tiles of 8192 log-weights, grid-stride, each copied
//      into shared memory while the CTA's previous tile is scanned: the tile
//      scan (pf_tile.cuh), a 16-byte record (k_t, S_t, i_last) and the tile's
//      cumulative weights v_i (sign bit: zero weight);
//   2. k_large_carries: one cluster of CTAs: the largest tile exponent K, the exact
//      prefix B_t = sum_{t' < t} S_t' 2^{k_t' - K} (128-bit fixed point), W = B_T, every
//      tile's offset map from B_t and B_{t+1} (the same function of a boundary for both
//      ends, so neighbouring tiles share their end exactly), and the multinomial's tile table;
//   3. k_large_assign (systematic, stratified): the tiles' offsets and their run-length
//      decode (pf_assign.cuh), warp by warp: a warp reads its share of a tile's v_i back
//      (not rescanned: 6-7% faster at 2^25 - 2^27 for the extra 4 B written and read per
//      particle) and meets no barrier; tiles that own too many offsets for that are left
//      to the whole CTA at the end.  Multinomial: the same pass decodes the guide table
//      (the first particle above each of P/4 evenly spaced targets), then k_large_draws
//      runs the draws, each through its guide entry and one window of v_i, or, where
//      that does not settle it, by binary searches over the tile table and the tile's v_i.
// The tiles, the exact boundaries and the per-tile arithmetic are those of the
// single-launch kernels, so the results follow the same rules.  A NaN/+inf or
// all-zero weight set records PF_ERR_DOMAIN in launch 1 or 2, and launch 3
// then writes nothing.
#include <cfloat>
#include <climits>

#include <cooperative_groups.h>

#include "pf_assign.cuh"

namespace pf {

namespace {

// What launch 2 hands to launch 3 (global memory).
struct LargeScalars {
    int ok;  // 0: a domain error was recorded, launch 3 writes nothing
    float W_hi, W_lo;
};

// A tile for launch 3: its offset map and its last positive element.
struct __align__(32) LargeMap {
    long long jlo;
    int noff;
    float x0, ir;
    int il;
};
static_assert(sizeof(LargeMap) == 32, "one sector a tile");

constexpr int kLargeTile = kTileMax;  // full tiles, 16 log-weights per thread

__device__ __forceinline__ i128 record_mass(uint4 r, int K) {
    const float sh = __uint_as_float(r.y);
    if (!(sh > 0.f)) return (i128)0;
    const int s = (int)r.x - K;
    return fixed_of(sh, s) + fixed_of(__uint_as_float(r.z), s);
}

// ---------------------------------------------------------------------------
// Launch 1: the tile scans.  A CTA's tiles are t = blockIdx.x + r gridDim.x;
// tile r + 1 is copied into one of two shared-memory buffers while tile r is
// scanned from the other.  P = 2^25 + 4096: 66 us with bulk copies (cp.async.bulk,
// whose plain order makes the scan's 16-byte reads conflict four ways), 61 us with
// per-thread copies into the conflict-free order.
// ---------------------------------------------------------------------------
constexpr size_t kScanSmem = ((sizeof(TileShared) + 15) & ~(size_t)15) + 2 * (size_t)kLargeTile * sizeof(float);

template <int KIND>
__global__ void __launch_bounds__(kThreads, 2) k_large_scan(SortedParams p, uint4* rec) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TileShared& sm = *reinterpret_cast<TileShared*>(smem_raw);
    float* slot = reinterpret_cast<float*>(smem_raw + ((sizeof(TileShared) + 15) & ~(size_t)15));
    grid_begin();
    const int tid = threadIdx.x;
    const int64_t PA = p.P + p.lead;
    const int n_mine = (p.n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;  // grid <= tiles
    auto start = [&](int r) {
        const int64_t t0 = (int64_t)(blockIdx.x + (int64_t)r * gridDim.x) * kLargeTile;
        stage_tile(p.lw + t0, (int)min((int64_t)kLargeTile, PA - t0), slot + (r & 1) * kLargeTile);
    };
    start(0);
    TileThread th;
    for (int r = 0; r < n_mine; ++r) {
        const int t = (int)blockIdx.x + r * (int)gridDim.x;
        const int64_t t0 = (int64_t)t * kLargeTile;
        const int n = (int)min((int64_t)kLargeTile, PA - t0);
        if (r + 1 < n_mine) {
            start(r + 1);
            async_wait<1>();
        } else {
            async_wait<0>();
        }
        __syncthreads();
        // a ragged last tile: its tail is not in the copy; read it from global memory
        const int lo = t == 0 ? p.lead : 0;
        const TileSummary ts = (n & 3) == 0 ? tile_scan_k<16, true>(slot + (r & 1) * kLargeTile, lo, n, sm, th)
                                            : tile_scan_k<16>(p.lw + t0, lo, n, sm, th);
        if (ts.bad && tid == 0) set_status(p.ctl + CTL_STATUS, ST_DOMAIN);
        write_tile_v<16>(p, th, t0, n);  // read back by launch 3
        if (tid == 0)
            rec[t] = make_uint4((uint32_t)ts.k, __float_as_uint(ts.bad ? NAN : ts.S.hi), __float_as_uint(ts.S.lo),
                                (uint32_t)ts.i_last);
        __syncthreads();  // the buffer and the tile scan's shared fields are reused
    }
}

// ---------------------------------------------------------------------------
// Launch 2: one cluster of kCarryCtas CTAs, each a contiguous range of tiles; the
// ranges' largest exponents and exact masses are exchanged through distributed
// shared memory.  Bound by the latency of its chain (128-bit shifts, two divisions, the
// strata's draws): at 4097 tiles 13 us for one CTA, for nine CTAs each summing all
// records, and for the cluster, whose share of records per thread stays an eighth.
// pm: the parameters of the offsets (multinomial: the guide's M bucket edges).
// ---------------------------------------------------------------------------
constexpr int kCarryCtas = 8;

template <int KIND>
__global__ void __cluster_dims__(kCarryCtas) __launch_bounds__(kThreads)
    k_large_carries(SortedParams pm, const uint4* rec, LargeMap* maps, TableEntry* table, LargeScalars* out) {
    namespace cg = cooperative_groups;
    __shared__ int red[kWarps];
    __shared__ i128 wsum[kWarps];
    __shared__ int cta_k;     // this CTA's largest exponent with weight (kBadRange: a NaN or +inf tile)
    __shared__ i128 cta_sum;  // this CTA's mass
    __shared__ long long jnext[kThreads + 1];
    constexpr int kBadRange = INT_MAX;
    grid_begin();
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int T = pm.n_tiles;
    const int per = ((T + kCarryCtas - 1) / kCarryCtas + 1) & ~1;
    const int t_lo = min(T, (int)blockIdx.x * per), t_hi = min(T, t_lo + per);
    // the largest exponent among tiles with weight, and the domain check
    constexpr int kBatch = 4;  // records in flight per thread
    int kmax = INT_MIN;
    for (int t0 = t_lo + tid; t0 < t_hi; t0 += kBatch * kThreads) {
        uint2 r[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
            r[u] = t0 + u * kThreads < t_hi ? *reinterpret_cast<const uint2*>(rec + t0 + u * kThreads)
                                            : make_uint2(0u, 0u);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const float sh = __uint_as_float(r[u].y);
            if (!(sh <= FLT_MAX)) kmax = kBadRange;
            else if (sh > 0.f) kmax = max(kmax, (int)r[u].x);
        }
    }
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) red[warp] = kmax;
    __syncthreads();
    kmax = __reduce_max_sync(0xffffffffu, lane < kWarps ? red[lane] : INT_MIN);
    if (tid == 0) cta_k = kmax;
    cluster.sync();
    int K = INT_MIN;
    for (int c = 0; c < kCarryCtas; ++c) K = max(K, *cluster.map_shared_rank(&cta_k, c));
    const bool ok = K != INT_MIN && K != kBadRange;  // the same in every CTA
    // this CTA's mass, then those before it and the total (integer sums: any order)
    if (ok) {
        i128 run = 0;
        for (int t0 = t_lo + tid; t0 < t_hi; t0 += kBatch * kThreads) {
            uint4 r[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u)
                r[u] = t0 + u * kThreads < t_hi ? rec[t0 + u * kThreads] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int u = 0; u < kBatch; ++u)
                if (t0 + u * kThreads < t_hi) run += record_mass(r[u], K);
        }
        run = warp_scan_i128(run, lane);
        if (lane == 31) wsum[warp] = run;
        __syncthreads();
        if (warp == 0) {
            const i128 v = warp_scan_i128(lane < kWarps ? wsum[lane] : (i128)0, lane);
            if (lane == 31) cta_sum = v;
        }
    }
    cluster.sync();
    i128 base = 0, Wt = 0;
    if (ok) {
        for (int c = 0; c < kCarryCtas; ++c) {
            const i128 v = *cluster.map_shared_rank(&cta_sum, c);
            if (c < (int)blockIdx.x) base += v;
            Wt += v;
        }
    }
    cluster.sync();  // no CTA leaves while another may still read its shared memory
    if (!ok) {
        if (tid == 0 && blockIdx.x == 0) {
            set_status(pm.ctl + CTL_STATUS, ST_DOMAIN);
            out->ok = 0;
        }
        return;
    }
    AssignShared as;
    as.Wt = Wt;
    as.K = K;
    const fpair W = fixed_to_pair(Wt);
    as.W_hi = W.hi;
    as.W_lo = W.lo;
    const fpair Pp = fast_two_sum((float)pm.P, (float)(pm.P - (int64_t)(float)pm.P));  // P exactly
    const fpair PW = pair_div(Pp, W);
    constexpr int kMapKind = KIND == KIND_MULTI ? KIND_SYS : KIND;
    const float u = kMapKind == KIND_SYS ? offset_uniform(pm) : 0.f;
    for (int t0 = t_lo; t0 < t_hi; t0 += kThreads) {
        const int t = t0 + tid;
        const uint4 r = t < t_hi ? rec[t] : make_uint4(0u, 0u, 0u, 0xffffffffu);
        const i128 mine = t < t_hi ? record_mass(r, K) : (i128)0;
        const i128 inc = warp_scan_i128(mine, lane);
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        const i128 ws = warp_scan_i128(lane < kWarps ? wsum[lane] : (i128)0, lane);  // every warp: the warps' totals
        const i128 before = shfl_i128(ws, max(warp, 1) - 1), round = shfl_i128(ws, kWarps - 1);
        const i128 B = base + (warp > 0 ? before : (i128)0) + inc - mine;
        base += round;
        // this tile's lower end; its upper one is the next tile's lower
        float x0 = 0.f, x0_end;
        const long long jlo = offsets_below<kMapKind>(pm, as, PW, B, u, x0);
        jnext[tid] = jlo;
        if (tid == kThreads - 1) jnext[kThreads] = offsets_below<kMapKind>(pm, as, PW, B + mine, u, x0_end);
        __syncthreads();
        if (t < t_hi) {
            LargeMap m;
            m.jlo = jlo;
            m.noff = (int)max(0LL, jnext[tid + 1] - jlo);
            m.x0 = x0;
            m.ir = PW.hi * pow2f((int)r.x - K);
            m.il = (int)r.w;
            maps[t] = m;
            if (KIND == KIND_MULTI) {
                const fpair b = fixed_to_pair(B);
                table[t] = {b.hi, b.lo, pow2f(K - (int)r.x), (int)r.w};
            }
        }
        // the next round writes wsum only after every thread has read it (the barrier
        // above), and jnext only after its own first barrier
    }
    if (tid == 0 && blockIdx.x == 0) *out = {1, W.hi, W.lo};
}

// ---------------------------------------------------------------------------
// Launch 3, systematic / stratified, and the multinomial's guide table g[b], b < M =
// P / 4, the first particle whose cumulative weight exceeds the bucket edge (b / M) W:
// the systematic assignment of M offsets with no uniform shift (p: the call's
// parameters, or those with anc = g, P = M, guide = 1; PA the call's P + lead).
// ---------------------------------------------------------------------------
constexpr int kMapBatch = 64;  // tiles whose maps a CTA holds at once

struct LargeShared {
    AssignShared as;
    LargeMap maps[kMapBatch];
};
static_assert(sizeof(LargeShared) % 16 == 0, "the staging buffers are 16-byte aligned");

// Bound by DRAM and its latency (systematic: 5 TB/s of reads and writes) and, with the
// strata's draws, by instruction issue (65% of the slots).  Maps formed by warp 0 behind
// a barrier per tile, and tiles staged by bulk copies behind another, had taken 77 us
// (systematic) and 112 us (stratified) at P = 2^25 + 4096; without any barrier between
// the maps' batches 53 and 79 us.  Asking L2 for the next share while decoding one: 56 and 77 us.
template <int KIND, int S>
__global__ void __launch_bounds__(kThreads, 2) k_large_assign(SortedParams p, int64_t PA, const LargeMap* maps,
                                                              const LargeScalars* sc) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LargeShared& sm = *reinterpret_cast<LargeShared*>(smem_raw);
    int32_t* stage = reinterpret_cast<int32_t*>(smem_raw + sizeof(LargeShared));
    grid_begin();
    const int tid = threadIdx.x;
    if (!sc->ok) return;  // launch 2 recorded a domain error
    const int n_mine = (p.n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;  // grid <= tiles
    warp_stage_init<KIND, kIoCap>(stage);
    TileThread th;
    TileSummary ts;
    for (int r0 = 0; r0 < n_mine; r0 += kMapBatch) {
        const int n = min(kMapBatch, n_mine - r0);
        if (tid < n) sm.maps[tid] = maps[(int)blockIdx.x + (r0 + tid) * (int)gridDim.x];
        __syncthreads();
        auto tile = [&](int r, bool heavy) {
            const LargeMap m = sm.maps[r];
            if ((m.noff > kWarpOffsets) != heavy) return;
            const int64_t t0 = (int64_t)((int)blockIdx.x + (r0 + r) * (int)gridDim.x) * kLargeTile;
            read_tile_v<16>(p.v_out + t0, (int)min((int64_t)kLargeTile, PA - t0), th);
            ts.i_last = m.il;
            // without SPILL: stratified, 10^8 particles 391 us, with it 396
            assign_tile<KIND, 16, kIoCap, S, true, false>(p, sm.as, {m.jlo, m.noff, m.x0, m.ir}, stage, th, ts,
                                                          t0 - p.lead);
        };
        bool any = false;
        for (int r = 0; r < n; ++r) {
            any |= sm.maps[r].noff > kWarpOffsets;
            tile(r, false);
        }
        if (any)  // block-uniform: the same maps in every thread
            for (int r = 0; r < n; ++r) tile(r, true);
        __syncthreads();  // the maps are replaced
    }
}

// ---------------------------------------------------------------------------
// Launch 4, multinomial: each draw first reads its guide entry and one 16-element window
// of v (quad-cooperatively, pf_assign.cuh); a lane whose four draws the guide did not all
// settle redoes its Philox block by the plain binary searches of Section 2's description
// over the tile table and the tile's cumulative weights, through L2 (same results).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads, 2) k_large_draws(SortedParams p, const TableEntry* table,
                                                             const LargeScalars* sc, const int32_t* g, int64_t M) {
    grid_begin();
    if (!sc->ok) return;
    const float Wh = sc->W_hi, Wl = sc->W_lo;
    const int64_t PA = p.P + p.lead;
    const int64_t nq = (p.P + 3) >> 2;  // four draws per Philox block
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    // the same number of passes in every thread of a CTA (the guided draws read their
    // windows quad-cooperatively); a lane past the end redraws block 0 and stores nothing
    for (int64_t q0 = (int64_t)blockIdx.x * kThreads; q0 < nq; q0 += stride) {
        const bool mine = q0 + threadIdx.x < nq;
        if (!__any_sync(0xffffffffu, mine)) continue;  // the whole warp is past the end
        const int64_t q = mine ? q0 + threadIdx.x : 0;
        const u32x4 r = philox((uint32_t)q, 0u, p.filter, TAG_MULTI, p.key0, p.key1);
        int32_t a[4];
        bool settled = true;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            bool ok;
            a[s] = multinomial_draw_guided(word_of(r, s), table, p.n_tiles, p.v_out, g, M, kLargeTile, PA, p.lead, Wh,
                                           Wl, ok);
            settled = settled && ok;
        }
        if (!settled)
            multinomial_draws4(r, table, p.n_tiles,
                               [&](int t, int64_t, int i) { return __ldcg(p.v_out + (int64_t)t * kLargeTile + i); },
                               kLargeTile, PA, p.lead, Wh, Wl, a);
        if (!mine) continue;
        const int64_t j = 4 * q;
        if (j + 3 < p.P && (((uintptr_t)(p.anc + j)) & 15u) == 0) {
            __stcs(reinterpret_cast<int4*>(p.anc + j), make_int4(a[0], a[1], a[2], a[3]));
        } else {
            for (int s = 0; s < 4; ++s)
                if (j + s < p.P) __stcs(p.anc + j + s, a[s]);
        }
    }
}

}  // namespace

namespace {
constexpr size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct LargeLayout {
    size_t rec, maps, table, scalars, v, g, total;
};

// Multinomial guide buckets: a quarter of the particles.
int64_t guide_buckets(int64_t P) { return (P + 3) / 4; }

LargeLayout large_layout(int kind, int64_t PA) {
    const size_t T = (size_t)((PA + kLargeTile - 1) / kLargeTile);
    const bool multi = kind == KIND_MULTI;
    LargeLayout l;
    l.rec = 0;
    l.maps = align256(T * sizeof(uint4));
    l.table = align256(l.maps + T * sizeof(LargeMap));
    l.scalars = align256(l.table + (multi ? T * sizeof(TableEntry) : 0));
    l.v = align256(l.scalars + sizeof(LargeScalars));
    l.g = align256(l.v + (size_t)PA * sizeof(float));
    l.total = l.g + (multi ? (size_t)guide_buckets(PA) * sizeof(int32_t) : 0);
    return l;
}

constexpr size_t kAssignSmem = sizeof(LargeShared) + 2 * (size_t)kIoCap * sizeof(int32_t);
constexpr int kGuideS = 8;  // guide: a warp's 512 elements hold ~128 bucket edges

template <int KIND>
cudaError_t launch_large_kind(SortedParams p, unsigned char* scratch, int num_sms, cudaStream_t s) {
    const int64_t PA = p.P + p.lead;
    const LargeLayout l = large_layout(KIND, PA);
    const int T = p.n_tiles;
    uint4* rec = reinterpret_cast<uint4*>(scratch + l.rec);
    LargeMap* maps = reinterpret_cast<LargeMap*>(scratch + l.maps);
    TableEntry* table = reinterpret_cast<TableEntry*>(scratch + l.table);
    LargeScalars* sc = reinterpret_cast<LargeScalars*>(scratch + l.scalars);
    p.v_out = reinterpret_cast<float*>(scratch + l.v);
    const int grid = T < 2 * num_sms ? T : 2 * num_sms;  // two resident CTAs per SM, grid-stride over tiles
    cudaError_t e = launch_overlapped(k_large_scan<KIND>, grid, kThreads, kScanSmem, s, p, rec);
    if (e != cudaSuccess) return e;
    SortedParams pm = p;  // of the offsets: the call's, or the guide's
    const int64_t M = guide_buckets(p.P);
    int32_t* g = reinterpret_cast<int32_t*>(scratch + l.g);
    if (KIND == KIND_MULTI) {
        pm.anc = g;
        pm.P = M;
        pm.Pd = (double)M;
        pm.guide = 1;
    }
    e = launch_overlapped(k_large_carries<KIND>, kCarryCtas, kThreads, 0, s, pm, rec, maps, table, sc);
    if (e != cudaSuccess) return e;
    constexpr int kMapKind = KIND == KIND_MULTI ? KIND_SYS : KIND;
    constexpr int S = KIND == KIND_MULTI ? kGuideS : warp_stage_per_lane(16);
    e = launch_overlapped(k_large_assign<kMapKind, S>, grid, kThreads, kAssignSmem, s, pm, PA, maps, sc);
    if constexpr (KIND == KIND_MULTI) {
        if (e != cudaSuccess) return e;
        const int64_t nq = (p.P + 3) >> 2;
        int64_t gd = (nq + kThreads - 1) / kThreads;
        if (gd > (int64_t)num_sms * 16) gd = (int64_t)num_sms * 16;
        e = launch_overlapped(k_large_draws, (unsigned)gd, kThreads, 0, s, p, table, sc, g, M);
    }
    return e;
}
}  // namespace

// Once per device: the scans' tile buffers and the assignment kernels' staging
// buffers exceed the default dynamic shared-memory limit.
cudaError_t prepare_large() {
    constexpr int S = warp_stage_per_lane(16);
    cudaError_t e = cudaFuncSetAttribute(k_large_assign<KIND_SYS, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kAssignSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_large_assign<KIND_STRAT, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kAssignSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_large_assign<KIND_SYS, kGuideS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kAssignSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_large_scan<KIND_MULTI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kScanSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_large_scan<KIND_STRAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kScanSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_large_scan<KIND_SYS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kScanSmem);
    return e;
}

size_t large_scratch_bytes(int kind, int64_t PA) { return large_layout(kind, PA).total; }

// p: the call's parameters with lw, anc, P, lead, keys, filter, ctl set; the
// tiles are set here.  scratch: large_scratch_bytes(kind, P + lead) bytes.
cudaError_t launch_large(int kind, SortedParams p, void* scratch, int num_sms, cudaStream_t s) {
    const int64_t PA = p.P + p.lead;
    const int64_t T = (PA + kLargeTile - 1) / kLargeTile;
    if (T < 1 || T > INT_MAX / 2 || num_sms < 1) return cudaErrorInvalidValue;
    p.tile = kLargeTile;
    p.n_tiles = (int)T;
    p.tiles_per_cta = 0;
    p.v_out = nullptr;
    p.c2_out = p.c1_out = nullptr;
    p.g_out = nullptr;
    p.guide = 0;
    unsigned char* sb = static_cast<unsigned char*>(scratch);
    switch (kind) {
    case KIND_MULTI: return launch_large_kind<KIND_MULTI>(p, sb, num_sms, s);
    case KIND_STRAT: return launch_large_kind<KIND_STRAT>(p, sb, num_sms, s);
    case KIND_SYS: return launch_large_kind<KIND_SYS>(p, sb, num_sms, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace pf

// Offspring/ancestor conversion for in-place particle moves (Section 2: the
// stratified and systematic schemes give offspring counts, the multinomial
// and Metropolis ones ancestors; converting between the two is direct).
//
// pf_permute rewrites any ancestor vector a into one with the same offspring
// counts o_i in which every particle with offspring keeps one of them in its
// own slot (out[i] = i); the other o_i - 1 copies of each such i (in
// increasing i) fill the slots of the particles without offspring (in
// increasing slot order).  Then out[out[j]] = out[j], so the states can be
// moved in place: row j is overwritten only if particle j has no offspring,
// and every row read belongs to a particle that keeps its slot.
//
// Passes, each over tiles of 4096 slots: offspring counts o (one atomic per run of
// equal neighbours in a row of 32: sorted ancestors, as the offset schemes give
// them, need one per survivor); per-tile sums of the extra copies max(o_i - 1, 0)
// and of the empty slots [o_i == 0], whose last CTA to finish forms their
// exclusive scans; the list E of the extra copies, each tile's run starts marked
// in shared memory and filled by a block max-scan (tiles with more than kPermPart
// extras are split over several CTAs); and the result, every slot written once in
// order: i where o_i > 0, else E at the rank of the empty slot.
//
// Bound by its launches and by L2 latency (five passes of 4 bytes a slot, of which
// only the first and the last touch the caller's arrays): one memset and four
// launches.  Stratified resampling, permutation and in-place move of 3 M rows of 64
// bytes: 113 us, 35 of them the permutation, 44 the rows (212 us in all with three
// memsets and seven launches and the rows in 128-bit chunks).
#include <climits>
#include <type_traits>

#include "pf_device.cuh"
#include "pf_index.h"
#include "pf_internal.h"
#include "pf_rows.cuh"

namespace pf {
namespace {

constexpr int kPermThreads = 512;
constexpr int kPermPer = 8;
constexpr int kPermTile = kPermThreads * kPermPer;
constexpr int kPermWarps = kPermThreads / 32;

// One count per ancestor.  A warp takes four rows of 32 consecutive entries; the
// first lane of each run of equal entries in a row adds the run's length.
__global__ void __launch_bounds__(256) k_perm_count(const int32_t* anc, int64_t P, int32_t* o, uint32_t* ctl) {
    grid_begin();
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t j0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 128; j0 < P; j0 += warps * 128) {
        int32_t a[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int64_t j = j0 + 32 * r + lane;
            a[r] = j < P ? anc[j] : INT_MIN;  // INT_MIN: past the end, counted nowhere
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (j0 + 32 * r + lane < P && (a[r] < 0 || a[r] >= P)) {
                set_status(ctl + CTL_STATUS, ST_INVALID);
                a[r] = INT_MIN;
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int32_t below = __shfl_up_sync(0xffffffffu, a[r], 1);
            const bool head = lane == 0 || below != a[r];
            const uint32_t heads = __ballot_sync(0xffffffffu, head);
            if (head && a[r] >= 0) {
                const uint32_t later = heads & ~(0xffffffffu >> (31 - lane));  // heads above this lane
                atomicAdd(o + a[r], (later ? __ffs((int)later) - 1 : 32) - lane);
            }
        }
    }
}

// Block exclusive scan of one int per thread (kPermThreads threads); *total gets the sum.
__device__ __forceinline__ int block_excl_scan(int x, int* red, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int h = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += h;
    }
    if (lane == 31) red[warp] = inc;
    __syncthreads();
    int w = lane < kPermWarps ? red[lane] : 0;
#pragma unroll
    for (int off = 1; off < kPermWarps; off <<= 1) {
        const int h = __shfl_up_sync(0xffffffffu, w, off);
        if (lane >= off) w += h;
    }
    total = __shfl_sync(0xffffffffu, w, kPermWarps - 1);
    const int base = warp > 0 ? __shfl_sync(0xffffffffu, w, warp - 1) : 0;
    __syncthreads();
    return base + inc - x;
}

// This thread's kPermPer counts of its tile (1 past the end: neither extra nor empty).
__device__ __forceinline__ void load_counts(const int32_t* o, int64_t i0, int64_t P, int (&c)[kPermPer]) {
    if (i0 + kPermPer <= P) {  // the counts start on a 256-byte boundary
#pragma unroll
        for (int q = 0; q < kPermPer / 4; ++q) {
            const int4 v = reinterpret_cast<const int4*>(o + i0)[q];
            c[4 * q] = v.x;
            c[4 * q + 1] = v.y;
            c[4 * q + 2] = v.z;
            c[4 * q + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < kPermPer; ++k) c[k] = i0 + k < P ? o[i0 + k] : 1;
    }
}

// Per-tile prefixes: extra copies, empty slots, and parts (CTAs of the listing pass).
struct TilePrefix {
    int32_t extra, dead, part;
};

// Tile sums; the last CTA to finish turns them into exclusive prefixes, pre[T] holding the totals.
__global__ void __launch_bounds__(kPermThreads) k_perm_tiles(const int32_t* o, int64_t P, TilePrefix* pre, int T,
                                                             uint32_t* ctl) {
    __shared__ int red[kPermWarps];
    __shared__ int last;
    grid_begin();
    int c[kPermPer];
    load_counts(o, (int64_t)blockIdx.x * kPermTile + (int64_t)threadIdx.x * kPermPer, P, c);
    int e = 0, d = 0;
#pragma unroll
    for (int k = 0; k < kPermPer; ++k) {
        e += c[k] > 1 ? c[k] - 1 : 0;
        d += c[k] == 0;
    }
    int te, td;
    block_excl_scan(e, red, te);
    block_excl_scan(d, red, td);
    if (threadIdx.x == 0) {
        pre[blockIdx.x] = {te, td, 0};
        __threadfence();
        last = atomicAdd(ctl + CTL_PERM_COUNT, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    int ce = 0, cd = 0, cp = 0;  // carries over rounds of kPermThreads tiles
    for (int base = 0; base < T; base += kPermThreads) {
        const int t = base + threadIdx.x;
        const int xe = t < T ? __ldcg(&pre[t].extra) : 0, xd = t < T ? __ldcg(&pre[t].dead) : 0;
        const int xp = perm_parts(xe);
        int se, sd, sp;
        const int pe = block_excl_scan(xe, red, se), pd = block_excl_scan(xd, red, sd);
        const int pp = block_excl_scan(xp, red, sp);
        if (t < T) pre[t] = {ce + pe, cd + pd, cp + pp};
        ce += se;
        cd += sd;
        cp += sp;
    }
    if (threadIdx.x == 0) {
        pre[T] = {ce, cd, cp};
        ctl[CTL_PERM_COUNT] = 0u;  // ready for the next call on this stream
    }
}

// Lists the extra copies: E[r], r < extras, in increasing particle order.  CTA b is
// part b of the listing: part pt of tile t, ranks [pt kPermPart, ...) of the tile's.
__global__ void __launch_bounds__(kPermThreads) k_perm_list(const int32_t* o, int64_t P, const TilePrefix* pre, int T,
                                                            int32_t* E) {
    __shared__ int red[kPermWarps];
    __shared__ __align__(16) int32_t mark[kPermPart + 4];
    grid_begin();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int b = blockIdx.x; b < pre[T].part; b += gridDim.x) {
        int lo = 0, hi = T - 1;  // the last tile with pre.part <= b
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (pre[mid].part <= b) lo = mid;
            else hi = mid - 1;
        }
        const int t = lo;
        const int s0 = (b - pre[t].part) * kPermPart;  // this part's ranks within the tile:
        const int s1 = perm_part_end(s0, pre[t + 1].extra - pre[t].extra);  // [s0, s1)
        int32_t* out = E + pre[t].extra + s0;
        const int shift = (int)(((uintptr_t)out >> 2) & 3u);  // to a 16-byte boundary
        const int end = s1 - s0 + shift;
        for (int i = 4 * tid; i < end; i += 4 * kPermThreads)
            *reinterpret_cast<int4*>(mark + i) = make_int4(-1, -1, -1, -1);
        const int64_t i0 = (int64_t)t * kPermTile + (int64_t)tid * kPermPer;
        int c[kPermPer];
        load_counts(o, i0, P, c);
        int e = 0, te;
#pragma unroll
        for (int k = 0; k < kPermPer; ++k) e += c[k] > 1 ? c[k] - 1 : 0;
        int r = block_excl_scan(e, red, te);  // also orders the clears before the marks
#pragma unroll
        for (int k = 0; k < kPermPer; ++k) {
            if (c[k] > 1) {
                const int r1 = r + c[k] - 1;
                if (r1 > s0 && r < s1) mark[max(r, s0) - s0 + shift] = (int32_t)(i0 + k);
                r = r1;
            }
        }
        __syncthreads();
        // running maximum over the marks, four entries a thread and round
        int carry = -1;
        for (int x0 = 0; x0 < end; x0 += 4 * kPermThreads) {
            const int x = x0 + 4 * tid;
            int4 v = make_int4(-1, -1, -1, -1);
            if (x < end) v = *reinterpret_cast<const int4*>(mark + x);
            v.y = max(v.x, v.y);
            v.z = max(v.y, v.z);
            v.w = max(v.z, v.w);
            int m = v.w;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int h = __shfl_up_sync(0xffffffffu, m, off);
                if (lane >= off) m = max(m, h);
            }
            int below = __shfl_up_sync(0xffffffffu, m, 1);
            if (lane == 0) below = -1;
            if (lane == 31) red[warp] = m;
            __syncthreads();
            below = max(max(below, carry), __reduce_max_sync(0xffffffffu, lane < warp ? red[lane] : -1));
            carry = max(carry, __reduce_max_sync(0xffffffffu, lane < kPermWarps ? red[lane] : -1));
            v.x = max(v.x, below);
            v.y = max(v.y, below);
            v.z = max(v.z, below);
            v.w = max(v.w, below);
            int32_t* g = out - shift + x;  // 16-byte aligned
            if (x >= shift && x + 4 <= end) {
                *reinterpret_cast<int4*>(g) = v;
            } else if (x < end) {
                if (x >= shift) g[0] = v.x;
                if (x + 1 >= shift && x + 1 < end) g[1] = v.y;
                if (x + 2 >= shift && x + 2 < end) g[2] = v.z;
                if (x + 3 < end) g[3] = v.w;
            }
            __syncthreads();  // red and (next part) mark are reused
        }
    }
}

// The result: a particle with offspring keeps its slot, the empty slots take E in order.
__global__ void __launch_bounds__(kPermThreads) k_perm_fill(const int32_t* o, int64_t P, const TilePrefix* pre,
                                                            const int32_t* E, int32_t* out) {
    __shared__ int red[kPermWarps];
    grid_begin();
    const int64_t i0 = (int64_t)blockIdx.x * kPermTile + (int64_t)threadIdx.x * kPermPer;
    int c[kPermPer];
    load_counts(o, i0, P, c);
    int d = 0, td;
#pragma unroll
    for (int k = 0; k < kPermPer; ++k) d += c[k] == 0;
    const int32_t* src = E + pre[blockIdx.x].dead + block_excl_scan(d, red, td);  // ranks below P: inside E
    int v[kPermPer];
#pragma unroll
    for (int k = 0; k < kPermPer; ++k) v[k] = c[k] == 0 ? *src++ : (int)(i0 + k);
    if (i0 + kPermPer <= P && (((uintptr_t)out) & 15u) == 0) {
#pragma unroll
        for (int q = 0; q < kPermPer / 4; ++q)
            reinterpret_cast<int4*>(out + i0)[q] = make_int4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    } else {
#pragma unroll
        for (int k = 0; k < kPermPer; ++k)
            if (i0 + k < P) out[i0 + k] = v[k];
    }
}

// Few particles: the whole permutation in one CTA and shared memory, where the passes above
// are five launches of two to three microseconds each whatever they move.  Counts and
// list lie at i + i / 32, so that threads reading their own consecutive entries meet no
// bank conflict.
// Bound by its serial phases, which grow with the particles a thread holds: 100, 4096, 8192,
// 16384 particles 3.6, 4.8, 7.1, 12.1 us against 13.5, 13.3, 13.7, 14.5 by the passes; the
// line is where shared memory ends, a little before the two meet.
constexpr int kPermSmall = 16384;  // both arrays in 132 KiB
constexpr int kPermSmallThreads = 1024;
constexpr int kPermSmallPer = kPermSmall / kPermSmallThreads;
constexpr int perm_small_at(int i) { return i + (i >> 5); }
constexpr size_t kPermSmallSmem = 2 * (size_t)(perm_small_at(kPermSmall)) * sizeof(int32_t);

__global__ void __launch_bounds__(kPermSmallThreads) k_perm_small(const int32_t* anc, int P, int32_t* out,
                                                                  uint32_t* ctl) {
    extern __shared__ int32_t perm_smem[];
    __shared__ int red[32];
    int32_t* o = perm_smem;
    int32_t* E = perm_smem + (kPermSmall + (kPermSmall >> 5));
    auto at = [](int i) { return i + (i >> 5); };
    grid_begin();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < P; i += kPermSmallThreads) {
        o[at(i)] = 0;
        E[at(i)] = -1;
    }
    __syncthreads();
    // counts: one addition per run of equal neighbours in a row of 32 (as k_perm_count)
    for (int j0 = 32 * warp; j0 < P; j0 += kPermSmallThreads) {
        const int j = j0 + lane;
        int32_t a = j < P ? anc[j] : INT_MIN;
        if (j < P && (a < 0 || a >= P)) {
            set_status(ctl + CTL_STATUS, ST_INVALID);
            a = INT_MIN;
        }
        const int32_t below = __shfl_up_sync(0xffffffffu, a, 1);
        const bool head = lane == 0 || below != a;
        const uint32_t heads = __ballot_sync(0xffffffffu, head);
        if (head && a >= 0) {
            const uint32_t later = heads & ~(0xffffffffu >> (31 - lane));
            atomicAdd(o + at(a), (later ? __ffs((int)later) - 1 : 32) - lane);
        }
    }
    __syncthreads();
    // extra copies and empty slots before this thread's entries: both below 2^15, one scan
    const int per = (P + kPermSmallThreads - 1) / kPermSmallThreads, i0 = tid * per, i1 = min(P, i0 + per);
    int x = 0;
    for (int i = i0; i < i1; ++i) {
        const int c = o[at(i)];
        x += c == 0 ? 1 : (c - 1) << 16;
    }
    int inc = x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int h = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += h;
    }
    if (lane == 31) red[warp] = inc;
    __syncthreads();
    const int before = inc - x + __reduce_add_sync(0xffffffffu, lane < warp ? red[lane] : 0);
    int r = before >> 16;
    for (int i = i0; i < i1; ++i) {
        const int c = o[at(i)];
        if (c > 1) {
            E[at(r)] = i;
            r += c - 1;
        }
    }
    __syncthreads();
    // running maximum over the marks
    int m = -1;
    for (int i = i0; i < i1; ++i) m = max(m, E[at(i)]);
    int mm = m;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int h = __shfl_up_sync(0xffffffffu, mm, off);
        if (lane >= off) mm = max(mm, h);
    }
    int carry = __shfl_up_sync(0xffffffffu, mm, 1);
    if (lane == 0) carry = -1;
    if (lane == 31) red[warp] = mm;  // every read of the sums is behind the barrier above
    __syncthreads();
    carry = max(carry, __reduce_max_sync(0xffffffffu, lane < warp ? red[lane] : -1));
    for (int i = i0; i < i1; ++i) E[at(i)] = carry = max(carry, E[at(i)]);
    __syncthreads();
    int d = before & 0xffff;
    for (int i = i0; i < i1; ++i) o[at(i)] = o[at(i)] == 0 ? E[at(d++)] : i;  // ranks below P: inside E
    __syncthreads();
    for (int i = tid; i < P; i += kPermSmallThreads) out[i] = o[at(i)];
}

// In-place gather: row j <- row perm[j] where they differ; a source must keep
// its own slot (perm[perm[j]] = perm[j]), else the row is left and
// PF_ERR_INVALID recorded.  Chunks as in the gather; a source row is read beside
// its own perm entry, before that is known to be itself (a row being overwritten
// meanwhile is read to no effect).  The next piece's entries of perm are asked for while
// this piece's rows are on their way.
//
// Bound by the reads in flight: a chunk waits for its entry of perm, then its row.
// us, row i of 3000017 moved where stratified resampling of exp(2 N(0,1)) weights moves it, rows
// of 32, 64, 96, 128 bytes, two chunks a thread without the early entries: 32, 51, 77, 80;
// four chunks a thread, a CTA for each piece: 25, 44, 80, 67; three a thread in one
// resident wave with the early entries: 27, 47, 67, 53.
template <typename VT, int U, bool POW2, typename Place = uint32_t>  // Place: as RowSplit
__global__ void __launch_bounds__(256) k_gather_inplace(VT* x, int64_t P, RowSplit split,
                                                        const int32_t* perm, uint32_t* ctl) {
    grid_begin();
    const int64_t total = P * split.vecs;
    const int64_t stride = (int64_t)gridDim.x * (256 * U);
    int64_t base = (int64_t)blockIdx.x * (256 * U) + threadIdx.x;
    int32_t a[U];  // this piece's entries of perm, and the chunks' places in their rows
    Place c[U];
    auto entries = [&](int64_t b, int32_t (&e)[U], Place (&at)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = b + u * 256;
            e[u] = -1;
            at[u] = 0;
            if (i < total) e[u] = perm[split.row<POW2>(i, at[u])];
        }
    };
    entries(base, a, c);
    for (; base < total; base += stride) {
        int32_t own[U];
        VT v[U];
        bool move[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = base + u * 256;
            Place cc;
            move[u] = i < total && a[u] != (int32_t)split.row<POW2>(i, cc);
            own[u] = -1;
            if (move[u] && a[u] >= 0 && a[u] < P) {
                own[u] = perm[a[u]];
                v[u] = load_chunk_cg(x + (int64_t)a[u] * split.vecs + c[u]);
            }
        }
        int32_t an[U];
        Place cn[U];
        entries(base + stride, an, cn);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (move[u]) {
                if (own[u] >= 0 && own[u] == a[u]) store_chunk_cs(x + base + u * 256, v[u]);
                else if (c[u] == 0) set_status(ctl + CTL_STATUS, ST_INVALID);
            }
            a[u] = an[u];
            c[u] = cn[u];
        }
    }
}

}  // namespace

// Scratch: the tile prefixes, then the counts o and the list E (16-byte loads of o: 256-byte aligned).
static size_t perm_counts_at(int64_t T) { return (((size_t)T + 1) * sizeof(TilePrefix) + 255) & ~(size_t)255; }

size_t permute_scratch_bytes(int64_t P) {
    if (P <= kPermSmall) return 0;  // one CTA, in shared memory
    const int64_t T = (P + kPermTile - 1) / kPermTile;
    return perm_counts_at(T) + (((size_t)P * sizeof(int32_t) + 255) & ~(size_t)255) + (size_t)P * sizeof(int32_t);
}

// Once per device.
cudaError_t prepare_permute() {
    return cudaFuncSetAttribute(k_perm_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPermSmallSmem);
}

cudaError_t launch_permute(const int32_t* anc, int64_t P, int32_t* out, void* scratch, uint32_t* ctl, int num_sms,
                           cudaStream_t s) {
    if (P <= kPermSmall) {
        return launch_overlapped(k_perm_small, 1, kPermSmallThreads, kPermSmallSmem, s, anc, (int)P, out, ctl);
    }
    const int T = (int)((P + kPermTile - 1) / kPermTile);
    TilePrefix* pre = static_cast<TilePrefix*>(scratch);
    int32_t* o = reinterpret_cast<int32_t*>((char*)scratch + perm_counts_at(T));
    int32_t* E = reinterpret_cast<int32_t*>((char*)o + (((size_t)P * sizeof(int32_t) + 255) & ~(size_t)255));
    cudaError_t e = cudaMemsetAsync(o, 0, (size_t)P * sizeof(int32_t), s);
    if (e != cudaSuccess) return e;
    int64_t blocks = (P + 1023) / 1024;  // 8 warps of 128 entries
    if (blocks > (int64_t)num_sms * 8) blocks = (int64_t)num_sms * 8;
    e = launch_overlapped(k_perm_count, (unsigned)blocks, 256, 0, s, anc, P, o, ctl);
    if (e == cudaSuccess) e = launch_overlapped(k_perm_tiles, (unsigned)T, kPermThreads, 0, s, o, P, pre, T, ctl);
    // at most T + P / kPermPart parts; a resident wave takes them in turn
    const int64_t parts = T + P / kPermPart, wave = (int64_t)num_sms * 4;
    if (e == cudaSuccess)
        e = launch_overlapped(k_perm_list, (unsigned)(parts < wave ? parts : wave), kPermThreads, 0, s, o, P, pre, T, E);
    if (e == cudaSuccess) e = launch_overlapped(k_perm_fill, (unsigned)T, kPermThreads, 0, s, o, P, pre, E, out);
    return e;
}

cudaError_t launch_gather_inplace(void* x, int64_t P, int64_t row_bytes, const int32_t* perm, uint32_t* ctl,
                                  int num_sms, cudaStream_t s) {
    auto go = [&](auto* p, auto unroll, int wave, int full) {
        using VT = std::remove_pointer_t<decltype(p)>;
        constexpr int U = decltype(unroll)::value;
        const int64_t vecs = row_bytes / (int64_t)sizeof(VT);
        const RowSplit split = row_split(vecs, P * vecs);
        const unsigned blocks = chunk_grid(P * vecs, 256 * U, num_sms, wave, full, wave);
        return launch_overlapped(split.wide() ? k_gather_inplace<VT, U, false, uint64_t>
                                 : split.pow2 ? k_gather_inplace<VT, U, true>
                                              : k_gather_inplace<VT, U, false>,
                                 blocks, 256, 0, s, p, P, split, perm, ctl);
    };
    const uintptr_t a = (uintptr_t)x | (uintptr_t)row_bytes;
    constexpr int kNever = 1 << 22;  // one resident wave however many pieces there are
    const std::integral_constant<int, 3> three;
    const std::integral_constant<int, 4> four;
    // 256-bit chunks: rows of one or two are read one row's length apart and do best with the
    // most reads in flight; longer rows with the wave (both sides measured above)
    if ((a & 31) == 0) {
        u32x8* q = static_cast<u32x8*>(x);
        return row_bytes <= 64 ? go(q, four, 4, 12) : go(q, three, 4, kNever);
    }
    if ((a & 15) == 0) return go(static_cast<uint4*>(x), four, 8, 40);
    // 4-byte chunks (1.2e7 rows of 4 and 12 bytes: 27 and 93 us as a wave, 33 and 110 in full)
    if ((a & 7) == 0) return go(static_cast<uint2*>(x), four, 5, kNever);
    return go(static_cast<uint32_t*>(x), four, 5, kNever);
}

}  // namespace pf

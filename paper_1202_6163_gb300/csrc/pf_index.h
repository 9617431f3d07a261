// Index arithmetic of the kernels, written so that host code can run it too: where a
// mistake would read or write out of range, it is checked on the CPU over more shapes than
// a GPU test can reach.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define PF_HD __host__ __device__ __forceinline__
#else
#define PF_HD inline
#endif

namespace pf {

// ---------------------------------------------------------------------------
// The strata of one warp of the stratified assignment, counted from its tile's first offset
// jlo.  Their uniforms lie in the warp's buffer by whole Philox blocks of four, from that of
// lane 0's lowest stratum on.
// ---------------------------------------------------------------------------
PF_HD long long strata_block(long long jlo, int k) { return (jlo + k) >> 2; }
// The place of stratum 0 (negative in all warps but the first) for a buffer from block g0 on.
PF_HD int strata_at(long long jlo, long long g0) { return (int)(jlo - 4 * g0); }
// The place of stratum k.  A lane without weight may ask for one below the buffer's (past the
// tile's end it may hold any coordinate); what it gets is not used.
PF_HD int strata_index(int at, int k) { return at + k < 0 ? 0 : at + k; }
// Whether a lane bounds each of its look-ups: its lowest stratum kb0 or its highest kl0 lies
// outside the tile (at the tile's ends, by rounding), or no element of it has weight (pos = 0).
// The strata of any other lane are lane 0's or later, and rise along the lane.
PF_HD bool strata_clamped(int kb0, int kl0, int kmax, uint32_t pos) { return kb0 < 0 || kl0 > kmax || pos == 0u; }

// ---------------------------------------------------------------------------
// Parts of the permutation's listing (pf_permute.cu): a tile's extra copies, up to P - 1 =
// 2^31 - 2 of them, kPermPart to a part.  Sums with kPermPart would pass 2^31.
// ---------------------------------------------------------------------------
constexpr int kPermPart = 8192;  // extras one CTA lists: twice a tile's mean share
PF_HD int perm_parts(int extras) { return extras / kPermPart + (extras % kPermPart != 0 ? 1 : 0); }
// The end of the part that starts at rank s0 < extras.
PF_HD int perm_part_end(int s0, int extras) { return s0 + (extras - s0 < kPermPart ? extras - s0 : kPermPart); }

// ---------------------------------------------------------------------------
// Runs and chunks of a tile's offsets (pf_assign.cuh), up to 2^31 - 1 of them in one tile.
// ---------------------------------------------------------------------------
// The end of the chunk of at most `chunk` offsets that starts at c0 < noff.
PF_HD int chunk_end(int c0, int noff, int chunk) { return c0 + (noff - c0 < chunk ? noff - c0 : chunk); }

// The pieces of four entries that thread t of `threads` stores of the `body` entries (a
// multiple of four) behind the first `head` of a run.  Unsigned: the step past the end of a
// run of 2^31 - 1 entries stays above every entry.
struct FillPieces {
    uint32_t x, end, step;
    PF_HD FillPieces(int head, int body, int t, int threads)
        : x((uint32_t)(head + 4 * t)), end((uint32_t)(head + body)), step(4u * (uint32_t)threads) {}
};

// ---------------------------------------------------------------------------
// Chunk index -> (row, place in the row) of the row moves, for rows of `vecs` chunks: a shift
// for a power of two; else, below 2^32 chunks, a multiplication by the rounded-up
// reciprocal 2^(32 + shift) / vecs less its leading bit (Granlund and Montgomery,
// "Division by invariant integers using multiplication", PLDI 1994, Fig. 4.1: exact
// for every 32-bit dividend); beyond, a 64-bit division.
// ---------------------------------------------------------------------------
PF_HD uint32_t mulhi32(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

struct RowSplit {
    int64_t vecs;
    int pow2, shift;      // shift: ceil(log2 vecs)
    uint32_t magic;       // 0: divide in 64 bits
    // Place: uint32_t, or, for rows that are `wide`, uint64_t.
    template <bool POW2, typename Place>
    PF_HD int64_t row(int64_t i, Place& place) const {
        if (POW2) {
            place = (Place)(i & (vecs - 1));
            return i >> shift;
        }
        int64_t j;
        if (magic != 0u) {
            const uint32_t n = (uint32_t)i, t = mulhi32(magic, n);
            j = (t + ((n - t) >> 1)) >> (shift - 1);
        } else {
            j = i / vecs;
        }
        place = (Place)(i - j * vecs);
        return j;
    }
    bool wide() const { return vecs > 0xffffffffLL; }  // a place takes more than 32 bits
};

inline RowSplit row_split(int64_t vecs, int64_t total) {
    RowSplit r{vecs, (vecs & (vecs - 1)) == 0, 0, 0u};
    while ((1LL << r.shift) < vecs) ++r.shift;
    if (!r.pow2 && total <= 0xffffffffLL && vecs <= 0x7fffffffLL)
        r.magic = (uint32_t)(((1ull << 32) * ((1ull << r.shift) - (uint64_t)vecs)) / (uint64_t)vecs + 1ull);
    return r;
}

}  // namespace pf

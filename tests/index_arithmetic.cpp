// Runs the kernels' shared index arithmetic (csrc/pf_index.h) on the CPU over shapes at the
// edges of what the entry points accept; prints the first violation and exits 1.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>

#include "pf_index.h"

#define REQUIRE(cond, ...)            \
    do {                              \
        if (!(cond)) {                \
            std::printf(__VA_ARGS__); \
            std::printf("\n");        \
            std::exit(1);             \
        }                             \
    } while (0)

// ---------------------------------------------------------------------------
// The stratified assignment's look-ups, warp by warp, over a tile of n elements KK to a
// thread (pf_assign.cuh, assign_warp): every index lies in the warp's buffer, UB strata at once or
// one 32 S after another.
// Lanes wholly past the tile's end hold: 0 the last element's weight, 1 zero, 2 anything.
// ---------------------------------------------------------------------------
static void strata_of_tile(std::mt19937& rng, int KK, int S, int UB, int n, const std::vector<float>& v, int noff, float x0,
                           float ir, long long jlo, int empty) {
    std::uniform_real_distribution<float> any(0.f, v[n - 1]);
    const int kmax = noff - 1;
    auto coordinate = [&](float x) { return std::fmaf(x, ir, x0); };
    for (int w = 0; w * 32 * KK < n; ++w) {
        std::vector<float> yb(32);
        std::vector<uint32_t> pos(32, 0u);
        std::vector<std::vector<float>> y(32, std::vector<float>(KK));
        for (int l = 0; l < 32; ++l) {
            const int e0 = (w * 32 + l) * KK;
            const bool past = e0 >= n;
            const float fill = empty == 0 ? v[n - 1] : (empty == 1 ? 0.f : any(rng));
            for (int i = 0; i < KK; ++i)
                if (e0 + i < n && v[e0 + i] > (e0 + i ? v[e0 + i - 1] : 0.f)) pos[l] |= 1u << i;
            for (int i = 0; i < KK; ++i) y[l][i] = coordinate(past ? fill : v[std::min(e0 + i, n - 1)]);
            yb[l] = coordinate(e0 == 0 ? 0.f : (e0 <= n ? v[e0 - 1] : (empty == 2 ? any(rng) : fill)));
        }
        auto stratum = [](float c) { return (int)std::floor(c); };
        auto bounded = [&](float c) { return std::min(std::max(stratum(c), 0), kmax); };
        const int k_first = bounded(yb[0]);
        int k_last = 0;
        for (int l = 0; l < 32; ++l) k_last = std::max({k_last, bounded(yb[l]), bounded(y[l][KK - 1])});
        k_last = std::min(k_last + 1, kmax);
        const long long g0 = pf::strata_block(jlo, k_first);
        const int blocks = (int)(pf::strata_block(jlo, k_last) - g0) + 1, at = pf::strata_at(jlo, g0);
        auto inside = [&](int index, int size, int l) {
            REQUIRE(index >= 0 && index < size, "strata: index %d of %d, warp %d lane %d, n %d noff %d KK %d, empty lanes %d",
                    index, size, w, l, n, noff, KK, empty);
        };
        if (4 * blocks <= UB) {
            for (int l = 0; l < 32; ++l) {
                const bool clamp = pf::strata_clamped(stratum(yb[l]), stratum(y[l][KK - 1]), kmax, pos[l]);
                inside(pf::strata_index(at, bounded(yb[l])), 4 * blocks, l);
                for (int i = 0; i < KK; ++i)
                    inside(clamp ? pf::strata_index(at, bounded(y[l][i])) : at + stratum(y[l][i]), 4 * blocks, l);
            }
            continue;
        }
        // one buffer of strata at a time
        std::vector<std::vector<int>> open(32, std::vector<int>(KK + 1, 1));
        int rounds = 0;
        for (int k0 = k_first; k0 < INT_MAX; ++rounds) {
            REQUIRE(rounds <= noff / (32 * S - 3) + 1, "strata: no end, n %d noff %d", n, noff);
            const int w_at = pf::strata_at(jlo, pf::strata_block(jlo, k0)), w_end = 32 * S - w_at;
            int next = INT_MAX;
            for (int l = 0; l < 32; ++l)
                for (int i = 0; i <= KK; ++i) {
                    if (!open[l][i]) continue;
                    const int k = bounded(i == KK ? yb[l] : y[l][i]);
                    if (k < w_end) {
                        inside(pf::strata_index(w_at, k), 32 * S, l);
                        open[l][i] = 0;
                    } else {
                        next = std::min(next, k);
                    }
                }
            k0 = next;
        }
    }
}

static void strata() {
    std::mt19937 rng(1);
    std::uniform_real_distribution<float> unit(0.f, 1.f);
    for (int round = 0; round < 1500; ++round) {
        const int KK = 4 << (round % 3), S = KK == 16 ? 20 : (KK == 8 ? 12 : 8), tile = 512 * KK;
        const int UB = 2 * (KK == 16 || round % 2 ? 640 : 512);
        // ragged lengths that end in every warp
        const int n = round % 5 ? 1 + (int)(rng() % tile) : 4153 % tile + 1;
        std::vector<float> v(n);
        const float spread = (float)(round % 4) * 1.5f;
        const int heavy = round % 7 == 0 ? -1 : (int)(rng() % n) % (round % 2 ? 64 : n);
        float s = 0.f;
        for (int i = 0; i < n; ++i) {
            float x = rng() % 9 ? std::exp(spread * (unit(rng) + unit(rng) - 1.f)) : 0.f;
            if (i == heavy) x += unit(rng) * 8.f * n;
            v[i] = s += x;
        }
        if (!(s > 0.f)) continue;
        const int noff = 1 + (int)(rng() % 65536);  // up to kWarpOffsets
        const float x0 = 2.f * unit(rng) - 1.f, ir = (float)noff / s;
        const long long jlo = (long long)(rng() % 2147000000u);
        for (int empty = 0; empty < 3; ++empty) strata_of_tile(rng, KK, S, UB, n, v, noff, x0, ir, jlo, empty);
    }
    // one particle of 30000 offsets in front of a last tile of 4153 particles
    std::vector<float> v(4153);
    for (int i = 0; i < 4153; ++i) v[i] = 30000.f + (float)i;
    for (int empty = 0; empty < 3; ++empty) strata_of_tile(rng, 16, 20, 1280, 4153, v, 34152, 0.25f, 1.f, 33550000, empty);
}

// ---------------------------------------------------------------------------
// The permutation's parts: they cover a tile's extra copies once, in order, up to the largest count.
// ---------------------------------------------------------------------------
static void permute_parts() {
    for (long long extras : {0LL, 1LL, 8191LL, 8192LL, 8193LL, 1000003LL, (1LL << 31) - 8194, (1LL << 31) - 8193,
                             (1LL << 31) - 8192, (1LL << 31) - 8191, (1LL << 31) - 2}) {
        const int x = (int)extras, parts = pf::perm_parts(x);
        long long at = 0;
        for (int b = 0; b < parts; ++b) {
            const int s0 = b * pf::kPermPart, s1 = pf::perm_part_end(s0, x);
            REQUIRE(s0 == at && s1 > s0 && s1 - s0 <= pf::kPermPart, "parts: [%d, %d) at %lld of %lld extras", s0, s1, at, extras);
            at = s1;
        }
        REQUIRE(at == extras, "parts: %d parts list %lld of %lld extras", parts, at, extras);
    }
}

// ---------------------------------------------------------------------------
// A tile's chunks and a run's pieces cover them once, up to the largest counts.
// ---------------------------------------------------------------------------
static void runs_and_chunks() {
    for (int noff : {1, 10236, 10237, 70001, INT_MAX - 10237, INT_MAX - 10236, INT_MAX - 10235, INT_MAX}) {
        for (int chunk : {10236, 8188, 2044}) {
            int c0 = 0;
            while (c0 < noff) {
                const int c1 = pf::chunk_end(c0, noff, chunk);
                REQUIRE(c1 > c0 && c1 - c0 <= chunk && c1 <= noff, "chunk [%d, %d) of %d", c0, c1, noff);
                c0 = c1;
            }
        }
    }
    for (int threads : {32, 512})
        for (int n : {0, 3, 4, 1283, 70001, INT_MAX - 2051, INT_MAX - 2047, INT_MAX - 1, INT_MAX})
            for (int head = 0; head < 4 && head <= n; ++head) {
                const int body = (n - head) & ~3;
                long long pieces = 0;
                for (int t = 0; t < threads; t += n > 1000000 && t + 3 < threads ? threads / 2 - 1 : 1) {
                    uint32_t at = (uint32_t)head + 4u * (uint32_t)t;
                    for (pf::FillPieces f(head, body, t, threads); f.x < f.end; f.x += f.step) {
                        REQUIRE(f.x == at && f.x + 4 <= (uint32_t)(head + body), "run of %d: piece at %u", n, f.x);
                        at += 4u * (uint32_t)threads;
                        ++pieces;
                    }
                    REQUIRE(at >= (uint32_t)(head + body), "run of %d: thread %d ends at %u", n, t, at);
                }
                REQUIRE(n > 1000000 || 4 * pieces == body, "run of %d: %lld pieces", n, pieces);
            }
}

// ---------------------------------------------------------------------------
// Row and place of a chunk, from one chunk a row to rows of more than 2^32 chunks, as the row
// moves choose them (power of two or not, wide or not).
// ---------------------------------------------------------------------------
static void rows() {
    std::mt19937_64 rng(2);
    std::vector<int64_t> lengths = {0x7fffffffLL, 0x80000000LL, 0x80000001LL, 0xffffffffLL, 1LL << 32, (1LL << 32) + 1,
                                    (1LL << 33) + 5, 1LL << 34, 16000000007LL};
    for (int64_t v = 1; v < 300; ++v) lengths.push_back(v);
    for (int k = 0; k < 300; ++k) lengths.push_back(1 + (int64_t)(rng() >> (33 + rng() % 29)));
    for (int64_t vecs : lengths)
        for (int64_t n : {1LL, 2LL, 3LL, 1000LL, 0xffffffffLL / vecs, 0xffffffffLL / vecs + 1, (1LL << 33) / vecs + 1}) {
            if (n < 1) continue;
            const int64_t total = n * vecs;
            const pf::RowSplit s = pf::row_split(vecs, total);
            auto check = [&](int64_t i) {
                if (i < 0 || i >= total) return;
                uint32_t narrow = 0;
                uint64_t wide = 0;
                const int64_t j = s.wide() ? s.row<false>(i, wide) : (s.pow2 ? s.row<true>(i, narrow) : s.row<false>(i, narrow));
                const int64_t place = s.wide() ? (int64_t)wide : (int64_t)narrow;
                REQUIRE(j == i / vecs && place == i % vecs, "rows of %lld: chunk %lld is (%lld, %lld)", (long long)vecs,
                        (long long)i, (long long)j, (long long)place);
            };
            for (int64_t i : {int64_t(0), vecs - 1, vecs, vecs + 1, total - vecs, total - 1}) check(i);
            for (int k = 0; k < 200; ++k) {
                const int64_t i = (int64_t)(rng() % (uint64_t)total);
                check(i);
                check(i - i % vecs);
                check(i - i % vecs - 1);
            }
        }
}

int main(int argc, char** argv) {
    const char* what = argc > 1 ? argv[1] : "";
    if (!std::strcmp(what, "strata")) strata();
    else if (!std::strcmp(what, "permute_parts")) permute_parts();
    else if (!std::strcmp(what, "runs_and_chunks")) runs_and_chunks();
    else if (!std::strcmp(what, "rows")) rows();
    else return 2;
    return 0;
}

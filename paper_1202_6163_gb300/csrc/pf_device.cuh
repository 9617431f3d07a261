// Device-side building blocks shared by the resampling kernels.
//
// Everything here is written for sm_103a (GB300): 32-wide warps, FP32 per
// element, FP64 only for per-tile carries (FP64 issue rate on this part is a
// small fraction of FP32), integer Philox.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "pf_internal.h"

namespace pf {

// ---------------------------------------------------------------------------
// Philox-4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 products
// whose halves are permuted and xored with the other counter words and the
// round key; the key advances by the Weyl increments each round.
// ---------------------------------------------------------------------------
struct u32x4 {
    uint32_t x, y, z, w;
};

// ROUNDS rounds of the same function: 10 is the default stream; 7 (listed in
// SC'11 among the Crush-resistant members) is the opt-in cheaper Metropolis stream.
template <int ROUNDS = 10>
__device__ __forceinline__ u32x4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                        uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        // one 32x32->64 product each (both halves used)
        const uint64_t a = (uint64_t)0xD2511F53u * c0;
        const uint64_t b = (uint64_t)0xCD9E8D57u * c2;
        c0 = (uint32_t)(b >> 32) ^ c1 ^ k0;
        c1 = (uint32_t)b;
        c2 = (uint32_t)(a >> 32) ^ c3 ^ k1;
        c3 = (uint32_t)a;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return {c0, c1, c2, c3};
}

// The ten-round function with the round keys given (kernel parameters: the keys are
// then operands of the xors, where advancing them costs two additions a round).
__device__ __forceinline__ u32x4 philox_keys(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, const PhiloxKeys& k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t a = (uint64_t)0xD2511F53u * c0;
        const uint64_t b = (uint64_t)0xCD9E8D57u * c2;
        c0 = (uint32_t)(b >> 32) ^ c1 ^ k.k0[r];
        c1 = (uint32_t)b;
        c2 = (uint32_t)(a >> 32) ^ c3 ^ k.k1[r];
        c3 = (uint32_t)a;
    }
    return {c0, c1, c2, c3};
}

__device__ __forceinline__ uint32_t word_of(const u32x4& r, int s) {
    return s == 0 ? r.x : (s == 1 ? r.y : (s == 2 ? r.z : r.w));
}

// u23: odd multiples of 2^-24 in (0,1); exact in float.  The word's top 23 bits
// make 1 + m 2^-23, and taking 1 - 2^-24 off leaves (2m + 1) 2^-24 exactly: no
// integer conversion, which issues at a quarter of the rate.
__device__ __forceinline__ float u23f(uint32_t x) {
    return __fsub_rn(__uint_as_float((x >> 9) | 0x3f800000u), 0x1.fffffep-1f);
}

// u32 = (2x+1) 2^-33 as an exact float pair (hi carries the top 24 bits).
__device__ __forceinline__ void u32_pair(uint32_t x, float& hi, float& lo) {
    hi = __uint2float_rn(x >> 8) * 0x1p-24f;
    lo = __uint2float_rn(((x & 0xFFu) << 1) | 1u) * 0x1p-33f;
}

__device__ __forceinline__ uint32_t draw_index(uint32_t x, uint32_t P) { return __umulhi(x, P); }

// ---------------------------------------------------------------------------
// Error-free transformations (Knuth's TwoSum) and float pairs.  The __f*_rn
// intrinsics keep the compiler from contracting or reordering them.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

struct fpair {
    float hi, lo;
};

__device__ __forceinline__ fpair pair_add(fpair a, fpair b) {
    float s, e;
    two_sum(a.hi, b.hi, s, e);
    e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
    const float hi = __fadd_rn(s, e);
    const float lo = __fsub_rn(e, __fsub_rn(hi, s));
    return {hi, lo};
}

// ---------------------------------------------------------------------------
// Tile reference.  A tile's weights are taken relative to 2^k (k near the
// tile's largest log-weight times log2 e), i.e. w_i = exp(lw_i - k ln 2).
// The reference k ln 2 is held as a float pair so that lw_i - k ln 2 is
// formed without rounding loss, and tiles with different k combine by exact
// binary scaling.
// ---------------------------------------------------------------------------
constexpr double kLn2 = 0.69314718055994530942;
constexpr float kLn2Hi = (float)kLn2;
constexpr float kLn2Lo = (float)(kLn2 - (double)(float)kLn2);
constexpr float kLog2e = 1.44269504088896340736f;

__device__ __forceinline__ int tile_exponent(float m) {
    // m = -inf (every weight zero in the tile): any k works, take 0.
    if (!(m > -INFINITY)) return 0;
    float km = fminf(fmaxf(m * kLog2e, -1.0e9f), 1.0e9f);
    return (int)ceilf(km);
}

__device__ __forceinline__ fpair tile_reference(int k) {
    const float kf = (float)k;  // |k| <= 1e9: exact enough; k below 2^24 is exact
    const float hi = __fmul_rn(kf, kLn2Hi);
    const float err = __fmaf_rn(kf, kLn2Hi, -hi);
    return {hi, __fmaf_rn(kf, kLn2Lo, err)};
}

// exp(lw - R) with R = (R.hi, R.lo): the subtraction is error-free and the
// residual d enters as the factor 1 + d + d^2/2 (for a reference k ln 2 beyond
// ~2^16 in magnitude, R.lo, and so d, reaches 4e-3, where the first-order
// factor alone would leave an error d^2/2 near 8e-6).  Zero for lw = -inf.
__device__ __forceinline__ float weight_rel(float lw, fpair R) {
    float s, e;
    two_sum(lw, -R.hi, s, e);
    const float d_lo = __fsub_rn(e, R.lo);
    const float x = expf(s);
    return x > 0.f ? __fmaf_rn(x, __fmaf_rn(d_lo, 0.5f * d_lo, d_lo), x) : 0.f;
}

// The same for two log-weights at once, in packed single precision (each half
// rounds as the scalar operation does, so the bits are weight_rel's), without
// the selection of zero for a zero weight: where expf gives 0 the result is 0,
// or NaN for lw = -inf (whose error term is inf - inf).
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }

__device__ __forceinline__ float2 weight_rel2(float2 lw, float2 neg_hi, float2 neg_lo) {
    const float2 s = __fadd2_rn(lw, neg_hi);
    const float2 bb = sub2(s, lw);
    const float2 e = __fadd2_rn(sub2(lw, sub2(s, bb)), sub2(neg_hi, bb));
    const float2 d = __fadd2_rn(e, neg_lo);
    const float2 x = make_float2(expf(s.x), expf(s.y));
    const float2 half = make_float2(0.5f, 0.5f);
    return __ffma2_rn(x, __ffma2_rn(d, __fmul2_rn(half, d), d), x);
}

// Minimum of three that propagates NaN (one instruction on this part).
__device__ __forceinline__ float fmin3_nan(float a, float b, float c) {
    float d;
    asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Maximum of three that propagates NaN.
__device__ __forceinline__ float fmax3_nan(float a, float b, float c) {
    float d;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// ---------------------------------------------------------------------------
// 64-bit fixed point (2^-48) <-> float without the 64-bit conversion
// instructions, which run on the FP64 pipe: 16 cycles a warp each on this part.
// Bit for bit the values of __float2ll_rn and of (float)(long long).
// ---------------------------------------------------------------------------
// __float2ll_rn(s 2^48) + __float2ll_rn(-c 2^48) for a compensated sum (s, c), s >= 0.
__device__ __forceinline__ long long fixed48_of(float s, float c) {
    const float sc = __fmul_rn(s, 0x1p48f), cc = __fmul_rn(-c, 0x1p48f);
    if (!(s < 64.f)) return __float2ll_rn(sc) + __float2ll_rn(cc);  // weights far above 1, or NaN: c may be large too
    // s < 64: Kahan's term is at most half an ulp of s, |c| <= 2^-19, so cc is below 2^30 and its
    // conversion to 32 bits exact; sc is an integer from 2^24 on
    const uint32_t b = __float_as_uint(sc);
    const int sh = (int)(b >> 23) - 150;
    const long long whole = (long long)((b & 0x7fffffu) | 0x800000u) << (sh > 0 ? sh : 0);
    return (sh > 0 ? whole : (long long)__float2int_rn(sc)) + (long long)__float2int_rn(cc);
}

// (float)v 2^-48 for v >= 0: the top 32 bits of v normalised, the rest kept as a
// sticky bit, so that one 32-bit conversion rounds to nearest as the 64-bit one.
__device__ __forceinline__ float fixed48_to_float(long long v) {
    const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
    const int sh = __clz((int)hi);  // 32 when hi = 0
    uint32_t top = __funnelshift_lc(lo, hi, sh);
    const uint32_t rest = sh < 32 ? lo << sh : 0u;
    top |= rest != 0u ? 1u : 0u;
    return __fmul_rn(__uint2float_rn(top), __uint_as_float((uint32_t)(127 - 16 - sh) << 23));
}

// First statement of a kernel launched by launch_overlapped, in every thread and before any
// access to global memory: waits for the work before this grid.  The kernel may be resident
// while that work still writes, so nothing it reads counts as read-only for its lifetime: no
// load through the read-only path (__ldg, ld.global.nc), and no const __restrict__ pointer, which
// lets the compiler choose that path (ld_input).  A grid of few CTAs
// first lets the next such launch take its place on the GPU; a larger one leaves that
// to its CTAs' exits, as a grid placed beside another that fills the SMs is spread
// unevenly over them (Metropolis at P = 65536: 17 us, 36 with the early start).
constexpr unsigned kEarlyStartCtas = 38;  // a quarter of this part's 152 SMs
__device__ __forceinline__ void grid_begin() {
    if (gridDim.x <= kEarlyStartCtas) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Status word and bounded waits.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void set_status(uint32_t* status, uint32_t code) {
    atomicCAS(status, 0u, code);
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint64_t ld_relaxed_u64(const uint64_t* p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint64_t ld_acquire_u64(const uint64_t* p) {
    uint64_t v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_u64(uint64_t* p, uint64_t v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void st_relaxed_u64(uint64_t* p, uint64_t v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint64_t tag_slot(uint32_t epoch, uint32_t bits) {
    return ((uint64_t)epoch << 32) | bits;
}

// 16-byte loads and stores of two epoch-tagged words.  Each 8-byte word is
// single-copy atomic and carries its own tag, so a reader that sees both tags
// current has both values whatever the order the halves arrived in.
__device__ __forceinline__ void ld_cg_v2(const uint64_t* p, uint64_t& a, uint64_t& b) {
    asm volatile("ld.global.cg.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

__device__ __forceinline__ void st_v2(uint64_t* p, uint64_t a, uint64_t b) {
    asm volatile("st.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}

// Reads of what earlier work on the stream may have written: log-weights, ancestors.
// kReadOnly, by the read-only path, which the compiler may move past stores and barriers: only
// in kernels launched the ordinary way, which start after that work.
constexpr bool kReadOnly = true;
template <bool RO = false, typename T>
__device__ __forceinline__ T ld_input(const T* p) {
    if constexpr (RO) return __ldg(p);
    return *p;
}

// The same as relaxed accesses at GPU scope (records another CTA polls).
__device__ __forceinline__ void ld_relaxed_v2(const uint64_t* p, uint64_t& a, uint64_t& b) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

__device__ __forceinline__ void st_relaxed_v2(uint64_t* p, uint64_t a, uint64_t b) {
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}

__device__ __forceinline__ void red_release_add_u32(uint32_t* p, uint32_t v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void st_v4_u32(uint32_t* p, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

__device__ __forceinline__ uint4 ld_cg_v4_u32(const uint32_t* p) {
    uint4 v;
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

// Float-pair (double-float) arithmetic for the few per-tile scalars that need
// more than float precision; FP64 issue on this part is far slower.
__device__ __forceinline__ fpair fast_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ fpair pair_mul(fpair a, fpair b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e));
    return fast_two_sum(p, e);
}

__device__ __forceinline__ fpair pair_div(fpair a, fpair b) {
    const float q1 = __fdiv_rn(a.hi, b.hi);
    // remainder a - q1 b, exactly enough for the second quotient digit
    const float p = __fmul_rn(q1, b.hi);
    const float pe = __fmaf_rn(q1, b.hi, -p);
    const float r = __fadd_rn(__fsub_rn(__fsub_rn(a.hi, p), pe), __fsub_rn(a.lo, __fmul_rn(q1, b.lo)));
    return fast_two_sum(q1, __fdiv_rn(r, b.hi));
}

__device__ __forceinline__ fpair pair_sub_f(fpair a, float b) {
    float s, e;
    two_sum(a.hi, -b, s, e);
    return fast_two_sum(s, __fadd_rn(e, a.lo));
}

// ceil and floor of a normalised pair below 2^24 in magnitude, as integers.
__device__ __forceinline__ long long pair_ceil(fpair a) {
    const float c = ceilf(a.hi);
    if (c != a.hi) return (long long)c;
    return (long long)a.hi + (long long)ceilf(a.lo);
}

__device__ __forceinline__ long long pair_floor(fpair a) {
    const float f = floorf(a.hi);
    if (f != a.hi) return (long long)f;
    return (long long)a.hi + (long long)floorf(a.lo);
}

// Spin (bounded) until *p carries epoch in its high word; returns false on timeout.
__device__ __forceinline__ bool wait_slot(const uint64_t* p, uint32_t epoch, uint64_t t_start,
                                          uint64_t limit_ns, uint32_t& bits) {
    for (uint32_t it = 0;; ++it) {
        const uint64_t v = ld_acquire_u64(p);
        if ((uint32_t)(v >> 32) == epoch) {
            bits = (uint32_t)v;
            return true;
        }
        if ((it & 63u) == 63u) {
            if (global_ns() - t_start > limit_ns) return false;
            __nanosleep(64);
        }
    }
}

// ---------------------------------------------------------------------------
// Asynchronous 16-byte copies global -> shared memory, past L1.  A thread's copies
// since its last commit form a group; the waits end by themselves.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void async_copy16(void* dst_smem, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst_smem)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// Waits until at most `left` of this thread's latest groups are incomplete.
template <int left>
__device__ __forceinline__ void async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(left) : "memory");
}

// ---------------------------------------------------------------------------
// Warp and block collectives.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Maximum that propagates NaN (max.NaN): a NaN operand gives NaN.
__device__ __forceinline__ float fmax_nan(float a, float b) {
    float d;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}

// Warp maximum of a float in one integer reduction: the bits of a float map to
// an int of the same order (negative values have their magnitude bits
// flipped), so redux.sync's signed maximum is the float maximum.  -inf stays
// the smallest value; a NaN maps above +inf.
__device__ __forceinline__ float warp_max_redux(float v) {
    int b = __float_as_int(v);
    b ^= (b >> 31) & 0x7fffffff;
    b = __reduce_max_sync(0xffffffffu, b);
    b ^= (b >> 31) & 0x7fffffff;
    return __int_as_float(b);
}

__device__ __forceinline__ int warp_max_i(int v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Inclusive warp scan of float pairs.
__device__ __forceinline__ fpair warp_scan_pair(fpair v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float h = __shfl_up_sync(0xffffffffu, v.hi, o);
        const float l = __shfl_up_sync(0xffffffffu, v.lo, o);
        if (lane >= o) v = pair_add({h, l}, v);
    }
    return v;
}

__device__ __forceinline__ float warp_scan_max(float v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float h = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v = fmaxf(v, h);
    }
    return v;
}

// Inclusive warp scan of doubles (carries only).
__device__ __forceinline__ double warp_scan_d(double v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double h = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += h;
    }
    return v;
}

}  // namespace pf

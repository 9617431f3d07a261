// Row moves in vector chunks, shared by the gather and the in-place gather: the
// chunk types (4 to 32 bytes), their loads and stores, and the grid (RowSplit, the split
// of a chunk's index into row and place, is in pf_index.h).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "pf_index.h"

namespace pf {

// 32-byte chunk: one 256-bit access.
struct __align__(32) u32x8 {
    uint32_t w[8];
};

template <typename VT>
__device__ __forceinline__ VT load_chunk(const VT* p) {
    return *p;
}
template <>
__device__ __forceinline__ u32x8 load_chunk<u32x8>(const u32x8* p) {
    u32x8 v;
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]), "=r"(v.w[4]), "=r"(v.w[5]), "=r"(v.w[6]),
                   "=r"(v.w[7])
                 : "l"(p));
    return v;
}

template <typename VT>
__device__ __forceinline__ VT load_chunk_cg(const VT* p) {  // data other threads may be writing
    return __ldcg(p);
}
template <>
__device__ __forceinline__ u32x8 load_chunk_cg<u32x8>(const u32x8* p) {
    u32x8 v;
    asm volatile("ld.global.cg.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]), "=r"(v.w[4]), "=r"(v.w[5]), "=r"(v.w[6]),
                   "=r"(v.w[7])
                 : "l"(p)
                 : "memory");
    return v;
}

template <typename VT>
__device__ __forceinline__ void store_chunk_cs(VT* p, VT v) {  // evicted first: not read again here
    __stcs(p, v);
}
template <>
__device__ __forceinline__ void store_chunk_cs<u32x8>(u32x8* p, u32x8 v) {
    asm volatile("st.global.cs.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v.w[0]), "r"(v.w[1]),
                 "r"(v.w[2]), "r"(v.w[3]), "r"(v.w[4]), "r"(v.w[5]), "r"(v.w[6]), "r"(v.w[7])
                 : "memory");
}

// CTAs for `total` chunks, `per_cta` each: beyond `from` CTAs per SM one resident wave of `wave`
// per SM that strides over the chunks, or, from `full` CTAs per SM on, a CTA per piece, whose
// staggered starts keep more reads in flight (gather of 2^22 rows of 64 bytes, 108 CTAs
// per SM: 88 us as a wave, 78 us in full; 2^20 rows, 27 per SM: 20.7 and 22.6 us).
inline unsigned chunk_grid(int64_t total, int per_cta, int num_sms, int wave, int full, int from) {
    int64_t blocks = (total + per_cta - 1) / per_cta;
    if (blocks > (int64_t)num_sms * from && blocks < (int64_t)num_sms * full) blocks = (int64_t)num_sms * wave;
    if (blocks > 0x7fffffffLL) blocks = 0x7fffffffLL;  // the kernels stride over what is left
    return (unsigned)(blocks < 1 ? 1 : blocks);
}

}  // namespace pf

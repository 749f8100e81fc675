// Cells in fixed point, shared by the link traversals (trace_mixed.cu, trace_fp64links.cu): the canvas is 2^31
// units wide, mirrored on the axes the ray runs down; a cell of level L is [X, X + 2^(31 - L)) per axis.
#pragma once

#include <cuda_fp16.h>

#include "canvox_internal.cuh"

namespace canvox {
namespace {

constexpr int kFix = 31;
constexpr uint32_t kLinkRecord = 1u << 31;  // a neighbour link that names an internal cell by its own record

// IEEE binary16 bits -> float (exact: every half is a float).
__device__ __forceinline__ float half_bits_to_float(unsigned h) { return __half2float(__ushort_as_half((unsigned short)h)); }
__device__ __forceinline__ float hsig(uint2 v) { return half_bits_to_float(v.y >> 16); }
__device__ __forceinline__ float hlo(unsigned w) { return half_bits_to_float(w & 0xFFFFu); }
__device__ __forceinline__ float hhi(unsigned w) { return half_bits_to_float(w >> 16); }
// x[a] for a runtime axis without indexing an array (which would put it in local memory).
template <typename V>
__device__ __forceinline__ V pick(int a, V x0, V x1, V x2) { return a == 0 ? x0 : (a == 1 ? x1 : x2); }

// How the pools of a canvas are addressed: by 32-bit byte offsets where they all end below 4 GiB (the address is then
// one instruction instead of three or four, five times a leaf step: 2 to 4 % on the depth-24 and -27 views, 33.8 ->
// 32.5 ms on the stereo pair of 2160^2), else by 64-bit ones; with more than 2^31 leaves the slots hold leaf numbers
// modulo 2^31 (leaf_index).
enum { kSmallPool = 0, kPlainPool = 1, kWrapPool = 2 };
inline int pool_kind(const Tree& t) {
    const int64_t span = (int64_t)1 << 32;
    if (t.n_wrap > 0) return kWrapPool;
    return t.n_rec <= span / 48 && t.n_leaf <= span / 8 ? kSmallPool : kPlainPool;  // (32 B a record, 48 B its links)
}
template <typename V>
__device__ __forceinline__ const V* byte_offset(const V* p, uint32_t bytes) {
    return reinterpret_cast<const V*>(reinterpret_cast<const char*>(p) + (size_t)bytes);
}

// Value of the leaf in slot k of record rec (slot value v < 0).
template <int kPool>
__device__ __forceinline__ uint2 load_leaf(const Tree& T, int32_t rec, int k, int32_t v) {
    if (kPool == kSmallPool) return __ldg(byte_offset(T.leaves, (uint32_t)~v * 8u));
    return __ldg(T.leaves + (kPool == kWrapPool ? leaf_index(T, rec, k, v) : (int64_t)(uint32_t)~v));
}

// Child index (not mirrored) at the bits `sh` <= 29 of the position q. (The shifts left lose bit 30 of q[2] only,
// the child of the root.)
__device__ __forceinline__ int child_index(const uint32_t q[3], int sh, uint32_t flip) {
    uint32_t k = ((q[0] >> sh) & 1u) ^ flip;
    k ^= ((q[1] << 1) >> sh) & 2u;
    k ^= ((q[2] << 2) >> sh) & 4u;
    return (int)k;
}
// The same for any bit (the root's children too).
__device__ __forceinline__ int child_index_any(const uint32_t q[3], int sh, uint32_t flip) {
    return (int)((((q[0] >> sh) & 1u) | (((q[1] >> sh) & 1u) << 1) | (((q[2] >> sh) & 1u) << 2)) ^ flip);
}

}  // namespace
}  // namespace canvox

// Cells in fixed point, shared by the link traversals (trace_mixed.cu, trace_fp64links.cu): the canvas is 2^31
// units wide, mirrored on the axes the ray runs down; a cell of level L is [X, X + 2^(31 - L)) per axis.
#pragma once

#include <cuda_fp16.h>

#include "canvox_internal.cuh"

namespace canvox {
namespace {

constexpr int kFix = 31;

// IEEE binary16 bits -> float (exact: every half is a float).
__device__ __forceinline__ float half_bits_to_float(unsigned h) { return __half2float(__ushort_as_half((unsigned short)h)); }
__device__ __forceinline__ float hsig(uint2 v) { return half_bits_to_float(v.y >> 16); }
__device__ __forceinline__ float hlo(unsigned w) { return half_bits_to_float(w & 0xFFFFu); }
__device__ __forceinline__ float hhi(unsigned w) { return half_bits_to_float(w >> 16); }
// x[a] for a runtime axis without indexing an array (which would put it in local memory).
template <typename V>
__device__ __forceinline__ V pick(int a, V x0, V x1, V x2) { return a == 0 ? x0 : (a == 1 ? x1 : x2); }

// Value of the leaf in slot k of record rec (slot value v < 0). kWrap: the canvas has more than 2^31 leaves (slots
// hold leaf numbers modulo 2^31); an instance without it reads the number straight from the slot.
template <bool kWrap>
__device__ __forceinline__ uint2 load_leaf(const Tree& T, int32_t rec, int k, int32_t v) {
    return __ldg(T.leaves + (kWrap ? leaf_index(T, rec, k, v) : (int64_t)(uint32_t)~v));
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

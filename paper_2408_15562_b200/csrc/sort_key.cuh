// Sort keys of (value, index) pairs, used by the tree builder (joint probabilities of candidates) and by the draft step
// (per-row and per-sequence top-k).  A key is a composite: an order-preserving image of a float in the high word, the
// complemented index in the low word, so equal values keep the lower index; 0 is no pair's key and ranks behind
// everything else.
#pragma once
#include <stdint.h>

// order-preserving map float -> uint32 (larger float, larger integer)
__device__ __forceinline__ uint32_t fspad_orderable(float f)
{
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float fspad_from_orderable(uint32_t o)
{
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}
__device__ __forceinline__ unsigned long long fspad_sort_key(float value, uint32_t index)
{
    // value + 0.0f turns -0.0 into +0.0, so the two zeros compare equal as they do for the float itself
    return ((unsigned long long)fspad_orderable(value + 0.0f) << 32) | (unsigned long long)(0xffffffffu - index);
}
__device__ __forceinline__ uint32_t fspad_key_index(unsigned long long key)
{
    return 0xffffffffu - (uint32_t)(key & 0xffffffffull);
}
__device__ __forceinline__ float fspad_key_value(unsigned long long key)
{
    return fspad_from_orderable((uint32_t)(key >> 32));
}


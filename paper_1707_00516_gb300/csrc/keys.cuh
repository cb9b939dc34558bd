// Sorting and merging of top-k keys, one a lane.
#pragma once

#include "common.cuh"

namespace fastid {

namespace {

__device__ __forceinline__ uint64_t shfl64(uint64_t v, int src) {
    uint32_t lo = __shfl_sync(0xffffffffu, (uint32_t)v, src);
    uint32_t hi = __shfl_sync(0xffffffffu, (uint32_t)(v >> 32), src);
    return ((uint64_t)hi << 32) | lo;
}
__device__ __forceinline__ uint64_t shfl_xor64(uint64_t v, int m) {
    uint32_t lo = __shfl_xor_sync(0xffffffffu, (uint32_t)v, m);
    uint32_t hi = __shfl_xor_sync(0xffffffffu, (uint32_t)(v >> 32), m);
    return ((uint64_t)hi << 32) | lo;
}

// Ascending bitonic sort of one key per lane across the warp.
__device__ __forceinline__ uint64_t warp_sort32(uint64_t v, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int j = size >> 1; j > 0; j >>= 1) {
            uint64_t p = shfl_xor64(v, j);
            bool up = (lane & size) == 0 || size == 32;
            bool lower = (lane & j) == 0;
            v = (lower == up) ? (v < p ? v : p) : (v < p ? p : v);
        }
    }
    return v;
}

// Given a sorted ascending (one key per lane) and b sorted ascending, return
// the 32 smallest of a U b, sorted ascending.
__device__ __forceinline__ uint64_t warp_merge32(uint64_t a, uint64_t b, int lane) {
    uint64_t br = shfl64(b, 31 - lane);
    uint64_t v = a < br ? a : br;  // bitonic: the 32 smallest
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        uint64_t p = shfl_xor64(v, j);
        bool lower = (lane & j) == 0;
        v = lower ? (v < p ? v : p) : (v < p ? p : v);
    }
    return v;
}

}  // namespace

}  // namespace fastid

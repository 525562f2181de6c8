// Which nodes' eccentricities the diameter of a symmetric graph still needs.  After an exact SSSP from s every node v has
// max(d(s, v), ecc(s) - d(s, v)) <= ecc(v) <= d(s, v) + ecc(s) (Takes and Kosters, "Determining the diameter of small
// world networks", CIKM 2011), so a node whose upper bound does not exceed the largest eccentricity seen cannot hold
// the diameter.
#pragma once

#include "common.cuh"

namespace cld {

// Sources of the next batch, by one block: every node whose upper bound exceeds the best eccentricity, or, when these
// are more than `most`, half of the batch from the largest upper bounds among them and half from the smallest lower
// bounds of all nodes with unknown eccentricity (thresholds by bisection over the value).  Returns their number, at
// every thread; s_n is a shared word.
__device__ __forceinline__ uint32_t bound_select(uint32_t k, uint32_t most, uint32_t best, const uint32_t* ub,
                                                 const uint32_t* lb, uint32_t* src, uint32_t& s_n) {
    constexpr uint32_t INF = 0xFFFFFFFFu;
    const auto count = [&](auto&& pred) -> uint32_t {  // nodes for which pred holds, at every thread
        __syncthreads();
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        uint32_t c = 0;
        for (uint32_t v = threadIdx.x; v < k; v += blockDim.x) c += pred(v) ? 1u : 0u;
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane_id() == 0 && c) atomicAdd(&s_n, c);
        __syncthreads();
        return s_n;
    };
    const uint32_t open = count([&](uint32_t v) { return ub[v] > best; });
    uint32_t hi_from = best + 1, lo_to = 0;  // take ub >= hi_from; lb < lo_to
    if (open > most) {
        uint32_t a = best + 1, b = INF;  // largest t with at least half of a batch at or above it
        while (a < b) {
            const uint32_t mid = a + (b - a) / 2 + 1;
            if (count([&](uint32_t v) { return ub[v] >= mid; }) >= most / 2) a = mid;
            else b = mid - 1;
        }
        hi_from = a;
        a = 0;
        b = INF;  // smallest t with at least half of a batch below it
        while (a < b) {
            const uint32_t mid = a + (b - a) / 2;
            if (count([&](uint32_t v) { return ub[v] > lb[v] && lb[v] < mid; }) >= most / 2) b = mid;
            else a = mid + 1;
        }
        lo_to = a;
    }
    __syncthreads();
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    for (int part = 0; part < 2; ++part) {
        const uint32_t cap = open <= most || part == 1 ? most : most / 2;
        for (uint32_t v = threadIdx.x; v < k; v += blockDim.x) {
            const bool high = ub[v] > best && ub[v] >= hi_from, low = ub[v] > lb[v] && lb[v] < lo_to;
            if (part == 0 ? high : low && !high) {
                const uint32_t at = atomicAdd(&s_n, 1u);
                if (at < cap) src[at] = v;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) s_n = min(s_n, cap);
        __syncthreads();
    }
    return s_n;
}

}  // namespace cld

// Sorting network on the registers of a group of lanes, shared by the sort tier and the
// format conversions.
#pragma once
#include "common.cuh"

namespace sg {

constexpr int ilog2(int x) { return x <= 1 ? 0 : 1 + ilog2(x / 2); }

// shared-memory index of element i: one gap per 8 elements, so that lanes writing K
// apart do not meet in a bank
__device__ __forceinline__ int st_ph(int i) { return i + (i >> 3); }
template <int N>
constexpr int st_span() { return N + N / 8; }

// Ascending bitonic sort of the N = G K keys of a group (element i = K lane + r).
template <int G, int K>
__device__ __forceinline__ void sort_keys(uint32_t (&key)[K], int lane) {
    constexpr int N = G * K;
#pragma unroll
    for (int k = 2; k <= N; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= K) {
                const int d = j / K;
                const bool asc = k == N || (lane & (k / K)) == 0;
                const bool take_min = asc == ((lane & d) == 0);
#pragma unroll
                for (int r = 0; r < K; ++r) {
                    const uint32_t o = __shfl_xor_sync(0xffffffffu, key[r], d, G);
                    key[r] = take_min ? min(key[r], o) : max(key[r], o);
                }
            } else {
#pragma unroll
                for (int r = 0; r < K; ++r) {
                    if (r & j) continue;
                    const bool asc = k == N || (k < K ? (r & k) == 0 : (lane & (k / K)) == 0);
                    const uint32_t a = key[r], b = key[r | j];
                    key[r] = asc ? min(a, b) : max(a, b);
                    key[r | j] = asc ? max(a, b) : min(a, b);
                }
            }
        }
    }
}

// Inclusive scan over a group of G lanes.
template <int G>
__device__ __forceinline__ int scan_g(int v, int lane) {
#pragma unroll
    for (int o = 1; o < G; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o, G);
        if (lane >= o) v += t;
    }
    return v;
}

}  // namespace sg

// tg_tiles.cuh -- a CTA's tile of edges visited grouped by a small key.
//
// The per-edge kernels give one thread to one (edge, class of slots); with the
// edges of a tile grouped by the key that fixes the slots' classes (the
// endpoints' types, and an edge label), a thread adds a group's values in
// registers and touches the histogram in shared memory once per group (a
// 64-bit shared-memory atomic runs at an eighth of the rate of a 32-bit one).
#pragma once

#include "tg_internal.cuh"

namespace tg {

template <int kKeys>
struct TileOrder {
    uint16_t order[kTile];      // the tile's edges (relative to its first) grouped by key
    uint8_t key[kTile];         // key by edge (kKeys <= 256)
    int count[kKeys];           // edges of each key
    int next[kKeys];
};

// groups the edges [begin, begin + n) by key_of(e) in [0, kKeys); begins and
// ends with a barrier
template <int kKeys, class F>
__device__ __forceinline__ void tile_order(int64_t begin, int n, TileOrder<kKeys> &o, F key_of) {
    __syncthreads();
    for (int k = threadIdx.x; k < kKeys; k += blockDim.x) o.count[k] = 0;
    __syncthreads();
    for (int x = threadIdx.x; x < n; x += blockDim.x) {
        const int k = key_of(begin + x);
        o.key[x] = (uint8_t)k;
        atomicAdd(&o.count[k], 1);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        int run = 0;
        for (int b = 0; b < kKeys; b += 32) {
            const int k = b + threadIdx.x;
            const int c = k < kKeys ? o.count[k] : 0;
            int inc = c;
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, d);
                if ((int)threadIdx.x >= d) inc += y;
            }
            if (k < kKeys) o.next[k] = run + inc - c;
            run += __shfl_sync(0xffffffffu, inc, 31);
        }
    }
    __syncthreads();
    for (int x = threadIdx.x; x < n; x += blockDim.x) o.order[atomicAdd(&o.next[o.key[x]], 1)] = (uint16_t)x;
    __syncthreads();
}

// the share of slice s of E of a tile's n grouped edges
__device__ __forceinline__ void slice_of(int n, int s, int E, int &b, int &e) {
    b = (int)((int64_t)n * s / E);
    e = (int)((int64_t)n * (s + 1) / E);
}

}  // namespace tg

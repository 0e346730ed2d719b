// tg_wedge_table.hpp -- sizes of the wedge anchors' counter tables and the
// anchors' classes (tg_wedge.cu).  Host and device code, and plain C++.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace tg {

// Wedge anchors by class: 0 a warp, 1-4 a CTA by table size, kHubClass hubs.
constexpr int kHubClass = 5;
constexpr int kFormBytes[kHubClass] = {0, 11 << 10, 30 << 10, 98 << 10, 200 << 10};   // table bytes (class 0: light_bytes)
struct WedgeLimits {
    int64_t light, hub;         // most wedges of class 0, and of the shared-memory classes
    int64_t bytes[4];           // table bytes of classes 1 to 4
};

// Layout of an anchor's counters: rw words per wedge end, F types per word,
// `bits` bits each.
struct Pack {
    int rw, F, bits;
};

// the smallest layout whose counters hold `most`
__host__ __device__ __forceinline__ Pack pack_of(int L, int64_t most) {
    Pack k;
    k.rw = 1;
    k.F = L;
    k.bits = 32 / L;
    if (most >> k.bits) {
        k.rw = 2;
        k.F = (L + 1) / 2;
        k.bits = 32 / k.F;
    }
    if (most >> k.bits) {
        k.rw = 4;
        k.F = 2;
        k.bits = 16;
    }
    return k;
}

// The layout of an anchor of W wedges with at most `most` lower neighbours of
// one type: a counter reaches neither number.  `most` alone would not do: a
// lower neighbour without a lower neighbour of its own has no wedge, so a
// star-like anchor has few wedges and any number of neighbours, and rows for
// all of them leave a light table (light_bytes) fewer slots than wedges.
__host__ __device__ __forceinline__ Pack anchor_pack(int L, int64_t W, int64_t most) {
    return pack_of(L, most < W ? most : W);
}

// Table of an anchor of W wedges: per slot a key and rw counter words, per
// wedge the slot it went to (uint16).  Two slots per wedge where `bytes` holds
// them, at least one (a slot per distinct end, so an insert finds one).
__host__ __device__ __forceinline__ int64_t table_need(int64_t W, int64_t slots, int rw) {
    return slots * (4 + 4 * rw) + ((2 * W + 3) & ~(int64_t)3);
}
__host__ __device__ __forceinline__ int64_t slots_for(int64_t W, int64_t bytes, int rw) {
    const int64_t fit = (bytes - table_need(W, 0, rw)) / (4 + 4 * rw), want = 2 * W + 16;
    return want < fit ? want : fit;
}

// bytes of a light anchor's table: its wedges may all end at distinct nodes,
// and its counters reach the number of its wedges
__host__ __device__ __forceinline__ int64_t light_bytes(int L, int64_t wedges) {
    return (table_need(wedges, 2 * wedges + 16, pack_of(L, wedges).rw) + 15) & ~(int64_t)15;
}

// class of an anchor of W wedges, or -1
__host__ __device__ __forceinline__ int wedge_class(const WedgeLimits &w, int L, int64_t W, int64_t most) {
    if (W <= 0) return -1;
    if (W <= w.light) return 0;
    if (W > w.hub) return kHubClass;
    const int rw = anchor_pack(L, W, most).rw;
    // two slots per wedge; in the largest form a slot per wedge is enough
    for (int f = 0; f < 4; ++f)
        if (table_need(W, (f < 3 ? 2 * W : W) + 16, rw) <= w.bytes[f] && W < (1 << 15)) return f + 1;
    return kHubClass;
}

}  // namespace tg

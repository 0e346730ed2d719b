// tg_local.cuh -- the triangles of a graph, each found once.
//
// Every triangle is found from its node u of lowest priority: its other two
// nodes a < b are both in N+(u), u's neighbours of higher priority, and b is
// in N+(a).  N+ lists are short on skewed graphs (the order is by degree:
// at most sqrt(2 m) entries, 342 on a 20 M-edge Chung-Lu graph whose hubs
// have degree 35,000), so the local graph of N+(u) fits shared memory.
// Intersecting the typed rows of every edge finds each triangle three times,
// and by binary searches in rows of hub length.
//
// Three forms by p = |N+(u)|:
//   p <= 32           warp per u; every pair of N+(u) is looked up in the
//                     lower node's N+ list by a binary search, one pair per
//                     lane (on the graph above 6.7e7 searches against
//                     1.8e9 entries that scanning the lists would read);
//   p <= the capacity CTA per u; every list N+(a), a in N+(u), is scanned by
//                     a warp (coalesced, four loads in flight) and tested
//                     against a bitmap of hashed ids of N+(u) in shared
//                     memory; the 5% that pass are collected in a queue per
//                     warp and looked up exactly, 32 at a time (a lookup at
//                     once would leave most lanes idle: few of 32 entries
//                     hit, but almost every 32 hold one that does);
//   larger            the same with the CTA's arrays in a global slice.
#pragma once

#include "tg_internal.cuh"

namespace tg {

constexpr int kTriWarpMax = 32;              // p of the warp form
constexpr int kTriMidMax = 128;              // p of the CTA form with kTriMidThreads threads
constexpr int kTriBigMax = 704;              // p of the CTA form with kTriBigThreads threads and shared memory
constexpr int kTriMidThreads = 128;
constexpr int kTriBigThreads = 256;
constexpr int kQueue = 64;                   // queue entries per warp

__device__ __forceinline__ uint32_t lg_hash(uint32_t id) { return id * 2654435761u; }

// pair x (0 <= x < p (p - 1) / 2) of a list -> positions k < l
__device__ __forceinline__ void pair_of(int x, int &k, int &l) {
    l = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)x)) * 0.5f);
    if (l * (l - 1) / 2 > x) --l;
    if (l * (l + 1) / 2 <= x) ++l;
    k = x - l * (l - 1) / 2;
}

// position in plus_adj of entry `key` (type << 29 | id) of N+(a), or -1
__device__ __forceinline__ int64_t plus_find(const GraphView &g, int32_t a, uint32_t key) {
    const int64_t lo = g.plus_off[a];
    uint32_t n = (uint32_t)(g.plus_off[a + 1] - lo);
    if (n == 0) return -1;
    const uint32_t *base = reinterpret_cast<const uint32_t *>(g.plus_adj) + lo;
    const uint32_t *b = base;
    while (n > 1) {
        const uint32_t half = n >> 1;
        b = __ldg(b + half) <= key ? b + half : b;
        n -= half;
    }
    return __ldg(b) == key ? lo + (b - base) : -1;
}

// The local list of one u held by a CTA: entries, edge ids, a bitmap of
// hashed ids and an exact hash (id -> list position).
struct LocalList {
    uint32_t *ent;              // [cap] type << 29 | id
    uint32_t *eid;              // [cap] edge id of {u, entry}
    uint32_t *keys;             // [1 << lgh] id or 0xffffffff
    uint16_t *vals;             // [1 << lgh] list position
    uint32_t *filter;           // [1 << (lgf - 5)] bitmap of hashed ids
    uint32_t *qpos;             // [kQueue] this warp's queue: position in plus_adj
    uint16_t *qrow;             // [kQueue] and the list position of the row's node
    int lgh, lgf;
};

__host__ __device__ inline int lg_at_least(int64_t v) {
    int l = 0;
    while (((int64_t)1 << l) < v) ++l;
    return l;
}

// bytes of the arrays of LocalList for lists of up to cap entries
__host__ __device__ inline size_t local_bytes(int cap, int lgf, int warps) {
    const size_t h = (size_t)1 << lg_at_least(2 * (int64_t)cap);
    return (size_t)cap * 8 + h * 6 + ((size_t)1 << lgf) / 8 + (size_t)warps * kQueue * 6;
}

__device__ __forceinline__ unsigned char *local_carve(LocalList &q, unsigned char *mem, int cap, int lgf, int warps,
                                                      int wid) {
    q.lgh = lg_at_least(2 * (int64_t)cap);
    q.lgf = lgf;
    q.ent = reinterpret_cast<uint32_t *>(mem);
    q.eid = q.ent + cap;
    q.keys = q.eid + cap;
    q.filter = q.keys + (1 << q.lgh);
    uint32_t *qp = q.filter + (1 << (lgf - 5));
    q.qpos = qp + wid * kQueue;
    q.vals = reinterpret_cast<uint16_t *>(qp + warps * kQueue);
    q.qrow = q.vals + (1 << q.lgh) + wid * kQueue;
    return reinterpret_cast<unsigned char *>(q.vals + (1 << q.lgh) + warps * kQueue);
}

// loads N+(u) (p entries) and builds the set; by the whole CTA
__device__ __forceinline__ void local_load(const GraphView &g, int64_t pb, int p, const LocalList &q) {
    for (int k = threadIdx.x; k < (1 << q.lgh); k += blockDim.x) q.keys[k] = 0xffffffffu;
    for (int k = threadIdx.x; k < (1 << (q.lgf - 5)); k += blockDim.x) q.filter[k] = 0u;
    __syncthreads();
    for (int k = threadIdx.x; k < p; k += blockDim.x) {
        const uint32_t e = (uint32_t)g.plus_adj[pb + k];
        q.ent[k] = e;
        q.eid[k] = (uint32_t)g.plus_eid[pb + k];
        const uint32_t id = e & (uint32_t)kIdMask, h = lg_hash(id);
        atomicOr(&q.filter[h >> (32 - q.lgf) >> 5], 1u << ((h >> (32 - q.lgf)) & 31u));
        uint32_t s = h >> (32 - q.lgh);
        while (atomicCAS(&q.keys[s], 0xffffffffu, id) != 0xffffffffu) s = (s + 1) & ((1u << q.lgh) - 1u);   // ids are distinct, load <= 1/2
        q.vals[s] = (uint16_t)k;
    }
    __syncthreads();
}

// list position of id, or -1
__device__ __forceinline__ int local_find(const LocalList &q, uint32_t id) {
    uint32_t s = lg_hash(id) >> (32 - q.lgh);
    for (;;) {                                              // ends at an empty slot: load <= 1/2
        const uint32_t k = q.keys[s];
        if (k == id) return q.vals[s];
        if (k == 0xffffffffu) return -1;
        s = (s + 1) & ((1u << q.lgh) - 1u);
    }
}

// Every pair a < b of N+(u) with b in N+(a), by the CTA's warps (rows a
// strided over the warps): fn(hit, ka, kb, pos) is called by whole warps for
// 32 candidates at a time (hit: lane holds a triangle; ka, kb: list
// positions of a and b; pos: b's position in plus_adj, i.e. of edge {a, b}).
template <class F>
__device__ __forceinline__ void local_pairs(const GraphView &g, int p, const LocalList &q, int lane, int wid,
                                            int nwarp, F fn) {
    int qn = 0;                                             // warp-uniform
    const int fs = 32 - q.lgf;
    auto work = [&](int first, int cnt) {
        __syncwarp();
        bool hit = false;
        int ka = 0, kb = -1;
        uint32_t pos = 0;
        if (lane < cnt) {
            pos = q.qpos[first + lane];
            ka = q.qrow[first + lane];
            kb = local_find(q, (uint32_t)__ldg(g.plus_adj + pos) & (uint32_t)kIdMask);
            hit = kb >= 0;
        }
        fn(hit, ka, kb, pos);
        __syncwarp();
    };
    for (int ka = wid; ka < p; ka += nwarp) {
        const uint32_t a = q.ent[ka] & (uint32_t)kIdMask;
        const int64_t pb = g.plus_off[a], pe = g.plus_off[a + 1];
        for (int64_t r0 = pb; r0 < pe; r0 += 128) {
            uint32_t ent[4];
            bool c[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int64_t at = r0 + 32 * v + lane;
                ent[v] = at < pe ? (uint32_t)__ldg(g.plus_adj + at) : 0xffffffffu;
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const uint32_t h = lg_hash(ent[v] & (uint32_t)kIdMask) >> fs;
                c[v] = r0 + 32 * v + lane < pe && ((q.filter[h >> 5] >> (h & 31u)) & 1u);
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const unsigned bal = __ballot_sync(0xffffffffu, c[v]);
                if (bal == 0) continue;
                if (c[v]) {
                    const int x = qn + __popc(bal & ((1u << lane) - 1u));
                    q.qpos[x] = (uint32_t)(r0 + 32 * v + lane);
                    q.qrow[x] = (uint16_t)ka;
                }
                qn += __popc(bal);
                if (qn >= 32) {                             // the queue never holds more than 31 + 32
                    work(qn - 32, 32);
                    qn -= 32;
                }
            }
        }
    }
    if (qn > 0) work(0, qn);
}

}  // namespace tg

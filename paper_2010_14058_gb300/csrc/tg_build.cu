// tg_build.cu -- device preprocessing of a typed graph (tg_build).
//
// From a caller CSR it builds, on the GPU:
//   * validation: row pointers, ranges, types < L, no self-loops, no repeated
//     entries, symmetric rows, no edge between two graphs of a batch;
//   * a node order by (graph, degree, id): the internal id of a node is its
//     rank, so comparisons of internal ids compare priorities;
//   * adjacency rows sorted by (type, internal id) with per-type offsets:
//     the typed neighbourhoods Gamma_x^t and typed degrees d_x^t of Def. 6-7;
//   * per node its higher-priority neighbours as one list, one entry per edge;
//   * edge ids in the caller's lexicographic (u < v) order, the two slots of
//     each edge and the edge id of every slot and list entry;
// and, before the first 4-node count (prepare_anchors):
//   * per-node typed degree sums delta_x[t][t'] = sum_{w in Gamma_x^t} d_w^t';
//   * work lists: wedge anchors by class.
// Sorting and scans use CUB device primitives.
// On a 20 M-edge Chung-Lu graph all of it takes 11.4 ms (28.2 before the edges
// came from the N+ lists instead of one global counter, the wedge counts from
// N+, the row sums from 32-byte sectors and the sort keys were packed): sorts
// 3.6, k_rows 1.5, k_edges 1.5, k_plus_fill 1.25, k_anchor_work 0.98, row sums
// 0.9 ms; bound by scattered reads of ids and slots.
#include <algorithm>
#include <cstdint>
#include <mutex>
#include <vector>

#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>

#include "tg_host.hpp"
#include "tg_local.cuh"

namespace tg {

namespace {

constexpr int kThreads = 256;

inline int blocks_for(int64_t items, int per_block) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > (1ll << 30)) b = 1ll << 30;
    return (int)b;
}

__global__ void k_check_rows(int64_t n, int64_t nnz, const int64_t *__restrict__ rp,
                             const uint8_t *__restrict__ types, int L, uint32_t *status) {
    int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (v > n) return;
    int64_t a = rp[v];
    bool bad = a < 0 || a > nnz;
    if (v == 0 && a != 0) bad = true;
    if (v == n && a != nnz) bad = true;
    if (v < n) {
        if (rp[v + 1] < a) bad = true;
        if (types[v] >= L) bad = true;
    }
    if (bad) set_status(status, ST_INVALID_GRAPH);
}

__global__ void k_check_cols(int64_t nnz, int64_t n, const int32_t *__restrict__ col, uint32_t *status) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= nnz) return;
    int32_t v = col[s];
    if (v < 0 || v >= n) set_status(status, ST_INVALID_GRAPH);
}

__global__ void k_degree_keys(int64_t n, const int64_t *__restrict__ rp, const int64_t *__restrict__ node_off,
                              int ngraphs, int deg_bits, unsigned long long *keys, int32_t *vals) {
    int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (v >= n) return;
    int lo = 0, hi = ngraphs;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (node_off[mid] <= v) lo = mid; else hi = mid;
    }
    unsigned long long d = (unsigned long long)(rp[v + 1] - rp[v]);
    keys[v] = ((unsigned long long)lo << deg_bits) | d;
    vals[v] = (int32_t)v;
}

__global__ void k_inverse(int64_t n, const int32_t *__restrict__ old_of, const int64_t *__restrict__ rp,
                          int32_t *new_of, int64_t *ndeg) {
    int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (x > n) return;
    if (x == n) { ndeg[n] = 0; return; }
    int32_t u = old_of[x];
    new_of[u] = (int32_t)x;
    ndeg[x] = rp[u + 1] - rp[u];
}

// Packed sort keys hold only the bits that n and the types need (a radix pass
// per 8 bits): row << (nb + 3) | type << nb | neighbour, nb = bits of a node id.
constexpr int kTypeBits = 3;

// warp per caller node u: the keys of its entries
__global__ void k_fill_keys(int64_t n, const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
                            const uint8_t *__restrict__ types, const int32_t *__restrict__ new_of,
                            const int64_t *__restrict__ rp_new, const int64_t *__restrict__ node_off, int ngraphs, int nb,
                            unsigned long long *keys, uint32_t *status) {
    int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kWarp;
    int lane = threadIdx.x & (kWarp - 1);
    if (warp >= n) return;
    int64_t u = warp;
    int32_t x = new_of[u];
    int64_t b = rp[u], e = rp[u + 1], base = rp_new[x];
    int64_t glo = 0, ghi = 0;
    if (ngraphs > 1) {
        int lo = 0, hi = ngraphs;
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (node_off[mid] <= u) lo = mid; else hi = mid;
        }
        glo = node_off[lo];
        ghi = node_off[lo + 1];
    }
    for (int64_t k = b + lane; k < e; k += kWarp) {
        int32_t v = col[k];
        if (ngraphs > 1 && (v < glo || v >= ghi)) set_status(status, ST_INVALID_GRAPH);
        keys[base + (k - b)] = ((unsigned long long)(uint32_t)x << (nb + kTypeBits)) |
                               ((unsigned long long)types[v] << nb) | (uint32_t)new_of[v];
    }
}

__global__ void k_gather_types(int64_t n, const int32_t *__restrict__ old_of, const uint8_t *__restrict__ ty,
                               uint8_t *out) {
    int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (x < n) out[x] = ty[old_of[x]];
}

// warp per internal row x: adjacency ids, self-loop / repeat checks, type
// offsets, typed degrees (one 32-byte sector per node), and the numbers of
// lower- and higher-priority neighbours
__global__ void k_rows(int64_t n, int L, int nb, const int64_t *__restrict__ rp,
                       const unsigned long long *__restrict__ keys, int32_t *adj, int32_t *toff, uint32_t *tdeg,
                       int32_t *pivot, int64_t *nplus, int32_t *most_lower, int64_t *long_type, uint32_t *status) {
    int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kWarp;
    int lane = threadIdx.x & (kWarp - 1);
    if (warp > n) return;
    if (warp == n) {
        if (lane == 0) nplus[n] = 0;
        return;
    }
    int64_t x = warp;
    int64_t b = rp[x], e = rp[x + 1];
    const unsigned long long id_mask = (1ull << nb) - 1ull;
    for (int64_t s = b + lane; s < e; s += kWarp) {
        unsigned long long k = keys[s];
        int32_t y = (int32_t)(k & id_mask);
        adj[s] = y;
        if ((int64_t)(k >> (nb + kTypeBits)) != x || y == x) set_status(status, ST_INVALID_GRAPH);
        if (s > b && keys[s - 1] == k) set_status(status, ST_INVALID_GRAPH);
    }
    // type t < L starts at the first slot whose packed type is >= t; the
    // end sentinel (t = L) is the row length
    if (lane < L) {
        const unsigned long long key = (unsigned long long)x << (nb + kTypeBits) | (unsigned long long)lane << nb;
        int64_t lo = b, hi = e;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            if (keys[mid] < key) lo = mid + 1; else hi = mid;
        }
        toff[x * (L + 1) + lane] = (int32_t)(lo - b);
    } else if (lane == L) {
        toff[x * (L + 1) + L] = (int32_t)(e - b);
    }
    // pivot: first slot of each type segment whose id exceeds x (the
    // neighbours of higher priority)
    __syncwarp();
    const int32_t sb = lane < L ? toff[x * (L + 1) + lane] : 0;
    const int32_t se = lane < L ? toff[x * (L + 1) + lane + 1] : 0;
    int32_t up = 0, down = 0;            // higher- and lower-priority neighbours of this type segment
    if (lane < L) {
        int64_t lo = b + sb, hi = b + se;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            if ((int32_t)(keys[mid] & id_mask) < (int32_t)x + 1) lo = mid + 1; else hi = mid;
        }
        pivot[x * L + lane] = (int32_t)(lo - b);
        up = se - (int32_t)(lo - b);
        down = (int32_t)(lo - b) - sb;
    }
    if (lane < kCRow) tdeg[x * kCRow + lane] = (uint32_t)(se - sb);
    if (se - sb >= kNarrowDegree) *long_type = 1;
    up = (int32_t)__reduce_add_sync(0xffffffffu, (unsigned)up);
    down = (int32_t)__reduce_max_sync(0xffffffffu, (unsigned)down);
    if (lane == 0) {
        nplus[x] = up;
        most_lower[x] = down;
    }
}

// Warp per node x: its higher-priority neighbours (the part of each type
// segment past the pivot), packed (type << 29 | id), into one contiguous
// list, and for every entry the key of its edge in the caller's order and its
// slot; nodes with more than kTriWarpMax of them are listed by class.
__global__ void k_plus_fill(GraphView g, const int32_t *__restrict__ old_of, int nb, int32_t *plus_adj,
                            uint32_t *plus_slot, unsigned long long *ekeys, uint32_t *epos, int32_t *mid, int32_t *big,
                            int32_t *huge, unsigned long long *counts) {
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kWarp;
    const int lane = threadIdx.x & (kWarp - 1);
    if (warp >= g.n) return;
    const int64_t x = warp, r = g.rp[x];
    int64_t out = g.plus_off[x];
    if (lane == 0) {
        const int64_t p = g.plus_off[x + 1] - out;
        if (p > kTriWarpMax) {
            const int c = p <= kTriMidMax ? 0 : p <= kTriBigMax ? 1 : 2;
            const unsigned long long at = atomicAdd(&counts[c], 1ull);
            (c == 0 ? mid : c == 1 ? big : huge)[at] = (int32_t)x;
            atomicMax(&counts[3], (unsigned long long)p);
        }
    }
    const unsigned long long ox = (unsigned long long)old_of[x];
    for (int q = 0; q < g.L; ++q) {
        const int64_t b = r + g.pivot[x * g.L + q], e = r + g.toff[x * (g.L + 1) + q + 1];
        for (int64_t k = b + lane; k < e; k += kWarp) {
            const int32_t y = g.adj[k];
            const unsigned long long oy = (unsigned long long)old_of[y];
            const int64_t at = out + (k - b);
            plus_adj[at] = (int32_t)(((uint32_t)q << kTypeShift) | (uint32_t)y);
            plus_slot[at] = (uint32_t)k;
            ekeys[at] = ox < oy ? ox << nb | oy : oy << nb | ox;
            epos[at] = (uint32_t)at;
        }
        out += e - b;
    }
}

// thread per edge id: endpoints, both slots, slot -> edge id, list entry -> edge id
__global__ void k_edges(int64_t m, int nb, const unsigned long long *__restrict__ ekeys,
                        const uint32_t *__restrict__ epos, const uint32_t *__restrict__ plus_slot, GraphView g,
                        const int32_t *__restrict__ new_of, int32_t *e_lo, int32_t *e_hi, int64_t *e_slot_lo,
                        int64_t *e_slot_hi, int32_t *slot_eid, int32_t *plus_eid, uint32_t *status) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= m) return;
    const unsigned long long k = ekeys[e];
    const int32_t a = new_of[(int32_t)(k >> nb)], c = new_of[(int32_t)(k & ((1ull << nb) - 1ull))];
    const int32_t x = min(a, c), y = max(a, c);
    const uint32_t at = epos[e];
    const int64_t s = plus_slot[at];            // slot of y in row x
    const int tx = g.ty[x];
    const int64_t b = seg_begin(g, y, tx), en = seg_end(g, y, tx);
    const int64_t r = lower_bound_i32(g.adj, b, en, x);
    if (r >= en || g.adj[r] != x) {             // one-sided entry
        set_status(status, ST_INVALID_GRAPH);
        return;
    }
    slot_eid[s] = (int32_t)e;
    slot_eid[r] = (int32_t)e;
    plus_eid[at] = (int32_t)e;
    e_lo[e] = x;
    e_hi[e] = y;
    e_slot_lo[e] = s;
    e_slot_hi[e] = r;
}

// Warp per node v: a higher-priority neighbour x of v is the anchor of the
// wedges x - v - w, w any neighbour of v below x: v's lower neighbours and
// those of N+(v) below x.  (Searching v's typed rows for x, anchor by anchor,
// took a binary search per pair and type: 11.0 ms on a 20 M-edge Chung-Lu
// graph against 0.98.)
__global__ void __launch_bounds__(256) k_anchor_work(GraphView g, unsigned long long *work) {
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kWarp;
    const int lane = threadIdx.x & (kWarp - 1);
    if (warp >= g.n) return;
    const int64_t v = warp, b = g.plus_off[v];
    const int p = (int)(g.plus_off[v + 1] - b);
    const int64_t lower = g.rp[v + 1] - g.rp[v] - p;
    for (int i0 = 0; i0 < p; i0 += kWarp) {
        const int32_t x = i0 + lane < p ? (int32_t)((uint32_t)g.plus_adj[b + i0 + lane] & (uint32_t)kIdMask) : -1;
        int below = 0;                          // entries of N+(v) below x
        for (int j0 = 0; j0 < p; j0 += kWarp) {
            const int32_t y =
                j0 + lane < p ? (int32_t)((uint32_t)g.plus_adj[b + j0 + lane] & (uint32_t)kIdMask) : INT32_MAX;
            const int cnt = min(kWarp, p - j0);
            for (int k = 0; k < cnt; ++k) below += __shfl_sync(0xffffffffu, y, k) < x ? 1 : 0;
        }
        if (x >= 0 && lower + below > 0) atomicAdd(&work[x], (unsigned long long)(lower + below));
    }
}

// per graph: its first slot and largest degree (its last internal node's);
// then the entries of all N+ lists and the status word, for one copy
__global__ void k_graph_info(GraphView g, int64_t *slot_off, int64_t *max_degree, int64_t *plus_total,
                             const uint32_t *status) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i > g.ngraphs) return;
    slot_off[i] = g.rp[g.node_off[i]];
    if (i == g.ngraphs) {
        plus_total[0] = g.plus_off[g.n];
        plus_total[1] = *status;
        return;
    }
    const int64_t last = g.node_off[i + 1] - 1;
    max_degree[i] = last >= g.node_off[i] ? g.rp[last + 1] - g.rp[last] : 0;
}

template <class F>
void cub_call(F f, cudaStream_t s) {
    size_t bytes = 0;
    TG_CK(f(nullptr, bytes));
    TBuf tmp(bytes, s);
    TG_CK(f(tmp.p, bytes));
}

int bits_for(int64_t v) {
    int b = 1;
    while (b < 63 && (1ll << b) <= v) ++b;
    return b;
}

// work << 4 | type of the listed nodes
__global__ void k_gather_work(int64_t c, const int32_t *__restrict__ ids, const int64_t *__restrict__ work,
                              const uint8_t *__restrict__ ty, int64_t *out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < c) out[i] = work[ids[i]] << 4 | ty[ids[i]];
}

uint32_t read_status(const DBuf &st, cudaStream_t s) {
    uint32_t v = 0;
    TG_CK(cudaMemcpyAsync(&v, st.p, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    TG_CK(cudaStreamSynchronize(s));
    return v;
}

}  // namespace

cudaMemPool_t device_pool() {
    static std::mutex mu;
    static cudaMemPool_t pools[64] = {};
    int dev = 0;
    TG_CK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) throw Error{TG_ERR_INVALID_ARG, "device index"};
    std::lock_guard<std::mutex> lock(mu);
    if (!pools[dev]) {
        cudaMemPoolProps props;
        std::memset(&props, 0, sizeof(props));
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        TG_CK(cudaMemPoolCreate(&pools[dev], &props));
        uint64_t keep = UINT64_MAX;
        TG_CK(cudaMemPoolSetAttribute(pools[dev], cudaMemPoolAttrReleaseThreshold, &keep));
    }
    return pools[dev];
}

int sm_count() {
    static int cached = 0;
    if (!cached) {
        int dev = 0;
        TG_CK(cudaGetDevice(&dev));
        TG_CK(cudaDeviceGetAttribute(&cached, cudaDevAttrMultiProcessorCount, dev));
    }
    return cached;
}

void build_graph(Graph &G, int32_t ngraphs, const int64_t *node_off_host, int64_t n, int64_t nnz,
                 const int64_t *row_ptr, const int32_t *col, const uint8_t *types, int32_t L,
                 const tg_options &opt, cudaStream_t s) {
    G.on(s);
    G.last_launches = 0;
    G.ngraphs = ngraphs;
    G.L = L;
    G.n = n;
    G.nnz = nnz;
    G.m = nnz / 2;
    G.opt = opt;
    TG_CK(cudaGetDevice(&G.device));
    G.h_node_off.assign(node_off_host, node_off_host + ngraphs + 1);

    G.status.alloc(sizeof(uint32_t));
    TG_CK(cudaMemsetAsync(G.status.p, 0, sizeof(uint32_t), s));
    uint32_t *status = G.status.as<uint32_t>();

    // inputs on the device (copied in when the caller passed host memory)
    TBuf rp_in(sizeof(int64_t) * (n + 1), s), col_in(sizeof(int32_t) * std::max<int64_t>(nnz, 1), s),
        ty_in(std::max<int64_t>(n, 1), s);
    TG_CK(cudaMemcpyAsync(rp_in.p, row_ptr, sizeof(int64_t) * (n + 1),
                          is_device_pointer(row_ptr) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
    if (nnz > 0)
        TG_CK(cudaMemcpyAsync(col_in.p, col, sizeof(int32_t) * nnz,
                              is_device_pointer(col) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
    if (n > 0)
        TG_CK(cudaMemcpyAsync(ty_in.p, types, n,
                              is_device_pointer(types) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
    G.node_off.alloc(sizeof(int64_t) * (ngraphs + 1));
    TG_CK(cudaMemcpyAsync(G.node_off.p, G.h_node_off.data(), sizeof(int64_t) * (ngraphs + 1),
                          cudaMemcpyHostToDevice, s));
    const int64_t *rp = rp_in.as<int64_t>();
    const int32_t *cl = col_in.as<int32_t>();
    const uint8_t *ty = ty_in.as<uint8_t>();

    // 1. ranges, row pointers, types
    ++G.last_launches;
    k_check_rows<<<blocks_for(n + 1, kThreads), kThreads, 0, s>>>(n, nnz, rp, ty, L, status);
    if (nnz > 0) ++G.last_launches;
    if (nnz > 0) k_check_cols<<<blocks_for(nnz, kThreads), kThreads, 0, s>>>(nnz, n, cl, status);
    TG_CK(cudaGetLastError());
    if (read_status(G.status, s) & ST_INVALID_GRAPH) throw Error{TG_ERR_INVALID_GRAPH, "row pointers, ids or types"};

    // 2. priority order: sort nodes by (graph, degree), stable in id
    G.old_of.alloc(sizeof(int32_t) * std::max<int64_t>(n, 1));
    G.rp.alloc(sizeof(int64_t) * (n + 1));
    TBuf new_of(sizeof(int32_t) * std::max<int64_t>(n, 1), s);
    {
        TBuf keys(sizeof(unsigned long long) * std::max<int64_t>(n, 1), s), keys2(sizeof(unsigned long long) * std::max<int64_t>(n, 1), s);
        TBuf vals(sizeof(int32_t) * std::max<int64_t>(n, 1), s);
        if (n > 0) {
            const int deg_bits = bits_for(std::max<int64_t>(nnz, 1));
            ++G.last_launches;
            k_degree_keys<<<blocks_for(n, kThreads), kThreads, 0, s>>>(n, rp, G.node_off.as<int64_t>(), ngraphs, deg_bits,
                                                                       keys.as<unsigned long long>(), vals.as<int32_t>());
            TG_CK(cudaGetLastError());
            const int end_bit = deg_bits + (ngraphs > 1 ? bits_for(ngraphs) : 0);
            cub_call([&](void *t, size_t &b) {
                return cub::DeviceRadixSort::SortPairs(t, b, keys.as<unsigned long long>(), keys2.as<unsigned long long>(),
                                                       vals.as<int32_t>(), G.old_of.as<int32_t>(), n, 0, end_bit, s);
            }, s);
        }
        TBuf ndeg(sizeof(int64_t) * (n + 1), s);
        ++G.last_launches;
        k_inverse<<<blocks_for(n + 1, kThreads), kThreads, 0, s>>>(n, G.old_of.as<int32_t>(), rp, new_of.as<int32_t>(),
                                                                   ndeg.as<int64_t>());
        TG_CK(cudaGetLastError());
        cub_call([&](void *t, size_t &b) {
            return cub::DeviceScan::ExclusiveSum(t, b, ndeg.as<int64_t>(), G.rp.as<int64_t>(), n + 1, s);
        }, s);
    }

    // 3. rows sorted by (type, internal id)
    const int nb = bits_for(std::max<int64_t>(n - 1, 1));
    G.adj.alloc(sizeof(int32_t) * std::max<int64_t>(nnz, 1));
    G.toff.alloc(sizeof(int32_t) * std::max<int64_t>(n * (L + 1), 1));
    G.tdeg.alloc(sizeof(uint32_t) * kCRow * std::max<int64_t>(n, 1));
    G.pivot.alloc(sizeof(int32_t) * std::max<int64_t>(n * L, 1));
    G.plus_off.alloc(sizeof(int64_t) * (n + 1));
    G.ty.alloc(std::max<int64_t>(n, 1));
    std::vector<int64_t> h_info(2 * (size_t)ngraphs + 4);    // see k_graph_info; last: a typed degree of kNarrowDegree or more
    TBuf info(sizeof(int64_t) * h_info.size(), s);
    TG_CK(cudaMemsetAsync(info.as<int64_t>() + 2 * ngraphs + 3, 0, sizeof(int64_t), s));
    TBuf nplus(sizeof(int64_t) * (n + 1), s);
    G.most_lower.alloc(sizeof(int32_t) * std::max<int64_t>(n, 1));
    {
        TBuf keys(sizeof(unsigned long long) * std::max<int64_t>(nnz, 1), s), keys2(sizeof(unsigned long long) * std::max<int64_t>(nnz, 1), s);
        if (n > 0) {
            ++G.last_launches;
            k_fill_keys<<<blocks_for(n * kWarp, kThreads), kThreads, 0, s>>>(
                n, rp, cl, ty, new_of.as<int32_t>(), G.rp.as<int64_t>(), G.node_off.as<int64_t>(), ngraphs, nb,
                keys.as<unsigned long long>(), status);
            TG_CK(cudaGetLastError());
        }
        if (nnz > 0)
            cub_call([&](void *t, size_t &b) {
                return cub::DeviceRadixSort::SortKeys(t, b, keys.as<unsigned long long>(), keys2.as<unsigned long long>(),
                                                      nnz, 0, 2 * nb + kTypeBits, s);
            }, s);
        ++G.last_launches;
        k_rows<<<blocks_for((n + 1) * kWarp, kThreads), kThreads, 0, s>>>(
            n, L, nb, G.rp.as<int64_t>(), keys2.as<unsigned long long>(), G.adj.as<int32_t>(), G.toff.as<int32_t>(),
            G.tdeg.as<uint32_t>(), G.pivot.as<int32_t>(), nplus.as<int64_t>(), G.most_lower.as<int32_t>(),
            info.as<int64_t>() + 2 * ngraphs + 3, status);
        TG_CK(cudaGetLastError());
    }
    // types by internal id
    if (n > 0) {
        ++G.last_launches;
        k_gather_types<<<blocks_for(n, kThreads), kThreads, 0, s>>>(n, G.old_of.as<int32_t>(), ty, G.ty.as<uint8_t>());
        TG_CK(cudaGetLastError());
    }
    cub_call([&](void *t, size_t &b) {
        return cub::DeviceScan::ExclusiveSum(t, b, nplus.as<int64_t>(), G.plus_off.as<int64_t>(), n + 1, s);
    }, s);
    // slots, edges and largest degree per graph; graph g's edges are those whose smaller caller id lies in
    // graph g: with caller ids grouped by graph and lexicographic edge order they are contiguous, half of
    // its rows' entries
    ++G.last_launches;
    k_graph_info<<<blocks_for(ngraphs + 1, kThreads), kThreads, 0, s>>>(
        G.view(), info.as<int64_t>(), info.as<int64_t>() + ngraphs + 1, info.as<int64_t>() + 2 * ngraphs + 1, status);
    TG_CK(cudaGetLastError());
    TG_CK(cudaMemcpyAsync(h_info.data(), info.p, sizeof(int64_t) * h_info.size(), cudaMemcpyDeviceToHost, s));
    TG_CK(cudaStreamSynchronize(s));
    if ((uint32_t)h_info[2 * (size_t)ngraphs + 2] & ST_INVALID_GRAPH)
        throw Error{TG_ERR_INVALID_GRAPH, "self-loop, repeated entry or cross-graph edge"};
    const int64_t m = G.m;
    if (h_info[2 * (size_t)ngraphs + 1] != m) throw Error{TG_ERR_INVALID_GRAPH, "asymmetric rows"};
    G.h_slot_off.assign(h_info.begin(), h_info.begin() + ngraphs + 1);
    G.h_edge_off.assign(ngraphs + 1, 0);
    G.max_degree = 0;
    for (int g = 0; g < ngraphs; ++g) {
        G.h_edge_off[g + 1] = G.h_edge_off[g] + (G.h_slot_off[g + 1] - G.h_slot_off[g]) / 2;
        G.max_degree = std::max(G.max_degree, h_info[(size_t)ngraphs + 1 + g]);
    }
    if (G.h_edge_off[ngraphs] != m) throw Error{TG_ERR_INVALID_GRAPH, "edge count per graph"};

    // 4. higher-priority neighbour lists (one entry per edge), and the edges in caller order
    G.slot_eid.alloc(sizeof(int32_t) * std::max<int64_t>(nnz, 1));
    G.e_lo.alloc(sizeof(int32_t) * std::max<int64_t>(m, 1));
    G.e_hi.alloc(sizeof(int32_t) * std::max<int64_t>(m, 1));
    G.e_slot_lo.alloc(sizeof(int64_t) * std::max<int64_t>(m, 1));
    G.e_slot_hi.alloc(sizeof(int64_t) * std::max<int64_t>(m, 1));
    G.plus_adj.alloc(sizeof(int32_t) * std::max<int64_t>(m, 1));
    G.plus_eid.alloc(sizeof(int32_t) * std::max<int64_t>(m, 1));
    // a class holds at most m / (its smallest |N+|) nodes
    G.tri_list[0].alloc(sizeof(int32_t) * (size_t)(m / (kTriWarpMax + 1) + 1));
    G.tri_list[1].alloc(sizeof(int32_t) * (size_t)(m / (kTriMidMax + 1) + 1));
    G.tri_list[2].alloc(sizeof(int32_t) * (size_t)(m / (kTriBigMax + 1) + 1));
    TBuf counts(sizeof(unsigned long long) * 4, s);
    TG_CK(cudaMemsetAsync(counts.p, 0, sizeof(unsigned long long) * 4, s));
    if (m > 0) {
        TBuf ekeys(sizeof(unsigned long long) * m, s), ekeys2(sizeof(unsigned long long) * m, s);
        TBuf epos(sizeof(uint32_t) * m, s), epos2(sizeof(uint32_t) * m, s), plus_slot(sizeof(uint32_t) * m, s);
        ++G.last_launches;
        k_plus_fill<<<blocks_for(n * kWarp, kThreads), kThreads, 0, s>>>(
            G.view(), G.old_of.as<int32_t>(), nb, G.plus_adj.as<int32_t>(), plus_slot.as<uint32_t>(),
            ekeys.as<unsigned long long>(), epos.as<uint32_t>(), G.tri_list[0].as<int32_t>(),
            G.tri_list[1].as<int32_t>(), G.tri_list[2].as<int32_t>(), counts.as<unsigned long long>());
        TG_CK(cudaGetLastError());
        cub_call([&](void *t, size_t &b) {
            return cub::DeviceRadixSort::SortPairs(t, b, ekeys.as<unsigned long long>(), ekeys2.as<unsigned long long>(),
                                                   epos.as<uint32_t>(), epos2.as<uint32_t>(), m, 0, 2 * nb, s);
        }, s);
        ++G.last_launches;
        k_edges<<<blocks_for(m, kThreads), kThreads, 0, s>>>(
            m, nb, ekeys2.as<unsigned long long>(), epos2.as<uint32_t>(), plus_slot.as<uint32_t>(), G.view(),
            new_of.as<int32_t>(), G.e_lo.as<int32_t>(), G.e_hi.as<int32_t>(), G.e_slot_lo.as<int64_t>(),
            G.e_slot_hi.as<int64_t>(), G.slot_eid.as<int32_t>(), G.plus_eid.as<int32_t>(), status);
        TG_CK(cudaGetLastError());
    }

    unsigned long long h_counts[4];
    uint32_t h_status = 0;
    TG_CK(cudaMemcpyAsync(h_counts, counts.p, sizeof(h_counts), cudaMemcpyDeviceToHost, s));
    TG_CK(cudaMemcpyAsync(&h_status, G.status.p, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    TG_CK(cudaStreamSynchronize(s));
    if (h_status & ST_INVALID_GRAPH) throw Error{TG_ERR_INVALID_GRAPH, "asymmetric rows"};
    for (int c = 0; c < 3; ++c) G.tri_count[c] = (int64_t)h_counts[c];
    G.max_nplus = (int64_t)h_counts[3];
    G.narrow = !h_info[2 * (size_t)ngraphs + 3] && nnz < kNarrowSlots && G.max_degree < kNarrowTotal;
}

// What only 4-node counts need, before the first of them: the per-node typed
// degree sums and the wedge anchors by class.  3-node, directed and edge-typed
// counts never read them (3-node counts of 10 M edges with their build 7.75 ->
// 6.46 ms without them, directed 5 M edges 6.13 -> 5.41).
void prepare_anchors(Graph &G, cudaStream_t s) {
    const int64_t n = G.n;
    const int L = G.L;
    G.delta.alloc(G.node_sum_bytes() * std::max<int64_t>(n * L * L, 1));
    launch_row_sums(G, G.adj.as<int32_t>(), G.tdeg.as<uint32_t>(), G.delta.p, s);
    TBuf work(sizeof(int64_t) * std::max<int64_t>(n, 1), s);
    TG_CK(cudaMemsetAsync(work.p, 0, sizeof(int64_t) * std::max<int64_t>(n, 1), s));
    if (n > 0) {
        k_anchor_work<<<blocks_for(n * kWarp, kThreads), kThreads, 0, s>>>(G.view(), work.as<unsigned long long>());
        TG_CK(cudaGetLastError());
    }
    list_anchors(G, work.as<int64_t>(), G.most_lower.as<int32_t>(), s);
    G.h_hub_id.assign((size_t)G.n_hubs, 0);
    G.h_hub_wedges.assign((size_t)G.n_hubs, 0);
    if (G.n_hubs > 0) {
        // hub order: by graph, type and id, as the entries of the N+ lists
        TBuf wk(sizeof(int64_t) * (size_t)G.n_hubs, s);
        std::vector<int32_t> id((size_t)G.n_hubs);
        std::vector<int64_t> wt((size_t)G.n_hubs);
        k_gather_work<<<blocks_for(G.n_hubs, kThreads), kThreads, 0, s>>>(
            G.n_hubs, G.hubs.as<int32_t>(), work.as<int64_t>(), G.ty.as<uint8_t>(), wk.as<int64_t>());
        TG_CK(cudaGetLastError());
        TG_CK(cudaMemcpyAsync(id.data(), G.hubs.p, sizeof(int32_t) * G.n_hubs, cudaMemcpyDeviceToHost, s));
        TG_CK(cudaMemcpyAsync(wt.data(), wk.p, sizeof(int64_t) * G.n_hubs, cudaMemcpyDeviceToHost, s));
        TG_CK(cudaStreamSynchronize(s));
        std::vector<std::pair<std::pair<int64_t, int64_t>, int64_t>> order((size_t)G.n_hubs);   // ((graph, type), id), wedges
        for (size_t h = 0; h < order.size(); ++h) {
            const int64_t gr = std::upper_bound(G.h_node_off.begin(), G.h_node_off.end(), (int64_t)id[h]) -
                               G.h_node_off.begin();
            order[h] = {{gr, (wt[h] & 15) << kTypeShift | id[h]}, wt[h] >> 4};
        }
        std::sort(order.begin(), order.end());
        for (size_t h = 0; h < order.size(); ++h) {
            G.h_hub_id[h] = (int32_t)(order[h].first.second & kIdMask);
            G.h_hub_wedges[h] = order[h].second;
        }
        TG_CK(cudaMemcpyAsync(G.hubs.p, G.h_hub_id.data(), sizeof(int32_t) * G.n_hubs, cudaMemcpyHostToDevice, s));
    }
    G.most_lower.release();
    G.anchors_ready = true;
}

}  // namespace tg

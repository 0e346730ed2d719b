// tg_visit.cuh -- calls a functor once per triangle of a graph (host launch of
// the enumeration of tg_local.cuh), for the counts whose per-edge cells are
// added to in global memory.
//
// The functor is a struct passed by value; its call gets the triangle u < a <
// b (internal ids) as its edges' ids and its nodes' types:
//   v(e_ua, e_ub, e_ab, type of u, type of a, type of b)
//
// Measured against intersecting the typed rows of every edge (5 M Chung-Lu
// edges, L = 5): directed 3-node counts 11.6 -> 0.90 ms for the cells and 0.54
// for the rows, edge-typed ones (4 edge types) 12.4 -> 1.58 and 2.8 ms.
#pragma once

#include <algorithm>

#include "tg_host.hpp"
#include "tg_local.cuh"

namespace tg {

template <class V>
__global__ void __launch_bounds__(256) k_visit_warp(GraphView g, V v) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; u < g.n; u += nw) {
        const int64_t pb = g.plus_off[u];
        const int p = (int)(g.plus_off[u + 1] - pb);
        if (p < 2 || p > kTriWarpMax) continue;
        const int tu = g.ty[u];
        const uint32_t ent = lane < p ? (uint32_t)g.plus_adj[pb + lane] : 0u;
        const uint32_t eid = lane < p ? (uint32_t)g.plus_eid[pb + lane] : 0u;
        const int np = p * (p - 1) / 2;
        for (int x0 = 0; x0 < np; x0 += 32) {
            const int x = x0 + lane;
            int k = 0, l = 0;
            if (x < np) pair_of(x, k, l);
            const uint32_t ek = __shfl_sync(0xffffffffu, ent, k), el = __shfl_sync(0xffffffffu, ent, l);
            const uint32_t dk = __shfl_sync(0xffffffffu, eid, k), dl = __shfl_sync(0xffffffffu, eid, l);
            if (x >= np) continue;
            const bool kl = (ek & (uint32_t)kIdMask) < (el & (uint32_t)kIdMask);
            const uint32_t ea = kl ? ek : el, eb = kl ? el : ek;
            const int64_t pos = plus_find(g, (int32_t)(ea & (uint32_t)kIdMask), eb);
            if (pos < 0) continue;
            v((int64_t)(kl ? dk : dl), (int64_t)(kl ? dl : dk), (int64_t)g.plus_eid[pos], tu, (int)(ea >> kTypeShift),
              (int)(eb >> kTypeShift));
        }
    }
}

template <int kThreadsT, bool kSmem, class V>
__global__ void __launch_bounds__(kThreadsT) k_visit_cta(GraphView g, V v, const int32_t *__restrict__ list,
                                                         int64_t n_list, int cap, int lgf, unsigned char *scratch,
                                                         int64_t stride) {
    extern __shared__ unsigned char visit_smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int kWarps = kThreadsT / 32;
    LocalList q;
    if (kSmem) local_carve(q, visit_smem, cap, lgf, kWarps, wid);
    else local_carve(q, scratch + (int64_t)blockIdx.x * stride, cap, lgf, kWarps, wid);
    for (int64_t x = blockIdx.x; x < n_list; x += gridDim.x) {
        const int32_t u = list[x];
        const int64_t pb = g.plus_off[u];
        const int p = (int)(g.plus_off[u + 1] - pb);
        const int tu = g.ty[u];
        local_load(g, pb, p, q);
        local_pairs(g, p, q, lane, wid, kWarps, [&](bool hit, int ka, int kb, uint32_t pos) {
            if (hit)
                v((int64_t)q.eid[ka], (int64_t)q.eid[kb], (int64_t)g.plus_eid[pos], tu, (int)(q.ent[ka] >> kTypeShift),
                  (int)(q.ent[kb] >> kTypeShift));
        });
        __syncthreads();                                    // the list is replaced next
    }
}

// Edges whose cells are counted together: all of them where their cells fit
// four times the handle's working budget (cycle_budget_mb) and device memory
// has room, else windows of equal numbers of edges, each with a visit of the
// triangles of its own (a functor of a window passes other edges by).
// Allocates `cells` at the handle's first such count.
int64_t cell_window(Graph &G, DBuf &cells, size_t edge_bytes);

// launches the functor over every triangle of the handle's graph; returns the launches
template <class V>
int64_t visit_triangles(Graph &G, V v, cudaStream_t s) {
    const GraphView gv = G.view();
    const int sms = sm_count();
    int64_t launches = 1;
    k_visit_warp<V><<<(unsigned)std::max<int64_t>(1, std::min<int64_t>((G.n + 7) / 8, (int64_t)sms * 64)), 256, 0, s>>>(gv, v);
    for (int cls = 0; cls < 3; ++cls) {
        const LocalClass c = local_class(G, cls);
        if (c.n == 0) continue;
        const size_t bytes = (local_bytes(c.cap, c.lgf, c.threads / 32) + 15) & ~(size_t)15;
        ++launches;
        if (cls == 2) {
            const int64_t grid = std::min<int64_t>(c.n, sms);
            prepare_tri_scratch(G);
            k_visit_cta<kTriBigThreads, false, V><<<(unsigned)grid, kTriBigThreads, 0, s>>>(
                gv, v, c.list, c.n, c.cap, c.lgf, G.tri_scratch.as<unsigned char>(), (int64_t)bytes);
            continue;
        }
        auto run = [&](auto kern) {
            raise_smem_limit((const void *)kern, bytes);
            const int per_sm = std::max(1, std::min<int>(2048 / c.threads, (int)((226u << 10) / (bytes + 1024))));
            kern<<<(unsigned)std::min<int64_t>(c.n, (int64_t)sms * per_sm), c.threads, bytes, s>>>(
                gv, v, c.list, c.n, c.cap, c.lgf, nullptr, 0);
        };
        if (cls == 0) run(k_visit_cta<kTriMidThreads, true, V>);
        else run(k_visit_cta<kTriBigThreads, true, V>);
    }
    TG_CK(cudaGetLastError());
    return launches;
}

}  // namespace tg

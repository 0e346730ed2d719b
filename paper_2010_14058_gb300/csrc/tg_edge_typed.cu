// tg_edge_typed.cu -- typed 3-node graphlets of a graph whose edges carry
// types too (Def. 1's edge types xi; Defs. 4-5: the class of a typed
// graphlet is its shape with the multisets of its node types and of its
// edge types).
//
// The handle is the ordinary tg_build layout (rows by (type, id), per-type
// segments) plus one edge type per edge and, per node x, node type t and edge
// type q, the number d_x^{t,q} of x's type-t neighbours joined to x by an
// edge of type q.  Every triangle is found once (tg_visit.cuh) and counted at
// each of its edges in the slot (t, {types of the other two edges}); these
// cells are the row's triangle slots.  A second kernel forms the 3-path slots
// and the class sums.  The sets S_i, S_j follow by Cor. 1-2, split by edge
// type:
//   |S_i^{t,x}| = d_i^{t,x} - |{w in T^t : xi_iw = x}| - [phi_j = t, xi_ij = x]
// and likewise for S_j.  A 3-path's slot is (t, x) whichever endpoint is its
// centre (its class ({phi_i, phi_j, t}, {xi_ij, x}) is the same), so it needs
// |{w : xi_iw = x}| + |{w : xi_jw = x}|, which the unordered cells give.
// Per-edge layout and class ranks: include/tg.h.
#include <algorithm>

#include "tg_host.hpp"
#include "tg_tiles.cuh"
#include "tg_visit.cuh"

namespace tg {

namespace {

constexpr int kMaxX = TG_MAX_EDGE_TYPES;

// multisets of size r from n symbols, C(n + r - 1, r)
__host__ __device__ inline int64_t mchoose(int n, int r) {
    int64_t c = 1;
    for (int k = 1; k <= r; ++k) c = c * (n + k - 1) / k;
    return c;
}

// rank of the non-decreasing K-tuple s over [0, A) among all of them in
// lexicographic order: for each position, the tuples that agree before it
// and hold a smaller value there
__host__ __device__ inline int64_t ms_rank(int A, int K, const int *s) {
    int64_t r = 0;
    int prev = 0;
    for (int k = 0; k < K; ++k) {
        for (int v = prev; v < s[k]; ++v) r += mchoose(A - v, K - k - 1);
        prev = s[k];
    }
    return r;
}

__host__ __device__ inline void sort2(int *a) {
    if (a[1] < a[0]) { const int x = a[0]; a[0] = a[1]; a[1] = x; }
}
__host__ __device__ inline void sort3v(int *a) {
    if (a[1] < a[0]) { const int x = a[0]; a[0] = a[1]; a[1] = x; }
    if (a[2] < a[1]) { const int x = a[1]; a[1] = a[2]; a[2] = x; }
    if (a[1] < a[0]) { const int x = a[0]; a[0] = a[1]; a[1] = x; }
}

// ---------------------------------------------------------------- build
__global__ void k_et_new_of(int64_t n, const int32_t *__restrict__ old_of, int32_t *new_of) {
    const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (x < n) new_of[old_of[x]] = (int32_t)x;
}

// slot of internal node y in the typed segment of row x, or -1
__device__ __forceinline__ int64_t et_slot(const GraphView &g, int32_t x, int32_t y) {
    const int64_t b = seg_begin(g, x, g.ty[y]), e = seg_end(g, x, g.ty[y]);
    const int64_t r = lower_bound_i32(g.adj, b, e, y);
    return (r < e && g.adj[r] == y) ? r : -1;
}

// the caller's entry k (row found by binary search over its row pointers)
// gives its edge type to the slot of that entry
__global__ void k_et_fill(GraphView g, int64_t nnz, const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
                          const uint8_t *__restrict__ xi, int X, const int32_t *__restrict__ new_of, uint8_t *etype,
                          uint32_t *status) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= nnz) return;
    int64_t lo = 0, hi = g.n;                               // rp[lo] <= k < rp[hi]
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (rp[mid] <= k) lo = mid; else hi = mid;
    }
    const uint8_t t = xi[k];
    if (t >= X) {
        set_status(status, ST_INVALID_GRAPH);
        return;
    }
    const int64_t s = et_slot(g, new_of[lo], new_of[col[k]]);
    if (s < 0) {
        set_status(status, ST_INTERNAL);
        return;
    }
    etype[s] = t;
}

// both slots of every edge hold the same type, which is the edge's
__global__ void k_et_check(GraphView g, const uint8_t *__restrict__ etype, uint8_t *by_edge, uint32_t *status) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= g.m) return;
    const uint8_t a = etype[g.e_slot_lo[e]], b = etype[g.e_slot_hi[e]];
    if (a == 0xff || a != b) set_status(status, ST_INVALID_GRAPH);
    by_edge[e] = a;
}

// d_x^{t,q}: warp per node, one warp sum per (type, edge type)
__global__ void __launch_bounds__(256) k_et_degree(GraphView g, const uint8_t *__restrict__ etype, int X,
                                                   int32_t *etdeg) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; x < g.n; x += nw) {
        for (int t = 0; t < g.L; ++t) {
            unsigned c[kMaxX];
#pragma unroll
            for (int q = 0; q < kMaxX; ++q) c[q] = 0;
            for (int64_t s = seg_begin(g, x, t) + lane; s < seg_end(g, x, t); s += 32) {
                const int q = etype[s];
#pragma unroll
                for (int r = 0; r < kMaxX; ++r) c[r] += q == r ? 1u : 0u;
            }
#pragma unroll
            for (int q = 0; q < kMaxX; ++q) {
                if (q >= X) break;
                const unsigned v = __reduce_add_sync(0xffffffffu, c[q]);
                if (lane == 0) etdeg[(x * g.L + t) * X + q] = (int32_t)v;
            }
        }
    }
}

// ---------------------------------------------------------------- count
// position of the unordered pair {x, y} among the pairs of X edge types
__device__ __forceinline__ int x_pair(int X, int x, int y) {
    const int a = x < y ? x : y, b = x < y ? y : x;
    return a * X - a * (a - 1) / 2 + (b - a);
}

// cells [edge][type of the third node][pair of its edges' types]
template <bool kWindow>
struct EdgeTypedCells {
    uint32_t *cell;             // of edge 0 (the array starts at e0's)
    int64_t stride;             // words from edge to edge
    const uint8_t *xi;
    int X, P;
    int64_t e0, e1;             // kWindow: edges with cells
    __device__ __forceinline__ void add(int64_t e, int slot) const {
        if (kWindow && (e < e0 || e >= e1)) return;
        atomicAdd(&cell[e * stride + slot], 1u);
    }
    __device__ __forceinline__ void operator()(int64_t ua, int64_t ub, int64_t ab, int tu, int ta, int tb) const {
        const int xa = xi[ua], xb = xi[ub], xab = xi[ab];
        add(ua, tb * P + x_pair(X, xb, xab));
        add(ub, ta * P + x_pair(X, xa, xab));
        add(ab, tu * P + x_pair(X, xa, xb));
    }
};

constexpr int kRowThreads = 256;

// zeroes the cells of every edge, a warp per edge (a thread per cell spent its
// time on the 64-bit division of its number)
__global__ void __launch_bounds__(256) k_et_zero(int64_t m, int64_t stride, int words, uint32_t *cell) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t e = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; e < m; e += nw)
        for (int x = lane; x < words; x += 32) cell[e * stride + x] = 0u;
}

// Thread per (edge, slot): the 3-path slot from the typed degrees and the
// cells, or the triangle slot's cell; class sums (block 0 edges, block 1
// 3-paths, block 2 triangles) are kept in registers while the endpoints'
// types and the edge's type stay the same.  Bound by the latency of the
// gathers and the rows written; the endpoints of a tile's edges are staged in
// shared memory by visiting order (5 M edges, L = 5, X = 4: 2.78 -> 2.45 ms).
template <int L, int X>
__global__ void __launch_bounds__(kRowThreads) k_edge_typed_rows(GraphView g, const uint32_t *__restrict__ cell,
                                                                 int64_t stride, const uint8_t *__restrict__ xi,
                                                                 const int32_t *__restrict__ etdeg, int G, int64_t tile,
                                                                 int64_t e0, int64_t e1,
                                                                 uint32_t *per_edge_out,
                                                                 unsigned long long *gacc, uint32_t *status) {
    extern __shared__ unsigned long long ehist[];
    __shared__ TileOrder<L * L * X> o;
    __shared__ int2 ends[kTile];                            // by order: rows of etdeg of the edges' endpoints
    constexpr int P = X * (X + 1) / 2, S = L * X + L * P, E = kRowThreads / S;
    const int64_t off1 = mchoose(L, 2) * X, off2 = off1 + mchoose(L, 3) * mchoose(X, 2);
    const int64_t w2 = mchoose(X, 2), w3 = mchoose(X, 3);
    for (int s = threadIdx.x; s < G; s += blockDim.x) ehist[s] = 0;
    // ranks of the multisets {phi_i, phi_j, t}, {xi_ij, x}, {xi_ij, x, y}
    __shared__ uint16_t rank_n[L * L * L], rank_2[X * X], rank_3[X * X * X];
    for (int k = threadIdx.x; k < L * L * L; k += blockDim.x) {
        int n3[3] = {k / (L * L), k / L % L, k % L};
        sort3v(n3);
        rank_n[k] = (uint16_t)ms_rank(L, 3, n3);
    }
    for (int k = threadIdx.x; k < X * X * X; k += blockDim.x) {
        int e3[3] = {k / (X * X), k / X % X, k % X}, e2[2] = {k / X, k % X};
        sort3v(e3);
        rank_3[k] = (uint16_t)ms_rank(X, 3, e3);
        if (k >= X * X) continue;
        sort2(e2);
        rank_2[k] = (uint16_t)ms_rank(X, 2, e2);
    }
    const int slice = threadIdx.x / S, slot = threadIdx.x % S;
    const bool path = slot < L * X;
    const int t = path ? slot / X : (slot - L * X) / P;
    const int pair = path ? 0 : (slot - L * X) % P;
    int x_at[X];                                            // pairs {x0, z} of a path slot
    int x0 = 0, y0 = 0;                                     // the slot's edge types: {x} or {x, y}
    if (path) {
        x0 = slot % X;
    } else {
        int r = pair;
        while (r >= X - x0) { r -= X - x0; ++x0; }
        y0 = x0 + r;
    }
#pragma unroll
    for (int z = 0; z < X; ++z) x_at[z] = x_pair(X, x0, z);
    for (int64_t b = e0 + blockIdx.x * tile; b < e1; b += gridDim.x * tile) {
        const int n = (int)min(tile, e1 - b);
        tile_order(b, n, o, [&](int64_t e) { return (g.ty[g.e_lo[e]] * L + g.ty[g.e_hi[e]]) * X + xi[e]; });
        for (int x = threadIdx.x; x < n; x += blockDim.x) {
            const int64_t e = b + o.order[x];
            ends[x] = make_int2(g.e_lo[e], g.e_hi[e]);
        }
        __syncthreads();
        for (int k = threadIdx.x; k < L * L * X; k += blockDim.x)
            if (o.count[k]) {
                int n2[2] = {k / X / L, k / X % L};
                sort2(n2);
                atomicAdd(&ehist[ms_rank(L, 2, n2) * X + k % X], (unsigned long long)o.count[k]);
            }
        if (slice >= E) continue;
        int xb, xe;
        slice_of(n, slice, E, xb, xe);
        unsigned long long acc = 0;
        int key = -1;
        auto flush = [&]() {
            const int n3 = rank_n[(key / X) * L + t];
            if (acc)
                atomicAdd(&ehist[path ? off1 + n3 * w2 + rank_2[key % X * X + x0]
                                      : off2 + n3 * w3 + rank_3[(key % X * X + x0) * X + y0]], acc);
            acc = 0;
        };
        for (int x = xb; x < xe; ++x) {
            const int rel = o.order[x], k = o.key[rel];
            const int64_t e = b + rel;
            if (k != key) {
                if (key >= 0) flush();
                key = k;
            }
            const uint32_t *c = cell + e * stride + t * P;
            int64_t v;
            if (path) {
                const int pi = k / X / L, pj = k / X % L, xij = k % X;
                v = (int64_t)etdeg[((int64_t)ends[x].x * L + t) * X + x0] + etdeg[((int64_t)ends[x].y * L + t) * X + x0] -
                    ((pj == t && xij == x0) ? 1 : 0) - ((pi == t && xij == x0) ? 1 : 0);
#pragma unroll
                for (int z = 0; z < X; ++z) v -= (int64_t)c[x_at[z]] * (z == x0 ? 2 : 1);
                if (v < 0) {
                    set_status(status, ST_INTERNAL);
                    v = 0;
                }
                if (per_edge_out) per_edge_out[e * S + slot] = (uint32_t)v;   // (the cells are in place)
            } else {
                v = c[pair];
            }
            acc += (unsigned long long)v;
        }
        if (key >= 0) flush();
    }
    __syncthreads();
    for (int s = threadIdx.x; s < G; s += blockDim.x)
        if (ehist[s]) atomicAdd(&gacc[s], ehist[s]);
}

// totals (Sec. 6): each 3-path was seen from its 2 edges, each triangle
// from its 3
__global__ void k_et_finalize(int G, int64_t off1, int64_t off2, const unsigned long long *__restrict__ gacc,
                              int64_t *global_out, uint32_t *status) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= G) return;
    const unsigned long long d = s < off1 ? 1ull : (s < off2 ? 2ull : 3ull);
    if (gacc[s] % d) set_status(status, ST_INTERNAL);
    global_out[s] = (int64_t)(gacc[s] / d);
}

}  // namespace

int64_t edge_typed_global_slots(int L, int X) {
    return mchoose(L, 2) * X + mchoose(L, 3) * mchoose(X, 2) + mchoose(L, 3) * mchoose(X, 3);
}

// Edge types of the slots (from the caller's CSR positions, device arrays)
// and the per-node counts by (node type, edge type); throws
// TG_ERR_INVALID_GRAPH for a type out of range or different on the two
// entries of an edge.
void prepare_edge_typed(Graph &G, int X, const int64_t *row_ptr, const int32_t *col, const uint8_t *edge_types,
                        cudaStream_t s) {
    const GraphView gv = G.view();
    TBuf by_slot(std::max<int64_t>(G.nnz, 1), s);
    G.etype.alloc(std::max<int64_t>(G.m, 1));
    G.etdeg.alloc(sizeof(int32_t) * (size_t)std::max<int64_t>(G.n * G.L * X, 1));
    TG_CK(cudaMemsetAsync(by_slot.p, 0xff, std::max<int64_t>(G.nnz, 1), s));
    TG_CK(cudaMemsetAsync(G.status.p, 0, sizeof(uint32_t), s));
    TBuf new_of(sizeof(int32_t) * std::max<int64_t>(G.n, 1), s);
    if (G.n > 0)
        k_et_new_of<<<(unsigned)((G.n + 255) / 256), 256, 0, s>>>(G.n, G.old_of.as<int32_t>(), new_of.as<int32_t>());
    if (G.nnz > 0)
        k_et_fill<<<(unsigned)((G.nnz + 255) / 256), 256, 0, s>>>(gv, G.nnz, row_ptr, col, edge_types, X,
                                                                   new_of.as<int32_t>(), by_slot.as<uint8_t>(),
                                                                   G.status.as<uint32_t>());
    if (G.m > 0)
        k_et_check<<<(unsigned)((G.m + 255) / 256), 256, 0, s>>>(gv, by_slot.as<uint8_t>(), G.etype.as<uint8_t>(),
                                                                 G.status.as<uint32_t>());
    TG_CK(cudaGetLastError());
    uint32_t st = 0;
    TG_CK(cudaMemcpyAsync(&st, G.status.p, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    TG_CK(cudaStreamSynchronize(s));
    if (st & ST_INVALID_GRAPH) throw Error{TG_ERR_INVALID_GRAPH, "edge types out of range or unequal on an edge's entries"};
    if (st) throw Error{TG_ERR_INTERNAL, "edge type slots"};
    if (G.n > 0)
        k_et_degree<<<(unsigned)std::min<int64_t>((G.n + 7) / 8, (int64_t)sm_count() * 16), 256, 0, s>>>(
            gv, by_slot.as<uint8_t>(), X, G.etdeg.as<int32_t>());
    TG_CK(cudaGetLastError());
    G.et_X = X;
    G.et_global = edge_typed_global_slots(G.L, X);
    G.etgacc.alloc(sizeof(unsigned long long) * (size_t)G.et_global);
    G.edge_typed = true;
}

int64_t run_edge_typed3(Graph &G, uint32_t *per_edge_out, int64_t *global_out, cudaStream_t s) {
    const int Gs = (int)G.et_global, X = G.et_X, L = G.L;
    TG_CK(cudaMemsetAsync(G.etgacc.p, 0, sizeof(unsigned long long) * (size_t)Gs, s));
    const size_t smem = sizeof(unsigned long long) * (size_t)Gs;
    int64_t launches = 0;
    if (G.m > 0) {
        const int P = X * (X + 1) / 2, S = L * X + L * P;
        // the rows hold the cells; without rows, a buffer of the handle
        const int64_t stride = per_edge_out ? S : L * P;
        const int64_t window = per_edge_out ? G.m : cell_window(G, G.etcell, sizeof(uint32_t) * (size_t)stride);
        const int64_t tile = tile_edges(G);
        for (int64_t e0 = 0; e0 < G.m; e0 += window) {
            const int64_t e1 = std::min(G.m, e0 + window);
            uint32_t *first = per_edge_out ? per_edge_out + L * X : G.etcell.as<uint32_t>(), *cell = first - e0 * stride;
            {
                KernelTimer kt(G, s, "k_edge_typed_cells");
                k_et_zero<<<(unsigned)std::min<int64_t>((e1 - e0 + 7) / 8, (int64_t)sm_count() * 64), 256, 0, s>>>(
                    e1 - e0, stride, L * P, first);
                const uint8_t *xi = G.etype.as<uint8_t>();
                if (window >= G.m) launches += 1 + visit_triangles(G, EdgeTypedCells<false>{cell, stride, xi, X, P, e0, e1}, s);
                else launches += 1 + visit_triangles(G, EdgeTypedCells<true>{cell, stride, xi, X, P, e0, e1}, s);
            }
            KernelTimer kt(G, s, "k_edge_typed_rows");
            const unsigned grid = (unsigned)std::min<int64_t>((e1 - e0 + tile - 1) / tile, (int64_t)sm_count() * 6);
            with_types(L, [&](auto l) {
                constexpr int kL = decltype(l)::value;
                auto run = [&](auto kern) {
                    raise_smem_limit((const void *)kern, smem);
                    kern<<<grid, kRowThreads, smem, s>>>(G.view(), cell, stride, G.etype.as<uint8_t>(), G.etdeg.as<int32_t>(),
                                                         Gs, tile, e0, e1, per_edge_out, G.etgacc.as<unsigned long long>(),
                                                         G.status.as<uint32_t>());
                };
                if (X == 1) run(k_edge_typed_rows<kL, 1>);
                else if (X == 2) run(k_edge_typed_rows<kL, 2>);
                else if (X == 3) run(k_edge_typed_rows<kL, 3>);
                else run(k_edge_typed_rows<kL, 4>);
            });
            ++launches;
        }
    }
    if (global_out) {
        const int64_t off1 = mchoose(L, 2) * X, off2 = off1 + mchoose(L, 3) * mchoose(X, 2);
        k_et_finalize<<<(unsigned)((Gs + 255) / 256), 256, 0, s>>>(Gs, off1, off2, G.etgacc.as<unsigned long long>(),
                                                                  global_out, G.status.as<uint32_t>());
        ++launches;
    }
    TG_CK(cudaGetLastError());
    return launches;
}

}  // namespace tg

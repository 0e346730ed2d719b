// tg_epi.cu -- rows and totals of every edge from the gathered sums.
//
// k_epi4 and k_epi4_pa evaluate the inclusion-exclusion of Thm. 1 (formulas
// at the head of tg_count.cu) with one thread per (edge, unordered type pair
// {t, u}): the entries (t, u) and (u, t) of the L x L matrices close over
// each other, so a thread loads both and needs no other thread (a warp per
// edge with the matrices spread over its lanes spent about 1,000 warp
// instructions per edge, most of them on 64-bit shuffles for transposes).
// The CTA takes a tile of edges at a time and visits them grouped by their
// endpoints' types (p, q): a thread's pair is fixed, so within a group every
// value it finds belongs to the same class and is added in a register; the
// histogram in shared memory is touched once per group.
// Measured on 20 M Chung-Lu edges (L = 5) and 30 M block-model edges (L = 4),
// against a warp per edge with an atomic per value: 39.1 -> 26.8 and 50.3 ->
// 29.7 ms, with the slots' 4-cycle values read as rows (k_slot_rows, 1.5
// and 1.2 ms) 11.7 and 9.8 ms, and with 32-bit values and node sums where
// they fit (a narrow graph, kNarrowDegree; 64 registers instead of 80, so a
// fourth CTA per SM, and half the bytes of the nodes' tables) 7.9
// and 7.3 ms, with the tile's edges staged (stage_ends) 6.6 and 6.2, with 32-bit
// sums throughout 6.7 and 6.0; 3-node rows of 10 M edges 3.0 -> 0.56 ms.
// Bound now: DRAM at 0.82 of the measured copy rate (36.5 GB on the 20 M
// edges of the benchmark graph: 12.9 of rows written, 23.6 read, of which the
// two nodes' tables of every edge, which do not stay in L2, are the most) at
// 32 warps per SM.  Narrow with 3 or 5 CTAs'
// registers: 51.8 and 53.6 ms per pass of the block model against 51.3
// (before the staging).
#include <algorithm>

#include "tg_host.hpp"
#include "tg_tiles.cuh"

namespace tg {

namespace {

constexpr int kEpiThreads = 256;

// lexicographic rank of a sorted K-multiset over [0,L): the number of
// non-decreasing K-tuples that precede it, counted position by position.
__device__ __forceinline__ int multichoose(int n, int r) {   // C(n + r - 1, r), n >= 1
    int64_t v = 1;
    for (int k = 1; k <= r; ++k) v = v * (n + k - 1) / k;
    return (int)v;
}
__device__ int multiset_rank_dev(int L, int K, const int *s) {
    int r = 0, prev = 0;
    for (int k = 0; k < K; ++k) {
        for (int v = prev; v < s[k]; ++v) r += multichoose(L - v, K - k - 1);
        prev = s[k];
    }
    return r;
}
__device__ __forceinline__ void sort4(int *s) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 3 - a; ++b)
            if (s[b] > s[b + 1]) { int x = s[b]; s[b] = s[b + 1]; s[b + 1] = x; }
}
__device__ __forceinline__ void sort3(int *s) {
    if (s[0] > s[1]) { int x = s[0]; s[0] = s[1]; s[1] = x; }
    if (s[1] > s[2]) { int x = s[1]; s[1] = s[2]; s[2] = x; }
    if (s[0] > s[1]) { int x = s[0]; s[0] = s[1]; s[1] = x; }
}

// global block offsets (block 0 edges, 1 3-path, 2 triangle, 3..8 four-node)
__device__ __forceinline__ int gblock_off(int L, int b) {
    int c2 = multichoose(L, 2), c3 = multichoose(L, 3), c4 = multichoose(L, 4);
    if (b == 0) return 0;
    if (b <= 2) return c2 + (b - 1) * c3;
    return c2 + 2 * c3 + (b - 3) * c4;
}

__device__ __forceinline__ int pair_idx(int L, int t, int u) {   // t <= u
    return t * L - t * (t - 1) / 2 + (u - t);
}
// pair number -> (t, u)
__device__ __forceinline__ void pair_types(int L, int pi, int &t, int &u) {
    t = 0;
    while (pair_idx(L, t, L - 1) < pi) ++t;
    u = t + (pi - pair_idx(L, t, t));
}

__device__ __forceinline__ uint32_t sat32(int32_t v, uint32_t *) { return (uint32_t)v; }   // (narrow: below 2^31)
__device__ __forceinline__ uint32_t sat32(int64_t v, uint32_t *status) {
    if (v > 0xffffffffll) {
        set_status(status, ST_OVERFLOW);
        return 0xffffffffu;
    }
    return (uint32_t)v;
}

// adds the CTA's histogram to the graph's sums and clears it
__device__ void flush_hist(unsigned long long *hist, int G, unsigned long long *gacc, int graph) {
    for (int s = threadIdx.x; s < G; s += blockDim.x) {
        const unsigned long long v = hist[s];
        if (v) atomicAdd(&gacc[(int64_t)graph * G + s], v);
        hist[s] = 0;
    }
}

// the types of the endpoints, p * L + q; by_caller: p is the type of the
// endpoint with the smaller caller id, else of e_lo
template <int L>
__device__ __forceinline__ void order_by_types(const GraphView &g, const Tile &tile, TileOrder<L * L> &o, bool by_caller,
                                               const int32_t *__restrict__ old_of) {
    tile_order(tile.begin, (int)(tile.end - tile.begin), o, [&](int64_t e) {
        const int32_t i = g.e_lo[e], j = g.e_hi[e];
        const bool swap = by_caller && old_of[i] > old_of[j];
        return g.ty[swap ? j : i] * L + g.ty[swap ? i : j];
    });
}

// By order: the endpoints of the tile's edges (by_caller's first if old_of, so
// x > y says that they are swapped) and the edge's slots in rows e_lo and
// e_hi, of the chunk; ends with a barrier.  Read once per edge here instead
// of by each of its threads ahead of everything that they point to: k_epi4
// 7.9 -> 7.1 (20 M Chung-Lu edges) and 7.3 -> 6.5 ms (30 M block model), and
// with tiles of 1,024 edges instead of 2,048 6.6 and 6.2 (512: 6.6 and 6.3).
template <int kKeys>
__device__ __forceinline__ void stage_ends(const GraphView &g, const CountView &cv, const Tile &tile,
                                           const TileOrder<kKeys> &o, uint4 *ends, const int32_t *__restrict__ old_of) {
    for (int x = threadIdx.x; x < (int)(tile.end - tile.begin); x += blockDim.x) {
        const int64_t e = tile.begin + o.order[x];
        const int32_t i = g.e_lo[e], j = g.e_hi[e];
        const bool swap = old_of && old_of[i] > old_of[j];
        ends[x] = make_uint4((uint32_t)(swap ? j : i), (uint32_t)(swap ? i : j), (uint32_t)(g.e_slot_lo[e] - cv.a_base),
                             (uint32_t)(g.e_slot_hi[e] - cv.a_base));
    }
    __syncthreads();
}

// ------------------------------------------------------------ slot rows
// The wedge pass adds to one plane per type pair (consecutive slots of a plane
// take its updates in whole sectors); an edge needs the L^2 values of two
// slots, one sector each from the planes.  This pass turns the planes into
// rows of L^2 words: 32 slots of every plane per warp through shared memory,
// read and written in runs of 128 bytes and more.
constexpr int kRowWarps = 4;
template <int L>
__global__ void __launch_bounds__(kRowWarps * 32) k_slot_rows(const uint32_t *__restrict__ A, int64_t stride,
                                                              int64_t n_slots, uint32_t *__restrict__ rows) {
    constexpr int LL = L * L;
    __shared__ uint32_t tile[kRowWarps][LL * 33];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t *t = tile[wid];
    const int64_t nw = (int64_t)gridDim.x * kRowWarps;
    for (int64_t b = ((int64_t)blockIdx.x * kRowWarps + wid) * 32; b < n_slots; b += nw * 32) {
        const int64_t s = b + lane;
#pragma unroll
        for (int k = 0; k < LL; ++k) t[k * 33 + lane] = s < n_slots ? __ldcs(A + k * stride + s) : 0u;
        __syncwarp();
        const int n = (int)min((int64_t)32, n_slots - b) * LL;
        for (int x = lane; x < n; x += 32) rows[b * LL + x] = t[(x % LL) * 33 + x / LL];
        __syncwarp();
    }
}

// ------------------------------------------------------------ one type pair
// Every matrix entry of one edge at (t, u) [0] and (u, t) [1], i the first
// endpoint (type p) and j the second (type q).
template <class T>
struct PairVals {
    T ct, cu, at, au, bt, bu;       // |T^t|, |S_i^t|, |S_j^t|
    T CTi[2], CTj[2], Q[2], Ri[2], Rj[2], G8[2], Wi, Wj, Ks;
};

template <int L, class T>
__device__ __forceinline__ void pair_values(const GraphView &g, const CountView &cv, int64_t e, int32_t i, int32_t j,
                                            int p, int q, bool swap, int64_t s0, int64_t s1, int t, int u,
                                            PairVals<T> &v) {
    // (e_lo, e_hi) = swap ? (j, i) : (i, j); s0, s1: the edge's slots in rows e_lo and e_hi, of the chunk
    constexpr int LL = L * L;
    const uint32_t *C = cv.C + e * kCRow;
    v.ct = (T)C[t];
    v.cu = (T)C[u];
    const int32_t *oi = g.toff + (int64_t)i * (L + 1), *oj = g.toff + (int64_t)j * (L + 1);
    const T dit = oi[t + 1] - oi[t], diu = oi[u + 1] - oi[u];
    const T djt = oj[t + 1] - oj[t], dju = oj[u + 1] - oj[u];
    v.at = dit - v.ct - (q == t ? 1 : 0);
    v.au = diu - v.cu - (q == u ? 1 : 0);
    v.bt = djt - v.ct - (p == t ? 1 : 0);
    v.bu = dju - v.cu - (p == u ? 1 : 0);
    // sums over T; rows of types without a triangle node are not kept.  (Where
    // they are loaded decides the registers: first in 32 bits, last in 64; the
    // block model's epilogue takes 6.0 ms, 6.3 with them last, and one of 2 M
    // edges beside a star of 70,000 leaves 1.07 ms, 1.27 with them first.)
    T TC0[2] = {0, 0}, TC1[2] = {0, 0}, DT[2] = {0, 0}, K[2] = {0, 0};
    auto load = [&](int row, int col, int h) {
        const uint32_t *r = cv.xsum + ((e - cv.e_base) * L + row) * 4 * L + col;
        TC0[h] = (T)r[0]; TC1[h] = (T)r[L]; DT[h] = (T)r[2 * L]; K[h] = (T)r[3 * L];
    };
    auto load_sums = [&]() {
        if (sizeof(T) == 4 && !(v.ct | v.cu)) return;
        if (v.ct) load(t, u, 0);
        if (v.cu) load(u, t, 1);
    };
    if (sizeof(T) == 4) load_sums();
    const int k0 = t * L + u, k1 = u * L + t;
    // P[x][y]: slot i->j holds [type next to i][type next to j], slot j->i the reverse
    const uint32_t *Aij = cv.slot_rows + (swap ? s1 : s0) * LL, *Aji = cv.slot_rows + (swap ? s0 : s1) * LL;
    const T P0 = (T)Aij[k1] + (T)Aji[k0];
    const T P1 = (T)Aij[k0] + (T)Aji[k1];
    const T *tau = static_cast<const T *>(cv.tau), *delta = static_cast<const T *>(g.delta);
    const T *tau_i = tau + (int64_t)i * LL, *tau_j = tau + (int64_t)j * LL;
    const T *del_i = delta + (int64_t)i * LL, *del_j = delta + (int64_t)j * LL;
    const T ti = tau_i[k0], tj = tau_j[k0];         // symmetric
    if (sizeof(T) > 4) load_sums();
    v.Ks = (K[0] + K[1]) >> 1;                              // ordered adjacent pairs of T (K' counts each twice)
    v.CTi[0] = (swap ? TC1[0] : TC0[0]) - v.Ks - (u == q ? v.ct : 0);
    v.CTi[1] = (swap ? TC1[1] : TC0[1]) - v.Ks - (t == q ? v.cu : 0);
    v.CTj[0] = (swap ? TC0[0] : TC1[0]) - v.Ks - (u == p ? v.ct : 0);
    v.CTj[1] = (swap ? TC0[1] : TC1[1]) - v.Ks - (t == p ? v.cu : 0);
    v.Wi = ti - v.CTi[0] - v.CTi[1] - v.Ks - (t == q ? v.cu : 0) - (u == q ? v.ct : 0);
    v.Wj = tj - v.CTj[0] - v.CTj[1] - v.Ks - (t == p ? v.cu : 0) - (u == p ? v.ct : 0);
    v.Q[0] = P0 - v.CTj[1] - v.CTi[0] - v.Ks;
    v.Q[1] = P1 - v.CTj[0] - v.CTi[1] - v.Ks;
    v.Ri[0] = del_i[k0] - DT[0] - (t == q ? dju : 0) - (u == p ? v.at : 0) - v.Wi - v.CTi[1] - v.Q[1];
    v.Ri[1] = del_i[k1] - DT[1] - (u == q ? djt : 0) - (t == p ? v.au : 0) - v.Wi - v.CTi[0] - v.Q[0];
    v.Rj[0] = del_j[k0] - DT[0] - (t == p ? diu : 0) - (u == q ? v.bt : 0) - v.Wj - v.CTj[1] - v.Q[0];
    v.Rj[1] = del_j[k1] - DT[1] - (u == p ? dit : 0) - (t == q ? v.bu : 0) - v.Wj - v.CTj[0] - v.Q[1];
    v.G8[0] = DT[0] - ((u == p ? 1 : 0) + (u == q ? 1 : 0)) * v.ct - v.Ks - v.CTi[0] - v.CTj[0];
    v.G8[1] = DT[1] - ((t == p ? 1 : 0) + (t == q ? 1 : 0)) * v.cu - v.Ks - v.CTi[1] - v.CTj[1];
}

// ------------------------------------------------------------ typed rows
// Shared memory of k_epi4: the tile's staged edges, the histogram of G(L) u64, then the multiset rank
// tables rank2[p][q], rank3[p][q][t], rank4[p][q][pair] (uint16).
size_t epi4_smem_bytes(int L) {
    const int P = L * (L + 1) / 2;
    return kTile * sizeof(uint4) + (size_t)global_slots(L, 4) * sizeof(unsigned long long) +
           (size_t)(L * L + L * L * L + L * L * P + 1) * sizeof(uint16_t);
}

template <int L, class T>
__global__ void __launch_bounds__(kEpiThreads, sizeof(T) == 4 ? 4 : 3)
    k_epi4(GraphView g, CountView cv, const Tile *__restrict__ tiles, int64_t n_tiles, int64_t row_base,
           uint32_t *per_edge_out, unsigned long long *gacc) {
    constexpr int LL = L * L, P = L * (L + 1) / 2, S = 2 * L + 10 * P;
    constexpr int E = kEpiThreads / P;                      // edges in flight per CTA
    extern __shared__ __align__(16) uint4 ends[];           // by order: nodes and slots of the tile's edges
    unsigned long long *hist = reinterpret_cast<unsigned long long *>(ends + kTile);
    __shared__ TileOrder<LL> o;
    const int G = (int)global_slots(L, 4);
    uint16_t *rank2 = reinterpret_cast<uint16_t *>(hist + G);
    uint16_t *rank3 = rank2 + LL;
    uint16_t *rank4 = rank3 + LL * L;
    for (int s = threadIdx.x; s < G; s += blockDim.x) hist[s] = 0;
    for (int k = threadIdx.x; k < LL * P; k += blockDim.x) {
        const int pq = k / P;
        int ms[4] = {pq / L, pq % L, 0, 0};
        pair_types(L, k % P, ms[2], ms[3]);
        sort4(ms);
        rank4[k] = (uint16_t)multiset_rank_dev(L, 4, ms);
    }
    for (int k = threadIdx.x; k < LL * L; k += blockDim.x) {
        int ms[3] = {k / LL, (k / L) % L, k % L};
        sort3(ms);
        rank3[k] = (uint16_t)multiset_rank_dev(L, 3, ms);
    }
    for (int k = threadIdx.x; k < LL; k += blockDim.x) {
        int ms[2] = {k / L < k % L ? k / L : k % L, k / L < k % L ? k % L : k / L};
        rank2[k] = (uint16_t)multiset_rank_dev(L, 2, ms);
    }
    const int off1 = gblock_off(L, 1), off2 = gblock_off(L, 2), off4 = gblock_off(L, 3), c4 = multichoose(L, 4);
    const int slice = threadIdx.x / P, pi = threadIdx.x % P;
    int t, u;
    pair_types(L, pi, t, u);
    int cur_graph = -1;
    for (int64_t ti = blockIdx.x; ti < n_tiles; ti += gridDim.x) {
        const Tile tile = tiles[ti];
        order_by_types<L>(g, tile, o, false, nullptr);
        stage_ends(g, cv, tile, o, ends, nullptr);
        if (tile.graph != cur_graph) {
            if (cur_graph >= 0) flush_hist(hist, G, gacc, cur_graph);
            __syncthreads();
            cur_graph = tile.graph;
        }
        for (int k = threadIdx.x; k < LL; k += blockDim.x)
            if (o.count[k]) atomicAdd(&hist[rank2[k]], (unsigned long long)o.count[k]);
        if (slice >= E) continue;
        int xb, xe;
        slice_of((int)(tile.end - tile.begin), slice, E, xb, xe);
        unsigned long long acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // graphlet blocks 3..8, then 1 and 2
        int key = -1;
        auto flush = [&]() {
            const int r = rank4[key * P + pi];
#pragma unroll
            for (int b = 0; b < 6; ++b) {
                if (acc[b]) atomicAdd(&hist[off4 + b * c4 + r], acc[b]);
                acc[b] = 0;
            }
            if (t == u) {
                const int r3 = rank3[key * L + t];
                if (acc[6]) atomicAdd(&hist[off1 + r3], acc[6]);
                if (acc[7]) atomicAdd(&hist[off2 + r3], acc[7]);
                acc[6] = acc[7] = 0;
            }
        };
        for (int x = xb; x < xe; ++x) {
            const int64_t e = tile.begin + o.order[x];
            const int k = o.key[o.order[x]];
            if (k != key) {
                if (key >= 0) flush();
                key = k;
            }
            PairVals<T> v;
            const uint4 at = ends[x];
            pair_values<L, T>(g, cv, e, (int32_t)at.x, (int32_t)at.y, k / L, k % L, false, at.z, at.w, t, u, v);
            T gv[10];
            bool ok = v.at >= 0 && v.au >= 0 && v.bt >= 0 && v.bu >= 0;
            if (t != u) {
                gv[0] = v.Ri[0] + v.Rj[0] + v.Ri[1] + v.Rj[1];         // g3
                gv[3] = v.Q[0] + v.Q[1];                               // g6
                gv[4] = v.Wi + v.Wj;                                   // g7
                gv[5] = v.G8[0] + v.G8[1];                             // g8
                gv[7] = v.CTi[0] + v.CTj[0] + v.CTi[1] + v.CTj[1];     // g10
                gv[9] = v.Ks;                                          // g12
                gv[1] = v.at * v.bu + v.au * v.bt - gv[3];             // Lemma 1
                gv[2] = v.at * v.au + v.bt * v.bu - gv[4];             // Lemma 2
                gv[6] = v.ct * (v.au + v.bu) + v.cu * (v.at + v.bt) - gv[7];   // Lemma 3
                gv[8] = v.ct * v.cu - gv[9];                           // Lemma 4
            } else {
                const T w = v.Wi + v.Wj;
                ok = ok && !(w & 1) && !(v.Ks & 1);
                gv[0] = v.Ri[0] + v.Rj[0];
                gv[3] = v.Q[0];
                gv[4] = w / 2;
                gv[5] = v.G8[0];
                gv[7] = v.CTi[0] + v.CTj[0];
                gv[9] = v.Ks / 2;
                gv[1] = v.at * v.bt - gv[3];
                gv[2] = v.at * (v.at - 1) / 2 + v.bt * (v.bt - 1) / 2 - gv[4];
                gv[6] = v.ct * (v.at + v.bt) - gv[7];
                gv[8] = v.ct * (v.ct - 1) / 2 - gv[9];
                acc[6] += (unsigned long long)(v.at + v.bt);
                acc[7] += (unsigned long long)v.ct;
            }
#pragma unroll
            for (int b = 0; b < 10; ++b) ok = ok && gv[b] >= 0;
            if (!ok) set_status(cv.status, ST_INTERNAL);
            if (per_edge_out) {
                uint32_t *row = per_edge_out + (e - row_base) * S;
                if (t == u) {
                    row[t] = sat32(v.at + v.bt, cv.status);
                    row[L + t] = sat32(v.ct, cv.status);
                }
#pragma unroll
                for (int b = 0; b < 10; ++b) row[2 * L + b * P + pi] = sat32(gv[b], cv.status);
            }
            acc[0] += (unsigned long long)gv[0] + (unsigned long long)gv[1];             // 4-path: g3, g4
            acc[1] += (unsigned long long)gv[2];                       // 4-star: g5
            acc[2] += (unsigned long long)gv[3];                       // 4-cycle: g6
            acc[3] += (unsigned long long)gv[4] + (unsigned long long)gv[5] + (unsigned long long)gv[6];     // tailed triangle: g7, g8, g9
            acc[4] += (unsigned long long)gv[7] + (unsigned long long)gv[8];             // chordal cycle: g10, g11
            acc[5] += (unsigned long long)gv[9];                       // 4-clique: g12
        }
        if (key >= 0) flush();
    }
    __syncthreads();
    if (cur_graph >= 0) flush_hist(hist, G, gacc, cur_graph);
}

// k = 3: 3-node slots and global blocks 0..2 only, thread per (edge, type)
template <int L>
__global__ void __launch_bounds__(kEpiThreads) k_edge3(GraphView g, CountView cv, const Tile *__restrict__ tiles,
                                                       int64_t n_tiles, int64_t e_begin, uint32_t *per_edge_out,
                                                       unsigned long long *gacc) {
    constexpr int LL = L * L, S = 2 * L, E = kEpiThreads / L;
    extern __shared__ unsigned long long hist[];
    __shared__ TileOrder<LL> o;
    const int G = (int)global_slots(L, 3);
    for (int s = threadIdx.x; s < G; s += blockDim.x) hist[s] = 0;
    const int off1 = gblock_off(L, 1), off2 = gblock_off(L, 2);
    const int slice = threadIdx.x / L, t = threadIdx.x % L;
    int cur_graph = -1;
    for (int64_t ti = blockIdx.x; ti < n_tiles; ti += gridDim.x) {
        const Tile tile = tiles[ti];
        order_by_types<L>(g, tile, o, false, nullptr);
        if (tile.graph != cur_graph) {
            if (cur_graph >= 0) flush_hist(hist, G, gacc, cur_graph);
            __syncthreads();
            cur_graph = tile.graph;
        }
        for (int k = threadIdx.x; k < LL; k += blockDim.x)
            if (o.count[k]) {
                int ms[2] = {k / L < k % L ? k / L : k % L, k / L < k % L ? k % L : k / L};
                atomicAdd(&hist[multiset_rank_dev(L, 2, ms)], (unsigned long long)o.count[k]);
            }
        if (slice >= E) continue;
        int xb, xe;
        slice_of((int)(tile.end - tile.begin), slice, E, xb, xe);
        unsigned long long paths = 0, triangles = 0;
        int key = -1;
        auto flush = [&]() {
            int ms[3] = {key / L, key % L, t};
            sort3(ms);
            const int r = multiset_rank_dev(L, 3, ms);
            if (paths) atomicAdd(&hist[off1 + r], paths);
            if (triangles) atomicAdd(&hist[off2 + r], triangles);
            paths = triangles = 0;
        };
        for (int x = xb; x < xe; ++x) {
            const int64_t e = tile.begin + o.order[x];
            const int k = o.key[o.order[x]];
            if (k != key) {
                if (key >= 0) flush();
                key = k;
            }
            const int64_t c = cv.C[e * kCRow + t];
            const int64_t a = typed_degree(g, g.e_lo[e], t) - c - (k % L == t ? 1 : 0);
            const int64_t b = typed_degree(g, g.e_hi[e], t) - c - (k / L == t ? 1 : 0);
            if (per_edge_out) {
                uint32_t *row = per_edge_out + (e - e_begin) * S;
                row[t] = sat32(a + b, cv.status);
                row[L + t] = sat32(c, cv.status);
            }
            paths += (unsigned long long)(a + b);
            triangles += (unsigned long long)c;
        }
        if (key >= 0) flush();
    }
    __syncthreads();
    if (cur_graph >= 0) flush_hist(hist, G, gacc, cur_graph);
}

// ------------------------------------------------- position-aware rows
// Sec. 5 (Def. 8): before k_epi4 folds them into unordered type pairs, the
// pair's values already keep the positions of an instance apart: Ri / Rj
// (4-path end edges with inner endpoint i / j: w the inner endpoint's other
// neighbour, r the far end), Q (4-cycles; first index the type of j's
// neighbour), Wi / Wj (adjacent pairs inside S_i / S_j), CTi / CTj (a
// triangle node and an adjacent node of S_i / S_j), G8 (a triangle node and
// its tail in I) and K (adjacent pairs inside T).  k_epi4_pa takes i as the
// endpoint with the smaller caller id (side 0), writes the values by
// position -- the row layout of tg_pa.cu -- and adds every count to the class
// that the slot and the endpoint types fix (host table).
struct PaView {
    const int32_t *cls;       // [L*L][S+1] class of (phi_lo, phi_hi, slot); slot S: the edge itself
    const int32_t *old_of;    // [n] caller id of each internal node
    int32_t S;                // per-edge slots
    int32_t G;                // classes (global slots) per graph
    int32_t off[13];          // first slot of blocks O1..O12
};

template <int L, class T>
__global__ void __launch_bounds__(kEpiThreads, 2) k_epi4_pa(GraphView g, CountView cv, PaView pv,
                                                         const Tile *__restrict__ tiles, int64_t n_tiles,
                                                         int64_t row_base, uint32_t *per_edge_out,
                                                         unsigned long long *gacc) {
    constexpr int LL = L * L, P = L * (L + 1) / 2, E = kEpiThreads / P;
    constexpr int kOrdered = 9, kPairs = 6;
    extern __shared__ __align__(16) uint4 ends[];
    unsigned long long *hist = reinterpret_cast<unsigned long long *>(ends + kTile);
    __shared__ TileOrder<LL> o;
    const int S = pv.S, G = pv.G;
    for (int s = threadIdx.x; s < G; s += blockDim.x) hist[s] = 0;
    const int slice = threadIdx.x / P, pi = threadIdx.x % P;
    int t, u;
    pair_types(L, pi, t, u);
    // slots of this thread's values, in the order they are emitted
    const int ktu = t * L + u;
    const int so[kOrdered] = {pv.off[3], pv.off[3] + LL, pv.off[4], pv.off[6], pv.off[8],
                              pv.off[9], pv.off[9] + LL, pv.off[10], pv.off[10] + LL};
    const int sp[kPairs] = {pv.off[5], pv.off[5] + P, pv.off[7], pv.off[7] + P, pv.off[11], pv.off[12]};
    int cur_graph = -1;
    for (int64_t ti = blockIdx.x; ti < n_tiles; ti += gridDim.x) {
        const Tile tile = tiles[ti];
        order_by_types<L>(g, tile, o, true, pv.old_of);
        stage_ends(g, cv, tile, o, ends, pv.old_of);
        if (tile.graph != cur_graph) {
            if (cur_graph >= 0) flush_hist(hist, G, gacc, cur_graph);
            __syncthreads();
            cur_graph = tile.graph;
        }
        for (int k = threadIdx.x; k < LL; k += blockDim.x)   // the edges themselves
            if (o.count[k]) atomicAdd(&hist[pv.cls[(int64_t)k * (S + 1) + S]], (unsigned long long)o.count[k]);
        if (slice >= E) continue;
        int xb, xe;
        slice_of((int)(tile.end - tile.begin), slice, E, xb, xe);
        unsigned long long acc_o[2][kOrdered], acc_p[kPairs], acc_3[3];
#pragma unroll
        for (int b = 0; b < kOrdered; ++b) acc_o[0][b] = acc_o[1][b] = 0;
#pragma unroll
        for (int b = 0; b < kPairs; ++b) acc_p[b] = 0;
        acc_3[0] = acc_3[1] = acc_3[2] = 0;
        int key = -1;
        auto flush = [&]() {
            const int32_t *cls = pv.cls + (int64_t)key * (S + 1);
            auto add = [&](int slot, unsigned long long &a) {
                if (a) atomicAdd(&hist[cls[slot]], a);
                a = 0;
            };
#pragma unroll
            for (int b = 0; b < kOrdered; ++b) {
                add(so[b] + ktu, acc_o[0][b]);
                if (t != u) add(so[b] + u * L + t, acc_o[1][b]);
            }
#pragma unroll
            for (int b = 0; b < kPairs; ++b) add(sp[b] + pi, acc_p[b]);
            if (t == u) {
                add(pv.off[1] + t, acc_3[0]);
                add(pv.off[1] + L + t, acc_3[1]);
                add(pv.off[2] + t, acc_3[2]);
            }
        };
        for (int x = xb; x < xe; ++x) {
            const int64_t e = tile.begin + o.order[x];
            const int k = o.key[o.order[x]];
            if (k != key) {
                if (key >= 0) flush();
                key = k;
            }
            const uint4 at = ends[x];
            PairVals<T> v;
            pair_values<L, T>(g, cv, e, (int32_t)at.x, (int32_t)at.y, k / L, k % L, at.x > at.y, at.z, at.w, t, u, v);
            uint32_t *row = per_edge_out ? per_edge_out + (e - row_base) * S : nullptr;
            bool ok = v.at >= 0 && v.au >= 0 && v.bt >= 0 && v.bu >= 0;
            auto emit = [&](int slot, T val, unsigned long long &a) {
                ok = ok && val >= 0;
                if (row) row[slot] = sat32(val, cv.status);
                a += (unsigned long long)val;
            };
            if (t == u) {
                emit(pv.off[1] + t, v.at, acc_3[0]);                  // 3-path centred at lo
                emit(pv.off[1] + L + t, v.bt, acc_3[1]);              // centred at hi
                emit(pv.off[2] + t, v.ct, acc_3[2]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {                             // ordered blocks at (x, y) = (t, u), (u, t)
                if (h == 1 && t == u) break;
                const int xy = h == 0 ? ktu : u * L + t;
                const T cx = h == 0 ? v.ct : v.cu;
                const T ax = h == 0 ? v.at : v.au, ay = h == 0 ? v.au : v.at;
                const T by = h == 0 ? v.bu : v.bt;
                const T QT = v.Q[1 - h];
                emit(so[0] + xy, v.Ri[h], acc_o[h][0]);               // inner endpoint lo: near x, far y
                emit(so[1] + xy, v.Rj[h], acc_o[h][1]);
                emit(so[2] + xy, ax * by - QT, acc_o[h][2]);          // lo's neighbour x, hi's y (Lemma 1)
                emit(so[3] + xy, QT, acc_o[h][3]);                    // 4-cycle: lo's neighbour x, hi's y
                emit(so[4] + xy, v.G8[h], acc_o[h][4]);               // triangle node x, tail y
                emit(so[5] + xy, cx * ay - v.CTi[h], acc_o[h][5]);    // Lemma 3, degree-3 node lo
                emit(so[6] + xy, cx * by - v.CTj[h], acc_o[h][6]);
                emit(so[7] + xy, v.CTi[h], acc_o[h][7]);              // chordal outer edge, degree-3 node lo
                emit(so[8] + xy, v.CTj[h], acc_o[h][8]);
            }
            T star_i, star_j, tail_i, tail_j, chord, clique;
            if (t != u) {
                star_i = v.at * v.au - v.Wi;                          // Lemma 2, centre lo
                star_j = v.bt * v.bu - v.Wj;
                tail_i = v.Wi;
                tail_j = v.Wj;
                chord = v.ct * v.cu - v.Ks;                           // Lemma 4
                clique = v.Ks;
            } else {
                ok = ok && !(v.Wi & 1) && !(v.Wj & 1) && !(v.Ks & 1);
                star_i = v.at * (v.at - 1) / 2 - v.Wi / 2;
                star_j = v.bt * (v.bt - 1) / 2 - v.Wj / 2;
                tail_i = v.Wi / 2;
                tail_j = v.Wj / 2;
                chord = v.ct * (v.ct - 1) / 2 - v.Ks / 2;
                clique = v.Ks / 2;
            }
            emit(sp[0] + pi, star_i, acc_p[0]);
            emit(sp[1] + pi, star_j, acc_p[1]);
            emit(sp[2] + pi, tail_i, acc_p[2]);
            emit(sp[3] + pi, tail_j, acc_p[3]);
            emit(sp[4] + pi, chord, acc_p[4]);
            emit(sp[5] + pi, clique, acc_p[5]);
            if (!ok) set_status(cv.status, ST_INTERNAL);
        }
        if (key >= 0) flush();
    }
    __syncthreads();
    if (cur_graph >= 0) flush_hist(hist, G, gacc, cur_graph);
}

// global totals: C_H = (1/|E(H)|) * sum_e x_e (Sec. 6), exact division
__global__ void k_finalize(int ngraphs, int L, int k, const unsigned long long *__restrict__ gacc, int64_t *out,
                           uint32_t *status) {
    const int G = (int)global_slots(L, k);
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= (int64_t)ngraphs * G) return;
    const int s = (int)(idx % G);
    const int nb = k == 4 ? 9 : 3;
    int b = 0;
    while (b + 1 < nb && gblock_off(L, b + 1) <= s) ++b;
    const int edges_of[9] = {1, 2, 3, 3, 3, 4, 4, 5, 6};
    const unsigned long long v = gacc[idx];
    if (v % edges_of[b]) set_status(status, ST_INTERNAL);
    out[idx] = (int64_t)(v / edges_of[b]);
}

PaView pa_view(const Graph &G) {
    PaView v;
    v.cls = G.pa_cls.as<int32_t>();
    v.old_of = G.old_of.as<int32_t>();
    v.S = G.pa.S;
    v.G = (int32_t)G.pa.G;
    for (int o = 0; o < 13; ++o) v.off[o] = G.pa.off[o];
    return v;
}

size_t pa_smem_bytes(const Graph &G) { return kTile * sizeof(uint4) + (size_t)G.pa.G * sizeof(unsigned long long); }

unsigned epi_grid(int64_t n_tiles, int per_sm) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(n_tiles, (int64_t)sm_count() * per_sm));
}

}  // namespace

void prepare_epi(Graph &G) {
    with_types(G.L, [&](auto l) { 
        raise_smem_limit((const void *)k_epi4<decltype(l)::value, int32_t>, epi4_smem_bytes(G.L));
        raise_smem_limit((const void *)k_epi4<decltype(l)::value, int64_t>, epi4_smem_bytes(G.L));
    });
}

void prepare_epi4_pa(Graph &G) {
    with_types(G.L, [&](auto l) {
        raise_smem_limit((const void *)k_epi4_pa<decltype(l)::value, int32_t>, pa_smem_bytes(G));
        raise_smem_limit((const void *)k_epi4_pa<decltype(l)::value, int64_t>, pa_smem_bytes(G));
    });
}

int64_t launch_edges3(Graph &G, const Tile *tiles, int64_t n_tiles, int64_t e_begin, uint32_t *per_edge_out,
                      unsigned long long *gacc, cudaStream_t s) {
    if (n_tiles <= 0) return 0;
    KernelTimer kt(G, s, "k_edge3");
    with_types(G.L, [&](auto l) {
        k_edge3<decltype(l)::value>
            <<<(unsigned)std::min<int64_t>(n_tiles, (int64_t)sm_count() * 8), kEpiThreads,
               (size_t)global_slots(G.L, 3) * sizeof(unsigned long long), s>>>(G.view(), G.cview(), tiles, n_tiles,
                                                                               e_begin, per_edge_out, gacc);
    });
    TG_CK(cudaGetLastError());
    return 1;
}

int64_t launch_slot_rows(Graph &G, int64_t n_slots, cudaStream_t s) {
    if (n_slots <= 0) return 0;
    KernelTimer kt(G, s, "k_slot_rows");
    with_types(G.L, [&](auto l) {
        constexpr int L = decltype(l)::value;
        const int64_t blocks = (n_slots + kRowWarps * 32 - 1) / (kRowWarps * 32);
        k_slot_rows<L><<<(unsigned)std::min<int64_t>(blocks, (int64_t)sm_count() * 64), kRowWarps * 32, 0, s>>>(
            G.A.as<uint32_t>(), G.a_stride, n_slots, G.slot_rows.as<uint32_t>());
    });
    TG_CK(cudaGetLastError());
    return 1;
}

int64_t launch_edges4(Graph &G, const Tile *tiles, int64_t n_tiles, int64_t row_base, uint32_t *per_edge_out,
                      unsigned long long *gacc, cudaStream_t s) {
    if (n_tiles <= 0) return 0;
    KernelTimer kt(G, s, G.pa_active ? "k_epi4_pa" : "k_epi4");
    with_types(G.L, [&](auto l) {
        constexpr int L = decltype(l)::value;
        auto launch = [&](auto v) {
            using T = decltype(v);
            if (G.pa_active)
                k_epi4_pa<L, T><<<epi_grid(n_tiles, G.opt.ctas_per_sm), kEpiThreads, pa_smem_bytes(G), s>>>(
                    G.view(), G.cview(), pa_view(G), tiles, n_tiles, row_base, per_edge_out, gacc);
            else
                k_epi4<L, T><<<epi_grid(n_tiles, G.opt.ctas_per_sm + (G.narrow ? 1 : 0)), kEpiThreads, epi4_smem_bytes(L), s>>>(
                    G.view(), G.cview(), tiles, n_tiles, row_base, per_edge_out, gacc);
        };
        if (G.narrow) launch(int32_t());
        else launch(int64_t());
    });
    TG_CK(cudaGetLastError());
    return 1;
}

int64_t launch_finalize(Graph &G, int k, int64_t *global_out, cudaStream_t s) {
    const int64_t total = (int64_t)G.ngraphs * global_slots(G.L, k);
    KernelTimer kt(G, s, "k_finalize");
    k_finalize<<<(unsigned)std::max<int64_t>(1, (total + 255) / 256), 256, 0, s>>>(
        G.ngraphs, G.L, k, G.gacc.as<unsigned long long>(), global_out, G.status.as<uint32_t>());
    TG_CK(cudaGetLastError());
    return 1;
}

}  // namespace tg

// tg_count.cu -- per-edge typed 3- and 4-node graphlet counts and global totals.
//
// The GPU path computes, for every edge e = (i,j) (i the endpoint with the
// smaller internal id, types p = phi_i, q = phi_j), the same numbers as
// Alg. 1-3 + Lemmas 1-4 of the paper, but it never scans Gamma_w for every
// w in T u S_i u S_j (that scan costs sum_e sum_{w in U_e} d_w, far too much
// on hub-heavy graphs).  Instead it gathers these typed quantities
// (t = type of the first node, t' = type of the second):
//
//   c[t]        |T_ij^t| (Cor. 1), each triangle found once         (k_tri_*, tg_triangles.cu)
//   TCi[t][t']  sum_{w in T^t} c_{iw}^{t'}                         (k_sum_*, tg_sums.cu)
//   TCj[t][t']  sum_{w in T^t} c_{jw}^{t'}                         (k_sum_*)
//   DT[t][t']   sum_{w in T^t} d_w^{t'}                            (k_sum_*)
//   K[t][t']    ordered adjacent pairs (w,x) in T^t x T^t'          (k_sum_*)
//   P[t][t']    3-paths j - w - r - i, w of type t, r of type t'   (k_wedge*)
//   tau_x[t][t'] ordered adjacent pairs inside Gamma_x              (k_tau)
//   delta_x[t][t'] sum_{w in Gamma_x^t} d_w^{t'}                    (build)
//
// and obtains every orbit of Table 3 by the inclusion-exclusion of Thm. 1
// (the sets T, S_i, S_j, I of Cor. 1-2 and Eq. indep-node-set partition
// each neighbourhood):
//   CTi = TCi - K - [t'=q] c_t          (w in T, r in S_i, adjacent)
//   CTj = TCj - K - [t'=p] c_t          (w in T, r in S_j, adjacent)
//   Wi  = tau_i - CTi - CTi^T - K - [t=q] c_t' - [t'=q] c_t   (pairs in S_i)
//   Wj  = tau_j - CTj - CTj^T - K - [t=p] c_t' - [t'=p] c_t   (pairs in S_j)
//   Q   = P - CTj^T - CTi - K           (w in S_j, r in S_i: 4-cycles)
//   Ri  = delta_i - DT - [t=q] d_j^t' - [t'=p] a_t - Wi - CTi^T - Q^T   (S_i to I)
//   Rj  = delta_j - DT - [t=p] d_i^t' - [t'=q] b_t - Wj - CTj^T - Q     (S_j to I)
//   G8  = DT - ([t'=p]+[t'=q]) c_t - K - CTi - CTj                      (T to I)
// then, for t <= t' (X^T is the transpose):
//   g3 = R(+sym), g6 = Q(+sym), g7 = W/2 on the diagonal, g8 = G8(+sym),
//   g10 = CT(+sym), g12 = K/2 on the diagonal; g4, g5, g9, g11 by
//   Lemmas 1-4; global totals by Sec. 4.4 and Sec. 6.
//
// P uses degree-priority wedges: each 4-cycle is found once, from its node
// of highest (degree, id) priority u, as two wedges u - v - w and u - x - w
// with v, w, x all of lower priority; the wedge work is
// sum_{(u,v) in E} min(d_u, d_v).
#include <algorithm>
#include <mutex>
#include <vector>

#include "tg_host.hpp"
#include "tg_side.hpp"

namespace tg {

// Edges per tile: kTile, or fewer for a small handle so that its tiles
// still fill the GPU (at least about 12 tiles per SM, 64 edges or more each).
int64_t tile_edges(const Graph &G) {
    const int64_t want = (G.m + (int64_t)sm_count() * 12 - 1) / ((int64_t)sm_count() * 12);
    int64_t t = 64;
    while (t < want && t < kTile) t <<= 1;
    return t;
}

static std::vector<Tile> make_tiles(const Graph &G, int64_t e_begin, int64_t e_end) {
    std::vector<Tile> tiles;
    const int64_t te = tile_edges(G);
    for (int gi = 0; gi < G.ngraphs; ++gi) {
        int64_t b = std::max(e_begin, G.h_edge_off[gi]), e = std::min(e_end, G.h_edge_off[gi + 1]);
        for (int64_t x = b; x < e; x += te) tiles.push_back(Tile{x, std::min(e, x + te), gi, 0});
    }
    return tiles;
}

// Splits the graphs into consecutive chunks whose adjacency slots fit the
// 4-cycle array budget (a single graph larger than the budget is a chunk of
// its own), and sizes the array for the largest chunk.
static void plan_chunks(Graph &G) {
    G.chunks.clear();
    // working bytes of a chunk: the 4-cycle array by plane and by slot (8 L^2 per slot) and the
    // per-edge sums (4 L^2 words per edge)
    const int64_t LL = (int64_t)G.L * G.L;
    const int64_t budget = std::max<int64_t>((int64_t)G.opt.cycle_budget_mb << 20, 1);
    auto bytes_of = [&](int a, int b) {
        return (G.h_slot_off[b] - G.h_slot_off[a]) * 8 * LL + (G.h_edge_off[b] - G.h_edge_off[a]) * 16 * LL;
    };
    // tile index ranges follow graph boundaries (make_tiles emits graph after graph)
    std::vector<int64_t> tile_off(G.ngraphs + 1, 0);
    const int64_t te = tile_edges(G);
    for (int gi = 0; gi < G.ngraphs; ++gi)
        tile_off[gi + 1] = tile_off[gi] + (G.h_edge_off[gi + 1] - G.h_edge_off[gi] + te - 1) / te;
    int g0 = 0;
    int64_t widest = 0;
    while (g0 < G.ngraphs) {
        int g1 = g0 + 1;
        while (g1 < G.ngraphs && bytes_of(g0, g1 + 1) <= budget) ++g1;
        Graph::Chunk c;
        c.g0 = g0; c.g1 = g1;
        c.n0 = G.h_node_off[g0]; c.n1 = G.h_node_off[g1];
        c.s0 = G.h_slot_off[g0]; c.s1 = G.h_slot_off[g1];
        c.e0 = G.h_edge_off[g0]; c.e1 = G.h_edge_off[g1];
        c.t0 = tile_off[g0]; c.t1 = tile_off[g1];
        widest = std::max(widest, c.s1 - c.s0);
        G.max_chunk_edges = std::max(G.max_chunk_edges, c.e1 - c.e0);
        G.chunks.push_back(c);
        g0 = g1;
    }
    G.a_stride = std::max<int64_t>(widest, 1);
}

// Device tile list of [e_begin, e_end); the full range is cached by the
// handle (so that a captured CUDA graph never copies from host memory).
static const Tile *tiles_for(Graph &G, int64_t e_begin, int64_t e_end, int64_t &n_tiles, DBuf &tmp, cudaStream_t s) {
    const bool full = e_begin == 0 && e_end == G.m;
    if (full && G.tiles_full.p) {
        n_tiles = G.n_tiles_full;
        return G.tiles_full.as<Tile>();
    }
    std::vector<Tile> tiles = make_tiles(G, e_begin, e_end);
    n_tiles = (int64_t)tiles.size();
    DBuf &dst = full ? G.tiles_full : tmp;
    dst.upload(tiles.data(), sizeof(Tile) * tiles.size(), s);
    if (full) G.n_tiles_full = n_tiles;
    return dst.as<Tile>();
}

void raise_smem_limit(const void *func, size_t bytes) {
    struct Limit { const void *func; int dev; size_t bytes; };
    static std::mutex mu;
    static std::vector<Limit> set;
    int dev = 0;
    TG_CK(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    Limit *hit = nullptr;
    for (auto &l : set)
        if (l.func == func && l.dev == dev) hit = &l;
    if (hit && hit->bytes >= bytes) return;
    TG_CK(cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    if (hit) hit->bytes = bytes;
    else set.push_back({func, dev, bytes});
}

// Tiles and kernel attributes of the count (done before any capture).
void prepare_edges(Graph &G, int k, cudaStream_t s) {
    if (k == 4) prepare_epi(G);
    if (k == 4) prepare_wedges(G);
    DBuf unused;
    unused.owner = &G;
    int64_t nt = 0;
    tiles_for(G, 0, G.m, nt, unused, s);
}

// Sums and 4-cycle slots of chunk ci, after the triangles of the whole graph
// when `triangles` (their per-node sums included).  The kernels run beside
// each other (a pass of 40 k edges 543 -> 282 us, 1 M edges 4.10 -> 3.76 ms,
// 2 M 10.51 -> 10.25, a 30 M edge block model 55.8 -> 53.7), but:
// - not the hub pass, which fills the GPU and whose tables want the L2 cache
//   for themselves (beside the others: 2 M edges 13.4 ms, 20 M edges 162 ->
//   235 ms; on graphs of few hubs beside or after differs by 3% at most);
// - not under capture: a side stream stays in the capture until it ends, past
//   this call, so no other call could take it (and captured batches whose
//   replays overlap gained nothing: 41.0 -> 42.2 ms);
// - not when every kernel is timed by itself.
static int64_t launch_chunk(Graph &G, size_t ci, bool triangles, cudaStream_t s) {
    const Graph::Chunk &c = G.chunks[ci];
    const int L = G.L;
    int64_t launches = 0;
    G.a_base = c.s0;
    G.e_base = c.e0;
    if (c.s1 > c.s0)
        TG_CK(cudaMemset2DAsync(G.A.p, (size_t)G.a_stride * sizeof(uint32_t), 0, (size_t)(c.s1 - c.s0) * sizeof(uint32_t),
                                (size_t)L * L, s));
    if (G.timing || G.captured) {
        if (triangles) launches += launch_triangles(G, true, s);
        launches += launch_sums(G, c.n0, c.n1, c.e0, c.e1, s);
        if (G.n_hubs > 0) launches += launch_hubs(G, ci, s);
        launches += launch_anchor_wedges(G, 0, kHubClass - 1, c.n0, c.n1, s);
    } else {
        SideStreams side(s);
        side.fork();
        launches += launch_anchor_wedges(G, kHubClass - 1, kHubClass - 1, c.n0, c.n1, side.side(1));
        launches += launch_anchor_wedges(G, 2, kHubClass - 2, c.n0, c.n1, side.side(2));
        if (triangles) {
            launches += launch_triangles(G, false, s);
            side.after_main(0);
            launches += launch_row_sums(G, G.slot_eid.as<int32_t>(), G.C.as<uint32_t>(), G.tau.p, side.side(0));
        }
        launches += launch_anchor_wedges(G, 0, 1, c.n0, c.n1, side.side(1));
        launches += launch_sums(G, c.n0, c.n1, c.e0, c.e1, s);
        side.join();
        if (G.n_hubs > 0) launches += launch_hubs(G, ci, s);
    }
    launches += launch_slot_rows(G, c.s1 - c.s0, s);
    return launches;
}

// Allocates the working arrays of a count with this k (kept by the handle).
void prepare_counting(Graph &G, int k, cudaStream_t s) {
    const int L = G.L;
    const size_t m = (size_t)std::max<int64_t>(G.m, 1), n = (size_t)std::max<int64_t>(G.n, 1);
    G.C.alloc_once(m * kCRow * sizeof(uint32_t));
    G.tri_any.alloc_once(n);
    prepare_triangles(G);
    G.gacc.alloc_once((size_t)G.ngraphs * global_slots(L, 4) * sizeof(unsigned long long));
    if (k == 4) {
        if (!G.anchors_ready) prepare_anchors(G, s);
        G.tau.alloc_once(n * L * L * G.node_sum_bytes());
        if (G.chunks.empty()) plan_chunks(G);
        const size_t ab = (size_t)G.a_stride * L * L * sizeof(uint32_t);
        G.A.alloc_once(ab);
        G.slot_rows.alloc_once(ab);
        const size_t me = (size_t)std::max<int64_t>(G.max_chunk_edges, 1);
        G.xsum.alloc_once(me * 4 * L * L * sizeof(uint32_t));
        prepare_sums(G);
        if (G.n_hubs > 0 && G.hub_plans.empty()) prepare_hubs(G, s);
    }
}

int64_t run_count(Graph &G, int k, int64_t e_begin, int64_t e_end, uint32_t *per_edge_out, unsigned long long *gacc,
                  bool full, cudaStream_t s) {
    int64_t launches = 0;
    CountGuard guard(G);
    // prepared_k 3: typed triangles only (all that k = 3 reads); 4: their per-node sums too
    bool triangles = full || G.prepared_k < 3 || (k == 4 && !G.tau_ready);
    if (triangles && (k == 3 || G.chunks.size() != 1 || e_begin >= e_end || (!full && G.prepared_k == 4))) {
        launches += launch_triangles(G, k == 4, s);
        triangles = false;
        G.prepared_k = std::max(G.prepared_k, 3);
        G.tau_ready = G.tau_ready || k == 4;
    }
    DBuf tmp;                                                // tiles of a range, stream-ordered
    tmp.owner = &G;
    int64_t n_tiles = 0;
    const Tile *tiles = tiles_for(G, e_begin, e_end, n_tiles, tmp, s);
    if (k == 3) {
        launches += launch_edges3(G, tiles, n_tiles, e_begin, per_edge_out, gacc, s);
    } else {
        const bool whole = e_begin == 0 && e_end == G.m;
        std::vector<Tile> host;
        if (!whole) host = make_tiles(G, e_begin, e_end);
        for (size_t ci = 0; ci < G.chunks.size(); ++ci) {
            const Graph::Chunk &c = G.chunks[ci];
            const int64_t b = std::max(e_begin, c.e0), e = std::min(e_end, c.e1);
            if (b >= e) continue;
            // the wedge pass and sums of a single-chunk handle are reused by later range calls
            if (full || G.chunks.size() > 1 || G.prepared_k != 4) {
                launches += launch_chunk(G, ci, triangles, s);
                if (G.chunks.size() == 1) G.prepared_k = 4;
                G.tau_ready = G.tau_ready || triangles;
            }
            const Tile *ct = tiles;
            int64_t nct = n_tiles;
            if (whole) {
                ct = tiles + c.t0;
                nct = c.t1 - c.t0;
            } else {
                int64_t a = 0;
                while (a < n_tiles && host[a].end <= b) ++a;
                int64_t y = a;
                while (y < n_tiles && host[y].begin < e) ++y;
                ct = tiles + a;
                nct = y - a;
            }
            G.a_base = c.s0;
            G.e_base = c.e0;
            launches += launch_edges4(G, ct, nct, e_begin, per_edge_out, gacc, s);
        }
    }
    if (tmp.p) TG_CK(cudaStreamSynchronize(s));
    guard.done = true;
    return launches;
}

}  // namespace tg

// tg_host.hpp -- host-side handle and helpers of libtg (not part of the ABI).
#pragma once

#include <cstdint>
#include <cstdio>
#include <cstring>
#include <memory>
#include <type_traits>
#include <utility>
#include <vector>
#include <cuda_runtime.h>

#include "tg.h"
#include "tg_error.hpp"
#include "tg_internal.cuh"

namespace tg {

// Raises (never lowers) a kernel's dynamic shared-memory limit.  The limit
// is a process-wide attribute of the function, so handles counted
// concurrently on several host threads must not shrink it under one another.
// Defined in tg_count.cu.
void raise_smem_limit(const void *func, size_t bytes);

// Largest light_anchor_max_wedges whose per-warp hashes of k_wedge_light fit
// one CTA's shared memory for L types.  Defined in tg_wedge.cu.
int light_anchor_limit(int L);

// Stream-ordered memory pool of the current device, owned by the library
// (release threshold kept at its maximum, so freed blocks are reused instead
// of returned to the CUDA driver).  Defined in tg_build.cu.
cudaMemPool_t device_pool();

// Whether `s` is being captured into a CUDA graph.
inline bool stream_captured(cudaStream_t s) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(s, &st);
    forget(e);
    return e == cudaSuccess && st != cudaStreamCaptureStatusNone;
}

// cudaMalloc and cudaFree are refused on a thread that captures a stream
// unless it asks for them.
template <class F>
cudaError_t relaxed(F f) {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    forget(cudaThreadExchangeStreamCaptureMode(&mode));
    const cudaError_t e = f();
    forget(cudaThreadExchangeStreamCaptureMode(&mode));
    return e;
}

// Stream of a handle's last call, and whether it was captured then (asked once
// per call, not per buffer: a small build has forty of them).
struct OwnerStream {
    cudaStream_t stream = nullptr;
    bool captured = false;
    void on(cudaStream_t s) {
        stream = s;
        captured = stream_captured(s);
    }
};

// Device buffer owned by a handle; freed by release() or the destructor.
// With an owner (the handle) it is allocated and freed stream-ordered on its
// stream from the library pool, so no call synchronises the device; without
// one, and while that stream is captured, it is cudaMalloc's and cudaFree's:
// an allocation that a capture takes up has memory behind it only while the
// captured graph runs, and the handle keeps the buffer.
struct DBuf {
    void *p = nullptr;
    size_t bytes = 0;
    const OwnerStream *owner = nullptr;
    bool plain = false;         // of cudaMalloc
    DBuf() = default;
    DBuf(const DBuf &) = delete;
    DBuf &operator=(const DBuf &) = delete;
    ~DBuf() { release(); }
    void alloc(size_t b) {
        release();
        if (b == 0) b = 16;
        plain = !owner || owner->captured;
        const cudaError_t e = plain ? relaxed([&] { return cudaMalloc(&p, b); })
                                    : cudaMallocFromPoolAsync(&p, b, device_pool(), owner->stream);
        if (e != cudaSuccess) p = nullptr;
        throw_cuda(e, "device memory of the handle");
        bytes = b;
    }
    // a copy of host memory, complete on return; after an error there is no buffer
    void upload(const void *src, size_t b, cudaStream_t s) {
        alloc(b);
        cudaError_t e = b ? cudaMemcpyAsync(p, src, b, cudaMemcpyHostToDevice, s) : cudaSuccess;
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) release();
        throw_cuda(e, "upload");
    }
    // for buffers that a captured batch points to: allocated once, and never
    // replaced while the handle lives
    void alloc_once(size_t b) {
        if (!p) alloc(b);
        else if (bytes < b) throw Error{TG_ERR_INTERNAL, "working array of another size"};
    }
    void release() {
        if (p) {
            forget(plain ? relaxed([&] { return cudaFree(p); }) : cudaFreeAsync(p, owner->stream));
        }
        p = nullptr;
        bytes = 0;
    }
    template <class T> T *as() const { return static_cast<T *>(p); }
};

// Temporary device buffer of one call, stream-ordered on `st`, from the
// same library pool (which keeps freed blocks mapped for the life of the
// process instead of returning them to the CUDA driver at synchronisations).
struct TBuf {
    void *p = nullptr;
    cudaStream_t s = nullptr;
    TBuf(size_t b, cudaStream_t st) : s(st) {
        if (b == 0) b = 16;
        TG_CK(cudaMallocFromPoolAsync(&p, b, device_pool(), s));
    }
    TBuf(const TBuf &) = delete;
    TBuf &operator=(const TBuf &) = delete;
    ~TBuf() { if (p) forget(cudaFreeAsync(p, s)); }
    template <class T> T *as() const { return static_cast<T *>(p); }
};

inline bool is_device_pointer(const void *p) {
    if (!p) return false;
    cudaPointerAttributes a;
    cudaError_t e = cudaPointerGetAttributes(&a, p);
    if (e != cudaSuccess) { (void)cudaGetLastError(); return false; }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Layout of the position-aware counts (Sec. 5): per-edge blocks O1..O12
// and the classes of each global block (tg_pa.cu).
struct PaLayout {
    int32_t L = 0, S = 0;               // types, per-edge slots
    int64_t G = 0;                      // classes per graph
    int32_t off[13] = {0};              // first slot of blocks O1..O12 (index 1..12)
    int64_t bsize[9] = {0};             // classes of each global block
    int64_t boff[10] = {0};             // first class of each global block; boff[9] = G
};

struct Graph : OwnerStream {
    int device = 0;
    int32_t ngraphs = 1, L = 1;
    int64_t n = 0, nnz = 0, m = 0;
    int64_t max_degree = 0;
    bool narrow = false;                                     // kNarrowDegree (tg_internal.cuh)
    std::vector<int64_t> h_node_off, h_edge_off, h_slot_off;
    // chunks of whole graphs counted one after another (bounds the 4-cycle array)
    struct Chunk { int32_t g0, g1; int64_t n0, n1, s0, s1, e0, e1, t0, t1; };
    std::vector<Chunk> chunks;
    int64_t a_stride = 0, a_base = 0;
    tg_options opt;

    // graph (built once)
    DBuf node_off, rp, adj, toff, tdeg, pivot, ty, old_of, slot_eid, e_lo, e_hi, e_slot_lo, e_slot_hi, delta;
    DBuf most_lower;                            // most lower-priority neighbours of one type, until prepare_anchors
    DBuf plus_off, plus_adj, plus_eid;
    // nodes by |N+| (tg_local.cuh): mid, big, and larger than shared memory
    // holds; the slices of the CTAs that list triangles and of those that sum
    DBuf tri_list[3], tri_scratch, sum_scratch;
    int64_t tri_count[3] = {0, 0, 0}, max_nplus = 0;
    // work lists
    DBuf anchors[kHubClass], anchor_wedges;     // wedge anchors by class (tg_wedge.cu); wedges of every node
    int64_t n_anchors[kHubClass] = {};
    // hub anchors in (graph, type, id) order and the pieces of their wedges (tg_hub.cu)
    DBuf hubs, hub_base, hub_nlow, hub_piece;
    int64_t n_hubs = 0;
    bool anchors_ready = false;                 // delta, anchors and hubs (prepare_anchors)
    std::vector<int32_t> h_hub_id;      // hub node ids
    std::vector<int64_t> h_hub_wedges;  // wedges of each hub
    // persistent hub pass (tg_hub.cu): per chunk, its ticket queue; the
    // table buffers shared by all chunks
    struct HubPlan {
        DBuf segs, groups, ntick, ctr;
        std::vector<HubGroup> h_groups;     // host copies (kept while the uploads may be in flight)
        std::vector<HubSegment> h_segs;
        std::vector<int64_t> h_ntick;       // tickets per (group, kind)
        int64_t n_tickets = 0, n_groups = 0, n_segs = 0;
    };
    std::vector<std::unique_ptr<HubPlan>> hub_plans;
    DBuf hub_tables;
    // directed counts (tg_directed.cu): edge labels, typed out-degrees, class tables, triangle cells
    DBuf dlab, doutdeg, dcls, darcs, dgacc, dcell;
    int64_t d_global = 0;
    bool directed = false;
    // edge-typed counts (tg_edge_typed.cu): edge type per edge, per-node
    // neighbour counts by (node type, edge type), the totals' accumulator,
    // triangle cells when there are no rows to hold them
    DBuf etype, etdeg, etgacc, etcell;
    int32_t et_X = 0;
    int64_t et_global = 0;
    bool edge_typed = false;
    int64_t hub_stride = 0, hub_buf_words = 0;  // words per hub table, per buffer
    bool hub_packed = false;                    // two 16-bit counters per word
    // counting state
    DBuf C, tau, A, gacc, status, tiles_full, stage_pe, stage_gl;
    DBuf xsum, tri_any, slot_rows;
    DBuf work;                          // [kWorkSlots] work counters (tg_set_work_counting)
    bool work_on = false;
    int64_t n_tiles_full = 0, max_chunk_edges = 0;
    int64_t e_base = 0;
    int32_t prepared_k = 0;             // 0: nothing, 3: C, 4: C and the chunk's per-slot and per-edge sums
    bool tau_ready = false;             // tau of the current C
    int64_t last_launches = 0;
    // per-kernel event timing (tg_set_timing)
    bool timing = false;
    struct TimerRec { const char *name; cudaEvent_t a, b; };
    std::vector<TimerRec> timer_pending;
    std::vector<cudaEvent_t> event_pool;
    std::vector<std::pair<const char *, std::pair<double, int64_t>>> timer_totals;
    // position-aware counting (Sec. 5): slot -> class table, raw class sums
    DBuf pa_cls, pa_gacc;
    PaLayout pa;
    bool pa_active = false;             // the per-edge epilogue writes position-aware rows
    // CUDA graph of the last batched count
    cudaGraphExec_t batch_exec = nullptr;
    int32_t batch_k = 0;
    const void *batch_pe = nullptr, *batch_gl = nullptr;
    cudaStream_t batch_stream = nullptr;

    size_t node_sum_bytes() const { return narrow ? sizeof(uint32_t) : sizeof(int64_t); }   // of a delta or tau value
    GraphView view() const {
        GraphView v;
        v.ngraphs = ngraphs; v.L = L; v.n = n; v.nnz = nnz; v.m = m;
        v.node_off = node_off.as<int64_t>();
        v.rp = rp.as<int64_t>();
        v.adj = adj.as<int32_t>();
        v.toff = toff.as<int32_t>();
        v.pivot = pivot.as<int32_t>();
        v.tdeg = tdeg.as<uint32_t>();
        v.ty = ty.as<uint8_t>();
        v.slot_eid = slot_eid.as<int32_t>();
        v.e_lo = e_lo.as<int32_t>();
        v.e_hi = e_hi.as<int32_t>();
        v.e_slot_lo = e_slot_lo.as<int64_t>();
        v.e_slot_hi = e_slot_hi.as<int64_t>();
        v.delta = delta.p;
        v.narrow = narrow;
        v.plus_off = plus_off.as<int64_t>();
        v.plus_adj = plus_adj.as<int32_t>();
        v.plus_eid = plus_eid.as<int32_t>();
        return v;
    }
    CountView cview() const {
        CountView c;
        c.C = C.as<uint32_t>();
        c.tau = tau.p;
        c.A = A.as<uint32_t>();
        c.slot_rows = slot_rows.as<uint32_t>();
        c.a_base = a_base;
        c.a_stride = a_stride;
        c.e_base = e_base;
        c.xsum = xsum.as<uint32_t>();
        c.tri_any = tri_any.as<uint8_t>();
        c.gacc = gacc.as<unsigned long long>();
        c.status = status.as<uint32_t>();
        c.work = work_on ? work.as<unsigned long long>() : nullptr;
        return c;
    }
    Graph() {
        for (DBuf *b : buffers()) b->owner = this;
    }
    std::vector<DBuf *> buffers() {
        std::vector<DBuf *> v;
        for (const DBuf *b : cbuffers()) v.push_back(const_cast<DBuf *>(b));
        return v;
    }
    std::vector<const DBuf *> cbuffers() const {
        return {&node_off, &rp, &adj, &toff, &tdeg, &pivot, &ty, &old_of, &slot_eid, &e_lo, &e_hi,
                             &e_slot_lo, &e_slot_hi, &delta, &most_lower, &anchors[0], &anchors[1], &anchors[2], &anchors[3], &anchors[4],
                             &anchor_wedges, &C, &tau, &A, &gacc, &status, &tiles_full, &stage_pe,
                             &stage_gl, &xsum, &tri_any, &slot_rows, &work, &hub_tables, &dlab, &doutdeg, &dcls, &darcs, &dgacc, &dcell, &etype, &etdeg, &etgacc, &etcell, &plus_off, &plus_adj, &plus_eid, &tri_list[0], &tri_list[1], &tri_list[2], &tri_scratch, &sum_scratch, &hubs, &hub_base, &hub_nlow, &hub_piece,
                &pa_cls, &pa_gacc};
    }
    int64_t device_bytes() const {
        int64_t s = 0;
        for (const DBuf *b : cbuffers()) s += (int64_t)b->bytes;
        return s;
    }
    ~Graph() {
        if (batch_exec) forget(cudaGraphExecDestroy(batch_exec));
        for (auto &r : timer_pending) { event_pool.push_back(r.a); event_pool.push_back(r.b); }
        for (cudaEvent_t e : event_pool) forget(cudaEventDestroy(e));
    }
    cudaEvent_t take_event() {
        if (!event_pool.empty()) { cudaEvent_t e = event_pool.back(); event_pool.pop_back(); return e; }
        cudaEvent_t e;
        TG_CK(cudaEventCreate(&e));
        return e;
    }
};

// What a count leaves in the handle's working arrays (prepared_k, tau_ready)
// is recorded once the launches that make it are enqueued; a count that ends
// with an error leaves nothing that a later one may rely on.
struct CountGuard {
    Graph &G;
    bool done = false;
    explicit CountGuard(Graph &g) : G(g) {}
    ~CountGuard() {
        if (done) return;
        G.prepared_k = 0;
        G.tau_ready = false;
    }
};

// Brackets one kernel launch with events when timing is on and the stream
// is not being captured.
struct KernelTimer {
    Graph &G;
    cudaStream_t s;
    const char *name;
    cudaEvent_t a = nullptr, b = nullptr;
    KernelTimer(Graph &g, cudaStream_t st, const char *nm) : G(g), s(st), name(nm) {
        if (!G.timing) return;
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        const cudaError_t e = cudaStreamIsCapturing(s, &cs);
        forget(e);
        if (e != cudaSuccess || cs != cudaStreamCaptureStatusNone) return;
        a = G.take_event();
        b = G.take_event();
        TG_CK(cudaEventRecord(a, s));
    }
    ~KernelTimer() {
        if (!a) return;
        const cudaError_t e = cudaEventRecord(b, s);
        if (e == cudaSuccess) G.timer_pending.push_back(Graph::TimerRec{name, a, b});
        else forget(e);
    }
};

inline void fill_defaults(tg_options *o) {
    std::memset(o, 0, sizeof(*o));
    o->light_edge_max_degree = 256;
    o->light_anchor_max_wedges = 64;
    o->anchor_table_budget_mb = 12288;
    o->ctas_per_sm = 3;
    o->cycle_budget_mb = 16384;
    o->hub_min_wedges = 1 << 14;
    o->hub_l2_mb = 192;
}

// number of SMs of the current device
int sm_count();

// build entry (tg_build.cu)
void build_graph(Graph &G, int32_t ngraphs, const int64_t *node_off_host, int64_t n, int64_t nnz,
                 const int64_t *row_ptr, const int32_t *col, const uint8_t *types, int32_t L,
                 const tg_options &opt, cudaStream_t s);

// One class of nodes u by |N+(u)| and its launch shape (tg_local.cuh).
struct LocalClass {
    int64_t n;                  // nodes
    const int32_t *list;
    int threads, cap, lgf;      // CTA size, list capacity, log2 bits of the id filter
};
LocalClass local_class(const Graph &G, int cls);

// out[x][t][q] = sums of rows[index[s]][q] over x's slots s of type t
int64_t launch_row_sums(Graph &G, const int32_t *index, const uint32_t *rows, void *out, cudaStream_t s);
// shared-memory limits and scratch of launch_triangles (before any capture)
void prepare_triangles(Graph &G);
// G.tri_scratch, of one size whichever kernels list the triangles
void prepare_tri_scratch(Graph &G);
// typed triangles per edge and, with_tau, the per-node sums of the whole
// graph (tg_triangles.cu); returns the kernel launches
int64_t launch_triangles(Graph &G, bool with_tau, cudaStream_t s);

// sums over the triangle nodes and 4-cliques of the edges [e0, e1) of whole
// graphs with nodes [n0, n1) (tg_sums.cu); prepare_sums before any capture
void prepare_sums(Graph &G);
int64_t launch_sums(Graph &G, int64_t n0, int64_t n1, int64_t e0, int64_t e1, cudaStream_t s);

// the hub anchors (tg_hub.cu): groups, items and ticket queues (before any
// capture), and the pass over the hubs of chunk ci
void prepare_hubs(Graph &G, cudaStream_t s);
int64_t launch_hubs(Graph &G, size_t ci, cudaStream_t s);

// f(std::integral_constant<int, L>) for the handle's L
template <class F>
void with_types(int L, F f) {
    switch (L) {
        case 1: f(std::integral_constant<int, 1>()); break;
        case 2: f(std::integral_constant<int, 2>()); break;
        case 3: f(std::integral_constant<int, 3>()); break;
        case 4: f(std::integral_constant<int, 4>()); break;
        case 5: f(std::integral_constant<int, 5>()); break;
        case 6: f(std::integral_constant<int, 6>()); break;
        case 7: f(std::integral_constant<int, 7>()); break;
        default: f(std::integral_constant<int, 8>()); break;
    }
}

// wedge anchors (tg_wedge.cu): class lists from the wedges and the most
// lower-priority neighbours of one type of every node (the hubs unsorted);
// the wedge pass of the anchors of [n0, n1) in the forms form_lo to form_hi
void prepare_anchors(Graph &G, cudaStream_t s);          // tg_build.cu, before any capture
void list_anchors(Graph &G, const int64_t *work, const int32_t *most, cudaStream_t s);
void prepare_wedges(Graph &G);
int64_t launch_anchor_wedges(Graph &G, int form_lo, int form_hi, int64_t n0, int64_t n1, cudaStream_t s);

// count entries (tg_count.cu)
void prepare_counting(Graph &G, int k, cudaStream_t s);
void prepare_edges(Graph &G, int k, cudaStream_t s);
// Runs the counting stages for edges [e_begin, e_end) into per_edge_out
// (row 0 = e_begin) and the raw sums gacc.  full: the whole graph, every
// stage recomputed (no cached state).  Returns the kernel launches.
int64_t run_count(Graph &G, int k, int64_t e_begin, int64_t e_end, uint32_t *per_edge_out,
                  unsigned long long *gacc, bool full, cudaStream_t s);
// edges per tile of the per-edge kernels (tg_count.cu)
int64_t tile_edges(const Graph &G);

// rows and raw sums of the edges of the tiles (tg_epi.cu)
void prepare_epi(Graph &G);
int64_t launch_edges3(Graph &G, const Tile *tiles, int64_t n_tiles, int64_t e_begin, uint32_t *per_edge_out,
                      unsigned long long *gacc, cudaStream_t s);
// the per-slot 4-cycle planes of a chunk as rows, one per slot
int64_t launch_slot_rows(Graph &G, int64_t n_slots, cudaStream_t s);
int64_t launch_edges4(Graph &G, const Tile *tiles, int64_t n_tiles, int64_t row_base, uint32_t *per_edge_out,
                      unsigned long long *gacc, cudaStream_t s);
int64_t launch_finalize(Graph &G, int k, int64_t *global_out, cudaStream_t s);
// Position-aware typed graphlets (tg_pa.cu; epilogue in tg_epi.cu).
PaLayout pa_layout(int L);
bool pa_labelling(int L, int block, int64_t rank, int32_t *labelling);
std::vector<int32_t> pa_class_table(const PaLayout &Y);
void prepare_position_aware(Graph &G, cudaStream_t s);
void prepare_epi4_pa(Graph &G);
int64_t launch_finalize_pa(Graph &G, int64_t *global_out, cudaStream_t s);
// Typed-graphlet weighted graph (tg_weights.cu).
void launch_weights(Graph &G, int k, const uint32_t *rows, int block, int64_t rank, int64_t *weights,
                    int64_t *degree, cudaStream_t s);
// Directed typed 3-node graphlets (tg_directed.cu).
int64_t directed_classes(int L);
bool directed_class_code(int L, int64_t rank, int32_t *types3, int32_t *arcs3);
void symmetrize_arcs(int64_t n, int64_t na, const int64_t *orp, const int32_t *ocol, int64_t *srp, int32_t *scol,
                     int32_t *src, cudaStream_t s);
void prepare_directed(Graph &G, int64_t na, const int32_t *src, const int32_t *ocol, cudaStream_t s);
int64_t run_directed3(Graph &G, uint32_t *per_edge_out, int64_t *global_out, cudaStream_t s);
// Edge-typed 3-node graphlets (tg_edge_typed.cu).
int64_t edge_typed_global_slots(int L, int X);
void prepare_edge_typed(Graph &G, int X, const int64_t *row_ptr, const int32_t *col, const uint8_t *edge_types,
                        cudaStream_t s);
int64_t run_edge_typed3(Graph &G, uint32_t *per_edge_out, int64_t *global_out, cudaStream_t s);
// Sparse per-edge counts (tg_sparse.cu): returns the number of nonzero
// pairs; writes them only while they fit `cap` (fits = false otherwise).
int64_t count_sparse(Graph &G, int k, int64_t *row_off, uint16_t *slot, uint32_t *value, int64_t cap, bool &fits,
                     cudaStream_t s);

}  // namespace tg

struct tg_graph {
    tg::Graph g;
};

// tg_wedge.cu -- the 4-cycle wedges of the anchors that are not hubs.
//
// For an anchor u, V_u = {v in Gamma_u : v < u} and, for v in V_u, the wedge
// ends {w in Gamma_v : w < u}.  Phase 0 counts, per wedge end w and per type
// t of the middle node, the wedges u - v - w (counters h_u[w][t]).  Phase 1
// revisits every wedge u - v - w: the other middles x of (u,w) of type t
// number h_u[w][t] - [phi_v = t]; each closes the 4-cycle u - v - w - x - u,
// which is recorded on
//   slot (v -> w): A[phi_u][t]   (v's other cycle neighbour u, w's is x)
//   slot (u -> v): A[t][phi_w]   (u's other cycle neighbour x, v's is w).
// A[s][t] of a slot (a -> b) counts 4-cycles a - b - y - z - a with
// phi_z = s (a's other neighbour) and phi_y = t (b's other neighbour).
//
// One group of threads per anchor: a warp, or a CTA of 64 to 1,024 threads
// by the size of its table.  The group first finds every run -- the part
// below u of v's type-t segment, one (v, t) per thread, all binary searches
// at once -- and a prefix over their lengths; then it walks the wedges of all
// runs as one list, a wedge per thread.  The counters live in a hash in
// shared memory whose size follows the anchor's wedges W (2 W slots where
// they fit; the ends of power-law anchors are almost all distinct).  A
// counter is at most the number of u's lower neighbours of its type, so all
// types of one end share one 32-bit word when that fits (L = 5: 63 per type),
// else two or four words.
//
// Measured against a hash of L 32-bit counters per end, cleared at full size
// per anchor, with a binary search per (v, t) and phase in sequence, and
// dense tables in HBM above 3,072 wedges: 30 M block-model edges 87.5 -> 26.5
// ms, 20 M Chung-Lu edges 18.6 -> 9.7 ms, 256 dense graphs 24.0 -> 8.1 ms.
// What it took, on the block model: the new tables with a search and a lookup
// per wedge and phase 54 ms; with the slot of every wedge kept (phase 1 reads
// its counter at once, and a wedge that is alone at its end stops there) and
// the runs followed instead of searched 26.5 ms; compiled to 56 registers
// since the insert is bounded 23.3 ms (six CTAs of 192 threads fit an SM, as
// launched; five did at 64: 6.0 -> 3.4 ms; Chung-Lu edges 8.6, dense graphs
// 7.3).  Bound now: instructions of
// the inserts (probes diverge) and the barriers between an anchor's phases.
#include <algorithm>

#include "tg_host.hpp"

namespace tg {

namespace {

// ------------------------------------------------------------ classes
// Threads per anchor, entries of the run list (entries beyond it are walked
// in chunks), and bytes of the table (the warp form's follow the option).
template <int kForm> struct Form;
template <> struct Form<0> { static constexpr int threads = 32, groups = 4, runs = 160; };
template <> struct Form<1> { static constexpr int threads = 64, groups = 1, runs = 256; };
template <> struct Form<2> { static constexpr int threads = 192, groups = 1, runs = 384; };
template <> struct Form<3> { static constexpr int threads = 512, groups = 1, runs = 1024; };
template <> struct Form<4> { static constexpr int threads = 1024, groups = 1, runs = 1536; };

template <int kForm>
__host__ __device__ constexpr size_t run_bytes() {          // start, off, sv, tv of Runs
    return (size_t)Form<kForm>::runs * 13 + 16;
}

template <int T>
__device__ __forceinline__ void group_sync() {
    if (T > 32) __syncthreads(); else __syncwarp();
}

// exclusive prefix of one value per thread over the group; total to all
template <int T>
__device__ __forceinline__ int32_t group_scan(int32_t v, int32_t *warp_tot, int32_t &total) {
    const int lane = threadIdx.x & 31;
    int32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (T == 32) {
        total = __shfl_sync(0xffffffffu, inc, 31);
        return inc - v;
    }
    const int wid = threadIdx.x >> 5;
    if (lane == 31) warp_tot[wid] = inc;
    __syncthreads();
    const int32_t mine = lane < T / 32 ? warp_tot[lane] : 0;
    int32_t run = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, run, o);
        if (lane >= o) run += y;
    }
    total = __shfl_sync(0xffffffffu, run, 31);
    const int32_t base = __shfl_sync(0xffffffffu, run - mine, wid);
    __syncthreads();                                        // warp_tot may be written again
    return base + inc - v;
}

constexpr int kWalkLanes = 8;               // lanes that walk one contiguous part of the wedges

// per-run sums of phase 1 over each kWalkLanes lanes (equal keys are
// contiguous): tail lanes add them to the 4-cycle slot of (u, v)
__device__ __forceinline__ void flush_runs(uint32_t *A, int64_t nnz, int L, const uint32_t *c, int key, int tw,
                                           int64_t sv, int lane) {
    const int sub = lane & (kWalkLanes - 1);
    unsigned same = 0;
#pragma unroll
    for (int s = 0; (1 << s) < kWalkLanes; ++s) {
        const int kk = __shfl_up_sync(0xffffffffu, key, 1 << s, kWalkLanes);
        if (sub >= (1 << s) && kk == key) same |= 1u << s;
    }
    const int knext = __shfl_down_sync(0xffffffffu, key, 1, kWalkLanes);
    const bool tail = key >= 0 && (sub == kWalkLanes - 1 || knext != key);
#pragma unroll
    for (int t = 0; t < kMaxL; ++t) {
        if (t >= L) break;
        uint32_t v = c[t];
#pragma unroll
        for (int s = 0; (1 << s) < kWalkLanes; ++s) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, v, 1 << s, kWalkLanes);
            if (same & (1u << s)) v += y;
        }
        if (tail && v) atomicAdd(&A[(int64_t)(t * L + tw) * nnz + sv], v);
    }
}

// The run list of one anchor (or of a chunk of its lower neighbours).
struct Runs {
    uint32_t *start;            // [runs] first adjacency slot
    int32_t *off;               // [runs + 1] first wedge
    uint32_t *sv;               // [runs / L] slot of v in u's row
    uint8_t *tv;                // [runs / L] v's type
};

struct Table {
    uint32_t *keys, *cnt;
    uint16_t *slot;             // [wedges] the slot of every wedge's end
    uint32_t cap;
    Pack pk;
    uint32_t *status;
};

// the slot of w, inserted if new (a free slot exists: cap >= the wedges,
// anchor_pack and slots_for; a full table would be reported, not probed on)
__device__ __forceinline__ uint32_t table_insert(const Table &tb, uint32_t w) {
    const uint32_t h0 = __umulhi(w * 2654435761u, tb.cap);
    uint32_t h = h0;
    for (;;) {
        uint32_t k = *(volatile uint32_t *)&tb.keys[h];
        if (k == 0xffffffffu) k = atomicCAS(&tb.keys[h], 0xffffffffu, w);
        if (k == 0xffffffffu || k == w) return h;
        h = h + 1 == tb.cap ? 0 : h + 1;
        if (h == h0) {
            set_status(tb.status, ST_INTERNAL);
            return h;
        }
    }
}

// One phase over the wedges of the listed runs (n entries, `total` wedges,
// the first one number x_base of the anchor).  Eight lanes take a contiguous
// part of the wedges, eight at a time, so each lane's run only moves on (a
// search per wedge cost more than the rest of the phase).
template <int T, int kRw, bool kFill>
__device__ __forceinline__ void walk(const GraphView &g, uint32_t *A, int64_t nnz, int tu, const Runs &r, int n,
                                     int32_t total, int32_t x_base, const Table &tb, int tid) {
    const int L = g.L;
    const int lane = threadIdx.x & 31;
    constexpr int kParts = T / kWalkLanes;
    const int32_t part = (total + kParts * kWalkLanes - 1) / (kParts * kWalkLanes) * kWalkLanes;
    const int32_t xb = (tid / kWalkLanes) * part, xe = min(total, xb + part);
    int32_t x = xb + (tid & (kWalkLanes - 1));
    int j = 0;                                              // last entry with off <= x
    if (x < xe) {
        int hi = n;
        while (hi - j > 1) {
            const int mid = (j + hi) >> 1;
            if (r.off[mid] <= x) j = mid; else hi = mid;
        }
    }
    const uint32_t inv = (65536u + L - 1) / L;              // j / L for j < 2048
    uint32_t low = 0;                                       // (kRw = 1) bit 0 of every type's field
    for (int t = 0; t < tb.pk.F; ++t) low |= 1u << (tb.pk.bits * t);
    for (int32_t step = 0; step < part; step += kWalkLanes, x += kWalkLanes) {   // group-uniform trip count
        const bool act = x < xe;
        if (act)
            while (r.off[j + 1] <= x) ++j;                  // off[n] = total > x
        if (kFill) {
            if (act) {
                const uint32_t w = (uint32_t)__ldg(g.adj + r.start[j] + (x - r.off[j]));
                const uint32_t h = table_insert(tb, w);
                tb.slot[x_base + x] = (uint16_t)h;
                const int tv = r.tv[(j * inv) >> 16];
                const int k = kRw == 1 ? 0 : kRw == 2 ? (tv >= tb.pk.F ? 1 : 0) : tv >> 1;
                atomicAdd(&tb.cnt[h * kRw + k], 1u << (tb.pk.bits * (tv - k * tb.pk.F)));
            }
        } else {
            uint32_t c[kMaxL];
#pragma unroll
            for (int t = 0; t < kMaxL; ++t) c[t] = 0;
            uint32_t any = 0;
            if (act) {
                const uint32_t h = tb.slot[x_base + x];
                uint32_t word[kRw];
                int ones = 0;
                uint32_t rest = 0;
#pragma unroll
                for (int k = 0; k < kRw; ++k) {
                    word[k] = tb.cnt[h * kRw + k];
                    ones += __popc(word[k]);
                    rest |= word[k] & ~low;
                }
                if (ones != 1 || rest) {                    // (else this wedge alone: it closes nothing)
                    const int tv = r.tv[(j * inv) >> 16];
                    const int64_t pos = (int64_t)r.start[j] + (x - r.off[j]);
                    const uint32_t mask = tb.pk.bits == 32 ? 0xffffffffu : (1u << tb.pk.bits) - 1u;
                    int f = 0, k = 0;
#pragma unroll
                    for (int t = 0; t < kMaxL; ++t) {
                        if (t >= L) break;
                        uint32_t wd = word[0];
#pragma unroll
                        for (int y = 1; y < kRw; ++y) wd = k == y ? word[y] : wd;
                        const uint32_t v = ((wd >> (tb.pk.bits * f)) & mask) - (t == tv ? 1u : 0u);
                        if (++f == tb.pk.F) { f = 0; ++k; }
                        c[t] = v;
                        any |= v;
                        if (v) atomicAdd(&A[(int64_t)(tu * L + t) * nnz + pos], v);
                    }
                }
            }
            if (__any_sync(0xffffffffu, any != 0)) {
                const int kv = (int)((j * inv) >> 16);      // (of every lane: a run's last lane adds its sums)
                flush_runs(A, nnz, L, c, act ? j : -1, j - kv * L, r.sv[kv], lane);
            }
        }
    }
}

template <int T, bool kFill>
__device__ __forceinline__ void walk_rw(const GraphView &g, uint32_t *A, int64_t nnz, int tu, const Runs &r, int n,
                                        int32_t total, int32_t x_base, const Table &tb, int tid) {
    if (tb.pk.rw == 1) walk<T, 1, kFill>(g, A, nnz, tu, r, n, total, x_base, tb, tid);
    else if (tb.pk.rw == 2) walk<T, 2, kFill>(g, A, nnz, tu, r, n, total, x_base, tb, tid);
    else walk<T, 4, kFill>(g, A, nnz, tu, r, n, total, x_base, tb, tid);
}

template <int kForm>
__global__ void __launch_bounds__(Form<kForm>::threads * Form<kForm>::groups)
    k_wedge(GraphView g, CountView cv, const int32_t *__restrict__ anchors, int64_t n_anchors,
            const int32_t *__restrict__ wedges, int64_t table_bytes, int64_t n0, int64_t n1) {
    using F = Form<kForm>;
    constexpr int T = F::threads;
    extern __shared__ uint32_t wsm[];
    __shared__ int32_t warp_tot[32];
    const int L = g.L;
    const int lane = threadIdx.x & 31, tid = threadIdx.x % T, grp = threadIdx.x / T;
    uint32_t *mem = wsm + grp * ((table_bytes + run_bytes<kForm>()) / 4);
    Runs r;
    r.start = mem + table_bytes / 4;
    r.off = reinterpret_cast<int32_t *>(r.start + F::runs);
    r.sv = reinterpret_cast<uint32_t *>(r.off + F::runs + 2);
    r.tv = reinterpret_cast<uint8_t *>(r.sv + F::runs);
    const int64_t nnz = cv.a_stride;
    uint32_t *A = cv.A - cv.a_base;                         // indexed by absolute slot
    const int vmax = F::runs / L;                           // lower neighbours per chunk
    for (int64_t a = (int64_t)blockIdx.x * F::groups + grp; a < n_anchors; a += (int64_t)gridDim.x * F::groups) {
        const int32_t u = anchors[a];
        if (u < n0 || u >= n1) continue;                    // anchor outside this chunk (uniform over the group)
        const int tu = g.ty[u];
        // u's lower neighbours by type: lane t < L its first slot, their number before it
        int32_t nt = 0;
        int64_t ub = 0;
        if (lane < L) {
            int64_t cut;
            seg_prefix(g, u, lane, u, ub, cut);
            nt = (int32_t)(cut - ub);
        }
        int32_t inc = nt;
#pragma unroll
        for (int o = 1; o < kMaxL; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        const int32_t uoff = inc - nt;
        const int32_t nV = __shfl_sync(0xffffffffu, inc, kMaxL - 1);
        const int32_t most = (int32_t)__reduce_max_sync(0xffffffffu, (unsigned)nt);
        Table tb;
        tb.pk = anchor_pack(L, wedges[u], most);
        tb.cap = (uint32_t)slots_for(wedges[u], table_bytes, tb.pk.rw);
        tb.status = cv.status;
        tb.keys = mem;
        tb.cnt = mem + tb.cap;
        tb.slot = reinterpret_cast<uint16_t *>(tb.cnt + (size_t)tb.cap * tb.pk.rw);
        group_sync<T>();                                    // the previous anchor's table is read
        for (uint32_t k = tid; k < tb.cap; k += T) tb.keys[k] = 0xffffffffu;
        for (uint32_t k = tid; k < tb.cap * tb.pk.rw; k += T) tb.cnt[k] = 0u;
        const int chunks = (nV + vmax - 1) / vmax;
        for (int phase = 0; phase < 2; ++phase) {
            int32_t x_base = 0;
            for (int ch = 0; ch < chunks; ++ch) {
                const int v0 = ch * vmax, nv = min(vmax, nV - v0), n = nv * L;
                if (phase == 0 || chunks > 1) {             // the runs of lower neighbours v0 .. v0 + nv - 1
                    if (chunks > 1) group_sync<T>();
                    int32_t run = 0;
                    for (int j0 = 0; j0 < n; j0 += T) {
                        const int j = j0 + tid;
                        const int kv = min(j, n - 1) / L, tw = j - kv * L;
                        int tv = 0;                         // (all lanes: shuffles)
#pragma unroll
                        for (int st = kMaxL / 2; st > 0; st >>= 1) {
                            const int32_t c = __shfl_sync(0xffffffffu, uoff, tv + st);
                            if (c <= v0 + kv) tv += st;
                        }
                        const int64_t sv = __shfl_sync(0xffffffffu, ub, tv) +
                                           (v0 + kv - __shfl_sync(0xffffffffu, uoff, tv));
                        int32_t len = 0;
                        if (j < n) {
                            int64_t b, cut;
                            seg_prefix(g, g.adj[sv], tw, u, b, cut);
                            len = (int32_t)(cut - b);
                            r.start[j] = (uint32_t)b;
                            if (tw == 0) {
                                r.sv[kv] = (uint32_t)sv;
                                r.tv[kv] = (uint8_t)tv;
                            }
                        }
                        int32_t tot;
                        const int32_t at = run + group_scan<T>(len, warp_tot, tot);
                        if (j < n) r.off[j] = at;
                        run += tot;
                    }
                    if (tid == 0) r.off[n] = run;
                }
                group_sync<T>();
                const int32_t total = r.off[n];
                if (phase == 0) walk_rw<T, true>(g, A, nnz, tu, r, n, total, x_base, tb, tid);
                else walk_rw<T, false>(g, A, nnz, tu, r, n, total, x_base, tb, tid);
                x_base += total;
            }
            group_sync<T>();
        }
    }
}

template <int kForm>
size_t form_bytes(int64_t table_bytes) {
    return Form<kForm>::groups * ((size_t)table_bytes + run_bytes<kForm>());
}

}  // namespace

int light_anchor_limit(int L) {
    int dev = 0, optin = 0;
    TG_CK(cudaGetDevice(&dev));
    TG_CK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    int w = 1;
    while (form_bytes<0>(light_bytes(L, 2 * w)) + 1024 <= (size_t)optin) w *= 2;
    return w;
}

WedgeLimits wedge_limits(const Graph &G) {
    WedgeLimits w;
    w.light = G.opt.light_anchor_max_wedges;
    w.hub = G.opt.hub_min_wedges;
    for (int f = 1; f < kHubClass; ++f) w.bytes[f - 1] = kFormBytes[f];
    return w;
}

static int64_t table_bytes_of(const Graph &G, int form) {
    return form == 0 ? light_bytes(G.L, G.opt.light_anchor_max_wedges) : kFormBytes[form];
}

template <class Fn>
static void each_form(const Graph &G, Fn f) {
    auto one = [&](auto form) {
        constexpr int kForm = decltype(form)::value;
        if (G.n_anchors[kForm] > 0) f(form, table_bytes_of(G, kForm), form_bytes<kForm>(table_bytes_of(G, kForm)));
    };
    one(std::integral_constant<int, 4>());                  // the largest anchors first
    one(std::integral_constant<int, 3>());
    one(std::integral_constant<int, 2>());
    one(std::integral_constant<int, 1>());
    one(std::integral_constant<int, 0>());
}

void prepare_wedges(Graph &G) {
    each_form(G, [&](auto form, int64_t, size_t smem) {
        raise_smem_limit((const void *)k_wedge<decltype(form)::value>, smem);
    });
}

int64_t launch_anchor_wedges(Graph &G, int form_lo, int form_hi, int64_t n0, int64_t n1, cudaStream_t s) {
    const GraphView gv = G.view();
    const CountView cv = G.cview();
    int64_t launches = 0;
    each_form(G, [&](auto form, int64_t table, size_t smem) {
        constexpr int kForm = decltype(form)::value;
        using F = Form<kForm>;
        if (kForm < form_lo || kForm > form_hi) return;
        static const char *names[5] = {"k_wedge_light", "k_wedge_64", "k_wedge_192", "k_wedge_512", "k_wedge_1024"};
        KernelTimer kt(G, s, names[kForm]);
        const int per_sm = std::max(1, std::min<int>(2048 / (F::threads * F::groups), (int)((226u << 10) / (smem + 1280))));
        const int64_t blocks = (G.n_anchors[kForm] + F::groups - 1) / F::groups;
        k_wedge<kForm><<<(unsigned)std::min<int64_t>(blocks, (int64_t)sm_count() * per_sm), F::threads * F::groups, smem, s>>>(
            gv, cv, G.anchors[kForm].as<int32_t>(), G.n_anchors[kForm], G.anchor_wedges.as<int32_t>(), table, n0, n1);
        ++launches;
    });
    TG_CK(cudaGetLastError());
    return launches;
}

// thread per node: class lists, their lengths (warp-aggregated counters), and
// the wedge counts the tables are sized by
__global__ void k_anchor_lists(int64_t n, int L, WedgeLimits lim, const int64_t *__restrict__ work,
                               const int32_t *__restrict__ most, int32_t *l0, int32_t *l1, int32_t *l2, int32_t *l3,
                               int32_t *l4, int32_t *hubs, unsigned long long *counts, int32_t *wedges) {
    const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    int cls = -1;
    if (x < n) {
        const int64_t W = work[x];
        cls = wedge_class(lim, L, W, most[x]);
        wedges[x] = (int32_t)min(W, (int64_t)INT32_MAX);
    }
#pragma unroll
    for (int c = 0; c <= kHubClass; ++c) {
        const unsigned b = __ballot_sync(0xffffffffu, cls == c);
        if (b == 0) continue;
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(&counts[c], (unsigned long long)__popc(b));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(b & ((1u << lane) - 1u));
        if (cls == c) (c == 0 ? l0 : c == 1 ? l1 : c == 2 ? l2 : c == 3 ? l3 : c == 4 ? l4 : hubs)[at] = (int32_t)x;
    }
}

void list_anchors(Graph &G, const int64_t *work, const int32_t *most, cudaStream_t s) {
    const int64_t n = G.n;
    const WedgeLimits lim = wedge_limits(G);
    TBuf counts(sizeof(unsigned long long) * (kHubClass + 1), s);
    TG_CK(cudaMemsetAsync(counts.p, 0, sizeof(unsigned long long) * (kHubClass + 1), s));
    G.anchor_wedges.alloc(sizeof(int32_t) * std::max<int64_t>(n, 1));
    for (int c = 0; c < kHubClass; ++c) G.anchors[c].alloc(sizeof(int32_t) * std::max<int64_t>(n, 1));
    G.hubs.alloc(sizeof(int32_t) * std::max<int64_t>(n, 1));
    if (n > 0) {
        k_anchor_lists<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(
            n, G.L, lim, work, most, G.anchors[0].as<int32_t>(), G.anchors[1].as<int32_t>(), G.anchors[2].as<int32_t>(),
            G.anchors[3].as<int32_t>(), G.anchors[4].as<int32_t>(), G.hubs.as<int32_t>(), counts.as<unsigned long long>(),
            G.anchor_wedges.as<int32_t>());
        TG_CK(cudaGetLastError());
    }
    unsigned long long h[kHubClass + 1];
    TG_CK(cudaMemcpyAsync(h, counts.p, sizeof(h), cudaMemcpyDeviceToHost, s));
    TG_CK(cudaStreamSynchronize(s));
    for (int c = 0; c < kHubClass; ++c) G.n_anchors[c] = (int64_t)h[c];
    G.n_hubs = (int64_t)h[kHubClass];
}

}  // namespace tg

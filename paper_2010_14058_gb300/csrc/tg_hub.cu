// tg_hub.cu -- the 4-cycle wedges of the hub anchors.
//
// An anchor u with very many wedges u - v - w (v, w of lower priority than u)
// is a hub: its counters h_u[w][t] (tg_wedge.cu) live in a node table in
// global memory, and all CTAs work on the wedges of the same few hubs so that
// the tables stay in L2.
//
// The work of a hub u is cut into pieces: a piece is one neighbour v of u
// below it and, for every type, up to kPart consecutive ends of v's row below
// u.  One warp works on a piece.  Its record (the slot of (u, v), and per
// type the first slot and the number of ends) is loaded by the lanes in one
// access, the next piece's while the current one is worked on, and the ends
// of all types are loaded together and then visited together, so a piece
// waits for two dependent accesses (ends, counters) however many runs it has.
// Within one type's 32 ends everything but the end is uniform.
// What decides its speed (20 M-edge Chung-Lu graph, 2.9e9 wedges): a walk over
// runs flattened to 32 wedges a step, with shuffles to find each lane's run
// and segmented sums, issued 740 warp instructions per 32 wedges and took
// 116 ms; pieces of 512 / 256 / 128 / 64 / 32 ends per type with groups of
// 2^22 wedges 137 / 123 / 115 / 110 / 117 ms (a warp's piece must be short
// beside a phase of its group), 64 with groups of 2^24 wedges 103, and five
// CTAs per SM 96 ms.  Of that, adding to the slots of (v, w) costs 27 ms, the
// fill's atomics 36 (their tables share L2 with the slots: 14.5 ms at the rate
// of random atomics that hit L2), reading the tables 18, the sums for (u, v) 6.
//
// The pass is one persistent launch over a ticket queue (below): per group,
// phase 0 fills the counters, phase 1 reads them, phase 2 clears them.
#include <algorithm>
#include <climits>
#include <vector>

#include <cub/device/device_scan.cuh>

#include "tg_host.hpp"

namespace tg {

namespace {

constexpr int kHubThreads = 256;
constexpr int kHubCtasPerSm = 5;                            // k_wedge_hub's launch bounds
constexpr int kPart = 64;                                  // most ends of one type in a piece

// record of a piece: [0] slot of (u, v), [1] hub << 4 | type of v, then per
// type its first end's slot and the number of ends
__host__ __device__ constexpr int piece_words(int L) { return 2 + 2 * L; }

struct HubView {
    const int32_t *hubs;        // hub node ids
    const int64_t *hub_base;    // first node of each hub's graph
    const int32_t *hub_nlow;    // nodes of each hub's graph with one-word rows
    const uint32_t *piece;      // [pieces][piece_words(L)]
};

// Table rows.  A counter h_u[w][t] is at most d_w^t, so a node w of degree
// below 2^(32 / L) has all its types in one word; the nodes of a graph are
// in degree order, so these are a prefix of its ids (L = 5: degree 63 and
// less, 96% of a Chung-Lu graph of average degree 20), and its table is a
// third of one with 16-bit counters throughout.
__host__ __device__ __forceinline__ int low_bits(int L) { return 32 / L; }

// thread per hub: its graph's first node and low nodes, its lower neighbours
__global__ void k_hub_info(GraphView g, const int32_t *__restrict__ hubs, int64_t n_hubs, int64_t *hub_base,
                           int32_t *hub_nlow, int64_t *nv) {
    const int64_t h = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (h > n_hubs) return;
    if (h == n_hubs) { nv[h] = 0; return; }
    const int32_t u = hubs[h];
    const int gr = graph_of_node(g, u);
    const int64_t base = g.node_off[gr];
    hub_base[h] = base;
    int64_t lo = base, hi = g.node_off[gr + 1];             // first node whose degree has no room in a field
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if ((g.rp[mid + 1] - g.rp[mid]) >> low_bits(g.L)) hi = mid; else lo = mid + 1;
    }
    hub_nlow[h] = (int32_t)(lo - base);
    int64_t acc = 0;
    for (int t = 0; t < g.L; ++t) {
        int64_t b, cut;
        seg_prefix(g, u, t, u, b, cut);
        acc += cut - b;
    }
    nv[h] = acc;
}

// pair x = lower neighbour number kv of hub h -> (slot of v in u's row, its type)
__device__ __forceinline__ int64_t pair_slot(const GraphView &g, int32_t u, int64_t kv, int &tv) {
    for (tv = 0; tv < g.L; ++tv) {
        int64_t b, cut;
        seg_prefix(g, u, tv, u, b, cut);
        if (kv < cut - b) return b + kv;
        kv -= cut - b;
    }
    return -1;                                              // (not reached: kv is below their number)
}

// Eight lanes per (hub, lower neighbour) pair, lane t on type t.  Counts the
// pair's pieces, or (kFill) writes them at first[pair].
template <bool kFill>
__global__ void __launch_bounds__(256) k_hub_pieces(GraphView g, const int32_t *__restrict__ hubs, int64_t n_hubs,
                                                    const int64_t *__restrict__ vbase, int64_t n_pairs, int64_t *count,
                                                    const int64_t *__restrict__ first, uint32_t *piece) {
    const int L = g.L;
    const int64_t x = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3;
    const int t = threadIdx.x & 7;
    const unsigned mask = __ballot_sync(0xffffffffu, x < n_pairs);
    if (x >= n_pairs) return;
    int64_t lo = 0, hi = n_hubs;                            // vbase[lo] <= x < vbase[hi]
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (vbase[mid] <= x) lo = mid; else hi = mid;
    }
    const int32_t u = hubs[lo];
    int tv;
    const int64_t sv = pair_slot(g, u, x - vbase[lo], tv);
    int64_t b = 0, cut = 0;
    if (t < L) seg_prefix(g, g.adj[sv], t, u, b, cut);
    const int32_t len = (int32_t)(cut - b);
    int32_t most = len;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) most = max(most, __shfl_xor_sync(mask, most, o, 8));
    const int32_t n = (most + kPart - 1) / kPart;
    if (!kFill) {
        if (t == 0) count[x] = n;
        return;
    }
    uint32_t *r = piece + first[x] * piece_words(L);
    for (int32_t k = 0; k < n; ++k, r += piece_words(L)) {
        if (t == 0) {
            r[0] = (uint32_t)sv;
            r[1] = (uint32_t)lo << 4 | (uint32_t)tv;
        }
        if (t < L) {
            const int32_t rest = len - k * kPart;
            r[2 + 2 * t] = (uint32_t)(b + (rest > 0 ? (int64_t)k * kPart : 0));
            r[3 + 2 * t] = (uint32_t)min(max(rest, 0), kPart);
        }
    }
}

// first piece of every hub
__global__ void k_hub_bounds(int64_t n_hubs, const int64_t *__restrict__ vbase, const int64_t *__restrict__ first,
                             int64_t *hub_piece) {
    const int64_t h = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (h <= n_hubs) hub_piece[h] = first[vbase[h]];
}

// One phase over the pieces [x0, x1) of one group (hub h's table at tbl +
// (h - h0) * stride), taken by the CTA's warps from the shared counter
// `next`.  Counters: one word per low node (above); for the others kPacked =
// two 16-bit counters per 32-bit word (types 2k and 2k+1; every count is at
// most the hub's degree, below 2^16 when this layout is chosen), else one
// word per type.  The tables are read and cleared at L2 (ld/st.cg): other
// CTAs of the same launch update them, so no L1 copy may be trusted.
template <int L, bool kPacked, bool kCount, int kPhase>
__device__ __forceinline__ void hub_pieces(const GraphView &g, const CountView &cv, const HubView &hv, int32_t h0,
                                           int64_t x0, int64_t x1, uint32_t *tbl, int64_t stride, int *next, uint32_t *s_rec,
                                           int lane) {
    constexpr int RW = kPacked ? (L + 1) / 2 : L;           // words per row of a node that is not low
    constexpr int lb = 32 / L;                              // bits per type in a low node's word
    constexpr uint32_t lm = lb == 32 ? 0xffffffffu : (1u << (lb & 31)) - 1u;
    constexpr int PW = piece_words(L);
    constexpr int kBatch = L <= 4 || kPhase != 1 ? L : (L + 1) / 2;   // types whose ends are in flight together
    const int64_t nnz = cv.a_stride;
    uint32_t *A = cv.A - cv.a_base;                         // indexed by absolute slot
    const int n = (int)(x1 - x0);
    unsigned wedges = 0, updates = 0;                       // (work counting) this lane's
    auto take = [&]() {
        int m = 0;
        if (lane == 0) m = atomicAdd(next, 1);
        return __shfl_sync(0xffffffffu, m, 0);
    };
    auto load = [&](int m) { return m < n && lane < PW ? __ldg(hv.piece + (x0 + m) * PW + lane) : 0u; };
    int m = take();
    uint32_t rec = load(m);
    while (m < n) {
        const int m2 = take();
        const uint32_t rec2 = load(m2);                     // the next piece's record, in flight meanwhile
        const uint32_t meta = __shfl_sync(0xffffffffu, rec, 1);
        const int32_t h = (int32_t)(meta >> 4);
        const int tv = (int)(meta & 15u);
        const int32_t nb = (int32_t)__ldg(hv.hub_base + h), nlow = __ldg(hv.hub_nlow + h);
        uint32_t *T = tbl + (int64_t)(h - h0) * stride;
        __syncwarp();
        if (lane < PW) s_rec[lane] = rec;                   // per type: s_rec[2 + 2 y] first slot, [3 + 2 y] ends
        __syncwarp();
        const int32_t most = (int32_t)__reduce_max_sync(0xffffffffu, lane >= 2 && lane < PW && (lane & 1) ? rec : 0u);
        uint32_t res0 = 0, res1 = 0;                        // lane (of 64) y * L + t: the sum for slot (u, v)
        uint32_t *Au = A;
        if (kPhase == 1) Au = A + (int64_t)(g.ty[hv.hubs[h]] * L) * nnz;
        for (int32_t r = lane; r - lane < most; r += 32) {  // warp-uniform trip count
#pragma unroll
            for (int y0 = 0; y0 < L; y0 += kBatch) {
                uint32_t off[kBatch];
                uint32_t low = 0;
#pragma unroll
                for (int b = 0; b < kBatch; ++b) {          // ends of type y0 + b
                    if (y0 + b >= L) break;
                    const int32_t rel =
                        r < (int32_t)s_rec[3 + 2 * (y0 + b)] ? __ldg(g.adj + s_rec[2 + 2 * (y0 + b)] + r) - nb : -1;
                    low |= (rel < nlow ? 1u : 0u) << b;
                    off[b] = rel < 0 ? 0xffffffffu
                                     : rel < nlow ? (uint32_t)rel : (uint32_t)nlow + (uint32_t)(rel - nlow) * RW;
                }
                if (kPhase == 0) {
                    const uint32_t inc = 1u << (lb * tv & 31), inch = kPacked ? 1u << (16 * (tv & 1)) : 1u;
                    const uint32_t word = (uint32_t)(kPacked ? tv >> 1 : tv);
#pragma unroll
                    for (int b = 0; b < kBatch; ++b)
                        if (y0 + b < L && off[b] != 0xffffffffu) {
                            const bool lo = (low >> b) & 1u;
                            atomicAdd(T + (lo ? off[b] : off[b] + word), lo ? inc : inch);
                            if (kCount) ++wedges;
                        }
                } else if (kPhase == 1) {
                    uint32_t word[kBatch][RW];
#pragma unroll
                    for (int b = 0; b < kBatch; ++b) {
                        if (y0 + b >= L) break;
                        const bool act = off[b] != 0xffffffffu, high = act && !((low >> b) & 1u);
                        word[b][0] = act ? __ldcg(T + off[b]) : 0u;
#pragma unroll
                        for (int k = 1; k < RW; ++k) word[b][k] = high ? __ldcg(T + off[b] + k) : 0u;
                    }
#pragma unroll
                    for (int b = 0; b < kBatch; ++b) {
                        if (y0 + b >= L) break;
                        const bool lo = (low >> b) & 1u, act = off[b] != 0xffffffffu;
                        // a low end that only this wedge reaches closes nothing
                        const bool some = act && !(lo && word[b][0] == 1u << (lb * tv & 31));
                        if (!__any_sync(0xffffffffu, some)) continue;
                        uint32_t *Ay = Au + s_rec[2 + 2 * (y0 + b)] + r;
#pragma unroll
                        for (int t = 0; t < L; ++t) {
                            const uint32_t hi = kPacked ? (word[b][t >> 1] >> (16 * (t & 1))) & 0xffffu : word[b][t];
                            uint32_t v = lo ? (word[b][0] >> (lb * t & 31)) & lm : hi;
                            v -= t == tv && act ? 1u : 0u;
                            if (v) {
                                atomicAdd(Ay, v);
                                if (kCount) ++updates;
                            }
                            Ay += nnz;
                            const uint32_t sum = __reduce_add_sync(0xffffffffu, v);
                            const int at = (y0 + b) * L + t;
                            if (at < 32) res0 += lane == at ? sum : 0u;
                            else res1 += lane == at - 32 ? sum : 0u;
                        }
                    }
                } else {
#pragma unroll
                    for (int b = 0; b < kBatch; ++b)
                        if (y0 + b < L && off[b] != 0xffffffffu) {
                            __stcg(T + off[b], 0u);
                            if (!((low >> b) & 1u))
                                for (int k = 1; k < RW; ++k) __stcg(T + off[b] + k, 0u);
                        }
                }
            }
        }
        if (kPhase == 1) {
            const int64_t sv = __shfl_sync(0xffffffffu, rec, 0);
            auto add = [&](int at, uint32_t v) {            // (y, t) = (at / L, at % L)
                if (v) {
                    atomicAdd(&A[(int64_t)((at % L) * L + at / L) * nnz + sv], v);
                    if (kCount) ++updates;
                }
            };
            add(lane, res0);
            if (L * L > 32) add(lane + 32, res1);
        }
        m = m2;
        rec = rec2;
    }
    if (kCount) {
        wedges = __reduce_add_sync(0xffffffffu, wedges);
        updates = __reduce_add_sync(0xffffffffu, updates);
        if (lane == 0 && wedges) atomicAdd(&cv.work[kWorkHubWedges], (unsigned long long)wedges);
        if (lane == 0 && updates) atomicAdd(&cv.work[kWorkHubSlotUpdates], (unsigned long long)updates);
    }
}

// The hub pass as one persistent launch over a ticket queue.  The hubs are
// cut into groups whose tables fit one of kHubBuffers table buffers; every
// group has four kinds of tickets, each a range of its pieces or table
// words: 0 fill the counters, 1 read them (4-cycle slot updates), 2 clear
// them by walking the pieces again or 3 by zeroing the group's table words.
// A CTA takes the next ticket from a device counter and, before working on
// it, waits until the tickets it needs are done: reading needs the group's
// fills, clearing its reads, and filling the clears of the group that used
// the same buffer before (kHubBuffers groups back).  Tickets are queued so
// that those are a few groups earlier, and a ticket is taken only by a
// running CTA, so every wait ends; each wait is bounded all the same and
// reports TG_ERR_TIMEOUT (the ticket is then skipped but still marked done,
// so no other wait depends on it forever).

constexpr int kHubBuffers = 3;
constexpr int kHubKinds = 4;
constexpr long long kSpinLimit = 1ll << 24;                // polls of 256 ns and more: several seconds

// range of ticket `local` of a (group, kind) run: pieces for kinds 0-2,
// table words of the group's buffer for kind 3
__device__ __forceinline__ void hub_ticket_range(const HubGroup &gr, int kind, int64_t local, int64_t &x0, int64_t &x1) {
    if (kind == 3) {
        x0 = local * kHubTicketWords;
        x1 = min(gr.zwords, x0 + kHubTicketWords);
    } else {
        x0 = gr.x0 + local * gr.tx;
        x1 = min(gr.x1, x0 + gr.tx);
    }
}

__device__ bool wait_done(const unsigned long long *ctr, unsigned long long target, uint32_t *status) {
    for (long long it = 0; it < kSpinLimit; ++it) {
        if (*(volatile const unsigned long long *)ctr >= target) return true;
        if (*(volatile const uint32_t *)status & ST_TIMEOUT) return false;   // another wait ran out: drain
        __nanosleep(256);
    }
    set_status(status, ST_TIMEOUT);
    return false;
}

template <int L, bool kPacked, bool kCount>
__global__ void __launch_bounds__(kHubThreads, kHubCtasPerSm)
    k_wedge_hub(GraphView g, CountView cv, HubView hv, const HubSegment *__restrict__ segs, int64_t n_segs,
                int64_t n_tickets, const HubGroup *__restrict__ groups, const int64_t *__restrict__ ntick,
                unsigned long long *ctr, uint32_t *tables, int64_t buf_words, int64_t stride) {
    __shared__ int64_t s_t, s_x0, s_x1;
    __shared__ int s_ok, s_group, s_kind, s_next;
    __shared__ uint32_t s_rec[kHubThreads / 32][piece_words(L)];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long *next = ctr;                         // ticket counter
    unsigned long long *done = ctr + 1;                     // [group][kind] tickets done
    long long c0 = 0;                                       // work counting: clock at the ticket's start
    int64_t seg = 0;                                        // (thread 0) run of the last ticket
    for (;;) {
        if (threadIdx.x == 0) {
            const int64_t t = (int64_t)atomicAdd(next, 1ull);
            if (kCount) c0 = clock64();
            bool ok = true;
            if (t < n_tickets) {
                // the run holding ticket t: a CTA's tickets rise, so it is this one or soon after
                while (seg + 1 < n_segs && segs[seg + 1].t0 <= t) ++seg;
                const HubSegment sg = segs[seg];
                int64_t x0, x1;
                hub_ticket_range(groups[sg.group], sg.kind, t - sg.t0, x0, x1);
                s_x0 = x0;
                s_x1 = x1;
                s_group = sg.group;
                s_kind = sg.kind;
                const int64_t q = sg.group;
                if (sg.kind == 1) {
                    ok = wait_done(&done[q * kHubKinds + 0], (unsigned long long)ntick[q * kHubKinds + 0], cv.status);
                } else if (sg.kind >= 2) {
                    ok = wait_done(&done[q * kHubKinds + 1], (unsigned long long)ntick[q * kHubKinds + 1], cv.status);
                } else if (q >= kHubBuffers) {
                    const int64_t p = q - kHubBuffers;
                    ok = wait_done(&done[p * kHubKinds + 2], (unsigned long long)ntick[p * kHubKinds + 2], cv.status) &&
                         wait_done(&done[p * kHubKinds + 3], (unsigned long long)ntick[p * kHubKinds + 3], cv.status);
                }
                __threadfence();
            }
            if (kCount) {
                const long long c1 = clock64();
                atomicAdd(&cv.work[kWorkHubWait], (unsigned long long)(c1 - c0));
                c0 = c1;
            }
            s_t = t;
            s_next = 0;
            s_ok = ok ? 1 : 0;
        }
        __syncthreads();
        const int64_t t = s_t;
        if (t >= n_tickets) break;                          // CTA-uniform
        const int group = s_group, kind = s_kind;
        const int64_t x0 = s_x0, x1 = s_x1;
        const HubGroup gr = groups[group];
        uint32_t *tbl = tables + (int64_t)gr.buf * buf_words;
        if (s_ok) {
            if (kind == 3) {
                for (int64_t x = x0 + threadIdx.x; x < x1; x += blockDim.x) __stcg(tbl + x, 0u);
            } else if (kind == 0) {
                hub_pieces<L, kPacked, kCount, 0>(g, cv, hv, gr.h0, x0, x1, tbl, stride, &s_next, s_rec[wid], lane);
            } else if (kind == 1) {
                hub_pieces<L, kPacked, kCount, 1>(g, cv, hv, gr.h0, x0, x1, tbl, stride, &s_next, s_rec[wid], lane);
            } else {
                hub_pieces<L, kPacked, kCount, 2>(g, cv, hv, gr.h0, x0, x1, tbl, stride, &s_next, s_rec[wid], lane);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&done[(int64_t)group * kHubKinds + kind], 1ull);
            if (kCount) atomicAdd(&cv.work[kWorkHubKind + kind], (unsigned long long)(clock64() - c0));
        }
    }
}

template <class T>
void exclusive_sum(const T *in, T *out, int64_t n, cudaStream_t s) {
    size_t tb = 0;
    TG_CK(cub::DeviceScan::ExclusiveSum(nullptr, tb, in, out, n, s));
    TBuf tmp(std::max<size_t>(tb, 16), s);
    TG_CK(cub::DeviceScan::ExclusiveSum(tmp.p, tb, in, out, n, s));
}

unsigned blocks(int64_t threads) { return (unsigned)std::max<int64_t>(1, (threads + 255) / 256); }

// words of the largest hub's counter table
int64_t words_per_table(const Graph &G, const std::vector<int32_t> &nlow) {
    const int64_t rw = G.hub_packed ? (G.L + 1) / 2 : G.L;
    int64_t most = 1;
    for (size_t h = 0; h < nlow.size(); ++h) {
        const size_t gr = std::upper_bound(G.h_node_off.begin(), G.h_node_off.end(), (int64_t)G.h_hub_id[h]) -
                          G.h_node_off.begin() - 1;
        most = std::max(most, nlow[h] + (G.h_node_off[gr + 1] - G.h_node_off[gr] - nlow[h]) * rw);
    }
    return most;
}

}  // namespace

// Pieces, groups and the ticket queue of every chunk (graph invariant, built
// before any capture).  Groups: consecutive hubs of one chunk, at most as
// many tables as half of hub_l2_mb holds and about 2^24 wedges; per group,
// fill and read tickets of at least two per CTA of the launch and clear
// tickets (zeroing the group's table words when that is cheaper than walking
// its pieces again: about 2.5e11 random stores and 5e12 bytes per second).
// Queue order: the clears of group s - 2, the reads of group s - 1, the fills
// of group s, for s = 0, 1, ...: every ticket waits on tickets at least one
// phase of another group earlier in the queue.
void prepare_hubs(Graph &G, cudaStream_t s) {
    const int L = G.L;
    const int64_t nh = G.n_hubs;
    const GraphView gv = G.view();
    G.hub_packed = G.max_degree < 65536;
    G.hub_base.alloc(sizeof(int64_t) * nh);
    G.hub_nlow.alloc(sizeof(int32_t) * nh);
    TBuf nv(sizeof(int64_t) * (nh + 1), s), vbase(sizeof(int64_t) * (nh + 1), s), bound(sizeof(int64_t) * (nh + 1), s);
    k_hub_info<<<blocks(nh + 1), 256, 0, s>>>(gv, G.hubs.as<int32_t>(), nh, G.hub_base.as<int64_t>(),
                                              G.hub_nlow.as<int32_t>(), nv.as<int64_t>());
    TG_CK(cudaGetLastError());
    exclusive_sum(nv.as<int64_t>(), vbase.as<int64_t>(), nh + 1, s);
    int64_t n_pairs = 0;
    TG_CK(cudaMemcpyAsync(&n_pairs, vbase.as<int64_t>() + nh, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    std::vector<int32_t> nlow((size_t)nh);
    TG_CK(cudaMemcpyAsync(nlow.data(), G.hub_nlow.p, sizeof(int32_t) * nh, cudaMemcpyDeviceToHost, s));
    TG_CK(cudaStreamSynchronize(s));
    G.hub_stride = words_per_table(G, nlow);
    // no more tables per buffer than there are hubs (a small graph's budget
    // would otherwise reserve hub_l2_mb for a few hubs)
    const int64_t fit = ((int64_t)G.opt.hub_l2_mb << 20) / 2 / (G.hub_stride * (int64_t)sizeof(uint32_t));
    const int64_t gmax = std::min<int64_t>(std::max<int64_t>(fit, 1), nh);
    G.hub_buf_words = gmax * G.hub_stride;
    const size_t tbytes = sizeof(uint32_t) * (size_t)(kHubBuffers * G.hub_buf_words);
    G.hub_tables.alloc(tbytes);
    TG_CK(cudaMemsetAsync(G.hub_tables.p, 0, tbytes, s));

    // pieces, in hub order
    TBuf count(sizeof(int64_t) * (n_pairs + 1), s), first(sizeof(int64_t) * (n_pairs + 1), s);
    TG_CK(cudaMemsetAsync(count.as<int64_t>() + n_pairs, 0, sizeof(int64_t), s));
    if (n_pairs > 0)
        k_hub_pieces<false><<<blocks(n_pairs * 8), 256, 0, s>>>(gv, G.hubs.as<int32_t>(), nh, vbase.as<int64_t>(), n_pairs,
                                                                count.as<int64_t>(), nullptr, nullptr);
    TG_CK(cudaGetLastError());
    exclusive_sum(count.as<int64_t>(), first.as<int64_t>(), n_pairs + 1, s);
    k_hub_bounds<<<blocks(nh + 1), 256, 0, s>>>(nh, vbase.as<int64_t>(), first.as<int64_t>(), bound.as<int64_t>());
    TG_CK(cudaGetLastError());
    std::vector<int64_t> hub_piece((size_t)nh + 1);
    TG_CK(cudaMemcpyAsync(hub_piece.data(), bound.p, sizeof(int64_t) * (nh + 1), cudaMemcpyDeviceToHost, s));
    TG_CK(cudaStreamSynchronize(s));
    G.hub_piece.alloc(sizeof(uint32_t) * piece_words(L) * (size_t)std::max<int64_t>(hub_piece[(size_t)nh], 1));
    if (n_pairs > 0)
        k_hub_pieces<true><<<blocks(n_pairs * 8), 256, 0, s>>>(gv, G.hubs.as<int32_t>(), nh, vbase.as<int64_t>(), n_pairs,
                                                               nullptr, first.as<int64_t>(), G.hub_piece.as<uint32_t>());
    TG_CK(cudaGetLastError());

    // ticket queues
    const int64_t ctas = (int64_t)sm_count() * kHubCtasPerSm;
    std::vector<std::unique_ptr<Graph::HubPlan>> plans;     // the handle gets all of them or, on an error, none
    for (size_t c = 0; c < G.chunks.size(); ++c) {
        auto plan = std::make_unique<Graph::HubPlan>();
        for (DBuf *d : {&plan->segs, &plan->groups, &plan->ntick, &plan->ctr}) d->owner = &G;
        std::vector<HubGroup> &groups = plan->h_groups;
        std::vector<int64_t> &ntick = plan->h_ntick;
        auto below = [&](int64_t n) {                       // hubs of earlier graphs (hub order is by graph first)
            return std::partition_point(G.h_hub_id.begin(), G.h_hub_id.end(), [&](int32_t id) { return id < n; }) -
                   G.h_hub_id.begin();
        };
        const int64_t hb1 = below(G.chunks[c].n1);
        for (int64_t h = below(G.chunks[c].n0); h < hb1;) {
            HubGroup gr{};
            gr.h0 = (int32_t)h;
            gr.buf = (int32_t)(groups.size() % kHubBuffers);
            int64_t wsum = 0;
            while (h < hb1 && h - gr.h0 < gmax && wsum < ((int64_t)1 << 24)) wsum += G.h_hub_wedges[(size_t)h++];
            gr.zwords = (h - gr.h0) * G.hub_stride;
            gr.x0 = hub_piece[(size_t)gr.h0];
            gr.x1 = hub_piece[(size_t)h];
            const int64_t n = gr.x1 - gr.x0;
            gr.tx = std::min<int64_t>(std::max<int64_t>((n + 2 * ctas - 1) / (2 * ctas), 8), 1 << 16);
            const int64_t nt = (n + gr.tx - 1) / gr.tx;
            const bool zero = gr.zwords * (int64_t)sizeof(uint32_t) <= 20 * wsum;
            ntick.push_back(nt);                                                     // fill
            ntick.push_back(nt);                                                     // read
            ntick.push_back(zero ? 0 : nt);                                          // clear by walking
            ntick.push_back(zero ? (gr.zwords + kHubTicketWords - 1) / kHubTicketWords : 0);   // clear by zeroing
            groups.push_back(gr);
        }
        const int64_t np = (int64_t)groups.size();
        std::vector<HubSegment> &segs = plan->h_segs;
        int64_t nt = 0;
        for (int64_t st = 0; st < np + 2; ++st) {
            auto emit = [&](int64_t q, int kind) {
                if (q < 0 || q >= np || ntick[q * kHubKinds + kind] == 0) return;
                segs.push_back(HubSegment{nt, (int32_t)q, kind});
                nt += ntick[q * kHubKinds + kind];
            };
            emit(st - 2, 2);
            emit(st - 2, 3);
            emit(st - 1, 1);
            emit(st, 0);
        }
        // every run waits only on runs queued before it (so each wait ends:
        // those tickets were taken by running CTAs)
        {
            std::vector<int64_t> pos((size_t)std::max<int64_t>(np * kHubKinds, 1), -1);
            for (int64_t k = 0; k < (int64_t)segs.size(); ++k) pos[(size_t)(segs[k].group * kHubKinds + segs[k].kind)] = k;
            for (int64_t k = 0; k < (int64_t)segs.size(); ++k) {
                const int64_t q = segs[k].group;
                const int kind = segs[k].kind;
                int64_t dep[2] = {-1, -1};
                if (kind == 1) dep[0] = q * kHubKinds;
                else if (kind >= 2) dep[0] = q * kHubKinds + 1;
                else if (q >= kHubBuffers) { dep[0] = (q - kHubBuffers) * kHubKinds + 2; dep[1] = dep[0] + 1; }
                for (int64_t d : dep)
                    if (d >= 0 && pos[(size_t)d] >= k) throw Error{TG_ERR_INTERNAL, "hub ticket order"};
            }
        }
        plan->n_groups = np;
        plan->n_segs = (int64_t)segs.size();
        plan->n_tickets = nt;
        if (np > 0) {
            plan->segs.alloc(sizeof(HubSegment) * segs.size());
            plan->groups.alloc(sizeof(HubGroup) * groups.size());
            plan->ntick.alloc(sizeof(int64_t) * ntick.size());
            plan->ctr.alloc(sizeof(unsigned long long) * (size_t)(1 + np * kHubKinds));
            TG_CK(cudaMemcpyAsync(plan->segs.p, segs.data(), sizeof(HubSegment) * segs.size(), cudaMemcpyHostToDevice, s));
            TG_CK(cudaMemcpyAsync(plan->groups.p, groups.data(), sizeof(HubGroup) * groups.size(),
                                  cudaMemcpyHostToDevice, s));
            TG_CK(cudaMemcpyAsync(plan->ntick.p, ntick.data(), sizeof(int64_t) * ntick.size(), cudaMemcpyHostToDevice,
                                  s));
        }
        plans.push_back(std::move(plan));
    }
    G.hub_plans = std::move(plans);
}

int64_t launch_hubs(Graph &G, size_t ci, cudaStream_t s) {
    Graph::HubPlan &P = *G.hub_plans[ci];
    if (P.n_tickets == 0) return 0;
    TG_CK(cudaMemsetAsync(P.ctr.p, 0, sizeof(unsigned long long) * (size_t)(1 + P.n_groups * kHubKinds), s));
    HubView hv;
    hv.hubs = G.hubs.as<int32_t>();
    hv.hub_base = G.hub_base.as<int64_t>();
    hv.hub_nlow = G.hub_nlow.as<int32_t>();
    hv.piece = G.hub_piece.as<uint32_t>();
    const int grid = sm_count() * kHubCtasPerSm;
    KernelTimer kt(G, s, "k_wedge_hub");
    with_types(G.L, [&](auto l) {
        constexpr int L = decltype(l)::value;
        auto launch = [&](auto kern) {
            kern<<<grid, kHubThreads, 0, s>>>(G.view(), G.cview(), hv, P.segs.as<HubSegment>(), P.n_segs, P.n_tickets,
                                              P.groups.as<HubGroup>(), P.ntick.as<int64_t>(),
                                              P.ctr.as<unsigned long long>(), G.hub_tables.as<uint32_t>(),
                                              G.hub_buf_words, G.hub_stride);
        };
        const bool count = G.work_on;                       // the work-counting form (diagnostics)
        if (G.hub_packed && !count) launch(k_wedge_hub<L, true, false>);
        else if (G.hub_packed) launch(k_wedge_hub<L, true, true>);
        else if (!count) launch(k_wedge_hub<L, false, false>);
        else launch(k_wedge_hub<L, false, true>);
    });
    TG_CK(cudaGetLastError());
    return 1;
}

}  // namespace tg

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
#include <vector>

#include <cub/device/device_scan.cuh>

#include <mutex>

#include "tg_host.hpp"

namespace tg {

namespace {


// ------------------------------------------------------------ hub anchors
// An anchor u with very many wedges (a hub) is counted by the whole GPU at
// once: every CTA works on the wedges of the same few hubs, against one node
// table per hub that all CTAs share, so the tables stay in L2 instead of one
// dense table per CTA streaming through HBM.  The wedges u - v - w (v, w of
// lower priority than u) of every hub are flattened into items, one per
// (hub, v, type of w) with at least one wedge; item_woff is the exclusive
// prefix of the items' wedge counts, so wedge x of the flattened order is
// w = adj[item_vb[it] + x - item_woff[it]] for the item it containing x.
// The counts are those of tg_wedge.cu: phase 0 fills h_u[w][t] (the
// number of type-t neighbours v of u below u that are adjacent to w),
// phase 1 adds h_u[w][t] - [t = t_v] to the 4-cycle slot of (v, w) and the
// per-(v, type of w) sums to the slot of (u, v), phase 2 clears the rows.
// All hubs of a chunk run in one persistent launch (k_wedge_hub below):
// hubs in groups, every (group, phase) cut into tickets, ticket waits on the
// phases it depends on.

struct HubView {
    const int32_t *hubs;        // hub node ids
    const int64_t *hub_base;    // first node of each hub's graph (read when batched)
    const int32_t *hub_nlow;    // nodes of each hub's graph with one-word rows (read when batched)
    int32_t nlow;               // the same when there is one graph
    const int64_t *woff;        // [n_items + 1] first wedge of each item
    const int4 *item;           // per item: adj position of its first w, adj position of v in the
                                // hub's row, hub index, type of u << 8 | type of v << 4 | type of w
    bool batched;               // several graphs: tables are indexed from each hub's graph's first node
};

constexpr int kHubThreads = 256;

// Table rows.  A counter h_u[w][t] is at most d_w^t, so a node w of degree
// below 2^(32 / L) has all its types in one word; the nodes of a graph are
// in degree order, so these are a prefix of its ids (L = 5: degree 63 and
// less, 96% of a Chung-Lu graph of average degree 20), and its table is a
// third of one with 16-bit counters throughout.
__host__ __device__ __forceinline__ int low_bits(int L) { return 32 / L; }

__global__ void k_hub_nv(GraphView g, const int32_t *__restrict__ hubs, int64_t n_hubs, int64_t *nv,
                         int64_t *hub_base, int32_t *hub_nlow) {
    const int64_t h = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (h > n_hubs) return;
    if (h == n_hubs) { nv[h] = 0; return; }
    const int32_t u = hubs[h];
    int64_t acc = 0;
    for (int t = 0; t < g.L; ++t) {
        int64_t b, cut;
        seg_prefix(g, u, t, u, b, cut);
        acc += cut - b;
    }
    nv[h] = acc;
    const int gr = graph_of_node(g, u);
    const int64_t base = g.node_off[gr];
    hub_base[h] = base;
    int64_t lo = base, hi = g.node_off[gr + 1];             // first node whose degree has no room in a field
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if ((g.rp[mid + 1] - g.rp[mid]) >> low_bits(g.L)) hi = mid; else lo = mid + 1;
    }
    hub_nlow[h] = (int32_t)(lo - base);
}

// CTA per hub: wedge count of every (v, type of w) of the hub
__global__ void __launch_bounds__(256) k_hub_cnt(GraphView g, const int32_t *__restrict__ hubs, int64_t n_hubs,
                                                 const int64_t *__restrict__ vbase, int32_t *cnt, int64_t *flag,
                                                 int32_t *sv_of, int32_t *hub_of) {
    __shared__ int64_t s_b[kMaxL + 1], s_cnt[kMaxL + 1];
    const int L = g.L;
    for (int64_t h = blockIdx.x; h < n_hubs; h += gridDim.x) {
        const int32_t u = hubs[h];
        __syncthreads();
        if (threadIdx.x == 0) {
            int64_t acc = 0;
            for (int t = 0; t < L; ++t) {
                int64_t b, cut;
                seg_prefix(g, u, t, u, b, cut);
                s_b[t] = b;
                s_cnt[t] = acc;
                acc += cut - b;
            }
            s_cnt[L] = acc;
        }
        __syncthreads();
        const int64_t nV = s_cnt[L], base = vbase[h];
        for (int64_t kv = threadIdx.x; kv < nV; kv += blockDim.x) {
            int tv = 0;
            while (tv + 1 < L && s_cnt[tv + 1] <= kv) ++tv;
            const int64_t sv = s_b[tv] + (kv - s_cnt[tv]);
            const int32_t v = g.adj[sv];
            sv_of[base + kv] = (int32_t)sv;
            hub_of[base + kv] = (int32_t)h;
            for (int tw = 0; tw < L; ++tw) {
                int64_t vb, vcut;
                seg_prefix(g, v, tw, u, vb, vcut);
                const int64_t idx = (base + kv) * L + tw;
                cnt[idx] = (int32_t)(vcut - vb);
                flag[idx] = vcut > vb ? 1 : 0;
            }
        }
    }
}

__global__ void k_hub_items(GraphView g, int64_t ni, const int32_t *__restrict__ cnt, const int64_t *__restrict__ pos,
                            const int32_t *__restrict__ sv_of, const int32_t *__restrict__ hub_of,
                            const int32_t *__restrict__ hubs, int4 *item, int64_t *icnt) {
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= ni) return;
    const int32_t c = cnt[idx];
    if (c == 0) return;
    const int64_t j = pos[idx], kv = idx / g.L;
    const int tw = (int)(idx - kv * g.L);
    const int32_t s = sv_of[kv];
    const int32_t v = g.adj[s];
    const int32_t h = hub_of[kv];
    item[j] = make_int4((int32_t)seg_begin(g, v, tw), s, h, (g.ty[hubs[h]] << 8) | (g.ty[v] << 4) | tw);
    icnt[j] = c;
}

__global__ void k_hub_bounds(int64_t n_hubs, int L, const int64_t *__restrict__ vbase, const int64_t *__restrict__ pos,
                             const int64_t *__restrict__ woff, int64_t *first_item, int64_t *first_wedge) {
    const int64_t h = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (h > n_hubs) return;
    const int64_t it = pos[vbase[h] * L];
    first_item[h] = it;
    first_wedge[h] = woff[it];
}

// largest j in [lo, hi) with woff[j] <= x, given woff[lo] <= x < woff[hi];
// a 32-way search by the whole warp
__device__ __forceinline__ int64_t hub_find_item(const int64_t *__restrict__ woff, int64_t lo, int64_t hi, int64_t x,
                                                 int lane) {
    while (hi - lo > 32) {
        const int64_t step = (hi - lo + 31) / 32;
        const int64_t p = lo + lane * step;
        const unsigned b = __ballot_sync(0xffffffffu, p < hi && woff[p] <= x);
        lo += (int64_t)(31 - __clz(b)) * step;
        hi = min(hi, lo + step);
    }
    const int64_t p = lo + lane;
    const unsigned b = __ballot_sync(0xffffffffu, p < hi && woff[p] <= x);
    return lo + (31 - __clz(b));
}

// One phase of the hub wedge pass over the wedges [x0r, x1r) of one group of
// hubs (items [i0, i1), first hub h0; hub h's table at tbl + (h - h0) *
// stride).  Warp wi of nwi takes one contiguous run of the range, 32 wedges
// at a time, one wedge per lane; the item window of the next 32 wedges is
// loaded while the current ones are worked on.  Counters: one word per node
// for the graph's low nodes (above); for the others kPacked = two 16-bit
// counters per 32-bit word (types 2k and 2k+1; every count is at most the
// hub's degree, below 2^16 when this layout is chosen), else one 32-bit
// counter per type.  The tables are read and cleared at L2 (ld/st.cg): other
// CTAs of the same launch update them, so no L1 copy may be trusted.
template <bool kPacked, bool kCount>
__device__ void hub_wedges(const GraphView &g, const CountView &cv, const HubView &hv, int64_t i0, int64_t i1,
                           int64_t x0r, int64_t x1r, int32_t h0, uint32_t *tbl, int64_t stride, int phase, int wi,
                           int nwi, int lane) {
    const int L = g.L;
    const int RW = kPacked ? (L + 1) / 2 : L;               // words per row of a node that is not low
    const int lb = low_bits(L);                             // bits per type in a low node's word
    const int64_t per = (((x1r - x0r) + nwi - 1) / nwi + 31) & ~(int64_t)31;
    int64_t x0 = x0r + wi * per;
    const int64_t xe = min(x1r, x0 + per);
    if (x0 >= xe) return;                                   // warp-uniform
    if (kCount && phase == 0 && lane == 0) atomicAdd(&cv.work[kWorkHubWedges], (unsigned long long)(xe - x0));
    const int64_t nnz = cv.a_stride;
    uint32_t *A = cv.A - cv.a_base;                         // indexed by absolute slot
    int64_t j = hub_find_item(hv.woff, i0, i1, x0, lane);
    int64_t wo = j + lane < i1 ? hv.woff[j + lane] : INT64_MAX;
    unsigned long long nupd_run = 0;                        // (work counting) the warp's slot updates
    for (; x0 < xe; x0 += 32) {
        // the wedges x0 .. x0+31 lie in items j .. j+31 (every item is non-empty)
        const int64_t x = x0 + lane;
        const bool act = x < xe;
        int k = 0;
#pragma unroll
        for (int st = 16; st > 0; st >>= 1) {
            const int64_t c = __shfl_sync(0xffffffffu, wo, k + st);
            if (c <= x) k += st;
        }
        const int64_t it = j + k;
        const int64_t wstart = __shfl_sync(0xffffffffu, wo, k);
        const int k31 = __shfl_sync(0xffffffffu, k, 31);
        const int64_t wnext = k31 < 31 ? __shfl_sync(0xffffffffu, wo, k31 < 31 ? k31 + 1 : 31)
                                       : (j + 32 < i1 ? hv.woff[j + 32] : INT64_MAX);
        // first item of the next 32 wedges (the item of x0 + 32), and its window
        const int64_t jn = (wnext <= x0 + 32) ? j + k31 + 1 : j + k31;
        const int64_t won = x0 + 32 < xe && jn + lane < i1 ? hv.woff[jn + lane] : INT64_MAX;
        int32_t svp = 0;
        int tw = 0;
        uint32_t c[kMaxL];
#pragma unroll
        for (int t = 0; t < kMaxL; ++t) c[t] = 0;
        if (act) {
            const int4 rec = hv.item[it];
            const int32_t hh = rec.z;
            const int tv = (rec.w >> 4) & 15;
            tw = rec.w & 15;
            svp = rec.y;
            const int64_t pos = (int64_t)rec.x + (x - wstart);
            const int32_t w = g.adj[pos];
            const int64_t base = hv.batched ? hv.hub_base[hh] : 0;
            const int32_t nlow = hv.batched ? hv.hub_nlow[hh] : hv.nlow;
            const int32_t rel = (int32_t)(w - base);
            const bool low = rel < nlow;
            uint32_t *row = tbl + (int64_t)(hh - h0) * stride + (low ? rel : nlow + (int64_t)(rel - nlow) * RW);
            if (phase == 0) {
                if (low) atomicAdd(row, 1u << (lb * tv));
                else if (kPacked) atomicAdd(row + (tv >> 1), 1u << (16 * (tv & 1)));
                else atomicAdd(row + tv, 1u);
            } else if (phase == 1) {
                const int tu = rec.w >> 8;
                uint32_t words[kMaxL];
                words[0] = __ldcg(row);
#pragma unroll
                for (int q = 1; q < kMaxL; ++q) words[q] = !low && q < RW ? __ldcg(row + q) : 0u;
                if (!low || words[0] != 1u << (lb * tv)) {  // (else this wedge alone: it closes nothing)
                    const uint32_t lm = lb == 32 ? 0xffffffffu : (1u << lb) - 1u;
#pragma unroll
                    for (int t = 0; t < kMaxL; ++t) {
                        if (t >= L) break;
                        const uint32_t hi = kPacked ? (words[t >> 1] >> (16 * (t & 1))) & 0xffffu : words[t];
                        const uint32_t h = low ? (words[0] >> (lb * t)) & lm : hi;
                        const uint32_t v = h - (t == tv ? 1u : 0u);
                        c[t] = v;
                        if (v) atomicAdd(&A[(int64_t)(tu * L + t) * nnz + pos], v);
                    }
                }
            } else {
                for (int q = 0; q < (low ? 1 : RW); ++q) __stcg(row + q, 0u);
            }
        }
        if (phase == 1) {
            // (work counting) the round's nonzero slot updates: per wedge, then per item sum
            unsigned nupd = 0;                              // (work counting) these 32 wedges' updates, warp-wide
            if (kCount) {
#pragma unroll
                for (int t = 0; t < kMaxL; ++t) nupd += t < L && c[t] ? 1u : 0u;
                nupd = __reduce_add_sync(0xffffffffu, nupd);
            }
            // per-item sums over the lanes of each item (items are contiguous runs of lanes)
            const int64_t key = act ? it : -1;
            const int64_t key0 = __shfl_sync(0xffffffffu, key, 0);
            if (__all_sync(0xffffffffu, !act || key == key0)) {
                // one item: warp sums, added by lane 0 (always active here)
#pragma unroll
                for (int t = 0; t < kMaxL; ++t) {
                    if (t >= L) break;
                    const uint32_t v = __reduce_add_sync(0xffffffffu, c[t]);
                    if (lane == 0 && v) atomicAdd(&A[(int64_t)(t * L + tw) * nnz + svp], v);
                    if (kCount) nupd += v ? 1u : 0u;       // (warp-uniform)
                }
            } else {
                unsigned same = 0;
#pragma unroll
                for (int s = 0; s < 5; ++s) {
                    const int64_t kk = __shfl_up_sync(0xffffffffu, key, 1 << s);
                    if (lane >= (1 << s) && kk == key) same |= 1u << s;
                }
                const int64_t knext = __shfl_down_sync(0xffffffffu, key, 1);
                const bool tail = act && (lane == 31 || knext != key);
#pragma unroll
                for (int t = 0; t < kMaxL; ++t) {
                    if (t >= L) break;
                    uint32_t v = c[t];
#pragma unroll
                    for (int s = 0; s < 5; ++s) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, v, 1 << s);
                        if (same & (1u << s)) v += y;
                    }
                    if (tail && v) atomicAdd(&A[(int64_t)(t * L + tw) * nnz + svp], v);
                    if (kCount) nupd += __popc(__ballot_sync(0xffffffffu, tail && v));
                }
            }
            if (kCount) nupd_run += nupd;
        }
        j = jn;
        wo = won;
    }
    if (kCount && lane == 0 && nupd_run) atomicAdd(&cv.work[kWorkHubSlotUpdates], nupd_run);
}

// The hub pass as one persistent launch over a ticket queue.  The hubs are
// cut into groups whose tables fit one of kHubBuffers table buffers; every
// group has four kinds of tickets, each a range of its wedges or table
// words: 0 fill the counters, 1 read them (4-cycle slot updates), 2 clear
// them by walking the wedges again or 3 by zeroing the group's table words.
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

// range of ticket `local` of a (group, kind) run: wedges for kinds 0-2,
// table words of the group's buffer for kind 3
__device__ __forceinline__ void hub_ticket_range(const HubGroup &gr, int kind, int64_t local, int64_t &x0, int64_t &x1) {
    if (kind == 3) {
        x0 = local * kHubTicketWords;
        x1 = min(gr.zwords, x0 + kHubTicketWords);
    } else {
        x0 = gr.w0 + local * gr.tw;
        x1 = min(gr.w1, x0 + gr.tw);
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

template <bool kPacked, bool kCount>
__global__ void __launch_bounds__(kHubThreads, 5) k_wedge_hub(GraphView g, CountView cv, HubView hv,
                                                           const HubSegment *__restrict__ segs, int64_t n_segs,
                                                           int64_t n_tickets, const HubGroup *__restrict__ groups,
                                                           const int64_t *__restrict__ ntick,
                                                           unsigned long long *ctr, uint32_t *tables, int64_t buf_words,
                                                           int64_t stride) {
    __shared__ int64_t s_t, s_x0, s_x1;
    __shared__ int s_ok, s_group, s_kind;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    unsigned long long *next = ctr;                         // ticket counter
    unsigned long long *done = ctr + 1;                     // [group][kind] tickets done
    long long c0 = 0;                                       // work counting: clock at the ticket's start
    for (;;) {
        if (threadIdx.x == 0) {
            const int64_t t = (int64_t)atomicAdd(next, 1ull);
            if (cv.work) c0 = clock64();
            bool ok = true;
            if (t < n_tickets) {
                int64_t lo = 0, hi = n_segs;                // the run holding ticket t: segs[lo].t0 <= t
                while (hi - lo > 1) {
                    const int64_t mid = (lo + hi) >> 1;
                    if (segs[mid].t0 <= t) lo = mid; else hi = mid;
                }
                const HubSegment sg = segs[lo];
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
            if (cv.work) {
                const long long c1 = clock64();
                atomicAdd(&cv.work[kWorkHubWait], (unsigned long long)(c1 - c0));
                c0 = c1;
            }
            s_t = t;
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
            } else {
                hub_wedges<kPacked, kCount>(g, cv, hv, gr.i0, gr.i1, x0, x1, gr.h0, tbl, stride, kind, wid, nwarp,
                                            lane);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&done[(int64_t)group * kHubKinds + kind], 1ull);
            if (cv.work) atomicAdd(&cv.work[kWorkHubKind + kind], (unsigned long long)(clock64() - c0));
        }
    }
}

int grid_for(int64_t items, int per_block, int cap) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (int)b;
}

}  // namespace

// Edges per tile: kTile, or fewer for a small handle so that its tiles
// still fill the GPU (at least about 12 tiles per SM, 64 edges or more each).
static int64_t tile_edges(const Graph &G) {
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
        return (G.h_slot_off[b] - G.h_slot_off[a]) * 8 * LL + (G.h_edge_off[b] - G.h_edge_off[a]) * LL * (G.wide_sums() ? 32 : 16);
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
    dst.alloc(sizeof(Tile) * std::max<size_t>(tiles.size(), 1));
    if (!tiles.empty()) {
        TG_CK(cudaMemcpyAsync(dst.p, tiles.data(), sizeof(Tile) * tiles.size(), cudaMemcpyHostToDevice, s));
        TG_CK(cudaStreamSynchronize(s));   // the host vector goes out of scope
    }
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
    unused.owner = &G.stream;
    int64_t nt = 0;
    tiles_for(G, 0, G.m, nt, unused, s);
}

// words of the largest hub's counter table
static int64_t hub_words_per_table(const Graph &G) {
    const int64_t rw = G.hub_packed ? (G.L + 1) / 2 : G.L;
    int64_t most = 1;
    for (size_t h = 0; h < G.h_hub_nlow.size(); ++h) {
        const size_t gr = std::upper_bound(G.h_node_off.begin(), G.h_node_off.end(), (int64_t)G.h_hub_id[h]) -
                          G.h_node_off.begin() - 1;
        const int64_t nodes = G.h_node_off[gr + 1] - G.h_node_off[gr];
        most = std::max(most, G.h_hub_nlow[h] + (nodes - G.h_hub_nlow[h]) * rw);
    }
    return most;
}

// hubs of one group: their tables fill at most half of hub_l2_mb (the
// persistent pass fills one group's tables while it reads the previous one's)
static int64_t hub_group_max(const Graph &G) {
    const int64_t per = G.hub_stride * (int64_t)sizeof(uint32_t);
    return std::max<int64_t>(((int64_t)G.opt.hub_l2_mb << 20) / 2 / per, 1);
}

constexpr int kHubCtasPerSm = 5;                            // k_wedge_hub's launch bounds

template <class T>
static void exclusive_sum(const T *in, T *out, int64_t n, cudaStream_t s) {
    size_t tb = 0;
    TG_CK(cub::DeviceScan::ExclusiveSum(nullptr, tb, in, out, n, s));
    TBuf tmp(std::max<size_t>(tb, 16), s);
    TG_CK(cub::DeviceScan::ExclusiveSum(tmp.p, tb, in, out, n, s));
}

static HubView hub_view(const Graph &G) {
    HubView h;
    h.hubs = G.hubs.as<int32_t>();
    h.hub_base = G.hub_base.as<int64_t>();
    h.hub_nlow = G.hub_nlow.as<int32_t>();
    h.nlow = G.h_hub_nlow.empty() ? 0 : G.h_hub_nlow[0];
    h.woff = G.item_woff.as<int64_t>();
    h.item = G.item_rec.as<int4>();
    h.batched = G.ngraphs > 1;
    return h;
}

// Wedge items of the hub anchors (graph invariant, built at the first count).
static void prepare_hubs(Graph &G, cudaStream_t s) {
    const int L = G.L;
    const int64_t nh = G.n_hubs;
    const GraphView gv = G.view();
    TBuf nv(sizeof(int64_t) * (nh + 1), s), vbase(sizeof(int64_t) * (nh + 1), s);
    G.hub_base.alloc(sizeof(int64_t) * nh);
    G.hub_nlow.alloc(sizeof(int32_t) * nh);
    k_hub_nv<<<grid_for(nh + 1, 256, 1 << 20), 256, 0, s>>>(gv, G.hubs.as<int32_t>(), nh, nv.as<int64_t>(),
                                                            G.hub_base.as<int64_t>(), G.hub_nlow.as<int32_t>());
    TG_CK(cudaGetLastError());
    exclusive_sum(nv.as<int64_t>(), vbase.as<int64_t>(), nh + 1, s);
    int64_t NV = 0;
    TG_CK(cudaMemcpyAsync(&NV, vbase.as<int64_t>() + nh, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    TG_CK(cudaStreamSynchronize(s));
    const int64_t NI = NV * L;
    TBuf cnt(sizeof(int32_t) * std::max<int64_t>(NI, 1), s), flag(sizeof(int64_t) * (NI + 1), s);
    TBuf pos(sizeof(int64_t) * (NI + 1), s);
    TBuf sv_of(sizeof(int32_t) * std::max<int64_t>(NV, 1), s), hub_of(sizeof(int32_t) * std::max<int64_t>(NV, 1), s);
    TG_CK(cudaMemsetAsync(flag.p, 0, sizeof(int64_t) * (NI + 1), s));
    k_hub_cnt<<<grid_for(nh, 1, sm_count() * 8), 256, 0, s>>>(gv, G.hubs.as<int32_t>(), nh, vbase.as<int64_t>(),
                                                               cnt.as<int32_t>(), flag.as<int64_t>(),
                                                               sv_of.as<int32_t>(), hub_of.as<int32_t>());
    TG_CK(cudaGetLastError());
    exclusive_sum(flag.as<int64_t>(), pos.as<int64_t>(), NI + 1, s);
    TG_CK(cudaMemcpyAsync(&G.n_items, pos.as<int64_t>() + NI, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    TG_CK(cudaStreamSynchronize(s));
    const int64_t ni = std::max<int64_t>(G.n_items, 1);
    G.item_rec.alloc(sizeof(int4) * ni);
    G.item_woff.alloc(sizeof(int64_t) * (G.n_items + 1));
    TBuf icnt(sizeof(int64_t) * (G.n_items + 1), s);
    TG_CK(cudaMemsetAsync(icnt.p, 0, sizeof(int64_t) * (G.n_items + 1), s));
    if (NI > 0) {
        k_hub_items<<<grid_for(NI, 256, 1 << 30), 256, 0, s>>>(gv, NI, cnt.as<int32_t>(), pos.as<int64_t>(),
                                                               sv_of.as<int32_t>(), hub_of.as<int32_t>(),
                                                               G.hubs.as<int32_t>(), G.item_rec.as<int4>(),
                                                               icnt.as<int64_t>());
        TG_CK(cudaGetLastError());
    }
    exclusive_sum(icnt.as<int64_t>(), G.item_woff.as<int64_t>(), G.n_items + 1, s);
    TBuf fi(sizeof(int64_t) * (nh + 1), s), fw(sizeof(int64_t) * (nh + 1), s);
    k_hub_bounds<<<grid_for(nh + 1, 256, 1 << 20), 256, 0, s>>>(nh, L, vbase.as<int64_t>(), pos.as<int64_t>(),
                                                                G.item_woff.as<int64_t>(), fi.as<int64_t>(),
                                                                fw.as<int64_t>());
    TG_CK(cudaGetLastError());
    G.h_hub_nlow.assign(nh, 0);
    TG_CK(cudaMemcpyAsync(G.h_hub_nlow.data(), G.hub_nlow.p, sizeof(int32_t) * nh, cudaMemcpyDeviceToHost, s));
    G.h_hub_item.assign(nh + 1, 0);
    G.h_hub_woff.assign(nh + 1, 0);
    TG_CK(cudaMemcpyAsync(G.h_hub_item.data(), fi.p, sizeof(int64_t) * (nh + 1), cudaMemcpyDeviceToHost, s));
    TG_CK(cudaMemcpyAsync(G.h_hub_woff.data(), fw.p, sizeof(int64_t) * (nh + 1), cudaMemcpyDeviceToHost, s));
    TG_CK(cudaStreamSynchronize(s));
    for (int64_t h = 0; h < nh; ++h)   // the items hold exactly the wedges the build counted
        if (G.h_hub_woff[h + 1] - G.h_hub_woff[h] != G.h_hub_wedges[h]) throw Error{TG_ERR_INTERNAL, "hub wedges"};
    G.hubs_ready = true;
}

// Ticket queues of the persistent hub pass, one per chunk (graph invariant,
// built before any capture): hubs in groups of at most hub_group_max tables
// and about 2^22 wedges; per group, fill and read tickets of at least 2 per
// CTA of the launch (1,024 to 8,192 wedges each) and clear tickets (zeroing
// the group's table words when that is cheaper than walking its wedges
// again).  Queue order: the clears of group s - 2, the reads of group s - 1,
// the fills of group s, for s = 0, 1, ...: every ticket waits on tickets at
// least one phase of another group earlier in the queue.
static void plan_hubs(Graph &G, cudaStream_t s) {
    const int64_t ctas = (int64_t)sm_count() * kHubCtasPerSm;
    G.hub_packed = G.max_degree < 65536;
    G.hub_stride = hub_words_per_table(G);
    // no more tables per buffer than there are hubs (a small graph's budget
    // would otherwise reserve hub_l2_mb for a few hubs)
    const int64_t gmax = std::min<int64_t>(hub_group_max(G), std::max<int64_t>(G.n_hubs, 1));
    G.hub_buf_words = gmax * G.hub_stride;
    const size_t tbytes = sizeof(uint32_t) * (size_t)(kHubBuffers * G.hub_buf_words);
    G.hub_tables.alloc(tbytes);
    TG_CK(cudaMemsetAsync(G.hub_tables.p, 0, tbytes, s));
    G.hub_plans.clear();
    for (const Graph::Chunk &c : G.chunks) {
        auto plan = std::make_unique<Graph::HubPlan>();
        for (DBuf *d : {&plan->segs, &plan->groups, &plan->ntick, &plan->ctr}) d->owner = &G.stream;
        const int64_t hb0 = std::lower_bound(G.h_hub_id.begin(), G.h_hub_id.end(), (int32_t)c.n0) - G.h_hub_id.begin();
        const int64_t hb1 = std::lower_bound(G.h_hub_id.begin(), G.h_hub_id.end(),
                                             (int32_t)std::min<int64_t>(c.n1, INT32_MAX)) - G.h_hub_id.begin();
        std::vector<HubGroup> &groups = plan->h_groups;
        std::vector<int64_t> &ntick = plan->h_ntick;
        for (int64_t h = hb0; h < hb1;) {
            int64_t h1 = h, wsum = 0;
            while (h1 < hb1 && h1 - h < gmax && wsum < ((int64_t)1 << 22)) wsum += G.h_hub_wedges[h1++];
            const int64_t w0 = G.h_hub_woff[h], w1 = G.h_hub_woff[h1];
            if (w1 > w0) {
                HubGroup gr;
                gr.i0 = G.h_hub_item[h];
                gr.i1 = G.h_hub_item[h1];
                gr.w0 = w0;
                gr.w1 = w1;
                gr.tw = std::min<int64_t>(std::max<int64_t>((wsum / (2 * ctas) + 255) & ~(int64_t)255, 1024), 8192);
                gr.zwords = (h1 - h) * G.hub_stride;
                gr.h0 = (int32_t)h;
                gr.buf = (int32_t)(groups.size() % kHubBuffers);
                const int64_t nw = (w1 - w0 + gr.tw - 1) / gr.tw;
                const bool zero = gr.zwords * (int64_t)sizeof(uint32_t) <= 32 * wsum;
                ntick.push_back(nw);                                                     // fill
                ntick.push_back(nw);                                                     // read
                ntick.push_back(zero ? 0 : nw);                                          // clear by walking
                ntick.push_back(zero ? (gr.zwords + kHubTicketWords - 1) / kHubTicketWords : 0);   // clear by zeroing
                groups.push_back(gr);
            }
            h = h1;
        }
        const int64_t ng = (int64_t)groups.size();
        std::vector<HubSegment> &segs = plan->h_segs;
        int64_t nt = 0;
        for (int64_t st = 0; st < ng + 2; ++st) {
            auto emit = [&](int64_t q, int kind) {
                if (q < 0 || q >= ng || ntick[q * kHubKinds + kind] == 0) return;
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
            std::vector<int64_t> pos((size_t)std::max<int64_t>(ng * kHubKinds, 1), -1);
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
        plan->n_groups = ng;
        plan->n_segs = (int64_t)segs.size();
        plan->n_tickets = nt;
        if (ng > 0) {
            plan->segs.alloc(sizeof(HubSegment) * segs.size());
            plan->groups.alloc(sizeof(HubGroup) * groups.size());
            plan->ntick.alloc(sizeof(int64_t) * ntick.size());
            plan->ctr.alloc(sizeof(unsigned long long) * (size_t)(1 + ng * kHubKinds));
            TG_CK(cudaMemcpyAsync(plan->segs.p, segs.data(), sizeof(HubSegment) * segs.size(), cudaMemcpyHostToDevice, s));
            TG_CK(cudaMemcpyAsync(plan->groups.p, groups.data(), sizeof(HubGroup) * groups.size(),
                                  cudaMemcpyHostToDevice, s));
            TG_CK(cudaMemcpyAsync(plan->ntick.p, ntick.data(), sizeof(int64_t) * ntick.size(), cudaMemcpyHostToDevice,
                                  s));
        }
        G.hub_plans.push_back(std::move(plan));
    }
}

// The hubs of chunk ci: one persistent launch over the chunk's tickets.
static int64_t launch_hubs(Graph &G, size_t ci, cudaStream_t s) {
    Graph::HubPlan &P = *G.hub_plans[ci];
    if (P.n_tickets == 0) return 0;
    TG_CK(cudaMemsetAsync(P.ctr.p, 0, sizeof(unsigned long long) * (size_t)(1 + P.n_groups * kHubKinds), s));
    const GraphView gv = G.view();
    const CountView cv = G.cview();
    const HubView hv = hub_view(G);
    const int grid = sm_count() * kHubCtasPerSm;
    KernelTimer kt(G, s, "k_wedge_hub");
    auto launch = [&](auto kern) {
        kern<<<grid, kHubThreads, 0, s>>>(gv, cv, hv, P.segs.as<HubSegment>(), P.n_segs, P.n_tickets,
                                          P.groups.as<HubGroup>(), P.ntick.as<int64_t>(), P.ctr.as<unsigned long long>(),
                                          G.hub_tables.as<uint32_t>(), G.hub_buf_words, G.hub_stride);
    };
    const bool count = cv.work != nullptr;                  // the work-counting form (diagnostics)
    if (G.hub_packed) {
        if (count) launch(k_wedge_hub<true, true>);
        else launch(k_wedge_hub<true, false>);
    } else {
        if (count) launch(k_wedge_hub<false, true>);
        else launch(k_wedge_hub<false, false>);
    }
    TG_CK(cudaGetLastError());
    return 1;
}

static int64_t launch_wedges(Graph &G, const Graph::Chunk &c, cudaStream_t s) {
    G.a_base = c.s0;
    const GraphView gv = G.view();
    const CountView cv = G.cview();
    const int sms = sm_count();
    int64_t launches = 0;
    const int L = G.L;
    if (c.s1 > c.s0)
        TG_CK(cudaMemset2DAsync(G.A.p, (size_t)G.a_stride * sizeof(uint32_t), 0, (size_t)(c.s1 - c.s0) * sizeof(uint32_t),
                                (size_t)L * L, s));
    if (G.n_hubs > 0) launches += launch_hubs(G, (size_t)(&c - G.chunks.data()), s);
    launches += launch_anchor_wedges(G, c.n0, c.n1, s);
    TG_CK(cudaGetLastError());
    return launches;
}

// Allocates the working arrays of a count with this k (kept by the handle).
void prepare_counting(Graph &G, int k, cudaStream_t s) {
    const int L = G.L;
    const size_t m = (size_t)std::max<int64_t>(G.m, 1), n = (size_t)std::max<int64_t>(G.n, 1);
    if (G.C.bytes < m * kCRow * sizeof(uint32_t)) G.C.alloc(m * kCRow * sizeof(uint32_t));
    if (G.tri_any.bytes < n) G.tri_any.alloc(n);
    if (G.tau.bytes < n * L * L * sizeof(int64_t)) G.tau.alloc(n * L * L * sizeof(int64_t));
    prepare_triangles(G);
    const size_t gbytes = (size_t)G.ngraphs * global_slots(L, 4) * sizeof(unsigned long long);
    if (G.gacc.bytes < gbytes) G.gacc.alloc(gbytes);
    if (k == 4) {
        if (G.chunks.empty()) plan_chunks(G);
        const size_t ab = (size_t)G.a_stride * L * L * sizeof(uint32_t);
        if (G.A.bytes < ab) G.A.alloc(ab);
        if (G.slot_rows.bytes < ab) G.slot_rows.alloc(ab);
        const size_t me = (size_t)std::max<int64_t>(G.max_chunk_edges, 1);
        const size_t xb = me * 4 * L * L * (G.wide_sums() ? sizeof(unsigned long long) : sizeof(uint32_t));
        if (G.xsum.bytes < xb) G.xsum.alloc(xb);
        prepare_sums(G);
        if (G.n_hubs > 0 && !G.hubs_ready) prepare_hubs(G, s);
        if (G.n_hubs > 0 && G.hub_plans.empty()) plan_hubs(G, s);
    }
}

int64_t run_count(Graph &G, int k, int64_t e_begin, int64_t e_end, uint32_t *per_edge_out, unsigned long long *gacc,
                  bool full, cudaStream_t s) {
    int64_t launches = 0;
    // prepared_k 3: typed triangles only (all that k = 3 reads); 4: their per-node sums too
    if (full || G.prepared_k < 3 || (k == 4 && !G.tau_ready)) {
        launches += launch_triangles(G, k == 4, s);
        G.prepared_k = std::max(G.prepared_k, 3);
        G.tau_ready = G.tau_ready || k == 4;
    }
    DBuf tmp;                                                // tiles of a range, stream-ordered
    tmp.owner = &G.stream;
    int64_t n_tiles = 0;
    const Tile *tiles = tiles_for(G, e_begin, e_end, n_tiles, tmp, s);
    if (k == 3) {
        launches += launch_edges3(G, tiles, n_tiles, e_begin, per_edge_out, gacc, s);
    } else {
        const bool whole = e_begin == 0 && e_end == G.m;
        std::vector<Tile> host;
        if (!whole) host = make_tiles(G, e_begin, e_end);
        for (const Graph::Chunk &c : G.chunks) {
            const int64_t b = std::max(e_begin, c.e0), e = std::min(e_end, c.e1);
            if (b >= e) continue;
            // the wedge pass and sums of a single-chunk handle are reused by later range calls
            if (full || G.chunks.size() > 1 || G.prepared_k != 4) {
                launches += launch_sums(G, c.n0, c.n1, c.e0, c.e1, s);
                launches += launch_wedges(G, c, s);
                launches += launch_slot_rows(G, c.s1 - c.s0, s);
                if (G.chunks.size() == 1) G.prepared_k = 4;
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
    return launches;
}

}  // namespace tg

// tg_sums.cu -- the sums over the triangle nodes of every edge, and its typed
// 4-cliques, from the local graphs of the lists N+(u) (tg_local.cuh).
//
// For every edge e = (i, j), i the endpoint of lower priority, and every type
// t with c_e^t > 0, row t of e holds 4 L words:
//   [0][q]  TCi  sum over w in T^t of c_{iw}^q
//   [1][q]  TCj  sum over w in T^t of c_{jw}^q
//   [2][q]  DT   sum over w in T^t of d_w^q
//   [3][q]  K'   K' + K'^T = 2 (ordered adjacent pairs of T^t x T^q)
// Every word fits 32 bits: DT adds up degrees of different nodes, so it is at
// most the number of adjacency entries, below 2^31; TCi and TCj are at most
// DT (c_{iw}^q <= d_w^q); and an unordered adjacent pair of T adds 2 to K' in
// all, so K' is at most twice the number of edges, below 2^31 too.
// A triangle u < a < b adds one 4 L-word term to row ty_b of {u, a}, row ty_a
// of {u, b} and row ty_u of {a, b}: one atomic instruction of 4 L lanes on
// consecutive words each.  The last part counts 4-cliques: with the local
// graph of N+(u) as a bit matrix B (columns grouped by type), the clique's
// other nodes of type q are n_q = popc(B_a & B_b) over type q's words; every
// 4-clique has one lowest node u, and n_q is added to {u, a} and {u, b} (whose
// sums over both nodes of a pair meet every pair twice) and 2 n_q to {a, b}.
// A set lookup per (edge, member, entry of the member's list), which this
// replaces, took 1.4e11 lookups on a 20 M-edge Chung-Lu graph; the words
// ANDed here are fewer than 2e9.
// Measured against one pass over every edge's typed intersection for the sums
// and one over every T list for the cliques: 61.4 + 62.9 + 32.7 -> 25.9 + 1.1
// (zeroing) ms on that graph, 18.2 + 12.0 -> 5.6 + 0.6 ms on 256 dense graphs
// of 14 M edges.  With each node's triangles kept in a list, so that its lists
// are scanned once and every warp step has 32 triangles, 25.3 -> 21.2 ms; with
// the number of types compiled in 18.5 ms (5.6 -> 4.3 ms).  What bounds it now:
// the atomics' instructions (one triangle of 4 L lanes per warp step) and
// their sectors in L2 (three rows of 80 bytes per triangle at L = 5).  Visiting
// the nodes u grouped by type, so that 1 / L of the rows of {a, b} is live,
// changed nothing (21.3 against 21.2 ms).
#include <algorithm>

#include "tg_host.hpp"
#include "tg_local.cuh"

namespace tg {

namespace {

constexpr int kSumWarps = 8;                 // warps per CTA of the warp form

// Per-warp staging of up to 32 triangles: what the lanes of add_terms read
// of each, worked out by one lane per triangle.
struct Stage {
    int64_t *at;                // [32][3] words of X: row ty_b of {u, a}, ty_a of {u, b}, ty_u of {a, b}
    uint32_t *kk;               // [32] list position of a << 16 | of b
    uint32_t *val;              // [32][2 L] triangle counts of {a, b}, then the nodes adjacent to u, a and b by type
};

__host__ __device__ inline size_t stage_words(int L) { return 32 * (7 + 2 * (size_t)L); }

__device__ __forceinline__ Stage stage_carve(uint32_t *mem, int L) {   // mem: 8-byte aligned
    Stage s;
    s.at = reinterpret_cast<int64_t *>(mem);
    s.kk = mem + 32 * 6;
    s.val = s.kk + 32;
    return s;
}

// the first L words of row e (of typed triangle counts by edge, or typed degrees by node)
__device__ __forceinline__ void load_c(const uint32_t *C, int64_t e, int L, uint32_t *out) {
    const uint4 *c = reinterpret_cast<const uint4 *>(C + e * kCRow);
    const uint4 lo = c[0], hi = L > 4 ? c[1] : make_uint4(0, 0, 0, 0);
    out[0] = lo.x;
    if (L > 1) out[1] = lo.y;
    if (L > 2) out[2] = lo.z;
    if (L > 3) out[3] = lo.w;
    if (L > 4) out[4] = hi.x;
    if (L > 5) out[5] = hi.y;
    if (L > 6) out[6] = hi.z;
    if (L > 7) out[7] = hi.w;
}

// the row of a local node: c_{u,node} and its typed degrees, 2 L words
__device__ __forceinline__ void load_vec(const GraphView &g, const uint32_t *C, uint32_t eid, int32_t id, int L,
                                         uint32_t *vec) {
    load_c(C, eid, L, vec);
    load_c(g.tdeg, id, L, vec + L);
}

// stages triangle number i of the warp (nq is filled in by the caller)
__device__ __forceinline__ void stage_put(const CountView &cv, int L, const Stage &s, int i, uint32_t ab, int ka, int kb,
                                          const uint32_t *ent, const uint32_t *eid, uint32_t tu) {
    const int row = 4 * L;
    s.at[3 * i] = ((int64_t)eid[ka] - cv.e_base) * (L * row) + (ent[kb] >> kTypeShift) * row;
    s.at[3 * i + 1] = ((int64_t)eid[kb] - cv.e_base) * (L * row) + (ent[ka] >> kTypeShift) * row;
    s.at[3 * i + 2] = ((int64_t)ab - cv.e_base) * (L * row) + tu * row;
    s.kk[i] = (uint32_t)ka << 16 | (uint32_t)kb;
    load_c(cv.C, ab, L, s.val + i * 2 * L);
}

// Adds the terms of the warp's `cnt` staged triangles.  vec: the local
// nodes' rows, du: the lane's word of u's own typed degrees (component 2).
// Lanes take 4 L words of one triangle, 32 / (4 L) triangles at a time.
template <int kL>
__device__ __forceinline__ void add_terms(uint32_t *X, const Stage &s, int cnt, const uint32_t *vec, uint32_t du,
                                          int lane) {
    constexpr int L = kL;
    const int row = 4 * L, per = 32 / row;
    const int grp = lane / row, comp = lane - grp * row;
    const int k = comp / L, q = comp - k * L;
    const int off = k == 2 ? L + q : q;                     // word of vec (components 0 and 2)
    const int val = k == 3 ? L + q : q;                     // word of the staged values (components 1 and 3)
    uint32_t *Xc = X + comp;
#pragma unroll 2
    for (int i = grp < per ? grp : cnt; i < cnt; i += per) {
        const uint32_t kk = s.kk[i];
        const uint32_t va = vec[(kk >> 16) * 2 * L + off], vb = vec[(kk & 0xffffu) * 2 * L + off];
        const uint32_t sv = s.val[i * 2 * L + val];
        // 0: u's counts of the other node; 1: {a, b}'s counts; 2: degrees; 3: the 4-cliques
        const uint32_t xa = k & 1 ? sv : vb, xb = k & 1 ? sv : va;
        const uint32_t xab = k == 0 ? va : k == 1 ? vb : k == 2 ? du : 2 * sv;
        if (xa) atomicAdd(Xc + s.at[3 * i], xa);
        if (xb) atomicAdd(Xc + s.at[3 * i + 1], xb);
        if (xab) atomicAdd(Xc + s.at[3 * i + 2], xab);
    }
}

// u's typed degree for the lanes of component 2
__device__ __forceinline__ uint32_t own_degree(const GraphView &g, int32_t u, int lane) {
    const int L = g.L, q = lane % L;
    return (lane / L) % 4 == 2 ? (uint32_t)typed_degree(g, u, q) : 0u;
}

// zeroes the rows that will be added to and read: (e, t) with c_e^t > 0
__global__ void __launch_bounds__(256) k_sum_zero(int64_t e0, int64_t e1, int L, const uint32_t *__restrict__ C,
                                                  uint32_t *X) {
    const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t e = e0 + x / kCRow;
    const int t = (int)(x % kCRow);
    if (e >= e1 || t >= L || C[e * kCRow + t] == 0) return;
    uint4 *r = reinterpret_cast<uint4 *>(X + ((e - e0) * L + t) * 4 * L);
    for (int k = 0; k < L; ++k) r[k] = make_uint4(0, 0, 0, 0);
}

// Warp per node u of [n0, n1) with 2 <= |N+(u)| <= kTriWarpMax: the bit
// matrix is one word per local node, type q's columns a mask of that word.
template <int kL>
__global__ void __launch_bounds__(kSumWarps * 32) k_sum_warp(GraphView g, CountView cv, int64_t n0, int64_t n1) {
    extern __shared__ uint32_t sw_smem[];
    constexpr int L = kL;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int per_warp = (int)stage_words(L) + 32 * 2 * L + 32 * 3;   // even: the staging is 8-byte aligned
    uint32_t *mem = sw_smem + wid * per_warp;
    const Stage s = stage_carve(mem, L);
    uint32_t *vec = mem + stage_words(L), *ents = vec + 32 * 2 * L, *eids = ents + 32, *B = eids + 32;
    uint32_t *X = cv.xsum;
    unsigned long long words = 0;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = n0 + ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5); u < n1; u += nw) {
        if (!cv.tri_any[u]) continue;
        const int64_t pb = g.plus_off[u];
        const int p = (int)(g.plus_off[u + 1] - pb);
        if (p > kTriWarpMax) continue;
        const uint32_t ent = lane < p ? (uint32_t)g.plus_adj[pb + lane] : 0xffffffffu;
        const uint32_t eid = lane < p ? (uint32_t)g.plus_eid[pb + lane] : 0u;
        __syncwarp();                                       // the previous node's shared rows are read
        ents[lane] = ent;
        eids[lane] = eid;
        B[lane] = 0u;
        if (lane < p) load_vec(g, cv.C, eid, (int32_t)(ent & (uint32_t)kIdMask), L, vec + lane * 2 * L);
        const uint32_t du = own_degree(g, (int32_t)u, lane);
        const uint32_t tu = g.ty[u];
        uint32_t mask[kMaxL];
#pragma unroll
        for (int q = 0; q < kMaxL; ++q)
            mask[q] = __ballot_sync(0xffffffffu, lane < p && (int)(ent >> kTypeShift) == q);
        __syncwarp();
        const int np = p * (p - 1) / 2;
        // every pair's place in the lower node's list, 32 pairs a round; found pairs as bits
        auto find = [&](int x, int &k, int &l) -> int64_t {
            pair_of(x, k, l);
            const uint32_t ek = ents[k], el = ents[l];
            if ((ek & (uint32_t)kIdMask) > (el & (uint32_t)kIdMask)) { const int y = k; k = l; l = y; }
            return plus_find(g, (int32_t)(ents[k] & (uint32_t)kIdMask), ents[l]);
        };
        uint32_t hits = 0;                                  // bit r: this lane's pair of round r is adjacent
        for (int r = 0; r * 32 < np; ++r) {
            const int x = r * 32 + lane;
            int k, l;
            if (x < np && find(x, k, l) >= 0) {
                hits |= 1u << r;
                atomicOr(&B[k], 1u << l);
                atomicOr(&B[l], 1u << k);
            }
        }
        __syncwarp();
        for (int r = 0; r * 32 < np; ++r) {
            const bool hit = (hits >> r) & 1u;
            const unsigned bal = __ballot_sync(0xffffffffu, hit);
            if (bal == 0) continue;
            if (hit) {
                int k, l;
                const int64_t pos = find(r * 32 + lane, k, l);
                const uint32_t e = (uint32_t)g.plus_eid[pos];
                const int at = __popc(bal & ((1u << lane) - 1u));
                stage_put(cv, L, s, at, e, k, l, ents, eids, tu);
                const uint32_t both = B[k] & B[l];
#pragma unroll
                for (int q = 0; q < kMaxL; ++q)
                    if (q < L) s.val[at * 2 * L + L + q] = __popc(both & mask[q]);
                words += 1;
            }
            __syncwarp();
            add_terms<kL>(X, s, __popc(bal), vec, du, lane);
            __syncwarp();
        }
    }
    if (cv.work && words) atomicAdd(&cv.work[kWorkCliqueProbes], words);
}

// words per row of the bit matrix: every type's columns start at a word; odd,
// so that rows spread over the shared-memory banks
__host__ __device__ inline int bit_words(int cap, int L) { return ((cap + 31) / 32 + L) | 1; }

__host__ __device__ inline size_t sum_bytes(int cap, int lgf, int warps, int L) {
    return 4 * ((((size_t)cap * bit_words(cap, L) + 1) & ~(size_t)1) + (size_t)cap * 2 * L +
                (size_t)warps * stage_words(L) + 2 * kMaxL + 2) +
           local_bytes(cap, lgf, warps);
}

// Triangles of one node: its list positions and the edge of the other two.
struct Found {
    uint32_t ab, kk;
};

__host__ __device__ inline int64_t most_found(int64_t cap) { return cap * (cap - 1) / 2; }

// CTA per listed node u of [n0, n1)
template <int kL, int kThreadsT, bool kSmem>
__global__ void __launch_bounds__(kThreadsT) k_sum_cta(GraphView g, CountView cv, const int32_t *__restrict__ list,
                                                       int64_t n_list, int64_t n0, int64_t n1, int cap, int lgf,
                                                       unsigned char *scratch, int64_t stride) {
    // kSmem: the arrays in shared memory, and in the CTA's global slice the
    // triangles of one node, so that its lists are scanned once; else the
    // arrays in the slice and a second scan
    extern __shared__ uint32_t sc_smem[];
    constexpr int L = kL;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int kWarps = kThreadsT / 32;
    uint32_t *mem = kSmem ? sc_smem : reinterpret_cast<uint32_t *>(scratch + (int64_t)blockIdx.x * stride);
    const int W = bit_words(cap, L);
    uint32_t *B = mem;
    uint32_t *vec = B + (((size_t)cap * W + 1) & ~(size_t)1);
    const Stage s = stage_carve(vec + (size_t)cap * 2 * L + wid * stage_words(L), L);
    int *ws = reinterpret_cast<int *>(vec + (size_t)cap * 2 * L + kWarps * stage_words(L));   // [L + 1] first word of a type
    int *shift = ws + kMaxL + 1;                            // [L] column of list position k of type t: k + shift[t]
    LocalList q;
    local_carve(q, reinterpret_cast<unsigned char *>(ws + 2 * kMaxL + 2), cap, lgf, kWarps, wid);
    uint32_t *X = cv.xsum;
    unsigned long long words = 0;
    __shared__ int s_found, s_next;
    Found *found = reinterpret_cast<Found *>(scratch + (int64_t)blockIdx.x * stride);
    for (int64_t x = blockIdx.x; x < n_list; x += gridDim.x) {
        const int32_t u = list[x];
        if (u < n0 || u >= n1 || !cv.tri_any[u]) continue;  // uniform over the CTA
        const int64_t pb = g.plus_off[u];
        const int p = (int)(g.plus_off[u + 1] - pb);
        const uint32_t tu = g.ty[u];
        const uint32_t du = own_degree(g, u, lane);
        for (int k = threadIdx.x; k < p * W; k += kThreadsT) B[k] = 0u;
        local_load(g, pb, p, q);                            // begins and ends with a barrier
        for (int k = threadIdx.x; k < p; k += kThreadsT)
            load_vec(g, cv.C, q.eid[k], (int32_t)(q.ent[k] & (uint32_t)kIdMask), L, vec + k * 2 * L);
        if (wid == 0) {                                     // the types' columns
            int start = 0, cnt = 0;
            if (lane < L) {
                int lo = 0, hi = p;                         // first entry of type >= lane
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if ((int)(q.ent[mid] >> kTypeShift) < lane) lo = mid + 1; else hi = mid;
                }
                start = lo;
            }
            const int next = __shfl_down_sync(0xffffffffu, start, 1);
            if (lane < L) cnt = (lane == L - 1 ? p : next) - start;
            int inc = (cnt + 31) / 32;
            const int own = inc;
#pragma unroll
            for (int o = 1; o < kMaxL; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane < L) {
                ws[lane] = inc - own;
                shift[lane] = 32 * (inc - own) - start;
                if (lane == L - 1) ws[L] = inc;
            }
        }
        if (threadIdx.x == 0) s_found = s_next = 0;
        __syncthreads();
        auto set_bits = [&](int ka, int kb) {
            const int ca = ka + shift[q.ent[ka] >> kTypeShift], cb = kb + shift[q.ent[kb] >> kTypeShift];
            atomicOr(&B[ka * W + (cb >> 5)], 1u << (cb & 31));
            atomicOr(&B[kb * W + (ca >> 5)], 1u << (ca & 31));
        };
        // stages one triangle per lane that has one and adds the warp's terms
        auto terms = [&](bool hit, uint32_t ab, int ka, int kb) {
            const unsigned bal = __ballot_sync(0xffffffffu, hit);
            if (bal == 0) return;
            if (hit) {
                const int at = __popc(bal & ((1u << lane) - 1u));
                stage_put(cv, L, s, at, ab, ka, kb, q.ent, q.eid, tu);
                const uint32_t *ra = B + ka * W, *rb = B + kb * W;
                int w = 0;
                for (int t = 0; t < L; ++t) {
                    uint32_t n = 0;
                    for (const int we = ws[t + 1]; w < we; ++w) n += __popc(ra[w] & rb[w]);
                    s.val[at * 2 * L + L + t] = n;
                }
                words += (unsigned)w;
            }
            __syncwarp();
            add_terms<kL>(X, s, __popc(bal), vec, du, lane);
            __syncwarp();
        };
        local_pairs(g, p, q, lane, wid, kWarps, [&](bool hit, int ka, int kb, uint32_t pos) {
            if (hit) set_bits(ka, kb);
            if (!kSmem) return;
            const unsigned bal = __ballot_sync(0xffffffffu, hit);
            if (bal == 0) return;
            int at = 0;
            if (lane == 0) at = atomicAdd(&s_found, __popc(bal));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & ((1u << lane) - 1u));
            if (hit) found[at] = Found{(uint32_t)g.plus_eid[pos], (uint32_t)ka << 16 | (uint32_t)kb};
        });
        __syncthreads();
        if (kSmem) {
            const int nf = s_found;
            for (;;) {
                int i = 0;
                if (lane == 0) i = atomicAdd(&s_next, 32);
                i = __shfl_sync(0xffffffffu, i, 0);
                if (i >= nf) break;
                Found f{0, 0};
                if (i + lane < nf) f = found[i + lane];
                terms(i + lane < nf, f.ab, (int)(f.kk >> 16), (int)(f.kk & 0xffffu));
            }
        } else {
            local_pairs(g, p, q, lane, wid, kWarps, [&](bool hit, int ka, int kb, uint32_t pos) {
                terms(hit, hit ? (uint32_t)g.plus_eid[pos] : 0u, ka, kb);
            });
        }
        __syncthreads();
    }
    if (cv.work && words) atomicAdd(&cv.work[kWorkCliqueProbes], words);
}

constexpr size_t kScratchBudget = (size_t)4 << 30;   // global slices of the lists beyond shared memory

int64_t huge_ctas(size_t bytes, int64_t n) {
    return std::max<int64_t>(1, std::min<int64_t>({n, (int64_t)sm_count(), (int64_t)(kScratchBudget / bytes)}));
}

size_t class_bytes(const Graph &G, const LocalClass &c) {
    return (sum_bytes(c.cap, c.lgf, c.threads / 32, G.L) + 15) & ~(size_t)15;
}

size_t warp_bytes(int L) { return sizeof(uint32_t) * kSumWarps * (stage_words(L) + 32 * 2 * (size_t)L + 32 * 3); }

// CTAs of a class and bytes of a CTA's global slice
struct SumShape {
    size_t smem, slice;
    int64_t ctas;
};

SumShape shape_of(const Graph &G, const LocalClass &c, int cls) {
    SumShape r;
    const size_t bytes = class_bytes(G, c);
    if (cls == 2) {
        r.smem = 0;
        r.slice = bytes;
        r.ctas = huge_ctas(bytes, c.n);
    } else {
        r.smem = bytes;
        r.slice = sizeof(Found) * (size_t)most_found(c.cap);
        const int per_sm = std::max(1, std::min<int>(2048 / c.threads, (int)((226u << 10) / (bytes + 1024))));
        r.ctas = std::min<int64_t>(c.n, (int64_t)sm_count() * per_sm);
    }
    return r;
}

template <int kL>
void prepare(Graph &G) {
    raise_smem_limit((const void *)k_sum_warp<kL>, warp_bytes(G.L));
    size_t scratch = 0;
    for (int cls = 0; cls < 3; ++cls) {
        const LocalClass c = local_class(G, cls);
        if (c.n == 0) continue;
        const SumShape r = shape_of(G, c, cls);
        if (cls == 0) raise_smem_limit((const void *)k_sum_cta<kL, kTriMidThreads, true>, r.smem);
        else if (cls == 1) raise_smem_limit((const void *)k_sum_cta<kL, kTriBigThreads, true>, r.smem);
        scratch = std::max(scratch, r.slice * (size_t)r.ctas);
    }
    if (scratch) G.sum_scratch.alloc_once(scratch);
}

template <int kL>
int64_t launch(Graph &G, int64_t n0, int64_t n1, int64_t e0, int64_t e1, cudaStream_t s) {
    G.e_base = e0;
    const GraphView gv = G.view();
    const CountView cv = G.cview();
    const int sms = sm_count();
    int64_t launches = 0;
    if (e1 <= e0) return 0;
    {
        KernelTimer kt(G, s, "k_sum_zero");
        k_sum_zero<<<(unsigned)(((e1 - e0) * kCRow + 255) / 256), 256, 0, s>>>(e0, e1, G.L, cv.C, cv.xsum);
        ++launches;
    }
    KernelTimer kt(G, s, "k_sum");
    {
        const size_t bytes = warp_bytes(G.L);
        const int per_sm = std::max(1, std::min<int>(2048 / (kSumWarps * 32), (int)((220u << 10) / (bytes + 1024))));
        k_sum_warp<kL><<<(unsigned)std::min<int64_t>((n1 - n0 + kSumWarps - 1) / kSumWarps, (int64_t)sms * per_sm * 8),
                         kSumWarps * 32, bytes, s>>>(gv, cv, n0, n1);
        ++launches;
    }
    for (int cls = 0; cls < 3; ++cls) {
        const LocalClass c = local_class(G, cls);
        if (c.n == 0) continue;
        const SumShape r = shape_of(G, c, cls);
        ++launches;
        auto run = [&](auto kern) {
            kern<<<(unsigned)r.ctas, c.threads, r.smem, s>>>(gv, cv, c.list, c.n, n0, n1, c.cap, c.lgf,
                                                             G.sum_scratch.as<unsigned char>(), (int64_t)r.slice);
        };
        if (cls == 0) run(k_sum_cta<kL, kTriMidThreads, true>);
        else if (cls == 1) run(k_sum_cta<kL, kTriBigThreads, true>);
        else run(k_sum_cta<kL, kTriBigThreads, false>);
    }
    TG_CK(cudaGetLastError());
    return launches;
}

}  // namespace

// the kernels are compiled per number of types: the terms' index arithmetic
// is most of their instructions
void prepare_sums(Graph &G) {
    with_types(G.L, [&](auto l) { prepare<decltype(l)::value>(G); });
}

int64_t launch_sums(Graph &G, int64_t n0, int64_t n1, int64_t e0, int64_t e1, cudaStream_t s) {
    int64_t launches = 0;
    with_types(G.L, [&](auto l) { launches = launch<decltype(l)::value>(G, n0, n1, e0, e1, s); });
    return launches;
}

}  // namespace tg

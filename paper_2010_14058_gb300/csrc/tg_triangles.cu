// tg_triangles.cu -- typed triangle counts per edge (Cor. 1) and per node.
//
// c_e^t = |Gamma_i^t cap Gamma_j^t| of every edge e = (i, j): every triangle
// is found once (tg_local.cuh) and adds 1 to the counts of its three edges.
// The counts are rows of kCRow words (one 32-byte sector per edge), so that
// later gathers of a row touch one sector.
// Measured on 20 M-edge Chung-Lu and 30 M-edge block-model graphs against an
// intersection of the typed rows per edge (4.3e9 binary searches): 41.9 ->
// 3.7 ms and 13.3 -> 4.2 ms.  What bounds it now: the scan of the lists (2.6e9
// entries, L2) and one scattered atomic per triangle.
#include <algorithm>

#include "tg_host.hpp"
#include "tg_local.cuh"
#include "tg_visit.cuh"

namespace tg {

namespace {

// kShare warps of a CTA per node u with |N+(u)| <= kTriWarpMax: one pair of
// N+(u) per lane, looked up in the lower node's N+ list.  A warp alone visits
// up to 16 sets of 32 pairs one after another, a chain of dependent reads
// that a graph of few nodes waits for (tri_share).
template <int kShare>
__global__ void __launch_bounds__(256) k_tri_warp(GraphView g, uint32_t *C, uint8_t *any) {
    constexpr int kNodes = 8 / kShare;                      // nodes per CTA at a time
    __shared__ uint8_t s_found[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int64_t u0 = (int64_t)blockIdx.x * kNodes; u0 < g.n; u0 += (int64_t)gridDim.x * kNodes) {
        const int64_t u = u0 + wid / kShare;
        const int64_t pb = u < g.n ? g.plus_off[u] : 0;
        const int p = u < g.n ? (int)(g.plus_off[u + 1] - pb) : kTriWarpMax + 1;
        if (kShare == 1 && p > kTriWarpMax) continue;
        if (kShare == 1 && p < 2) {
            if (lane == 0) any[u] = 0;
            continue;
        }
        bool found = false;
        if (p <= kTriWarpMax && p >= 2) {
            const uint32_t tu = g.ty[u];
            const uint32_t ent = lane < p ? (uint32_t)g.plus_adj[pb + lane] : 0u;
            const uint32_t eid = lane < p ? (uint32_t)g.plus_eid[pb + lane] : 0u;
            const int np = p * (p - 1) / 2;
            for (int x0 = wid % kShare * 32; x0 < np; x0 += 32 * kShare) {
                const int x = x0 + lane;
                int k = 0, l = 0;
                if (x < np) pair_of(x, k, l);
                const uint32_t ek = __shfl_sync(0xffffffffu, ent, k), el = __shfl_sync(0xffffffffu, ent, l);
                const uint32_t dk = __shfl_sync(0xffffffffu, eid, k), dl = __shfl_sync(0xffffffffu, eid, l);
                if (x >= np) continue;
                const bool kl = (ek & (uint32_t)kIdMask) < (el & (uint32_t)kIdMask);
                const int64_t pos = plus_find(g, (int32_t)((kl ? ek : el) & (uint32_t)kIdMask), kl ? el : ek);
                if (pos < 0) continue;
                found = true;
                atomicAdd(&C[(int64_t)dk * kCRow + (el >> kTypeShift)], 1u);
                atomicAdd(&C[(int64_t)dl * kCRow + (ek >> kTypeShift)], 1u);
                atomicAdd(&C[(int64_t)g.plus_eid[pos] * kCRow + tu], 1u);
            }
        }
        found = __any_sync(0xffffffffu, found);
        if (kShare == 1) {
            if (lane == 0) any[u] = found ? 1 : 0;
            continue;
        }
        if (lane == 0) s_found[wid] = found ? 1 : 0;
        __syncthreads();
        if (wid % kShare == 0 && lane == 0 && p <= kTriWarpMax) {
            uint8_t f = 0;
            for (int k = 0; k < kShare; ++k) f |= s_found[wid + k];
            any[u] = f;
        }
        __syncthreads();
    }
}

// Warps per node of k_tri_warp: eight or two where the warps of all nodes then
// still run at once, else one.  3-node passes on kept handles (one warp ->
// shared): 3,398 nodes and 34,547 edges 44.9 -> 38.8 us, 3,000 nodes and
// 60,000 edges 58 -> 46; 700 nodes and 20,000 edges 35 us.  On more nodes the
// warps of other nodes hide the chain.
int tri_share(int64_t n) {
    const int64_t warps = (int64_t)sm_count() * 64;
    return 8 * n <= warps ? 8 : 2 * n <= warps ? 2 : 1;
}

// CTA per listed node u: the counts of u's own edges in shared memory (or,
// kSmem = false, in the CTA's global slice), those of {a, b} added in place.
template <int kThreadsT, bool kSmem>
__global__ void __launch_bounds__(kThreadsT) k_tri_cta(GraphView g, uint32_t *C, uint8_t *any, const int32_t *__restrict__ list,
                                                       int64_t n_list, int cap, int lgf, unsigned char *scratch,
                                                       int64_t stride) {
    extern __shared__ unsigned char tri_smem[];
    const int L = g.L;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int kWarps = kThreadsT / 32;
    LocalList q;
    uint32_t *cnt;
    if (kSmem) {
        cnt = reinterpret_cast<uint32_t *>(tri_smem);
        local_carve(q, tri_smem + (size_t)cap * L * 4, cap, lgf, kWarps, wid);
    } else {
        unsigned char *mem = scratch + (int64_t)blockIdx.x * stride;
        cnt = reinterpret_cast<uint32_t *>(mem);
        local_carve(q, mem + (size_t)cap * L * 4, cap, lgf, kWarps, wid);
    }
    for (int64_t x = blockIdx.x; x < n_list; x += gridDim.x) {
        const int32_t u = list[x];
        const int64_t pb = g.plus_off[u];
        const int p = (int)(g.plus_off[u + 1] - pb);
        const uint32_t tu = g.ty[u];
        for (int k = threadIdx.x; k < p * L; k += kThreadsT) cnt[k] = 0;
        local_load(g, pb, p, q);                            // begins and ends with a barrier
        local_pairs(g, p, q, lane, wid, kWarps, [&](bool hit, int ka, int kb, uint32_t pos) {
            if (!hit) return;
            atomicAdd(&cnt[ka * L + (q.ent[kb] >> kTypeShift)], 1u);
            atomicAdd(&cnt[kb * L + (q.ent[ka] >> kTypeShift)], 1u);
            atomicAdd(&C[(int64_t)g.plus_eid[pos] * kCRow + tu], 1u);
        });
        __syncthreads();
        bool found = false;
        for (int k = threadIdx.x; k < p * L; k += kThreadsT) {
            const uint32_t v = cnt[k];
            if (v) atomicAdd(&C[(int64_t)q.eid[k / L] * kCRow + k % L], v);
            found = found || v;
        }
        found = __syncthreads_or(found);
        if (threadIdx.x == 0) any[u] = found ? 1 : 0;
    }
}

// out[x][t][q] = sum over x's slots s of type t of rows[index[s]][q] (rows of
// kCRow words): with the edges' typed triangle counts tau_x[t][t'] = sum_{w in
// Gamma_x^t} c_{xw}^{t'}, the ordered adjacent pairs inside Gamma_x by type;
// with the nodes' typed degrees delta_x[t][t'] = sum_{w in Gamma_x^t} d_w^t'.
// Eight lanes read one row (a 32-byte sector), so a warp takes four slots at
// a time and a type's sums need two shuffles (a lane per slot with L sums
// each left most lanes idle in segments of a few slots and needed L 64-bit
// warp sums per type: 3.7 ms for delta and 3.0 for tau on a 20 M-edge
// Chung-Lu graph against 0.9 and 1.27).  Rows of more than kLongRow slots: a
// CTA per node.
constexpr int64_t kLongRow = 1024;

__device__ __forceinline__ unsigned long long seg_row_sum(const int32_t *__restrict__ index,
                                                          const uint32_t *__restrict__ rows, int64_t s, int64_t e,
                                                          int64_t step, int q) {
    unsigned long long acc = 0;
    for (; s + 3 * step < e; s += 4 * step) {
        uint32_t v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = __ldg(rows + (int64_t)__ldg(index + s + k * step) * kCRow + q);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc += v[k];
    }
    for (; s < e; s += step) acc += __ldg(rows + (int64_t)__ldg(index + s) * kCRow + q);
    return acc;
}

template <class Out>
__global__ void __launch_bounds__(256) k_row_sums(GraphView g, const int32_t *__restrict__ index,
                                                  const uint32_t *__restrict__ rows, Out *out) {
    const int L = g.L;
    const int lane = threadIdx.x & 31, q = lane & 7, sub = lane >> 3;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; x < g.n; x += nw) {
        const int64_t b = g.rp[x];
        if (g.rp[x + 1] - b > kLongRow) continue;
        int32_t to = lane <= L ? g.toff[x * (L + 1) + lane] : 0;
        for (int t = 0; t < L; ++t) {
            const int64_t s = b + __shfl_sync(0xffffffffu, to, t), e = b + __shfl_sync(0xffffffffu, to, t + 1);
            unsigned long long acc = 0;
            if (e > s) {
                acc = seg_row_sum(index, rows, s + sub, e, 4, q);
                acc += __shfl_xor_sync(0xffffffffu, acc, 8);
                acc += __shfl_xor_sync(0xffffffffu, acc, 16);
            }
            if (lane < L) out[(x * L + t) * L + lane] = (Out)acc;
        }
    }
}

template <class Out>
__global__ void __launch_bounds__(256) k_row_sums_long(GraphView g, const int32_t *__restrict__ index,
                                                       const uint32_t *__restrict__ rows, Out *out) {
    __shared__ unsigned long long part[8][kMaxL];
    __shared__ int64_t found[256];
    __shared__ int n_found;
    const int L = g.L;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, q = lane & 7, sub = lane >> 3;
    // the CTA's nodes are gridDim apart (long rows are the last ids of a
    // graph), looked over 256 at a time
    for (int64_t x0 = blockIdx.x; x0 < g.n; x0 += (int64_t)gridDim.x * 256) {
        if (threadIdx.x == 0) n_found = 0;
        __syncthreads();
        const int64_t y = x0 + (int64_t)threadIdx.x * gridDim.x;
        if (y < g.n && g.rp[y + 1] - g.rp[y] > kLongRow) found[atomicAdd(&n_found, 1)] = y;
        __syncthreads();
        const int n = n_found;
        for (int k = 0; k < n; ++k) {
            const int64_t x = found[k];
            for (int t = 0; t < L; ++t) {
                const int64_t s = seg_begin(g, x, t), e = seg_end(g, x, t);
                unsigned long long acc = seg_row_sum(index, rows, s + wid * 4 + sub, e, 32, q);
                acc += __shfl_xor_sync(0xffffffffu, acc, 8);
                acc += __shfl_xor_sync(0xffffffffu, acc, 16);
                if (lane < kMaxL) part[wid][lane] = acc;
                __syncthreads();
                if (threadIdx.x < L) {
                    unsigned long long sum = 0;
                    for (int w = 0; w < 8; ++w) sum += part[w][threadIdx.x];
                    out[(x * L + t) * L + threadIdx.x] = (Out)sum;
                }
                __syncthreads();
            }
        }
        __syncthreads();                                    // the list is replaced next
    }
}

}  // namespace

int64_t launch_row_sums(Graph &G, const int32_t *index, const uint32_t *rows, void *out, cudaStream_t s) {
    if (G.n == 0) return 0;
    const int sms = sm_count();
    auto launch = [&](auto *o) {
        using Out = std::remove_pointer_t<decltype(o)>;
        k_row_sums<Out><<<(unsigned)std::min<int64_t>((G.n + 7) / 8, (int64_t)sms * 64), 256, 0, s>>>(G.view(), index, rows, o);
        if (G.max_degree <= kLongRow) return 1;
        k_row_sums_long<Out><<<(unsigned)std::min<int64_t>(G.n, (int64_t)sms * 8), 256, 0, s>>>(G.view(), index, rows, o);
        return 2;
    };
    const int64_t launches = G.narrow ? launch(static_cast<uint32_t *>(out)) : launch(static_cast<int64_t *>(out));
    TG_CK(cudaGetLastError());
    return launches;
}

LocalClass local_class(const Graph &G, int cls) {
    LocalClass c;
    c.n = G.tri_count[cls];
    c.list = G.tri_list[cls].as<int32_t>();
    c.threads = cls == 0 ? kTriMidThreads : kTriBigThreads;
    const int pmax = (int)std::max<int64_t>(G.max_nplus, 1);
    if (cls == 0) c.cap = kTriMidMax;
    else if (cls == 1) c.cap = (std::min(pmax, kTriBigMax) + 31) & ~31;
    else c.cap = pmax;
    c.lgf = cls == 0 ? 13 : cls == 1 ? 15 : std::min(22, lg_at_least(64 * (int64_t)c.cap));
    return c;
}

static size_t tri_bytes(const Graph &G, const LocalClass &c) {
    return ((size_t)c.cap * G.L * 4 + local_bytes(c.cap, c.lgf, c.threads / 32) + 15) & ~(size_t)15;
}

int64_t cell_window(Graph &G, DBuf &cells, size_t edge_bytes) {
    if (!cells.p) {
        const int64_t budget = std::max<int64_t>((int64_t)G.opt.cycle_budget_mb << 22, 1);
        int64_t n = std::min<int64_t>(G.m, std::max<int64_t>(budget / (int64_t)edge_bytes, kTile));
        for (;;) {
            try {
                cells.alloc(edge_bytes * (size_t)n);
                break;
            } catch (const Error &e) {                      // no room: half as many edges at a time
                if (e.status != TG_ERR_OOM || n <= kTile) throw;
                n = std::max<int64_t>((n + 1) / 2, kTile);
            }
        }
    }
    const int64_t most = (int64_t)(cells.bytes / edge_bytes);
    const int64_t windows = (G.m + most - 1) / most;
    return (G.m + windows - 1) / windows;
}

void prepare_tri_scratch(Graph &G) {
    const LocalClass c = local_class(G, 2);
    if (c.n > 0) G.tri_scratch.alloc_once(tri_bytes(G, c) * (size_t)std::min<int64_t>(c.n, sm_count()));
}

void prepare_triangles(Graph &G) {
    prepare_tri_scratch(G);
    for (int cls = 0; cls < 2; ++cls) {
        const LocalClass c = local_class(G, cls);
        if (c.n == 0) continue;
        const size_t bytes = tri_bytes(G, c);
        if (cls == 0) raise_smem_limit((const void *)k_tri_cta<kTriMidThreads, true>, bytes);
        else raise_smem_limit((const void *)k_tri_cta<kTriBigThreads, true>, bytes);
    }
}

int64_t launch_triangles(Graph &G, bool with_tau, cudaStream_t s) {
    const GraphView gv = G.view();
    const CountView cv = G.cview();
    const int sms = sm_count();
    int64_t launches = 0;
    if (G.m > 0) {
        KernelTimer kt(G, s, "k_tri");
        TG_CK(cudaMemsetAsync(G.C.p, 0, (size_t)G.m * kCRow * sizeof(uint32_t), s));
        const int share = tri_share(G.n);
        const unsigned grid = (unsigned)std::min<int64_t>((G.n * share + 7) / 8, (int64_t)sms * 64);
        if (share == 8) k_tri_warp<8><<<grid, 256, 0, s>>>(gv, cv.C, cv.tri_any);
        else if (share == 2) k_tri_warp<2><<<grid, 256, 0, s>>>(gv, cv.C, cv.tri_any);
        else k_tri_warp<1><<<grid, 256, 0, s>>>(gv, cv.C, cv.tri_any);
        ++launches;
        for (int cls = 0; cls < 3; ++cls) {
            const LocalClass c = local_class(G, cls);
            if (c.n == 0) continue;
            const size_t bytes = tri_bytes(G, c);
            ++launches;
            if (cls == 2) {
                const int64_t grid = std::min<int64_t>(c.n, sms);
                k_tri_cta<kTriBigThreads, false><<<(unsigned)grid, kTriBigThreads, 0, s>>>(
                    gv, cv.C, cv.tri_any, c.list, c.n, c.cap, c.lgf, G.tri_scratch.as<unsigned char>(), (int64_t)bytes);
                continue;
            }
            auto launch = [&](auto kern) {
                const int per_sm = std::max(1, std::min<int>(2048 / c.threads, (int)((220u << 10) / (bytes + 1024))));
                kern<<<(unsigned)std::min<int64_t>(c.n, (int64_t)sms * per_sm), c.threads, bytes, s>>>(
                    gv, cv.C, cv.tri_any, c.list, c.n, c.cap, c.lgf, nullptr, 0);
            };
            if (cls == 0) launch(k_tri_cta<kTriMidThreads, true>);
            else launch(k_tri_cta<kTriBigThreads, true>);
        }
    }
    if (G.n > 0 && with_tau) {
        KernelTimer kt(G, s, "k_tau");
        launches += launch_row_sums(G, G.slot_eid.as<int32_t>(), cv.C, cv.tau, s);
    }
    TG_CK(cudaGetLastError());
    return launches;
}

}  // namespace tg

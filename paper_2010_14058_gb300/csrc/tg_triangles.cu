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

namespace tg {

namespace {

// Warp per node u with 2 <= |N+(u)| <= kTriWarpMax: one pair of N+(u) per
// lane, looked up in the lower node's N+ list.
__global__ void __launch_bounds__(256) k_tri_warp(GraphView g, uint32_t *C, uint8_t *any) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; u < g.n; u += nw) {
        const int64_t pb = g.plus_off[u];
        const int p = (int)(g.plus_off[u + 1] - pb);
        if (p > kTriWarpMax) continue;
        if (p < 2) {
            if (lane == 0) any[u] = 0;
            continue;
        }
        bool found = false;
        const uint32_t tu = g.ty[u];
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
            const int64_t pos = plus_find(g, (int32_t)((kl ? ek : el) & (uint32_t)kIdMask), kl ? el : ek);
            if (pos < 0) continue;
            found = true;
            atomicAdd(&C[(int64_t)dk * kCRow + (el >> kTypeShift)], 1u);
            atomicAdd(&C[(int64_t)dl * kCRow + (ek >> kTypeShift)], 1u);
            atomicAdd(&C[(int64_t)g.plus_eid[pos] * kCRow + tu], 1u);
        }
        found = __any_sync(0xffffffffu, found);
        if (lane == 0) any[u] = found ? 1 : 0;
    }
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

// Warp per node x: tau_x[t][t'] = sum_{w in Gamma_x^t} c_{xw}^{t'}, the
// ordered adjacent pairs inside Gamma_x by type.
__global__ void __launch_bounds__(256) k_tau(GraphView g, CountView cv) {
    const int lane = threadIdx.x & 31;
    const int L = g.L;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; x < g.n; x += nw) {
        for (int t = 0; t < L; ++t) {
            unsigned long long acc[kMaxL];
#pragma unroll
            for (int q = 0; q < kMaxL; ++q) acc[q] = 0;
            for (int64_t s = seg_begin(g, x, t) + lane; s < seg_end(g, x, t); s += 32) {
                const uint4 *c = reinterpret_cast<const uint4 *>(cv.C + (int64_t)g.slot_eid[s] * kCRow);
                const uint4 lo = c[0];
                acc[0] += lo.x; acc[1] += lo.y; acc[2] += lo.z; acc[3] += lo.w;
                if (L > 4) {
                    const uint4 hi = c[1];
                    acc[4] += hi.x; acc[5] += hi.y; acc[6] += hi.z; acc[7] += hi.w;
                }
            }
#pragma unroll
            for (int q = 0; q < kMaxL; ++q) {
                if (q >= L) break;
                unsigned long long v = acc[q];
                for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
                if (lane == 0) cv.tau[(x * L + t) * L + q] = (int64_t)v;
            }
        }
    }
}

}  // namespace

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

void prepare_triangles(Graph &G) {
    for (int cls = 0; cls < 3; ++cls) {
        const LocalClass c = local_class(G, cls);
        if (c.n == 0) continue;
        const size_t bytes = tri_bytes(G, c);
        if (cls == 0) raise_smem_limit((const void *)k_tri_cta<kTriMidThreads, true>, bytes);
        else if (cls == 1) raise_smem_limit((const void *)k_tri_cta<kTriBigThreads, true>, bytes);
        else if (G.local_scratch.bytes < bytes * (size_t)sm_count()) G.local_scratch.alloc(bytes * (size_t)sm_count());
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
        k_tri_warp<<<(unsigned)std::min<int64_t>((G.n + 7) / 8, (int64_t)sms * 64), 256, 0, s>>>(gv, cv.C, cv.tri_any);
        ++launches;
        for (int cls = 0; cls < 3; ++cls) {
            const LocalClass c = local_class(G, cls);
            if (c.n == 0) continue;
            const size_t bytes = tri_bytes(G, c);
            ++launches;
            if (cls == 2) {
                const int64_t grid = std::min<int64_t>(c.n, sms);
                k_tri_cta<kTriBigThreads, false><<<(unsigned)grid, kTriBigThreads, 0, s>>>(
                    gv, cv.C, cv.tri_any, c.list, c.n, c.cap, c.lgf, G.local_scratch.as<unsigned char>(), (int64_t)bytes);
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
        k_tau<<<(unsigned)std::min<int64_t>((G.n + 7) / 8, (int64_t)sms * 16), 256, 0, s>>>(gv, cv);
        ++launches;
    }
    TG_CK(cudaGetLastError());
    return launches;
}

}  // namespace tg

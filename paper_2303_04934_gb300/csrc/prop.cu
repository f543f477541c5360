// The whole SCC of a graph without hubs in one cooperative launch, and the
// batches that remain after the first SCC of a graph with hubs (prop.cuh).
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "common.cuh"
#include "engine.cuh"
#include "internal.h"
#include "prop.cuh"

namespace scc {
namespace {

constexpr int kPropBlock = 256;
constexpr int kPropRegions = 1024;
constexpr int kPropWarps = kPropBlock / kWarp;
// Arcs per thread up to which searches only pull (a pass over all of them is
// then one hop of every path). Pulling against marking, run alone: 2D torus 524 k
// vertices (6.7 arcs a thread) 19.7 / 21.9 ms, 3D torus 512 k (5.9) 1.35 / 1.50,
// k-NN 200 k x 5 (6.4) 0.88 / 1.02, k-NN 400 k x 3 (7.7) 2.8 / 2.3, 3D torus 1 M
// (11.6) 2.4 / 1.9, 2D torus 1 M (13.5) 31 / 16.
constexpr long long kPropPullArcs = 7;
// Vertices from which the first batch has a head start (of at most n / 4 ns):
// 3D torus 256^3 28 -> 11 ms with it. Below, a search is bound by its hops and
// the wave of the head start would only come on top.
constexpr int kPropHeadMin = 1 << 20;

struct PropDev {
    PropCtl c;
    unsigned int region[kPropRegions];  // active vertices of each of the equal runs of bitmap words
};

struct PropParams {
    PropGraph<PropMax> G;
    uint32_t k0;
    PropDev* dev;
    // fresh: trim, decide by the largest degree, canonical labels into out;
    // otherwise the classes are given in label (kDone: finished), N active
    int fresh;
    const int32_t* label;
    unsigned long long N;
    long long m;
    uint64_t seed;
    int32_t* minid;
    int32_t* out;
};

// The active vertex of rank p (one warp; the regions hold the bitmap's counts).
__device__ int prop_select(const uint32_t* act, long long nw, const unsigned int* region, unsigned long long p) {
    const int lane = lane_id();
    const long long len = (nw + kPropRegions - 1) / kPropRegions;
    int r = 0;
    for (;; r += 32) {  // 32 regions at a time
        if (r >= kPropRegions) return -1;
        const int incl = warp_incl_scan((int)ld_volatile(&region[r + lane]));
        const unsigned int tot = (unsigned int)__shfl_sync(kFull, incl, 31);
        if (p < tot) {
            const uint32_t m = __ballot_sync(kFull, (unsigned int)incl > (unsigned int)p);
            const int j = __ffs(m) - 1;
            p -= j ? (unsigned int)__shfl_sync(kFull, incl, j - 1) : 0u;
            r += j;
            break;
        }
        p -= tot;
    }
    for (long long b = r * len; b < min((r + 1) * len, nw); b += 32) {
        const uint32_t x = b + lane < min((r + 1) * len, nw) ? ld_volatile(&act[b + lane]) : 0u;
        const int incl = warp_incl_scan(__popc(x));
        const unsigned int tot = (unsigned int)__shfl_sync(kFull, incl, 31);
        if (p < tot) {
            const uint32_t m = __ballot_sync(kFull, (unsigned int)incl > (unsigned int)p);
            const int j = __ffs(m) - 1;
            const uint32_t xj = __shfl_sync(kFull, x, j);
            const int ej = __shfl_sync(kFull, incl - __popc(x), j);
            return (int)((b + j) * 32 + __fns(xj, 0, (int)p - ej + 1));
        }
        p -= tot;
    }
    return -1;
}

// Two instantiations, so that neither form of the search takes registers from the other.
template <bool kPull>
__global__ void __launch_bounds__(kPropBlock, 4) k_prop(const __grid_constant__ PropParams P) {
    using S = GridScope;
    __shared__ PropShared sh;
    __shared__ unsigned int s_n;
    __shared__ uint32_t s_q[kPropWarps][kPropQueue];
    __shared__ uint32_t s_mk[kPropWarps][kPropMarks];
    const PropGraph<PropMax>& G = P.G;
    PropMax op{P.k0};
    PropCtl* ctl = &P.dev->c;
    const int lane = lane_id();
    uint32_t* q = s_q[threadIdx.x >> 5];
    uint32_t* mk = s_mk[threadIdx.x >> 5];
    // a head start pays where a search is bound by throughput, not by its hops
    const uint64_t head_ns = P.fresh && G.n >= kPropHeadMin && !kPull ? (uint64_t)(G.n / 4) : 0;
    const PropSlice sl = prop_slice<S>(G.n);
    unsigned long long active = P.N;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    // ---- state of every vertex; with fresh, vertices without in- or out-arcs
    // are finished (Sec. 4.1)
    {
        const long long len = (sl.nw + kPropRegions - 1) / kPropRegions;
        unsigned int cnt = 0, mx = 0;
        unsigned long long best = 0;  // the vertex of the largest smaller degree
        for (long long i = 0; i < sl.cnt; ++i) {
            const long long w = sl.word(i), v = w * 32 + lane;
            if (w >= sl.nw) break;
            bool a = false;
            uint32_t lab = 0;
            if (v < G.n) {
                if (P.fresh) {
                    const int d0 = G.off[0][v + 1] - G.off[0][v], d1 = G.off[1][v + 1] - G.off[1][v];
                    a = d0 > 0 && d1 > 0;
                    mx = max(mx, (unsigned int)max(d0, d1));
                    if (head_ns && a) best = max(best, prop_pack((uint32_t)min(d0, d1), op.key((uint32_t)v)));
                    G.rep[v] = (int)v;
                    P.minid[v] = (int)v;
                } else {
                    const int32_t l = P.label[v];
                    a = l >= 0;
                    lab = (uint32_t)l;
                }
                const unsigned long long st =
                    a ? prop_pack(lab, head_ns ? 0u : op.key((uint32_t)v)) : PropMax::none();
                G.s[0][v] = st;
                G.s[1][v] = st;
            }
            const uint32_t m = __ballot_sync(kFull, a);
            if (lane == 0) {
                G.act[w] = m;
                G.d[0][w] = 0;
                G.d[1][w] = 0;
                cnt += __popc(m);
                if (P.fresh && m) atomicAdd(&P.dev->region[w / len], (unsigned int)__popc(m));
            }
        }
        if (P.fresh) {
            for (int d = 16; d >= 1; d >>= 1) {
                mx = max(mx, __shfl_xor_sync(kFull, mx, d));
                best = max(best, __shfl_xor_sync(kFull, best, d));
            }
            if (lane == 0) {
                atomicAdd(&s_n, cnt);
                atomicMax(&ctl->max_deg, mx);
                if (best) atomicMax(&ctl->best, best);
            }
            __syncthreads();
            if (threadIdx.x == 0 && s_n) atomicAdd(&ctl->active0, (unsigned long long)s_n);
        }
        if (!S::sync(&ctl->bar, &ctl->err)) return;
    }
    if (P.fresh) {
        active = ld_volatile(&ctl->active0);
        // that vertex becomes the largest source
        if (head_ns && active > 0) op.k0 = op.vertex((uint32_t)ld_volatile(&ctl->best)) ^ prop_unmix(0xffffffffu);
        const unsigned long long md = ld_volatile(&ctl->max_deg);
        if (prop_skewed(md, (unsigned long long)G.n, (unsigned long long)P.m)) {
            if (blockIdx.x == 0 && threadIdx.x == 0) ctl->status = 1;
            return;
        }
        // the first pivot of the seeded order: statistics only (its SCC's
        // size), found before any bit is cleared
        if (active > 0 && blockIdx.x == 0 && threadIdx.x < 32) {
            Feistel f;
            f.init(P.seed, active);
            const int v = prop_select(G.act, sl.nw, P.dev->region, f.perm(0, active));
            if (lane == 0) ctl->pivot = v;
        }
        if (!S::sync(&ctl->bar, &ctl->err)) return;
    }
    if (!prop_batches<S, kPull>(G, op, ctl, sh, q, mk, active, head_ns)) return;
    if (!P.fresh) return;
    // ---- canonical labels: the smallest vertex of each SCC
    const int proot = active > 0 && ld_volatile(&ctl->pivot) >= 0 ? ld_volatile(&G.rep[ld_volatile(&ctl->pivot)]) : -1;
    unsigned int first = 0;
    int last = -1;
    for (long long i = 0; i < sl.cnt; ++i) {
        const long long w = sl.word(i), v = w * 32 + lane;
        if (w >= sl.nw) break;
        const int r = v < G.n ? G.rep[v] : -1;
        first += r >= 0 && r == proot;
        const bool ok = r >= 0 && r != (int)v;
        const uint32_t okm = __ballot_sync(kFull, ok);
        if (okm == 0) continue;
        const int key0 = __shfl_sync(kFull, r, __ffs(okm) - 1);
        const uint32_t peers = __ballot_sync(kFull, ok && r != key0) == 0 ? okm : __match_any_sync(kFull, ok ? r : -1);
        if (ok && lane == __ffs(peers & okm) - 1 && r != last) {
            last = r;
            if (ld_volatile(&P.minid[r]) > (int)v) atomicMin(&P.minid[r], (int)v);
        }
    }
    for (int d = 16; d >= 1; d >>= 1) first += __shfl_xor_sync(kFull, first, d);
    if (lane == 0 && first) atomicAdd(&ctl->first, first);
    if (!S::sync(&ctl->bar, &ctl->err)) return;
    for (long long i = 0; i < sl.cnt; ++i) {
        const long long v = sl.word(i) * 32 + lane;
        if (v < G.n) P.out[v] = ld_volatile(&P.minid[G.rep[v]]);
    }
}

}  // namespace

size_t prop_dev_bytes() { return sizeof(PropDev); }

// Whether the searches of a graph without hubs only pull.
bool prop_pulls(long long m, int num_sms) { return m <= kPropPullArcs * 4ll * num_sms * kPropBlock; }

int run_prop(const PropArgs& a, PropResult* res, cudaStream_t st) {
    PropParams P;
    memset(&P, 0, sizeof(P));
    P.G = PropGraph<PropMax>{{a.off, a.toff}, {a.adj, a.tadj}, a.n, {a.sf, a.sb}, {a.df, a.db}, a.act, a.rep};
    P.k0 = (uint32_t)mix64(a.seed);
    P.dev = reinterpret_cast<PropDev*>(a.dev);
    P.fresh = a.label == nullptr;
    P.label = a.label;
    P.N = (unsigned long long)a.N;
    P.m = a.m;
    P.seed = a.seed;
    P.minid = a.minid;
    P.out = a.out;
    static int per_sm = -1;
    if (per_sm < 0) {  // of the two forms, the fewer
        int x = 0, y = 0;
        SCC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&x, k_prop<false>, kPropBlock, 0));
        SCC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&y, k_prop<true>, kPropBlock, 0));
        if (std::min(x, y) < 1) return SCC_ERR_CUDA;
        per_sm = std::min(x, y);
    }
    const long long nw = ((long long)a.n + 31) / 32;
    const int full = per_sm * a.num_sms;
    const int grid = (int)std::max<long long>(1, std::min<long long>(full, (nw + kPropWarps - 1) / kPropWarps));
    const bool pull = a.pull;
    SCC_CUDA(cudaMemsetAsync(P.dev, 0, sizeof(PropDev), st));
    void* args[] = {(void*)&P};
    SCC_CUDA(cudaLaunchCooperativeKernel(pull ? (const void*)k_prop<true> : (const void*)k_prop<false>, dim3(grid), dim3(kPropBlock), args, 0, st));
    count_launch();
    PropCtl c;
    SCC_CUDA(cudaMemcpyAsync(&c, P.dev, sizeof(c), cudaMemcpyDeviceToHost, st));
    SCC_CUDA(cudaStreamSynchronize(st));
    if (c.err) return c.err;
    res->status = c.status;
    res->active = (int64_t)c.active0;
    res->first = (int32_t)c.first;
    res->batches = c.batches;
    res->searches = c.searches;
    res->items = c.items;
    res->arcs = c.arcs;
    return SCC_OK;
}

}  // namespace scc

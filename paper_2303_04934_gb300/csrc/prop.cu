// The whole SCC of a graph without hubs in one cooperative launch, and the
// batches that remain after the first SCC of a graph with hubs (prop.cuh).
#include <algorithm>
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
// Arcs per thread up to which searches only pull (a pass over all of them is then
// one hop of every path), pulling against marking, ms. scc_run: 2D torus 63 k vertices
// 1.38 / 2.55, 155 k 1.35 / 1.58, 262 k 1.8 / 1.7, DAG of 131 k vertices (387 k arcs, 2.5 a
// thread) 1.02 / 1.34, k-NN 200 k x 5 (6.4) 0.83 / 0.83, but 3D torus 262 k (472 k arcs, 3)
// 1.18 / 0.91, 2D 423 k 3.44 / 2.11. reach_multi, 64 sources: 2D torus 262 k (3.4) 2.98 /
// 4.44, 360 k (4.6) 4.00 / 4.27, 3D 512 k (5.9) 0.56 / 0.65, but 2D 524 k (6.7) 8.02 / 6.51,
// k-NN 200 k x 5 0.40 / 0.30. Since warps relax narrow waves themselves (kPropNarrow)
// marking is ahead on some graphs from 3 arcs a thread on; on others pulling still is.
constexpr long long kPropPullArcs = 7;
// ... in reach_multi on graphs of about one arc a vertex, long paths, above all:
// cycles of 300 k vertices, one source and 7: 764 / 526, 337 / 526, of 524 k 1559 / 917,
// 846 / 916 (by rounds of the engine 1233, 1244).
constexpr long long kReachPullPath = 3;
// Vertices from which the first batch has a head start (of at most n / 4 ns):
// 3D torus 256^3 28 -> 11 ms with it. Below, a search is bound by its hops and
// the wave of the head start would only come on top.
constexpr int kPropHeadMin = 1 << 20;

struct PropDev {
    PropCtl c;
    unsigned int region[kPropRegions];  // active vertices of each of the equal runs of bitmap words
};

// The graph contracted along mutual arcs (prop_contract).
struct PropCon {
    int32_t* cid;      // n: a vertex's node, -1 when it is not active
    int32_t* lead;     // n: the smallest vertex of a node
    int32_t* beg[2];   // n: a node's row, in the graph and in its transpose
    int32_t* end[2];   // n (the number of its arcs, then where the next arc goes)
    int32_t* adj[2];   // m
    int32_t* rep;      // n: a node of the node's SCC
    int32_t* min;      // n: the smallest vertex of the SCC (by rep)
    uint32_t* act;     // n / 32
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
    unsigned long long pull_arcs;  // up to so many arcs the searches only pull
    unsigned long long arcs;  // arcs of the graphs without hubs (m, but in a group)
    uint64_t seed;
    int32_t* minid;
    int32_t* out;
    PropCon con;  // fresh
    // fresh, a group of a batch's graphs as one graph (null: one graph): labels
    // of the graphs with mesh[g], from their own first vertex, into out
    const long long* vbase;
    const unsigned char* mesh;
    int g0, g1;
    unsigned long long* times;
    int time_words;
    uint64_t idle_ns;
};

// The group's graph that holds vertex v (the last one that starts at or before it).
__device__ __forceinline__ int prop_graph_of(const PropParams& P, long long v) {
    const long long x = P.vbase[P.g0] + v;
    int lo = P.g0, hi = P.g1;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (P.vbase[mid] <= x) lo = mid;
        else hi = mid;
    }
    return lo;
}

// The records of the group's graphs: their searches share the launch's time.
__device__ __forceinline__ void prop_times(const PropParams& P, uint64_t t0) {
    if (P.times == nullptr || blockIdx.x != 0) return;
    for (int g = P.g0 + (int)threadIdx.x; g < P.g1; g += blockDim.x)
        if (P.mesh[g]) {
            unsigned long long* t = P.times + (size_t)P.time_words * g;
            for (int k = 0; k < P.time_words; ++k) t[k] = k < 5 ? t0 : 0;
            t[5] = globaltimer_ns();
        }
}

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

// A cooperative grid that also reads graph arrays it wrote itself.
struct PropScope : PropGrid {
    __device__ __forceinline__ static int32_t ld(const int32_t* p) { return *p; }
};

// ------------------------------------------------------------ contraction --
// The root of v's set (parents only ever shrink, so the walk ends).
__device__ __forceinline__ int con_find(int32_t* p, int v) {
    for (;;) {
        const int a = ld_volatile(&p[v]);
        if (a == v) return v;
        const int b = ld_volatile(&p[a]);
        if (b == a) return a;
        *(volatile int32_t*)&p[v] = b;  // path halving: b is further up, and smaller
        v = b;
    }
}
// The same after the unions, read-only: a halving store from a walk that started
// earlier could put an inner vertex back over a root already stored.
__device__ __forceinline__ int con_root(const int32_t* p, int v) {
    for (;;) {
        const int a = ld_volatile(&p[v]);
        if (a == v) return v;
        v = a;
    }
}
__device__ __forceinline__ bool con_unite(int32_t* p, int a, int b) {
    for (;;) {
        a = con_find(p, a);
        b = con_find(p, b);
        if (a == b) return false;
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        if (atomicCAS(&p[a], a, b) == a) return true;
    }
}

// Vertices joined by mutual arcs lie in one SCC, so they can be one vertex of the
// searches. On a lattice or a k-NN graph many arcs are mutual: merging along
// them leaves a 2D torus (p = 0.5) half of its vertices and k-NN (k = 5) 2%, and
// takes more than that off the searches' hops and raises, which is what they
// cost (2D torus 512^2, rounds of a synchronous model: 2570 -> 1051 hops, 6.2 M ->
// 1.1 M raises). A 3D torus (p = 0.3) keeps three quarters and gains less than
// building the contracted rows costs; so a sixteenth of the words is tried
// first, and the graph is contracted when two fifths of its vertices have a
// smaller mutual neighbour (2D torus 47%, 3D 31%, k-NN 78%). Run alone: 2D torus
// 512^2 6.0 -> 2.2 ms, 724^2 17.9 -> 4.8, 1227^2 25 -> 12, k-NN 1 M x 5 1.8 -> 1.3.
//
// Union-find over the mutual arcs (found by looking each out-neighbour up in the
// vertex's in-row, both rows at hand; the first kConRow arcs of each are enough):
// a forest of smallest neighbours first, by plain stores, then the arcs it left
// open; uniting all arcs from single vertices took k-NN's (1 M x 5) walks through
// long chains of parents, 0.90 ms. Then nodes numbered in vertex order within a warp's words, then rows: counted,
// placed by one counter per warp, filled. A node's arcs keep their multiplicity.
constexpr int kConRow = 32;
constexpr unsigned kConSample = 16;  // one word in so many
// Mean row up to which the searches of a contracted graph may only pull: k-NN (1 M
// x 5) keeps 3,845 nodes with 8 arcs each, most of them at a few large clusters,
// whose rows a pull reads in every pass (first batch 407 against 242 us).
constexpr unsigned kConPullRow = 4;
// Vertices from which a graph is contracted: the passes take 50-110 us on small
// ones, which critical lattices get back early and others late. The run with it /
// without, us, at 8 k, 16 k, 33 k, 50 k, 66 k and 90 k vertices: 2D torus p = 0.5 347 /
// 326, 419 / 462, 620 / 735, 749 / 830, 766 / 1057, 1135 / 1542; p = 0.65 197 / 119, 216 /
// 143, 245 / 173, 266 / 205, 284 / 233, 306 / 276; k-NN k = 5 212 / 177, 243 / 186, 294 /
// 221, 331 / 310, 358 / 325, 396 / 431; k = 3 231 / 237, 288 / 313, 356 / 356, 389 / 518, 421
// / 612, 462 / 807; graphs that are tried and not contracted +2%.
constexpr int kConMin = 1 << 16;

template <class S>
__device__ bool prop_contract(const PropGraph<PropMax>& G, const PropCon& C, PropCtl* ctl, unsigned long long active,
                              bool* done) {
    const int lane = lane_id();
    const PropSlice P = prop_slice<S>(G.n);
    int32_t* parent = G.rep;
    *done = false;
    // f(v, u) for the mutual arcs of v to smaller vertices
    auto mutual = [&](int v, auto&& f) {
        const int o0 = G.off[0][v], o1 = o0 + min(G.end[0][v] - o0, kConRow);
        const int i0 = G.off[1][v], i1 = i0 + min(G.end[1][v] - i0, kConRow);
        for (int e = o0; e < o1; ++e) {
            const int u = G.adj[0][e];
            if (u >= v) continue;
            bool in = false;
            for (int k = i0; k < i1 && !in; ++k) in = G.adj[1][k] == u;
            if (in) f(u);
        }
    };
    // ---- every vertex under its smallest mutual neighbour that is smaller than
    // itself: a forest, by plain stores, whose edges are so many merges for
    // certain; in a sample of the words and then in the others
    const bool sample = P.nw >= 64 * kConSample;
    unsigned long long merged = 0;
    for (int part = sample ? 0 : 1; part < 2; ++part) {
        unsigned int got = 0;
        for (long long i = 0; i < P.cnt; ++i) {
            const long long w = P.word(i);
            if (w >= P.nw) break;
            if (sample && ((w % kConSample) == 0) != (part == 0)) continue;
            if (!((G.act[w] >> lane) & 1u)) continue;
            const int v = (int)(w * 32) + lane;
            int least = v;
            mutual(v, [&](int u) { least = min(least, u); });
            if (least < v) {
                *(volatile int32_t*)&parent[v] = least;
                ++got;
            }
        }
        __syncwarp();
        got = __reduce_add_sync(kFull, got);
        if (lane == 0 && got) atomicAdd(&ctl->merged[part], got);
        unsigned long long m;
        if (!S::sync_then(&ctl->bar, &ctl->err, m, [&] { return (unsigned long long)ld_volatile(&ctl->merged[part]); }))
            return false;
        if (part == 0 && m * kConSample * 5 < active * 2) return true;
        if (part == 1 && !sample && m * 5 < active * 2) return true;
        merged += m;
    }
    // ---- the forest's roots, then the other mutual arcs: most of their ends
    // have one root by now, and the walks are short
    auto flatten = [&]() {
        for (long long i = 0; i < P.cnt; ++i) {
            const long long w = P.word(i);
            if (w >= P.nw) break;
            if (!((G.act[w] >> lane) & 1u)) continue;
            const int v = (int)(w * 32) + lane;
            const int r = con_root(parent, v);
            if (r != v) *(volatile int32_t*)&parent[v] = r;
        }
        __syncwarp();
    };
    flatten();
    if (!S::sync(&ctl->bar, &ctl->err)) return false;
    // rounds that put every root under the smallest root beside it, while a
    // round merges a sixteenth of the vertices. A link that a smaller one
    // replaces is made again below, where every arc is looked at once more
    for (int r = 0; merged * 16 >= active; r = r == 2 ? 0 : r + 1) {
        unsigned int got = 0;
        for (long long i = 0; i < P.cnt; ++i) {
            const long long w = P.word(i);
            if (w >= P.nw) break;
            if (!((G.act[w] >> lane) & 1u)) continue;
            const int v = (int)(w * 32) + lane;
            const int a = parent[v];
            mutual(v, [&](int u) {
                const int b = parent[u], hi = max(a, b), lo = min(a, b);
                if (hi != lo && ld_volatile(&parent[hi]) > lo) got += atomicMin(&parent[hi], lo) == hi;
            });
        }
        __syncwarp();
        got = __reduce_add_sync(kFull, got);
        if (S::block() == 0 && threadIdx.x == 0) ctl->hooked[(r + 1) % 3] = 0;
        if (lane == 0 && got) atomicAdd(&ctl->hooked[r], got);
        if (!S::sync_then(&ctl->bar, &ctl->err, merged,
                          [&] { return (unsigned long long)ld_volatile(&ctl->hooked[r]); }))
            return false;
        flatten();
        if (!S::sync(&ctl->bar, &ctl->err)) return false;
    }
    for (long long i = 0; i < P.cnt; ++i) {
        const long long w = P.word(i);
        if (w >= P.nw) break;
        if (!((G.act[w] >> lane) & 1u)) continue;
        const int v = (int)(w * 32) + lane;
        mutual(v, [&](int u) {
            if (ld_volatile(&parent[u]) != ld_volatile(&parent[v])) con_unite(parent, u, v);
        });
    }
    __syncwarp();
    if (!S::sync(&ctl->bar, &ctl->err)) return false;
    // ---- roots; a warp's nodes are numbered together
    flatten();
    unsigned int mine = 0;
    for (long long i = 0; i < P.cnt; ++i) {
        const long long w = P.word(i);
        if (w >= P.nw) break;
        const int v = (int)(w * 32) + lane;
        mine += __popc(__ballot_sync(kFull, ((G.act[w] >> lane) & 1u) && ld_volatile(&parent[v]) == v));
    }
    unsigned int base = 0;
    if (lane == 0 && mine) base = atomicAdd(&ctl->nodes, mine);
    base = __shfl_sync(kFull, base, 0);
    for (long long i = 0; i < P.cnt; ++i) {
        const long long w = P.word(i);
        if (w >= P.nw) break;
        const int v = (int)(w * 32) + lane;
        const bool root = ((G.act[w] >> lane) & 1u) && ld_volatile(&parent[v]) == v;
        const uint32_t m = __ballot_sync(kFull, root);
        if (root) {
            const unsigned int c = base + __popc(m & lanemask_lt());
            C.cid[v] = (int)c;
            C.lead[c] = v;
            C.end[0][c] = 0;
            C.end[1][c] = 0;
        }
        base += __popc(m);
    }
    if (!S::sync(&ctl->bar, &ctl->err)) return false;
    const unsigned int n2 = ld_volatile(&ctl->nodes);
    // ---- arcs between nodes, counted; every vertex learns its node
    for (long long i = 0; i < P.cnt; ++i) {
        const long long w = P.word(i);
        if (w >= P.nw) break;
        if (!((G.act[w] >> lane) & 1u)) continue;
        const int v = (int)(w * 32) + lane;
        const int r = parent[v];
        const int a = C.cid[r];
        if ((unsigned int)a >= n2) {  // never: r is a root, and every root has a node
            atomicCAS(&ctl->err, 0, SCC_ERR_INTERNAL);
            continue;
        }
        if (r != v) *(volatile int32_t*)&C.cid[v] = a;
        const int o0 = G.off[0][v], o1 = G.end[0][v];
        int cnt = 0;
        row_steps<4>(o0, o1, 0, 1, [&](const uint32_t (&x)[4]) {
            int u[4], b[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) u[k] = x[k] != kNoArc ? G.adj[0][x[k]] : -1;
#pragma unroll
            for (int k = 0; k < 4; ++k) b[k] = u[k] >= 0 ? parent[u[k]] : -1;
#pragma unroll
            for (int k = 0; k < 4; ++k) b[k] = b[k] >= 0 ? C.cid[b[k]] : -1;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if ((unsigned int)b[k] < n2 && b[k] != a) {
                    ++cnt;
                    atomicAdd(&C.end[1][b[k]], 1);
                }
        });
        if (cnt) atomicAdd(&C.end[0][a], cnt);
    }
    __syncwarp();
    if (!S::sync(&ctl->bar, &ctl->err)) return false;
    // ---- a warp's nodes get their rows together
    const PropSlice Q = prop_slice<S>((int32_t)n2);
#pragma unroll 1
    for (int d = 0; d < 2; ++d) {
        unsigned int sum = 0, most = 0;
        for (long long i = 0; i < Q.cnt; ++i) {
            const long long c = Q.word(i) * 32 + lane;
            const unsigned int k = c < n2 ? (unsigned int)ld_volatile(&C.end[d][c]) : 0u;
            sum += k;
            most = max(most, k);
        }
        sum = __reduce_add_sync(kFull, sum);
        most = __reduce_max_sync(kFull, most);
        if (lane == 0 && most > (unsigned int)kPropHub) atomicMax(&ctl->max_row2, most);
        unsigned int at = 0;
        if (lane == 0 && sum) at = atomicAdd(&ctl->arcs2[d], sum);
        at = __shfl_sync(kFull, at, 0);
        for (long long i = 0; i < Q.cnt; ++i) {
            const long long w = Q.word(i), c = w * 32 + lane;
            if (w >= Q.nw) break;
            const int k = c < n2 ? ld_volatile(&C.end[d][c]) : 0;
            const int incl = warp_incl_scan(k);
            if (c < n2) {
                C.beg[d][c] = (int)at + incl - k;
                C.end[d][c] = (int)at + incl - k;
            }
            at += (unsigned int)__shfl_sync(kFull, incl, 31);
        }
    }
    if (!S::sync(&ctl->bar, &ctl->err)) return false;
    const unsigned int arcs = ld_volatile(&ctl->arcs2[0]);
    // ---- the rows; afterwards end[d][c] is where row c ends
    for (long long i = 0; i < P.cnt; ++i) {
        const long long w = P.word(i);
        if (w >= P.nw) break;
        if (!((G.act[w] >> lane) & 1u)) continue;
        const int v = (int)(w * 32) + lane;
        const int a = ld_volatile(&C.cid[v]);
        if ((unsigned int)a >= n2) continue;
        const int o0 = G.off[0][v], o1 = G.end[0][v];
        row_steps<4>(o0, o1, 0, 1, [&](const uint32_t (&x)[4]) {
            int b[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) b[k] = x[k] != kNoArc ? G.adj[0][x[k]] : -1;
#pragma unroll
            for (int k = 0; k < 4; ++k) b[k] = b[k] >= 0 ? ld_volatile(&C.cid[b[k]]) : -1;
            int p[4], t[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool arc = (unsigned int)b[k] < n2 && b[k] != a;
                p[k] = arc ? atomicAdd(&C.end[0][a], 1) : -1;
                t[k] = arc ? atomicAdd(&C.end[1][b[k]], 1) : -1;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (p[k] >= 0 && (unsigned int)max(p[k], t[k]) < arcs) {
                    C.adj[0][p[k]] = b[k];
                    C.adj[1][t[k]] = a;
                }
        });
    }
    __syncwarp();
    if (!S::sync(&ctl->bar, &ctl->err)) return false;
    *done = true;
    return ld_volatile(&ctl->err) == 0;
}

// The state of the contracted graph's nodes: all active, in one class.
template <class S>
__device__ __forceinline__ void prop_node_state(const PropGraph<PropMax>& N, const PropMax& op, const PropCon& C) {
    const PropSlice Q = prop_slice<S>(N.n);
    for (long long i = 0; i < Q.cnt; ++i) {
        const long long w = Q.word(i), c = w * 32 + lane_id();
        if (w >= Q.nw) break;
        if (c < N.n) {
            const unsigned long long st = prop_pack(0, op.key((uint32_t)c));
            N.s[0][c] = st;
            N.s[1][c] = st;
            C.rep[c] = (int)c;
            C.min[c] = C.lead[c];
        }
        const uint32_t m = __ballot_sync(kFull, c < N.n);
        if (lane_id() == 0) {
            N.act[w] = m;
            N.d[0][w] = 0;
            N.d[1][w] = 0;
        }
    }
}

// The contracted graph's nodes as a graph.
__device__ __forceinline__ PropGraph<PropMax> prop_nodes(const PropParams& P, const PropCtl* ctl) {
    const PropCon& C = P.con;
    PropGraph<PropMax> N;
    for (int d = 0; d < 2; ++d) {
        N.off[d] = C.beg[d];
        N.end[d] = C.end[d];
        N.adj[d] = C.adj[d];
        N.s[d] = P.G.s[d];
        N.d[d] = P.G.d[d];
    }
    N.n = (int32_t)ld_volatile(&ctl->nodes);
    N.act = C.act;
    N.rep = C.rep;
    return N;
}

// The labels of all vertices from the SCCs of the nodes.
template <class S>
__device__ __forceinline__ bool prop_node_labels(const PropParams& P, const PropGraph<PropMax>& N, PropCtl* ctl) {
    const int lane = lane_id();
    const PropCon& C = P.con;
    const PropGraph<PropMax>& G = P.G;
    const PropSlice sl = prop_slice<S>(G.n);
    const PropSlice Q = prop_slice<S>(N.n);
    for (long long i = 0; i < Q.cnt; ++i) {
        const long long w = Q.word(i), c = w * 32 + lane;
        if (w >= Q.nw) break;
        const int r = c < N.n ? C.rep[c] : -1;
        const unsigned int x = c < N.n ? (unsigned int)C.lead[c] : 0u;
        const uint32_t peers = __match_any_sync(kFull, r);
        const unsigned int least = __reduce_min_sync(peers, x);
        if (r >= 0 && lane == __ffs(peers) - 1 && (unsigned int)ld_volatile(&C.min[r]) > least)
            atomicMin(&C.min[r], (int)least);
    }
    if (!S::sync(&ctl->bar, &ctl->err)) return false;
    auto label = [&](int c) { return ld_volatile(&C.min[ld_volatile(&C.rep[c])]); };
    const int pv = P.vbase == nullptr ? ld_volatile(&ctl->pivot) : -1;
    const int pc = pv >= 0 ? ld_volatile(&C.cid[pv]) : -1;
    const int pl = (unsigned int)pc < (unsigned int)N.n ? label(pc) : -1;
    unsigned int first = 0;
    for (long long i = 0; i < sl.cnt; ++i) {
        const long long v = sl.word(i) * 32 + lane;
        if (v >= G.n) continue;
        int first_v = 0;
        if (P.vbase != nullptr) {
            const int g = prop_graph_of(P, v);
            if (!P.mesh[g]) continue;
            first_v = (int)(P.vbase[g] - P.vbase[P.g0]);
        }
        const int c = ld_volatile(&C.cid[v]);
        const int l = (unsigned int)c < (unsigned int)N.n ? label(c) : (int)v;
        first += l == pl;
        P.out[v] = l - first_v;
    }
    __syncwarp();
    first = __reduce_add_sync(kFull, first);
    if (lane == 0 && first) atomicAdd(&ctl->first, first);
    return true;
}

// The whole run on a graph without hubs.
__global__ void __launch_bounds__(kPropBlock, 4) k_prop(const __grid_constant__ PropParams P) {
    using S = PropScope;
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
    const bool pull = P.arcs <= P.pull_arcs;  // few arcs a thread: the searches only pull
    const uint64_t head_ns = P.vbase == nullptr && G.n >= kPropHeadMin && !pull ? (uint64_t)(G.n / 4) : 0;
    const PropSlice sl = prop_slice<S>(G.n);
    const uint64_t t0 = globaltimer_ns();
    unsigned long long active;
    if (threadIdx.x == 0) {
        s_n = 0;
        sh.idle_ns = P.idle_ns;
    }
    __syncthreads();
    // ---- state of every vertex; vertices without in- or out-arcs are finished
    // (Sec. 4.1)
    {
        const long long len = (sl.nw + kPropRegions - 1) / kPropRegions;
        unsigned int cnt = 0, mx = 0;
        unsigned long long best = 0;  // the vertex of the largest smaller degree
        for (long long i = 0; i < sl.cnt; ++i) {
            const long long w = sl.word(i), v = w * 32 + lane;
            if (w >= sl.nw) break;
            bool a = false;
            if (v < G.n) {
                const int d0 = G.end[0][v] - G.off[0][v], d1 = G.end[1][v] - G.off[1][v];
                a = d0 > 0 && d1 > 0 && (P.vbase == nullptr || P.mesh[prop_graph_of(P, v)]);
                mx = max(mx, (unsigned int)max(d0, d1));
                if (head_ns && a) best = max(best, prop_pack((uint32_t)min(d0, d1), op.key((uint32_t)v)));
                G.rep[v] = (int)v;
                P.minid[v] = (int)v;
                if (!a) P.con.cid[v] = -1;
                const unsigned long long st =
                    a ? prop_pack(0, head_ns ? 0u : op.key((uint32_t)v)) : PropMax::none();
                G.s[0][v] = st;
                G.s[1][v] = st;
            }
            const uint32_t m = __ballot_sync(kFull, a);
            if (lane == 0) {
                G.act[w] = m;
                G.d[0][w] = 0;
                G.d[1][w] = 0;
                cnt += __popc(m);
                if (m) atomicAdd(&P.dev->region[w / len], (unsigned int)__popc(m));
            }
        }
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
        if (!S::sync(&ctl->bar, &ctl->err)) return;
    }
    active = ld_volatile(&ctl->active0);
    // that vertex becomes the largest source
    if (head_ns && active > 0) op.k0 = op.vertex((uint32_t)ld_volatile(&ctl->best)) ^ prop_unmix(0xffffffffu);
    const unsigned long long md = ld_volatile(&ctl->max_deg);
    if (P.vbase == nullptr && prop_skewed(md, (unsigned long long)G.n, (unsigned long long)P.m)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl->status = 1;
        return;
    }
    // the first pivot of the seeded order: statistics only (its SCC's
    // size), found before any bit is cleared
    if (P.vbase == nullptr && active > 0 && blockIdx.x == 0 && threadIdx.x < 32) {
        Feistel f;
        f.init(P.seed, active);
        const int v = prop_select(G.act, sl.nw, P.dev->region, f.perm(0, active));
        if (lane == 0) ctl->pivot = v;
    }
    if (!S::sync(&ctl->bar, &ctl->err)) return;
    bool contracted = false;
    if (active > 0 && G.n >= kConMin && !prop_contract<S>(G, P.con, ctl, active, &contracted)) return;
    if (contracted) {
        const PropGraph<PropMax> N = prop_nodes(P, ctl);
        const unsigned long long arcs2 = ld_volatile(&ctl->arcs2[0]);
        op.k0 = P.k0;
        prop_node_state<S>(N, op, P.con);
        if (!S::sync(&ctl->bar, &ctl->err)) return;
        // a node's row is as long as its vertices' rows together
        if (ld_volatile(&ctl->max_row2) > (unsigned int)kPropHub) {  // k_prop_hubs goes on
            if (blockIdx.x == 0 && threadIdx.x == 0) ctl->status = 2;
            return;
        }
        const bool pull2 = arcs2 <= P.pull_arcs && arcs2 <= kConPullRow * (unsigned long long)N.n;
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl->form = kFormContracted | (pull2 ? kFormPull : 0);
        if (!(pull2 ? prop_batches<S, true, false>(N, op, ctl, sh, q, mk, (unsigned long long)N.n, 0)
                    : prop_batches<S, false, false>(N, op, ctl, sh, q, mk, (unsigned long long)N.n, 0)))
            return;
        if (!prop_node_labels<S>(P, N, ctl)) return;
        prop_times(P, t0);
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->form = pull ? kFormPull : head_ns ? kFormHeadStart : 0;
    if (!(pull ? prop_batches<S, true, false>(G, op, ctl, sh, q, mk, active, 0)
               : prop_batches<S, false, false>(G, op, ctl, sh, q, mk, active, head_ns)))
        return;
    // ---- canonical labels: the smallest vertex of each SCC
    const int proot = P.vbase == nullptr && active > 0 && ld_volatile(&ctl->pivot) >= 0 ? ld_volatile(&G.rep[ld_volatile(&ctl->pivot)]) : -1;
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
        if (v >= G.n) continue;
        int first_v = 0;
        if (P.vbase != nullptr) {
            const int g = prop_graph_of(P, v);
            if (!P.mesh[g]) continue;
            first_v = (int)(P.vbase[g] - P.vbase[P.g0]);
        }
        P.out[v] = ld_volatile(&P.minid[G.rep[v]]) - first_v;
    }
    prop_times(P, t0);
}

// What may have long rows: the rest of a graph with hubs, whose first SCC is done
// (classes in label), or (status 2) the contracted graph that k_prop left. A
// kernel of its own: the same searches in k_prop, called from the same places,
// cost the lattices of 1 k to 131 k vertices 3-6%, whether they ran or not.
__global__ void __launch_bounds__(kPropBlock, 4) k_prop_hubs(const __grid_constant__ PropParams P) {
    using S = PropScope;
    __shared__ PropShared sh;
    __shared__ uint32_t s_q[kPropWarps][kPropQueue];
    __shared__ uint32_t s_mk[kPropWarps][kPropMarks];
    const PropMax op{P.k0};
    PropCtl* ctl = &P.dev->c;
    const int lane = lane_id();
    uint32_t* q = s_q[threadIdx.x >> 5];
    uint32_t* mk = s_mk[threadIdx.x >> 5];
    const uint64_t t0 = globaltimer_ns();
    if (threadIdx.x == 0) sh.idle_ns = P.idle_ns;
    __syncthreads();
    if (P.fresh) {
        if (ld_volatile(&ctl->status) != 2) return;
        const PropGraph<PropMax> N = prop_nodes(P, ctl);
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl->form = kFormContracted;
        if (!prop_list_hubs<S>(N, ctl, P.minid)) return;
        if (!prop_batches<S, false, true>(N, op, ctl, sh, q, mk, (unsigned long long)N.n, 0)) return;
        if (!prop_node_labels<S>(P, N, ctl)) return;
        prop_times(P, t0);
        return;
    }
    const PropGraph<PropMax>& G = P.G;
    const PropSlice sl = prop_slice<S>(G.n);
    unsigned int mx = 0;
    for (long long i = 0; i < sl.cnt; ++i) {
        const long long w = sl.word(i), v = w * 32 + lane;
        if (w >= sl.nw) break;
        const int32_t lab = v < G.n ? P.label[v] : kDone;
        if (lab >= 0) mx = max(mx, (unsigned int)max(G.end[0][v] - G.off[0][v], G.end[1][v] - G.off[1][v]));
        if (v < G.n) {
            const unsigned long long st = lab >= 0 ? prop_pack((uint32_t)lab, op.key((uint32_t)v)) : PropMax::none();
            G.s[0][v] = st;
            G.s[1][v] = st;
        }
        const uint32_t m = __ballot_sync(kFull, lab >= 0);
        if (lane == 0) {
            G.act[w] = m;
            G.d[0][w] = 0;
            G.d[1][w] = 0;
        }
    }
    mx = __reduce_max_sync(kFull, mx);
    if (lane == 0 && mx > (unsigned int)kPropHub) atomicMax(&ctl->max_deg, mx);
    if (!S::sync(&ctl->bar, &ctl->err)) return;
    if (ld_volatile(&ctl->max_deg) > (unsigned int)kPropHub) {
        if (!prop_list_hubs<S>(G, ctl, P.minid)) return;
        prop_batches<S, false, true>(G, op, ctl, sh, q, mk, P.N, 0);
    } else {
        prop_batches<S, false, false>(G, op, ctl, sh, q, mk, P.N, 0);
    }
}

__global__ void k_prop_err(const PropCtl* c, int* err) {
    if (c->err != 0) atomicCAS(err, 0, c->err);
}

}  // namespace

size_t prop_dev_bytes() { return sizeof(PropDev); }

// Whether a reach_multi search of a graph without hubs only pulls (four blocks an
// SM, as k_prop).
bool reach_pulls(long long n, long long m, int num_sms) {
    return m <= (4 * m < 5 * n ? kReachPullPath : kPropPullArcs) * 4 * num_sms * kPropBlock;
}

// Resident blocks per SM (the first call is outside any stream capture).
int prop_blocks_per_sm(int* out) {
    static int per_sm = -1;
    if (per_sm < 0) {
        int x = 0, y = 0;  // one grid for both: k_prop_hubs goes on at k_prop's barrier
        SCC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&x, k_prop, kPropBlock, 0));
        SCC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&y, k_prop_hubs, kPropBlock, 0));
        if (std::min(x, y) < 1) return SCC_ERR_CUDA;
        per_sm = std::min(x, y);
    }
    *out = per_sm;
    return SCC_OK;
}

// hubs: k_prop_hubs, on the rest of a graph or after k_prop.
static int launch_prop(const PropArgs& a, bool hubs, cudaStream_t st) {
    PropParams P;
    memset(&P, 0, sizeof(P));
    P.G = PropGraph<PropMax>{{a.off, a.toff}, {a.off + 1, a.toff + 1}, {a.adj, a.tadj}, a.n, {a.sf, a.sb}, {a.df, a.db}, a.act, a.rep};
    P.k0 = (uint32_t)mix64(a.seed);
    P.dev = reinterpret_cast<PropDev*>(a.dev);
    P.fresh = a.label == nullptr;
    P.label = a.label;
    P.N = (unsigned long long)a.N;
    P.m = a.m;
    P.seed = a.seed;
    P.minid = a.minid;
    P.out = a.out;
    P.arcs = (unsigned long long)(a.vbase ? a.mesh_arcs : a.m);
    if (P.fresh) {
        const size_t n = (size_t)a.n;
        int32_t* w = a.con_n;
        P.con.cid = w;
        P.con.lead = w + n;
        for (int d = 0; d < 2; ++d) {
            P.con.beg[d] = w + (2 + d) * n;
            P.con.end[d] = w + (4 + d) * n;
            P.con.adj[d] = a.con_m + (size_t)d * (size_t)a.m;
        }
        P.con.rep = w + 6 * n;
        P.con.min = w + 7 * n;
        P.con.act = reinterpret_cast<uint32_t*>(w + 8 * n);
    }
    P.vbase = a.vbase;
    P.mesh = a.mesh;
    P.g0 = a.g0;
    P.g1 = a.g1;
    P.times = a.times;
    P.time_words = a.time_words;
    P.idle_ns = a.idle_ns ? a.idle_ns : kPropIdleTimeoutNs;
    int per_sm = 0;
    SCC_TRY(prop_blocks_per_sm(&per_sm));
    const long long nw = ((long long)a.n + 31) / 32;
    const int full = per_sm * a.num_sms;
    const int grid = (int)std::max<long long>(1, std::min<long long>(full, (nw + kPropWarps - 1) / kPropWarps));
    P.pull_arcs = (unsigned long long)(kPropPullArcs * grid * kPropBlock);
    if (!hubs || !P.fresh) SCC_CUDA(cudaMemsetAsync(P.dev, 0, sizeof(PropDev), st));
    void* args[] = {(void*)&P};
    SCC_CUDA(cudaLaunchCooperativeKernel(hubs ? (const void*)k_prop_hubs : (const void*)k_prop, dim3(grid),
                                         dim3(kPropBlock), args, 0, st));
    count_launch();
    return SCC_OK;
}

int enqueue_prop(const PropArgs& a, int* err, cudaStream_t st) {
    SCC_TRY(launch_prop(a, false, st));
    if (a.n >= kConMin) SCC_TRY(launch_prop(a, true, st));  // ends at once unless it is needed
    k_prop_err<<<1, 1, 0, st>>>(&reinterpret_cast<PropDev*>(a.dev)->c, err);
    SCC_LAUNCH();
    return SCC_OK;
}

int run_prop(const PropArgs& a, PropResult* res, cudaStream_t st) {
    PropCtl c;
    for (bool hubs = a.label != nullptr;; hubs = true) {
        SCC_TRY(launch_prop(a, hubs, st));
        SCC_CUDA(cudaMemcpyAsync(&c, a.dev, sizeof(c), cudaMemcpyDeviceToHost, st));
        SCC_CUDA(cudaStreamSynchronize(st));
        if (c.err) return c.err;
        if (hubs || c.status != 2) break;
    }
    res->status = c.status == 1;
    res->form = c.form;
    res->active = (int64_t)c.active0;
    res->first = (int32_t)c.first;
    res->batches = c.batches;
    res->searches = c.searches;
    res->items = c.items;
    res->arcs = c.arcs;
    return SCC_OK;
}

}  // namespace scc

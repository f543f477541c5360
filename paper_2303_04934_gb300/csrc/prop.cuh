// Signature propagation: the SCCs of a graph from the largest source reaching
// each vertex and the largest source each vertex reaches (sm_103a).
//
// Alg. 1 (Wang, Dong, Gu, Sun, SIGMOD 2023) labels a vertex after a batch by
// its old class, the largest source of the batch that reaches it and the
// largest one it reaches; a vertex whose two are equal lies in that source's
// SCC. With every active vertex a source of the batch, that signature is all
// the labelling needs, so the searches keep it and nothing else: two values
// per vertex instead of a table of (vertex, source) pairs, and an arc is
// followed again only when its tail's value grew. A batch of all vertices
// finishes at least one SCC of every class and splits the others; five to seven
// batches finish a lattice or a k-NN graph.
//
// State: one 64-bit word per vertex and direction, class << 32 | key, where key
// is a seeded bijection of the vertex id (so the order of the sources is random
// and a value names its vertex without a table). A raise is one 64-bit
// atomicMax; the class in the high word makes the arc test (both ends of one
// class, both not finished) part of the same 8-byte read. A finished vertex has
// the high word kPropDone.
//
// Schedule. What bounds these searches on a large-diameter graph is the chain
// of dependent accesses along its paths, not bandwidth, so nothing in a search
// waits for a barrier: vertices whose value grew are bits of a dirty bitmap, a
// warp owns a contiguous run of its words, polls them, takes the set bits and
// relaxes those vertices' arcs, marking the heads it raised in whichever warp's
// words they lie. A search ends when every block is idle at once, which a
// counter of idle blocks detects; a check of the whole bitmap between two grid
// barriers then confirms it (a mark may lie unseen in a block that went idle
// before it), or resumes the search.
//
// Measured against batches of doubling size whose searches kept every pair (the
// whole create + run + destroy, GB300): 2D torus 33^2 2.59 -> 0.42 ms, 256^2
// 11.7 -> 1.31, k-NN of 1 M points 13.9 -> 2.05, 3D torus 256^3 12.8 -> 9.2
// (41 -> 9.1 when the first pivot misses the giant SCC). Of 9.2 ms the head
// start takes 4.2: its wave is a few vertices per warp wide, so it is bound by
// the time of a hop (about 20 us there), not by traffic.
#pragma once
#include "common.cuh"
#include "engine.cuh"

namespace scc {

constexpr uint32_t kPropDone = 0xffffffffu;
constexpr int kPropQueue = 256;    // vertices a warp gathers before it works on them
constexpr int kPropMarks = 384;    // marks a warp gathers before it publishes them
constexpr int kPropBigRow = 64;    // rows longer than this are relaxed by the whole warp
constexpr int kPropPoll = 2;       // bitmap words of each direction a lane polls at a time
constexpr int kPropUnroll = 4;     // arcs of a row in flight per lane
constexpr unsigned kPropSweepMin = 1;  // a sweep follows while the last one raised n values or more
constexpr int kPropTrimPasses = 3; // trimming passes at the start of a batch, at most
constexpr uint64_t kPropIdleTimeoutNs = 20000000000ull;  // an idle block gives up after 20 s (others may work that long)

// A bijection of the 32-bit integers (the finaliser of MurmurHash3, Appleby) and its inverse.
__host__ __device__ __forceinline__ uint32_t prop_mix(uint32_t x) {
    x ^= x >> 16;
    x *= 0x85ebca6bu;
    x ^= x >> 13;
    x *= 0xc2b2ae35u;
    x ^= x >> 16;
    return x;
}
__host__ __device__ __forceinline__ uint32_t prop_unmix(uint32_t x) {
    x ^= x >> 16;
    x *= 0x7ed1b41du;  // 0xc2b2ae35^-1 mod 2^32
    x ^= (x >> 13) ^ (x >> 26);
    x *= 0xa5cb9243u;  // 0x85ebca6b^-1 mod 2^32
    x ^= x >> 16;
    return x;
}

struct PropGraph {
    const int32_t *off, *adj, *toff, *tadj;
    int32_t n;
    uint32_t k0;  // key(v) = prop_mix(v ^ k0)
    unsigned long long *sf, *sb;  // forward (from ancestors) and backward state
    uint32_t *act;                // active vertices
    uint32_t *df, *db;            // dirty vertices, per direction
    int32_t* rep;                 // a vertex of v's SCC, the same for all of it
    __device__ __forceinline__ uint32_t key(uint32_t v) const { return prop_mix(v ^ k0); }
    __device__ __forceinline__ uint32_t vertex(uint32_t key) const { return prop_unmix(key) ^ k0; }
};

struct PropCtl {
    GridBarrier bar;
    int err;
    int idle;                 // idle blocks
    unsigned int found;       // last check that found a dirty word
    unsigned long long count[4];  // vertices finished by a counting step, a ring over the steps
    unsigned long long items, arcs;
    unsigned long long active0;  // active vertices after the first trim
    unsigned int max_deg;
    unsigned long long best;  // smaller degree << 32 | key of the vertex that becomes the largest source
    int batches, searches;
    int pivot;
    int status;  // 0 finished, 1 a skewed graph (nothing done but the first trim)
    unsigned int first;  // vertices in the first pivot's SCC
};

__device__ __forceinline__ unsigned long long prop_pack(uint32_t lab, uint32_t key) {
    return ((unsigned long long)lab << 32) | key;
}

struct PropShared {
    int idle;  // idle warps of the block
    int exit;  // the search is over (or failed)
    int ok;
};

// the run of bitmap words of this warp
template <class S>
__device__ __forceinline__ void prop_slice(int32_t n, long long& w0, long long& w1) {
    const long long nw = ((long long)n + 31) / 32;
    const long long warps = (long long)S::blocks() * (blockDim.x >> 5);
    const long long wid = (long long)S::block() * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long per = (nw + warps - 1) / warps;
    w0 = min(wid * per, nw);
    w1 = min(w0 + per, nw);
}

// A warp's queue of vertices (| direction << 31) in shared memory.
struct PropQueue {
    uint32_t* buf;  // kPropQueue entries
    int cnt;        // warp-uniform
};
// Calls f(has, v, dir) warp-collectively for the queued vertices, 32 at a time.
template <class F>
__device__ __forceinline__ void prop_drain(PropQueue& Q, F&& f) {
    __syncwarp();
    for (int i = lane_id(); i - lane_id() < Q.cnt; i += 32) {
        const bool has = i < Q.cnt;
        const uint32_t c = has ? Q.buf[i] : 0u;
        f(has, (int)(c & 0x7fffffffu), (int)(c >> 31));
    }
    Q.cnt = 0;
    __syncwarp();
}
// Queues the set bits of the lanes' words x (direction 0) and y (direction 1),
// word0 + lane each; f is called when the queue is full.
template <class F>
__device__ __forceinline__ void prop_queue_bits(PropQueue& Q, uint32_t x, uint32_t y, long long word0, F&& f) {
    const uint32_t v0 = (uint32_t)(word0 + lane_id()) * 32u;
    while (__any_sync(kFull, (x | y) != 0)) {
        int nx = __popc(x), ny = __popc(y);
        int incl = warp_incl_scan(nx + ny);
        int total = __shfl_sync(kFull, incl, 31);
        if (Q.cnt + total > kPropQueue) {  // warp-uniform
            if (Q.cnt) prop_drain(Q, f);
            if (total > kPropQueue) {
                nx = min(nx, kPropQueue / 64);
                ny = min(ny, kPropQueue / 64);
                incl = warp_incl_scan(nx + ny);
                total = __shfl_sync(kFull, incl, 31);
            }
        }
        int k = Q.cnt + incl - nx - ny;
        for (int i = 0; i < nx; ++i) {
            Q.buf[k++] = v0 + (uint32_t)(__ffs(x) - 1);
            x &= x - 1;
        }
        for (int i = 0; i < ny; ++i) {
            Q.buf[k++] = (v0 + (uint32_t)(__ffs(y) - 1)) | 0x80000000u;
            y &= y - 1;
        }
        Q.cnt += total;
    }
}
// f(has, v) for the active vertices of the warp's words [w0, w1).
template <class F>
__device__ __forceinline__ void prop_for_active(const uint32_t* act, long long w0, long long w1, uint32_t* q, F&& f) {
    PropQueue Q{q, 0};
    auto g = [&](bool has, int v, int) { f(has, v); };
    for (long long b = w0; b < w1; b += 32) {
        const long long w = b + lane_id();
        const uint32_t x = w < w1 ? act[w] : 0u;
        prop_queue_bits(Q, x, 0u, b, g);
    }
    prop_drain(Q, g);
}

// The marks of a warp's raises, kept in shared memory until one fence covers
// them: whoever takes a mark then sees the raise.
struct PropMarks {
    uint32_t* buf;  // kPropMarks entries of the warp: vertex | direction << 31
    int cnt;        // warp-uniform
};
template <class S>
__device__ __forceinline__ void prop_flush(const PropGraph& G, PropMarks& M) {
    if (M.cnt == 0) return;
    __syncwarp();
    S::fence();
    for (int i = lane_id(); i < M.cnt; i += 32) {
        const uint32_t c = M.buf[i], w = c & 0x7fffffffu;
        atomicOr(&(c >> 31 ? G.db : G.df)[w >> 5], 1u << (w & 31));
    }
    M.cnt = 0;
    __syncwarp();
}

// Relax the arcs of v in direction dir (0: G with sf, 1: G^T with sb); all
// lanes of the warp call.
template <class S>
__device__ __forceinline__ void prop_relax(const PropGraph& G, bool has, int v, int dir, PropMarks& M,
                                           unsigned long long& arcs) {
    const int lane = lane_id();
    const int32_t* off = dir ? G.toff : G.off;
    const int32_t* adj = dir ? G.tadj : G.adj;
    unsigned long long* s = dir ? G.sb : G.sf;
    int o0 = 0, o1 = 0;
    unsigned long long st = 0;
    if (has) {
        st = ld_volatile(&s[v]);
        o0 = S::ld(&off[v]);
        o1 = S::ld(&off[v + 1]);
    }
    const uint32_t lab = (uint32_t)(st >> 32);
    // the source named by the value may itself have been reached by a larger one
    if (has) {
        const uint32_t r = G.vertex((uint32_t)st);
        if (r != (uint32_t)v && r < (uint32_t)G.n) {
            const unsigned long long t = ld_volatile(&s[r]);
            if ((uint32_t)(t >> 32) == lab && t > st) {
                st = t;
                atomicMax(&s[v], t);
            }
        }
    }
    constexpr int U = kPropUnroll;
    auto raise = [&](const int (&w)[U], const unsigned long long (&t)[U], unsigned long long to, unsigned long long* ts,
                     int tdir) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool up = w[u] >= 0 && (uint32_t)(t[u] >> 32) == (uint32_t)(to >> 32) && t[u] < to;
            if (up) atomicMax(&ts[w[u]], to);
            const uint32_t m = __ballot_sync(kFull, up);
            if (up) M.buf[M.cnt + __popc(m & lanemask_lt())] = (uint32_t)w[u] | ((uint32_t)tdir << 31);
            M.cnt += __popc(m);
        }
        if (M.cnt > kPropMarks - 32 * U) prop_flush<S>(G, M);
    };
    const bool big = o1 - o0 > kPropBigRow;
    const int len = big ? 0 : o1 - o0;
    arcs += (unsigned long long)len;
    const int most = __reduce_max_sync(kFull, len);
    for (int k = 0; k < most; k += U) {
        int w[U];
        unsigned long long t[U];
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = k + u < len ? S::ld(&adj[o0 + k + u]) : -1;
#pragma unroll
        for (int u = 0; u < U; ++u) t[u] = w[u] >= 0 ? ld_volatile(&s[w[u]]) : 0ull;
        raise(w, t, st, s, dir);
    }
    uint32_t bm = __ballot_sync(kFull, big);
    while (bm) {  // long rows by the whole warp
        const int l = __ffs(bm) - 1;
        bm &= bm - 1;
        const unsigned long long bst = __shfl_sync(kFull, st, l);
        const int b0 = __shfl_sync(kFull, o0, l), b1 = __shfl_sync(kFull, o1, l);
        const int bdir = __shfl_sync(kFull, dir, l);
        const int32_t* ba = bdir ? G.tadj : G.adj;
        unsigned long long* bs = bdir ? G.sb : G.sf;
        for (int e = b0; e < b1; e += 32 * U) {
            int w[U];
            unsigned long long t[U];
#pragma unroll
            for (int u = 0; u < U; ++u) w[u] = e + 32 * u + lane < b1 ? S::ld(&ba[e + 32 * u + lane]) : -1;
#pragma unroll
            for (int u = 0; u < U; ++u) t[u] = w[u] >= 0 ? ld_volatile(&bs[w[u]]) : 0ull;
            raise(w, t, bst, bs, bdir);
        }
        if (lane == 0) arcs += (unsigned long long)(b1 - b0);
    }
}

// One pull of v: both values become the largest of the in-class neighbours'
// (and, with jump, of the source each names). v's words are written by its
// owner alone, so there is no atomic. Returns bit d set when direction d grew.
template <class S>
__device__ __forceinline__ int prop_pull(const PropGraph& G, bool has, int v, bool jump) {
    unsigned long long s0[2] = {0, 0}, st[2] = {0, 0};
    int e0[2] = {0, 0}, e1[2] = {0, 0};
    const int32_t* const adj[2] = {G.tadj, G.adj};  // the forward value comes from in-neighbours
    unsigned long long* const s[2] = {G.sf, G.sb};
    if (has) {
        e0[0] = S::ld(&G.toff[v]);
        e1[0] = S::ld(&G.toff[v + 1]);
        e0[1] = S::ld(&G.off[v]);
        e1[1] = S::ld(&G.off[v + 1]);
        s0[0] = ld_volatile(&G.sf[v]);
        s0[1] = ld_volatile(&G.sb[v]);
    }
    const uint32_t lab = (uint32_t)(s0[0] >> 32);
    st[0] = s0[0];
    st[1] = s0[1];
    if (jump && has) {
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            const uint32_t r = G.vertex((uint32_t)s0[d]);
            const unsigned long long t = r != (uint32_t)v && r < (uint32_t)G.n ? ld_volatile(&s[d][r]) : 0ull;
            if ((uint32_t)(t >> 32) == lab) st[d] = max(st[d], t);
        }
    }
    constexpr int U = kPropUnroll;
    const bool big = has && max(e1[0] - e0[0], e1[1] - e0[1]) > kPropBigRow;
    int n0 = big ? 0 : e1[0] - e0[0], n1 = big ? 0 : e1[1] - e0[1];
    for (int k = 0; k < max(n0, n1); k += U) {
        int w[2][U];
        unsigned long long t[2][U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            w[0][u] = k + u < n0 ? S::ld(&adj[0][e0[0] + k + u]) : -1;
            w[1][u] = k + u < n1 ? S::ld(&adj[1][e0[1] + k + u]) : -1;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            t[0][u] = w[0][u] >= 0 ? ld_volatile(&s[0][w[0][u]]) : 0ull;
            t[1][u] = w[1][u] >= 0 ? ld_volatile(&s[1][w[1][u]]) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (w[0][u] >= 0 && (uint32_t)(t[0][u] >> 32) == lab) st[0] = max(st[0], t[0][u]);
            if (w[1][u] >= 0 && (uint32_t)(t[1][u] >> 32) == lab) st[1] = max(st[1], t[1][u]);
        }
    }
    uint32_t bm = __ballot_sync(kFull, big);
    while (bm) {  // long rows by the whole warp
        const int l = __ffs(bm) - 1;
        bm &= bm - 1;
        const uint32_t blab = __shfl_sync(kFull, lab, l);
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            const int b0 = __shfl_sync(kFull, e0[d], l), b1 = __shfl_sync(kFull, e1[d], l);
            unsigned long long m = 0;
            for (int e = b0 + lane_id(); e < b1; e += 32 * U) {
                int w[U];
                unsigned long long t[U];
#pragma unroll
                for (int u = 0; u < U; ++u) w[u] = e + 32 * u < b1 ? S::ld(&adj[d][e + 32 * u]) : -1;
#pragma unroll
                for (int u = 0; u < U; ++u) t[u] = w[u] >= 0 ? ld_volatile(&s[d][w[u]]) : 0ull;
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (w[u] >= 0 && (uint32_t)(t[u] >> 32) == blab) m = max(m, t[u]);
            }
            for (int dd = 16; dd >= 1; dd >>= 1) m = max(m, __shfl_xor_sync(kFull, m, dd));
            if (lane_id() == l) st[d] = max(st[d], m);
        }
    }
    int up = 0;
#pragma unroll
    for (int d = 0; d < 2; ++d)
        if (has && st[d] > s0[d]) {
            *(volatile unsigned long long*)&s[d][v] = st[d];
            up |= 1 << d;
        }
    return up;
}

// A warp's idle state within its block, and the block's within the grid.
template <class S>
struct PropIdle {
    PropCtl* ctl;
    PropShared& sh;
    bool idle = false;
    uint64_t t0 = 0;
    __device__ __forceinline__ PropIdle(PropCtl* c, PropShared& s) : ctl(c), sh(s) {}
    __device__ __forceinline__ void wake() {
        if (!idle) return;
        idle = false;
        if (lane_id() == 0 && atomicSub(&sh.idle, 1) == (int)(blockDim.x >> 5) && S::blocks() > 1)
            atomicSub(&ctl->idle, 1);
    }
    // after a pass over the warp's words that found nothing: true when the
    // search is over (or a wait ran out)
    __device__ __forceinline__ bool rest() {
        if (!idle) {
            idle = true;
            if (lane_id() == 0) {
                S::fence();
                if (atomicAdd(&sh.idle, 1) == (int)(blockDim.x >> 5) - 1) {
                    if (S::blocks() > 1) atomicAdd(&ctl->idle, 1);
                    else atomicExch(&sh.exit, 1);
                }
            }
            __syncwarp();
            t0 = globaltimer_ns();
        } else if (threadIdx.x == 0 && S::blocks() > 1) {
            if (ld_volatile(&ctl->idle) >= S::blocks()) {
                atomicExch(&sh.exit, 1);
            } else if (globaltimer_ns() - t0 > kPropIdleTimeoutNs) {
                atomicCAS(&ctl->err, 0, SCC_ERR_TIMEOUT);
                atomicExch(&sh.exit, 1);
            }
        }
        const int ex = lane_id() == 0 ? ld_volatile(&sh.exit) : 0;
        return __shfl_sync(kFull, ex, 0) != 0;
    }
};
// Ends a check (every block has arrived at its first barrier and looked for
// work left): *more says whether any block found some. False: a barrier timed out.
template <class S>
__device__ __forceinline__ bool prop_checked(PropCtl* ctl, PropShared& sh, unsigned int check, bool left, bool* more) {
    if (__any_sync(kFull, left) && lane_id() == 0) atomicMax(&ctl->found, check);
    if (S::block() == 0 && threadIdx.x == 0) *(volatile int*)&ctl->idle = 0;  // no block counts itself in between the two barriers
    if (!S::sync(&ctl->bar, &ctl->err)) return false;
    *more = ld_volatile(&ctl->found) == check;
    if (threadIdx.x == 0) sh.idle = sh.exit = 0;
    __syncthreads();
    return ld_volatile(&ctl->err) == 0;
}

// A search by pulling alone. With one word per warp a lane keeps its vertex's
// two values and the first arcs of both its rows in registers, so a pass, and
// with it a hop, costs one round of loads; the value's own source is looked at
// in the same round.
template <class S>
__device__ bool prop_search_pull(const PropGraph& G, PropCtl* ctl, PropShared& sh, unsigned int& check,
                                 unsigned long long& items) {
    long long w0, w1;
    prop_slice<S>(G.n, w0, w1);
    if (threadIdx.x == 0) sh.idle = sh.exit = 0;
    __syncthreads();
    auto pass = [&](bool jump) {
        bool up = false;
        for (long long w = w0; w < w1; ++w) {
            const uint32_t x = G.act[w];
            if (x == 0) continue;  // warp-uniform
            const bool has = (x >> lane_id()) & 1u;
            const int c = prop_pull<S>(G, has, (int)(w * 32) + lane_id(), jump);
            up |= c != 0;
            if (c) ++items;
        }
        return __any_sync(kFull, up) != 0;
    };
    constexpr int U = kPropUnroll;
    const bool one = w1 - w0 == 1;
    const int v = (int)(w0 * 32) + lane_id();
    const bool has = one && ((G.act[w0] >> lane_id()) & 1u);
    unsigned long long st[2] = {0, 0};
    int w[2][U], len[2] = {0, 0};
#pragma unroll
    for (int u = 0; u < U; ++u) w[0][u] = w[1][u] = -1;
    if (has) {
        st[0] = ld_volatile(&G.sf[v]);
        st[1] = ld_volatile(&G.sb[v]);
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            const int32_t* off = d ? G.off : G.toff;
            const int32_t* adj = d ? G.adj : G.tadj;
            const int e0 = S::ld(&off[v]);
            len[d] = S::ld(&off[v + 1]) - e0;
#pragma unroll
            for (int u = 0; u < U; ++u) w[d][u] = u < len[d] ? S::ld(&adj[e0 + u]) : -1;
        }
    }
    const uint32_t lab = (uint32_t)(st[0] >> 32);
    const bool fits = __all_sync(kFull, max(len[0], len[1]) <= U) != 0;
    auto pass_one = [&]() {
        unsigned long long t[2][U], j[2];
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            const unsigned long long* s = d ? G.sb : G.sf;
            const uint32_t r = G.vertex((uint32_t)st[d]);
            j[d] = has && r < (uint32_t)G.n ? ld_volatile(&s[r]) : 0ull;
#pragma unroll
            for (int u = 0; u < U; ++u) t[d][u] = w[d][u] >= 0 ? ld_volatile(&s[w[d][u]]) : 0ull;
        }
        bool up = false;
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            unsigned long long m = st[d];
            if ((uint32_t)(j[d] >> 32) == lab) m = max(m, j[d]);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (w[d][u] >= 0 && (uint32_t)(t[d][u] >> 32) == lab) m = max(m, t[d][u]);
            if (has && m > st[d]) {
                st[d] = m;
                *(volatile unsigned long long*)&(d ? G.sb : G.sf)[v] = m;
                up = true;
                ++items;
            }
        }
        return __any_sync(kFull, up) != 0;
    };
    for (;;) {
        PropIdle<S> id(ctl, sh);
        for (;;) {
            if (one && fits ? pass_one() : pass(true)) id.wake();
            else if (id.rest()) break;
        }
        if (!S::sync(&ctl->bar, &ctl->err)) return false;
        ++check;
        const bool left = one && fits ? pass_one() : pass(false);
        bool more = false;
        if (!prop_checked<S>(ctl, sh, check, left, &more)) return false;
        if (!more) return true;
    }
}

// One search: relax until no vertex is dirty. Every thread of the scope calls
// it; `check` numbers the checks of the launch (the same in every block). With
// a deadline (globaltimer ns; 0: none) it may end early, vertices still dirty.
// Returns false when a wait ran out (the caller returns at once).
template <class S>
__device__ bool prop_search(const PropGraph& G, PropCtl* ctl, PropShared& sh, uint32_t* q, uint32_t* mk,
                            unsigned int& check, uint64_t deadline, unsigned long long& items,
                            unsigned long long& arcs) {
    const int lane = lane_id();
    long long w0, w1;
    prop_slice<S>(G.n, w0, w1);
    if (threadIdx.x == 0) sh.idle = sh.exit = 0;
    __syncthreads();
    PropMarks M{mk, 0};
    PropQueue Q{q, 0};
    long long turn = 0;  // the word whose sources are looked at next
    auto relax = [&](bool has, int v, int dir) { prop_relax<S>(G, has, v, dir, M, arcs); };
    for (;;) {
        PropIdle<S> id(ctl, sh);
        for (;;) {
            // the words of the whole run are polled before any work: a wave
            // touches a few vertices in each, which then share one step
            bool did = false;
            for (long long b = w0; b < w1; b += 32 * kPropPoll) {
                uint32_t x[kPropPoll], y[kPropPoll];
#pragma unroll
                for (int j = 0; j < kPropPoll; ++j) {
                    const long long w = b + 32 * j + lane;
                    x[j] = w < w1 ? ld_volatile(&G.df[w]) : 0u;
                    y[j] = w < w1 ? ld_volatile(&G.db[w]) : 0u;
                }
                uint32_t any = 0;
#pragma unroll
                for (int j = 0; j < kPropPoll; ++j) any |= x[j] | y[j];
                if (!__any_sync(kFull, any != 0)) continue;
                if (!did) {
                    did = true;
                    id.wake();
                }
#pragma unroll
                for (int j = 0; j < kPropPoll; ++j) {
                    const long long w = b + 32 * j + lane;
                    if (x[j]) x[j] = atomicExch(&G.df[w], 0u);
                    if (y[j]) y[j] = atomicExch(&G.db[w], 0u);
                }
                S::fence();
#pragma unroll
                for (int j = 0; j < kPropPoll; ++j) {
                    items += (unsigned long long)(__popc(x[j]) + __popc(y[j]));
                    prop_queue_bits(Q, x[j], y[j], b + 32 * j, relax);
                }
            }
            if (did) {
                prop_drain(Q, relax);
                prop_flush<S>(G, M);
            }
            // nothing dirty: look whether the source that a vertex of the next
            // word names was itself reached by a larger one (paths are walked
            // hop by hop; this takes the rest of one in a step)
            if (!did && w1 > w0) {
                if (++turn >= w1 - w0) turn = 0;
                const long long w = w0 + turn;
                const uint32_t x = G.act[w];
                uint32_t up[2] = {0, 0};
                if (x != 0) {  // warp-uniform
                    const bool has = (x >> lane) & 1u;
                    const long long v = w * 32 + lane;
                    unsigned long long st[2], t[2];
                    st[0] = has ? ld_volatile(&G.sf[v]) : 0ull;
                    st[1] = has ? ld_volatile(&G.sb[v]) : 0ull;
#pragma unroll
                    for (int d = 0; d < 2; ++d) {
                        const uint32_t r = G.vertex((uint32_t)st[d]);
                        t[d] = has && r != (uint32_t)v && r < (uint32_t)G.n ? ld_volatile(&(d ? G.sb : G.sf)[r]) : 0ull;
                    }
#pragma unroll
                    for (int d = 0; d < 2; ++d) {
                        const bool u = t[d] > st[d] && (t[d] >> 32) == (st[d] >> 32);
                        if (u) atomicMax(&(d ? G.sb : G.sf)[v], t[d]);
                        up[d] = __ballot_sync(kFull, u);
                    }
                }
                if (up[0] | up[1]) {
                    did = true;
                    id.wake();
                    S::fence();
                    __syncwarp();
                    if (lane == 0 && up[0]) atomicOr(&G.df[w], up[0]);
                    if (lane == 0 && up[1]) atomicOr(&G.db[w], up[1]);
                }
            }
            if (!did && id.rest()) break;
            if (deadline) {
                const uint64_t now = lane == 0 ? globaltimer_ns() : 0;
                if (__shfl_sync(kFull, now, 0) > deadline) break;
            }
        }
        // every block is here: look for marks that no poll saw
        if (!S::sync(&ctl->bar, &ctl->err)) return false;
        ++check;
        bool left = false;
        if (!deadline)
            for (long long w = w0 + lane; w < w1; w += 32) left |= (ld_volatile(&G.df[w]) | ld_volatile(&G.db[w])) != 0;
        bool more = false;
        if (!prop_checked<S>(ctl, sh, check, left, &more)) return false;
        if (!more) return true;
    }
}

// Whether a vertex w != v of v's class is in the row.
template <class S>
__device__ __forceinline__ bool prop_any_in_class(const int32_t* adj, int o0, int o1, const unsigned long long* s,
                                                  uint32_t lab) {
    for (int e = o0; e < o1; e += 2) {
        const int w0 = S::ld(&adj[e]);
        const int w1 = e + 1 < o1 ? S::ld(&adj[e + 1]) : w0;
        const uint32_t l0 = (uint32_t)(ld_volatile(&s[w0]) >> 32), l1 = (uint32_t)(ld_volatile(&s[w1]) >> 32);
        if (l0 == lab || l1 == lab) return true;
    }
    return false;
}

// The vertices finished by a counting step, summed over the scope. The counters
// are a ring indexed by the step (the same number in every block), so that no
// block reads one that a faster block already adds to; ends at a barrier.
template <class S>
__device__ __forceinline__ bool prop_count(PropCtl* ctl, unsigned int& step, unsigned long long mine,
                                           unsigned long long& sum) {
    for (int d = 16; d >= 1; d >>= 1) mine += __shfl_xor_sync(kFull, mine, d);
    if (S::block() == 0 && threadIdx.x == 0) ctl->count[(step + 1) & 3] = 0;
    if (lane_id() == 0 && mine) atomicAdd(&ctl->count[step & 3], mine);
    if (!S::sync(&ctl->bar, &ctl->err)) return false;
    sum = ld_volatile(&ctl->count[step & 3]);
    ++step;
    return true;
}

// The batches from the state in sf/sb/act until every active vertex is
// finished (`active` of them): trimming inside the classes, the two searches,
// the labelling. Self-loops must not be in the graph. The ring of counters
// starts zero. pull: the searches only pull. head_ns: time limit of the first batch's head start (0: none);
// with it the state's keys start zero, and the first batch sets them.
template <class S>
__device__ bool prop_batches(const PropGraph& G, PropCtl* ctl, PropShared& sh, uint32_t* q, uint32_t* mk,
                             unsigned long long active, bool pull, uint64_t head_ns) {
    const int lane = lane_id();
    long long w0, w1;
    prop_slice<S>(G.n, w0, w1);
    unsigned int check = 0;
    unsigned long long items = 0, arcs = 0, done = 0;
    int batches = 0;
    unsigned int step = 0;
    while (done < active) {
        // ---- vertices with no arc from, or no arc to, a vertex of their class
        for (int pass = 0; pass < kPropTrimPasses; ++pass) {
            unsigned long long cnt = 0;
            prop_for_active(G.act, w0, w1, q, [&](bool has, int v) {
                if (!has) return;
                const uint32_t lab = (uint32_t)(ld_volatile(&G.sf[v]) >> 32);
                const int o0 = S::ld(&G.off[v]), o1 = S::ld(&G.off[v + 1]);
                const int i0 = S::ld(&G.toff[v]), i1 = S::ld(&G.toff[v + 1]);
                if (prop_any_in_class<S>(G.adj, o0, o1, G.sf, lab) &&
                    prop_any_in_class<S>(G.tadj, i0, i1, G.sf, lab))
                    return;
                *(volatile unsigned long long*)&G.sf[v] = prop_pack(kPropDone, 0);
                *(volatile unsigned long long*)&G.sb[v] = prop_pack(kPropDone, 0);
                G.rep[v] = v;
                atomicAnd(&G.act[v >> 5], ~(1u << (v & 31)));
                ++cnt;
            });
            unsigned long long got = 0;
            if (!prop_count<S>(ctl, step, cnt, got)) return false;
            done += got;
            if (got * 8 < active - done) break;
        }
        if (done >= active) break;
        if (pull) {
            if (!prop_search_pull<S>(G, ctl, sh, check, items)) return false;
        } else {
            // ---- every active vertex is a source. A head start: the largest
            // source alone, so that a giant SCC is flooded once before the
            // others' values wander through it
            unsigned long long grew = 2 * (active - done);
            if (batches == 0 && head_ns) {
                const uint32_t b = G.vertex(0xffffffffu);
                if (S::block() == 0 && threadIdx.x == 0) {
                    const unsigned long long st = G.sf[b];
                    if ((uint32_t)(st >> 32) != kPropDone) {
                        G.sf[b] = G.sb[b] = st | 0xffffffffull;
                        G.df[b >> 5] = G.db[b >> 5] = 1u << (b & 31);
                    }
                }
                if (!S::sync(&ctl->bar, &ctl->err)) return false;
                if (!prop_search<S>(G, ctl, sh, q, mk, check, globaltimer_ns() + head_ns, items, arcs)) return false;
                unsigned long long cnt = 0;
                for (long long w = w0; w < w1; ++w) {
                    const uint32_t x = G.act[w];
                    if (x == 0) continue;  // warp-uniform
                    const long long v = w * 32 + lane;
                    bool f = false, r = false;
                    if ((x >> lane) & 1u) {
                        const unsigned long long sf = G.sf[v], sb = G.sb[v];
                        const uint32_t key = G.key((uint32_t)v);
                        f = (uint32_t)sf < key;
                        r = (uint32_t)sb < key;
                        if (f) G.sf[v] = prop_pack((uint32_t)(sf >> 32), key);
                        if (r) G.sb[v] = prop_pack((uint32_t)(sb >> 32), key);
                    }
                    const uint32_t mf = __ballot_sync(kFull, f), mr = __ballot_sync(kFull, r);
                    if (lane == 0) {
                        G.df[w] |= mf;
                        G.db[w] |= mr;
                        cnt += __popc(mf) + __popc(mr);
                    }
                }
                if (!prop_count<S>(ctl, step, cnt, grew)) return false;
            } else {
                for (long long w = w0 + lane; w < w1; w += 32) {
                    const uint32_t x = G.act[w];
                    if (x) {
                        G.df[w] = x;
                        G.db[w] = x;
                    }
                }
                if (!S::sync(&ctl->bar, &ctl->err)) return false;
            }
            // ---- sweeps that pull every active vertex (no atomics, coalesced
            // rows) while a sweep raises much of the graph; the last one leaves
            // the vertices it raised dirty
            while (grew * kPropSweepMin >= (unsigned long long)G.n) {
                unsigned long long cnt = 0;
                for (long long w = w0; w < w1; ++w) {
                    const uint32_t x = G.act[w];
                    if (x == 0) continue;  // warp-uniform
                    const bool has = (x >> lane) & 1u;
                    const int c = prop_pull<S>(G, has, (int)(w * 32) + lane, false);
                    const uint32_t cf = __ballot_sync(kFull, c & 1), cb = __ballot_sync(kFull, c & 2);
                    if (lane == 0) {
                        G.df[w] = cf;
                        G.db[w] = cb;
                        cnt += __popc(cf) + __popc(cb);
                    }
                }
                items += cnt;
                if (!prop_count<S>(ctl, step, cnt, grew)) return false;
            }
            if (!prop_search<S>(G, ctl, sh, q, mk, check, 0, items, arcs)) return false;
        }
        // ---- labelling (Alg. 1): equal maxima finish a vertex, the others'
        // class becomes the hash of the old one and the two maxima
        unsigned long long cnt = 0;
        prop_for_active(G.act, w0, w1, q, [&](bool has, int v) {
            if (!has) return;
            const unsigned long long f = ld_volatile(&G.sf[v]), r = ld_volatile(&G.sb[v]);
            if (f == r) {
                G.sf[v] = G.sb[v] = prop_pack(kPropDone, 0);
                const uint32_t r = G.vertex((uint32_t)f);
                if (r >= (uint32_t)G.n) atomicCAS(&ctl->err, 0, SCC_ERR_INTERNAL);  // never: a value names a vertex
                G.rep[v] = r < (uint32_t)G.n ? (int32_t)r : v;
                atomicAnd(&G.act[v >> 5], ~(1u << (v & 31)));
                ++cnt;
            } else {
                const int32_t lab = class_hash((int32_t)(uint32_t)(f >> 32), (int32_t)(uint32_t)f, (int32_t)(uint32_t)r);
                G.sf[v] = G.sb[v] = prop_pack((uint32_t)lab, G.key((uint32_t)v));
            }
        });
        unsigned long long got = 0;
        if (!prop_count<S>(ctl, step, cnt, got)) return false;
        done += got;
        ++batches;
    }
    for (int d = 16; d >= 1; d >>= 1) {
        items += __shfl_xor_sync(kFull, items, d);
        arcs += __shfl_xor_sync(kFull, arcs, d);
    }
    if (lane == 0 && items) atomicAdd(&ctl->items, items);
    if (lane == 0 && arcs) atomicAdd(&ctl->arcs, arcs);
    if (S::block() == 0 && threadIdx.x == 0) {
        ctl->batches = batches;
        ctl->searches = (int)check;
    }
    return true;
}

}  // namespace scc

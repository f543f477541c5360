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
// warp owns runs of its words, polls them, takes the set bits and
// relaxes those vertices' arcs, marking the heads it raised in whichever warp's
// words they lie; a few it relaxes at once itself (kPropNarrow), and a hub's row
// is shared by the idle warps (prop_share). A search ends when every block is idle
// at once, which a counter of idle blocks detects; a check of the whole bitmap
// between two grid barriers then confirms it (a mark may lie unseen in a block that
// went idle before it), or resumes the search.
//
// Measured against batches of doubling size whose searches kept every pair (the
// whole create + run + destroy, GB300): 2D torus 33^2 1.37 -> 0.24 ms, 256^2
// 11.8 -> 1.15, k-NN of 1 M points 12.2 -> 1.5, 3D torus 256^3 12.8 -> 6.4
// (41 -> 6.4 when the first pivot misses the giant SCC), about half of which is
// the head start: its wave is a few vertices per warp wide, so it is bound by the
// time of a hop, not by traffic.
#pragma once
#include "common.cuh"
#include "engine.cuh"

namespace scc {

constexpr uint32_t kPropDone = 0xffffffffu;
constexpr int kPropQueue = 256;    // vertices a warp gathers before it works on them
constexpr int kPropMarks = 384;    // marks a warp gathers before it publishes them
constexpr int kPropBigRow = 64;    // rows longer than this are relaxed by the whole warp
constexpr int kPropUnroll = 4;     // arcs of a row in flight per lane
constexpr int kPropHub = 4096;     // rows longer than this are shared by the idle warps of the grid ...
constexpr int kPropPiece = 512;    // ... in pieces of this many arcs
constexpr int kPropTasks = 24;     // rows shared at a time
// So few raised vertices are relaxed at once by the warp that raised them, so many
// times in a row: a hop through a mark is a fence, the mark, a poll, its exchange
// and a fence more (4 us against 0.9 on a two-way path). reach_multi, ms: ladder of 1 M
// vertices 1850 -> 790, 3D torus of 1 M 2.43 -> 1.33 (4 vertices 1.79, 8 1.53; 32 and 8
// hops 1.40); SCC of the 3D torus 256^3 8.4 -> 6.2 (4: 7.7, 8: 7.2).
constexpr int kPropNarrow = 32;
constexpr int kPropHops = 32;
constexpr int kPropTrimPasses = 3; // trimming passes at the start of a batch, at most
constexpr uint64_t kPropIdleTimeoutNs = 20000000000ull;  // an idle block gives up when no block woke for 20 s

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

// A long row that the warps share: a warp takes the next piece by one addition
// to `next`, which holds the number of pieces beside it, so a claim on a slot that
// has ended, or holds another row by now, is judged by that row's own count.
struct PropTask {
    unsigned long long next;  // pieces << 32 | next piece; 0: free
    unsigned int read;        // claimed pieces whose claimers have read v
    uint32_t v;               // vertex | direction << 31
};

struct PropCtl {
    GridBarrier bar;
    // idle blocks (low 16 bits, signed) under a count of the blocks that woke, and
    // the slots of rows with pieces to take: read as one word
    alignas(8) unsigned int idle;
    unsigned int open;
    unsigned int taken;       // slots in use
    int err;
    PropTask task[kPropTasks];
    int32_t* hub;             // the vertices with a row of more than kPropHub arcs
    unsigned int nhub;        // their number
    unsigned int found;       // last check that found work left
    unsigned long long count[4];  // vertices finished by a counting step, a ring over the steps
    unsigned long long items, arcs;
    unsigned long long active0;  // active vertices after the first trim
    unsigned int max_deg, max_row2;  // the longest row: of an active vertex, of the contracted graph
    unsigned long long best;  // smaller degree << 32 | key of the vertex that becomes the largest source
    int batches, searches;
    int pivot;
    unsigned int merged[2];    // vertices merged by mutual arcs: in the sample, in the rest
    unsigned int hooked[3];    // ... and by a round, a ring over the rounds
    unsigned int nodes;        // vertices of the contracted graph
    unsigned int arcs2[2];     // arcs of the contracted graph and of its transpose
    int status;  // 0 finished, 1 a skewed graph (nothing done but the first trim), 2 contracted, with long rows
    unsigned int first;  // vertices in the first pivot's SCC
    int form;            // kForm* taken
};

struct PropShared {
    uint64_t idle_ns;  // the limit of an idle block's wait, kept by its first thread:
    uint64_t t0;       // since when it waits (0: to be set)
    unsigned int woken, polls;  // the count of woken blocks last seen; looks since then
    int idle;  // idle warps of the block
    int exit;  // the search is over (or failed)
    unsigned int open;  // rows that have pieces to take
};

__device__ __forceinline__ unsigned long long prop_pack(uint32_t lab, uint32_t key) {
    return ((unsigned long long)lab << 32) | key;
}

// ----------------------------------------------------------------- values --
// What a search spreads along the arcs: a value per vertex and direction that
// only grows. gains: whether a vertex holding t grows by mine; raise: the same
// in memory. part: what a vertex holding a can take from t, folded over its
// neighbours before it is compared with a (more) and put into it (with).

// the largest source, inside a class (state class << 32 | key)
struct PropMax {
    using Val = unsigned long long;
    static constexpr int kDirs = 2;  // from ancestors along G, from descendants along G^T
    static constexpr bool kNamed = true;  // a value names a vertex, whose own value may be larger
    uint32_t k0;  // key(v) = prop_mix(v ^ k0)
    __device__ __forceinline__ uint32_t key(uint32_t v) const { return prop_mix(v ^ k0); }
    __device__ __forceinline__ uint32_t vertex(uint32_t key) const { return prop_unmix(key) ^ k0; }
    __device__ __forceinline__ uint32_t named(Val x) const { return vertex((uint32_t)x); }
    __device__ __forceinline__ static Val load(const Val* p, size_t i) { return ld_volatile(&p[i]); }
    __device__ __forceinline__ static void store(Val* p, size_t i, Val x) { *(volatile Val*)&p[i] = x; }
    __device__ __forceinline__ static bool gains(Val mine, Val t) { return (t >> 32) == (mine >> 32) && t < mine; }
    using Part = uint32_t;  // the key, 0 outside the class
    __device__ __forceinline__ static Part part(Val a, Val t) { return (t >> 32) == (a >> 32) ? (uint32_t)t : 0u; }
    __device__ __forceinline__ static Part fold(Part a, Part b) { return max(a, b); }
    __device__ __forceinline__ static Val with(Val a, Part p) { return (a & ~0xffffffffull) | p; }
    __device__ __forceinline__ static bool more(Part p, Val a) { return p > (uint32_t)a; }
    __device__ __forceinline__ static void raise(Val* p, size_t i, Val mine) { atomicMax(&p[i], mine); }
    __device__ __forceinline__ static Val none() { return prop_pack(kPropDone, 0); }  // takes and gives nothing
};
// the set of sources, 64 or 128 of them (mask words v, or 2 v and 2 v + 1)
struct PropOr {
    using Val = unsigned long long;
    static constexpr int kDirs = 1;
    static constexpr bool kNamed = false;
    __device__ __forceinline__ uint32_t named(Val) const { return 0; }
    __device__ __forceinline__ static Val load(const Val* p, size_t i) { return ld_volatile(&p[i]); }
    __device__ __forceinline__ static void store(Val* p, size_t i, Val x) { *(volatile Val*)&p[i] = x; }
    __device__ __forceinline__ static bool gains(Val mine, Val t) { return (mine & ~t) != 0; }
    using Part = Val;
    __device__ __forceinline__ static Part part(Val, Val t) { return t; }
    __device__ __forceinline__ static Part fold(Part a, Part b) { return a | b; }
    __device__ __forceinline__ static Val with(Val a, Part p) { return a | p; }
    __device__ __forceinline__ static bool more(Part p, Val a) { return (p & ~a) != 0; }
    __device__ __forceinline__ static void raise(Val* p, size_t i, Val mine) { atomicOr(&p[i], mine); }
    __device__ __forceinline__ static Val none() { return 0; }
};
// A vertex's two words are one 16-byte access: a pull search of a lattice is
// bound by the sectors its loads touch, and two loads of 8 bytes touched a
// sector twice (128 sources on a 2D torus 504^2: 5.0 -> 3.5 ms).
struct PropOr2 {
    struct alignas(16) Val {
        unsigned long long lo, hi;
    };
    static constexpr int kDirs = 1;
    static constexpr bool kNamed = false;
    __device__ __forceinline__ uint32_t named(Val) const { return 0; }
    __device__ __forceinline__ static Val load(const Val* p, size_t i) {
        Val x;
        asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(x.lo), "=l"(x.hi) : "l"(p + i) : "memory");
        return x;
    }
    __device__ __forceinline__ static void store(Val* p, size_t i, Val x) {
        asm volatile("st.volatile.global.v2.u64 [%0], {%1, %2};" ::"l"(p + i), "l"(x.lo), "l"(x.hi) : "memory");
    }
    __device__ __forceinline__ static bool gains(Val mine, Val t) { return ((mine.lo & ~t.lo) | (mine.hi & ~t.hi)) != 0; }
    using Part = Val;
    __device__ __forceinline__ static Part part(const Val&, const Val& t) { return t; }
    __device__ __forceinline__ static Part fold(Part a, Part b) { return {a.lo | b.lo, a.hi | b.hi}; }
    __device__ __forceinline__ static Val with(Val a, Part p) { return {a.lo | p.lo, a.hi | p.hi}; }
    __device__ __forceinline__ static bool more(Part p, Val a) { return ((p.lo & ~a.lo) | (p.hi & ~a.hi)) != 0; }
    __device__ __forceinline__ static void raise(Val* p, size_t i, Val mine) {
        if (mine.lo) atomicOr(&p[i].lo, mine.lo);
        if (mine.hi) atomicOr(&p[i].hi, mine.hi);
    }
    __device__ __forceinline__ static Val none() { return {0, 0}; }
};
template <class V>
__device__ __forceinline__ V prop_shfl(const V& x, int l) {
    if constexpr (sizeof(V) == 8) return __shfl_sync(kFull, x, l);
    else return {__shfl_sync(kFull, x.lo, l), __shfl_sync(kFull, x.hi, l)};
}
template <class V>
__device__ __forceinline__ V prop_shfl_xor(const V& x, int d) {
    if constexpr (sizeof(V) <= 8) return __shfl_xor_sync(kFull, x, d);
    else return {__shfl_xor_sync(kFull, x.lo, d), __shfl_xor_sync(kFull, x.hi, d)};
}

template <class Op>
struct PropGraph {
    using Val = typename Op::Val;
    const int32_t* off[2];  // the graph, its transpose: row v of [k] is adj[k][off[k][v] .. end[k][v])
    const int32_t* end[2];
    const int32_t* adj[2];
    int32_t n;
    Val* s[Op::kDirs];            // values; direction 1 travels along the transpose
    uint32_t* d[Op::kDirs];       // dirty vertices
    uint32_t* act;                // active vertices (null: all)
    int32_t* rep;                 // a vertex of v's SCC, the same for all of it
    __device__ __forceinline__ uint32_t active(long long w) const {
        if (act) return act[w];
        const long long left = (long long)n - w * 32;
        return left >= 32 ? kFull : (1u << left) - 1u;
    }
};

// The bitmap words of a warp: runs of 2^l words dealt out to the warps in turn,
// so that a busy part of the graph is shared by many warps (3D torus 256^3, the
// head start and the searches of the first batch: runs of 32 words 4.98 ms, of 8
// 5.62, one run a warp 7.37). Word i of the warp, i < cnt, may be past the end
// (>= nw).
struct PropSlice {
    long long nw, wid, warps;
    int l;
    long long cnt;
    __device__ __forceinline__ long long word(long long i) const {
        return ((((i >> l) * warps) + wid) << l) + (i & ((1 << l) - 1));
    }
};
template <class S>
__device__ __forceinline__ PropSlice prop_slice(int32_t n) {
    PropSlice P;
    P.nw = ((long long)n + 31) / 32;
    P.warps = (long long)S::blocks() * (blockDim.x >> 5);
    P.wid = (long long)S::block() * (blockDim.x >> 5) + (threadIdx.x >> 5);
    P.l = P.nw >= 64 * P.warps ? 5 : P.nw >= 16 * P.warps ? 3 : 0;
    const long long runs = (P.nw + (1 << P.l) - 1) >> P.l;
    P.cnt = ((runs + P.warps - 1 - P.wid) / P.warps) << P.l;
    return P;
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
// Moves set bits of the lanes' words x (direction 0) and y (direction 1) into
// the queue, a lane's both at the same word: all of them if they fit, else some.
__device__ __forceinline__ void prop_queue_bits(PropQueue& Q, uint32_t& x, uint32_t& y, long long word) {
    const uint32_t v0 = (uint32_t)word * 32u;
    int nx = __popc(x), ny = __popc(y);
    int incl = warp_incl_scan(nx + ny);
    int total = __shfl_sync(kFull, incl, 31);
    if (Q.cnt + total > kPropQueue) {  // warp-uniform
        if (Q.cnt) return;             // after the next drain
        nx = min(nx, kPropQueue / 64);
        ny = min(ny, kPropQueue / 64);
        incl = warp_incl_scan(nx + ny);
        total = __shfl_sync(kFull, incl, 31);
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
// Gathers vertices from the warp's words, take(w, x, y) giving each lane's two
// bitmap words, and calls f for them: the words are all looked at before any
// work where the queue holds what they hold (a wave touches a few vertices in
// each, which then share one step). Returns whether there was any. One place
// calls f: its code is long, and copies of it cost more than they save. When no
// bits are left, more(Q) may fill the queue with what f found.
template <class T, class F, class M>
__device__ __forceinline__ bool prop_gather(const PropSlice& P, PropQueue& Q, T&& take, F&& f, M&& more) {
    bool did = false;
    uint32_t x = 0, y = 0;
    long long w = 0;
    for (long long b = 0;;) {
        bool left = __any_sync(kFull, (x | y) != 0);
        while (!left && b < P.cnt) {
            const long long i = b + lane_id();
            w = P.word(i);
            x = y = 0;
            left = take(i < P.cnt && w < P.nw, w, x, y);
            b += 32;
        }
        if (left) {
            did = true;
            prop_queue_bits(Q, x, y, w);
            left = __any_sync(kFull, (x | y) != 0);
        }
        if (!left && b < P.cnt) continue;
        if (Q.cnt == 0) return did;
        prop_drain(Q, f);
        if (!left) more(Q);
    }
}
// f(has, v) for the active vertices of the warp's words.
template <class Op, class F>
__device__ __forceinline__ void prop_for_active(const PropGraph<Op>& G, const PropSlice& P, uint32_t* q, F&& f) {
    PropQueue Q{q, 0};
    prop_gather(
        P, Q,
        [&](bool in, long long w, uint32_t& x, uint32_t&) {
            x = in ? G.active(w) : 0u;
            return __any_sync(kFull, x != 0) != 0;
        },
        [&](bool has, int v, int) { f(has, v); }, [](PropQueue&) {});
}

// The marks of a warp's raises, kept in shared memory until one fence covers
// them: whoever takes a mark then sees the raise.
struct PropMarks {
    uint32_t* buf;  // kPropMarks entries of the warp: vertex | direction << 31
    int cnt;        // warp-uniform
};
template <class S, class Op>
__device__ __forceinline__ void prop_flush(const PropGraph<Op>& G, PropMarks& M) {
    if (M.cnt == 0) return;
    __syncwarp();
    S::fence();
    for (int i = lane_id(); i < M.cnt; i += 32) {
        const uint32_t c = M.buf[i], w = c & 0x7fffffffu;
        atomicOr(&(Op::kDirs > 1 && (c >> 31) ? G.d[Op::kDirs - 1] : G.d[0])[w >> 5], 1u << (w & 31));
    }
    M.cnt = 0;
    __syncwarp();
}

// Puts the row of c (vertex | direction << 31) up for the warps to share: the
// slot, or -1 when all are in use. One thread calls.
template <class S>
__device__ __forceinline__ int prop_post(PropCtl* ctl, uint32_t c, int len) {
    constexpr unsigned int kAll = (1u << kPropTasks) - 1;
    unsigned int t = ld_volatile(&ctl->taken);
    for (int i = 0; i < kPropTasks && (t & kAll) != kAll; ++i) {
        const int j = __ffs(~t) - 1;
        t = atomicOr(&ctl->taken, 1u << j);
        if ((t >> j) & 1u) continue;
        PropTask& T = ctl->task[j];
        // open before there is a piece to claim: whoever takes the last one then
        // closes the slot for certain (a claim may come from an earlier look)
        *(volatile uint32_t*)&T.v = c;
        atomicOr(&ctl->open, 1u << j);
        S::fence();
        atomicExch(&T.next, (unsigned long long)((len - 1) / kPropPiece + 1) << 32);
        return j;
    }
    return -1;
}
// The next piece of the row in slot j, if any is left: its vertex | direction
// << 31 in *c. One thread calls. The slot is free once every claimer has read v.
template <class S>
__device__ __forceinline__ bool prop_claim(PropCtl* ctl, int j, uint32_t* c, unsigned int* piece) {
    PropTask& T = ctl->task[j];
    const unsigned long long x = atomicAdd(&T.next, 1ull);
    const unsigned int p = (unsigned int)x, pieces = (unsigned int)(x >> 32);
    if (p >= pieces) return false;
    S::fence();
    *c = ld_volatile(&T.v);
    *piece = p;
    if (p + 1 == pieces) atomicAnd(&ctl->open, ~(1u << j));
    S::fence();
    if (atomicAdd(&T.read, 1u) + 1 == pieces) {
        *(volatile unsigned int*)&T.read = 0;
        atomicExch(&T.next, 0ull);
        S::fence();
        atomicAnd(&ctl->taken, ~(1u << j));
    }
    return true;
}

// The warp marks the heads it raised among t, whose vertices are w (< 0: none).
template <class S, class Op>
__device__ __forceinline__ void prop_raise(const PropGraph<Op>& G, const int (&w)[kPropUnroll],
                                           const typename Op::Val (&t)[kPropUnroll], const typename Op::Val& to,
                                           typename Op::Val* ts, int tdir, PropMarks& M) {
#pragma unroll
    for (int u = 0; u < kPropUnroll; ++u) {
        const bool up = w[u] >= 0 && Op::gains(to, t[u]);
        if (up) Op::raise(ts, w[u], to);
        const uint32_t m = __ballot_sync(kFull, up);
        if (up) M.buf[M.cnt + __popc(m & lanemask_lt())] = (uint32_t)w[u] | ((uint32_t)tdir << 31);
        M.cnt += __popc(m);
    }
    if (M.cnt > kPropMarks - 32 * kPropUnroll) prop_flush<S>(G, M);
}
// Arcs [b0, b1) of a row of direction dir, whose vertex holds st, by the warp.
template <class S, class Op>
__device__ __forceinline__ void prop_relax_row(const PropGraph<Op>& G, const typename Op::Val& st, int b0, int b1, int dir,
                                               PropMarks& M) {
    using Val = typename Op::Val;
    constexpr int U = kPropUnroll;
    const int32_t* adj = dir ? G.adj[1] : G.adj[0];
    Val* s = dir ? G.s[Op::kDirs - 1] : G.s[0];
    row_steps<U>(b0, b1, lane_id(), 32, [&](const uint32_t (&x)[U]) {
        int w[U];
        Val t[U];
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = x[u] != kNoArc ? S::ld(&adj[x[u]]) : -1;
#pragma unroll
        for (int u = 0; u < U; ++u) t[u] = w[u] >= 0 ? Op::load(s, w[u]) : Op::none();
        prop_raise<S>(G, w, t, st, s, dir, M);
    });
}

// A hub's row is long: by one warp it takes 9 ns an arc, with all others waiting
// for what lies behind it. So it is put up in pieces, and idle warps take some: the
// row of `put` (vertex | direction << 31; kFull: none) first, then those in
// `slots`. Returns the number of marks in mk. Only searches of graphs that have
// such rows are compiled with it (kHubs): lattices lost 4-6% to its registers.
// One call, 64 sources, GB300, by one warp against shared: a star of 1 M two-way
// arcs 24.3 -> 0.13 ms, 16 stars of 65 k 13.5 -> 0.30; SCC of the 16 stars 49.7 ->
// 2.0 ms; pieces of 1024 there 2.2, of 256 2.0. The bound: a contracted k-NN graph of
// 1 M points has rows of up to 3.3 k arcs, which cost its run 1089 -> 1146 us when
// shared, and one of a 2D torus 700^2 with p = 0.7 rows of 8 k, 629 -> 525.
template <class S, class Op>
__device__ __noinline__ int prop_share(const PropGraph<Op> G, PropCtl* ctl, uint32_t put, uint32_t slots, uint32_t* mk,
                                       int cnt) {
    constexpr int D = Op::kDirs - 1;
    PropMarks M{mk, cnt};
    unsigned long long arcs = 0;
    auto row = [&](uint32_t c, int& b0, int& b1) {
        const int v = (int)(c & 0x7fffffffu), d = (int)(c >> 31);
        b0 = S::ld(&(d ? G.off[1] : G.off[0])[v]);
        b1 = S::ld(&(d ? G.end[1] : G.end[0])[v]);
    };
    int whole = 0;  // no slot was free: one piece, the row
    if (put != kFull) {
        int b0, b1, j = -1;
        row(put, b0, b1);
        if (lane_id() == 0) j = prop_post<S>(ctl, put, b1 - b0);
        j = __shfl_sync(kFull, j, 0);
        if (j >= 0) slots = 1u << j;
        else whole = 1;
    }
    for (; slots | whole; slots &= slots - 1) {
        for (;;) {
            uint32_t c = put;
            int b0, b1;
            if (!whole) {
                unsigned int piece = 0;
                bool got = false;
                if (lane_id() == 0) got = prop_claim<S>(ctl, __ffs(slots) - 1, &c, &piece);
                if (!__shfl_sync(kFull, (int)got, 0)) break;
                c = __shfl_sync(kFull, c, 0);
                piece = __shfl_sync(kFull, piece, 0);
                row(c, b0, b1);
                b0 += (int)piece * kPropPiece;
                if (b1 - b0 > kPropPiece) b1 = b0 + kPropPiece;
            } else {
                row(c, b0, b1);
            }
            const int d = D ? (int)(c >> 31) : 0;
            prop_relax_row<S>(G, Op::load(d ? G.s[D] : G.s[0], c & 0x7fffffffu), b0, b1, d, M);
            arcs += (unsigned long long)(b1 - b0);
            if (whole) break;
        }
        whole = 0;
    }
    if (lane_id() == 0 && arcs) atomicAdd(&ctl->arcs, arcs);
    return M.cnt;
}

// Spread v's value along its arcs in direction dir; all lanes of the warp call.
// again: the vertices are those the warp has just raised. A long row among them is
// left to the owner of its mark, where the raises of many warps meet: a star of
// 131 k two-way arcs, 64 sources, 0.98 ms without that, 0.1 with it.
template <class S, bool kHubs, class Op>
__device__ __forceinline__ void prop_relax(const PropGraph<Op>& G, const Op& op, PropCtl* ctl, bool has, int v, int dir,
                                           bool again, PropMarks& M, unsigned long long& arcs) {
    using Val = typename Op::Val;
    constexpr int D = Op::kDirs - 1;
    const int lane = lane_id();
    if constexpr (D == 0) dir = 0;
    const int32_t* off = dir ? G.off[1] : G.off[0];
    const int32_t* end = dir ? G.end[1] : G.end[0];
    const int32_t* adj = dir ? G.adj[1] : G.adj[0];
    Val* s = dir ? G.s[D] : G.s[0];
    int o0 = 0, o1 = 0;
    Val st = Op::none();
    if (has) {
        st = Op::load(s, v);
        o0 = S::ld(&off[v]);
        o1 = S::ld(&end[v]);
    }
    if constexpr (Op::kNamed) {
        if (has) {
            const uint32_t r = op.named(st);
            if (r != (uint32_t)v && r < (uint32_t)G.n) {
                const Val t = Op::load(s, r);
                if (Op::gains(t, st)) {
                    st = t;
                    Op::raise(s, v, t);
                }
            }
        }
    }
    constexpr int U = kPropUnroll;
    const bool big = o1 - o0 > kPropBigRow;
    const int len = big ? 0 : o1 - o0;
    arcs += (unsigned long long)len;
    const int most = __reduce_max_sync(kFull, len);
    for (int k = 0; k < most; k += U) {
        int w[U];
        Val t[U];
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = k + u < len ? S::ld(&adj[o0 + k + u]) : -1;
#pragma unroll
        for (int u = 0; u < U; ++u) t[u] = w[u] >= 0 ? Op::load(s, w[u]) : Op::none();
        prop_raise<S>(G, w, t, st, s, dir, M);
    }
    for (uint32_t bm = __ballot_sync(kFull, big); bm; bm &= bm - 1) {  // long rows by the whole warp
        const int l = __ffs(bm) - 1;
        if (again) {
            if (lane == l) {
                S::fence();
                atomicOr(&(dir ? G.d[D] : G.d[0])[v >> 5], 1u << (v & 31));
            }
            continue;
        }
        const Val bst = prop_shfl(st, l);
        const int b0 = __shfl_sync(kFull, o0, l), b1 = __shfl_sync(kFull, o1, l);
        const int bdir = D ? __shfl_sync(kFull, dir, l) : 0;
        if constexpr (kHubs)
            if (b1 - b0 > kPropHub && S::blocks() > 1) {
                M.cnt = prop_share<S, Op>(G, ctl, (uint32_t)__shfl_sync(kFull, v, l) | ((uint32_t)bdir << 31), 0, M.buf, M.cnt);
                continue;
            }
        prop_relax_row<S>(G, bst, b0, b1, bdir, M);
        if (lane == 0) arcs += (unsigned long long)(b1 - b0);
    }
}

// One pull of v: its values take what its in-class neighbours (and, with jump,
// the vertex each names) hold. v's words are written by its owner
// alone, so there is no atomic. Returns bit d set when direction d grew. Rows of
// more than `most_row` arcs are left out.
template <class S, class Op>
__device__ __forceinline__ int prop_pull(const PropGraph<Op>& G, const Op& op, bool has, int v, bool jump,
                                         int most_row = INT32_MAX) {
    using Val = typename Op::Val;
    constexpr int D = Op::kDirs, U = kPropUnroll;
    using Part = typename Op::Part;
    Val s0[D];
    Part st[D];
    int e0[D], len[D];
    bool big = false;
    int most = 0;
#pragma unroll
    for (int d = 0; d < D; ++d) {  // a value that travels along a graph comes in along the other
        const int32_t* off = G.off[1 - d];
        e0[d] = has ? S::ld(&off[v]) : 0;
        len[d] = has ? S::ld(&G.end[1 - d][v]) - e0[d] : 0;
        if (len[d] > most_row) len[d] = 0;
        s0[d] = has ? Op::load(G.s[d], v) : Op::none();
    }
#pragma unroll
    for (int d = 0; d < D; ++d) {
        st[d] = Part{};
        if (Op::kNamed && jump && has) {
            const uint32_t r = op.named(s0[d]);
            if (r != (uint32_t)v && r < (uint32_t)G.n) st[d] = Op::part(s0[d], Op::load(G.s[d], r));
        }
        big |= len[d] > kPropBigRow;
        most = max(most, len[d]);
    }
    if (big) most = 0;
    for (int k = 0; k < most; k += U) {
        int w[D][U];
        Val t[D][U];
#pragma unroll
        for (int d = 0; d < D; ++d)
#pragma unroll
            for (int u = 0; u < U; ++u) w[d][u] = k + u < len[d] ? S::ld(&G.adj[1 - d][e0[d] + k + u]) : -1;
#pragma unroll
        for (int d = 0; d < D; ++d)
#pragma unroll
            for (int u = 0; u < U; ++u) t[d][u] = w[d][u] >= 0 ? Op::load(G.s[d], w[d][u]) : Op::none();
#pragma unroll
        for (int d = 0; d < D; ++d)
#pragma unroll
            for (int u = 0; u < U; ++u) st[d] = Op::fold(st[d], Op::part(s0[d], t[d][u]));
    }
    uint32_t bm = __ballot_sync(kFull, big);
    while (bm) {  // long rows by the whole warp
        const int l = __ffs(bm) - 1;
        bm &= bm - 1;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const int b0 = __shfl_sync(kFull, e0[d], l), b1 = b0 + __shfl_sync(kFull, len[d], l);
            const Val own = prop_shfl(s0[d], l);
            Part m = Part{};
            row_steps<U>(b0, b1, lane_id(), 32, [&](const uint32_t (&x)[U]) {
                int w[U];
                Val t[U];
#pragma unroll
                for (int u = 0; u < U; ++u) w[u] = x[u] != kNoArc ? S::ld(&G.adj[1 - d][x[u]]) : -1;
#pragma unroll
                for (int u = 0; u < U; ++u) t[u] = w[u] >= 0 ? Op::load(G.s[d], w[u]) : Op::none();
#pragma unroll
                for (int u = 0; u < U; ++u) m = Op::fold(m, Op::part(own, t[u]));
            });
            for (int x = 16; x >= 1; x >>= 1) m = Op::fold(m, prop_shfl_xor(m, x));
            if (lane_id() == l) st[d] = Op::fold(st[d], m);
        }
    }
    int up = 0;
#pragma unroll
    for (int d = 0; d < D; ++d)
        if (has && Op::more(st[d], s0[d])) {
            Op::store(G.s[d], v, Op::with(s0[d], st[d]));
            up |= 1 << d;
        }
    return up;
}

// The grid, with a barrier that takes one round trip less than grid_sync: the
// arrivals are tickets of a count that only grows (zero at the launch), so a
// block need not read a generation before it arrives, and no last arrival has to
// release the others. What all threads read behind it is read by one thread of
// each block (f) and handed round, instead of by every warp from one word. Create,
// run and destroy of a 2D torus 33^2 264 -> 240 us, 256^2 1216 -> 1133, k-NN of 1 M
// points 1541 -> 1482.
struct PropGrid : GridScope {
    template <class F>
    __device__ __forceinline__ static bool sync_then(GridBarrier* b, int* err, unsigned long long& val, F&& f) {
        __shared__ unsigned long long s_val;
        __shared__ int s_ok;
        __syncthreads();
        if (threadIdx.x == 0) {
            int ok = 1;
            __threadfence();
            if (gridDim.x > 1) {
                unsigned long long* at = reinterpret_cast<unsigned long long*>(b);
                const unsigned long long end = (atomicAdd(at, 1ull) / gridDim.x + 1) * gridDim.x;
                const uint64_t t0 = globaltimer_ns();
                for (int it = 0; ld_volatile(at) < end; ++it) {
                    if (gridDim.x > 128) __nanosleep(32);  // so many polls get in the way of the arrivals
                    if ((it & 63) == 63 && globaltimer_ns() - t0 > kBarrierTimeoutNs) {
                        atomicCAS(err, 0, SCC_ERR_TIMEOUT);
                        ok = 0;
                        break;
                    }
                }
                __threadfence();
            }
            s_val = f();
            s_ok = ok;
        }
        __syncthreads();
        val = s_val;
        return s_ok != 0;
    }
    __device__ __forceinline__ static bool sync(GridBarrier* b, int* err) {
        unsigned long long x;
        return sync_then(b, err, x, [] { return 0ull; });
    }
};

// A warp's idle state within its block, and the block's within the grid.
template <class S, bool kHubs>
struct PropIdle {
    PropCtl* ctl;
    PropShared& sh;
    bool idle = false;
    __device__ __forceinline__ PropIdle(PropCtl* c, PropShared& s) : ctl(c), sh(s) {}
    __device__ __forceinline__ void wake() {
        if (!idle) return;
        idle = false;
        if (lane_id() == 0 && atomicSub(&sh.idle, 1) == (int)(blockDim.x >> 5) && S::blocks() > 1)
            atomicAdd(&ctl->idle, 0xffffu);  // one idle block less, one woken more
    }
    // after a pass over the warp's words that found nothing: true when the
    // search is over (or a wait ran out); open: the rows to help with
    __device__ __forceinline__ bool rest(uint32_t& open) {
        if (!idle) {
            idle = true;
            if (lane_id() == 0) {
                S::fence();
                if (atomicAdd(&sh.idle, 1) == (int)(blockDim.x >> 5) - 1) {
                    if (S::blocks() > 1) atomicAdd(&ctl->idle, 1u);
                    else atomicExch(&sh.exit, 1);
                }
            }
            if (threadIdx.x == 0) {
                sh.t0 = 0;
                sh.polls = 0;
            }
            __syncwarp();
        } else if (threadIdx.x == 0 && S::blocks() > 1) {
            const unsigned long long x = ld_volatile(reinterpret_cast<unsigned long long*>(&ctl->idle));
            if (kHubs) *(volatile unsigned int*)&sh.open = (unsigned int)(x >> 32);
            const unsigned int seen = (unsigned int)x & 0xffff0000u;
            if ((int)(int16_t)(unsigned int)x >= S::blocks()) {
                atomicExch(&sh.exit, 1);
            } else if ((++sh.polls & 63) == 0) {  // the timer is slow to read
                const uint64_t now = globaltimer_ns();
                if (seen != sh.woken || sh.t0 == 0) {  // a chain of vertices may keep others at work for as long as it is
                    sh.woken = seen;
                    sh.t0 = now;
                } else if (now - sh.t0 > sh.idle_ns) {
                    atomicCAS(&ctl->err, 0, SCC_ERR_TIMEOUT);
                    atomicExch(&sh.exit, 1);
                }
            }
        }
        const int ex = lane_id() == 0 ? ld_volatile(&sh.exit) : 0;
        if (kHubs) open = __shfl_sync(kFull, lane_id() == 0 ? ld_volatile(&sh.open) : 0u, 0);
        return __shfl_sync(kFull, ex, 0) != 0;
    }
};
// Ends a check (every block has arrived at its first barrier and looked for
// work left): *more says whether any block found some. False: a barrier timed out.
template <class S>
__device__ __forceinline__ bool prop_checked(PropCtl* ctl, PropShared& sh, unsigned int check, bool left, bool* more) {
    if (__any_sync(kFull, left) && lane_id() == 0) atomicMax(&ctl->found, check);
    if (S::block() == 0 && threadIdx.x == 0) *(volatile unsigned int*)&ctl->idle = 0;  // no block counts itself in between the two barriers
    unsigned long long x;
    if (!S::sync_then(&ctl->bar, &ctl->err, x, [&] {
            sh.idle = sh.exit = 0;
            sh.open = 0;
            return (unsigned long long)(uint32_t)ld_volatile(&ctl->err) << 32 | ld_volatile(&ctl->found);
        }))
        return false;
    *more = (uint32_t)x == check;
    return (x >> 32) == 0;
}

// A search by pulling alone. With one word per warp a lane keeps its vertex's
// values and the first arcs of its rows in registers, so a pass, and with it a
// hop, costs one round of loads (a longer row one more for every kPropUnroll
// arcs); the vertex a value names is looked at in the same round.
template <class S, class Op>
__device__ bool prop_search_pull(const PropGraph<Op>& G, const Op op, PropCtl* ctl, PropShared& sh, unsigned int& check,
                                 unsigned long long& items) {
    using Val = typename Op::Val;
    using Part = typename Op::Part;
    constexpr int D = Op::kDirs, U = kPropUnroll;
    const PropSlice P = prop_slice<S>(G.n);
    const int lane = lane_id();
    if (threadIdx.x == 0) {
        sh.idle = sh.exit = 0;
        sh.open = 0;
    }
    __syncthreads();
    const bool one = P.cnt == 1 && P.word(0) < P.nw;
    const int v = (int)(P.word(0) * 32) + lane;
    const bool has = one && ((G.active(P.word(0)) >> lane) & 1u);
    Val st[D];
    int w[D][U], e0[D], len[D], most = 0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
        st[d] = has ? Op::load(G.s[d], v) : Op::none();
        e0[d] = has ? S::ld(&G.off[1 - d][v]) : 0;
        len[d] = has ? S::ld(&G.end[1 - d][v]) - e0[d] : 0;
        most = max(most, len[d]);
#pragma unroll
        for (int u = 0; u < U; ++u) w[d][u] = u < len[d] ? S::ld(&G.adj[1 - d][e0[d] + u]) : -1;
    }
    most = __reduce_max_sync(kFull, most);
    const bool fits = one && most <= 4 * U;
    auto pass_one = [&]() {
        Val t[D][U], j[D];
        Part m[D];
#pragma unroll
        for (int d = 0; d < D; ++d) {
            j[d] = Op::none();
            if constexpr (Op::kNamed) {
                const uint32_t r = op.named(st[d]);
                if (has && r < (uint32_t)G.n) j[d] = Op::load(G.s[d], r);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) t[d][u] = w[d][u] >= 0 ? Op::load(G.s[d], w[d][u]) : Op::none();
        }
#pragma unroll
        for (int d = 0; d < D; ++d) {
            m[d] = Op::part(st[d], j[d]);
#pragma unroll
            for (int u = 0; u < U; ++u) m[d] = Op::fold(m[d], Op::part(st[d], t[d][u]));
        }
        for (int k = U; k < most; k += U) {  // warp-uniform
            int x[D][U];
#pragma unroll
            for (int d = 0; d < D; ++d)
#pragma unroll
                for (int u = 0; u < U; ++u) x[d][u] = k + u < len[d] ? S::ld(&G.adj[1 - d][e0[d] + k + u]) : -1;
#pragma unroll
            for (int d = 0; d < D; ++d)
#pragma unroll
                for (int u = 0; u < U; ++u) t[d][u] = x[d][u] >= 0 ? Op::load(G.s[d], x[d][u]) : Op::none();
#pragma unroll
            for (int d = 0; d < D; ++d)
#pragma unroll
                for (int u = 0; u < U; ++u) m[d] = Op::fold(m[d], Op::part(st[d], t[d][u]));
        }
        bool up = false;
#pragma unroll
        for (int d = 0; d < D; ++d)
            if (has && Op::more(m[d], st[d])) {
                st[d] = Op::with(st[d], m[d]);
                Op::store(G.s[d], v, st[d]);
                up = true;
                ++items;
            }
        return __any_sync(kFull, up) != 0;
    };
    auto pass_all = [&](bool jump) {
        bool up = false;
        for (long long i = 0; i < P.cnt; ++i) {
            const long long wd = P.word(i);
            const uint32_t x = wd < P.nw ? G.active(wd) : 0u;
            if (x == 0) continue;  // warp-uniform
            const int c = prop_pull<S>(G, op, (x >> lane) & 1u, (int)(wd * 32) + lane, jump);
            up |= c != 0;
            items += (unsigned long long)__popc(c);
        }
        return __any_sync(kFull, up) != 0;
    };
    for (;;) {
        PropIdle<S, false> id(ctl, sh);
        uint32_t open;
        for (;;) {
            if (fits ? pass_one() : pass_all(true)) id.wake();
            else if (id.rest(open)) break;
        }
        if (!S::sync(&ctl->bar, &ctl->err)) return false;
        ++check;
        const bool left = fits ? pass_one() : pass_all(false);
        bool more = false;
        if (!prop_checked<S>(ctl, sh, check, left, &more)) return false;
        if (!more) return true;
    }
}

// One search: spread until no vertex is dirty. Every thread of the scope calls
// it; `check` numbers the checks of the launch (the same in every block). With
// a deadline (globaltimer ns; 0: none) it may end early, vertices still dirty.
// Returns false when a wait ran out (the caller returns at once).
template <class S, bool kHubs, class Op>
__device__ bool prop_search(const PropGraph<Op>& G, const Op op, PropCtl* ctl, PropShared& sh, uint32_t* q, uint32_t* mk,
                            unsigned int& check, uint64_t deadline, unsigned long long& items,
                            unsigned long long& arcs) {
    using Val = typename Op::Val;
    constexpr int D = Op::kDirs;
    const int lane = lane_id();
    const PropSlice P = prop_slice<S>(G.n);
    if (threadIdx.x == 0) {
        sh.idle = sh.exit = 0;
        sh.open = 0;
    }
    __syncthreads();
    PropMarks M{mk, 0};
    PropQueue Q{q, 0};
    long long turn = 0;  // the word whose named vertices are looked at next
    for (;;) {
        PropIdle<S, kHubs> id(ctl, sh);
        uint32_t help = 0;  // rows of others to help with
        for (;;) {
            int hops = 0;
            bool did = prop_gather(
                P, Q,
                [&](bool in, long long w, uint32_t& x, uint32_t& y) {
                    x = in ? ld_volatile(&G.d[0][w]) : 0u;
                    y = D > 1 && in ? ld_volatile(&G.d[D - 1][w]) : 0u;
                    if (!__any_sync(kFull, (x | y) != 0)) return false;
                    id.wake();
                    if (x) x = atomicExch(&G.d[0][w], 0u);
                    if (y) y = atomicExch(&G.d[D - 1][w], 0u);
                    S::fence();
                    items += (unsigned long long)(__popc(x) + __popc(y));
                    return __any_sync(kFull, (x | y) != 0) != 0;
                },
                [&](bool has, int v, int dir) { prop_relax<S, kHubs>(G, op, ctl, has, v, dir, hops > 0, M, arcs); },
                [&](PropQueue& Q) {
                    if (M.cnt > kPropNarrow || hops == kPropHops) return;
                    ++hops;
                    __syncwarp();
                    if (lane < M.cnt) Q.buf[lane] = M.buf[lane];
                    Q.cnt = M.cnt;
                    M.cnt = 0;
                    __syncwarp();
                });
            if constexpr (kHubs)
                if (help) {
                    id.wake();
                    M.cnt = prop_share<S, Op>(G, ctl, kFull, help, M.buf, M.cnt);
                    if (lane == 0) atomicAnd(&sh.open, ~help);  // no pieces left there
                    help = 0;
                    did = true;
                }
            if (did) prop_flush<S>(G, M);
            // nothing dirty: look whether the vertex that a value of the next
            // word names holds a larger one itself (paths are walked hop by
            // hop; this takes the rest of one in a step)
            if constexpr (Op::kNamed) {
                if (!did && P.cnt > 0 && !deadline) {
                    if (++turn >= P.cnt) turn = 0;
                    const long long w = P.word(turn);
                    const uint32_t a = w < P.nw ? G.active(w) : 0u;
                    uint32_t up[D];
                    uint32_t any = 0;
                    if (a != 0) {  // warp-uniform
                        const bool has = (a >> lane) & 1u;
                        const long long v = w * 32 + lane;
                        Val st[D], t[D];
#pragma unroll
                        for (int d = 0; d < D; ++d) st[d] = has ? Op::load(G.s[d], v) : Op::none();
#pragma unroll
                        for (int d = 0; d < D; ++d) {
                            const uint32_t r = op.named(st[d]);
                            t[d] = has && r != (uint32_t)v && r < (uint32_t)G.n ? Op::load(G.s[d], r) : Op::none();
                        }
#pragma unroll
                        for (int d = 0; d < D; ++d) {
                            const bool u = has && Op::gains(t[d], st[d]);
                            if (u) Op::raise(G.s[d], v, t[d]);
                            up[d] = __ballot_sync(kFull, u);
                            any |= up[d];
                        }
                    }
                    if (any) {
                        did = true;
                        id.wake();
                        S::fence();
                        __syncwarp();
#pragma unroll
                        for (int d = 0; d < D; ++d)
                            if (lane == 0 && up[d]) atomicOr(&G.d[d][w], up[d]);
                    }
                }
            }
            if (!did && id.rest(help)) break;
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
            for (long long i = lane; i < P.cnt; i += 32) {
                const long long w = P.word(i);
                if (w >= P.nw) continue;
#pragma unroll
                for (int d = 0; d < D; ++d) left |= ld_volatile(&G.d[d][w]) != 0;
            }
        bool more = false;
        if (!prop_checked<S>(ctl, sh, check, left, &more)) return false;
        if (!more) return true;
    }
}

// Whether a vertex w != v of v's class (lab) is in v's row [o0, o1): by one thread
// (lanes = 1), or by the warp, all of whose lanes call.
template <class S, int kLanes>
__device__ __forceinline__ bool prop_any_in_class(const int32_t* adj, int o0, int o1, const unsigned long long* s,
                                                  uint32_t lab, int v) {
    constexpr int U = kLanes == 1 ? 2 : kPropUnroll;
    bool found = false;
    row_steps<U>(o0, o1, kLanes == 1 ? 0 : lane_id(), kLanes, [&](const uint32_t (&x)[U]) {
        int w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = x[u] != kNoArc ? S::ld(&adj[x[u]]) : v;
        uint32_t l[U];
#pragma unroll
        for (int u = 0; u < U; ++u) l[u] = (uint32_t)(ld_volatile(&s[w[u]]) >> 32);
#pragma unroll
        for (int u = 0; u < U; ++u) found |= l[u] == lab && w[u] != v;
        if constexpr (kLanes > 1) found = __any_sync(kFull, found) != 0;
        return !found;
    });
    return found;
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
    const unsigned int at = step++ & 3;
    return S::sync_then(&ctl->bar, &ctl->err, sum, [&] { return ld_volatile(&ctl->count[at]); });
}

// The active vertices with a row of more than kPropHub arcs, into hub (a word a
// vertex), their number ctl->nhub. Ends at a barrier.
template <class S>
__device__ __forceinline__ bool prop_list_hubs(const PropGraph<PropMax>& G, PropCtl* ctl, int32_t* hub) {
    const PropSlice P = prop_slice<S>(G.n);
    for (long long i = 0; i < P.cnt; ++i) {
        const long long w = P.word(i);
        if (w >= P.nw) break;
        if (!((G.act[w] >> lane_id()) & 1u)) continue;
        const int v = (int)(w * 32) + lane_id();
        if (max(S::ld(&G.end[0][v]) - S::ld(&G.off[0][v]), S::ld(&G.end[1][v]) - S::ld(&G.off[1][v])) > kPropHub)
            hub[atomicAdd(&ctl->nhub, 1u)] = v;
    }
    if (S::block() == 0 && threadIdx.x == 0) ctl->hub = hub;
    __syncwarp();
    return S::sync(&ctl->bar, &ctl->err);
}

// The long rows that a sweep left out, in pieces dealt out to all warps, 32 hubs
// at a time: a piece's vertex is raised by an atomic, and is dirty if it was.
// Returns the raises.
template <class S>
__device__ __forceinline__ unsigned long long prop_pull_hubs(const PropGraph<PropMax>& G, const PropSlice& P,
                                                             const int32_t* hub, unsigned int nhub) {
    constexpr int U = kPropUnroll;
    const int lane = lane_id();
    unsigned long long cnt = 0;
    long long first = 0;  // the warp that takes the next piece
    for (unsigned int j0 = 0; j0 < nhub; j0 += 32) {
        const int v = j0 + lane < nhub ? hub[j0 + lane] : -1;
        const bool on = v >= 0 && ((G.act[v >> 5] >> (v & 31)) & 1u);
        for (int d = 0; d < 2; ++d) {
            const int b0 = on ? S::ld(&G.off[1 - d][v]) : 0, len = on ? S::ld(&G.end[1 - d][v]) - b0 : 0;
            const int mine = len > kPropHub ? (len - 1) / kPropPiece + 1 : 0;
            const int incl = warp_incl_scan(mine);  // 2^31 / kPropPiece and 32 in all at most
            const int all = __shfl_sync(kFull, incl, 31);
            long long p = P.wid - first;
            if (p < 0) p += P.warps;
            first = (first + all) % P.warps;
            for (; p < all; p += P.warps) {
                const int l = __popc(__ballot_sync(kFull, incl <= (int)p));  // the first lane with incl > p
                const int hv = __shfl_sync(kFull, v, l), hlen = __shfl_sync(kFull, len, l);
                const int at = ((int)p - __shfl_sync(kFull, incl - mine, l)) * kPropPiece;
                const int lo = __shfl_sync(kFull, b0, l) + at;
                const unsigned long long own = PropMax::load(G.s[d], hv);
                uint32_t m = 0;
                row_steps<U>(lo, lo + min(hlen - at, kPropPiece), lane, 32, [&](const uint32_t (&x)[U]) {
                    int w[U];
                    unsigned long long t[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) w[u] = x[u] != kNoArc ? S::ld(&G.adj[1 - d][x[u]]) : -1;
#pragma unroll
                    for (int u = 0; u < U; ++u) t[u] = w[u] >= 0 ? PropMax::load(G.s[d], w[u]) : PropMax::none();
#pragma unroll
                    for (int u = 0; u < U; ++u) m = max(m, PropMax::part(own, t[u]));
                });
                m = __reduce_max_sync(kFull, m);
                if (lane == 0 && PropMax::more(m, own)) {
                    PropMax::raise(G.s[d], hv, PropMax::with(own, m));
                    atomicOr(&G.d[d][hv >> 5], 1u << (hv & 31));
                    ++cnt;
                }
            }
        }
    }
    __syncwarp();
    return cnt;
}

// The batches from the state in sf/sb/act until every active vertex is
// finished (`active` of them): trimming inside the classes, the two searches,
// the labelling. The ring of counters starts zero. kPull: the searches only pull. head_ns: time limit of the first batch's head start (0: none);
// with it the state's keys start zero, and the first batch sets them. kHubs: there
// are rows of more than kPropHub arcs, those of the vertices that prop_list_hubs
// listed.
template <class S, bool kPull, bool kHubs>
__device__ __noinline__ bool prop_batches(const PropGraph<PropMax> G, const PropMax op, PropCtl* ctl, PropShared& sh, uint32_t* q, uint32_t* mk,
                             unsigned long long active, uint64_t head_ns) {
    const int lane = lane_id();
    const PropSlice P = prop_slice<S>(G.n);
    unsigned long long *const sf = G.s[0], *const sb = G.s[1];
    unsigned int check = 0;
    unsigned long long items = 0, arcs = 0, done = 0;
    int batches = 0;
    unsigned int step = 0;
    while (done < active) {
        // ---- vertices with no arc from, or no arc to, a vertex of their class
        for (int pass = 0; pass < kPropTrimPasses; ++pass) {
            unsigned long long cnt = 0;
            prop_for_active(G, P, q, [&](bool has, int v) {
                uint32_t lab = 0;
                int o0 = 0, o1 = 0, i0 = 0, i1 = 0;
                if (has) {
                    lab = (uint32_t)(ld_volatile(&sf[v]) >> 32);
                    o0 = S::ld(&G.off[0][v]);
                    o1 = S::ld(&G.end[0][v]);
                    i0 = S::ld(&G.off[1][v]);
                    i1 = S::ld(&G.end[1][v]);
                }
                // a hub is left to the searches, which share its row
                const bool is_hub = kHubs && max(o1 - o0, i1 - i0) > kPropHub;
                // a thread looks at the first arcs of its rows, where most have a
                // neighbour in the class; the rest of a long row without one there
                // is read by the whole warp (rows of more than 64 arcs by the warp
                // from the start: k-NN of 300 k points 545 -> 590 us a run)
                const int oe = o0 + min(o1 - o0, kPropBigRow), ie = i0 + min(i1 - i0, kPropBigRow);
                bool more0 = false, more1 = false;
                bool stays = is_hub;
                if (has && !is_hub) {
                    stays = prop_any_in_class<S, 1>(G.adj[0], o0, oe, sf, lab, v);
                    more0 = !stays && oe < o1;
                    if (stays || more0) {
                        stays = prop_any_in_class<S, 1>(G.adj[1], i0, ie, sf, lab, v);
                        more1 = !stays && ie < i1;
                        stays = stays || more1;
                    }
                }
                for (uint32_t bm = __ballot_sync(kFull, stays && (more0 || more1)); bm; bm &= bm - 1) {
                    const int l = __ffs(bm) - 1, hv = __shfl_sync(kFull, v, l);
                    const uint32_t hl = __shfl_sync(kFull, lab, l);
                    bool in = true;
                    if (__shfl_sync(kFull, (int)more0, l))
                        in = prop_any_in_class<S, 32>(G.adj[0], __shfl_sync(kFull, oe, l), __shfl_sync(kFull, o1, l), sf,
                                                      hl, hv);
                    if (in && __shfl_sync(kFull, (int)more1, l))
                        in = prop_any_in_class<S, 32>(G.adj[1], __shfl_sync(kFull, ie, l), __shfl_sync(kFull, i1, l), sf,
                                                      hl, hv);
                    if (lane == l) stays = in;
                }
                if (!has || stays) return;
                *(volatile unsigned long long*)&sf[v] = prop_pack(kPropDone, 0);
                *(volatile unsigned long long*)&sb[v] = prop_pack(kPropDone, 0);
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
        if constexpr (kPull) {
            if (!prop_search_pull<S>(G, op, ctl, sh, check, items)) return false;
        } else {
            // ---- every active vertex is a source. A head start: the largest
            // source alone, so that a giant SCC is flooded once before the
            // others' values wander through it
            unsigned long long grew = 2 * (active - done);
            if (batches == 0 && head_ns) {
                const uint32_t b = op.vertex(0xffffffffu);
                if (S::block() == 0 && threadIdx.x == 0) {
                    const unsigned long long st = sf[b];
                    if ((uint32_t)(st >> 32) != kPropDone) {
                        sf[b] = sb[b] = st | 0xffffffffull;
                        G.d[0][b >> 5] = G.d[1][b >> 5] = 1u << (b & 31);
                    }
                }
                if (!S::sync(&ctl->bar, &ctl->err)) return false;
                if (!prop_search<S, kHubs>(G, op, ctl, sh, q, mk, check, globaltimer_ns() + head_ns, items, arcs)) return false;
                unsigned long long cnt = 0;
                for (long long i = 0; i < P.cnt; ++i) {
                    const long long w = P.word(i);
                    const uint32_t x = w < P.nw ? G.act[w] : 0u;
                    if (x == 0) continue;  // warp-uniform
                    const long long v = w * 32 + lane;
                    bool f = false, r = false;
                    if ((x >> lane) & 1u) {
                        const unsigned long long a = sf[v], b2 = sb[v];
                        const uint32_t key = op.key((uint32_t)v);
                        f = (uint32_t)a < key;
                        r = (uint32_t)b2 < key;
                        if (f) sf[v] = prop_pack((uint32_t)(a >> 32), key);
                        if (r) sb[v] = prop_pack((uint32_t)(b2 >> 32), key);
                    }
                    const uint32_t mf = __ballot_sync(kFull, f), mr = __ballot_sync(kFull, r);
                    if (lane == 0) {
                        G.d[0][w] |= mf;
                        G.d[1][w] |= mr;
                        cnt += __popc(mf) + __popc(mr);
                    }
                }
                if (!prop_count<S>(ctl, step, cnt, grew)) return false;
            } else {
                for (long long i = lane; i < P.cnt; i += 32) {
                    const long long w = P.word(i);
                    const uint32_t x = w < P.nw ? G.act[w] : 0u;
                    if (x) {
                        G.d[0][w] = x;
                        G.d[1][w] = x;
                    }
                }
                if (!S::sync(&ctl->bar, &ctl->err)) return false;
            }
            // ---- sweeps that pull every active vertex (no atomics, coalesced
            // rows) while the last one raised as many values as vertices were
            // active at first: a sweep costs 12-25 ps a value, marking 42 ps a
            // raise. The last one leaves the vertices it raised dirty
            while (grew >= active) {
                unsigned long long cnt = 0;
                for (long long i = 0; i < P.cnt; ++i) {
                    const long long w = P.word(i);
                    const uint32_t x = w < P.nw ? G.act[w] : 0u;
                    if (x == 0) continue;  // warp-uniform
                    const bool has = (x >> lane) & 1u;
                    const int c = prop_pull<S>(G, op, has, (int)(w * 32) + lane, false, kHubs ? kPropHub : INT32_MAX);
                    const uint32_t cf = __ballot_sync(kFull, c & 1), cb = __ballot_sync(kFull, c & 2);
                    if (lane == 0) {
                        G.d[0][w] = cf;
                        G.d[1][w] = cb;
                        cnt += __popc(cf) + __popc(cb);
                    }
                }
                if constexpr (kHubs) {
                    __syncwarp();
                    if (!S::sync(&ctl->bar, &ctl->err)) return false;
                    cnt += prop_pull_hubs<S>(G, P, ld_volatile(&ctl->hub), ld_volatile(&ctl->nhub));
                }
                items += cnt;
                if (!prop_count<S>(ctl, step, cnt, grew)) return false;
            }
            if (!prop_search<S, kHubs>(G, op, ctl, sh, q, mk, check, 0, items, arcs)) return false;
        }
        // ---- labelling (Alg. 1): equal maxima finish a vertex, the others'
        // class becomes the hash of the old one and the two maxima
        unsigned long long cnt = 0;
        prop_for_active(G, P, q, [&](bool has, int v) {
            if (!has) return;
            const unsigned long long f = ld_volatile(&sf[v]), r = ld_volatile(&sb[v]);
            if (f == r) {
                sf[v] = sb[v] = prop_pack(kPropDone, 0);
                const uint32_t r = op.vertex((uint32_t)f);
                if (r >= (uint32_t)G.n) atomicCAS(&ctl->err, 0, SCC_ERR_INTERNAL);  // never: a value names a vertex
                G.rep[v] = r < (uint32_t)G.n ? (int32_t)r : v;
                atomicAnd(&G.act[v >> 5], ~(1u << (v & 31)));
                ++cnt;
            } else {
                const int32_t lab = class_hash((int32_t)(uint32_t)(f >> 32), (int32_t)(uint32_t)f, (int32_t)(uint32_t)r);
                sf[v] = sb[v] = prop_pack((uint32_t)lab, op.key((uint32_t)v));
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

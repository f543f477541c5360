// Least-element lists (Sec. 5.2, Alg. 5: the BGSS LE-lists algorithm) of the
// undirected graph under the arcs of G, unweighted (sm_103a).
//
// Source v_j (position j of a seeded vertex order) belongs to L(u) iff its hop
// distance to u is smaller than that of every earlier source. Alg. 5 takes the
// sources in batches of 1, 2, 4, ... and runs one multi-source BFS per batch:
//
//   * the BFS is level-synchronous (VGC does not apply: BFS order matters,
//     Sec. 5.2) in one cooperative launch over all batches, a grid barrier
//     after each level;
//   * a frontier item is a (vertex, source) pair; a pair (w, s) is new when it
//     enters the batch's hash table of visited pairs (insert-if-absent, the
//     "parallel hash table" of Sec. 5.2), and it is only tried when level + 1 <
//     delta(w), the distance from w to the closest source of the earlier
//     batches (the pruning of Alg. 5);
//   * new pairs go, with their distance, straight to the log of candidate
//     entries (u, s, d); the entries of one level are the next level's
//     frontier, so a pair is written once and no pass collects the table;
//   * at the end of a batch its part of the log lowers delta(u) (Alg. 5
//     "delta(u) <- min") and the table is emptied.
//
// What bounds it is arcs examined: a few gathers and a table probe each. They
// are spread evenly: a warp takes up to 32 frontier items and walks their arcs
// as one range, four arcs a lane at a time, and rows of more than kLeHub arcs
// are queued in pieces as their pair is logged. New pairs gather in shared
// memory and take places in the log 32 or more at a time, one atomic each. R-MAT
// with 262 k vertices: 15.6 -> 1.54 ms (a warp an item, two atomics on single
// words per 32 arcs, a hub's row by one warp); 79 levels, 35 M arcs. A lattice is
// bound by the level instead, a barrier and a chain of eight accesses: 13.9 ->
// 6.6 us each (90 k vertices, 1415 levels: 19.8 -> 9.4 ms).
//
// A pair with d(s, w) < delta_b(w) is reached at its BFS distance (every vertex
// on a shortest path from s also passes the test), and no other pair is ever
// inserted, so after all batches the candidates at u, sorted by source
// position and kept while their distance strictly decreases (Alg. 5 "sort ...
// filter out triples that violate constraints"), are exactly L(u).
//
// A table over its load limit or a full candidate log stops the launch; the
// host grows the buffer and relaunches from the start of the batch.
#include <algorithm>
#include <climits>
#include <vector>

#include "common.cuh"
#include "engine.cuh"
#include "internal.h"

namespace scc {
namespace {

constexpr unsigned long long kEmpty = ~0ull;
constexpr int kLeProbe = 64;        // probes of an insert before the table counts as full
constexpr int kLeHub = 256;         // longer rows are walked in pieces of this many arcs or more ...
constexpr int kLePieces = 256;      // ... at most so many a row
constexpr int kLeStep = 4;          // arcs a lane takes at a time
constexpr int kLeStage = 32 + 32 * kLeStep;
constexpr int kLeBlock = 1024;      // one block an SM: the fewest to arrive at a barrier
constexpr int kLeWarps = kLeBlock / 32;
constexpr int kLeTableFull = 1, kLeLogFull = 2;

struct LeCtl {
    GridBarrier bar;
    int err;
    int status;                    // 0 done, 1 grow the table, 2 grow the log
    int batch;                     // the batch to resume at
    // Rings over the levels (their index runs on across batches): a level reads
    // its own slot, writes the next one and clears the one after, so a block
    // still deciding about the previous level never sees the next level's writes.
    unsigned long long fr_n[3];    // pairs of the level
    unsigned long long hub_n[3];   // pieces of long rows of the level
    int full[3];                   // kLeTableFull | kLeLogFull met while writing the level
    unsigned long long ins;        // pairs of the batch at which the launch stopped
    unsigned long long log_n;      // candidates of the finished batches
    int levels;                    // BFS levels run (statistics)
    unsigned long long edges;      // arcs examined (statistics)
};

struct LeParams {
    const int32_t* soff;
    const int32_t* sadj;
    int32_t n;
    const int32_t* order;
    const long long* bounds;
    int nb;
    int32_t* delta;
    unsigned long long* keys;  // visited pairs of the batch: w << 32 | s
    unsigned long long mask;   // table capacity - 1
    unsigned long long* log_key;  // u << 32 | s
    int32_t* log_d;
    unsigned long long log_cap;
    int2* row[2];              // rows of a level's pairs (by its parity): first arc, arcs (0: queued)
    unsigned long long* hub_key[2];  // pieces of a level (by its parity): the pair, or kEmpty,
    int32_t* hub_arc[2];             // and the first arc
    unsigned long long hub_cap;
    LeCtl* ctl;
};

__device__ __forceinline__ int le_piece(int deg) {
    const int p = (int)(((long long)deg + kLePieces - 1) / kLePieces);
    return p <= kLeHub ? kLeHub : (int)min(((long long)p + 127) / 128 * 128, 1ll << 30);
}

// Insert-if-absent of key, whose first slot h held cur (or may hold kEmpty);
// true if the key is new. A slot is read before its atomic: most pairs tried are
// there already (R-MAT, 262 k vertices: 1.58 ms by the atomic alone, 1.54 so;
// lattices within 1%). Sets *full past the probe limit.
__device__ __forceinline__ bool le_insert(const LeParams& P, unsigned long long key, unsigned long long h,
                                          unsigned long long cur, int* full) {
    for (int i = 0; i < kLeProbe; ++i) {
        if (cur == key) return false;
        if (cur == kEmpty) {
            cur = atomicCAS(&P.keys[h], kEmpty, key);
            if (cur == kEmpty) return true;
            if (cur == key) return false;
        }
        h = (h + 1) & P.mask;
        cur = ld_volatile(&P.keys[h]);
    }
    atomicOr(full, kLeTableFull);
    return false;
}

// What a level found, the same for every thread of the grid.
struct LeLevel {
    unsigned long long n, hub_n;
    int full;
};

// The barrier after a level, with slot o3 of the rings read behind it. One
// thread a block adds to a count that only grows and polls it, instead of a last
// arrival that releases the others, and reads the slot for its block: a level of
// a lattice is mostly this and a chain of eight accesses, and with the common
// barrier and every warp reading the slot's words itself it was 9.8 us, now 6.6.
// Ends by the time limit.
__device__ __forceinline__ bool le_sync(LeCtl* ctl, unsigned int& target, int o3, LeLevel& lv) {
    __shared__ LeLevel s_lv;
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        target += gridDim.x;
        __threadfence();
        atomicAdd(&ctl->bar.count, 1u);
        int ok = 1;
        const uint64_t t0 = globaltimer_ns();
        for (int it = 0; (int)(ld_volatile(&ctl->bar.count) - target) < 0; ++it)
            if ((it & 63) == 63 && globaltimer_ns() - t0 > kBarrierTimeoutNs) {
                atomicCAS(&ctl->err, 0, SCC_ERR_TIMEOUT);
                ok = 0;
                break;
            }
        __threadfence();
        s_lv.n = ld_volatile(&ctl->fr_n[o3]);
        s_lv.hub_n = ld_volatile(&ctl->hub_n[o3]);
        s_lv.full = ld_volatile(&ctl->full[o3]);
        s_ok = ok;
    }
    __syncthreads();
    lv = s_lv;
    return s_ok != 0;
}

// One level's output: the slot of the rings, the parity of the pieces, where
// the level begins in the log, and its distance.
struct LeOut {
    unsigned long long* n;
    unsigned long long* hub_n;
    int* full;
    int par;
    unsigned long long beg;
    int32_t d;
};

// The pair key of row [a0, a0 + deg) to place `at` of the level, and the row's
// pieces to the queue (a row that does not fit there is walked whole by the warp
// that meets it).
__device__ __forceinline__ void le_put(const LeParams& P, const LeOut& o, unsigned long long key, int a0, int deg,
                                       unsigned long long at) {
    if (deg > kLeHub) {
        const int piece = le_piece(deg);
        const unsigned long long k = (unsigned long long)((deg - 1) / piece + 1);
        const unsigned long long q = atomicAdd(o.hub_n, k);
        const bool fits = q + k <= P.hub_cap;
        for (unsigned long long j = 0; j < k && q + j < P.hub_cap; ++j) {
            P.hub_key[o.par][q + j] = fits ? key : kEmpty;
            P.hub_arc[o.par][q + j] = a0 + (int)j * piece;
        }
        if (fits) deg = 0;
    }
    P.row[o.par][at] = make_int2(a0, deg);  // at < the table's slots: each pair has one
    const unsigned long long x = o.beg + at;
    if (x < P.log_cap) {
        P.log_key[x] = key;
        P.log_d[x] = o.d;
    } else {
        atomicOr(o.full, kLeLogFull);
    }
}

// The warp's staged pairs to the log.
__device__ __forceinline__ void le_flush(const LeParams& P, const LeOut& o, const unsigned long long* stage, int& cnt) {
    __syncwarp();
    unsigned long long base = 0;
    if (lane_id() == 0) base = atomicAdd(o.n, (unsigned long long)cnt);
    base = __shfl_sync(kFull, base, 0);
    for (int i = lane_id(); i < cnt; i += 32) {
        const unsigned long long key = stage[i];
        const int a0 = __ldg(&P.soff[key >> 32]), deg = __ldg(&P.soff[(key >> 32) + 1]) - a0;
        le_put(P, o, key, a0, deg, base + i);
    }
    cnt = 0;
    __syncwarp();
}

// The block's leftovers (fewer than 32 a warp) by one atomic of the block.
__device__ __forceinline__ void le_flush_block(const LeParams& P, const LeOut& o, const unsigned long long* stage,
                                               int& cnt) {
    __shared__ int s_cnt[kLeWarps];
    __shared__ unsigned long long s_base;
    const int warp = threadIdx.x >> 5, lane = lane_id();
    if (lane == 0) s_cnt[warp] = cnt;
    if (!__syncthreads_or(cnt)) return;
    // the rows while the atomic is under way
    unsigned long long key = 0;
    int a0 = 0, a1 = 0;
    if (lane < cnt) {
        key = stage[lane];
        a0 = __ldg(&P.soff[key >> 32]);
        a1 = __ldg(&P.soff[(key >> 32) + 1]);
    }
    int inc = lane < kLeWarps ? s_cnt[lane] : 0;
    for (int d = 1; d < 32; d <<= 1) {
        const int x = __shfl_up_sync(kFull, inc, d);
        if (lane >= d) inc += x;
    }
    const int all = __shfl_sync(kFull, inc, 31), before = __shfl_sync(kFull, inc, warp) - cnt;
    if (threadIdx.x == 0) s_base = atomicAdd(o.n, (unsigned long long)all);
    __syncthreads();
    if (lane < cnt) le_put(P, o, key, a0, a1 - a0, s_base + before + lane);
    cnt = 0;
}

// kLeStep arcs a lane: to w[j] from a pair of source s[j] (w[j] < 0: none).
__device__ __forceinline__ void le_arcs(const LeParams& P, const LeOut& o, const int (&w)[kLeStep],
                                        const uint32_t (&src)[kLeStep], unsigned long long* stage, int& cnt) {
    bool go[kLeStep];
    unsigned long long key[kLeStep], h[kLeStep], cur[kLeStep];
    // delta changes between batches only, before a barrier: plain loads, so the
    // hubs' words come from L1
#pragma unroll
    for (int j = 0; j < kLeStep; ++j) go[j] = w[j] >= 0 && o.d < P.delta[w[j]];
#pragma unroll
    for (int j = 0; j < kLeStep; ++j) {
        key[j] = (unsigned long long)(uint32_t)w[j] << 32 | src[j];
        h[j] = mix64(key[j]) & P.mask;
        cur[j] = go[j] ? ld_volatile(&P.keys[h[j]]) : kEmpty;
    }
#pragma unroll
    for (int j = 0; j < kLeStep; ++j) {
        const bool nw = go[j] && le_insert(P, key[j], h[j], cur[j], o.full);
        const uint32_t m = __ballot_sync(kFull, nw);
        if (nw) stage[cnt + __popc(m & lanemask_lt())] = key[j];
        cnt += __popc(m);
    }
    if (cnt >= 32) le_flush(P, o, stage, cnt);
}

// Arcs [e, end) of the row of u, by the whole warp.
__device__ __forceinline__ void le_row(const LeParams& P, const LeOut& o, uint32_t src, int e, int end,
                                       unsigned long long* stage, int& cnt) {
    for (long long e0 = e; e0 < end; e0 += 32 * kLeStep) {
        int w[kLeStep];
        uint32_t s[kLeStep];
#pragma unroll
        for (int j = 0; j < kLeStep; ++j) {
            const long long x = e0 + 32 * j + lane_id();
            w[j] = x < end ? __ldg(&P.sadj[x]) : -1;
            s[j] = src;
        }
        le_arcs(P, o, w, s, stage, cnt);
    }
}

__global__ void __launch_bounds__(kLeBlock, 1) k_le_lists(LeParams P) {
    __shared__ unsigned long long s_stage[kLeWarps][kLeStage];
    LeCtl* ctl = P.ctl;
    const int lane = lane_id();
    unsigned long long* stage = s_stage[threadIdx.x >> 5];
    int cnt = 0;  // staged pairs of the warp
    const long long gtid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long gstride = (long long)gridDim.x * blockDim.x;
    const long long wid = gtid >> 5, nwarps = gstride >> 5;
    unsigned long long edges = 0;
    const unsigned long long load_limit = (P.mask + 1) / 4 * 3;
    unsigned long long base = ld_volatile(&ctl->log_n);  // the log's end before the batch
    unsigned long long g = 0;                            // levels so far: the rings' index
    int b = ld_volatile(&ctl->batch);
    int status = 0;
    unsigned long long ins = 0;
    unsigned int target = 0;  // arrivals at the barrier so far
    for (; b < P.nb; ++b) {
        // ---- the batch's sources at distance 0
        const long long p0 = P.bounds[b], p1 = P.bounds[b + 1];
        {
            const int o3 = (int)(g % 3);
            const LeOut o{&ctl->fr_n[o3], &ctl->hub_n[o3], &ctl->full[o3], (int)(g & 1), base, 0};
            for (long long q = p0 + (gtid - lane); q < p1; q += gstride) {
                const long long p = q + lane;
                bool nw = false;
                unsigned long long key = 0;
                if (p < p1) {
                    const int s = P.order[p];
                    key = ((unsigned long long)(uint32_t)s << 32) | (uint32_t)s;
                    if (P.delta[s] > 0) {
                        const unsigned long long h = mix64(key) & P.mask;
                        nw = le_insert(P, key, h, kEmpty, o.full);
                    }
                }
                const uint32_t m = __ballot_sync(kFull, nw);
                if (nw) stage[cnt + __popc(m & lanemask_lt())] = key;
                cnt += __popc(m);
                if (cnt >= 32) le_flush(P, o, stage, cnt);
            }
            __syncwarp();
            le_flush_block(P, o, stage, cnt);
        }
        // Every block takes the same decisions below: it reads only counters
        // and flags that no block writes again before the next barrier.
        LeLevel lv;
        if (!le_sync(ctl, target, (int)(g % 3), lv)) return;
        unsigned long long beg = base, n_lev = lv.n;
        int full = lv.full;
        ins = n_lev;
        if (ins > load_limit) full |= kLeTableFull;
        // ---- BFS levels
        for (int lev = 0; !full; ++lev, ++g) {
            const int o3 = (int)((g + 1) % 3);
            const LeOut o{&ctl->fr_n[o3], &ctl->hub_n[o3], &ctl->full[o3], (int)((g + 1) & 1), beg + n_lev, lev + 1};
            const long long nh = (long long)min(lv.hub_n, P.hub_cap);
            if (gtid == 0) {  // read last level, written next level
                const int z = (int)((g + 2) % 3);
                ctl->fr_n[z] = 0;
                ctl->hub_n[z] = 0;
                ctl->full[z] = 0;
                ctl->levels += 1;
            }
            // the queued pieces, a warp each
            for (long long i = wid; i < nh; i += nwarps) {
                const unsigned long long key = P.hub_key[g & 1][i];
                if (key == kEmpty) continue;
                const int u = (int)(key >> 32);
                const int a0 = __ldg(&P.soff[u]), a1 = __ldg(&P.soff[u + 1]), e = P.hub_arc[g & 1][i];
                const int piece = le_piece(a1 - a0);
                const int end = a1 - e > piece ? e + piece : a1;
                le_row(P, o, (uint32_t)key, e, end, stage, cnt);
                if (lane == 0) edges += (unsigned long long)(end - e);
            }
            // the other rows, up to 32 a warp as one range of arcs
            const long long per = max(1ll, min(32ll, ((long long)n_lev + nwarps - 1) / nwarps));
            for (long long i0 = wid * per; i0 < (long long)n_lev; i0 += nwarps * per) {
                // once a buffer is full the batch starts over and the rest of
                // the level is moot: stop taking items
                if (i0 >= nwarps * per) {
                    int stop = lane == 0 ? ld_volatile(o.full) : 0;
                    if (__shfl_sync(kFull, stop, 0) != 0) break;
                }
                uint32_t src = 0;
                int a0 = 0, deg = 0;
                if (lane < per && i0 + lane < (long long)n_lev) {
                    src = (uint32_t)P.log_key[beg + i0 + lane];
                    const int2 r = P.row[g & 1][i0 + lane];
                    a0 = r.x;
                    deg = r.y;
                    edges += (unsigned long long)deg;
                }
                for (uint32_t m = __ballot_sync(kFull, deg > kLeHub); m; m &= m - 1) {  // found no room in the queue
                    const int l = __ffs(m) - 1;
                    const int x = __shfl_sync(kFull, a0, l), d = __shfl_sync(kFull, deg, l);
                    le_row(P, o, __shfl_sync(kFull, src, l), x, x + d, stage, cnt);
                }
                if (deg > kLeHub) deg = 0;
                int inc = deg;
                for (int d = 1; d < 32; d <<= 1) {
                    const int x = __shfl_up_sync(kFull, inc, d);
                    if (lane >= d) inc += x;
                }
                const int total = __shfl_sync(kFull, inc, 31);
                const int first = a0 - (inc - deg);  // arc t of the range is arc first + t of its row
                for (int t0 = 0; t0 < total; t0 += 32 * kLeStep) {
                    int w[kLeStep];
                    uint32_t s[kLeStep];
#pragma unroll
                    for (int j = 0; j < kLeStep; ++j) {
                        const int t = t0 + 32 * j + lane;
                        int l = 0;  // the row of t: the first lane with inc > t
#pragma unroll
                        for (int d = 16; d >= 1; d >>= 1)
                            if (__shfl_sync(kFull, inc, l + d - 1) <= t) l += d;
                        const int f = __shfl_sync(kFull, first, l);
                        s[j] = __shfl_sync(kFull, src, l);
                        w[j] = t < total ? __ldg(&P.sadj[f + t]) : -1;
                    }
                    le_arcs(P, o, w, s, stage, cnt);
                }
            }
            __syncwarp();
            le_flush_block(P, o, stage, cnt);
            if (!le_sync(ctl, target, o3, lv)) return;
            beg += n_lev;
            n_lev = lv.n;
            full = lv.full;
            ins += n_lev;
            if (ins > load_limit) full |= kLeTableFull;
            if (n_lev == 0) {  // an empty next frontier ends the batch
                ++g;
                break;
            }
        }
        if (full) {  // the host grows a buffer and resumes at this batch
            status = full & kLeTableFull ? 1 : 2;
            break;
        }
        // ---- the batch's pairs lower delta; an empty table for the next batch
        for (long long i = gtid; i < (long long)ins; i += gstride) {
            const int u = (int)(P.log_key[base + i] >> 32), d = P.log_d[base + i];
            if (d < P.delta[u]) atomicMin(&P.delta[u], d);
        }
        if (b + 1 < P.nb)
            for (long long h = gtid; h <= (long long)(P.mask >> 1); h += gstride)
                reinterpret_cast<ulonglong2*>(P.keys)[h] = make_ulonglong2(kEmpty, kEmpty);
        base += ins;
        LeLevel lv0;
        if (!le_sync(ctl, target, (int)(g % 3), lv0)) return;
    }
    if (gtid == 0) {
        ctl->status = status;
        ctl->batch = b;
        ctl->log_n = base;
        ctl->ins = ins;
    }
    for (int d = 16; d >= 1; d >>= 1) edges += __shfl_xor_sync(kFull, edges, d);
    if (lane == 0 && edges) atomicAdd(&ctl->edges, edges);
}

// ------------------------------------------------------------ assembly --
__global__ void k_le_count(const unsigned long long* __restrict__ log_key, long long total, int32_t* cnt) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x)
        atomicAdd(&cnt[log_key[i] >> 32], 1);
}
__global__ void k_le_scatter(const unsigned long long* __restrict__ log_key, const int32_t* __restrict__ log_d,
                             long long total, int32_t* cursor, int32_t* gs, int32_t* gd) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const unsigned long long key = log_key[i];
        const int p = atomicAdd(&cursor[key >> 32], 1);
        gs[p] = (int32_t)(uint32_t)key;
        gd[p] = log_d[i];
    }
}
// In-place heapsort of k (source, distance) entries by the source's position.
__device__ void heap_sift(int32_t* gs, int32_t* gd, int i, int k, const int32_t* __restrict__ rank) {
    for (;;) {
        int c = 2 * i + 1;
        if (c >= k) return;
        if (c + 1 < k && rank[gs[c + 1]] > rank[gs[c]]) ++c;
        if (rank[gs[c]] <= rank[gs[i]]) return;
        const int ts = gs[i], td = gd[i];
        gs[i] = gs[c];
        gd[i] = gd[c];
        gs[c] = ts;
        gd[c] = td;
        i = c;
    }
}
__device__ void heap_sort(int32_t* gs, int32_t* gd, int k, const int32_t* __restrict__ rank) {
    for (int i = k / 2 - 1; i >= 0; --i) heap_sift(gs, gd, i, k, rank);
    for (int e = k - 1; e > 0; --e) {
        const int ts = gs[0], td = gd[0];
        gs[0] = gs[e];
        gd[0] = gd[e];
        gs[e] = ts;
        gd[e] = td;
        heap_sift(gs, gd, 0, e, rank);
    }
}

// One thread per vertex: its candidates sorted by source position, kept while
// their distance strictly decreases; keep[u] = the survivors (compacted to the
// front of the vertex's range).
__global__ void k_le_filter(int32_t n, const int32_t* __restrict__ pos, const int32_t* __restrict__ rank, int32_t* gs,
                            int32_t* gd, int32_t* keep) {
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += (long long)gridDim.x * blockDim.x) {
        const int a0 = pos[u], a1 = pos[u + 1];
        if (a1 - a0 <= 32) {
            for (int i = a0 + 1; i < a1; ++i) {  // insertion sort by the source's position
                const int s = gs[i], d = gd[i], r = rank[s];
                int j = i - 1;
                while (j >= a0 && rank[gs[j]] > r) {
                    gs[j + 1] = gs[j];
                    gd[j + 1] = gd[j];
                    --j;
                }
                gs[j + 1] = s;
                gd[j + 1] = d;
            }
        } else {
            heap_sort(gs + a0, gd + a0, a1 - a0, rank);
        }
        int k = a0, best = INT_MAX;
        for (int i = a0; i < a1; ++i)
            if (gd[i] < best) {
                best = gd[i];
                gs[k] = gs[i];
                gd[k] = gd[i];
                ++k;
            }
        keep[u] = k - a0;
    }
}
__global__ void k_le_compact(int32_t n, const int32_t* __restrict__ pos, const int32_t* __restrict__ kpos,
                             const int32_t* __restrict__ gs, const int32_t* __restrict__ gd, int64_t* le_off,
                             int32_t* le_src, int32_t* le_dist) {
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += (long long)gridDim.x * blockDim.x) {
        const int k0 = kpos[u], k1 = kpos[u + 1], a0 = pos[u];
        le_off[u] = k0;
        if (u == n - 1) le_off[n] = k1;
        for (int i = 0; i < k1 - k0; ++i) {
            le_src[k0 + i] = gs[a0 + i];
            le_dist[k0 + i] = gd[a0 + i];
        }
    }
}
__global__ void k_le_rank(int32_t n, const int32_t* __restrict__ order, int32_t* rank, int32_t* delta) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        rank[order[i]] = (int32_t)i;
        delta[i] = INT_MAX;
    }
}

inline int grid_for(int64_t work, int per_block, int cap) {
    int64_t g = (work + per_block - 1) / per_block;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, cap));
}

}  // namespace

int le_lists_compute(const int32_t* soff, const int32_t* sadj, int32_t n, const int32_t* order, int num_sms,
                     LeResult* res, cudaStream_t s, long long init_cap, long long init_log) {
    *res = LeResult();
    if (n == 0) return SCC_OK;
    Scratch tmp(s);
    // batches of 1, 2, 4, ... sources (Alg. 5)
    std::vector<long long> bounds{0};
    for (long long sz = 1, pos = 0; pos < n; sz *= 2) {
        pos = std::min<long long>(n, pos + sz);
        bounds.push_back(pos);
    }
    const int nb = (int)bounds.size() - 1;
    long long* bounds_d = nullptr;
    int32_t *rank = nullptr, *delta = nullptr;
    LeCtl* ctl = nullptr;
    SCC_TRY(tmp.alloc(&bounds_d, bounds.size()));
    SCC_TRY(tmp.alloc(&rank, (size_t)n));
    SCC_TRY(tmp.alloc(&delta, (size_t)n));
    SCC_TRY(tmp.alloc(&ctl, 1));
    SCC_CUDA(cudaMemcpyAsync(bounds_d, bounds.data(), sizeof(long long) * bounds.size(), cudaMemcpyHostToDevice, s));
    k_le_rank<<<grid_for(n, 1024, num_sms * 16), 256, 0, s>>>(n, order, rank, delta);
    SCC_LAUNCH();
    SCC_CUDA(cudaMemsetAsync(ctl, 0, sizeof(LeCtl), s));
    // buffers: the table (and the queue of long rows' pieces) and the candidate
    // log, grown on demand
    unsigned long long cap = 1024;
    while (cap < (init_cap > 0 ? (unsigned long long)init_cap : 4ull * (unsigned long long)n)) cap <<= 1;
    unsigned long long log_cap = init_log > 0 ? (unsigned long long)init_log : (unsigned long long)n * 24 + 1024;
    unsigned long long* keys = nullptr;
    unsigned long long *hk0 = nullptr, *hk1 = nullptr, *lk = nullptr;
    int32_t *ha0 = nullptr, *ha1 = nullptr, *ld = nullptr;
    int2 *row0 = nullptr, *row1 = nullptr;
    const auto hub_cap = [&] { return cap / 4 + 1024; };
    auto alloc_table = [&]() -> int {
        tmp.release(keys);
        tmp.release(row0);
        tmp.release(row1);
        tmp.release(hk0);
        tmp.release(hk1);
        tmp.release(ha0);
        tmp.release(ha1);
        SCC_TRY(tmp.alloc(&keys, (size_t)cap));
        SCC_TRY(tmp.alloc(&row0, (size_t)cap));
        SCC_TRY(tmp.alloc(&row1, (size_t)cap));
        SCC_TRY(tmp.alloc(&hk0, (size_t)hub_cap()));
        SCC_TRY(tmp.alloc(&hk1, (size_t)hub_cap()));
        SCC_TRY(tmp.alloc(&ha0, (size_t)hub_cap()));
        SCC_TRY(tmp.alloc(&ha1, (size_t)hub_cap()));
        SCC_CUDA(cudaMemsetAsync(keys, 0xff, (size_t)cap * 8, s));
        return SCC_OK;
    };
    SCC_TRY(alloc_table());
    SCC_TRY(tmp.alloc(&lk, (size_t)log_cap));
    SCC_TRY(tmp.alloc(&ld, (size_t)log_cap));
    int per_sm = 0;
    SCC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_le_lists, kLeBlock, 0));
    if (per_sm < 1) return SCC_ERR_INTERNAL;
    const int grid = num_sms;
    for (int attempt = 0;; ++attempt) {
        if (attempt > 64) return SCC_ERR_CAPACITY;
        LeParams P;
        P.soff = soff;
        P.sadj = sadj;
        P.n = n;
        P.order = order;
        P.bounds = bounds_d;
        P.nb = nb;
        P.delta = delta;
        P.keys = keys;
        P.mask = cap - 1;
        P.row[0] = row0;
        P.row[1] = row1;
        P.log_key = lk;
        P.log_d = ld;
        P.log_cap = log_cap;
        P.hub_key[0] = hk0;
        P.hub_key[1] = hk1;
        P.hub_arc[0] = ha0;
        P.hub_arc[1] = ha1;
        P.hub_cap = hub_cap();
        P.ctl = ctl;
        void* args[] = {(void*)&P};
        SCC_CUDA(cudaLaunchCooperativeKernel((const void*)k_le_lists, dim3(grid), dim3(kLeBlock), args, 0, s));
        count_launch();
        LeCtl h;
        SCC_CUDA(cudaMemcpyAsync(&h, ctl, sizeof(LeCtl), cudaMemcpyDeviceToHost, s));
        SCC_CUDA(cudaStreamSynchronize(s));
        if (h.err) return h.err;
        res->levels = h.levels;
        res->edges = h.edges;
        res->launches = attempt + 1;
        if (h.status == 0) {
            res->candidates = (long long)h.log_n;
            break;
        }
        // grow the full buffer; the batch starts over (its pairs were never logged)
        if (h.status == 1) {
            cap *= 2;
            SCC_TRY(alloc_table());
        } else {
            const unsigned long long need = std::max(2 * log_cap, h.log_n + 2 * h.ins + 1024);
            unsigned long long* nk = nullptr;
            int32_t* nd = nullptr;
            SCC_TRY(tmp.alloc(&nk, (size_t)need));
            SCC_TRY(tmp.alloc(&nd, (size_t)need));
            SCC_CUDA(cudaMemcpyAsync(nk, lk, 8 * h.log_n, cudaMemcpyDeviceToDevice, s));
            SCC_CUDA(cudaMemcpyAsync(nd, ld, 4 * h.log_n, cudaMemcpyDeviceToDevice, s));
            tmp.release(lk);
            tmp.release(ld);
            lk = nk;
            ld = nd;
            log_cap = need;
            SCC_CUDA(cudaMemsetAsync(keys, 0xff, (size_t)cap * 8, s));  // the batch's partial pairs
        }
        h.status = 0;
        h.err = 0;
        h.bar = GridBarrier{0, 0};
        for (int r = 0; r < 3; ++r) {
            h.fr_n[r] = h.hub_n[r] = 0;
            h.full[r] = 0;
        }
        SCC_CUDA(cudaMemcpyAsync(ctl, &h, sizeof(LeCtl), cudaMemcpyHostToDevice, s));
        SCC_CUDA(cudaStreamSynchronize(s));  // h is a stack variable
    }
    // ---- assembly: group the candidates by vertex, sort and filter each list
    const long long total = res->candidates;
    if (total > (long long)INT32_MAX - 1) return SCC_ERR_CAPACITY;
    int32_t *cnt = nullptr, *pos = nullptr, *cursor = nullptr, *gs = nullptr, *gd = nullptr, *keep = nullptr,
            *kpos = nullptr;
    void* stmp = nullptr;
    SCC_TRY(tmp.alloc(&cnt, (size_t)n + 1));
    SCC_TRY(tmp.alloc(&pos, (size_t)n + 1));
    SCC_TRY(tmp.alloc(&cursor, (size_t)n + 1));
    SCC_TRY(tmp.alloc(&keep, (size_t)n + 1));
    SCC_TRY(tmp.alloc(&kpos, (size_t)n + 1));
    SCC_TRY(tmp.alloc(&gs, (size_t)std::max<long long>(total, 1)));
    SCC_TRY(tmp.alloc(&gd, (size_t)std::max<long long>(total, 1)));
    SCC_TRY(tmp.alloc(reinterpret_cast<unsigned char**>(&stmp), scan_tmp_bytes(n)));
    SCC_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int32_t) * ((size_t)n + 1), s));
    const int g2 = grid_for(std::max<long long>(total, n), 1024, num_sms * 16);
    k_le_count<<<g2, 256, 0, s>>>(lk, total, cnt);
    SCC_LAUNCH();
    SCC_TRY(launch_scan(cnt, pos, n, stmp, s));
    SCC_CUDA(cudaMemcpyAsync(cursor, pos, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, s));
    k_le_scatter<<<g2, 256, 0, s>>>(lk, ld, total, cursor, gs, gd);
    SCC_LAUNCH();
    k_le_filter<<<grid_for(n, 256, num_sms * 16), 256, 0, s>>>(n, pos, rank, gs, gd, keep);
    SCC_LAUNCH();
    SCC_TRY(launch_scan(keep, kpos, n, stmp, s));
    int32_t kept = 0;
    SCC_CUDA(cudaMemcpyAsync(&kept, kpos + n, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    SCC_CUDA(cudaStreamSynchronize(s));
    // the result, kept by the caller
    SCC_TRY(dalloc_t(&res->off, (size_t)n + 1, s));
    SCC_TRY(dalloc_t(&res->src, (size_t)std::max(kept, 1), s));
    SCC_TRY(dalloc_t(&res->dist, (size_t)std::max(kept, 1), s));
    res->total = kept;
    k_le_compact<<<grid_for(n, 256, num_sms * 16), 256, 0, s>>>(n, pos, kpos, gs, gd, res->off, res->src, res->dist);
    SCC_LAUNCH();
    SCC_CUDA(cudaStreamSynchronize(s));
    return SCC_OK;
}

}  // namespace scc

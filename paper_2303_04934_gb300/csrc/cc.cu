// Connected components of the undirected graph under the arcs of G (Sec. 5.1;
// sm_103a) by union-find on a sample of the arcs first, as a forest of parent
// pointers with parent[x] <= x, so that a tree's root is its smallest vertex
// and the final roots are the labels:
//
//   1. parent[v] = the smallest of v and the sampled neighbours of v (its first
//      kCcOut out-arcs and kCcIn in-arcs), by plain stores; then every other
//      sampled arc joins its two trees (k_cc_seed, k_cc_link).
//   2. Every parent becomes its tree's root (k_cc_flat) and the most frequent
//      root of 1024 vertices spread over the graph is taken as the large tree
//      (k_cc_giant).
//   3. The arcs that were not sampled (k_cc_rest). A vertex of the large tree
//      skips its rows: an arc between it and a vertex of another tree is read
//      from the other end's row of G or of G^T, and an arc between two of its
//      vertices joins nothing. Without a tree that holds an eighth of the
//      vertices nobody is skipped and the rows of G cover every arc. Rows of
//      more than kCcRow arcs are cut into pieces of kCcPiece for k_cc_big.
//   4. labels_out[v] = the root of v (k_cc_labels).
//
// Joining a few sampled neighbours of each vertex, taking the most frequent root
// of 1024 probes for the large component and skipping its vertices afterwards is
// Afforest (Sutton, Ben-Nun, Barak, IPDPS 2018); the passes by atomicMin and their
// flattening are this file's.
//
// The paper's LDD-UF-JTB (Alg. 4) takes the same labels from a low-diameter
// decomposition of the symmetrised graph, a search of tens of rounds, and then
// tests every arc for joining two clusters. On R-MAT with 4.2 M vertices and
// 25 M arcs that was 0.97 ms for the search, 0.51 for the arcs and 0.14 for the
// labels, and 3.2 ms before the first of them for the symmetric CSR; now the
// sample is 0.18, the other arcs 0.04 and the labels 0.014 (1.81 -> 0.29 ms a
// call; 5.1 -> 0.32 ms the first). By bytes (offsets of both graphs, a sector an
// active vertex and sample, the copies and parents) it is bound at about
// 0.09 ms; what is left is gathers of parents from L2 and 16 launches. The
// decomposition has no graph left on which it is ahead: lattices 4.4 -> 0.62 ms
// (2-D, 8.4 M vertices), small graphs 0.56 -> 0.26.
#include <algorithm>
#include <climits>
#include <vector>

#include "common.cuh"
#include "engine.cuh"
#include "internal.h"

namespace scc {
namespace {

constexpr int kBlk = 256;
constexpr int kUfLimit = 1 << 20;  // attempts of one union before it reports an error
constexpr int kCcOut = 2;          // sampled out-arcs of a vertex
constexpr int kCcIn = 1;           // sampled in-arcs of a vertex
constexpr int kCcSample = kCcOut + kCcIn;
constexpr int kCcRow = 32;         // longer rows go to k_cc_big ...
constexpr int kCcPiece = 1024;     // ... in pieces of this many arcs, a warp each
constexpr int kCcProbe = 1024;     // vertices whose roots name the large tree

inline int grid_for(int64_t work, int per_block, int cap) {
    int64_t g = (work + per_block - 1) / per_block;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, cap));
}

// Row v of the symmetric CSR: G's row, then G^T's (one warp per vertex). Rows of
// more than kSymRow arcs are listed in pieces of so many (v, or ~v for the row of
// G^T; first arc) and copied by k_sym_big: a hub's row by one warp held the pass
// up (R-MAT of 262 k vertices, 8 M entries, first LE-lists 1.84 -> 1.63 ms).
constexpr int kSymRow = 1024;
__device__ __forceinline__ void sym_copy(const int32_t* __restrict__ src, int32_t* __restrict__ dst, int cnt) {
    for (int e = lane_id(); e < cnt; e += 128) {
        int32_t x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = e + 32 * j < cnt ? src[e + 32 * j] : 0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (e + 32 * j < cnt) dst[e + 32 * j] = x[j];
    }
}
__global__ void __launch_bounds__(kBlk) k_sym_rows(const int32_t* __restrict__ off, const int32_t* __restrict__ adj,
                                                   const int32_t* __restrict__ toff, const int32_t* __restrict__ tadj,
                                                   int32_t n, int32_t* __restrict__ soff, int32_t* __restrict__ sadj,
                                                   int2* __restrict__ piece, unsigned int* npiece, unsigned int cap) {
    const int lane = lane_id();
    const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long v = w0; v < n; v += nw) {
        const int a0 = off[v], a1 = off[v + 1], b0 = toff[v], b1 = toff[v + 1];
        const long long s0 = (long long)a0 + b0;
        if (lane == 0) soff[v] = (int32_t)s0;
        for (int d = 0; d < 2; ++d) {
            const int lo = d == 0 ? a0 : b0, hi = d == 0 ? a1 : b1;
            if (hi - lo <= kSymRow) {
                sym_copy((d == 0 ? adj : tadj) + lo, sadj + (d == 0 ? s0 : s0 + (a1 - a0)), hi - lo);
                continue;
            }
            const int k = (int)(((long long)hi - lo + kSymRow - 1) / kSymRow);
            unsigned int at = 0;
            if (lane == 0) at = atomicAdd(npiece, (unsigned int)k);
            at = __shfl_sync(kFull, at, 0);
            for (int j = lane; j < k; j += 32)
                if (at + j < cap) piece[at + j] = make_int2(d == 0 ? (int)v : ~(int)v, lo + j * kSymRow);
        }
    }
    if (w0 == 0 && lane == 0) soff[n] = off[n] + toff[n];
}
__global__ void __launch_bounds__(kBlk) k_sym_big(const int32_t* __restrict__ off, const int32_t* __restrict__ adj,
                                                  const int32_t* __restrict__ toff, const int32_t* __restrict__ tadj,
                                                  int32_t* __restrict__ sadj, const int2* __restrict__ piece,
                                                  const unsigned int* npiece, unsigned int cap) {
    const unsigned int np = min(*npiece, cap);
    const unsigned int nw = (gridDim.x * blockDim.x) >> 5;
    for (unsigned int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < np; k += nw) {
        const int2 q = piece[k];
        const bool t = q.x < 0;
        const int v = t ? ~q.x : q.x;
        const int end = t ? toff[v + 1] : off[v + 1];
        // entry e of a row of G is e + toff[v] in the symmetric CSR, of G^T e + off[v + 1]
        sym_copy((t ? tadj : adj) + q.y, sadj + ((long long)q.y + (t ? off[v + 1] : toff[v])), min(end - q.y, kSymRow));
    }
}

// ------------------------------------------------------------- union-find --
// parent[x] <= x always (a root is hooked under a smaller one), so the
// concurrent halving writes keep every parent a vertex of the same tree, and a
// walk towards the root ends: each step goes to a smaller vertex.
__device__ __forceinline__ int32_t uf_find(int32_t* parent, int32_t x) {
    for (;;) {
        const int32_t p = ld_volatile(&parent[x]);
        if (p >= x) return x;
        const int32_t gp = ld_volatile(&parent[p]);
        if (gp >= p) return p;
        parent[x] = gp;  // halving
        x = gp;
    }
}
// A root without writes, for the passes in which no trees join and each
// vertex's owner stores its root (a halving store could put an older ancestor
// over it). Plain loads: the few words that most walks end in come from L1.
__device__ __forceinline__ int32_t uf_root(const int32_t* parent, int32_t x) {
    for (;;) {
        const int32_t p = parent[x];
        if (p >= x) return x;
        x = p;
    }
}
__device__ __forceinline__ void uf_union(int32_t* parent, int32_t a, int32_t b, int* err) {
    for (int it = 0; it < kUfLimit; ++it) {
        const int32_t ra = uf_find(parent, a), rb = uf_find(parent, b);
        if (ra == rb) return;
        const int32_t lo = ra < rb ? ra : rb, hi = ra < rb ? rb : ra;
        const int32_t old = atomicCAS(&parent[hi], hi, lo);
        if (old == hi) return;
        a = lo;
        b = old;
    }
    atomicExch(err, SCC_ERR_INTERNAL);
}

// A vertex of x's set by plain loads and no writes (a filter in front of
// uf_union): a parent pointer only ever holds a vertex of the same set, and
// sets only merge, so even a stale chain of pointers stays inside x's set. If
// the chains from two vertices meet, the two are connected already.
__device__ __forceinline__ int32_t uf_peek(const int32_t* parent, int32_t x) {
    for (int it = 0; it < 64; ++it) {
        const int32_t p = parent[x];
        if (p == x) break;
        x = p;
    }
    return x;
}

// The block's sum of c into *out, by one atomic (one a warp on a single word was
// 50 us on 4.2 M vertices).
__device__ __forceinline__ void cc_add(unsigned long long* out, unsigned long long c) {
    __shared__ unsigned long long sum;
    if (threadIdx.x == 0) sum = 0;
    __syncthreads();
    for (int d = 16; d >= 1; d >>= 1) c += __shfl_xor_sync(kFull, c, d);
    if (lane_id() == 0 && c) atomicAdd(&sum, c);
    __syncthreads();
    if (threadIdx.x == 0 && sum) atomicAdd(out, sum);
}

// sample[j n + v] = the sampled neighbours of v: its first kCcOut out-arcs and
// kCcIn in-arcs, v itself where the row is shorter; parent[v] = the smallest of
// v and these. Bound by the latency of off -> adj: one vertex a thread keeps as
// many chains in flight as the chip holds threads. The passes below read the
// copy, 12 coalesced bytes a vertex instead of four offsets and three sectors.
__global__ void __launch_bounds__(kBlk) k_cc_seed(const int32_t* __restrict__ off, const int32_t* __restrict__ adj,
                                                  const int32_t* __restrict__ toff, const int32_t* __restrict__ tadj,
                                                  int32_t n, int32_t* __restrict__ sample, int32_t* __restrict__ parent) {
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
        const int a0 = off[v], a1 = off[v + 1], b0 = toff[v], b1 = toff[v + 1];
        int32_t w[kCcSample], lo = (int32_t)v;
#pragma unroll
        for (int j = 0; j < kCcOut; ++j) w[j] = a1 - a0 > j ? adj[a0 + j] : (int32_t)v;
#pragma unroll
        for (int j = 0; j < kCcIn; ++j) w[kCcOut + j] = b1 - b0 > j ? tadj[b0 + j] : (int32_t)v;
#pragma unroll
        for (int j = 0; j < kCcSample; ++j) {
            sample[(long long)j * n + v] = w[j];
            lo = min(lo, w[j]);
        }
        parent[v] = lo;
    }
}

// Every sampled arc between two trees hooks the larger root under the smaller:
// each parent was its tree's root before the launch, so all values read and
// written here are such roots, and of several hooks of one root the smallest
// stays (the arcs of the others are met again by a later pass). An atomic
// without a result instead of a find-and-CAS loop: joining the trees to the end
// here, with walks that go on while every tree changes, was 213 us on R-MAT with
// 262 k vertices and 263-368 us with 4.2 M, where two passes of hooks and their
// flattening take 27 and 84.
__global__ void __launch_bounds__(kBlk) k_cc_hook(const int32_t* __restrict__ sample, int32_t n, int32_t* parent,
                                                  const int32_t* giant, const int32_t* unless) {
    if (unless && *unless >= 0) return;
    const int32_t gt = giant ? *giant : -1;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
        const int32_t a = parent[v];
        if (a == gt) continue;
        int32_t b[kCcSample];
#pragma unroll
        for (int j = 0; j < kCcSample; ++j) b[j] = sample[(long long)j * n + v];
#pragma unroll
        for (int j = 0; j < kCcSample; ++j) b[j] = b[j] == (int32_t)v ? a : parent[b[j]];
#pragma unroll
        for (int j = 0; j < kCcSample; ++j)
            if (b[j] != a) {
                const int32_t lo = min(a, b[j]), hi = max(a, b[j]);
                if (lo < parent[hi]) atomicMin(&parent[hi], lo);
            }
    }
}

// parent[v] = the root of v, four vertices a thread whose walks go side by side.
// A walk of more than six steps reads past L1 and stores where it is, its own
// word only, so the walks that run at once shorten one another's: a path graph
// numbered in order, whose seeded forest is one chain, takes 0.5 ms at 4.2 M
// vertices, and seconds without. For the same reason each thread starts all its
// walks at once and the grid has a thread for every four vertices: a walk goes to
// smaller vertices and blocks start in order, so none passes a vertex whose own
// walk is yet to start.
__global__ void __launch_bounds__(kBlk) k_cc_flat(int32_t n, int32_t* parent, const int32_t* unless) {
    if (unless && *unless >= 0) return;
    const long long v = 4 * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
    if (v >= n) return;
    const int k = n - v < 4 ? (int)(n - v) : 4;
    int32_t p0[4], r[4];
    if (k == 4) {
        const int4 q = *reinterpret_cast<const int4*>(parent + v);
        p0[0] = q.x;
        p0[1] = q.y;
        p0[2] = q.z;
        p0[3] = q.w;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) p0[j] = j < k ? parent[v + j] : 0;  // parent[0] = 0
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) r[j] = p0[j];
    uint32_t on = 15;  // the walks under way
    for (int it = 0; on; ++it) {
        int32_t p[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            p[j] = !(on >> j & 1) ? r[j] : it < 6 ? parent[r[j]] : ld_volatile(&parent[r[j]]);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (p[j] < r[j]) {
                r[j] = p[j];
                if (it >= 6 && j < k) *(volatile int32_t*)&parent[v + j] = p[j];
            } else {
                on &= ~(1u << j);
            }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (j < k && r[j] != p0[j]) parent[v + j] = r[j];
}

// giant = the most frequent root of kCcProbe vertices at equal distances if at
// least an eighth of them have it, or -1 (or *unless if that names one). One
// block of kCcProbe threads.
__global__ void __launch_bounds__(kCcProbe) k_cc_giant(const int32_t* __restrict__ parent, int32_t n, int32_t* giant,
                                                       const int32_t* unless) {
    if (unless && *unless >= 0) {
        if (threadIdx.x == 0) *giant = *unless;
        return;
    }
    __shared__ int32_t key[2 * kCcProbe];
    __shared__ int cnt[2 * kCcProbe];
    __shared__ unsigned long long best;
    const int t = threadIdx.x;
    for (int j = t; j < 2 * kCcProbe; j += kCcProbe) {
        key[j] = -1;
        cnt[j] = 0;
    }
    if (t == 0) best = 0;
    __syncthreads();
    const int32_t r = parent[(long long)t * n / kCcProbe];
    uint32_t slot = ((uint32_t)r * 2654435769u) >> 21;  // 11 bits: 2 kCcProbe slots
    for (int it = 0; it < 2 * kCcProbe; ++it) {         // kCcProbe keys at most: a free slot is met
        const int32_t k = atomicCAS(&key[slot], -1, r);
        if (k == -1 || k == r) break;
        slot = (slot + 1) & (2 * kCcProbe - 1);
    }
    const int c = atomicAdd(&cnt[slot], 1) + 1;
    atomicMax(&best, (unsigned long long)(uint32_t)c << 32 | (uint32_t)r);
    __syncthreads();
    if (t == 0) *giant = (int)(best >> 32) >= kCcProbe / 8 ? (int32_t)(uint32_t)best : -1;
}

// One row (arcs [a, b) of adj) of u: four targets at a time, then their peeks,
// as independent loads.
__device__ __forceinline__ unsigned long long cc_row(const int32_t* __restrict__ adj, int a, int b, int step, int32_t u,
                                                     int32_t* parent, int* err) {
    unsigned long long c = 0;
    for (long long e0 = a; e0 < b; e0 += 4 * step) {
        int32_t w[4], p[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = e0 + j * step < b ? adj[e0 + j * step] : u;
#pragma unroll
        for (int j = 0; j < 4; ++j) p[j] = uf_peek(parent, w[j]);
        const int32_t pu = uf_peek(parent, u);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (p[j] != pu) {
                ++c;
                uf_union(parent, pu, p[j], err);
            }
    }
    return c;
}

// The rows of the vertices outside the large tree, a thread a vertex; the warp
// lists the pieces of its long rows together (piece = (u, or ~u for the row of
// G^T; first arc)).
__global__ void __launch_bounds__(kBlk) k_cc_rest(const int32_t* __restrict__ off, const int32_t* __restrict__ adj,
                                                  const int32_t* __restrict__ toff, const int32_t* __restrict__ tadj,
                                                  int32_t n, int32_t* parent, const int32_t* giant,
                                                  unsigned long long* joined, unsigned long long* trees, int2* piece,
                                                  unsigned long long* npiece, long long cap, int* err) {
    const int lane = lane_id();
    const int32_t gt = *giant;
    unsigned long long c = 0, nt = 0;
    for (long long v0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) - lane; v0 < n;
         v0 += (long long)gridDim.x * blockDim.x) {
        const long long v = v0 + lane;
        const int32_t pv = v < n ? parent[v] : -1;
        const bool live = v < n && (gt < 0 || pv != gt);
        nt += pv == (int32_t)v;
        if (!__any_sync(kFull, live)) continue;
        // both rows' ends at once: most of these vertices have no arcs
        int lo[2] = {0, 0}, hi[2] = {0, 0};
        if (live) {
            lo[0] = off[v];
            hi[0] = off[v + 1];
            if (gt >= 0) {
                lo[1] = toff[v];
                hi[1] = toff[v + 1];
            }
        }
        if (!__any_sync(kFull, lo[0] < hi[0] || lo[1] < hi[1])) continue;
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            const int32_t* aj = d == 0 ? adj : tadj;
            const int a = lo[d], b = hi[d];
            const bool big = b - a > kCcRow;
            if (!big && a < b) c += cc_row(aj, a, b, 1, (int32_t)v, parent, err);
            for (uint32_t m = __ballot_sync(kFull, big); m; m &= m - 1) {
                const int l = __ffs(m) - 1;
                const int la = __shfl_sync(kFull, a, l), lb = __shfl_sync(kFull, b, l);
                const int k = (int)(((long long)lb - la + kCcPiece - 1) / kCcPiece);
                unsigned long long at = 0;
                if (lane == 0) at = atomicAdd(npiece, (unsigned long long)k);
                at = __shfl_sync(kFull, at, 0);
                const int32_t u = (int32_t)(v0 + l);
                for (int j = lane; j < k; j += 32) {
                    if ((long long)at + j < cap) piece[at + j] = make_int2(d == 0 ? u : ~u, la + j * kCcPiece);
                    else atomicExch(err, SCC_ERR_INTERNAL);  // cannot happen: a piece is more than 32 arcs of its row
                }
            }
            __syncwarp();
        }
    }
    cc_add(joined, c);
    __syncthreads();
    cc_add(trees, nt);
}
__global__ void __launch_bounds__(kBlk) k_cc_big(const int32_t* __restrict__ off, const int32_t* __restrict__ adj,
                                                 const int32_t* __restrict__ toff, const int32_t* __restrict__ tadj,
                                                 int32_t* parent, unsigned long long* joined,
                                                 const int2* __restrict__ piece, const unsigned long long* npiece,
                                                 long long cap, int* err) {
    const int lane = lane_id();
    const long long np = min((long long)*npiece, cap);
    unsigned long long c = 0;
    for (long long k = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < np;
         k += ((long long)gridDim.x * blockDim.x) >> 5) {
        const int2 q = piece[k];
        const int32_t u = q.x < 0 ? ~q.x : q.x;
        const int end = q.x < 0 ? toff[u + 1] : off[u + 1];
        const int b = end - q.y > kCcPiece ? q.y + kCcPiece : end;
        c += cc_row(q.x < 0 ? tadj : adj, q.y + lane, b, 32, u, parent, err);
    }
    cc_add(joined, c);
}

__global__ void __launch_bounds__(kBlk) k_cc_labels(int32_t n, const int32_t* parent, int32_t* out,
                                                    unsigned long long* comps) {
    unsigned long long c = 0;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
        const int32_t r = uf_root(parent, (int32_t)v);
        out[v] = r;
        c += r == (int32_t)v;
    }
    cc_add(comps, c);
}
__global__ void k_iota(int32_t n, int32_t* a) {
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x)
        a[v] = (int32_t)v;
}
}  // namespace

int64_t sym_piece_cap(int64_t mt) { return 4 * (mt / (kSymRow + 1)) + 2; }

int launch_sym_csr(const int32_t* off, const int32_t* adj, const int32_t* toff, const int32_t* tadj, int32_t n,
                   int32_t* soff, int32_t* sadj, void* piece, int64_t cap, int num_sms, cudaStream_t s) {
    unsigned int* npiece = reinterpret_cast<unsigned int*>(piece);  // the first entry holds their number
    int2* const list = reinterpret_cast<int2*>(piece) + 1;
    SCC_CUDA(cudaMemsetAsync(npiece, 0, sizeof(int2), s));
    k_sym_rows<<<num_sms * 8, kBlk, 0, s>>>(off, adj, toff, tadj, n, soff, sadj, list, npiece, (unsigned int)cap);
    SCC_LAUNCH();
    k_sym_big<<<num_sms * 8, kBlk, 0, s>>>(off, adj, toff, tadj, sadj, list, npiece, (unsigned int)cap);
    SCC_LAUNCH();
    return SCC_OK;
}

int launch_iota(int32_t n, int32_t* a, int num_sms, cudaStream_t s) {
    k_iota<<<grid_for(n, kBlk * 4, num_sms * 16), kBlk, 0, s>>>(n, a);
    SCC_LAUNCH();
    return SCC_OK;
}

size_t cc_sample_size(int64_t n) { return (size_t)n * kCcSample; }
int64_t cc_piece_cap(int64_t mt) { return 2 * (mt / (kCcRow + 1)) + 2; }

int launch_cc(const int32_t* off, const int32_t* adj, const int32_t* toff, const int32_t* tadj, int32_t n,
              int32_t* sample, int32_t* parent, int32_t* out, unsigned long long* counters, int32_t* giant, void* piece,
              long long piece_cap, int* err, int num_sms, cudaStream_t s, cudaEvent_t* ev) {
    const int g = grid_for(n, kBlk, num_sms * 32);
    const int gf = grid_for(n, 4 * kBlk, INT_MAX);
    if (ev) cudaEventRecord(ev[0], s);
    k_cc_seed<<<g, kBlk, 0, s>>>(off, adj, toff, tadj, n, sample, parent);
    SCC_LAUNCH();
    k_cc_flat<<<gf, kBlk, 0, s>>>(n, parent, nullptr);
    SCC_LAUNCH();
    k_cc_hook<<<g, kBlk, 0, s>>>(sample, n, parent, nullptr, nullptr);
    SCC_LAUNCH();
    k_cc_flat<<<gf, kBlk, 0, s>>>(n, parent, nullptr);
    SCC_LAUNCH();
    k_cc_giant<<<1, kCcProbe, 0, s>>>(parent, n, giant, nullptr);
    SCC_LAUNCH();
    k_cc_hook<<<g, kBlk, 0, s>>>(sample, n, parent, giant, nullptr);
    SCC_LAUNCH();
    k_cc_flat<<<gf, kBlk, 0, s>>>(n, parent, nullptr);
    SCC_LAUNCH();
    k_cc_giant<<<1, kCcProbe, 0, s>>>(parent, n, giant + 1, nullptr);
    SCC_LAUNCH();
    for (int r = 0; r < 2; ++r) {
        k_cc_hook<<<g, kBlk, 0, s>>>(sample, n, parent, nullptr, giant + 1);
        SCC_LAUNCH();
        k_cc_flat<<<gf, kBlk, 0, s>>>(n, parent, giant + 1);
        SCC_LAUNCH();
    }
    k_cc_giant<<<1, kCcProbe, 0, s>>>(parent, n, giant + 2, giant + 1);
    SCC_LAUNCH();
    if (ev) cudaEventRecord(ev[1], s);
    k_cc_rest<<<g, kBlk, 0, s>>>(off, adj, toff, tadj, n, parent, giant + 2, &counters[0], &counters[1], (int2*)piece, &counters[3],
                                 piece_cap, err);
    SCC_LAUNCH();
    k_cc_big<<<num_sms * 8, kBlk, 0, s>>>(off, adj, toff, tadj, parent, &counters[0], (const int2*)piece, &counters[3],
                                          piece_cap, err);
    SCC_LAUNCH();
    if (ev) cudaEventRecord(ev[2], s);
    k_cc_labels<<<g, kBlk, 0, s>>>(n, parent, out, &counters[2]);
    SCC_LAUNCH();
    if (ev) cudaEventRecord(ev[3], s);
    return SCC_OK;
}

}  // namespace scc

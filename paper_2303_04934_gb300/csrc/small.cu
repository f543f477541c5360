// Small graphs: intake and transposition by one block (sm_103a).
#include "common.cuh"
#include "internal.h"

namespace scc {
namespace {

constexpr int kSmallVerts = 8192, kSmallArcs = 1 << 16;  // a graph that one block takes in

// Intake and transposition of a small graph by one block: the offsets copied and
// checked, the targets copied, checked and counted in shared memory, the counts
// scanned into the rows of G^T, each arc's source placed. out: [0] an offset or
// a target out of range (nothing else is written then), [1] the longest row, [2]
// self-loops (G^T is not built if there are any). What bounds a small graph is
// not this work but the ten launches, three synchronisations and thirteen
// temporaries of the general path: creating a graph of 1089 vertices 177 -> 57 us,
// of 8192 vertices and 59 k arcs 190 -> 118 (the block itself takes 60 of these;
// much larger ones are better off with the whole chip, so the limits lie there).
// Long rows are placed by the whole block, so no thread walks one alone.
constexpr int kSmallBlk = 1024;
constexpr int kSmallRow = 32;
__global__ void __launch_bounds__(kSmallBlk) k_small_graph(const int32_t* off_src, const int32_t* adj_src, int32_t n,
                                                           int32_t m, int32_t* off, int32_t* adj, int32_t* toff,
                                                           int32_t* tadj, int* out) {
    __shared__ int s_cnt[kSmallVerts + 1];
    __shared__ int s_long[kSmallArcs / (kSmallRow + 1) + 1];  // rows of more than kSmallRow arcs
    __shared__ int s_nlong, s_bad, s_most, s_self;
    __shared__ int s_wsum[32];
    const int t = threadIdx.x;
    if (t == 0) s_nlong = s_bad = s_most = s_self = 0;
    for (int i = t; i <= n; i += kSmallBlk) s_cnt[i] = 0;
    __syncthreads();
    int most = 0;
    bool bad = false;
    for (int i = t; i <= n; i += kSmallBlk) {
        const int a = off_src[i];
        off[i] = a;
        if (i == 0 && a != 0) bad = true;
        if (i == n) {
            if (a != m) bad = true;
        } else {
            const int b = off_src[i + 1];
            if (a > b || a < 0 || b > m) bad = true;  // with off[0] = 0 and off[n] = m: not increasing somewhere
            else most = max(most, b - a);
        }
    }
    for (int e = t; e < m; e += kSmallBlk) {
        const int w = adj_src[e];
        adj[e] = w;
        if ((unsigned)w < (unsigned)n) atomicAdd(&s_cnt[w], 1);
        else bad = true;
    }
    most = __reduce_max_sync(kFull, most);
    if (lane_id() == 0) atomicMax(&s_most, most);
    if (bad) s_bad = 1;
    __syncthreads();
    if (s_bad) {
        if (t == 0) out[0] = 1;
        return;
    }
    // exclusive scan of the counts, kPer consecutive ones a thread
    constexpr int kPer = kSmallVerts / kSmallBlk;
    int sum = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) sum += t * kPer + j < n ? s_cnt[t * kPer + j] : 0;
    int incl = warp_incl_scan(sum);
    if (lane_id() == 31) s_wsum[t >> 5] = incl;
    __syncthreads();
    if (t < 32) {
        const int x = s_wsum[t];
        s_wsum[t] = warp_incl_scan(x) - x;
    }
    __syncthreads();
    int run = s_wsum[t >> 5] + incl - sum;
#pragma unroll
    for (int j = 0; j < kPer; ++j)
        if (t * kPer + j < n) {
            const int c = s_cnt[t * kPer + j];
            s_cnt[t * kPer + j] = run;
            toff[t * kPer + j] = run;
            run += c;
        }
    if (t == 0) toff[n] = m;
    __syncthreads();
    int self = 0;
    auto place = [&](int u, int w) {
        self += u == w;
        tadj[atomicAdd(&s_cnt[w], 1)] = u;
    };
    for (int u = t; u < n; u += kSmallBlk) {
        const int a = off[u], b = off[u + 1];
        if (b - a > kSmallRow) {
            s_long[atomicAdd(&s_nlong, 1)] = u;
            continue;
        }
        for (int e0 = a; e0 < b; e0 += 4) {
            int w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = e0 + j < b ? adj[e0 + j] : -1;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (w[j] >= 0) place(u, w[j]);
        }
    }
    __syncthreads();
    for (int i = t >> 5; i < s_nlong; i += kSmallBlk / 32) {  // a warp a long row
        const int u = s_long[i], b = off[u + 1];
        for (int e = off[u] + lane_id(); e < b; e += 32) place(u, adj[e]);
    }
    if (self) atomicAdd(&s_self, self);
    __syncthreads();
    if (t == 0) {
        out[0] = 0;
        out[1] = s_most;
        out[2] = s_self;
    }
}

}  // namespace

bool small_graph(int32_t n, int64_t m) { return n >= 1 && n <= kSmallVerts && m <= kSmallArcs; }

int launch_small_graph(const int32_t* off_src, const int32_t* adj_src, int32_t n, int64_t m, int32_t* off, int32_t* adj,
                       int32_t* toff, int32_t* tadj, int* out, cudaStream_t s) {
    k_small_graph<<<1, kSmallBlk, 0, s>>>(off_src, adj_src, n, (int32_t)m, off, adj, toff, tadj, out);
    SCC_LAUNCH();
    return SCC_OK;
}

}  // namespace scc

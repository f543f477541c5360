// reach_multi: the set of sources reaching each vertex, as one or two mask
// words per vertex, spread along the arcs by the barrier-free search of
// prop.cuh (one launch: masks cleared, sources checked and set, the search).
//
// On a graph with hubs nearly every source reaches, or is reached from, one
// giant SCC, and a search that carries 64 masks through it raises every vertex
// of it many times over. There the hub's own forward and backward sets come
// first, by the engine's bitmap searches with dense rounds (one bit per vertex,
// each row read once and mostly not to its end): a source that reaches the hub
// reaches all that the hub reaches, so those vertices start with the set H of
// the sources that do, and the search only adds what lies outside. The set of
// vertices the hub reaches is closed under arcs and carries H throughout, so a
// source of H stops at its border.
//
// Measured (both directions, GB300): R-MAT of 4 M vertices, 64 sources 14.6 ->
// 2.30 ms, 3D torus of 1 M vertices, 7 sources 3.15 -> 1.31, against one search of
// 64-bit masks by the engine's rounds. The R-MAT time is the hub's four bitmap
// searches; the masks' own search ends after a few hops.
#include <algorithm>
#include <climits>
#include <cstring>

#include "common.cuh"
#include "engine.cuh"
#include "internal.h"
#include "prop.cuh"

namespace scc {
namespace {

constexpr int kReachBlock = 256;
constexpr int kReachWarps = kReachBlock / kWarp;

// The grid with the common barrier: there are four in a call, and with PropGrid's
// the pulling loop came out 5% slower (2D torus 504^2, 64 sources 3.1 -> 3.3 ms).
struct ReachScope : GridScope {
    template <class F>
    __device__ __forceinline__ static bool sync_then(GridBarrier* b, int* err, unsigned long long& val, F&& f) {
        __shared__ unsigned long long s_val;
        if (!grid_sync(b, err)) return false;
        if (threadIdx.x == 0) s_val = f();
        __syncthreads();
        val = s_val;
        return true;
    }
};

template <class Op>
struct ReachParams {
    PropGraph<Op> G;  // off[0], adj[0]: the direction of the search
    PropCtl* ctl;     // zero; status 2: a source is out of range
    const int32_t* src;
    int k;
    const uint32_t* from_hub;  // vertices the hub reaches in the direction of the search (null: no hub)
    const uint32_t* to_hub;    // vertices that reach it
    uint64_t idle_ns;
};

__device__ __forceinline__ unsigned long long bit_of(const unsigned long long&, int j) { return 1ull << j; }
__device__ __forceinline__ PropOr2::Val bit_of(const PropOr2::Val&, int j) {
    return {j < 64 ? 1ull << j : 0ull, j < 64 ? 0ull : 1ull << (j - 64)};
}

// kHubs: for a graph with rows of more than kPropHub arcs
template <class Op, bool kPull, bool kHubs>
__global__ void __launch_bounds__(kReachBlock, 4) k_reach(const __grid_constant__ ReachParams<Op> P) {
    using S = ReachScope;
    using Val = typename Op::Val;
    __shared__ uint32_t s_q[kReachWarps][kPropQueue];
    __shared__ uint32_t s_mk[kReachWarps][kPropMarks];
    __shared__ PropShared sh;
    __shared__ Val s_hub;  // sources that reach the hub
    __shared__ int s_bad;
    const PropGraph<Op>& G = P.G;
    PropCtl* ctl = P.ctl;
    const int lane = lane_id();
    uint32_t* q = s_q[threadIdx.x >> 5];
    uint32_t* mk = s_mk[threadIdx.x >> 5];
    const PropSlice sl = prop_slice<S>(G.n);
    if (threadIdx.x == 0) {
        sh.idle_ns = P.idle_ns;
        s_hub = Op::none();
        s_bad = 0;
    }
    __syncthreads();
    // every block looks at the sources: all see the same ones out of range
    for (int j = threadIdx.x; j < P.k; j += blockDim.x) {
        const int v = P.src[j];
        if (v < 0 || v >= G.n) s_bad = 1;
        else if (P.to_hub && ((P.to_hub[v >> 5] >> (v & 31)) & 1u)) Op::raise(&s_hub, 0, bit_of(Val{}, j));
    }
    __syncthreads();
    if (s_bad) {
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl->status = 2;
        return;
    }
    const Val hub = s_hub;
    for (long long i = 0; i < sl.cnt; ++i) {
        const long long w = sl.word(i), v = w * 32 + lane;
        if (w >= sl.nw) break;
        const uint32_t x = P.from_hub ? P.from_hub[w] : 0u;
        if (v < G.n) Op::store(G.s[0], v, (x >> lane) & 1u ? hub : Op::none());
        if (!kPull && lane == 0) G.d[0][w] = 0;
    }
    if (!S::sync(&ctl->bar, &ctl->err)) return;
    if (blockIdx.x == 0)
        for (int j = threadIdx.x; j < P.k; j += blockDim.x) {
            const int v = P.src[j];
            Op::raise(G.s[0], v, bit_of(Val{}, j));
            if (!kPull) atomicOr(&G.d[0][v >> 5], 1u << (v & 31));
        }
    if (!S::sync(&ctl->bar, &ctl->err)) return;
    unsigned int check = 0;
    unsigned long long items = 0, arcs = 0;
    if constexpr (kPull) prop_search_pull<S>(G, Op{}, ctl, sh, check, items);
    else prop_search<S, kHubs>(G, Op{}, ctl, sh, q, mk, check, 0, items, arcs);
}

// The vertex of the largest smaller degree, degree << 32 | vertex.
__global__ void k_hub(const int32_t* __restrict__ off, const int32_t* __restrict__ toff, int32_t n,
                      unsigned long long* best) {
    unsigned long long b = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const int d = min(off[v + 1] - off[v], toff[v + 1] - toff[v]);
        b = max(b, ((unsigned long long)(uint32_t)d << 32) | (uint32_t)v);
    }
    for (int d = 16; d >= 1; d >>= 1) b = max(b, __shfl_xor_sync(kFull, b, d));
    if (lane_id() == 0 && b > ld_volatile(best)) atomicMax(best, b);
}

__global__ void k_longest_row(const int32_t* __restrict__ off, int32_t n, unsigned long long* best) {
    unsigned long long b = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        b = max(b, (unsigned long long)(off[v + 1] - off[v]));
    for (int d = 16; d >= 1; d >>= 1) b = max(b, __shfl_xor_sync(kFull, b, d));
    if (lane_id() == 0 && b > ld_volatile(best)) atomicMax(best, b);
}

template <class Op>
int launch_reach(const ReachArgs& a, cudaStream_t st) {
    ReachParams<Op> P;
    memset(&P, 0, sizeof(P));
    P.G.off[0] = a.off;
    P.G.off[1] = a.toff;
    P.G.end[0] = a.off + 1;
    P.G.end[1] = a.toff + 1;
    P.G.adj[0] = a.adj;
    P.G.adj[1] = a.tadj;
    P.G.n = a.n;
    P.G.s[0] = reinterpret_cast<typename Op::Val*>(a.mask);
    P.G.d[0] = a.dirty;
    P.ctl = reinterpret_cast<PropCtl*>(a.dev);
    P.src = a.src;
    P.k = a.k;
    P.from_hub = a.from_hub;
    P.to_hub = a.to_hub;
    P.idle_ns = a.idle_ns ? a.idle_ns : kPropIdleTimeoutNs;
    static int per_sm = -1;
    if (per_sm < 0) {
        int x = INT_MAX;
        for (const void* k : {(const void*)k_reach<Op, true, false>, (const void*)k_reach<Op, false, false>,
                              (const void*)k_reach<Op, false, true>}) {
            int y = 0;
            SCC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&y, k, kReachBlock, 0));
            x = std::min(x, y);
        }
        if (x < 1) return SCC_ERR_CUDA;
        per_sm = x;
    }
    const long long nw = ((long long)a.n + 31) / 32;
    const int grid =
        (int)std::max<long long>(1, std::min<long long>(per_sm * a.num_sms, (nw + kReachWarps - 1) / kReachWarps));
    const void* const kernel = a.pull             ? (const void*)k_reach<Op, true, false>
                               : a.row > kPropHub ? (const void*)k_reach<Op, false, true>
                                                  : (const void*)k_reach<Op, false, false>;
    SCC_CUDA(cudaMemsetAsync(P.ctl, 0, sizeof(PropCtl), st));
    void* args[] = {(void*)&P};
    SCC_CUDA(cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(kReachBlock), args, 0, st));
    count_launch();
    PropCtl c;
    SCC_CUDA(cudaMemcpyAsync(&c, P.ctl, sizeof(c), cudaMemcpyDeviceToHost, st));
    SCC_CUDA(cudaStreamSynchronize(st));
    if (c.status == 2) return SCC_ERR_INVALID_ARG;
    return c.err;
}

}  // namespace

int run_reach(const ReachArgs& a, cudaStream_t st) {
    return a.words == 1 ? launch_reach<PropOr>(a, st) : launch_reach<PropOr2>(a, st);
}

// One device word, cleared, filled by `launch` and read back.
template <class F>
static int word_of(unsigned long long* tmp, int32_t* out, cudaStream_t st, F&& launch) {
    SCC_CUDA(cudaMemsetAsync(tmp, 0, sizeof(unsigned long long), st));
    launch();
    SCC_LAUNCH();
    unsigned long long b = 0;
    SCC_CUDA(cudaMemcpyAsync(&b, tmp, sizeof(b), cudaMemcpyDeviceToHost, st));
    SCC_CUDA(cudaStreamSynchronize(st));
    *out = (int32_t)(uint32_t)b;
    return SCC_OK;
}

int longest_row(const int32_t* off, int32_t n, unsigned long long* tmp, int num_sms, int32_t* most, cudaStream_t st) {
    return word_of(tmp, most, st, [&] { k_longest_row<<<num_sms * 4, 256, 0, st>>>(off, n, tmp); });
}

int find_hub(const int32_t* off, const int32_t* toff, int32_t n, unsigned long long* tmp, int num_sms, int32_t* hub,
             cudaStream_t st) {
    return word_of(tmp, hub, st, [&] { k_hub<<<num_sms * 4, 256, 0, st>>>(off, toff, n, tmp); });
}

}  // namespace scc

// Placement stage of the paper's heuristic (Section 3.2.2, Algorithms 2 and 3) in one launch: every run
// of cuts gets a path of unused nodes at the largest bandwidth threshold for which one of the trial
// colourings has a colourful path (Eq. 8 + K-PATH).
//
// Algorithm 2 bisects over the sorted bandwidths and asks the colour-coding table at each probe whether a
// path exists.  The answer is monotone in the threshold for every colouring, so the bisection ends at the
// widest bottleneck over the colourings, and that comes out of one pass over the table if it holds
// bottlenecks instead of bits:
//   W[C][v] = largest over paths with colour set C that end at v of the smallest bandwidth on the path,
//   W[C + colour(v')][v'] = max over u of min(W[C][u], bw[u][v']).
// The node sets reachable at a threshold t are exactly those with W >= t, so the path that the bisection
// would rebuild (lowest end vertex, then lowest predecessors, at the final threshold, first colouring that
// has one) can be read from the same table.
//
// A block takes one colouring at a time, the table in shared memory, the colour sets of a size in
// parallel over its warps (a lane owns the vertices lane and lane + 32).  The blocks' bottlenecks meet in
// one 64-bit maximum per run (bottleneck, lower colouring first) and a grid barrier; the winner's path is
// in global memory by then.  What bounds a run is the latency of its few steps: with 24 colourings of 50
// nodes and runs of one to three cuts about 4 us each, where a bisection took 11 probes of a launch, two
// copies and a synchronisation (45 us) each.
#include "pp_internal.cuh"

namespace pp {

namespace {

constexpr int kMatchThreads = 512;
constexpr int kMatchWarps = kMatchThreads / 32;
constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr int kSpinLimit = 1 << 22;

__device__ __forceinline__ int lowest(uint32_t lo, uint32_t hi) { return lo ? __ffs(lo) - 1 : hi ? 31 + __ffs(hi) : -1; }

__global__ void __launch_bounds__(kMatchThreads, 1) k_match(const MatchDev d)
{
    extern __shared__ __align__(16) uint32_t smem_match[];
    const int n = d.n, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    uint32_t *s_bw = smem_match;       // [n][n]
    uint32_t *W = smem_match + n * n;  // [2^kk][n]
    __shared__ uint8_t s_col[64];
    __shared__ int s_nodes[64], s_path[PP_KPATH_MAX_K];
    __shared__ uint32_t s_thr[64];
    __shared__ unsigned long long s_used, s_key;
    __shared__ int s_ok;
    MatchCtl *ctl = d.ctl;
    for (int e = tid; e < n * n; e += kMatchThreads) s_bw[e] = (e / n == e % n) ? 0u : d.bw[e];
    if (tid < 64) {
        s_nodes[tid] = -1;
        s_thr[tid] = 0u;
    }
    if (tid == 0) s_used = 0ull;
    __syncthreads();
    bool fail = false;
    for (int run = 0; run < d.n_runs && !fail; ++run) {
        const int first = d.runs[run].first, kk = d.runs[run].cuts + 1;
        const uint32_t nsets = 1u << kk, all = nsets - 1u;
        const int sv = s_nodes[first], uv = s_nodes[first + kk - 1];
        unsigned long long alive = ~s_used;
        if (sv >= 0) alive |= 1ull << sv;
        if (uv >= 0) alive |= 1ull << uv;
        unsigned long long best = 0ull;  // (bottleneck, ~colouring) of this block
        for (int t = blockIdx.x; t < d.trials; t += gridDim.x) {
            __syncthreads();
            for (uint32_t e = tid; e < nsets * n; e += kMatchThreads) W[e] = 0u;
            if (tid < n) s_col[tid] = (uint8_t)(((unsigned long long)d.draws[(size_t)t * n + tid] * (unsigned)kk) >> 32);
            __syncthreads();
            if (tid < n && ((alive >> tid) & 1ull) && (sv < 0 || sv == tid)) W[(1u << s_col[tid]) * n + tid] = kFull;
            // this lane's two vertices as path ends; a node that is not available has no colour
            const int v0 = lane, v1 = lane + 32;
            const uint32_t c0 = v0 < n && ((alive >> v0) & 1ull) ? 1u << s_col[v0] : 0u;
            const uint32_t c1 = v1 < n && ((alive >> v1) & 1ull) ? 1u << s_col[v1] : 0u;
            for (int size = 1; size < kk; ++size) {
                __syncthreads();
                for (uint32_t C = 1 + wid; C < all; C += kMatchWarps) {
                    if (__popc(C) != size) continue;
                    const uint32_t *row = W + C * n;
                    // vertices a path with these colours ends at; the end vertex ends every walk
                    uint32_t lo = __ballot_sync(kFull, v0 < n && row[v0 < n ? v0 : 0] != 0u && v0 != uv);
                    uint32_t hi = __ballot_sync(kFull, v1 < n && row[v1 < n ? v1 : 0] != 0u && v1 != uv);
                    uint32_t w0 = 0u, w1 = 0u;
                    while (lo | hi) {
                        const int u = lowest(lo, hi);
                        if (lo) lo &= lo - 1; else hi &= hi - 1;
                        const uint32_t x = row[u];
                        w0 = max(w0, min(x, s_bw[u * n + (v0 < n ? v0 : 0)]));
                        w1 = max(w1, min(x, s_bw[u * n + (v1 < n ? v1 : 0)]));
                    }
                    if (c0 & ~C) W[(C | c0) * n + v0] = w0;  // one source set per entry: no other warp writes it
                    if (c1 & ~C) W[(C | c1) * n + v1] = w1;
                }
            }
            __syncthreads();
            if (wid == 0) {
                const uint32_t *row = W + all * n;
                const uint32_t x0 = v0 < n && (uv < 0 || uv == v0) ? row[v0] : 0u;
                const uint32_t x1 = v1 < n && (uv < 0 || uv == v1) ? row[v1] : 0u;
                const uint32_t b = __reduce_max_sync(kFull, max(x0, x1));
                const unsigned long long key = ((unsigned long long)b << 32) | (uint32_t)~t;
                if (b != 0u && key > best) {
                    best = key;
                    int v = lowest(__ballot_sync(kFull, x0 >= b), __ballot_sync(kFull, x1 >= b));
                    uint32_t C = all;
                    for (int i = kk - 1; i >= 0; --i) {
                        if (lane == 0) s_path[i] = v;
                        if (i == 0) break;
                        C &= ~(1u << s_col[v]);
                        const uint32_t *prev = W + C * n;
                        const bool h0 = v0 < n && v0 != uv && prev[v0 < n ? v0 : 0] >= b && s_bw[(v0 < n ? v0 : 0) * n + v] >= b;
                        const bool h1 = v1 < n && v1 != uv && prev[v1 < n ? v1 : 0] >= b && s_bw[(v1 < n ? v1 : 0) * n + v] >= b;
                        v = lowest(__ballot_sync(kFull, h0), __ballot_sync(kFull, h1));
                    }
                    __syncwarp();
                }
            }
        }
        __syncthreads();
        int32_t *slots = d.paths + (size_t)(run & 1) * gridDim.x * PP_KPATH_MAX_K;
        if (wid == 0 && best != 0ull && lane < kk) slots[blockIdx.x * PP_KPATH_MAX_K + lane] = s_path[lane];
        __syncwarp();
        if (tid == 0) {
            if (best != 0ull) atomicMax(&ctl->best[run], best);
            __threadfence();
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&ctl->arrived) : "memory");
            const uint32_t target = gridDim.x * (uint32_t)(run + 1);
            uint32_t seen;
            int spins = 0;
            do {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&ctl->arrived) : "memory");
            } while (seen < target && ++spins < kSpinLimit);
            s_ok = seen >= target;
            s_key = __ldcg(&ctl->best[run]);
        }
        __syncthreads();
        if (!s_ok) return;  // the host finds its record unwritten
        const unsigned long long key = s_key;
        if (key == 0ull) {
            fail = true;
        } else {
            const int owner = (int)(~(uint32_t)key % gridDim.x);
            const int node = tid < kk ? __ldcg(slots + owner * PP_KPATH_MAX_K + tid) : 0;
            if (tid < kk) s_nodes[first + tid] = node;
            if (tid < kk - 1) s_thr[first + tid] = (uint32_t)(key >> 32);
            if (tid < kk) atomicOr(&s_used, 1ull << node);
            __syncthreads();
        }
    }
    if (blockIdx.x == 0) {
        for (int j = tid; j <= d.n_cuts; j += kMatchThreads) d.out->nodes[j] = fail ? -1 : s_nodes[j];
        for (int j = tid; j < d.n_cuts; j += kMatchThreads) d.out->threshold[j] = s_thr[j];
        if (tid == 0) d.out->status = fail ? (int)PP_INFEASIBLE : (int)PP_OK;
    }
}

}  // namespace

size_t match_smem_bytes(int n, int kk) { return ((size_t)n * n + ((size_t)n << kk)) * 4; }

cudaError_t launch_match(const MatchDev &d, int kk_max, int sms, cudaStream_t s)
{
    const size_t sm = match_smem_bytes(d.n, kk_max);
    cudaError_t e = cudaFuncSetAttribute(k_match, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(d.trials < sms ? d.trials : sms));
    cfg.blockDim = dim3(kMatchThreads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_match, d);
}

}  // namespace pp

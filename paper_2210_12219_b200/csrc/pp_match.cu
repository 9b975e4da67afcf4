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
// parallel over its warps (a lane owns the vertices lane and lane + 32; a size with few sets splits the
// predecessors of a set among several warps, which meet in shared maxima).  Between runs the blocks
// exchange one record each: bottleneck, colouring and path, every 64-bit word tagged with the run, so that
// a reader that sees the tags has the words and neither side needs a fence or a second trip.
//
// What bounds a run is the latency of its few steps.  24 colourings of 50 nodes, five runs of one to three
// cuts: 79 000 cycles when a warp walked its predecessors one by one, a run read its draws and its bounds
// from global memory and the blocks met in a 64-bit maximum, a fence and a counter (35 000 table, 22 000
// meeting, 13 000 setting up, 6 000 path); 39 000 now, the stage's call 58 -> 40 us.  A bisection took 11
// probes of a launch, two copies and a synchronisation (45 us) for each run.
#include "pp_internal.cuh"

#include <cstring>

namespace pp {

namespace {

constexpr int kShortPath = 4;
constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr int kSpinLimit = 1 << 22;
constexpr int kMaxRuns = 64;
constexpr int kRecordWords = 8;  // of a block: two records of four words, by the parity of the run
constexpr int kAhead = 4;      // predecessors at a time
constexpr int kPadWords = 64;  // a lane without a second vertex reads this far beyond a row, and drops what it read
constexpr int kWordNodes = 9;  // nodes of a path in the third word of a record, the others in the fourth; 6 bits each

struct Binomials {
    uint16_t c[PP_KPATH_MAX_K + 1][PP_KPATH_MAX_K + 1];
};
constexpr Binomials binomials()
{
    Binomials t{};
    for (int n = 0; n <= PP_KPATH_MAX_K; ++n)
        for (int r = 0; r <= n; ++r) t.c[n][r] = r == 0 || r == n ? 1 : t.c[n - 1][r - 1] + t.c[n - 1][r];
    return t;
}
__constant__ const Binomials kSets = binomials();

__device__ __forceinline__ int lowest(uint32_t lo, uint32_t hi) { return lo ? __ffs(lo) - 1 : hi ? 31 + __ffs(hi) : -1; }

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// WORDS > 0: bandwidths, draws and runs travel as parameters of the launch.  Up to 8 KB that costs a call 2 us
// less than a copy in front of it; of 16 KB the parameters take longer than the copy (a launch carries all of
// its struct, 0.3 us for each KB beyond four).
template <int WORDS>
struct MatchIn {
    uint32_t v[WORDS];
};
template <>
struct MatchIn<0> {};

// Paths of up to kShortPath vertices have no work for more than eight warps, and every barrier costs by the warp
// (three runs of four vertices and less: 21.7 us a call with 512 threads, 20.9 with 256; ten vertices 118 and 140).
template <int kMatchThreads, int WORDS>
__global__ void __launch_bounds__(kMatchThreads, 1) k_match(const __grid_constant__ MatchDev d, const __grid_constant__ MatchIn<WORDS> in)
{
    constexpr int kMatchWarps = kMatchThreads / 32;
    extern __shared__ __align__(16) uint32_t smem_match[];
    const int n = d.n, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    uint32_t *s_bw = smem_match;       // [n][n]
    uint32_t *W = smem_match + n * n + kPadWords;  // [2^kk][n]
    uint16_t *s_set = reinterpret_cast<uint16_t *>(W + ((size_t)n << d.kk));  // colour sets by size, ascending in a size
    __shared__ uint8_t s_col[64];
    __shared__ int s_nodes[64], s_base[PP_KPATH_MAX_K + 1];
    __shared__ uint32_t s_thr[64];
    __shared__ MatchRun s_runs[kMaxRuns];
    __shared__ unsigned long long s_top[kMatchWarps], s_path[2];
    PP_BLOCK_BOUNDS(chk);
    [[maybe_unused]] const size_t n_w = (size_t)n << d.kk, n_bw = (size_t)n * n + kPadWords;  // entries of the tables
    const uint32_t *g_bw = d.bw, *g_draws = d.draws;
    const MatchRun *g_runs = d.runs;
    if constexpr (WORDS > 0) {
        g_bw = in.v;
        // an address of their own: neighbouring threads read neighbouring words, which the constant bank would
        // serve one after another
        asm volatile("" : "+l"(g_bw));
        g_draws = g_bw + n * n;
        g_runs = reinterpret_cast<const MatchRun *>(g_bw + match_runs_at(n, d.trials));
    }
    // the records of the launch before this one lie in the other half: no tag in it for the launch after
    if (blockIdx.x == 0)
        for (int i = tid; i < kRecordWords * d.stride; i += kMatchThreads) d.records[(size_t)(d.half ^ 1) * kRecordWords * d.stride + i] = 0ull;
    const uint32_t draw = tid < n ? g_draws[(size_t)blockIdx.x * n + tid] : 0u;  // of the block's first colouring
    uint32_t part[PP_KPATH_MAX_N * PP_KPATH_MAX_N / kMatchThreads];  // of the bandwidths, on their way while the sets are listed
#pragma unroll
    for (int i = 0; i < PP_KPATH_MAX_N * PP_KPATH_MAX_N / kMatchThreads; ++i) {
        const int e = tid + i * kMatchThreads;
        part[i] = e < n * n ? g_bw[e] : 0u;
    }
    if (tid < d.n_runs) s_runs[tid] = g_runs[tid];
    if (tid < 64) {
        s_nodes[tid] = -1;
        s_thr[tid] = 0u;
    }
    // the sets of `size` of d.kk colours; those of fewer colours are the first of them
    for (int size = wid; size <= d.kk; size += kMatchWarps) {
        int at = 0;
        for (int s = 0; s < size; ++s) at += kSets.c[d.kk][s];
        if (lane == 0) s_base[size] = at;
        for (uint32_t C0 = 0; C0 < 1u << d.kk; C0 += 32) {
            const uint32_t C = C0 + lane;
            const bool mine = C < 1u << d.kk && __popc(C) == size;
            const uint32_t all = __ballot_sync(kFull, mine);
            if (mine) s_set[at + __popc(all & ((1u << lane) - 1u))] = (uint16_t)C;
            at += __popc(all);
        }
    }
#pragma unroll
    for (int i = 0; i < PP_KPATH_MAX_N * PP_KPATH_MAX_N / kMatchThreads; ++i) {
        const int e = tid + i * kMatchThreads;
        if (e < n * n) s_bw[e] = part[i];
    }
    __syncthreads();
    if (tid < n) s_bw[tid * n + tid] = 0u;
    // colours of a colouring for a path of `vertices`, and an empty table
    auto prepare = [&](uint32_t dr, int vertices) {
        for (uint32_t e = tid; e < (uint32_t)n << vertices; e += kMatchThreads)
            if (PP_IN_BOUNDS(chk, e, n_w)) W[e] = 0u;
        if (tid < n) s_col[tid] = (uint8_t)__umulhi(dr, (uint32_t)vertices);
    };
    prepare(draw, s_runs[0].cuts + 1);
    unsigned long long used = 0ull;
    bool fail = false;
    for (int run = 0; run < d.n_runs && !fail; ++run) {
        const int first = s_runs[run].first, kk = s_runs[run].cuts + 1;
        const uint32_t all = (1u << kk) - 1u;
        const int sv = s_nodes[first], uv = s_nodes[first + kk - 1];
        unsigned long long alive = ~used;
        if (sv >= 0) alive |= 1ull << sv;
        if (uv >= 0) alive |= 1ull << uv;
        unsigned long long best = 0ull;  // (bottleneck, ~colouring) of this block
        int node = 0;                    // of the first warp's lane i: node i of its path
        for (int t = blockIdx.x; t < d.trials; t += gridDim.x) {
            if (t != (int)blockIdx.x) {
                __syncthreads();  // the path has been read from the table
                prepare(tid < n ? g_draws[(size_t)t * n + tid] : 0u, kk);
            }
            __syncthreads();
            if (tid < n && tid != uv && ((alive >> tid) & 1ull) && (sv < 0 || sv == tid) && PP_IN_BOUNDS(chk, (1u << s_col[tid]) * n + tid, n_w)) W[(1u << s_col[tid]) * n + tid] = kFull;
            // this lane's two vertices as path ends; a node that is not available has no colour
            const int v0 = lane, v1 = lane + 32;
            const int r0 = v0 < n ? v0 : 0, r1 = v1 < n ? v1 : 0;
            const uint32_t c0 = v0 < n && ((alive >> v0) & 1ull) ? 1u << s_col[v0] : 0u;
            const uint32_t c1 = v1 < n && ((alive >> v1) & 1ull) ? 1u << s_col[v1] : 0u;
            for (int size = 1; size < kk; ++size) {
                const int sets = kSets.c[kk][size], base = s_base[size];
                const int cut = sets > kMatchWarps ? 0 : __clz(sets - 1) - __clz(kMatchWarps - 1);  // log2 of the warps to a set
                // the end vertex ends every walk: it is entered with the last colour only
                const uint32_t e0 = v0 == uv && size < kk - 1 ? 0u : c0, e1 = v1 == uv && size < kk - 1 ? 0u : c1;
                const int share = (n + (1 << cut) - 1) >> cut;
                __syncthreads();
                for (int item = wid; item < sets << cut; item += kMatchWarps) {
                    const uint32_t C = s_set[base + (item >> cut)];
                    const int from = (item & ((1 << cut) - 1)) * share, to = min(from + share, n);
                    const uint32_t *row = W + C * n, *bw = s_bw + lane;
                    uint32_t w0 = 0u, w1 = 0u;
                    int u = from;
                    for (; u + kAhead <= to; u += kAhead) {
#pragma unroll
                        for (int i = 0; i < kAhead; ++i) {
                            if (!PP_IN_BOUNDS(chk, C * n + u + i, n_w) || !PP_IN_BOUNDS(chk, lane + (u + i) * n + 32, n_bw)) break;
                            const uint32_t x = row[u + i];
                            w0 = max(w0, min(x, bw[(u + i) * n]));
                            w1 = max(w1, min(x, bw[(u + i) * n + 32]));
                        }
                    }
                    if (u < to) {
#pragma unroll
                        for (int i = 0; i < kAhead - 1; ++i) {
                            const int ui = min(u + i, to - 1);  // the last one again where there are none left
                            if (!PP_IN_BOUNDS(chk, C * n + ui, n_w) || !PP_IN_BOUNDS(chk, lane + ui * n + 32, n_bw)) break;
                            const uint32_t x = row[ui];
                            w0 = max(w0, min(x, bw[ui * n]));
                            w1 = max(w1, min(x, bw[ui * n + 32]));
                        }
                    }
                    // one source set per entry: no other set writes it
                    if (cut == 0) {
                        if ((e0 & ~C) && PP_IN_BOUNDS(chk, (C | e0) * n + v0, n_w)) W[(C | e0) * n + v0] = w0;
                        if ((e1 & ~C) && PP_IN_BOUNDS(chk, (C | e1) * n + v1, n_w)) W[(C | e1) * n + v1] = w1;
                    } else {
                        if ((e0 & ~C) && w0 && PP_IN_BOUNDS(chk, (C | e0) * n + v0, n_w)) atomicMax(&W[(C | e0) * n + v0], w0);
                        if ((e1 & ~C) && w1 && PP_IN_BOUNDS(chk, (C | e1) * n + v1, n_w)) atomicMax(&W[(C | e1) * n + v1], w1);
                    }
                }
            }
            __syncthreads();
            if (wid == 0) {
                const uint32_t *row = W + all * n;
                const uint32_t x0 = v0 < n && (uv < 0 || uv == v0) && PP_IN_BOUNDS(chk, all * n + v0, n_w) ? row[v0] : 0u;
                const uint32_t x1 = v1 < n && (uv < 0 || uv == v1) && PP_IN_BOUNDS(chk, all * n + v1, n_w) ? row[v1] : 0u;
                const uint32_t b = __reduce_max_sync(kFull, max(x0, x1));
                const unsigned long long key = ((unsigned long long)b << 32) | (uint32_t)~t;
                if (b != 0u && key > best) {
                    best = key;
                    int v = lowest(__ballot_sync(kFull, x0 >= b), __ballot_sync(kFull, x1 >= b));
                    uint32_t C = all;
                    const bool in0 = (v0 < n) & (v0 != uv), in1 = (v1 < n) & (v1 != uv);
                    for (int i = kk - 1; i >= 0; --i) {
                        if (lane == i) node = v;
                        if (i == 0) break;
                        C &= ~(1u << s_col[v]);
                        const uint32_t *prev = W + C * n;
                        const bool ok = PP_IN_BOUNDS(chk, C * n + max(r0, r1), n_w) && PP_IN_BOUNDS(chk, max(r0, r1) * n + v, n_bw);
                        const bool h0 = ok && (min(prev[r0], s_bw[r0 * n + v]) >= b) & in0;
                        const bool h1 = ok && (min(prev[r1], s_bw[r1 * n + v]) >= b) & in1;
                        v = lowest(__ballot_sync(kFull, h0), __ballot_sync(kFull, h1));
                    }
                }
            }
        }
        // records of this parity were read by every block before it posted the run in between
        unsigned long long *rec = d.records + ((size_t)d.half * 2 + (run & 1)) * d.stride * 4;
        const unsigned long long tag = (unsigned long long)(run + 1);
        if (wid == 0) {
            const uint32_t id = lane < kk && best != 0ull ? (uint32_t)node : 0u;
            const uint32_t n0 = __reduce_or_sync(kFull, lane < 5 ? id << (6 * lane) : 0u);
            const uint32_t n1 = __reduce_or_sync(kFull, lane >= 5 && lane < kWordNodes ? id << (6 * (lane - 5)) : 0u);
            const uint32_t n2 = __reduce_or_sync(kFull, lane >= kWordNodes && lane < PP_KPATH_MAX_K ? id << (6 * (lane - kWordNodes)) : 0u);
            const unsigned long long word = lane == 0   ? tag << 32 | best >> 32
                                            : lane == 1 ? tag << 32 | (uint32_t)best
                                            : lane == 2 ? tag << 56 | (unsigned long long)n1 << 30 | n0
                                                        : tag << 56 | n2;
            if (lane < 4) st_relaxed(rec + (size_t)blockIdx.x * 4 + lane, word);
        }
        if (run + 1 < d.n_runs) {  // while the records travel
            __syncthreads();
            prepare(draw, s_runs[run + 1].cuts + 1);
        }
        unsigned long long key = 0ull, p0 = 0ull, p1 = 0ull;
        bool late = false;
        if (tid < d.posts) {
            const unsigned long long *r = rec + (size_t)tid * 4;
            int spins = 0;
            for (;;) {
                const unsigned long long a = ld_relaxed(r), b = ld_relaxed(r + 1);
                p0 = ld_relaxed(r + 2);
                p1 = ld_relaxed(r + 3);
                if (a >> 32 == tag && b >> 32 == tag && p0 >> 56 == tag && p1 >> 56 == tag) {
                    key = a << 32 | (uint32_t)b;
                    break;
                }
                if (++spins >= d.polls) {
                    late = true;
                    break;
                }
            }
        }
        const uint32_t hi = __reduce_max_sync(kFull, (uint32_t)(key >> 32));
        const uint32_t lo = __reduce_max_sync(kFull, (uint32_t)(key >> 32) == hi ? (uint32_t)key : 0u);
        if (lane == 0) s_top[wid] = (unsigned long long)hi << 32 | lo;
        if (__syncthreads_or(late)) return;  // the host finds its record unwritten
        unsigned long long top = 0ull;
        for (int i = 0; i < ((int)gridDim.x + 31) / 32; ++i) top = max(top, s_top[i]);
        if (top >> 32 == 0ull) {
            fail = true;
        } else {
            if (key == top) {
                s_path[0] = p0;
                s_path[1] = p1;
            }
            __syncthreads();
            p0 = s_path[0];
            p1 = s_path[1];
            for (int i = 0; i < kk; ++i) {
                const int at = (int)((i < kWordNodes ? p0 >> (6 * i) : p1 >> (6 * (i - kWordNodes))) & 63);
                used |= 1ull << at;
                if (tid == i) s_nodes[first + i] = at;
            }
            if (tid < kk - 1) s_thr[first + tid] = (uint32_t)(top >> 32);
            __syncthreads();
        }
    }
    if (PP_BROKEN(chk) && tid == 0) d.out->bounds = 1;
    if (blockIdx.x == 0) {
        for (int j = tid; j <= d.n_cuts; j += kMatchThreads) d.out->nodes[j] = fail ? -1 : s_nodes[j];
        for (int j = tid; j < d.n_cuts; j += kMatchThreads) d.out->threshold[j] = s_thr[j];
        if (tid == 0) d.out->status = fail ? (int)PP_INFEASIBLE : (int)PP_OK;
    }
}

}  // namespace

PP_CHECKS_OF(match)

size_t match_smem_bytes(int n, int kk) { return ((size_t)n * n + kPadWords + ((size_t)n << kk)) * 4 + ((size_t)2 << kk); }

size_t match_record_bytes(int sms) { return (size_t)2 * kRecordWords * 8 * sms; }

namespace {

template <int THREADS, int WORDS>
cudaError_t launch_match_of(const MatchDev &d, const MatchIn<WORDS> &in, cudaStream_t s)
{
    const size_t sm = match_smem_bytes(d.n, d.kk);
    cudaError_t e = allow_shared(k_match<THREADS, WORDS>, 2048);
    if (e != cudaSuccess) return e;
    MatchDev q = d;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(d.trials < d.stride ? d.trials : d.stride));
    q.posts = (int)cfg.gridDim.x;
    q.polls = kSpinLimit;
    if (const int polls = q.posts < q.stride ? starved_polls() : 0) {  // test hook: a block that never comes
        ++q.posts;
        q.polls = polls;
    }
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_match<THREADS, WORDS>, q, in);
}

template <int WORDS>
cudaError_t launch_match_in(const MatchDev &d, const MatchIn<WORDS> &in, cudaStream_t s)
{
    return d.kk <= kShortPath ? launch_match_of<256>(d, in, s) : launch_match_of<512>(d, in, s);
}

constexpr int kParamWords = 2000;

}  // namespace

cudaError_t launch_match(const MatchDev &d, const uint32_t *in, size_t words, cudaStream_t s)
{
    if (d.bw) return launch_match_in<0>(d, MatchIn<0>{}, s);
    MatchIn<kParamWords> params;
    std::memcpy(params.v, in, words * 4);
    return launch_match_in<kParamWords>(d, params, s);
}

bool match_as_params(size_t words) { return words <= (size_t)kParamWords; }

}  // namespace pp

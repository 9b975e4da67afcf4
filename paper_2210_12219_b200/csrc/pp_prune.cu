// The exact search as a sparse frontier with a bound, one launch for the whole solve.
//
// The dense sweep (pp_sweep*.cu) computes every state of the recurrence
//   dp[S'][w][c'] = min over c in [lo_w(c'), c'-1] of g[c],
//   g[c] = min over v in S = S'\{w} of max(dp[S][v][c], gamma[c][v][w]).
// Values never fall along a plan, so a state that is no better than a complete plan already known
// cannot be part of a better one.  The levels are walked in the order of the number of nodes used,
// and a plan with fewer nodes wins a tie; a state is therefore kept only while its value is
//   < the best final value found on a lower level, and
//   <= the best one found on the level that is being written (another node set may still win the tie).
// Likewise a state whose remaining layers need more memory than the unused nodes have together
// cannot be completed.  What is left is exact: every state on a plan of value beta* survives, so the
// final choice and the backtrack see what they would see in the dense table.  On the named
// configurations and on the paper's evaluation graphs 0.1 to 5 % of the node sets keep a state; what
// bounds the solve is then the latency of a handful of levels, not the table.
//
// Values are 32-bit keys of the fp64 quotients (one correctly rounded division per layer and link):
// 0 for +0.0, all ones for +inf, else 1 + (bits - base) >> shift, base and shift such that the
// smallest and the largest possible quotient fit.  A key stands for a class of neighbouring doubles
// (relative width about 2^-28), and since the map is monotone the minima and maxima of keys are the
// keys of the minima and maxima.  The plan found is therefore optimal and canonical unless the class
// of beta* holds a quotient smaller than the plan's own bottleneck.  That is checked at the end; if it
// does, the search runs again (block 0 alone) with keys that resolve exactly this class.  A rank
// compression as the dense search has it would be exact at once, but ranking 30 000 quotients takes
// longer (0.03 ms) than the search.
//
// One cooperative launch: blocks meet at a barrier in global memory once per level.
//   level 2   one group of lanes per ordered pair (v, w): the keys of the link (kept in `gam` for the
//             later levels), the base state of v, the row of ({v, w}, w)
//   level j   the node sets of the frontier are a list; a group of lanes takes (S, w), reads the rows
//             of S that can still matter, and writes the row of (S + w, w) if any of its states does
//   end       once a level has little work block 0 goes on alone (its barrier costs nothing); it walks
//             back by the threshold rule, checks the class of beta*, and writes the result record
// A group of G lanes holds a row, P consecutive cut positions per lane.
#include <algorithm>
#include <cstring>
#include <functional>

#include "pp_thresholds.cuh"

namespace pp {

namespace {

constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr uint32_t kInfKey = 0xFFFFFFFFu;
constexpr int kClusterBlocks = 8, kClusterRounds = 2;
constexpr int kWideK = 10;  // nodes up to which short rows take two positions a lane (k = 14, L = 60: 192 us, with four 144)
constexpr int kSharedRounds = 3;  // k = 6, L = 12: 17 -> 12 us a solve; k = 7 (5 rounds) no gain, k = 8 a loss
constexpr size_t kSharedBytes = 220 * 1024;
constexpr int kAhead = 8;             // steps of a window scan whose compute times are asked for at a time
constexpr int kSpinLimit = 1 << 22;  // polls of a barrier before the kernel gives up
// The second search is block 0's alone, at 0.2 us a row it keeps.  After a first one of more node sets than this a
// caller that has the dense search, which is exact at once, gets to run that (k = 14, L = 100, every state kept:
// 25.6 -> 0.3 ms on the device; a search that a bound thins out has a few hundred sets at k = 18).
constexpr uint32_t kAloneSets = 1024;
constexpr int kAloneRounds = 2;      // a level of at most this many rounds of one block is done by block 0 alone
// P = 8 (129 to 256 layers): 20 warps, more of a level's targets in a round.  Against 16 warps, mean of nine
// instances each at L = 135, 200, 240: k = 18 34.0, 32.1, 29.1 -> 31.5, 28.9, 26.1 us a solve, k = 17 33.7, 29.1, 28.6 ->
// 32.4, 28.0, 26.3, k = 13 and 15 within 2 %; k = 11 26.8, 25.9, 25.4 -> 27.4, 26.7, 25.7, where 16 would do.
__host__ __device__ constexpr int prune_threads(int P) { return P == 8 ? 640 : P <= 16 ? 512 : 256; }

// Which class of doubles a key stands for.
struct KeyMap {
    unsigned long long base;
    int shift;
    uint32_t zoom;  // 0, or the class that is resolved exactly: smaller values become 0, larger ones +inf
    __device__ __forceinline__ uint32_t operator()(double x) const
    {
        const unsigned long long b = (unsigned long long)__double_as_longlong(x);
        if (b == 0ull) return 0u;
        const uint32_t key = 1u + (uint32_t)((b - base) >> shift);
        if (!zoom) return key;
        return key < zoom ? 0u : key > zoom ? kInfKey : 1u + (uint32_t)((b - base) & ((1ull << shift) - 1ull));
    }
};

// first value that is not worth keeping on `level`, given the best final state known
__device__ __forceinline__ uint32_t limit_of(unsigned long long best, int level)
{
    if (best == kNoBest) return kInfKey;
    const uint32_t val = (uint32_t)(best >> 30);
    return ((int)(best >> 25) & 31) < level ? val : val + 1u;
}

// smallest of a group's keys
template <int G>
__device__ __forceinline__ uint32_t group_min(uint32_t u)
{
    if constexpr (G == 32) {
        u = __reduce_min_sync(kFull, u);
    } else {
#pragma unroll
        for (int o = G >> 1; o; o >>= 1) u = min(u, __shfl_xor_sync(kFull, u, o, G));
    }
    return u;
}

// Shared memory: the part common to the block, then one strip per group of lanes.
struct PruneLayout {
    size_t bits, M, cap, bw, Wp, speed, gmin, lo, code, strips, total;
};
__host__ __device__ inline PruneLayout prune_layout(int L, int k, int Lp, int groups, size_t strip, bool codes, bool compute)
{
    PruneLayout p;
    size_t o = 0;
    auto take = [&o](size_t bytes) { size_t at = o; o = (o + bytes + 15) & ~(size_t)15; return at; };
    p.bits = take((size_t)Lp * 8);
    p.M = take((size_t)(L + 1) * 8);
    p.cap = take((size_t)k * 8);
    p.bw = take((size_t)k * k * 4);
    p.Wp = take(compute ? (size_t)(L + 1) * 8 : 0);
    p.speed = take(compute ? (size_t)k * 4 : 0);
    p.gmin = take((size_t)k * k * 4);  // the tables of the search by thresholds lie from here on, before the others do
    p.lo = take((size_t)k * Lp * 2);
    p.code = take(codes ? (size_t)k * Lp * sizeof(WindowCode) : 0);
    p.strips = o;
    p.total = o + (size_t)groups * strip;
    return p;
}
// Window codes where a warp works off several rows of every node: short chains, few blocks.
template <int G, int P, bool CT>
constexpr bool kCodes = G * P <= 64 && !CT;

// strip of a group: its window minima, then the ids of the source rows
template <int G, int P>
constexpr size_t kStripBytes = ((size_t)(Strip<G, P>::kSize + PP_MAX_K) * 4 + 15) & ~(size_t)15;

// Long rows of the first level: a team of four warps to a row, so that no lane has a chain of P divisions and P
// window minima while most warps of the GPU have no row at all (level of 156 rows of 337 positions, P = 16:
// 14 300 cycles by one warp a row, 6500 so; 306 rows of 200, P = 8: 6400 and 4200).  Up to two rounds of them; with more rows
// than that a warp a row keeps the SMs as busy.
constexpr int kTeam = 128;
template <int G, int P, bool CT>
constexpr bool kByTeams = !CT && G == 32 && P >= 8;

// Barrier of a team, and whether any of its threads says so.
__device__ __forceinline__ bool team_any(int team, bool mine)
{
    uint32_t any;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(any)
                 : "r"((uint32_t)mine), "r"(2 + team), "n"(kTeam)
                 : "memory");
    return any != 0u;
}

// What another block may have written: past L1.  SM: the tables are in shared memory.
template <bool SM, typename T>
__device__ __forceinline__ T ld_now(const T *p)
{
    if constexpr (SM) return *p;
    else return __ldcg(p);
}

// P keys of a row; CA: as they are, through L1 or in shared memory
template <int P, bool CA>
__device__ __forceinline__ void load_row(const uint32_t *p, uint32_t (&x)[P])
{
    if constexpr (P == 2) {
        const uint2 t = CA ? *reinterpret_cast<const uint2 *>(p) : __ldcg(reinterpret_cast<const uint2 *>(p));
        x[0] = t.x; x[1] = t.y;
    } else {
#pragma unroll
        for (int i = 0; i < P; i += 4) {
            const uint4 t = CA ? *reinterpret_cast<const uint4 *>(p + i) : __ldcg(reinterpret_cast<const uint4 *>(p + i));
            x[i] = t.x; x[i + 1] = t.y; x[i + 2] = t.z; x[i + 3] = t.w;
        }
    }
}
template <int P>
__device__ __forceinline__ void store_row(uint32_t *p, const uint32_t (&x)[P])
{
    if constexpr (P == 2) {
        *reinterpret_cast<uint2 *>(p) = make_uint2(x[0], x[1]);
    } else {
#pragma unroll
        for (int i = 0; i < P; i += 4) *reinterpret_cast<uint4 *>(p + i) = make_uint4(x[i], x[i + 1], x[i + 2], x[i + 3]);
    }
}

// The same at index i of a table of n entries: checked in the bounds-checking build, where a value from outside
// reads as 0 and a row as +inf.
template <bool SM, typename T>
__device__ __forceinline__ T ld_at(const Bounds &chk, const T *table, size_t i, size_t n)
{
    return PP_IN_BOUNDS(chk, i, n) ? ld_now<SM>(table + i) : T(0);
}
template <typename T>
__device__ __forceinline__ void st_at(const Bounds &chk, T *table, size_t i, size_t n, T x)
{
    if (PP_IN_BOUNDS(chk, i, n)) table[i] = x;
}
template <int P, bool CA>
__device__ __forceinline__ void load_row_at(const Bounds &chk, const uint32_t *table, size_t i, size_t n, uint32_t (&x)[P])
{
    if (PP_IN_BOUNDS(chk, i, n) && PP_IN_BOUNDS(chk, i + P - 1, n)) {
        load_row<P, CA>(table + i, x);
    } else {
#pragma unroll
        for (int q = 0; q < P; ++q) x[q] = kInfKey;
    }
}
template <int P>
__device__ __forceinline__ void store_row_at(const Bounds &chk, uint32_t *table, size_t i, size_t n, const uint32_t (&x)[P])
{
    if (PP_IN_BOUNDS(chk, i, n) && PP_IN_BOUNDS(chk, i + P - 1, n)) store_row<P>(table + i, x);
}

// All blocks of the grid; false when the wait ran out, here or in another block (the caller reports it and
// leaves by the end of the kernel, so that the counters are cleared).  A level's word holds the blocks
// that have arrived above the node sets it added (32 bits each), so that the last poll brings both; *best,
// polled along, may miss what the last blocks found, which only makes it a weaker bound.  (Reading both after
// the barrier cost another trip to L2, 600 cycles a level: k = 16, L = 136 28.7 -> 26.8 us, k = 10, L = 50 48.8 -> 47.9.)
__device__ __forceinline__ bool grid_barrier(const PruneDev &d, unsigned long long *word, unsigned long long *best, uint32_t *added)
{
    __shared__ int s_ok;
    PruneCtl *ctl = d.ctl;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long seen;
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(word), "l"(1ull << 32) : "memory");
        int spins = 0;
        uint32_t failed = 0;
        do {
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(*best) : "l"(&ctl->best) : "memory");
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(seen) : "l"(word) : "memory");
            if ((++spins & 1023) == 0) asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(failed) : "l"(&ctl->failed) : "memory");
        } while ((uint32_t)(seen >> 32) < d.arrivals && spins < d.polls && !failed);
        *added = (uint32_t)seen;
        s_ok = (uint32_t)(seen >> 32) >= d.arrivals;
        if (!s_ok) asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(&ctl->failed), "r"(1u) : "memory");
    }
    __syncthreads();
    return s_ok != 0;
}

// The inputs travel as a kernel parameter (4 KB for chains of up to 128 layers, 18 KB for the longest): no
// copy to queue in front of the search and to wait for.
template <int N, bool CT>
struct PruneIn {
    unsigned long long bits[N], M[N + 1], cap[PP_MAX_K];
    uint32_t bw[PP_MAX_K * PP_MAX_K];
};
template <int N>
struct PruneIn<N, true> {
    unsigned long long bits[N], M[N + 1], cap[PP_MAX_K];
    uint32_t bw[PP_MAX_K * PP_MAX_K], speed[PP_MAX_K];
    unsigned long long Wp[N + 1];
};

// SM: the tables of the search in shared memory, one block (launch_prune).  TH: the search by thresholds first, with its tables
// as tlay has them.
template <int G, int P, bool CT, bool SM, bool TH>
__global__ void __launch_bounds__(prune_threads(P), 1) k_prune(const PruneDev d, const ThresholdLayout tlay,
                                                               const __grid_constant__ PruneIn<G * P, CT> params)
{
    constexpr int kThreads = prune_threads(P), kWarps = kThreads / 32, kGroups = kThreads / G, kPerWarp = 32 / G;
    extern __shared__ __align__(16) unsigned char smem_prune[];
    const int k = d.k, L = d.L, Lp = d.Lp, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int sl = lane & (G - 1), gb = lane & ~(G - 1);  // position in the group, first lane of the group
    const int at = sl * P;                                // this lane's first cut position
    const bool in_row = at < Lp;
    const int at0 = in_row ? at : 0;
    const PruneLayout lay = prune_layout(L, k, Lp, kGroups, kStripBytes<G, P>, kCodes<G, P, CT>, CT);
    double *s_bits = reinterpret_cast<double *>(smem_prune + lay.bits);
    unsigned long long *s_M = reinterpret_cast<unsigned long long *>(smem_prune + lay.M);
    unsigned long long *s_cap = reinterpret_cast<unsigned long long *>(smem_prune + lay.cap);
    uint32_t *s_bw = reinterpret_cast<uint32_t *>(smem_prune + lay.bw);
    uint32_t *s_gmin = reinterpret_cast<uint32_t *>(smem_prune + lay.gmin);
    int16_t *s_lo = reinterpret_cast<int16_t *>(smem_prune + lay.lo);
    [[maybe_unused]] unsigned long long *s_Wp = reinterpret_cast<unsigned long long *>(smem_prune + lay.Wp);
    [[maybe_unused]] uint32_t *s_speed = reinterpret_cast<uint32_t *>(smem_prune + lay.speed);
    [[maybe_unused]] WindowCode *s_code = reinterpret_cast<WindowCode *>(smem_prune + lay.code);
    uint32_t *s_strip = reinterpret_cast<uint32_t *>(smem_prune + lay.strips + (size_t)(tid / G) * kStripBytes<G, P>);
    uint32_t *s_ids = s_strip + Strip<G, P>::kSize;
    __shared__ unsigned long long s_best;  // best final state the block knows of
    __shared__ unsigned int s_pick[kWarps];
    __shared__ int s_cut[PP_MAX_K], s_node[PP_MAX_K];
    __shared__ unsigned long long s_worst;  // bits of the plan's bottleneck
    __shared__ unsigned long long s_low;    // bits of the smallest quotient in the optimum's class
    __shared__ uint32_t s_cnt;
    __shared__ int s_fail;
    [[maybe_unused]] constexpr int kTeams = kThreads / kTeam, kOwn = (G * P + kTeam - 1) / kTeam;
    [[maybe_unused]] const int team = tid / kTeam, in_team = tid % kTeam;
    [[maybe_unused]] uint32_t *team_row =  // two rows, in the strips of the team's warps
        reinterpret_cast<uint32_t *>(smem_prune + lay.strips + (size_t)team * (kTeam / G) * kStripBytes<G, P>);
    __shared__ uint32_t s_team[kWarps][2];
    PruneCtl *ctl = d.ctl;
    __shared__ uint32_t s_count[SM ? 64 : 1];
    unsigned char *tables = smem_prune + lay.total;  // SM: in the layout they have in global memory
    const SparseLayout tl = sparse_layout(k, Lp);
    uint32_t *t_live = SM ? reinterpret_cast<uint32_t *>(tables + tl.live) : d.live;
    unsigned long long *t_rowmap = SM ? reinterpret_cast<unsigned long long *>(tables + tl.rowmap) : d.rowmap;
    uint32_t *t_list = SM ? reinterpret_cast<uint32_t *>(tables + tl.list) : d.list;
    uint32_t *t_gam = SM ? reinterpret_cast<uint32_t *>(tables + tl.gam) : d.gam;
    uint32_t *t_gmin = SM ? reinterpret_cast<uint32_t *>(tables + tl.gmin) : d.gmin;
    uint32_t *t_rows = SM ? reinterpret_cast<uint32_t *>(tables + tl.rows) : d.rows;
    [[maybe_unused]] uint32_t *t_seg = SM ? t_rows + (((size_t)k << (k - 1)) * Lp) : d.seg;
    // entries of the tables
    [[maybe_unused]] const Bounds chk{&ctl->err};
    [[maybe_unused]] const size_t n_sets = (size_t)1 << k, n_map = (size_t)k << k, n_gam = (size_t)k * k * Lp, n_rows = (size_t)d.row_cap * Lp,
                                  n_seg = (size_t)k * L * Lp;
    const double kInf = __longlong_as_double(0x7FF0000000000000ll);
    const int top = k < L ? k : L;
    const uint32_t full = (1u << k) - 1u;
    const int npairs = k * (k - 1) / 2;

    unsigned long long t_start = 0;
    if ((TH || blockIdx.x == 0) && tid == 0) asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t_start));
    // ---- inputs ----
    // read through an address of their own: neighbouring threads read neighbouring words, which the constant
    // bank would serve one after another
    const PruneIn<G * P, CT> *in = &params;
    asm volatile("" : "+l"(in));
    [[maybe_unused]] unsigned long long *s_raw = reinterpret_cast<unsigned long long *>(smem_prune + tlay.raw);
    for (int c = tid; c < Lp; c += kThreads) {
        const unsigned long long x = c < L ? in->bits[c] : 0ull;
        s_bits[c] = (double)x;
        if constexpr (TH) s_raw[c] = x << 10 | (unsigned)c;
    }
    for (int c = tid; c <= L; c += kThreads) s_M[c] = in->M[c];
    for (int e = tid; e < k * k; e += kThreads) s_bw[e] = in->bw[e];
    if (tid < k) s_cap[tid] = in->cap[tid];
    if (SM && tid < 64) s_count[tid] = 0u;
    if (tid == 0) s_best = kNoBest;
    if constexpr (CT) {
        for (int c = tid; c <= L; c += kThreads) s_Wp[c] = in->Wp[c];
        if (tid < k) s_speed[tid] = in->speed[tid];
    }
    __syncthreads();
    bool solved = false;  // by thresholds
    int writer = 0;       // the block that has the result
    int m = 0, w_end = 0, status = (int)PP_INFEASIBLE;
    double beta = kInf;
    if constexpr (TH) {
        if (CT || d.whole == 0) {
            const ThresholdIn tin{L, k, s_raw, s_M, s_cap, s_bw, CT ? s_Wp : nullptr, CT ? s_speed : nullptr};
            const int outcome = threshold_search<(G * P + 31) / 32, CT, kThreads>(d, tin, tlay, smem_prune, chk, s_cut, s_node, &writer, &m, &beta);
            solved = outcome != kThresholdOpen;
            if (outcome == kThresholdSolved) status = m > 0 ? (int)PP_OK : (int)PP_ERR_CUDA;
            if (outcome == kThresholdGaveUp) status = (int)PP_ERR_CUDA;
            if (m < 0) {
                m = 0;
                beta = kInf;
            }
            __syncthreads();
        }
    }
    for (int e = tid; e < k * k; e += kThreads) s_gmin[e] = kInfKey;
    if (sl == 0) s_strip[Strip<G, P>::kNone] = kInfKey;
    auto set_window = [&](int w, int c, int l) {
        s_lo[w * Lp + c] = (int16_t)l;
        if constexpr (kCodes<G, P, CT>) s_code[w * Lp + c] = window_code<G, P, uint32_t>(c, l);
    };
    // window starts: lo[w][c'] = earliest previous cut c >= 0 such that layers c+1..c' fit on w, c' itself when
    // not even layer c' alone does; by bisection, a lane has four positions of a node in flight (runs of
    // neighbouring positions, found by stepping on from one to the next: 9300 cycles at k = 13, L = 337)
    if (solved) {
    } else if (d.lo)  // a problem that is solved again and again has them on the device
        for (int w = wid; w < k; w += kWarps)
            for (int c = lane; c < Lp; c += 32) set_window(w, c, c < L ? (int)d.lo[w * L + c] : c);
    else
    for (int w = wid; w < k; w += kWarps) {
        constexpr int kU = G * P >= 128 ? 4 : G * P >= 64 ? 2 : 1;
        const unsigned long long capw = s_cap[w];
        for (int c0 = lane; c0 < Lp; c0 += 32 * kU) {
            unsigned long long thr[kU];
            int l[kU], last[kU];  // l: largest index <= last with M[l] < thr, 0 when there is none
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                last[u] = min(c0 + 32 * u, L - 1);
                const unsigned long long need = s_M[last[u] + 1];
                thr[u] = need > capw ? need - capw : 0ull;
                l[u] = 0;
            }
#pragma unroll
            for (int step = G * P / 2; step; step >>= 1)
#pragma unroll
                for (int u = 0; u < kU; ++u)
                    if (l[u] + step <= last[u] && s_M[l[u] + step] < thr[u]) l[u] += step;
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int c = c0 + 32 * u;
                if (c < Lp) set_window(w, c, c < L ? l[u] : c);
            }
        }
    }
    __syncthreads();
    const unsigned long long total = s_M[L];
    const uint32_t tight_levels = d.tight_levels, whole = d.whole;
    __shared__ double s_room[384];  // memory of a set of nodes, seven of them at a time
    if (tight_levels)
        for (int e = tid; e < 384; e += kThreads) {
            double sum = 0.0;
            for (int b = 0; b < 7; ++b) {
                const int v = (e >> 7) * 7 + b;
                if (((e >> b) & 1) && v < k) sum += (double)s_cap[v];
            }
            s_room[e] = sum;
        }
    __syncthreads();

    KeyMap key_of{d.key_base, d.key_shift, 0u};
    bool dense = false;
    int nblk = SM ? 1 : (int)gridDim.x;  // blocks that work on the search: 1 once block 0 goes on alone

    // base state of one node: layers 0..c on v
    auto base_key = [&](int v, int c) -> uint32_t {
        if (s_M[c + 1] > s_cap[v]) return kInfKey;
        if constexpr (CT) return s_speed[v] ? key_of(__ddiv_rn((double)s_Wp[c + 1], (double)s_speed[v])) : kInfKey;
        return 0u;
    };
    // layers 0..c have to hold this much for the nodes outside S2 to hold the rest
    auto must_hold = [&](uint32_t S2) -> unsigned long long {
        const uint32_t rest = full & ~S2;
        double room = s_room[rest & 127u] + s_room[128 + (rest >> 7 & 127u)] + s_room[256 + (rest >> 14)];
        room *= 1.0 + 1e-9;  // rounding of the sums must not drop a state
        return room < (double)total ? total - (unsigned long long)room : 0ull;
    };
    auto note_final = [&](uint32_t x, int level, uint32_t S2, int w) {
        const unsigned long long cand = pack_best(x, level, S2, w);
        if (cand < *reinterpret_cast<volatile unsigned long long *>(&s_best)) atomicMin(&s_best, cand);
    };
    // row of (S2, w) from g: window minimum, then drop what cannot matter, note a final state; returns
    // whether the group keeps the row, and its smallest value
    auto make_row = [&](const uint32_t (&g)[P], uint32_t (&out)[P], uint32_t S2, int w, int level, uint32_t lim, bool on,
                        uint32_t &rmin) -> bool {
        if constexpr (!CT) {
            if constexpr (kCodes<G, P, CT>) window_min<G, P>(g, s_code + (size_t)w * Lp + at0, s_strip, sl, kInfKey, out);
            else window_min_direct<G, P>(g, s_lo + (size_t)w * Lp + at0, s_strip, sl, kInfKey, out);
        } else {
            // the compute time of the last partition depends on both its ends: every output scans its
            // window, nearest start first, until the compute time alone is too much
#pragma unroll
            for (int i = 0; i < P; ++i) s_strip[at + i] = g[i];
            __syncwarp();
            uint32_t cur[P];
            cur[0] = at > 0 ? s_strip[at - 1] : kInfKey;
#pragma unroll
            for (int i = 1; i < P; ++i) cur[i] = g[i - 1];
#pragma unroll
            for (int i = 0; i < P; ++i) out[i] = kInfKey;
            const size_t seg = (size_t)w * L * Lp + at0;
            for (int d0 = 0; d0 < L; d0 += kAhead) {  // the loads of kAhead steps are in flight together
                uint32_t x[kAhead][P];
#pragma unroll
                for (int u = 0; u < kAhead; ++u) load_row_at<P, true>(chk, t_seg, seg + (size_t)min(d0 + u, L - 1) * Lp, n_seg, x[u]);
                bool more = false;
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    const int dd = d0 + u;
#pragma unroll
                    for (int i = 0; i < P; ++i) {
                        out[i] = min(out[i], max(cur[i], x[u][i]));
                        more |= x[u][i] < lim;
                    }
#pragma unroll
                    for (int i = P - 1; i > 0; --i) cur[i] = cur[i - 1];
                    cur[0] = at - 2 - dd >= 0 ? s_strip[at - 2 - dd] : kInfKey;
                }
                if (!more || at + P - 1 - kAhead - d0 < 0) break;
            }
        }
        const bool tight = (tight_levels >> level) & 1u;
        const unsigned long long must = tight ? must_hold(S2) : 0ull;
        uint32_t least = kInfKey, x = kInfKey;
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const int c = at + i;
            if (!on || out[i] >= lim || c >= L || (tight && s_M[c + 1] < must)) out[i] = kInfKey;
            least = min(least, out[i]);
            if (c == L - 1) x = out[i];
        }
        if (x != kInfKey) note_final(x, level, S2, w);
        rmin = group_min<G>(least);
        return rmin != kInfKey;
    };
    // end of a level: the block's best final state goes to the others; false = a barrier gave up
    // and s_cnt has the node sets it added to the frontier
    auto level_end = [&](unsigned long long best_before, int level) -> bool {
        __syncthreads();
        if (nblk == 1) {
            if (tid == 0) s_cnt = SM ? s_count[(key_of.zoom ? 32 : 0) + level] : (uint32_t)__ldcg(ctl->count + (key_of.zoom ? 32 : 0) + level);
            __syncthreads();
            return true;
        }
        if (tid == 0 && s_best < best_before)
            asm volatile("red.relaxed.gpu.global.min.u64 [%0], %1;" ::"l"(&ctl->best), "l"(s_best) : "memory");
        unsigned long long seen = kNoBest;
        uint32_t added = 0;
        if (d.clustered) {
            asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
            if (tid == 0) {
                seen = __ldcg(&ctl->best);
                added = (uint32_t)__ldcg(ctl->count + level);
            }
        } else if (!grid_barrier(d, ctl->count + level, &seen, &added)) {
            return false;
        }
        if (tid == 0) {
            s_cnt = added;
            if (seen < s_best) s_best = seen;
        }
        __syncthreads();
        return true;
    };

    bool found = solved || (!CT && whole != 0);
    if (found && !solved) {
        m = 1;
        beta = 0.0;
        w_end = __ffs(whole) - 1;
        status = (int)PP_OK;
        if (tid < PP_MAX_K) {
            s_cut[tid] = -1;
            s_node[tid] = tid == 0 ? w_end : -1;
        }
    }
    auto next_place = [&](int level) -> uint32_t {  // of a level's node sets in the frontier
        const int at = (key_of.zoom ? 32 : 0) + level;
        if constexpr (SM) return atomicAdd(&s_count[at], 1u);
        else return (uint32_t)atomicAdd(ctl->count + at, 1ull);
    };
    while (!found) {
        const int slots = nblk * kWarps, my_slot = wid * nblk + (nblk == 1 ? 0 : (int)blockIdx.x);
        // node sets of three nodes and more start without rows (those of two nodes are all written below)
        for (uint32_t S = (nblk == 1 ? 0 : blockIdx.x) * kThreads + tid; S < (1u << k); S += nblk * kThreads)
            if (__popc(S) > 2) st_at(chk, t_live, S, n_sets, 0u);
        if constexpr (CT) {
            // compute times of every run of layers: seg[(w * L + d) * Lp + c'] = layers c'-d .. c' on w
            const int n = k * L * Lp;
            for (int e = (nblk == 1 ? 0 : (int)blockIdx.x) * kThreads + tid; e < n; e += nblk * kThreads) {
                const int r = e / Lp, c2 = e - r * Lp, w = r / L, first = c2 - (r - w * L);
                uint32_t key = kInfKey;
                const uint32_t sp = s_speed[w];
                if (c2 < L && first >= 0 && sp != 0 && s_M[c2 + 1] - s_M[first] <= s_cap[w])
                    key = key_of(__ddiv_rn((double)(s_Wp[c2 + 1] - s_Wp[first]), (double)sp));
                st_at(chk, t_seg, e, n_seg, key);
            }
            if (tid == 0)
                for (int v = 0; v < k; ++v) {
                    const uint32_t x = base_key(v, L - 1);
                    if (x != kInfKey) s_best = min(s_best, pack_best(x, 1, 1u << v, v));
                }
            if (!level_end(kNoBest, 1)) goto gave_up;
        }
        // ---- two nodes: the keys of every link, the rows of every pair ----
        if (top >= 2) {
            const unsigned long long before = s_best;
            const int items = k * (k - 1);
            bool by_teams = false;
            if constexpr (kByTeams<G, P, CT>) {
                by_teams = items <= 2 * nblk * kTeams;
                if (by_teams) {
                    for (int it = team * nblk + (nblk == 1 ? 0 : (int)blockIdx.x); it < items; it += nblk * kTeams) {
                        const int v = it / (k - 1), o = it - v * (k - 1), w = o + (o >= v ? 1 : 0);
                        const uint32_t link = s_bw[v * k + w], S2 = (1u << v) | (1u << w);
                        const double div = (double)link;
                        uint32_t x[kOwn], out[kOwn], gm = kInfKey, least = kInfKey;
                        int lo[kOwn], t[kOwn];  // t: log2 of the window's length, -1: no window
#pragma unroll
                        for (int q = 0; q < kOwn; ++q) {
                            const int c = in_team + q * kTeam;
                            uint32_t key = kInfKey;
                            x[q] = out[q] = kInfKey;
                            lo[q] = 0;
                            t[q] = -1;
                            if (c < L) {
                                if (link != 0) key = key_of(__ddiv_rn(s_bits[c], div));
                                if (c < L - 1) gm = min(gm, key);
                                x[q] = max(key, base_key(v, c));
                                lo[q] = s_lo[w * Lp + c];
                                if (lo[q] < c) t[q] = 31 - __clz(c - lo[q]);
                            }
                            if (c < Lp) {
                                st_at(chk, t_gam, (size_t)(w * k + v) * Lp + c, n_gam, key);
                                team_row[c] = x[q];
                            }
                        }
                        // sparse table of the row, one level at a time: out = min over [lo, c - 1]
                        uint32_t *cur = team_row, *next = team_row + Lp;
                        for (int s = 0;; ++s) {
                            bool more = false;
#pragma unroll
                            for (int q = 0; q < kOwn; ++q) more |= t[q] > s;
                            more = team_any(team, more);
#pragma unroll
                            for (int q = 0; q < kOwn; ++q)
                                if (t[q] == s) out[q] = min(cur[in_team + q * kTeam - 1], cur[lo[q] + (1 << s) - 1]);
                            if (!more) break;
#pragma unroll
                            for (int q = 0; q < kOwn; ++q) {
                                const int c = in_team + q * kTeam;
                                if (c < Lp) {
                                    if (c >= 1 << s) x[q] = min(x[q], cur[c - (1 << s)]);
                                    next[c] = x[q];
                                }
                            }
                            uint32_t *const swap = cur;
                            cur = next;
                            next = swap;
                        }
                        const uint32_t lim = limit_of(*reinterpret_cast<volatile unsigned long long *>(&s_best), 2);
                        const bool tight = (tight_levels >> 2) & 1u;
                        const unsigned long long must = tight ? must_hold(S2) : 0ull;
#pragma unroll
                        for (int q = 0; q < kOwn; ++q) {
                            const int c = in_team + q * kTeam;
                            if (out[q] >= lim || c >= L || (tight && s_M[c + 1] < must)) out[q] = kInfKey;
                            least = min(least, out[q]);
                            if (c == L - 1 && out[q] != kInfKey) note_final(out[q], 2, S2, w);
                        }
                        least = __reduce_min_sync(kFull, least);
                        gm = __reduce_min_sync(kFull, gm);
                        if (lane == 0) {
                            s_team[wid][0] = least;
                            s_team[wid][1] = gm;
                        }
                        team_any(team, false);
#pragma unroll
                        for (int i = 0; i < kTeam / 32; ++i) {
                            least = min(least, s_team[team * (kTeam / 32) + i][0]);
                            gm = min(gm, s_team[team * (kTeam / 32) + i][1]);
                        }
                        const int a = v < w ? v : w, b = v < w ? w : v;
                        const int pr = a * (2 * k - a - 1) / 2 + (b - a - 1);
                        const uint32_t id = 2u * (uint32_t)pr + (w == b ? 1u : 0u);
                        if (least != kInfKey)
#pragma unroll
                            for (int q = 0; q < kOwn; ++q) {
                                const int c = in_team + q * kTeam;
                                if (c < Lp) st_at(chk, t_rows, (size_t)id * Lp + c, n_rows, out[q]);
                            }
                        if (in_team == 0) {
                            st_at(chk, t_gmin, w * k + v, k * k, gm);
                            st_at(chk, t_rowmap, (size_t)S2 * k + w, n_map, ((unsigned long long)least << 32) | id);
                            if (w == b) {
                                st_at(chk, t_list, pr, n_sets, S2);
                                st_at(chk, t_live, S2, n_sets, S2);
                            }
                        }
                    }
                }
            }
            for (int base = by_teams ? items : my_slot * kPerWarp; base < items; base += slots * kPerWarp) {
                const int it = base + lane / G;
                const bool on = it < items;
                const int v = on ? it / (k - 1) : 0, x = on ? it - v * (k - 1) : 0, w = x + (x >= v ? 1 : 0);
                const uint32_t link = on ? s_bw[v * k + w] : 0u;
                const double div = (double)link;
                uint32_t g[P], out[P], gm = kInfKey, rmin;
#pragma unroll
                for (int i = 0; i < P; ++i) {
                    const int c = at + i;
                    g[i] = (link != 0 && c < L) ? key_of(__ddiv_rn(s_bits[c], div)) : kInfKey;
                    if (c < L - 1) gm = min(gm, g[i]);
                }
                if (on && in_row) store_row_at<P>(chk, t_gam, (size_t)(w * k + v) * Lp + at, n_gam, g);
                gm = group_min<G>(gm);
                if (on && sl == 0) st_at(chk, t_gmin, w * k + v, k * k, gm);
#pragma unroll
                for (int i = 0; i < P; ++i) {
                    const int c = at + i;
                    g[i] = c < L ? max(g[i], base_key(v, c)) : kInfKey;
                }
                const uint32_t S2 = (1u << v) | (1u << w);
                const uint32_t lim = limit_of(*reinterpret_cast<volatile unsigned long long *>(&s_best), 2);
                const bool keep = make_row(g, out, S2, w, 2, lim, on, rmin);
                const int a = v < w ? v : w, b = v < w ? w : v;
                const int pr = a * (2 * k - a - 1) / 2 + (b - a - 1);
                const uint32_t id = 2u * (uint32_t)pr + (w == b ? 1u : 0u);
                if (keep && in_row) store_row_at<P>(chk, t_rows, (size_t)id * Lp + at, n_rows, out);
                if (on && sl == 0) {
                    st_at(chk, t_rowmap, (size_t)S2 * k + w, n_map, ((unsigned long long)rmin << 32) | id);
                    if (w == b) {
                        st_at(chk, t_list, pr, n_sets, S2);
                        st_at(chk, t_live, S2, n_sets, S2);
                    }
                }
                __syncwarp();
            }
            if (!level_end(before, 2)) goto gave_up;
            for (int e = tid; e < k * k; e += kThreads) s_gmin[e] = (e / k != e % k) ? ld_at<SM>(chk, t_gmin, e, k * k) : kInfKey;
            __syncthreads();
        }

        // ---- three nodes and more ----
        uint32_t beg = 0, cnt = (uint32_t)npairs;
        unsigned long long used = 2ull * npairs;  // rows: one per item, kept or not, so that ids need no counter
        bool alone = nblk == 1;
        for (int level = 3; level <= top && cnt; ++level) {
            const int nw = k - (level - 1);
            const uint32_t recip_nw = 0xFFFFFFFFu / (uint32_t)nw + 1u;  // floor(it / nw) by a multiplication: it < 2^27
            const unsigned long long items = (unsigned long long)cnt * nw;
            if (used + items > d.row_cap) {
                dense = true;
                break;
            }
            if (!alone && items <= (unsigned long long)(kGroups * kAloneRounds)) {
                if (blockIdx.x != 0) break;
                alone = true;
                nblk = 1;
            }
            const unsigned long long before = s_best;
            const int my = alone ? wid : my_slot, all = alone ? kWarps : slots;
            for (unsigned long long base = (unsigned long long)my * kPerWarp; base < items; base += (unsigned long long)all * kPerWarp) {
                const unsigned long long it = base + lane / G;
                const bool on = it < items;
                const uint32_t li = on ? (nw > 1 ? __umulhi((uint32_t)it, recip_nw) : (uint32_t)it) : 0u;
                const uint32_t S = ld_at<SM>(chk, t_list, beg + li, n_sets);
                const int w = select_bit(full & ~S, on ? (int)((uint32_t)it - li * (uint32_t)nw) : 0);
                const uint32_t rows_of_S = ld_at<SM>(chk, t_live, S, n_sets);
                const uint32_t lim = limit_of(*reinterpret_cast<volatile unsigned long long *>(&s_best), level);
                // source rows that can still matter: their smallest value and the link's smallest key
                uint32_t src = 0;
#pragma unroll
                for (int v0 = 0; v0 < PP_MAX_K; v0 += G) {
                    if (v0 >= k) break;
                    const int v = v0 + sl;
                    bool ok = false;
                    if (v < k && ((S >> v) & 1u)) {
                        const unsigned long long e = ld_at<SM>(chk, t_rowmap, (size_t)S * k + v, n_map);
                        s_ids[v] = (uint32_t)e;
                        ok = on && ((rows_of_S >> v) & 1u) && max((uint32_t)(e >> 32), s_gmin[w * k + v]) < lim;
                    }
                    const uint32_t hit = __ballot_sync(kFull, ok);
                    src |= (G == 32 ? hit : ((hit >> gb) & ((1u << (G & 31)) - 1u))) << v0;
                }
                if (!__any_sync(kFull, src != 0)) continue;
                __syncwarp();
                uint32_t g[P];
#pragma unroll
                for (int i = 0; i < P; ++i) g[i] = kInfKey;
                while (src != 0) {  // two sources at a time: their loads are in flight together
                    const int v = __ffs(src) - 1;
                    src &= src - 1;
                    const int v2 = src ? __ffs(src) - 1 : v;
                    src &= src - 1;
                    if (in_row) {
                        uint32_t a[P], b[P], a2[P], b2[P];
                        load_row_at<P, SM>(chk, t_rows, (size_t)s_ids[v] * Lp + at, n_rows, a);
                        load_row_at<P, SM>(chk, t_gam, (size_t)(w * k + v) * Lp + at, n_gam, b);
                        load_row_at<P, SM>(chk, t_rows, (size_t)s_ids[v2] * Lp + at, n_rows, a2);
                        load_row_at<P, SM>(chk, t_gam, (size_t)(w * k + v2) * Lp + at, n_gam, b2);
#pragma unroll
                        for (int i = 0; i < P; ++i) g[i] = min(g[i], min(max(a[i], b[i]), max(a2[i], b2[i])));
                    }
                }
                uint32_t gm = g[0], out[P], rmin;
#pragma unroll
                for (int i = 1; i < P; ++i) gm = min(gm, g[i]);
                if (!__any_sync(kFull, gm < lim)) continue;
                const uint32_t S2 = S | (1u << w);
                if (make_row(g, out, S2, w, level, lim, on, rmin)) {
                    const uint32_t id = (uint32_t)(used + it);
                    if (in_row) store_row_at<P>(chk, t_rows, (size_t)id * Lp + at, n_rows, out);
                    if (sl == 0) {
                        st_at(chk, t_rowmap, (size_t)S2 * k + w, n_map, ((unsigned long long)rmin << 32) | id);
                        if (PP_IN_BOUNDS(chk, S2, n_sets) && atomicOr(t_live + S2, 1u << w) == 0u)
                            st_at(chk, t_list, beg + cnt + next_place(level), n_sets, S2);
                    }
                }
                __syncwarp();
            }
            used += items;
            if (!level_end(before, level)) goto gave_up;
            beg += cnt;
            cnt = s_cnt;
        }
        if (blockIdx.x != 0 || dense) break;  // block 0 finishes
        if (!SM && tid == 0 && gridDim.x > 1 && !d.clustered && !key_of.zoom) s_best = min(s_best, __ldcg(&ctl->best));
        __syncthreads();
        const unsigned long long best = s_best;
        if (best == kNoBest) break;  // no plan

        // ---- final choice, backtrack: the lowest (c, v) whose value is within the optimum's class ----
        status = (int)PP_OK;
        m = (int)(best >> 25) & 31;
        const uint32_t vstar = (uint32_t)(best >> 30);
        uint32_t S = (uint32_t)(best >> 5) & 0xFFFFFu;
        int w = (int)best & 31, c2 = L - 1;
        if (tid < PP_MAX_K) s_cut[tid] = s_node[tid] = -1;
        if (tid == 0) {
            s_low = ~0ull;
            s_fail = 0;
        }
        __syncthreads();
        // Half of the warps walk back, the others look for the smallest quotient in the optimum's class.  With the
        // tables in shared memory one warp does the walk, lanes over the positions: a node takes it less time
        // than the two barriers a step that several warps need (k = 6, L = 12 from host arrays: 32.1 -> 31.2 us).
        constexpr int kBack = SM ? 1 : kWarps / 2;
        if (wid < kBack) {
            for (int j = m - 1; j >= 0; --j) {
                if (tid == 0) {
                    s_node[j] = w;
                    if (j < m - 1) s_cut[j] = c2;
                }
                if (j == 0) break;
                const uint32_t from = S & ~(1u << w);
                const int lo = s_lo[(size_t)w * Lp + c2], np = __popc(from);
                const uint32_t rows_of = np > 1 ? ld_at<SM>(chk, t_live, from, n_sets) : from;
                unsigned int pick = 0xFFFFFFFFu;
                if constexpr (SM)
                    for (int c0 = lo; c0 < c2 && pick == 0xFFFFFFFFu; c0 += 32) {
                        const int c = min(c0 + lane, c2 - 1);
                        for (uint32_t rem = from; rem; rem &= rem - 1) {
                            const int v = __ffs(rem) - 1;
                            const unsigned long long e = np > 1 ? ld_at<SM>(chk, t_rowmap, (size_t)from * k + v, n_map) : 0ull;
                            const bool ok = ((rows_of >> v) & 1u) && (uint32_t)(e >> 32) <= vstar;
                            uint32_t x = max(np > 1 ? ld_at<SM>(chk, t_rows, (size_t)(ok ? (uint32_t)e : 0u) * Lp + c, n_rows) : base_key(v, c),
                                             ld_at<SM>(chk, t_gam, (size_t)(w * k + v) * Lp + c, n_gam));
                            if constexpr (CT) x = max(x, ld_at<SM>(chk, t_seg, (size_t)(w * L + c2 - c - 1) * Lp + c2, n_seg));
                            if (ok && x <= vstar) pick = min(pick, ((unsigned)c << 5) | (unsigned)v);
                        }
                        pick = __reduce_min_sync(kFull, pick);
                    }
                for (int vi = wid; !SM && vi < np; vi += kBack) {
                    const int v = select_bit(from, vi);
                    const unsigned long long e = np > 1 ? ld_at<SM>(chk, t_rowmap, (size_t)from * k + v, n_map) : 0ull;
                    if (!((rows_of >> v) & 1u) || (uint32_t)(e >> 32) > vstar) continue;
                    const size_t row = (size_t)(uint32_t)e * Lp, gm = (size_t)(w * k + v) * Lp;
                    constexpr int kChunks = 4;  // of 32 positions, their loads in flight together
                    bool hit_one = false;
                    for (int c0 = lo; c0 < c2 && !hit_one; c0 += 32 * kChunks) {
                        uint32_t x[kChunks];
#pragma unroll
                        for (int u = 0; u < kChunks; ++u) {
                            const int c = c0 + 32 * u + lane;
                            x[u] = kInfKey;
                            if (c < c2) {
                                x[u] = max(np > 1 ? ld_at<SM>(chk, t_rows, row + c, n_rows) : base_key(v, c), ld_at<SM>(chk, t_gam, gm + c, n_gam));
                                if constexpr (CT) x[u] = max(x[u], ld_at<SM>(chk, t_seg, (size_t)(w * L + c2 - c - 1) * Lp + c2, n_seg));
                            }
                        }
#pragma unroll
                        for (int u = 0; u < kChunks; ++u) {
                            const unsigned int hits = __ballot_sync(kFull, x[u] <= vstar);
                            if (hits && !hit_one) {
                                pick = min(pick, ((unsigned)(c0 + 32 * u + __ffs(hits) - 1) << 5) | (unsigned)v);
                                hit_one = true;
                            }
                        }
                    }
                }
                if constexpr (!SM) {
                    if (lane == 0) s_pick[wid] = pick;
                    asm volatile("bar.sync 1, %0;" ::"n"(kBack * 32) : "memory");
                    pick = __reduce_min_sync(kFull, s_pick[lane < kBack ? lane : 0]);
                    asm volatile("bar.sync 1, %0;" ::"n"(kBack * 32) : "memory");
                }
                if (pick == 0xFFFFFFFFu) {  // cannot happen on a consistent frontier; report, do not trap
                    s_fail = 1;
                    break;
                }
                S = from;
                w = (int)(pick & 31u);
                c2 = (int)(pick >> 5);
            }
        } else if (!key_of.zoom && key_of.shift != 0 && vstar != 0u) {
            // They lie within 2^-24 of the lower end of the class (a class spans at most 2^27 of the 2^52
            // mantissas), so that a multiplication per link and two per layer find the few candidates; few
            // links have a quotient below the optimum at all.
            constexpr double kNear = 1.0 / (1 << 23);
            constexpr int kOthers = kWarps - kBack;
            const double edge = __longlong_as_double((long long)(key_of.base + ((unsigned long long)(vstar - 1u) << key_of.shift)));
            auto candidate = [&](double q) {
                if (key_of(q) == vstar) atomicMin(&s_low, (unsigned long long)__double_as_longlong(q));
            };
            for (int p0 = 0; p0 < k * k; p0 += 32 * kOthers) {
                const int p = p0 + lane * kOthers + wid - kBack, w2 = p / k, v2 = p - w2 * k;
                const bool has = p < k * k && s_gmin[p] <= vstar;
                const double link = has ? (double)s_bw[v2 * k + w2] : 0.0;
                for (uint32_t hits = __ballot_sync(kFull, has); hits; hits &= hits - 1) {
                    const double div = __shfl_sync(kFull, link, __ffs(hits) - 1), near = edge * div;
                    for (int c = lane; c < L - 1; c += 32) {
                        const double b = s_bits[c];
                        if (fabs(b - near) <= near * kNear) candidate(__ddiv_rn(b, div));
                    }
                }
            }
            if constexpr (CT) {  // compute times: for every end of a run the starts that come near, by bisection
                for (int e = tid - kBack * 32; e < k * L; e += kOthers * 32) {
                    const int w2 = e / L, last = e - w2 * L;
                    const double div = (double)s_speed[w2], near = edge * div, work = (double)s_Wp[last + 1];
                    if (div == 0.0) continue;
                    int a = 0, b = last + 1;
                    while (a < b) {
                        const int mid = (a + b) >> 1;
                        if ((double)s_Wp[mid] < work - near - near * kNear) a = mid + 1; else b = mid;
                    }
                    for (; a <= last && (double)s_Wp[a] <= work - near + near * kNear; ++a)
                        candidate(__ddiv_rn((double)(s_Wp[last + 1] - s_Wp[a]), div));
                }
            }
        }
        __syncthreads();
        if (s_fail) {
            status = (int)PP_ERR_CUDA;
            break;
        }
        // the plan's own bottleneck
        if (wid == 0) {
            double x = 0.0;
            if (tid < m - 1) x = __ddiv_rn(s_bits[s_cut[tid]], (double)s_bw[s_node[tid] * k + s_node[tid + 1]]);
            if constexpr (CT) {
                if (tid < m) {
                    const int first = tid ? s_cut[tid - 1] + 1 : 0, last = tid < m - 1 ? s_cut[tid] : L - 1;
                    const double y = __ddiv_rn((double)(s_Wp[last + 1] - s_Wp[first]), (double)s_speed[s_node[tid]]);
                    x = y > x ? y : x;
                }
            }
            unsigned long long bits = (unsigned long long)__double_as_longlong(x);
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                const unsigned long long other = __shfl_xor_sync(kFull, bits, o);
                bits = other > bits ? other : bits;
            }
            if (tid == 0) s_worst = bits;
        }
        __syncthreads();
        const unsigned long long worst = s_worst;
        beta = __longlong_as_double((long long)worst);
        // exact unless the class of the optimum holds a quotient smaller than the plan's own bottleneck
        if (key_of.zoom || s_low >= worst) break;
        if (d.fallback && beg + cnt > kAloneSets) {
            dense = true;
            break;
        }
        key_of.zoom = vstar;  // once more, this class resolved
        nblk = 1;
        if (tid == 0) s_best = kNoBest;
        __syncthreads();
    }

    goto result;
gave_up:  // a jump: leaving the loops by a flag cost every solve 0.3 % (k = 18, L = 200)
    status = (int)PP_ERR_CUDA;
    // ---- result ----
result:
    __syncthreads();
#ifdef PP_DEBUG_BOUNDS
    if ((int)blockIdx.x == writer && __ldcg(&ctl->err) != 0) {
        status = (int)PP_ERR_CUDA;
        beta = kInf;
        m = 0;
    }
    __syncthreads();
    if (SM && tid == 0) ctl->err = 0;
#endif
    if ((int)blockIdx.x == writer) {
        if (!dense && tid < PP_MAX_K) {
            d.out->cuts[tid] = m ? s_cut[tid] : -1;
            d.out->placement[tid] = m ? s_node[tid] : -1;
        }
        if (tid == 0) {
            if (!dense) {
                d.out->beta_ms = beta;
                d.out->status = status;
                d.out->m = m;
            }
            unsigned long long t_end;
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t_end));
            d.note->ns = (long long)(t_end - t_start);
            d.note->dense = dense ? 1 : 0;
            d.note->thresholds = !TH || (!CT && d.whole != 0) ? 0 : solved ? 1 : 2;
        }
    }
    if constexpr (SM) return;  // the counters in global memory are as they were
    // The last block to leave clears the counters for the next launch.  Every block comes here, also one whose
    // wait ran out.
    __shared__ uint32_t s_left;
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_left = atomicAdd(&ctl->left, 1u);
    }
    __syncthreads();
    if (s_left == gridDim.x - 1) {
        if (tid < 64) ctl->count[tid] = 0ull;
        if (tid == 0) {
            ctl->best = kNoBest;
            ctl->left = ctl->failed = 0u;
            ctl->err = 0;
        }
    }
}

struct PruneShape {
    int G, P;
};
// Lanes and positions a lane of a row.  Short rows of few nodes take two positions a lane: there are warps
// to spare, and the time of a level is that of a lane's own chain of instructions.
PruneShape prune_shape(int L, int k)
{
    PruneShape s = L <= 64 && k <= kWideK ? PruneShape{8, 2} : PruneShape{4, 4};
    while (s.G * s.P < L && s.G < 32) s.G *= 2;
    while (s.G * s.P < L) s.P *= 2;
    return s;
}

// targets of the widest level if it is kept whole
unsigned long long widest_level(int k)
{
    unsigned long long widest = 1, binom = 1;
    for (int j = 1; j <= k; ++j) {
        binom = binom * (unsigned)(k - j + 1) / (unsigned)j;  // C(k, j)
        widest = std::max(widest, binom * (unsigned)(k - j));
    }
    return widest;
}

// Shared memory of a block that holds the whole search; 0 when it does not fit or the widest level takes
// more than kSharedRounds rounds of a block's groups.  With the tables in shared memory a round takes 1.4 us
// against 3.3 in global memory, and there is no barrier of blocks (2 us a level and more).
template <int G, int P, bool CT>
size_t shared_bytes(int L, int k, int Lp)
{
    constexpr int groups = prune_threads(P) / G;
    if (k > 10 || widest_level(k) > (unsigned long long)kSharedRounds * groups) return 0;
    const size_t rows = ((size_t)k << (k - 1)) * Lp * 4, seg = CT ? (size_t)k * L * Lp * 4 : 0;
    const size_t all = prune_layout(L, k, Lp, groups, kStripBytes<G, P>, kCodes<G, P, CT>, CT).total + sparse_layout(k, Lp).rows + rows + seg;
    return all <= kSharedBytes ? all : 0;
}

constexpr size_t kOwnShared = 8192;  // static shared memory of k_prune, at most
// Whether the search by thresholds is tried first.  us a call, the bounded search / by thresholds, mean of five to 25 instances:
//   Eq. 1    cnn chains (L = 50, k = 8) 59.6 / 45.6, (50, 12) 69.0 / 50.3, (30, 9) 56.7 / 44.0; geometric graphs (14, 8) 45.9 / 37.6, (50, 12)
//            48.9 / 39.2, (60, 9) 45.1 / 38.5; blocks (50, 10) 67.8 / 56.5, (14, 11) 82.6 / 55.3; stages (30, 9) 43.8 / 34.8, (60, 8) 48 / 46
//   Eq. 2    cnn (50, 7) 51.3 / 46.4, (50, 8) 47.3 / 42.5, (14, 8) 45.2 / 40.6; uniform (40, 8) 53.4 / 45.1; blocks (50, 8) 43.5 / 41.2
// It runs in a block's shared memory and by one block a threshold, so that it loses where most rows of more than eight or
// nine nodes live.  Under Eq. 2 that cannot be told beforehand: cnn (50, 10) is 54.8 / 54.0 in the mean of 60 instances, 42 / 39 for an easy one
// and 73 / 95 for a hard one; there k <= 8, whose sets all have room.  Under Eq. 1, where the windows of the bounded search are scans, k
// <= 12; three of 60 of (50, 12) lose, 98 / 117 the most.  Chains that two nodes can hold end on the second level of the bounded
// search (Eq. 2, stages (64, 8) 32.4 / 33.9).  L <= 64: at 128 blocks lose (k = 8, 44.0 / 47.6).
// kThresholdRows: rows of as many nodes as the chain takes at least; uniform chains, whose optimum takes 6 of 10 nodes, have 2500
// and more and lose (Eq. 2, (50, 10) 51 / 78).
constexpr unsigned kThresholdRows = 1500;
// Three kinds of input lose by it whatever their size, and are seen beforehand (mean of eight instances, the bounded search / by thresholds):
//   no set of nodes holds the chain, which the bounded search sees on its first levels: Eq. 2 (50, 7) 30 / 36, (64, 8) 31 / 41, Eq. 1 (50, 8) 35 / 42
//   terms over more than kThresholdOctaves powers of two, of which the first round leaves too many between two blocks' thresholds: Eq. 2 (50, 7)
//     of near-equal layers and links with one far smaller layer and one far slower link 50 / 54 and, closer still, 51 / 58, (64, 8) 55 / 62 and
//     55 / 67, Eq. 1 (50, 5) 44 / 47 and 44 / 48 (but six nodes 52 / 51, eight 64 / 58)
//   stacks of identical layers, all of whose rows are alive at the optimum: Eq. 2 (50, 7) 42 / 48, (64, 8) 42 / 50 (24 layers 51 / 47 and 44 / 42),
//     Eq. 1 (50, 5) 43 / 46, (50, 10) 62 / 65, (64, 12) 72 / 81 (but (50, 6) 55 / 52, (50, 8) 63 / 60, (24, 12) 70 / 60)
constexpr int kThresholdOctaves = 20, kThresholdPlainK = 8;  // nodes under Eq. 2, at most
bool threshold_takes(const PruneDev &d, const PruneHost &h, bool compute)
{
    const int L = d.L, k = d.k;
    const uint64_t *cap = h.cap, total = h.M[L];
    if (L > 32 * kThresholdW || k > (compute ? kThresholdK : kThresholdPlainK)) return false;
    if ((!compute || k <= 5) && (d.key_top - d.key_base) >> 52 > (unsigned)kThresholdOctaves) return false;
    if (L > 32 && (!compute || k <= 5 || k >= 10)) {
        int alike = 0;
        for (int c = 0; c + 2 < L; ++c) alike += h.bits[c] == h.bits[c + 1] ? 1 : 0;
        if (2 * alike > L) return false;
    }
    uint64_t sorted[PP_MAX_K];
    std::copy(cap, cap + k, sorted);
    std::sort(sorted, sorted + k, std::greater<uint64_t>());
    int need = 0;
    uint64_t left = total;
    for (; need < k && left > 0; ++need) left -= std::min(left, sorted[need]);
    if (left > 0) return false;
    unsigned rows = 0, binom = 1;
    for (int j = 1; j <= need; ++j) {
        binom = binom * (unsigned)(k - j + 1) / (unsigned)j;  // C(k, j)
        rows += binom * (unsigned)j;
    }
    return rows <= kThresholdRows && (compute || need > 2);
}
// Where it comes before the search in one block's shared memory: Eq. 1, k = 6, 35 layers 40 to 52 / 33 to 45, 25 layers 30 to 41 / 31 to 41;
// k = 5, 50 layers 36.8 / 31.5 (and 2 for the scratch that the search behind it may need), 25 30.6 / 32.
bool threshold_before_shared(const PruneDev &d, const PruneHost &h)
{
    return h.Wp && d.k >= 5 && d.k * d.L >= 200 && threshold_takes(d, h, true);
}

// Eq. 2: a grid that takes every SM for itself gains 9 to 40 % a solve, and takes from solves on other streams what a cluster of eight
// blocks leaves them.  us a solve, one, two, four, eight handles on streams of their own, the bounded search and by thresholds: uniform
// (24, 7) 28.1, 14.4, 8.4, 7.7 and 20.8, 16.9, 18.2, 19.0; cnn (50, 8) 27.8, 15.3, 8.6, 4.8 and 22.2, 20.7, 20.9, 20.9 (by 24 and by 74 blocks
// 25.7, 17.0, -, 5.4 and 22.8, 14.0, -, 11.1).  Solves on the legacy stream run one after another in any case; Eq. 1 knows no other.
bool on_legacy_stream(cudaStream_t s) { return s == nullptr || s == cudaStreamLegacy; }

template <int G, int P, bool CT>
cudaError_t launch_shape(const PruneDev &d, const PruneHost &h, int sms, cudaStream_t s)
{
    PruneIn<G * P, CT> in;
    std::memcpy(in.bits, h.bits, (size_t)d.L * 8);
    std::memcpy(in.M, h.M, (size_t)(d.L + 1) * 8);
    std::memcpy(in.cap, h.cap, (size_t)d.k * 8);
    std::memcpy(in.bw, h.bw, (size_t)d.k * d.k * 4);
    if constexpr (CT) {
        std::memcpy(in.Wp, h.Wp, (size_t)(d.L + 1) * 8);
        std::memcpy(in.speed, h.speed, (size_t)d.k * 4);
    }
    constexpr int threads = prune_threads(P), groups = threads / G;
    PruneDev q = d;
    q.clustered = 0;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = s;
    cfg.attrs = attr;
    const bool before_shared = threshold_before_shared(d, h);
    const size_t all = before_shared ? 0 : shared_bytes<G, P, CT>(d.L, d.k, d.Lp);
    if (all) {
        cudaError_t e = allow_shared(k_prune<G, P, CT, true, false>, 4096);
        if (e != cudaSuccess) return e;
        q.row_cap = (unsigned long long)d.k << (d.k - 1);
        cfg.dynamicSmemBytes = all;
        return cudaLaunchKernelEx(&cfg, k_prune<G, P, CT, true, false>, q, ThresholdLayout{}, in);
    }
    // blocks: one round over the targets of the widest level if it is kept whole; a single block where
    // two rounds of it do, its barrier costs next to nothing
    const unsigned long long widest = widest_level(d.k);
    int blocks = (int)std::min<unsigned long long>((widest + groups - 1) / groups, (unsigned long long)sms);
    if (blocks <= 2) blocks = 1;
    const PruneLayout lay = prune_layout(d.L, d.k, d.Lp, groups, kStripBytes<G, P>, kCodes<G, P, CT>, CT);
    size_t sm = lay.total;
    ThresholdLayout tlay{};
    auto kernel = k_prune<G, P, CT, false, false>;
    static_assert(kWideK >= kThresholdPlainK, "Eq. 2 by thresholds has rows of two positions a lane");
    if constexpr (G * P <= 32 * kThresholdW && (CT || P == 2)) {
        if (before_shared || (blocks > 1 && (CT || on_legacy_stream(s)) && threshold_takes(d, h, CT))) {
            tlay = threshold_layout(d.L, d.k, (G * P + 31) / 32, CT, lay.gmin, kBlockShared - kOwnShared);
            sm = std::max(sm, tlay.total);
            blocks = sms;
            kernel = k_prune<G, P, CT, false, true>;
        }
    }
    // up to kClusterRounds rounds of 8 blocks: one cluster, whose barrier is the hardware's (0.3 us; one in
    // global memory 1.5 to 2)
    const bool cluster = tlay.set_cap == 0 && blocks > 1 && widest <= (unsigned long long)kClusterRounds * kClusterBlocks * groups;
    if (cluster) blocks = kClusterBlocks;
    cudaError_t e = allow_shared(kernel, kOwnShared);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.dynamicSmemBytes = sm;
    if (cluster) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)blocks;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    } else {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    }
    cfg.numAttrs = blocks > 1 ? 1 : 0;
    q.clustered = cluster ? 1 : 0;
    q.arrivals = (uint32_t)blocks;
    q.polls = kSpinLimit;
    if (const int polls = blocks > 1 && !cluster ? starved_polls() : 0) {  // test hook: a block that never comes
        ++q.arrivals;
        q.polls = polls;
    }
#ifdef PP_DEBUG_BOUNDS
    int late = 0;
    if (const int polls = tlay.set_cap ? late_polls(&late) : 0) {
        q.late = (uint32_t)late + 1u;
        q.polls = polls;
    }
#endif
    return cudaLaunchKernelEx(&cfg, kernel, q, tlay, in);
}

}  // namespace

PP_CHECKS_OF(prune)

int prune_row_pad(int L, int k)
{
    const int P = prune_shape(L, k).P;
    return (L + P - 1) / P * P;
}

void prune_ctl_init(PruneCtl *c)
{
    *c = PruneCtl{};
    c->best = kNoBest;
}

// base and shift of the keys of all values between lo and hi (the smallest and the largest positive one)
void prune_key_range(double lo, double hi, PruneDev *d)
{
    unsigned long long a, b;
    static_assert(sizeof a == sizeof lo, "doubles are 64 bits");
    std::memcpy(&a, &lo, 8);
    std::memcpy(&b, &hi, 8);
    d->key_base = a;
    d->key_top = b;
    d->key_shift = 0;
    while (((b - a) >> d->key_shift) >= 0x80000000ull) ++d->key_shift;
}

// The nodes that hold the whole chain, and the levels on which some choice of nodes leaves too little
// memory for some rest of it: even the k - j smallest nodes together hold everything on the others.
void prune_node_bounds(const uint64_t *cap, uint64_t total, PruneDev *d)
{
    uint64_t sorted[PP_MAX_K];
    d->whole = 0;
    for (int v = 0; v < d->k; ++v) {
        sorted[v] = cap[v];
        d->whole |= (cap[v] >= total ? 1u : 0u) << v;
    }
    std::sort(sorted, sorted + d->k);
    d->tight_levels = 0;
    double sum = 0.0;
    for (int n = 0; n <= d->k; ++n) {
        if (sum < (double)total) d->tight_levels |= 1u << (d->k - n);
        if (n < d->k) sum += (double)sorted[n];
    }
}

// F<G, P, CT> of the shape of a row of L layers among k nodes; Eq. 1 stops at 256 layers
#define PP_SHAPES(CASE) CASE(8, 2) CASE(16, 2) CASE(32, 2) CASE(4, 4) CASE(8, 4) CASE(16, 4) CASE(32, 4) CASE(32, 8)

bool prune_in_shared(const PruneDev &d, const PruneHost &h) { return !threshold_before_shared(d, h) && prune_in_shared(d.L, d.k, true); }

bool prune_in_shared(int L, int k, bool compute)
{
    const PruneShape sh = prune_shape(L, k);
    const int Lp = prune_row_pad(L, k);
    switch (sh.G * 100 + sh.P) {
#define PP_CASE(g, p) \
    case g * 100 + p: return (compute ? shared_bytes<g, p, true>(L, k, Lp) : shared_bytes<g, p, false>(L, k, Lp)) != 0;
        PP_SHAPES(PP_CASE)
#undef PP_CASE
        case 3216: return !compute && shared_bytes<32, 16, false>(L, k, Lp) != 0;
        case 3232: return !compute && shared_bytes<32, 32, false>(L, k, Lp) != 0;
    }
    return false;
}

cudaError_t launch_prune(const PruneDev &d, const PruneHost &h, int sms, cudaStream_t s)
{
    const PruneShape sh = prune_shape(d.L, d.k);
    switch (sh.G * 100 + sh.P) {
#define PP_CASE(g, p) \
    case g * 100 + p: return h.Wp ? launch_shape<g, p, true>(d, h, sms, s) : launch_shape<g, p, false>(d, h, sms, s);
        PP_SHAPES(PP_CASE)
#undef PP_CASE
        case 3216: return launch_shape<32, 16, false>(d, h, sms, s);
        case 3232: return launch_shape<32, 32, false>(d, h, sms, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace pp
